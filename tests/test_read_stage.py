"""The pinned read-back stage against a stand-in for the CUDA runtime with two
devices: like the runtime, it records an event only on a stream of the event's
own device."""
import os
import subprocess

from paper_2605_30878_gb300 import build

PROGRAM = r'''
#include <cstdio>
#include <cstdlib>
#include "lbm_read_stage.h"
struct CUstream_st { int device; };
struct CUevent_st { int device; };
static int current = 0, memory = 0, events = 0, fail_events = 0;
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = current; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { current = d; return cudaSuccess; }
cudaError_t cudaStreamGetDevice(cudaStream_t s, int* d) { *d = s ? s->device : current; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = malloc(n); ++memory; return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); --memory; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    if (fail_events) { *e = nullptr; return cudaErrorMemoryAllocation; }
    *e = new CUevent_st{current}; ++events; return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete e; --events; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    return e->device == (s ? s->device : current) ? cudaSuccess : cudaErrorInvalidResourceHandle;
}
}
using lbmgpu::ReadStage;
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
    CUstream_st s0{0}, s1{1};
    for (int again = 0; again < 2; ++again)
        for (current = 0; current < 2;) {
            const int was = current;
            for (cudaStream_t s : {&s1, &s0, (cudaStream_t)nullptr}) {
                ReadStage& st = ReadStage::of(s);
                CHECK(st.ready());
                CHECK(current == was);
                for (cudaEvent_t e : st.landed) CHECK(cudaEventRecord(e, s) == cudaSuccess);
            }
            CHECK(memory == 2);
            CHECK(events == 4);
            if (was == 1) {
                ReadStage::release_all();
                CHECK(memory == 0 && events == 0 && current == was);
            }
            ++current;
        }
    current = 0;
    fail_events = 1;
    CHECK(!ReadStage::of(&s1).ready() && memory == 0 && events == 0);
    fail_events = 0;
    CHECK(ReadStage::of(&s1).ready());
    ReadStage::release_all();
    CHECK(memory == 0 && events == 0);
    return 0;
}
'''


def test_stage_belongs_to_the_device_of_the_stream(tmp_path):
    src, exe = tmp_path / "stage.cpp", tmp_path / "stage"
    src.write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())) or "/usr/local/cuda", "include")
    r = subprocess.run(["g++", "-std=c++17", "-I" + build.CSRC, "-I" + cuda, str(src), "-o", str(exe), "-pthread"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
