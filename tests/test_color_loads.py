"""The color kernels read what the kernel in front of them writes, and may be
resident while it still runs: nothing of it over the read-only path, whose data
must be constant for a kernel's whole life.  Checked in the sources (the two
functions that every color kernel calls), since results do not show it."""
import os
import re

import pytest

from paper_2605_30878_gb300 import build


def _after_wait(file, name):
    with open(os.path.join(build.CSRC, file)) as f:
        s = f.read()
    start = s.index("__forceinline__ void %s(" % name)
    body = s[start:s.index("\n}\n", start)]
    assert body.count("pdl_wait();") == 1
    return body.split("{", 1)[0], body.split("pdl_wait();")[1]


@pytest.mark.parametrize("file,name", [("lbm_kernels.cuh", "phi_node"), ("lbm_kernels_pair.cuh", "phi_pair")])
def test_color_kernels_load_populations_fresh(file, name):
    head, body = _after_wait(file, name)
    assert "__restrict__ Bst" not in head
    assert "__ldg" not in body and "Ld::Constant" not in body
    loads = re.findall(r"\b(?:PS::(?:template )?(?:load_\w+|accumulate)|pull_pair|ld)\b[^(]*\(", body)
    assert len(loads) == 2 and all("Ld::Fresh" in x for x in loads), loads
    assert not re.search(r"[=+]\s*\*", body), "a plain dereference on the right-hand side"


@pytest.mark.parametrize("entry,launch", [("lbm_profile_steps", "launch_one_step("), ("lbm_batch_tune", "batch_launch_step(")])
def test_steps_launched_without_a_graph_wait_for_the_state(entry, launch):
    """The step kernels read N over the read-only path: the kernel that wrote the
    first step's N must have completed before one can be resident."""
    with open(os.path.join(build.CSRC, "lbm_api.cu")) as f:
        s = f.read()
    start = s.index("lbm_status %s(" % entry)
    assert "cudaStreamSynchronize(" in s[start:s.index(launch, start)]
