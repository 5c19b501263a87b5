// Two-node step and color kernels (float arithmetic, FP32 or FP16 population
// storage).
//
// Every thread updates the two x-adjacent nodes A = (x0 + 2t, y, z) and
// B = (x0 + 2t + 1, y, z) of its row, with the arithmetic of k_step and k_color:
// the same sums in the same order and NodeUpdate's per-node update, so the
// kernels round alike.  What bounds them on 192^3 (D3Q19, one GB300): with FP32
// the DRAM (step 196 bytes per fluid node in 192 us, 7.1 TB/s; color 108 bytes
// in 120 us, 6.3 TB/s), with FP16 storage instruction issue and latency (step
// 124 bytes in 145 us, color 72 bytes in 102 us; ~1000 and ~620 instructions per
// warp of 64 nodes).  Since A's index is even, the pair shares
//   - its mask (one 8-byte load),
//   - its streaming pulls along y and z (one two-wide load per direction with
//     c_x = 0; directions with c_x != 0 pull from odd offsets, two loads),
//   - its shared-memory stencil values (two-wide loads; the rows a +/- x
//     direction needs come from three aligned two-wide loads, shared by the
//     directions of that row; values at odd offsets enter by scalar operations,
//     see H2),
//   - its stores of N*, f, u and p (one two-wide store each),
// which halves the load/store and address instructions per node of the
// one-node kernel.  The float arithmetic of the two nodes runs on packed
// pairs (NodeUpdate<..., F2>: one add/mul/fma.f32x2 for both nodes, each lane
// rounded as the one-node kernel's scalar operation), which halves the float
// instructions too.  Blocks are TX/2 x TY x TZ threads covering TX x TY x TZ
// nodes; the halo tile is copied by the same halo_issue/halo_complete as
// k_step's (TMA boxes (TX + 8) x (TY + 2) x (TZ + 2) on interior tiles).  A node of
// the pair that is not fluid gets zero velocity and pressure; its population
// slots receive values that nothing reads (every pull of a fluid node reads
// fluid sources or its own slots, as the diagnostics and state transfer do).
#pragma once

#include "lbm_kernels.cuh"

namespace lbmgpu {

// TXn nodes along x (64: the single-domain kernel and batch shape 5; 32:
// batch shapes 0 and 3, narrower tiles for small domains' ragged x ends) and
// TYn along y (0: 4 in 2D, 2 in 3D; batch shape 0 takes 8 and 4)
template <int Q, int TXn = 64, int TYn = 0>
struct PairTile {
    static constexpr int D = Lattice<Q>::D;
    static constexpr int BX = TXn / 2;             // threads along x
    static constexpr int TX = TXn;                 // nodes along x
    static constexpr int TY = TYn ? TYn : (D == 2 ? 4 : 2);
    static constexpr int TZ = D == 2 ? 1 : 2;
    static constexpr int XO = 4;                   // halo origin x0 - 4: 16-byte aligned for tiled copies
    static constexpr int HX = TX + 2 * XO;
    static constexpr int HY = TY + 2;
    static constexpr int HZ = D == 2 ? 1 : TZ + 2;
    static constexpr int HN = HX * HY * HZ;
    static constexpr int THREADS = BX * TY * TZ;
    __host__ __device__ static constexpr int off(int cx, int cy, int cz) { return cx + HX * (cy + HY * cz); }
};

// 32 nodes wide, as batch shape 0.
template <int Q> using NarrowTile = PairTile<Q, 32, Q == 9 ? 8 : 4>;

// Resident blocks per SM the pair kernel is compiled for (registers per thread
// <= 65536 / (THREADS * blocks)): 7 with density contrast (72 registers), 8
// without (64).  us per step with 6, 7 and 8: 192^3 FP16 storage 255, 250, 255
// and FP32 316, 317, 317, twelve 3D domains, both kinds, 304, 294, 291, 128^3
// packing (no contrast) 107.9, 108.0, 106.7.
template <bool CONTRAST, int THREADS = 128> struct PairBlocks {
    static constexpr int value = (CONTRAST ? 7 : 8) * 128 / THREADS;
};

// The values at halo slots hc + o and hc + o + 1 (hc even): one aligned
// two-wide load for even o, else the odd half of the pair below and the even
// half of the pair above (loads of the same address are shared by the compiler
// across directions).
template <int HN>
__device__ __forceinline__ H2 halo_pair(const float* s, int hc, int o, int* err) {
    if ((o & 1) == 0) return {*reinterpret_cast<const float2*>(s + idx_checked(hc + o, HN - 1, err)), false};
    const float2 lo = *reinterpret_cast<const float2*>(s + idx_checked(hc + o - 1, HN - 1, err));
    const float2 hi = *reinterpret_cast<const float2*>(s + idx_checked(hc + o + 1, HN - 1, err));
    return {make_float2(lo.y, hi.x), true};
}

// The pair of nodes of a thread: A = (xa, y, z) and B = (xa + 1, y, z), their
// bounce-back masks (one 8-byte load).
struct PairNode {
    int xa, y, z, nodeA;
    bool in_grid, b_in;                            // A in the grid; B too (it may be a padding column)
    bool fluidA, fluidB;
    uint2 m;
    __device__ __forceinline__ PairNode(const StepParams<float>& P, const uint32_t* __restrict__ mask, int x0, int y0,
                                        int z0, int* err) {
        xa = x0 + 2 * threadIdx.x;
        y = y0 + threadIdx.y;
        z = z0 + threadIdx.z;
        in_grid = xa < P.nx && y < P.ny && z < P.nz;
        b_in = in_grid && xa + 1 < P.nx;
        nodeA = in_grid ? idx_checked(xa + P.px * (y + P.ny * z), P.plane - 1, err) : 0;
        m = make_uint2(MASK_NOT_FLUID, MASK_NOT_FLUID);
        if (in_grid) m = __ldg(reinterpret_cast<const uint2*>(mask + nodeA));
        fluidA = !(m.x & MASK_NOT_FLUID);
        fluidB = !(m.y & MASK_NOT_FLUID);
    }
};

// The pair's moving populations after streaming, in storage units (the
// deviation form never reads N[0]).
template <int Q, typename S>
__device__ __forceinline__ void pull_pair(const StepParams<float>& P, const S* __restrict__ N, const PairNode& pn,
                                          float (&NA)[Q], float (&NB)[Q], int* err) {
    using L = Lattice<Q>;
    using PS = PopStore<S>;
    const int pl = (int)P.plane, nodeA = pn.nodeA;
    const auto* mv = PS::moving(N, pl);
    NA[0] = NB[0] = 0.f;
    if (!pn.in_grid) return;
    const Wrap W(pn.xa, pn.y, pn.z, P.nx, P.ny, P.nz, P.px);
    // the column A pulls from x - 1, and the one the pair's last node pulls from
    // x + 1, relative to A (B's left neighbour is A, A's right one B)
    const int dl = W.xm, dr = pn.b_in ? (pn.xa + 2 == P.nx ? 2 - P.nx : 2) : W.xp;
    auto at = [&](int node) { return mv + pop_at<Q>(idx_checked(node, P.plane, err)); };
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const int cx = L::cx(i), cy = L::cy(i), cz = L::cz(i);
        const int row = nodeA + W.off(0, -cy, -cz);
        if (cx == 0) {
            const float2 v = PS::load_units2(at(row), pop_dir(i));
            NA[i] = v.x;
            NB[i] = v.y;
        } else if (cx > 0) {
            NA[i] = (float)PS::load_units(at(row + dl), pop_dir(i));
            NB[i] = (float)PS::load_units(at(row), pop_dir(i));
        } else {
            const float v = (float)PS::load_units(at(row), pop_dir(i) + 1);      // B's column: A is even
            NB[i] = (float)PS::load_units(at(row + dr), pop_dir(i));
            NA[i] = pn.b_in ? v : NB[i];
        }
    }
    // halfway bounce-back: directions whose neighbour is not fluid read the node's own opposite slot
    if (pn.fluidA && (pn.m.x & MASK_DIRS)) {
#pragma unroll
        for (int i = 1; i < Q; ++i)
            if ((pn.m.x >> i) & 1u) NA[i] = (float)PS::load_units(at(nodeA), pop_dir(L::opp(i)));
    }
    if (pn.fluidB && (pn.m.y & MASK_DIRS)) {
#pragma unroll
        for (int i = 1; i < Q; ++i)
            if ((pn.m.y >> i) & 1u) NB[i] = (float)PS::load_units(at(nodeA), pop_dir(L::opp(i)) + 1);
    }
}

// Whole sectors (FP32 storage): a pair without a fluid node writes zeros to
// its slots (nodeP, its first node; -1: outside the padded rows) when another
// pair of its group of 8 nodes (32 bytes, one sector of every plane, since
// planes start at multiples of 64 nodes) stores its update.  The L2 then writes
// back whole sectors, where a partly written one would first be read from DRAM
// (a batch of 64 domains of 48^3 to 128^3: 10% less DRAM read per step kernel
// launch, 6% faster).  Nothing reads these slots: a fluid node pulls from fluid
// nodes or its own slots, and u, p stay 0 at nodes that are not fluid.  With
// FP16 storage the extra instructions cost more than the traffic saved (its
// k_step is issue-bound: 0.77 of its roofline with the fill, 0.80 without).
// Every lane of the warp calls it.
template <int Q, typename S>
__device__ __forceinline__ void fill_sectors(const StepParams<float>& P, const StepBuffers<float, S>& b, int nodeP,
                                             bool stores, bool ok) {
    if constexpr (sizeof(S) == 4) {
        using PS = PopStore<S>;
        constexpr int kGroupShift = 3;
        unsigned lane;
        asm("mov.u32 %0, %%laneid;" : "=r"(lane));
        const int group = nodeP >= 0 ? (nodeP >> kGroupShift) : -1 - (int)lane;
        const unsigned same = __match_any_sync(0xffffffffu, group);
        const unsigned writers = __ballot_sync(0xffffffffu, stores);
        if (!stores && nodeP >= 0 && ok && (same & writers) && idx_ok(nodeP, P.plane - 1, b.err)) {
            const int pl = (int)P.plane;
            auto* __restrict__ Nm = PS::moving(b.Nout, pl) + pop_at<Q>(nodeP);
#pragma unroll
            for (int i = 1; i < Q; ++i) PS::store_zero2(Nm + pop_dir(i));
            const float2 zero = make_float2(0.f, 0.f);
            *reinterpret_cast<float2*>(PS::rest(b.Nout) + nodeP) = zero;
#pragma unroll
            for (int a = 0; a < Lattice<Q>::D; ++a) {
                *reinterpret_cast<float2*>(b.u_out + a * pl + nodeP) = zero;
                *reinterpret_cast<float2*>(b.flux + a * pl + nodeP) = zero;
            }
            *reinterpret_cast<float2*>(b.p + nodeP) = zero;
        }
    }
}

// The update of a pair whose moments n2 holds, and its stores: stencils of the
// color ph(cx, cy, cz) and the previous velocity us(a, cx, cy, cz) at the
// pair's lattice neighbours, over +/- pairs in the order of k_step.
template <int Q, typename S, bool CONTRAST, class Node, class PhiAt, class VelAt>
__device__ __forceinline__ void pair_update(const StepParams<float>& P, const StepBuffers<float, S>& b, Node& n2,
                                            int nodeA, bool fluidA, bool fluidB, PhiAt phi_at, VelAt u_at) {
    using L = Lattice<Q>;
    using PS = PopStore<S>;
    constexpr int D = L::D;
    const int pl = (int)P.plane;
    const F2 ph = phi_at(0, 0, 0);
    F2 g[3] = {F2(0.f), F2(0.f), F2(0.f)}, lap(0.f);
    F2 du[3][3] = {{F2(0.f), F2(0.f), F2(0.f)}, {F2(0.f), F2(0.f), F2(0.f)}, {F2(0.f), F2(0.f), F2(0.f)}};
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        if (L::opp(i) < i) continue;
        const int cx = L::cx(i), cy = L::cy(i), cz = L::cz(i);
        const float wi = float(3.0 * L::w(i)), wl = float(6.0 * L::w(i));   // grad: 3 w_i, lap: 6 w_i
        const auto pp = phi_at(cx, cy, cz), pm = phi_at(-cx, -cy, -cz);
        const F2 dphi = pp - pm;
        if (cx) g[0] = fma(F2(float(cx) * wi), dphi, g[0]);
        if (cy) g[1] = fma(F2(float(cy) * wi), dphi, g[1]);
        if (cz) g[2] = fma(F2(float(cz) * wi), dphi, g[2]);
        lap = fma(F2(wl), (pp - ph) + (pm - ph), lap);
        if (CONTRAST) {
#pragma unroll
            for (int bb = 0; bb < D; ++bb) {
                const F2 dub = u_at(bb, cx, cy, cz) - u_at(bb, -cx, -cy, -cz);
                if (cx) du[0][bb] = fma(F2(float(cx) * wi), dub, du[0][bb]);
                if (cy) du[1][bb] = fma(F2(float(cy) * wi), dub, du[1][bb]);
                if (cz) du[2][bb] = fma(F2(float(cz) * wi), dub, du[2][bb]);
            }
        }
    }
    n2.compute(P, ph, g, lap, du);

    // u and p of the pair in one store per field; 0 at a node that is not fluid
    // (the velocity halo reads 0 at solid nodes)
#pragma unroll
    for (int a = 0; a < D; ++a) {
        *reinterpret_cast<float2*>(b.u_out + a * pl + nodeA) =
            make_float2(fluidA ? n2.u[a].lo() : 0.f, fluidB ? n2.u[a].hi() : 0.f);
        const F2 f = n2.kflux * n2.gp[a];
        *reinterpret_cast<float2*>(b.flux + a * pl + nodeA) = make_float2(f.lo(), f.hi());
    }
    *reinterpret_cast<float2*>(b.p + nodeA) = make_float2(fluidA ? n2.p.lo() : 0.f, fluidB ? n2.p.hi() : 0.f);
    if ((fluidA && !(n2.uu.lo() < 1e30f)) || (fluidB && !(n2.uu.hi() < 1e30f))) atomicOr(b.err, kErrNonFinite);

    float sNA = 0.f, sNB = 0.f;                             // moving populations as stored (FP16 storage)
    auto* __restrict__ Nmov = PS::moving(b.Nout, pl) + pop_at<Q>(nodeA);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        if (L::opp(i) < i) continue;
        const int o = L::opp(i);
        F2 ni, no;
        n2.dir(i, ni, no);
        PS::store_units2(Nmov, pop_dir(i), ni.lo(), ni.hi(), sNA, sNB);
        PS::store_units2(Nmov, pop_dir(o), no.lo(), no.hi(), sNA, sNB);
    }
    float2 rn;
    if constexpr (PS::kExact) {
        const F2 n0 = n2.rest_N(P);
        rn = make_float2(n0.lo(), n0.hi());
    } else {
        rn = make_float2(Node::rest_N_from_sum(sNA), Node::rest_N_from_sum(sNB));
    }
    *reinterpret_cast<float2*>(PS::rest(b.Nout) + nodeA) = rn;
}

// The pair tile at (x0, y0, z0); maps != nullptr: tiled halo copies (the
// caller checked the tile needs no periodic image in y and z and initialised
// the barrier).
template <int Q, typename S, bool CONTRAST, int TXn = 64, int TYn = 0>
__device__ __forceinline__ void step_pair_tile(const StepParams<float>& P, const StepBuffers<float, S>& b,
                                               float* s_phi, float* s_u, int x0, int y0, int z0,
                                               const CUtensorMap* tm_phi, const CUtensorMap* tm_u,
                                               uint64_t* bar) {
    using Tl = PairTile<Q, TXn, TYn>;
    constexpr int D = Lattice<Q>::D;
    constexpr bool kUnits = !PopStore<S>::kExact;
    int* const err = b.err;
    const bool interior = tm_phi != nullptr;
    const PairNode pn(P, b.mask, x0, y0, z0, err);
    pdl_wait();
    HaloFix<Tl, float, CONTRAST> fx;
    if (!halo_issue<Tl, float, CONTRAST>(P, b.phi, b.u_in, err, s_phi, s_u, x0, y0, z0, tm_phi, tm_u, bar, fx)) return;

    // the pair's populations, pulled while the halo is in flight
    const bool fluidA = pn.fluidA, fluidB = pn.fluidB;
    const int nodeA = pn.nodeA, xa = pn.xa, y = pn.y, z = pn.z;
    float NA[Q], NB[Q];
    pull_pair<Q, S>(P, b.Nin, pn, NA, NB, err);
    // the moments of both nodes (one packed lane each) while the halo copy
    // completes; the pulled values are then dead, which keeps them out of the
    // registers the stencils need
    NodeUpdate<Q, kUnits, CONTRAST, F2> n2;
    {
        F2 N2[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) N2[i] = F2(NA[i], NB[i]);
        n2.moments(N2);
    }
    const bool halo_ok = halo_complete<Tl, float>(err, interior, bar, s_phi, s_u, fx);
    __syncthreads();
    fill_sectors<Q, S>(P, b, xa < P.px && y < P.ny && z < P.nz ? xa + P.px * (y + P.ny * z) : -1, fluidA || fluidB, halo_ok);
    if (!(fluidA || fluidB) || !halo_ok) return;

    // isotropic stencils of both nodes, over +/- pairs in the order of k_step
    const int hcA = (2 * threadIdx.x + Tl::XO) + Tl::HX * ((threadIdx.y + 1) + Tl::HY * (D == 2 ? 0 : threadIdx.z + 1));
    auto ph = [&](int cx, int cy, int cz) { return halo_pair<Tl::HN>(s_phi, hcA, Tl::off(cx, cy, cz), err); };
    auto us = [&](int a, int cx, int cy, int cz) {
        return halo_pair<D * Tl::HN>(s_u, hcA + a * Tl::HN, Tl::off(cx, cy, cz), err);
    };
    pair_update<Q, S, CONTRAST>(P, b, n2, nodeA, fluidA, fluidB, ph, us);
}

// The color tile at (x0, y0, z0), two nodes per thread, packed: color_tile's
// arithmetic.  Warps without a bounce-back direction skip its selects.
template <int Q, typename S, int TXn = 64, int TYn = 0>
__device__ __forceinline__ void color_pair_tile(const StepParams<float>& P, const StepBuffers<float, S>& b,
                                                float* s_phi, float* s_f, int x0, int y0, int z0, int early,
                                                const CUtensorMap* tm_phi, const CUtensorMap* tm_f, uint64_t* bar) {
    using Tl = PairTile<Q, TXn, TYn>;
    using L = Lattice<Q>;
    using PS = PopStore<S>;
    constexpr int D = L::D;
    int* const err = b.err;
    const PairNode pn(P, b.mask, x0, y0, z0, err);
    pdl_wait();
    if (early) pdl_trigger();
    HaloFix<Tl, float, true> fx;
    if (!halo_issue<Tl, float, true>(P, b.phi, b.flux, err, s_phi, s_f, x0, y0, z0, tm_phi, tm_f, bar, fx)) return;
    float NA[Q], NB[Q];
    pull_pair<Q, S>(P, b.Nout, pn, NA, NB, err);
    const S* const Ncst = b.Nout;
    float2 n0 = make_float2(0.f, 0.f);
    float2 lov = n0;
    if (pn.in_grid) {
        n0 = PS::load_rest2(PS::rest(Ncst), pn.nodeA);
        lov = *reinterpret_cast<const float2*>(b.phi_lo + pn.nodeA);
    }
    const bool halo_ok = halo_complete<Tl, float>(err, tm_phi != nullptr, bar, s_phi, s_f, fx);
    __syncthreads();
    const uint32_t bounce = ((pn.fluidA ? pn.m.x : 0u) | (pn.fluidB ? pn.m.y : 0u)) & MASK_DIRS;
    const bool any_bounce = __any_sync(0xffffffffu, bounce != 0u);
    if (!pn.in_grid || !halo_ok) return;
    const int hc = (2 * threadIdx.x + Tl::XO) + Tl::HX * ((threadIdx.y + 1) + Tl::HY * (D == 2 ? 0 : threadIdx.z + 1));
    const float2 phv = halo_pair<Tl::HN>(s_phi, hc, 0, err).v;
    float2 out = make_float2(phv.x, pn.b_in ? phv.y : 0.f);     // not fluid: kept
    if (pn.fluidA || pn.fluidB) {
        F2 N2[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) N2[i] = F2(NA[i], NB[i]);
        const F2 phi(phv.x, phv.y), rest(n0.x, n0.y);
        F2 r, lo(lov.x, lov.y);
        if (!any_bounce) {
            auto ph = [&](int i) {
                return halo_pair<Tl::HN>(s_phi, hc, -Tl::off(L::cx(i), L::cy(i), L::cz(i)), err);
            };
            auto fl = [&](int i, int a) {
                return halo_pair<D * Tl::HN>(s_f, hc + a * Tl::HN, -Tl::off(L::cx(i), L::cy(i), L::cz(i)), err);
            };
            r = color_update<Q, !PS::kExact, F2>(P, phi, rest, N2, ph, fl, lo);
        } else {
            auto ph = [&](int i) {
                const float2 v = halo_pair<Tl::HN>(s_phi, hc, -Tl::off(L::cx(i), L::cy(i), L::cz(i)), err).v;
                return F2((pn.m.x >> i) & 1u ? phv.x : v.x, (pn.m.y >> i) & 1u ? phv.y : v.y);
            };
            auto fl = [&](int i, int a) {
                const float2 v = halo_pair<D * Tl::HN>(s_f, hc + a * Tl::HN, -Tl::off(L::cx(i), L::cy(i), L::cz(i)), err).v;
                const float2 own = halo_pair<D * Tl::HN>(s_f, hc + a * Tl::HN, 0, err).v;
                return F2((pn.m.x >> i) & 1u ? -own.x : v.x, (pn.m.y >> i) & 1u ? -own.y : v.y);
            };
            r = color_update<Q, !PS::kExact, F2>(P, phi, rest, N2, ph, fl, lo);
        }
        if (pn.fluidA) out.x = r.lo();
        if (pn.fluidB) out.y = r.hi();
        *reinterpret_cast<float2*>(b.phi_lo + pn.nodeA) = make_float2(lo.lo(), lo.hi());
    }
    *reinterpret_cast<float2*>(b.phi_out + pn.nodeA) = out;
}

template <int Q, typename S, bool CONTRAST, int TXn, int TYn>
__global__ void __launch_bounds__(PairTile<Q, TXn, TYn>::THREADS, PairBlocks<CONTRAST>::value)
    k_step_pair(StepParams<float> P, StepBuffers<float, S> b, const __grid_constant__ CUtensorMap tm_phi,
                const __grid_constant__ CUtensorMap tm_u, int tma) {
    using Tl = PairTile<Q, TXn, TYn>;
    constexpr int D = Tl::D;
    __shared__ __align__(128) float s_phi[Tl::HN];
    __shared__ __align__(128) float s_u[CONTRAST ? D * Tl::HN : 2];
    __shared__ __align__(8) uint64_t s_bar;
    const int x0 = blockIdx.x * Tl::TX, y0 = blockIdx.y * Tl::TY, z0 = blockIdx.z * Tl::TZ;
    // tiles whose halo needs no periodic image in y and z (x images are patched)
    const bool interior = tma && y0 >= 1 && y0 + Tl::TY + 1 <= P.ny &&
                          (D == 2 || (z0 >= 1 && z0 + Tl::TZ + 1 <= P.nz));
    if (interior) {
        if (threadIdx.x + threadIdx.y + threadIdx.z == 0) mbar_init(&s_bar, 1);
        __syncthreads();                                      // the barrier exists before anyone waits on it
    }
    step_pair_tile<Q, S, CONTRAST, TXn, TYn>(P, b, s_phi, s_u, x0, y0, z0, interior ? &tm_phi : nullptr, &tm_u, &s_bar);
}

// Resident blocks per SM of the color kernel: 8 (64 registers).  With 6, 7, 8:
// 192^3 FP32 130, 122, 119 us per launch, FP16 storage 103, 101, 97.
template <int THREADS = 128> struct ColorBlocks { static constexpr int value = 8 * 128 / THREADS; };

template <int Q, typename S, int TXn, int TYn>
__global__ void __launch_bounds__(PairTile<Q, TXn, TYn>::THREADS, ColorBlocks<>::value)
    k_color_pair(StepParams<float> P, StepBuffers<float, S> b, const __grid_constant__ CUtensorMap tm_phi,
                 const __grid_constant__ CUtensorMap tm_f, int tma, int early) {
    using Tl = PairTile<Q, TXn, TYn>;
    constexpr int D = Tl::D;
    __shared__ __align__(128) float s_phi[Tl::HN];
    __shared__ __align__(128) float s_f[D * Tl::HN];
    __shared__ __align__(8) uint64_t s_bar;
    // tiles in the reverse of k_step_pair's order, as k_color
    const int x0 = (gridDim.x - 1 - blockIdx.x) * Tl::TX, y0 = (gridDim.y - 1 - blockIdx.y) * Tl::TY,
              z0 = (gridDim.z - 1 - blockIdx.z) * Tl::TZ;
    const bool interior = tma && y0 >= 1 && y0 + Tl::TY + 1 <= P.ny &&
                          (D == 2 || (z0 >= 1 && z0 + Tl::TZ + 1 <= P.nz));
    if (interior) {
        if (threadIdx.x + threadIdx.y + threadIdx.z == 0) mbar_init(&s_bar, 1);
        __syncthreads();
    }
    color_pair_tile<Q, S, TXn, TYn>(P, b, s_phi, s_f, x0, y0, z0, early, interior ? &tm_phi : nullptr, &tm_f, &s_bar);
}

// Batched form: one pair tile of one domain per block, the domain's
// parameters in its constant-memory slot (as k_step_batched): 64 nodes wide
// for tile shape 5, 32 for tile shapes 0 and 3.
template <int Q, typename S, bool CONTRAST, int TXn = 64, int TYn = 0>
__global__ void __launch_bounds__(PairTile<Q, TXn, TYn>::THREADS,
                                  (PairBlocks<CONTRAST, PairTile<Q, TXn, TYn>::THREADS>::value))
    k_step_pair_batched(const int4* __restrict__ tiles, const CUtensorMap* __restrict__ maps, int parity) {
    using Tl = PairTile<Q, TXn, TYn>;
    constexpr int D = Tl::D;
    __shared__ __align__(128) float s_phi[Tl::HN];
    __shared__ __align__(128) float s_u[CONTRAST ? D * Tl::HN : 2];
    __shared__ __align__(8) uint64_t s_bar;
    const int4 t = __ldg(tiles + blockIdx.x);          // {slot, x0, y0, z0}
    const BatchEntry<float, S>& e = c_batch<float, S>[idx_checked(t.x, kBatchSlots, c_batch<float, S>[0].b[0].err)];
    const int y0 = t.z, z0 = t.w;
    if (kDebugBounds && !(idx_ok(t.y, e.P.nx, e.b[0].err) && idx_ok(y0, e.P.ny, e.b[0].err) &&
                          idx_ok(z0, e.P.nz, e.b[0].err))) {
        pdl_wait();
        return;                                         // a tile outside its domain
    }
    const bool tma = maps != nullptr && e.tma && y0 >= 1 && y0 + Tl::TY + 1 <= e.P.ny &&
                     (D == 2 || (z0 >= 1 && z0 + Tl::TZ + 1 <= e.P.nz));
    if (tma) {
        if (threadIdx.x + threadIdx.y + threadIdx.z == 0) mbar_init(&s_bar, 1);
        __syncthreads();                                      // the barrier exists before anyone waits on it
    }
    step_pair_tile<Q, S, CONTRAST, TXn, TYn>(e.P, e.b[parity], s_phi, s_u, t.y, y0, z0,
                                             tma ? slot_phi_map(maps, t.x, parity) : nullptr,
                                             slot_u_map(maps, t.x, parity), &s_bar);
}

template <int Q, typename S, int TXn = 64, int TYn = 0>
__global__ void __launch_bounds__(PairTile<Q, TXn, TYn>::THREADS, (ColorBlocks<PairTile<Q, TXn, TYn>::THREADS>::value))
    k_color_pair_batched(const int4* __restrict__ tiles, const CUtensorMap* __restrict__ maps, int parity, int early) {
    using Tl = PairTile<Q, TXn, TYn>;
    constexpr int D = Tl::D;
    __shared__ __align__(128) float s_phi[Tl::HN];
    __shared__ __align__(128) float s_f[D * Tl::HN];
    __shared__ __align__(8) uint64_t s_bar;
    const int4 t = __ldg(tiles + (gridDim.x - 1 - blockIdx.x));     // reverse order, as k_color
    const BatchEntry<float, S>& e = c_batch<float, S>[idx_checked(t.x, kBatchSlots, c_batch<float, S>[0].b[0].err)];
    const int y0 = t.z, z0 = t.w;
    if (kDebugBounds && !(idx_ok(t.y, e.P.nx, e.b[0].err) && idx_ok(y0, e.P.ny, e.b[0].err) &&
                          idx_ok(z0, e.P.nz, e.b[0].err))) {
        pdl_wait();
        return;                                         // a tile outside its domain
    }
    const bool tma = maps != nullptr && e.tma && y0 >= 1 && y0 + Tl::TY + 1 <= e.P.ny &&
                     (D == 2 || (z0 >= 1 && z0 + Tl::TZ + 1 <= e.P.nz));
    if (tma) {
        if (threadIdx.x + threadIdx.y + threadIdx.z == 0) mbar_init(&s_bar, 1);
        __syncthreads();
    }
    color_pair_tile<Q, S, TXn, TYn>(e.P, e.b[parity], s_phi, s_f, t.y, y0, z0, early,
                                    tma ? slot_phi_map(maps, t.x, parity) : nullptr, slot_flux_map(maps, t.x), &s_bar);
}

}  // namespace lbmgpu
