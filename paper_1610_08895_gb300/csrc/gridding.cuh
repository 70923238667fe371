// Device helpers shared by the two forms of the interpolation G: weights evaluated in
// the kernels (gridding.cu) and G stored as a sparse matrix (gridding_csr.cu).
#pragma once
#include "common.cuh"
#include "plan.hpp"

namespace pdgb {

// The J tap weights phi(frac + J/2 - 1 - a) of one axis, from the plan's per-tap Chebyshev
// interpolants in x = 2 frac - 1 (FP32: degree 10, interpolation error ~3e-11 of phi(0);
// FP64: degree 18, fitted in extended precision, below 1e-17 of phi(0)). phi is even, so tap
// J-1-a is tap a at -x: with the polynomial split into even and odd parts p = E(x^2) + x O(x^2),
// one pass gives both E + x O (tap a) and E - x O (tap J-1-a). In FP64, where the GPU has 1/64
// of its FP32 rate, the 8 x 2 evaluations of I0 were most of both kernels (phi_256_f64 of
// perf/cases.py: 8.4 ms with them, 4.7 ms with the polynomials).
template <typename R, int J>
__device__ __forceinline__ void kb_taps(R frac, R* w, R two_over_j, R beta, const kb_poly_t<R>& kp) {
    constexpr int DEG = sizeof(R) == 4 ? KB_DEG : KB_DEG64;
    if constexpr (sizeof(R) == 8) {
        if (!kp.use) {
#pragma unroll
            for (int a = 0; a < J; ++a) w[a] = kb_weight<R>(frac + R(J / 2 - 1 - a), two_over_j, beta);
            return;
        }
    }
    const R x = R(2) * frac - R(1), x2 = x * x;
    constexpr int OUT = sizeof(R) == 8 ? kb_outer(J) : 0;
    if constexpr (sizeof(R) == 8) {
        // FP64, outermost taps: the weight falls to 1e-7 of phi(0) and less there, so a fit that is
        // exact to phi(0) is not to the weight itself (1.7e-12 of it at J = 8). s = q (2 - q), q the
        // distance to the kernel's end in half-widths, has no cancellation at that end.
#pragma unroll
        for (int a = 0; a < OUT; ++a) {
            const double q0 = (a + 1 - frac) * two_over_j, q1 = (a + frac) * two_over_j;
            const double s0 = q0 * (2.0 - q0), s1 = q1 * (2.0 - q1);
            double w0 = kp.e[kb_edge_deg(J)], w1 = w0;
#pragma unroll
            for (int k = kb_edge_deg(J) - 1; k >= 0; --k) {
                w0 = fma(w0, s0, kp.e[k]);
                w1 = fma(w1, s1, kp.e[k]);
            }
            w[a] = w0;
            w[J - 1 - a] = w1;
        }
    }
#pragma unroll
    for (int a = OUT; a < J / 2; ++a) {
        R ev = kp.c[a][DEG], od = kp.c[a][DEG - 1];
#pragma unroll
        for (int k = DEG - 2; k >= 2; k -= 2) ev = fma(ev, x2, kp.c[a][k]);
#pragma unroll
        for (int k = DEG - 3; k >= 1; k -= 2) od = fma(od, x2, kp.c[a][k]);
        if constexpr (sizeof(R) == 4) {
            // the constant term last, with the part that its rounding left: one rounding of w
            ev = fma(ev, x2, kp.lo[a]);
            w[a] = kp.c[a][0] + fma(x, od, ev);
            w[J - 1 - a] = kp.c[a][0] + fma(-x, od, ev);
        } else {
            ev = fma(ev, x2, kp.c[a][0]);
            w[a] = fma(x, od, ev);
            w[J - 1 - a] = fma(-x, od, ev);
        }
    }
}

// ---------------------------------------------------------------- active segments
// Warp 0 lists the tile's segments whose block is active (all of them when active is
// null) in act_seg[0..nact) and the prefix sums of their lengths in act_pre[0..nact];
// returns nact to every thread (the caller syncs before use).
__device__ __forceinline__ void list_active_segments(int seg0, int nseg_t, const int32_t* __restrict__ seg_block,
                                                     const int32_t* __restrict__ active,
                                                     const int32_t* __restrict__ seg_start, int* act_seg,
                                                     int* act_pre, int* nact_out) {
    if ((threadIdx.x >> 5) != 0) return;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    int nact = 0, total = 0;
    for (int base = 0; base < nseg_t; base += 32) {
        const int k = base + lane;
        const bool ok = k < nseg_t && (active == nullptr || active[seg_block[seg0 + k]]);
        const int len = ok ? seg_start[seg0 + k + 1] - seg_start[seg0 + k] : 0;
        const unsigned bal = __ballot_sync(0xffffffffu, ok);
        int incl = len;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (ok) {
            const int pos = nact + __popc(bal & below);
            act_seg[pos] = seg0 + k;
            act_pre[pos] = total + incl - len;
        }
        total += __shfl_sync(0xffffffffu, incl, 31);
        nact += __popc(bal);
    }
    if (lane == 0) { act_pre[nact] = total; *nact_out = nact; }
}

// Cell (ky, kx) of F Z x from the half grid (columns 0 .. nx, column panels): the image
// is real, so the columns kx > nx are conj(b[-ky][-kx]).
template <typename C2>
__device__ __forceinline__ C2 half_grid_at(const C2* __restrict__ gh, int ky, int kx, const Geo& g) {
    if (kx <= g.nx) return gh[panel_off(ky, kx, g.Ky)];
    const C2 v = gh[panel_off((g.Ky - ky) & (g.Ky - 1), g.Kx - kx, g.Ky)];
    return mk<C2>(v.x, -v.y);
}

// ---------------------------------------------------------------- reductions
// Warp-level segmented sum: the lanes with ok add (a, b) to their local segment ls;
// lane 0 adds each segment's warp total into part[2 ls], part[2 ls + 1] (FP64 slots
// owned by this warp), always in the same order. The at most 32 terms of one warp are
// summed in the working precision A (a fixed shuffle tree of non-negative terms:
// relative error below 6 units of A's rounding), every sum above that in FP64.
template <typename A>
__device__ __forceinline__ void warp_seg_add(bool ok, int ls, A a, A b, double* part) {
    unsigned todo = __ballot_sync(0xffffffffu, ok);
    while (todo) {
        const int key = __shfl_sync(0xffffffffu, ls, __ffs(todo) - 1);
        const bool mine = ok && ls == key;
        const unsigned mask = __ballot_sync(0xffffffffu, mine);
        const A x = warp_sum(mine ? a : A(0)), y = warp_sum(mine ? b : A(0));
        if ((threadIdx.x & 31) == 0) { part[2 * key] += (double)x; part[2 * key + 1] += (double)y; }
        todo &= ~mask;
    }
}

// value of visibility m to grid: MODE 0 the input (user order); MODE 1 the dual change
// v_new - v_old with v_new = scale_i r (step 8), writing v_new.
template <typename R, int MODE>
__device__ __forceinline__ cplx_t<R> grid_value(int m, const cplx_t<R>* __restrict__ src,
                                                const cplx_t<R>* __restrict__ rbuf, cplx_t<R>* __restrict__ v,
                                                const int32_t* __restrict__ perm, R sc) {
    if (MODE == 0) return vis_conj(perm[m], src[vis_index(perm[m])]);
    const cplx_t<R> r = rbuf[m], vo = v[m];
    const cplx_t<R> vn = cscale(r, sc);
    v[m] = vn;
    return csub(vn, vo);
}

// U += the tile's E x E window (tile and halo, wrapped periodically), the window's value
// of cell (ey, ex) given by val(ey, ex). The U reads of a batch of cells go out together.
template <typename R, class V>
__device__ __forceinline__ void add_window(cplx_t<R>* __restrict__ U, int oy, int ox, const Geo& g, const V& val) {
    using C2 = cplx_t<R>;
    const int E = g.ext;
    constexpr int EB = 8;
    for (int i0 = threadIdx.x; i0 < E * E; i0 += EB * (int)blockDim.x) {
        C2 uo[EB];
        int64_t off[EB];
#pragma unroll
        for (int k = 0; k < EB; ++k) {
            const int i = i0 + k * (int)blockDim.x;
            off[k] = -1;
            if (i < E * E) {
                const int ey = i / E, ex = i - ey * E;
                off[k] = panel_off((oy + ey) & (g.Ky - 1), (ox + ex) & (g.Kx - 1), g.Ky);
                uo[k] = U[off[k]];
            }
        }
#pragma unroll
        for (int k = 0; k < EB; ++k) {
            if (off[k] < 0) break;
            const int i = i0 + k * (int)blockDim.x;
            const int ey = i / E, ex = i - ey * E;
            U[off[k]] = cadd(uo[k], val(ey, ex));
        }
    }
}

// Thread 0: the next item (claimed in order by whichever CTA is free) whose tile is on, into
// *it; its number w is returned (>= n * batch: none left). A batch goes image by image (image
// w / n) where G is evaluated: the visibilities are read or written in user order, at random, and
// one image's stay in the L2 cache meanwhile (eight images of 1024^2, 4.19M points each: Phi 1405 ->
// 837 us). Where G is stored the images of an item follow one another (image w % batch): its rows
// come from HBM once for all of them (four images of 512^2, 524,288 points, complex rows: Phi^H 467
// us, image by image 512).
template <bool STORED>
__device__ __forceinline__ int claim_item(int* sched, const TileItem* __restrict__ items, int n, int batch,
                                          const int32_t* __restrict__ tile_on, TileItem* it) {
    for (;;) {
        const int w = atomicAdd(sched, 1);
        if (w >= n * batch) return w;
        const TileItem t = items[STORED ? w / batch : w % n];
        if (tile_on && !tile_on[t.tile]) continue;
        *it = t;
        return w;
    }
}
// The same over a list of tiles.
template <bool STORED>
__device__ __forceinline__ int claim_tile(int* next, const int32_t* __restrict__ list, int n, int batch,
                                          const int32_t* __restrict__ tile_on) {
    for (;;) {
        const int w = atomicAdd(next, 1);
        if (w >= n * batch || !tile_on || tile_on[list[STORED ? w / batch : w % n]]) return w;
    }
}
// Thread 0 of each CTA at the end: the last one sets the counters back for the next launch on the
// same grid (the forward FFT sets them too).
__device__ __forceinline__ void leave_items(int* sched) {
    if (atomicAdd(sched + 1, 1) == (int)gridDim.x - 1) {
        sched[0] = 0;
        sched[1] = 0;
    }
}

#define PD_J_DISPATCH(J_, CALL)                          \
    switch (J_) {                                        \
        case 2: { constexpr int JJ = 2; CALL; } break;   \
        case 4: { constexpr int JJ = 4; CALL; } break;   \
        case 6: { constexpr int JJ = 6; CALL; } break;   \
        case 8: { constexpr int JJ = 8; CALL; } break;   \
        case 10: { constexpr int JJ = 10; CALL; } break; \
        case 12: { constexpr int JJ = 12; CALL; } break; \
        case 14: { constexpr int JJ = 14; CALL; } break; \
        case 16: { constexpr int JJ = 16; CALL; } break; \
        default: return cudaErrorInvalidValue;           \
    }

// G held as a sparse matrix (gridding_csr.cu), J <= 8: the same contracts as the
// on-the-fly launchers of gridding.cu, which hand over to these when the plan's
// g_mode is PD_G_CSR.
template <typename R, int J, int MODE>
cudaError_t launch_degrid_csr(const pd_plan* p, const cplx_t<R>* grid, cplx_t<R>* out, const DualArgs* a,
                              cudaStream_t s, int batch);
template <typename R, int J, int MODE>
cudaError_t launch_grid_csr(const pd_plan* p, const cplx_t<R>* src, const DualArgs* a, const int32_t* tiles,
                            const int32_t* count, cplx_t<R>* U, int* next_tile, cudaStream_t s, int batch);

}  // namespace pdgb
