// Sparse interpolation G (degridding) and its adjoint G^T (gridding) with a
// separable J x J Kaiser-Bessel kernel evaluated on the fly (Sec. 2; the paper's
// experiments use 8 x 8 kernels, Sec. 5), fused with the data-fidelity dual
// update of Algorithm 1 step 8 (l2-ball projection, eq. proj-L2) and the
// gridding of the dual change for step 9.
//
// Visibilities are stored in (tile, block, super-cell, row, column) order of the first
// cell of their footprint: each (tile, block) pair is a contiguous segment. Per tile, the
// segments of active blocks are listed in shared memory and worked on as one
// concatenated range, so inactive blocks cost nothing and batches stay full. A point at
// continuous grid coordinate g has base cell floor(g) (kept mod K) and fraction g - floor(g) (working precision, computed in FP64 at plan
// time); its taps are the cells floor(g) - J/2 + 1 ... floor(g) + J/2 (mod K),
// with weight phi(fraction + J/2 - 1 - a) for tap a; what is stored is the first of them.
//
// Both directions work tile by tile (one CTA owns a T x T tile at a time) on the
// tile plus a halo of J - 1 cells after it:
// * degridding stages that window of F Z x (held as its half grid: the columns
//   kx <= nx, the others by conjugate symmetry) in shared memory and gathers from it;
// * gridding accumulates the window in shared memory and adds the whole window
//   (tile and halo) to U. The windows of two tiles of one colour (tile row and column
//   parity) are disjoint. In FP32 with J <= 8 (k_grid_mma) one launch takes the tiles colour
//   by colour and adds overlapping windows in the order of the tiles; the other kernels take
//   one launch per colour. Either way every cell's sum has a fixed order.
#include <algorithm>

#include "gridding.cuh"

namespace pdgb {

// ---------------------------------------------------------------- degridding
// The global inputs of one point to degrid (MODE 1 also its y and v).
template <typename R> struct DegridIn {
    cplx_t<R> yy, vv;
    R fx, fy;
    int c, m;
};

template <typename R, int MODE>
__device__ __forceinline__ void degrid_load(DegridIn<R>& in, int pos, int& j, const int* act_seg, const int* act_pre,
                                            const int32_t* __restrict__ seg_start, const int32_t* __restrict__ cell,
                                            const R* __restrict__ fxs, const R* __restrict__ fys,
                                            const cplx_t<R>* __restrict__ y, const cplx_t<R>* __restrict__ v) {
    while (act_pre[j + 1] <= pos) ++j;
    const int m = seg_start[act_seg[j]] + pos - act_pre[j];
    in.m = m;
    in.c = cell[m];
    in.fx = fxs[m];
    in.fy = fys[m];
    if (MODE == 1) {
        in.yy = y[m];
        in.vv = v[m];
    }
}

// Stage the E x E window of the half grid at (oy, ox) in shared memory (pitch EP, even) twice,
// the second copy (E * EP further) shifted left by one column. The window starts on a column
// panel, so a thread takes two cells (16 bytes) at a time, consecutive threads along a panel,
// with all of a thread's loads of a batch in flight.
__device__ __forceinline__ void stage_window_pairs(float2* win, const float2* __restrict__ gh, int oy, int ox, int E,
                                                   int EP, const Geo& g) {
    constexpr int UB = 2;
    const int per = 2 * E, slots = ((E + 3) >> 2) * per;       // slots of a panel: (row, half)
    for (int i0 = threadIdx.x; i0 < slots; i0 += UB * (int)blockDim.x) {
        float4 q[UB];
        int o[UB];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int i = i0 + u * (int)blockDim.x;
            const int pn = i / per, r = i - pn * per;
            const int ey = r >> 1, ex = 4 * pn + 2 * (r & 1);
            o[u] = i < slots && ex < E ? ey * EP + ex : -1;
            if (o[u] < 0) continue;
            const int ky = (oy + ey) & (g.Ky - 1), kx = (ox + ex) & (g.Kx - 1);
            if (kx < g.nx) {
                q[u] = *reinterpret_cast<const float4*>(gh + panel_off(ky, kx, g.Ky));
            } else {
                const float2 a = half_grid_at(gh, ky, kx, g), b = half_grid_at(gh, ky, kx + 1, g);
                q[u] = make_float4(a.x, a.y, b.x, b.y);
            }
        }
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            if (o[u] < 0) continue;
            *reinterpret_cast<float4*>(win + o[u]) = q[u];
            float2* w2 = win + E * EP + o[u];
            if (o[u] > 0) w2[-1] = make_float2(q[u].x, q[u].y);   // column 0 goes to the row above's spare slot
            w2[0] = make_float2(q[u].z, q[u].w);
        }
    }
}

// Bound by the shared-memory pipe (32 16-byte window reads a point). Four CTAs per SM: five
// leave 48 registers and spill (16.8M points, half active, 4096^2 grid: 222 us against 231;
// packed multiply-adds of the (re, im) pairs did not help either way: 238 us).
// MODE 0 (plain): out_user[perm[m]] = (G grid)_m for every visibility of the listed tiles.
// MODE 1 (pd): for visibilities of active blocks r = v + G b - y, with FP64 sums of
// ||r||^2 and ||G b - y||^2 per (tile, block) segment (per-warp slots, summed in warp order).
template <typename R, int J, int MODE>
__global__ void __launch_bounds__(256, J <= 8 ? (sizeof(R) == 4 ? 4 : 3) : 1) k_degrid(const cplx_t<R>* __restrict__ grid, cplx_t<R>* __restrict__ out,
                                                const cplx_t<R>* __restrict__ y, const cplx_t<R>* __restrict__ v,
                                                cplx_t<R>* __restrict__ rbuf, const int32_t* __restrict__ cell,
                                                const R* __restrict__ fxs, const R* __restrict__ fys,
                                                const int32_t* __restrict__ perm,
                                                const int32_t* __restrict__ seg_start,
                                                const int32_t* __restrict__ seg_block,
                                                const int32_t* __restrict__ active,
                                                const TileItem* __restrict__ items,
                                                const int32_t* __restrict__ nitems,
                                                const int32_t* __restrict__ tile_on, double* __restrict__ seg_part,
                                                int max_segs, Geo g, R two_over_j, R beta, const kb_poly_t<R> kp,
                                                int* __restrict__ sched, int batch, int64_t gstride,
                                                int64_t ostride) {
    using C2 = cplx_t<R>;
    extern __shared__ __align__(16) unsigned char smraw[];
    // FP32: the window twice, row stride EP (even), the second copy shifted left by one
    // column, so every footprint row is J/2 aligned 16-byte pairs in one of the copies.
    // FP64: one copy, row stride E.
    constexpr bool PAIRS = sizeof(R) == 4;
    const int EP = PAIRS ? ((g.ext + 2) & ~1) : g.ext;
    C2* win = reinterpret_cast<C2*>(smraw);                              // [ext][EP] (x2 in FP32)
    double* part = reinterpret_cast<double*>(win + (PAIRS ? 2 : 1) * g.ext * EP);  // [8 warps][max_segs][2]
    int* act_seg = reinterpret_cast<int*>(part + 16 * max_segs);        // [max_segs]
    int* act_pre = act_seg + max_segs;                                   // [max_segs + 1]
    __shared__ int nact_s, item_s;
    __shared__ TileItem ti_s;
    const int E = g.ext, T = g.tile;
    const int warp = threadIdx.x >> 5;
    const int n = *nitems;
    if (threadIdx.x == 0) item_s = claim_item<false>(sched, items, n, batch, tile_on, &ti_s);
    for (;;) {
        __syncthreads();
        const int w = item_s;
        if (w >= n * batch) break;
        const TileItem ti = ti_s;
        const int t = ti.tile, img = w / n;
        const cplx_t<R>* gimg = grid + (int64_t)img * gstride;
        cplx_t<R>* oimg = MODE == 0 ? out + (int64_t)img * ostride : out;
        const int ty = t / g.ntx, tx = t - ty * g.ntx;
        const int oy = ty * T, ox = tx * T;
        const int seg0 = ti.seg0, nseg_t = ti.nseg;
        list_active_segments(seg0, nseg_t, seg_block, MODE == 1 ? active : nullptr, seg_start, act_seg, act_pre,
                             &nact_s);
        if constexpr (PAIRS) {
            stage_window_pairs(win, gimg, oy, ox, E, EP, g);
        } else {
            for (int i = threadIdx.x; i < E * E; i += blockDim.x) {
                const int ey = i / E, ex = i - ey * E;
                win[ey * EP + ex] = half_grid_at(gimg, (oy + ey) & (g.Ky - 1), (ox + ex) & (g.Kx - 1), g);
            }
        }
        if (MODE == 1)
            for (int i = threadIdx.x; i < 16 * nseg_t; i += blockDim.x) part[i] = 0.0;
        __syncthreads();
        // this part's positions of the tile's active points
        const int nact = nact_s, all = act_pre[nact];
        const int first = (int)((int64_t)all * ti.part / ti.parts), total = (int)((int64_t)all * (ti.part + 1) / ti.parts);
        double* mypart = part + 2 * nseg_t * warp;
        int j = 0;   // segment cursor: positions only grow, so it only moves forward
        // the inputs of the point blockDim.x positions ahead are loaded while this one is worked on
        DegridIn<R> nx{};
        if (first + (int)threadIdx.x < total)
            degrid_load<R, MODE>(nx, first + threadIdx.x, j, act_seg, act_pre, seg_start, cell, fxs, fys, y, v);
        for (int base = first; base < total; base += blockDim.x) {
            const int pos = base + threadIdx.x;
            const bool ok = pos < total;
            const DegridIn<R> in = nx;
            const int jcur = j;
            if (pos + (int)blockDim.x < total)
                degrid_load<R, MODE>(nx, pos + blockDim.x, j, act_seg, act_pre, seg_start, cell, fxs, fys, y, v);
            R ar = R(0), ad = R(0);     // squares in the working precision (exact for FP64)
            if (ok) {
                const int m = in.m;
                R wx[J], wy[J];
                kb_taps<R, J>(in.fx, wx, two_over_j, beta, kp);
                kb_taps<R, J>(in.fy, wy, two_over_j, beta, kp);
                const int c = in.c;
                const int r0 = (c >> 16) - oy, c0 = (c & 0xFFFF) - ox;   // footprint origin in the window
                R sx = 0, sy = 0;
                if constexpr (PAIRS) {
                    const float4* bp = reinterpret_cast<const float4*>(
                        (c0 & 1) ? win + E * EP + r0 * EP + c0 - 1 : win + r0 * EP + c0);
#pragma unroll
                    for (int b = 0; b < J; ++b) {
                        R rx = 0, ry = 0;
#pragma unroll
                        for (int a = 0; a < J / 2; ++a) {
                            const float4 q = bp[(b * EP >> 1) + a];
                            rx += wx[2 * a] * q.x + wx[2 * a + 1] * q.z;
                            ry += wx[2 * a] * q.y + wx[2 * a + 1] * q.w;
                        }
                        sx += wy[b] * rx;
                        sy += wy[b] * ry;
                    }
                } else {
                    const C2* bp = win + r0 * EP + c0;
#pragma unroll
                    for (int b = 0; b < J; ++b) {
                        R rx = 0, ry = 0;
#pragma unroll
                        for (int a = 0; a < J; ++a) {
                            const C2 gv = bp[b * EP + a];
                            rx += wx[a] * gv.x;
                            ry += wx[a] * gv.y;
                        }
                        sx += wy[b] * rx;
                        sy += wy[b] * ry;
                    }
                }
                if (MODE == 0) {
                    oimg[vis_index(perm[m])] = vis_conj(perm[m], mk<C2>(sx, sy));
                } else {
                    const R dx = sx - in.yy.x, dy = sy - in.yy.y;
                    const C2 r = mk<C2>(in.vv.x + dx, in.vv.y + dy);
                    rbuf[m] = r;
                    ar = r.x * r.x + r.y * r.y;
                    ad = dx * dx + dy * dy;
                }
            }
            if (MODE == 1) warp_seg_add(ok, jcur, ar, ad, mypart);
        }
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) item_s = claim_item<false>(sched, items, n, batch, tile_on, &ti_s);
        if (MODE == 1) {
            for (int k = threadIdx.x; k < nact; k += blockDim.x) {
                double sr = 0.0, sd = 0.0;
                for (int wp = 0; wp < (int)(blockDim.x >> 5); ++wp) {
                    sr += part[2 * nseg_t * wp + 2 * k];
                    sd += part[2 * nseg_t * wp + 2 * k + 1];
                }
                const int64_t slot = (int64_t)ti.slot0 + act_seg[k] - seg0;
                seg_part[2 * slot] = sr;
                seg_part[2 * slot + 1] = sd;
            }
        }
    }
    if (threadIdx.x == 0) leave_items(sched);
}

// Per-block FP64 norms summed over the block's seg_part slots in a fixed order (one CTA per
// block: thread-strided partial sums, then a fixed tree; one warp per block took 48 us for the
// 1,500 slots of each of 64 blocks in tiles of 8 cells), the ball scale
// c_i = max(0, 1 - eps_i/||r_i||) of step 8 (so v_new = c_i r_i = z - P_B(z)), and the
// residual norm ||G_i b - y_i|| for the adaptive probabilities of Sec. 4.
// norm_only (active == nullptr: every block): only the residual norm is written.
template <typename R>
__global__ void __launch_bounds__(128) k_block_norms(const double* __restrict__ part, const int32_t* __restrict__ bss,
                              const int32_t* __restrict__ bsl, const int32_t* __restrict__ active,
                              const double* __restrict__ eps, double* __restrict__ bnorm, R* __restrict__ scale,
                              double* __restrict__ res_norm, int d, int norm_only) {
    __shared__ double sh[32];
    const int i = blockIdx.x;
    if (active && !active[i]) return;
    double sr = 0.0, sd = 0.0;
    const int end = bss[i + 1];
    for (int k0 = bss[i] + threadIdx.x; k0 < end; k0 += 4 * (int)blockDim.x) {
        double2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = k0 + u * (int)blockDim.x;
            v[u] = k < end ? *reinterpret_cast<const double2*>(part + 2 * (int64_t)bsl[k]) : make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) { sr += v[u].x; sd += v[u].y; }
    }
    sr = block_sum(sr, sh);
    sd = block_sum(sd, sh);
    if (threadIdx.x != 0) return;
    if (norm_only) {
        res_norm[i] = sqrt(sd);
        return;
    }
    bnorm[2 * i] = sr;
    bnorm[2 * i + 1] = sd;
    const double nr = sqrt(sr);
    const double sc = nr > eps[i] ? 1.0 - eps[i] / nr : 0.0;
    scale[i] = (R)sc;
    res_norm[i] = sqrt(sd);
}

// ---------------------------------------------------------------- gridding
// Generic J: one thread per visibility, shared-memory atomics per tap.
template <typename R, int J, int MODE>
__global__ void __launch_bounds__(256) k_grid(const cplx_t<R>* __restrict__ src, const cplx_t<R>* __restrict__ rbuf,
                                              cplx_t<R>* __restrict__ v, const R* __restrict__ scale,
                                              const int32_t* __restrict__ active, const int32_t* __restrict__ cell,
                                              const R* __restrict__ fxs, const R* __restrict__ fys,
                                              const int32_t* __restrict__ perm, const int32_t* __restrict__ seg_start,
                                              const int32_t* __restrict__ seg_block,
                                              const int32_t* __restrict__ tile_seg_start,
                                              const int32_t* __restrict__ list, const int32_t* __restrict__ count,
                                              const int32_t* __restrict__ tile_on, cplx_t<R>* __restrict__ U,
                                              int max_segs,
                                              Geo g, R two_over_j, R beta, const kb_poly_t<R> kp) {
    extern __shared__ __align__(16) unsigned char smraw[];
    R* acc = reinterpret_cast<R*>(smraw);   // [ext*ext] re then [ext*ext] im
    int* act_seg = reinterpret_cast<int*>(acc + 2 * g.ext * g.ext);
    int* act_pre = act_seg + max_segs;
    __shared__ int nact_s;
    const int E = g.ext, EE = E * E;
    const int n = *count;
    for (int w = blockIdx.x; w < n; w += gridDim.x) {
        const int t = list[w];
        if (tile_on && !tile_on[t]) continue;
        const int ty = t / g.ntx, tx = t - ty * g.ntx;
        const int oy = ty * g.tile, ox = tx * g.tile;
        const int seg0 = tile_seg_start[t], nseg_t = tile_seg_start[t + 1] - seg0;
        list_active_segments(seg0, nseg_t, seg_block, MODE == 1 ? active : nullptr, seg_start, act_seg, act_pre,
                             &nact_s);
        for (int i = threadIdx.x; i < 2 * EE; i += blockDim.x) acc[i] = R(0);
        __syncthreads();
        const int total = act_pre[nact_s];
        int j = 0;
        for (int pos = threadIdx.x; pos < total; pos += blockDim.x) {
            while (act_pre[j + 1] <= pos) ++j;
            const int sg = act_seg[j];
            const int m = seg_start[sg] + pos - act_pre[j];
            const cplx_t<R> dv = grid_value<R, MODE>(m, src, rbuf, v, perm, MODE == 1 ? scale[seg_block[sg]] : R(0));
            R wx[J], wy[J];
            kb_taps<R, J>(fxs[m], wx, two_over_j, beta, kp);
            kb_taps<R, J>(fys[m], wy, two_over_j, beta, kp);
            const int c = cell[m];
            R* rowp = acc + ((c >> 16) - oy) * E + ((c & 0xFFFF) - ox);
#pragma unroll
            for (int b = 0; b < J; ++b) {
                const R wr = wy[b] * dv.x, wi = wy[b] * dv.y;
#pragma unroll
                for (int a = 0; a < J; ++a) {
                    atomicAdd(rowp + b * E + a, wx[a] * wr);
                    atomicAdd(rowp + b * E + a + EE, wx[a] * wi);
                }
            }
        }
        __syncthreads();
        add_window<R>(U, oy, ox, g, [&](int ey, int ex) { return mk<cplx_t<R>>(acc[ey * E + ex], acc[ey * E + ex + EE]); });
        __syncthreads();
    }
}

// J <= 8 without atomics inside a tile. Warp w of the CTA takes the 8 x 8 super-cells of
// column w of the tile (T/8 warps), so its points' footprints cover the window columns
// 8w .. 8w + 15 only: each warp accumulates into a private window of T + 7 rows and 16
// columns, and the CTA sums the (at most two) windows that cover each cell at the end of
// the tile. Cells are split into 64 classes by (window row mod 8, window column mod 8);
// lane l owns classes (l / 4, 2 (l % 4) + {0, 1}). A J x J footprint (J <= 8) holds at
// most one cell of each class, so the lanes of a warp never touch the same cell. The
// points of a super-cell arrive sorted by base row: over one base row (a "super-row") a
// class has one footprint row and two candidate columns (c and c + 8 of the warp's
// window), and the lane keeps one running sum per candidate cell in registers, adding
// them to its window when the row changes.
// Staging (one lane per point, 32 points per chunk) writes per-class records that make
// the lane's work a fixed-address read: for row class r the weight times the value,
// phi_y(tap) d; for column class c the weight of its tap, negated when the class cell is
// the high candidate (the weights are positive, so the sign carries the choice and the
// lane splits it with max(w, 0) and max(-w, 0)). The staging lane rotates its taps into
// class order in registers (three conditional shifts), so the column record is two
// aligned 16-byte stores and one 8-byte read per lane and point.
constexpr int GW_MAXW = 16;    // warps per CTA: one per super-cell column (tile <= 128)
constexpr int GW_RREC = 9;     // row records per staged point (8, padded against bank conflicts)
constexpr int GW_CREC = 12;    // column record reals per staged point (8, padded: 16-byte rows, no conflicts)
constexpr int GW_WP = 18;      // window pitch (complex): the 16 columns of one super-cell column's footprints,
                               // padded so that the 8 rows a warp's flush touches start in distinct banks

template <typename R> __device__ __forceinline__ void ld2r(const R* p, R& a, R& b) {
    if constexpr (sizeof(R) == 4) {
        const float2 q = *reinterpret_cast<const float2*>(p);
        a = q.x; b = q.y;
    } else {
        const double2 q = *reinterpret_cast<const double2*>(p);
        a = q.x; b = q.y;
    }
}
template <typename R> __device__ __forceinline__ void st4(R* p, R a, R b, R c, R d) {
    if constexpr (sizeof(R) == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
    } else {
        *reinterpret_cast<double2*>(p) = make_double2(a, b);
        *reinterpret_cast<double2*>(p + 2) = make_double2(c, d);
    }
}
// lo, hi += the class weight's low / high part times ry
template <typename C2, typename R> __device__ __forceinline__ void acc_cand(C2& lo, C2& hi, R w, C2 ry) {
    R wl, wh;
    if constexpr (sizeof(R) == 8) {      // by the sign bit: a comparison would take the FP64 pipe
        const bool neg = __double2hiint(w) < 0;
        wl = neg ? 0.0 : w;
        wh = neg ? -w : 0.0;
    } else {
        wl = w > R(0) ? w : R(0);
        wh = w < R(0) ? -w : R(0);
    }
    lo.x += wl * ry.x; lo.y += wl * ry.y;
    hi.x += wh * ry.x; hi.y += wh * ry.y;
}

// p[0] += a, p[1] += b (two adjacent complex cells, 16-byte aligned in FP32)
template <typename C2> __device__ __forceinline__ void add2(C2* p, C2 a, C2 b) {
    if constexpr (sizeof(C2) == 8) {
        float4* q = reinterpret_cast<float4*>(p);
        float4 t = *q;
        t.x += a.x; t.y += a.y; t.z += b.x; t.w += b.y;
        *q = t;
    } else {
        p[0] = cadd(p[0], a);
        p[1] = cadd(p[1], b);
    }
}

// Shared memory of one CTA of nw warps (ms: most segments of a tile).
template <typename R>
__host__ __device__ constexpr size_t grid8w_smem(int T, int nw, int ms) {
    return (size_t)nw * (T + 7) * GW_WP * 2 * sizeof(R)                       // windows
           + (size_t)nw * 32 * (GW_RREC * 2 + GW_CREC) * sizeof(R)           // records
           + (size_t)nw * (ms * (T / 8 > 0 ? T / 8 : 1) + 1) * sizeof(R)      // range scales
           + (size_t)nw * (2 * (ms * (T / 8 > 0 ? T / 8 : 1)) + 1) * sizeof(int)   // range starts, prefixes
           + (size_t)(2 * ms + 1) * sizeof(int);                              // active segment lists
}

// The raw inputs of one staged point, loaded a chunk ahead.
template <typename R> struct GridIn {
    cplx_t<R> a, b;     // MODE 1: r and v_old; MODE 0: the input value (a)
    R fx, fy, sc;
    int c, m;
};

template <typename R, int MODE>
__device__ __forceinline__ void grid_load(GridIn<R>& in, int pos, int& j, const int* rpre, const int* rstart,
                                          const R* rscale, const cplx_t<R>* __restrict__ src,
                                          const cplx_t<R>* __restrict__ rbuf, const cplx_t<R>* __restrict__ v,
                                          const int32_t* __restrict__ cell, const R* __restrict__ fxs,
                                          const R* __restrict__ fys, const int32_t* __restrict__ perm) {
    while (rpre[j + 1] <= pos) ++j;
    const int m = rstart[j] + pos - rpre[j];
    in.m = m;
    in.fx = fxs[m];
    in.fy = fys[m];
    in.c = cell[m];
    if (MODE == 1) {
        in.a = rbuf[m];
        in.b = v[m];
        in.sc = rscale[j];
    } else {
        in.a = vis_conj(perm[m], src[vis_index(perm[m])]);
    }
}

template <typename R, int J, int MODE>
__global__ void __launch_bounds__(GW_MAXW * 32) k_grid8w(
    const cplx_t<R>* __restrict__ src, const cplx_t<R>* __restrict__ rbuf, cplx_t<R>* __restrict__ v,
    const R* __restrict__ scale, const int32_t* __restrict__ active, const int32_t* __restrict__ cell,
    const R* __restrict__ fxs, const R* __restrict__ fys, const int32_t* __restrict__ perm,
    const int32_t* __restrict__ seg_start, const int32_t* __restrict__ seg_block,
    const int32_t* __restrict__ tile_seg_start, const int32_t* __restrict__ sc_start,
    const int32_t* __restrict__ list, const int32_t* __restrict__ count, const int32_t* __restrict__ tile_on,
    cplx_t<R>* __restrict__ U, int max_segs, Geo g, R two_over_j, R beta, const kb_poly_t<R> kp,
    int* __restrict__ next_tile, int batch, int64_t istride, int64_t ustride) {
    static_assert(J <= 8 && J % 2 == 0, "class ownership needs J <= 8");
    using C2 = cplx_t<R>;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int T = g.tile, WR = T + 7, WS = WR * GW_WP;
    const int nsd = T / 8 > 0 ? T / 8 : 1, nsc = nsd * nsd;    // super-cells per side, per tile
    const int nw = blockDim.x >> 5;                             // = nsd
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rcap = max_segs * nsd;                            // ranges a warp can hold
    C2* wins = reinterpret_cast<C2*>(smraw);                    // [nw][WR][GW_WP]
    C2* win = wins + (size_t)warp * WS;
    C2* rrec = wins + (size_t)nw * WS + (size_t)warp * 32 * GW_RREC;
    R* crec = reinterpret_cast<R*>(wins + (size_t)nw * WS + (size_t)nw * 32 * GW_RREC) + (size_t)warp * 32 * GW_CREC;
    R* rscale = reinterpret_cast<R*>(wins + (size_t)nw * WS + (size_t)nw * 32 * GW_RREC) + (size_t)nw * 32 * GW_CREC +
                (size_t)warp * (rcap + 1);
    int* ints = reinterpret_cast<int*>(reinterpret_cast<R*>(wins + (size_t)nw * WS + (size_t)nw * 32 * GW_RREC) +
                                       (size_t)nw * 32 * GW_CREC + (size_t)nw * (rcap + 1));
    int* rstart = ints + warp * (2 * rcap + 1);
    int* rpre = rstart + rcap;                                  // [rcap + 1]
    int* act_seg = ints + nw * (2 * rcap + 1);
    int* act_pre = act_seg + max_segs;
    __shared__ int nact_s, tile_s;
    const int lcy = lane >> 2, lcx = (lane & 3) * 2;
    const int n = *count;
    for (;;) {
        // tiles are taken from the heaviest-first list one at a time by whichever CTA is free
        if (threadIdx.x == 0) tile_s = claim_tile<false>(next_tile, list, n, batch, tile_on);
        __syncthreads();
        const int w = tile_s;
        if (w >= n * batch) break;
        const int t = list[w % n], img = w / n;   // image by image of a batch
        const cplx_t<R>* simg = MODE == 0 ? src + (int64_t)img * istride : src;
        cplx_t<R>* Uimg = U + (int64_t)img * ustride;
        const int ty = t / g.ntx, tx = t - ty * g.ntx;
        const int oy = ty * T, ox = tx * T;
        const int seg0 = tile_seg_start[t], nseg_t = tile_seg_start[t + 1] - seg0;
        list_active_segments(seg0, nseg_t, seg_block, MODE == 1 ? active : nullptr, seg_start, act_seg, act_pre,
                             &nact_s);
        for (int i = lane; i < WS; i += 32) win[i] = mk<C2>(R(0), R(0));
        __syncthreads();
        // this warp's ranges: the super-cells of column `warp` of every active segment
        const int nact = nact_s, nr = nact * nsd;
        if (lane == 0) rpre[0] = 0;
        for (int base = 0; base < nr; base += 32) {
            const int k = base + lane;
            int len = 0, st0 = 0;
            R scv = R(0);
            if (k < nr) {
                const int jj = k / nsd, srow = k - jj * nsd;
                const int sg = act_seg[jj];
                const int sc = srow * nsd + warp;
                st0 = sc_start[(int64_t)sg * (nsc + 1) + sc];
                len = sc_start[(int64_t)sg * (nsc + 1) + sc + 1] - st0;
                if (MODE == 1) scv = scale[seg_block[sg]];
            }
            int incl = len;
            for (int o = 1; o < 32; o <<= 1) {
                const int yv = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += yv;
            }
            const int before = base > 0 ? rpre[base] : 0;
            __syncwarp();
            if (k < nr) {
                rstart[k] = st0;
                rscale[k] = scv;
                rpre[k + 1] = before + incl;
            }
            __syncwarp();
        }
        const int total = nr > 0 ? rpre[nr] : 0;
        // chunks of 32 consecutive points of the warp's ranges
        const int nchunk = (total + 31) >> 5;
        int j = 0;            // this lane's range cursor (its positions only grow)
        GridIn<R> in{};
        if (nchunk > 0 && lane < total)
            grid_load<R, MODE>(in, lane, j, rpre, rstart, rscale, simg, rbuf, v, cell, fxs, fys, perm);
        for (int chunk = 0; chunk < nchunk; ++chunk) {
            const int fill = min(32, total - chunk * 32);
            int mykey = -1;   // footprint row of this lane's staged point
            if (lane < fill) {
                C2 d;
                if (MODE == 1) {
                    const C2 vn = cscale(in.a, in.sc);       // step 8: v_new = c_i r
                    v[in.m] = vn;
                    d = csub(vn, in.b);
                } else {
                    d = in.a;
                }
                R wx[J], wy[J];
                kb_taps<R, J>(in.fx, wx, two_over_j, beta, kp);
                kb_taps<R, J>(in.fy, wy, two_over_j, beta, kp);
                const int r0 = (in.c >> 16) - oy, c0 = (in.c & 0xFFFF) - ox;   // footprint origin in the window
                C2* rr = rrec + lane * GW_RREC;
#pragma unroll
                for (int b = 0; b < 8; ++b) {
                    const R wv = b < J ? wy[b] : R(0);
                    rr[(r0 + b) & 7] = mk<C2>(wv * d.x, wv * d.y);
                }
                // class c = (gam + a) mod 8 takes tap a = (c - gam) mod 8; its cell is the high
                // candidate (window column c + 8) when gam + a >= 8, i.e. when c < gam
                const int gam = c0 & 7;                             // c0 = 8 warp + gam
                R cw[8];
#pragma unroll
                for (int a = 0; a < 8; ++a) cw[a] = a < J ? wx[a] : R(0);
#pragma unroll
                for (int sh = 1; sh < 8; sh <<= 1) {
                    const bool on = (gam & sh) != 0;
                    R t[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) t[c] = on ? cw[(c - sh) & 7] : cw[c];
#pragma unroll
                    for (int c = 0; c < 8; ++c) cw[c] = t[c];
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) cw[c] = c < gam ? -cw[c] : cw[c];
                R* cr = crec + lane * GW_CREC;
                st4(cr, cw[0], cw[1], cw[2], cw[3]);
                st4(cr + 4, cw[4], cw[5], cw[6], cw[7]);
                mykey = r0;
            }
            // the next chunk's loads go out now and land while this one is accumulated
            const int nxt = (chunk + 1) * 32 + lane;
            if (nxt < total)
                grid_load<R, MODE>(in, nxt, j, rpre, rstart, rscale, simg, rbuf, v, cell, fxs, fys, perm);
            __syncwarp();
            // runs of consecutive points with the same footprint row: one set of running sums
            // per run, added to the window at its end
            const int prevk = __shfl_up_sync(0xffffffffu, mykey, 1);
            unsigned starts = __ballot_sync(0xffffffffu, lane < fill && (lane == 0 || mykey != prevk));
            while (starts) {
                const int q0 = __ffs(starts) - 1;
                starts &= starts - 1;
                const int q1 = starts ? __ffs(starts) - 1 : fill;
                const int r0 = __shfl_sync(0xffffffffu, mykey, q0);
                // the run's first point starts the running sums, the others add to them two at a time
                C2 lo0 = mk<C2>(R(0), R(0)), hi0 = lo0, lo1 = lo0, hi1 = lo0;
                int q = q0;
                for (; q + 1 < q1; q += 2) {
                    const C2 ra = rrec[q * GW_RREC + lcy], rb = rrec[(q + 1) * GW_RREC + lcy];
                    R a0, a1, b0, b1;
                    ld2r(crec + q * GW_CREC + lcx, a0, a1);
                    ld2r(crec + (q + 1) * GW_CREC + lcx, b0, b1);
                    acc_cand(lo0, hi0, a0, ra);
                    acc_cand(lo1, hi1, a1, ra);
                    acc_cand(lo0, hi0, b0, rb);
                    acc_cand(lo1, hi1, b1, rb);
                }
                if (q < q1) {
                    const C2 ry = rrec[q * GW_RREC + lcy];
                    R a0, a1;
                    ld2r(crec + q * GW_CREC + lcx, a0, a1);
                    acc_cand(lo0, hi0, a0, ry);
                    acc_cand(lo1, hi1, a1, ry);
                }
                C2* cp = win + (r0 + ((lcy - r0) & 7)) * GW_WP + lcx;
                add2(cp, lo0, lo1);
                add2(cp + 8, hi0, hi1);
            }
            __syncwarp();
        }
        __syncthreads();
        // U += the windows (tile and halo): column ex of the tile window lies in warp
        // ex/8's window (local column ex mod 8) and in warp ex/8 - 1's (local ex mod 8 + 8)
        add_window<R>(Uimg, oy, ox, g, [&](int ey, int ex) {
            const int w0 = ex >> 3, lc = ex & 7;
            C2 sum = mk<C2>(R(0), R(0));
            if (w0 < nw) sum = wins[(size_t)w0 * WS + ey * GW_WP + lc];
            if (w0 >= 1) sum = cadd(sum, wins[(size_t)(w0 - 1) * WS + ey * GW_WP + lc + 8]);
            return sum;
        });
        __syncthreads();
    }
}

// ---------------------------------------------------------------- gridding, FP32, J <= 8
// The window of one super-cell (8 x 8 footprint origins) is a 16 x 16 patch, and gridding
// its points is a contraction over them: patch[r][c] = sum_m wy_m[r] (d_m wx_m[c]). A warp
// runs it on the tensor cores: M = 16 patch rows, N = 2 x 16 patch columns (re, im), K = 16
// points. Every FP32 operand is split exactly into three bf16 values, each rounded to nearest
// (8 + 8 + 8 significant bits), and the six products down to 2^-16 of the leading one are
// accumulated. What is dropped has an rms of 5.7e-9 of the product and 5.3e-8 at most (4M random
// pairs), the rounding of an FP32 product 2.5e-8 and 6.0e-8. The sum of 16 points is added to
// FP32 registers. The tensor core truncates its sums: left at that, Phi^H was up to 8% further
// from 64-bit arithmetic at J = 6 than with chains of FP32 multiply-adds (512^2 image: 1.58e-7 ->
// 1.70e-7), so the leading products go through it twice and what the first sum lost is added with
// the smaller products (1.53e-7; J = 4, 6 and 8: 3% to 25% below the chains; 16.8M points on 4096^2
// cells, half of them active: 390 -> 400 us).
// A CTA works on one part of a tile at a time. The part's points, super-cell by super-cell
// (each padded to a multiple of 16), are cut into chunks of 32 that are shared out evenly
// among the CTA's working warps; at the end of a super-cell (or of its share) a warp stores
// the patch to the slot super-cell + warp, which no other pair has; the slots are then summed,
// in a fixed order, into the part's window. One more warp keeps the others fed: it claims
// the next item and lists its points while they work on the current one, and it adds the
// finished window to U with bulk reductions, one per column panel (rows of a panel are
// contiguous in U), while they work on the next.
// What bounds it: instruction issue and the barriers between the phases of an item (about 30 warp
// instructions a point, half of them in the contraction) with 16 warps per SM by registers. 16.8M
// points, half of them active, on a 4096^2 grid: 400 us, against 478 us for FP32 multiply-adds in
// four launches; 65,536 points on 512^2, where the densest tile was the critical path of each launch:
// 30 against 164 us; 1.05M on 1024^2: 56 against 296 us. A batch of dense images is the exception:
// eight of 1024^2 with 4.19M points each, Phi^H 1.92 ms, in four launches 1.73. Slower (timed on an
// earlier form, 360 us at 16.8M points): 2048-point parts (459 us), 3 or 15 working warps (442, 448
// us), 80 or 96 registers for more warps (496, 410 us), waits in the order of the tiles' weight
// instead of their colour (3.3 ms: chains of neighbours).
// Staging (one lane per point) writes the taps by class (patch row / column mod 8),
// negated when the tap falls in the upper half of the patch: 18 floats a point, each read
// once, by the lane whose fragment needs it.
constexpr int GM_F = 18;       // floats per staged point: 8 row classes, 8 column classes, re, im
constexpr int GM_WP = 18;      // patch pitch (complex)
constexpr int GM_PS = 16 * GM_WP;   // patch slot (complex)
constexpr int GM_MAXW = 16;    // warps per CTA, the feeding one included

__device__ __forceinline__ int ld_acquire(const int32_t* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// One work item, listed by the feeding warp: which tile and part, and its chunks.
struct GridItem {
    int tile, img, part, parts;   // tile < 0: none left
    int nact, total, cbeg, nchunk;
};

// Shared memory of a CTA with nc working warps (ms: most segments of a tile); the item
// lists are kept twice.
__host__ __device__ constexpr size_t grid_mma_lists(int nsc, int ms) {
    return (size_t)nsc * sizeof(int2) + (size_t)(nsc + 1) * sizeof(int) + (size_t)ms * sizeof(float) +
           (size_t)(2 * nsc * ms + 1) * sizeof(int);
}
__host__ __device__ constexpr size_t grid_mma_smem(int T, int nc, int ms) {
    const int nsd = T / 8, nsc = nsd * nsd;
    return (size_t)(T + 8) * (T + 8) * sizeof(float2) + (size_t)(nsc + nc) * GM_PS * sizeof(float2) +
           (size_t)nc * 32 * GM_F * sizeof(float) + 2 * ((grid_mma_lists(nsc, ms) + 15) / 16 * 16) +
           (size_t)ms * sizeof(int);
}

__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// x = s0 + s1 + s2 for two values at a time, each part rounded to nearest to bf16 (8 bits; the last one
// exactly), a in the low and b in the high half: the parts' signs differ, so that the dropped
// products have no bias.
__device__ __forceinline__ uint32_t bf16_pair(float2 v) {
    uint32_t p;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p) : "f"(v.y), "f"(v.x));
    return p;
}
__device__ __forceinline__ void split3(float a, float b, uint32_t* s) {
    float2 r = make_float2(a, b);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        s[i] = bf16_pair(r);
        if (i < 2) r = ffma2(make_float2(__uint_as_float(s[i] << 16), __uint_as_float(s[i] & 0xffff0000u)),
                             make_float2(-1.f, -1.f), r);
    }
}
// 0xffff in the half of each negative operand
__device__ __forceinline__ uint32_t sign_mask(float a, float b) {
    uint32_t m;
    asm("prmt.b32 %0, %1, %2, 0xFFBB;" : "=r"(m) : "r"(__float_as_uint(a)), "r"(__float_as_uint(b)));
    return m;
}

// acc += the 16 staged points of group grp, all of one super-cell.
// acc[n][e]: n = {re low, re high, im low, im high} columns, e = the fragment's 4 elements.
__device__ __forceinline__ void grid_mma_group(const float* __restrict__ st, int grp, int g, int t, float (*acc)[4]) {
    const int p0 = 16 * grp + 4 * t;
    const int ps = p0 ^ ((g & 1) << 4);
    const float4 wy = *reinterpret_cast<const float4*>(st + g * 32 + ps);
    const float4 wx = *reinterpret_cast<const float4*>(st + (8 + g) * 32 + ps);
    const float4 dr = *reinterpret_cast<const float4*>(st + 16 * 32 + p0);
    const float4 di = *reinterpret_cast<const float4*>(st + 17 * 32 + p0);
    uint32_t A[3][4];
    {
        const uint32_t m0 = sign_mask(wy.x, wy.y), m1 = sign_mask(wy.z, wy.w);
        uint32_t u[3], v[3];
        split3(fabsf(wy.x), fabsf(wy.y), u);
        split3(fabsf(wy.z), fabsf(wy.w), v);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            A[i][0] = u[i] & ~m0; A[i][1] = u[i] & m0; A[i][2] = v[i] & ~m1; A[i][3] = v[i] & m1;
        }
    }
    const uint32_t m0 = sign_mask(wx.x, wx.y), m1 = sign_mask(wx.z, wx.w);
#pragma unroll
    for (int h = 0; h < 2; ++h) {                       // real, imaginary part
        const float4 dv = h ? di : dr;
        uint32_t u[3], v[3];
        split3(fabsf(wx.x) * dv.x, fabsf(wx.y) * dv.y, u);
        split3(fabsf(wx.z) * dv.z, fabsf(wx.w) * dv.w, v);
#pragma unroll
        for (int hi = 0; hi < 2; ++hi) {                // low, high half of the patch columns
            uint32_t b0[3], b1[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                b0[i] = hi ? u[i] & m0 : u[i] & ~m0;
                b1[i] = hi ? v[i] & m1 : v[i] & ~m1;
            }
            // The tensor core truncates its sums. m is the sum of the leading products as it comes,
            // t that added to the running sum and rounded; d starts from what that rounding left, adds
            // the leading products again (less m: what the truncation left) and then the smaller ones.
            float* ac = acc[2 * h + hi];
            float m[4] = {0.f, 0.f, 0.f, 0.f}, d[4], t[4];
            mma_bf16(m, A[0], b0[0], b1[0]);
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                const float2 a2 = make_float2(ac[e], ac[e + 1]);
                const float2 t2 = fadd2(a2, make_float2(m[e], m[e + 1]));
                const float2 d2 = ffma2(t2, make_float2(-1.f, -1.f), a2);
                t[e] = t2.x; t[e + 1] = t2.y; d[e] = d2.x; d[e + 1] = d2.y;
            }
            mma_bf16(d, A[0], b0[0], b1[0]);
            mma_bf16(d, A[2], b0[0], b1[0]);
            mma_bf16(d, A[0], b0[2], b1[2]);
            mma_bf16(d, A[1], b0[1], b1[1]);
            mma_bf16(d, A[1], b0[0], b1[0]);
            mma_bf16(d, A[0], b0[1], b1[1]);
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                const float2 s2 = fadd2(make_float2(t[e], t[e + 1]), make_float2(d[e], d[e + 1]));
                ac[e] = s2.x; ac[e + 1] = s2.y;
            }
        }
    }
}

// w[0..J) (tap a falls in class (o + a) mod 8) into class order, negated for o + a >= 8,
// zero for classes without a tap
template <int J> __device__ __forceinline__ void class_order(const float* w, int o, float* out) {
#pragma unroll
    for (int a = 0; a < 8; ++a) out[a] = a < J ? w[a] : 0.f;
#pragma unroll
    for (int sh = 1; sh < 8; sh <<= 1) {
        const bool on = (o & sh) != 0;
        float q[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) q[c] = on ? out[(c - sh) & 7] : out[c];
#pragma unroll
        for (int c = 0; c < 8; ++c) out[c] = q[c];
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) out[c] = c < o ? -out[c] : out[c];
}

// The lists of one item in shared memory.
struct GridLists {
    int2* sinfo;      // [nsc] first slot and number of slots of each super-cell
    int* ps;          // [nsc + 1] padded start of each super-cell
    float* rscale;    // [ms] ball scale of each active segment
    int* rstart;      // [nsc * ms] first point of each range (super-cell * nact + segment)
    int* rpre;        // [nsc * ms + 1] prefix sums of the ranges' lengths
    __device__ GridLists(unsigned char* base, int nsc, int ms) {
        sinfo = reinterpret_cast<int2*>(base);
        ps = reinterpret_cast<int*>(sinfo + nsc);
        rscale = reinterpret_cast<float*>(ps + nsc + 1);
        rstart = reinterpret_cast<int*>(rscale + ms);
        rpre = rstart + nsc * ms;
    }
};

// The point at position pos of the item's padded order (super-cell sc from ps[sc] on); sc,
// k and jj are this lane's super-cell, range and active-segment cursors (k = sc * nact +
// jj), moved forward to it. False past the super-cell's points.
template <int MODE>
__device__ __forceinline__ bool grid_mma_load(GridIn<float>& in, int pos, int& sc, int& k, int& jj, int nsc, int nact,
                                              const GridLists& L, const float2* __restrict__ src,
                                              const float2* __restrict__ rbuf, const float2* __restrict__ v,
                                              const int32_t* __restrict__ cell, const float* __restrict__ fxs,
                                              const float* __restrict__ fys, const int32_t* __restrict__ perm) {
    while (sc + 1 < nsc && L.ps[sc + 1] <= pos) ++sc;
    const int up = pos - L.ps[sc] + L.rpre[sc * nact];
    if (up >= L.rpre[(sc + 1) * nact]) return false;
    while (L.rpre[k + 1] <= up) {
        ++k;
        jj = jj + 1 == nact ? 0 : jj + 1;
    }
    const int m = L.rstart[k] + up - L.rpre[k];
    in.m = m;
    in.fx = fxs[m];
    in.fy = fys[m];
    in.c = cell[m];
    if (MODE == 1) {
        in.a = rbuf[m];
        in.b = v[m];
        in.sc = L.rscale[jj];
    } else {
        const int q = perm[m];
        in.a = vis_conj(q, src[vis_index(q)]);
    }
    return true;
}

template <int J, int MODE>
__global__ void __launch_bounds__(GM_MAXW * 32) k_grid_mma(
    const float2* __restrict__ src, const float2* __restrict__ rbuf, float2* __restrict__ v,
    const float* __restrict__ scale, const int32_t* __restrict__ active, const int32_t* __restrict__ cell,
    const float* __restrict__ fxs, const float* __restrict__ fys, const int32_t* __restrict__ perm,
    const int32_t* __restrict__ seg_block, const int32_t* __restrict__ sc_start, const int4* __restrict__ tile_info, const int32_t* __restrict__ tile_on,
    const int2* __restrict__ items, const int32_t* __restrict__ nitems, int32_t* pend, float2* U, int max_segs, Geo g,
    const KbPoly kp, int* sched, int32_t* gave_up, int polls, int batch, int64_t istride, int64_t ustride) {
    static_assert(J <= 8 && J % 2 == 0, "a super-cell's window is 16 x 16 for J <= 8");
    extern __shared__ __align__(16) unsigned char smraw[];
    const int T = g.tile, nsd = T >> 3, nsc = nsd * nsd, W = T + 8;
    const int nc = (blockDim.x >> 5) - 1, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int NT = blockDim.x, NCT = nc * 32;                   // all threads, working threads
    float2* wbuf = reinterpret_cast<float2*>(smraw);            // [W / 4][W][4] the window, in U's panel layout
    float2* slots = wbuf + W * W;                               // [nsc + nc][16][GM_WP]
    float* st = reinterpret_cast<float*>(slots + (size_t)(nsc + nc) * GM_PS) + (size_t)warp * 32 * GM_F;   // [GM_F][32]
    unsigned char* lbase = reinterpret_cast<unsigned char*>(slots + (size_t)(nsc + nc) * GM_PS) +
                           (size_t)nc * 32 * GM_F * sizeof(float);
    const size_t lsz = (grid_mma_lists(nsc, max_segs) + 15) / 16 * 16;
    __shared__ GridItem item_s[2];
    // barriers: 1, 2 item listed (even, odd); 3 slots written; 4 window written; 5 window free; 6 halfway
    if (warp == nc) {
        // ---------------------------------------------------------------- the feeding warp
        int* act_seg = reinterpret_cast<int*>(lbase + 2 * lsz);
        const int nlist = *nitems, nitem = nlist * batch;
        // claims the next item with an active block (items are claimed in order by whichever CTA is
        // free, all images of a batch before the next item) and lists it in buffer b
        auto prepare = [&](int b) -> bool {
            const GridLists L(lbase + b * lsz, nsc, max_segs);
            int w, img;
            int2 it;
            int4 ti;
            for (;;) {
                w = lane == 0 ? atomicAdd(sched, 1) : 0;
                w = __shfl_sync(0xffffffffu, w, 0);
                if (w >= nitem) {
                    if (lane == 0) item_s[b].tile = -1;
                    return false;
                }
                it = items[w / batch];
                img = w % batch;
                ti = tile_info[it.x];
                if (!tile_on || tile_on[it.x]) break;
            }
            int nact = 0;
            const unsigned below = (1u << lane) - 1u;
            for (int base = 0; base < ti.y; base += 32) {
                const int k = base + lane;
                int blk = 0;
                bool on = k < ti.y;
                if (on) blk = seg_block[ti.x + k];
                if (MODE == 1 && on) on = active[blk] != 0;
                const unsigned bal = __ballot_sync(0xffffffffu, on);
                if (on) {
                    const int pos = nact + __popc(bal & below);
                    act_seg[pos] = ti.x + k;
                    if (MODE == 1) L.rscale[pos] = scale[blk];
                }
                nact += __popc(bal);
            }
            __syncwarp();
            // ranges super-cell * nact + segment, with the prefix sums of their lengths
            const int nr = nact * nsc;
            int tot = 0;
            if (lane == 0) L.rpre[0] = 0;
            for (int base = 0; base < nr; base += 128) {
                int s0[4], s1[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = base + u * 32 + lane;
                    s0[u] = s1[u] = 0;
                    if (k < nr) {
                        const int sc = k / nact;
                        const int32_t* p = sc_start + (int64_t)act_seg[k - sc * nact] * (nsc + 1) + sc;
                        s0[u] = p[0];
                        s1[u] = p[1];
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = base + u * 32 + lane;
                    int incl = s1[u] - s0[u];
                    for (int o = 1; o < 32; o <<= 1) {
                        const int yv = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += yv;
                    }
                    if (k < nr) {
                        L.rstart[k] = s0[u];
                        L.rpre[k + 1] = tot + incl;
                    }
                    tot += __shfl_sync(0xffffffffu, incl, 31);
                }
            }
            __syncwarp();
            // every super-cell starts at a multiple of 16, so that the 16 points of a group share it
            int padded = 0;
            for (int base = 0; base < nsc; base += 32) {
                const int sc = base + lane;
                const int pl = sc < nsc && nact ? (L.rpre[(sc + 1) * nact] - L.rpre[sc * nact] + 15) & ~15 : 0;
                int incl = pl;
                for (int o = 1; o < 32; o <<= 1) {
                    const int yv = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += yv;
                }
                if (sc < nsc) L.ps[sc] = padded + incl - pl;
                padded += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) L.ps[nsc] = padded;
            __syncwarp();
            // this part's chunks of the tile, shared out to nu warps with at least one chunk each
            const int allch = (padded + 31) >> 5;
            const int cbeg = (int)((int64_t)allch * it.y / ti.z);
            const int nchunk = (int)((int64_t)allch * (it.y + 1) / ti.z) - cbeg, nu = min(nc, nchunk);
            for (int sc = lane; sc < nsc; sc += 32) {
                const int c0 = max((L.ps[sc] >> 5) - cbeg, 0), c1 = min(((L.ps[sc + 1] - 1) >> 5) - cbeg, nchunk - 1);
                int2 si = make_int2(0, 0);
                if (L.ps[sc + 1] > L.ps[sc] && c0 <= c1) {   // chunk c belongs to warp ((c + 1) nu - 1) / nchunk
                    const int w0 = ((c0 + 1) * nu - 1) / nchunk, w1 = ((c1 + 1) * nu - 1) / nchunk;
                    si = make_int2(sc + w0, w1 - w0 + 1);
                }
                L.sinfo[sc] = si;
            }
            if (lane == 0) item_s[b] = GridItem{it.x, img, it.y, ti.z, nact, padded, cbeg, nchunk};
            return true;
        };
        bool have = prepare(0);
        __syncwarp();
        bar_arrive(1, NT);
        for (int i = 0; have; ++i) {
            const int b = i & 1;
            bar_sync(6, 64);                                    // the working warps are halfway through item i
            const bool next = prepare(b ^ 1);
            __syncwarp();
            bar_arrive(1 + (b ^ 1), NT);
            bar_sync(4, NT);                                    // item i's window is complete
            // The windows of neighbouring tiles overlap, and so do a tile's parts: they are added to
            // U in the order of the items, so that the sums do not depend on timing. Earlier items
            // are claimed earlier and a CTA takes its items in order, so the first unfinished one
            // is being worked on and never waits: this wait ends. Its limit is a safeguard (some
            // seconds), after which the launch sets its flag and goes on: the adds are atomic, so that
            // U is still complete and only the order of its sums is lost.
            const GridItem& im = item_s[b];
            const int ty = im.tile / g.ntx, tx = im.tile - ty * g.ntx;
            int32_t* pd = pend + (int64_t)im.img * g.ntiles;
            if (lane < 9) {
                const int t2 = ((ty + lane / 3 - 1) & (g.nty - 1)) * g.ntx + ((tx + lane % 3 - 1) & (g.ntx - 1));
                const int upto = t2 == im.tile ? im.parts - im.part : 0;
                if (t2 == im.tile || tile_info[t2].w < tile_info[im.tile].w) {
                    int tries = 0;
                    while (ld_acquire(pd + t2) > upto)
                        if (++tries > polls) { atomicExch(gave_up, 1); break; }
                }
            }
            __syncwarp();
            asm volatile("fence.proxy.async;" ::: "memory");
            // panel pn of the window: W rows of 32 bytes, in two pieces where they wrap around the grid
            float2* Uimg = U + (int64_t)im.img * ustride;
            const int oy = ty * T, r0 = min(W, g.Ky - oy);
            for (int pn = lane; pn < W / 4; pn += 32) {
                float2* dst = Uimg + panel_off(oy, (tx * T + 4 * pn) & (g.Kx - 1), g.Ky);
                const uint32_t sa = (uint32_t)__cvta_generic_to_shared(wbuf + pn * W * 4);
                asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;" ::"l"(dst),
                             "r"(sa), "r"(r0 * 32) : "memory");
                if (r0 < W)
                    asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;" ::"l"(
                                     dst - (int64_t)oy * PW), "r"(sa + r0 * 32), "r"((W - r0) * 32) : "memory");
            }
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncwarp();
            if (next) bar_arrive(5, NT);                        // the window's buffer is free
            asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
            asm volatile("fence.proxy.async;" ::: "memory");
            __threadfence();
            __syncwarp();
            if (lane == 0) atomicSub(pd + im.tile, 1);
            have = next;
        }
        return;
    }
    // -------------------------------------------------------------------- the working warps
    const int fg = lane >> 2, ft = lane & 3;                    // fragment row / column of this lane
    // where this warp stands in the current item
    GridIn<float> in{};
    int sc, k, jj, ch0, ch1, nact, total, oy, ox;
    const float2* simg = src;
    bool ok;
    auto setup = [&](int b) {
        const GridItem& im = item_s[b];
        const GridLists L(lbase + b * lsz, nsc, max_segs);
        const int ty = im.tile / g.ntx;
        oy = ty * T;
        ox = (im.tile - ty * g.ntx) * T;
        nact = im.nact;
        total = im.total;
        if (MODE == 0) simg = src + (int64_t)im.img * istride;
        const int nu = min(nc, im.nchunk);
        ch0 = warp < nu ? im.cbeg + (int)((int64_t)im.nchunk * warp / nu) : 0;
        ch1 = warp < nu ? im.cbeg + (int)((int64_t)im.nchunk * (warp + 1) / nu) : 0;
        sc = k = jj = 0;
        ok = false;
        if (ch0 < ch1) {
            const int pos = ch0 * 32 + lane;
            int hi = nsc;     // last super-cell with ps[sc] <= pos
            while (hi - sc > 1) {
                const int mid = (sc + hi) >> 1;
                if (L.ps[mid] <= pos) sc = mid; else hi = mid;
            }
            const int nr = nact * nsc, up = min(pos - L.ps[sc] + L.rpre[sc * nact], L.rpre[nr] - 1);
            hi = nr;          // last range with rpre[k] <= up
            while (hi - k > 1) {
                const int mid = (k + hi) >> 1;
                if (L.rpre[mid] <= up) k = mid; else hi = mid;
            }
            jj = k % nact;
            ok = pos < total && grid_mma_load<MODE>(in, pos, sc, k, jj, nsc, nact, L, simg, rbuf, v, cell, fxs, fys, perm);
        }
    };
    for (int c = 0; c < GM_F; ++c) st[c * 32 + lane] = 0.f;
    bar_sync(1, NT);
    if (item_s[0].tile < 0) return;
    setup(0);
    for (int i = 0;; ++i) {
        const int b = i & 1;
        const GridLists L(lbase + b * lsz, nsc, max_segs);
        float acc[4][4] = {};
        int cur = -1;         // the super-cell the sums belong to
        auto flush = [&]() {
            float2* cp = slots + (size_t)(cur + warp) * GM_PS + fg * GM_WP + 2 * ft;
#pragma unroll
            for (int hi = 0; hi < 2; ++hi)
#pragma unroll
                for (int u = 0; u < 2; ++u)             // patch rows fg and fg + 8
                    *reinterpret_cast<float4*>(cp + u * 8 * GM_WP + hi * 8) =
                        make_float4(acc[hi][2 * u], acc[2 + hi][2 * u], acc[hi][2 * u + 1], acc[2 + hi][2 * u + 1]);
        };
        const int half = (ch0 + ch1) >> 1;
        if (warp == 0 && ch0 >= ch1) bar_arrive(6, 64);
        for (int chunk = ch0; chunk < ch1; ++chunk) {
            if (warp == 0 && chunk == half) bar_arrive(6, 64);
            const int mysc = sc;
            if (ok) {
                float2 d;
                if (MODE == 1) {
                    const float2 vn = cscale(in.a, in.sc);       // step 8: v_new = c_i r
                    v[in.m] = vn;
                    d = csub(vn, in.b);
                } else {
                    d = in.a;
                }
                const int r0 = (in.c >> 16) - oy, c0 = (in.c & 0xFFFF) - ox;   // footprint origin in the window
                float wt[J], cw[8];
                kb_taps<float, J>(in.fy, wt, 0.f, 0.f, kp);
                class_order<J>(wt, r0 & 7, cw);
#pragma unroll
                for (int c = 0; c < 8; ++c) st[c * 32 + (lane ^ ((c & 1) << 4))] = cw[c];
                const int gam = c0 & 7;
                kb_taps<float, J>(in.fx, wt, 0.f, 0.f, kp);
                class_order<J>(wt, gam, cw);
#pragma unroll
                for (int c = 0; c < 8; ++c) st[(8 + c) * 32 + (lane ^ ((c & 1) << 4))] = cw[c];
                st[16 * 32 + lane] = d.x;
                st[17 * 32 + lane] = d.y;
            } else {          // no point here: value zero, with the (finite) weights of an earlier one
                st[16 * 32 + lane] = 0.f;
                st[17 * 32 + lane] = 0.f;
            }
            // the next chunk's loads go out now and land while this one is accumulated
            const int nxt = (chunk + 1) * 32 + lane;
            ok = chunk + 1 < ch1 && nxt < total &&
                 grid_mma_load<MODE>(in, nxt, sc, k, jj, nsc, nact, L, simg, rbuf, v, cell, fxs, fys, perm);
            __syncwarp();
#pragma unroll
            for (int grp = 0; grp < 2; ++grp) {
                if (chunk * 32 + grp * 16 >= total) break;
                const int key = __shfl_sync(0xffffffffu, mysc, grp * 16);
                if (key != cur) {
                    if (cur >= 0) flush();
                    cur = key;
#pragma unroll
                    for (int q = 0; q < 16; ++q) (&acc[0][0])[q] = 0.f;
                }
                grid_mma_group(st, grp, fg, ft, acc);
            }
            __syncwarp();
        }
        if (cur >= 0) flush();
        // the next item's first loads go out before this one's window is put together
        bar_sync(1 + (b ^ 1), NT);
        const bool more = item_s[b ^ 1].tile >= 0;
        if (more) setup(b ^ 1);
        bar_sync(3, NCT);
        if (i > 0) bar_sync(5, NT);
        // the window, block of 8 x 8 cells by block, two cells a lane: block (by, bx) is covered by
        // the patches of the super-cells (by, bx) .. (by - 1, bx - 1)
        for (int by = 0, bx = warp; ; bx += nc) {
            while (bx > nsd) { bx -= nsd + 1; ++by; }
            if (by > nsd) break;
            float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int a = q >> 1, c = q & 1, sy = by - a, sx = bx - c;
                if (sy < 0 || sy >= nsd || sx < 0 || sx >= nsd) continue;
                const int2 si = L.sinfo[sy * nsd + sx];
                const float2* sp = slots + si.x * GM_PS + (8 * a + fg) * GM_WP + 8 * c + 2 * ft;
#pragma unroll 1
                for (int e = 0; e < si.y; ++e, sp += GM_PS) {
                    const float4 x = *reinterpret_cast<const float4*>(sp);
                    sum.x += x.x; sum.y += x.y; sum.z += x.z; sum.w += x.w;
                }
            }
            const int ex = 8 * bx + 2 * ft;
            *reinterpret_cast<float4*>(wbuf + ((ex >> 2) * W + 8 * by + fg) * 4 + (ex & 3)) = sum;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        bar_sync(4, NT);
        if (!more) return;
    }
}

// ---------------------------------------------------------------- launchers

template <typename R, int J, int MODE>
static cudaError_t launch_degrid(const pd_plan* p, const cplx_t<R>* grid, cplx_t<R>* out, const DualArgs* a,
                                 cudaStream_t s, int batch = 1) {
    if constexpr (J <= 8)
        if (p->g_mode == PD_G_CSR) return launch_degrid_csr<R, J, MODE>(p, grid, out, a, s, batch);
    const Geo& g = p->g;
    const int ms = std::max(p->max_tile_segs, 1);
    const size_t win = sizeof(R) == 4 ? (size_t)2 * g.ext * ((g.ext + 2) & ~1) : (size_t)g.ext * g.ext;
    const size_t smem = win * sizeof(cplx_t<R>) + (size_t)16 * ms * sizeof(double) + (size_t)(2 * ms + 1) * sizeof(int);
    cudaError_t e = ensure_smem(k_degrid<R, J, MODE>, smem);
    if (e) return e;
    // items are claimed one at a time: launch only as many CTAs as are resident at once
    int per_sm = 0;
    // 256 threads, or 128 where the items hold fewer points than would keep those busy and are enough
    // to fill the GPU all the same (FP32; J = 12, 300,007 points on 1024^2 cells: 68 -> 45 us; 64
    // images of 256^2, 65,536 points, J = 8: 273 -> 220 us; too few items, 800 of 125 points: 25 -> 27 us)
    const bool small = sizeof(R) == 4 && p->M < (int64_t)p->n_ditems * 192 &&
                       (int64_t)p->n_ditems * batch >= (int64_t)p->num_sms * 8;
    const int NT = small ? 128 : 256;
    if ((e = occupancy(&per_sm, k_degrid<R, J, MODE>, NT, smem))) return e;
    const int ctas = (int)std::min<int64_t>((int64_t)p->n_ditems * batch, (int64_t)std::max(per_sm, 1) * p->num_sms);
    k_degrid<R, J, MODE><<<ctas, NT, smem, s>>>(
        grid, out, a ? (const cplx_t<R>*)a->y : nullptr, a ? (const cplx_t<R>*)a->v : nullptr,
        (cplx_t<R>*)p->rbuf, p->cell, (const R*)p->fx, (const R*)p->fy, p->perm, p->seg_start, p->seg_block,
        a ? a->block_active : nullptr, a ? a->ditems : p->ditems, a ? a->nditems : p->counts_all + 2,
        a ? a->tile_on : nullptr, p->seg_part, ms, g, R(2.0 / g.J), R(g.beta), kb_poly<R>(p), p->sched + 4, batch,
        (int64_t)(g.nx / 4 + 1) * 4 * g.Ky, (int64_t)p->M);
    return cudaGetLastError();
}

template <typename R>
cudaError_t degrid_plain(const pd_plan* p, const cplx_t<R>* grid, cplx_t<R>* out_user, cudaStream_t s, int batch) {
    cudaError_t e = cudaSuccess;
    PD_J_DISPATCH(p->g.J, (e = launch_degrid<R, JJ, 0>(p, grid, out_user, nullptr, s, batch)));
    return e;
}

template <typename R>
static cudaError_t block_norms(const pd_plan* p, const int32_t* active, const double* eps, double* res_norm,
                               int norm_only, cudaStream_t s) {
    k_block_norms<R><<<p->d, 128, 0, s>>>(p->seg_part, p->block_slot_start, p->block_slot_list,
                                                             active, eps, p->blk_norm, (R*)p->blk_scale, res_norm,
                                                             p->d, norm_only);
    return cudaGetLastError();
}

template <typename R>
cudaError_t degrid_dual(const pd_plan* p, const cplx_t<R>* grid, const DualArgs& a, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    prof_mark(PH_DEGRID, 0, s);
    PD_J_DISPATCH(p->g.J, (e = launch_degrid<R, JJ, 1>(p, grid, nullptr, &a, s)));
    prof_mark(PH_DEGRID, 1, s);
    if (e) return e;
    prof_mark(PH_NORMS, 0, s);
    e = block_norms<R>(p, a.block_active, a.eps, a.res_norm, 0, s);
    prof_mark(PH_NORMS, 1, s);
    return e;
}

template <typename R>
cudaError_t degrid_res_norms(const pd_plan* p, const cplx_t<R>* grid, const cplx_t<R>* y, double* res_norm,
                             cudaStream_t s) {
    // every block: the residual part of the pd-mode pass (its r output goes to the
    // plan's scratch and v is not needed, so y stands in for it), then ||G_i b - y_i||
    DualArgs a{y, (void*)y, nullptr, nullptr, res_norm, nullptr, p->ditems, p->counts_all + 2};
    cudaError_t e = cudaSuccess;
    PD_J_DISPATCH(p->g.J, (e = launch_degrid<R, JJ, 1>(p, grid, nullptr, &a, s)));
    return e ? e : block_norms<R>(p, nullptr, nullptr, res_norm, 1, s);
}

// Whether the plan grids with k_grid_mma (FP32 taps evaluated in the kernel, J <= 8, and the
// segment lists fit), its warps per CTA and its part size.
void grid_setup(pd_plan* p) {
    const Geo& g = p->g;
    const int ms = std::max(p->max_tile_segs, 1);
    // Seven working warps and the feeding one: 2 CTAs per SM by registers (at 16.8M points on a
    // 4096^2 grid 3 / 5 / 7 / 10 / 15 working warps take 445 / 415 / 360 / 485 / 448 us).
    p->grid_warps = 8;
    // Parts of a tile are added to U one after the other, so only a tile well above a CTA's
    // share of the points is split (at the same size 2048 points a part cost 23% more than
    // whole tiles of up to 9100).
    p->grid_part = (int)std::max<int64_t>(4096, p->M / (2 * p->num_sms));
    bool ok = p->prec == PD_F32 && g.J <= 8 && p->g_mode == PD_G_ON_THE_FLY && g.tile >= SC;
    const size_t smem = ok ? grid_mma_smem(g.tile, p->grid_warps - 1, ms) : 0;
    ok = ok && smem <= (size_t)p->max_smem - 1024;
    p->grid_smem = ok ? smem : 0;
}

// Tests only (pd_test_ordered_adds): one part too many pending for the first item's tile, so that
// the waits for it run out.
__global__ void k_hold(const int2* items, const int32_t* nitems, int32_t* pend) {
    if (*nitems > 0) pend[items[0].x] += 1;
}

template <int J, int MODE>
static cudaError_t launch_grid_mma(const pd_plan* p, const float2* src, const DualArgs* a, int32_t* pend, float2* U,
                                   int32_t* gave_up, cudaStream_t s, int batch) {
    const Geo& g = p->g;
    cudaError_t e;
    // A batch goes item by item, all images of each: image by image, overlapping tiles of one image wait
    // for one another with nothing else to do meanwhile (64 images of 256^2, 65,536 points: Phi^H 997
    // us, so 734; eight of 1024^2, 4.19M points: 2119, 1920).
    // Items with few points are held up by the feeding warps, one chain of loads and adds an item:
    // three working warps then, and twice the CTAs (the 64 images: 734 us with seven, 590 / 517 / 556
    // with four / three / two; eight of 512^2, 100,001 points: 320, 256 / 222 / 231, with 1.05M, 630 an
    // item: 568, 514 / 497 / 596). Not for one image, whose items are one or two a CTA, nor where they
    // hold many more points (the eight of 1024^2, 2300 an item: 2105, 2192 / 2728 / 3624 image by image).
    const bool few = batch > 1 && p->M <= (int64_t)p->n_items * 800 && (int64_t)p->n_items * batch >= (int64_t)p->num_sms * 8;
    const int warps = few ? 4 : p->grid_warps;
    const size_t smem = few ? grid_mma_smem(g.tile, warps - 1, std::max(p->max_tile_segs, 1)) : p->grid_smem;
    if ((e = ensure_smem(k_grid_mma<J, MODE>, smem))) return e;
    int per_sm = 1;
    if ((e = occupancy(&per_sm, k_grid_mma<J, MODE>, warps * 32, smem))) return e;
    const int ctas = (int)std::min<int64_t>((int64_t)p->n_items * batch, (int64_t)std::max(per_sm, 1) * p->num_sms);
    if (p->test_hold) k_hold<<<1, 1, 0, s>>>(a ? a->items : p->items, a ? a->nitems : p->nitems, pend);
    k_grid_mma<J, MODE><<<ctas, warps * 32, smem, s>>>(
        src, (const float2*)p->rbuf, a ? (float2*)a->v : nullptr, (const float*)p->blk_scale,
        a ? a->block_active : nullptr, p->cell, (const float*)p->fx, (const float*)p->fy, p->perm,
        p->seg_block, p->seg_sc_start, p->tile_info, a ? a->tile_on : nullptr, a ? a->items : p->items,
        a ? a->nitems : p->nitems, pend, U, std::max(p->max_tile_segs, 1), g, p->kbpoly, p->sched + 8, gave_up,
        p->wait_polls, batch, (int64_t)p->M, (int64_t)g.Kx * g.Ky);
    return cudaGetLastError();
}

#define PD_J8_DISPATCH(J_, CALL)                         \
    switch (J_) {                                        \
        case 2: { constexpr int JJ = 2; CALL; } break;   \
        case 4: { constexpr int JJ = 4; CALL; } break;   \
        case 6: { constexpr int JJ = 6; CALL; } break;   \
        case 8: { constexpr int JJ = 8; CALL; } break;   \
        default: return cudaErrorInvalidValue;           \
    }

template <typename R, int J, int MODE>
static cudaError_t launch_grid_j(const pd_plan* p, const cplx_t<R>* src, const DualArgs* a, const int32_t* tiles,
                                 const int32_t* count, cplx_t<R>* U, int* next_tile, cudaStream_t s, int batch) {
    if constexpr (J <= 8)
        if (p->g_mode == PD_G_CSR) return launch_grid_csr<R, J, MODE>(p, src, a, tiles, count, U, next_tile, s, batch);
    const Geo& g = p->g;
    const int ms = std::max(p->max_tile_segs, 1);
    const size_t lists = (size_t)(2 * ms + 1) * sizeof(int);
    const R toj = R(2.0 / g.J), beta = R(g.beta);
    const int ctas = std::min(g.ntiles, p->num_sms * 4);
    const cplx_t<R>* rb = (const cplx_t<R>*)p->rbuf;
    cplx_t<R>* vv = a ? (cplx_t<R>*)a->v : nullptr;
    const int32_t* act = a ? a->block_active : nullptr;
    cudaError_t e;
    if constexpr (J <= 8) {
        const int nw = std::max(1, g.tile / SC);
        const size_t smem8 = grid8w_smem<R>(g.tile, nw, ms);
        if ((e = ensure_smem(k_grid8w<R, J, MODE>, smem8))) return e;
        int per_sm = 0;
        int ctas8 = std::min(g.ntiles * batch, p->num_sms * 16);
        if (occupancy(&per_sm, k_grid8w<R, J, MODE>, nw * 32, smem8) ==
                cudaSuccess && per_sm > 0)
            ctas8 = std::min(ctas8, per_sm * p->num_sms);
        k_grid8w<R, J, MODE><<<ctas8, nw * 32, smem8, s>>>(
            src, rb, vv, (const R*)p->blk_scale, act, p->cell, (const R*)p->fx, (const R*)p->fy, p->perm,
            p->seg_start, p->seg_block, p->tile_seg_start, p->seg_sc_start, tiles, count, a ? a->tile_on : nullptr, U, ms, g, toj, beta,
            kb_poly<R>(p), next_tile, batch, (int64_t)p->M, (int64_t)g.Kx * g.Ky);
    } else {
        const size_t smem = (size_t)2 * g.ext * g.ext * sizeof(R) + lists;
        if ((e = ensure_smem(k_grid<R, J, MODE>, smem))) return e;
        for (int b = 0; b < batch; ++b)        // kernels wider than 8: one launch per image
            k_grid<R, J, MODE><<<ctas, 256, smem, s>>>(src ? src + (int64_t)b * p->M : src, rb, vv,
                                                      (const R*)p->blk_scale, act, p->cell, (const R*)p->fx,
                                                      (const R*)p->fy, p->perm, p->seg_start, p->seg_block,
                                                      p->tile_seg_start, tiles, count, a ? a->tile_on : nullptr,
                                                      U + (int64_t)b * g.Kx * g.Ky, ms, g, toj, beta, kb_poly<R>(p));
    }
    return cudaGetLastError();
}

// One launch per tile colour (their windows are disjoint within a colour), each taking
// its tiles from a dynamically claimed position of its list.
template <typename R>
static cudaError_t launch_grid(const pd_plan* p, int mode, const cplx_t<R>* src, const DualArgs* a,
                               const int32_t* const* tiles, const int32_t* counts4, cplx_t<R>* U, cudaStream_t s,
                               int batch = 1, int32_t* pend = nullptr, int32_t* gave_up = nullptr) {
    const Geo& g = p->g;
    cudaError_t e = cudaSuccess;
    prof_mark(PH_GRID, 0, s);
    if constexpr (sizeof(R) == 4) {
        if (p->grid_smem) {
            int32_t* pd = pend ? pend : p->pend;
            int32_t* gu = a ? a->gave_up : gave_up;
            if (!gu) gu = p->sched + 10;
            if (mode == 0) PD_J8_DISPATCH(g.J, (e = launch_grid_mma<JJ, 0>(p, src, a, pd, U, gu, s, batch)))
            else PD_J8_DISPATCH(g.J, (e = launch_grid_mma<JJ, 1>(p, src, a, pd, U, gu, s, 1)))
            prof_mark(PH_GRID, 1, s);
            return e;
        }
    }
    if ((e = cudaMemsetAsync(p->sched, 0, 4 * sizeof(int32_t), s))) return e;
    for (int c = 0; c < 4 && !e; ++c) {
        if (mode == 0) {
            PD_J_DISPATCH(g.J, (e = launch_grid_j<R, JJ, 0>(p, src, a, tiles[c], counts4 + c, U, p->sched + c, s,
                                                            batch)));
        } else {
            PD_J_DISPATCH(g.J, (e = launch_grid_j<R, JJ, 1>(p, src, a, tiles[c], counts4 + c, U, p->sched + c, s,
                                                            1)));
        }
    }
    prof_mark(PH_GRID, 1, s);
    return e ? e : cudaGetLastError();
}

template <typename R>
cudaError_t grid_plain(const pd_plan* p, const cplx_t<R>* y_user, cplx_t<R>* U, cudaStream_t s, int batch, int32_t* pend,
                       int32_t* gave_up) {
    // U = G^T y: every window is added to a zeroed grid
    cudaError_t e;
    const int64_t cells = (int64_t)batch * p->g.Kx * p->g.Ky;
    if (p->grid_smem) e = grid_begin(p, nullptr, pend ? pend : p->pend, (float4*)U, cells / 2, batch, s);
    else e = cudaMemsetAsync(U, 0, (size_t)cells * sizeof(cplx_t<R>), s);
    if (e) return e;
    const int q = p->g.ntiles / 4;
    const int32_t* lists[4] = {p->colour_tiles, p->colour_tiles + q, p->colour_tiles + 2 * q, p->colour_tiles + 3 * q};
    return launch_grid<R>(p, 0, y_user, nullptr, lists, p->colour_counts, U, s, batch, pend, gave_up);
}

template <typename R>
cudaError_t grid_dual(const pd_plan* p, const DualArgs& a, const int32_t* const* tiles, const int32_t* counts4,
                      cplx_t<R>* U, cudaStream_t s) {
    return launch_grid<R>(p, 1, nullptr, &a, tiles, counts4, U, s);
}

template cudaError_t degrid_plain<float>(const pd_plan*, const float2*, float2*, cudaStream_t, int);
template cudaError_t degrid_plain<double>(const pd_plan*, const double2*, double2*, cudaStream_t, int);
template cudaError_t degrid_res_norms<float>(const pd_plan*, const float2*, const float2*, double*, cudaStream_t);
template cudaError_t degrid_res_norms<double>(const pd_plan*, const double2*, const double2*, double*, cudaStream_t);
template cudaError_t degrid_dual<float>(const pd_plan*, const float2*, const DualArgs&, cudaStream_t);
template cudaError_t degrid_dual<double>(const pd_plan*, const double2*, const DualArgs&, cudaStream_t);
template cudaError_t grid_plain<float>(const pd_plan*, const float2*, float2*, cudaStream_t, int, int32_t*, int32_t*);
template cudaError_t grid_plain<double>(const pd_plan*, const double2*, double2*, cudaStream_t, int, int32_t*, int32_t*);
template cudaError_t grid_dual<float>(const pd_plan*, const DualArgs&, const int32_t* const*, const int32_t*,
                                      float2*, cudaStream_t);
template cudaError_t grid_dual<double>(const pd_plan*, const DualArgs&, const int32_t* const*, const int32_t*,
                                       double2*, cudaStream_t);

}  // namespace pdgb
