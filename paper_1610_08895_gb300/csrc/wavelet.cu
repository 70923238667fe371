// Sparsity dictionary Psi = b^{-1/2} [Psi_1 ... Psi_b] (Sec. 3: a collection of b
// bases, the Dirac basis and Daubechies wavelets db1..db8), and the sparsity dual
// update of Algorithm 1 steps 13-14.
//
// Periodic separable filter banks: analysis a_k = sum_j h_j x_{(2k+j) mod m},
// d_k = sum_j g_j x_{(2k+j) mod m}, g_j = (-1)^j h_{L-1-j}; rows then columns;
// L levels in the packed layout (coarsest approximation top-left). Synthesis is
// the transpose. Each CTA stages one input tile plus its filter halo in shared
// memory, filters rows then columns there, and writes the four sub-bands.
//
// Step 13 is s <- s + w - S_alpha(s + w) = clip(s + w, -alpha, alpha) (Moreau,
// eq. prox-L1), fused into the analysis epilogue; the change ds = s_new - s_old
// is synthesised and added to s~ (step 14) so that inactive bases cost nothing.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>

#include "common.cuh"
#include "host_math.hpp"
#include "plan.hpp"

namespace pdgb {

constexpr int AT = 32;   // analysis output tile edge (per sub-band)
constexpr int ST = 64;   // synthesis output tile edge
constexpr int NT_W = 256;

template <typename R> __device__ __forceinline__ R clip(R v, R a) { return v > a ? a : (v < -a ? -a : v); }

// -------------------------------------------------------------------- analysis
// The filter pair of one basis in registers: h (low-pass) and g_j = (-1)^j h_{LF-1-j}.
template <typename R, int LF>
__device__ __forceinline__ void load_filters(const R* __restrict__ filt, int k, R* h, R* g) {
#pragma unroll
    for (int j = 0; j < LF; ++j) {
        h[j] = filt[k * MAX_FILTER + j];
        g[j] = ((j & 1) ? R(-1) : R(1)) * filt[k * MAX_FILTER + LF - 1 - j];
    }
}

// Dispatch on the filter length of basis k (2, 4, ..., 16: db1 .. db8) to a body with the
// length as a compile-time constant (fully unrolled taps, filters in registers).
#define PD_LF_DISPATCH(lf_, CALL)                           \
    switch (lf_) {                                          \
        case 2: { constexpr int LF = 2; CALL; } break;      \
        case 4: { constexpr int LF = 4; CALL; } break;      \
        case 6: { constexpr int LF = 6; CALL; } break;      \
        case 8: { constexpr int LF = 8; CALL; } break;      \
        case 10: { constexpr int LF = 10; CALL; } break;    \
        case 12: { constexpr int LF = 12; CALL; } break;    \
        case 14: { constexpr int LF = 14; CALL; } break;    \
        default: { constexpr int LF = 16; CALL; } break;    \
    }

constexpr int ARB = 4;   // analysis outputs per thread along a row (row pass) or column (column pass)

// One analysis level of basis k on an output tile of ty x tx per sub-band at (oy0, ox0)
// of the (my x mx) region. Staged input rows have an odd pitch IWP and the row-pass
// results a pitch tx + 1, so that threads walking down a column hit distinct banks.
// Row pass: a thread computes ARB consecutive outputs of one input row from
// LF + 2 ARB - 2 staged values (consecutive threads take consecutive rows); column
// pass: ARB consecutive output rows of one column, the low-pass half (LL, LH) and then
// the high-pass half (HL, HH). MODE 0 writes the scaled coefficients, MODE 1 the
// step-13 update of s and its change ds.
template <typename R, int MODE, int LF>
__device__ __forceinline__ void dwt_body(const R* __restrict__ src, R* __restrict__ ll_out, R* __restrict__ out,
                                         R* __restrict__ ds, const R* __restrict__ wt, const R* __restrict__ filt,
                                         int k, int my, int mx,
                                         int oy0, int ox0, int ty, int tx, bool last, int64_t boff, int nx,
                                         int64_t ll_off, R scale, R alpha, R* sm) {
    constexpr int NX = LF + 2 * ARB - 2;               // staged values per ARB outputs
    const int hy = my >> 1, hx = mx >> 1;
    const int IH = 2 * ty + LF - 2, IW = 2 * tx + LF - 2, IWP = IW | 1, TP = tx + 1;
    R* in = sm;                                        // [IH][IWP]
    R* ra = in + IH * IWP;                             // [IH][TP]
    R* rd = ra + IH * TP;                              // [IH][TP]
    R h[LF], g[LF];
    load_filters<R, LF>(filt, k, h, g);
    stage_batched<8>(in, IH * IWP, [&](int i) {
        const int r = i / IWP, cc = i - r * IWP;
        const int gy = (2 * oy0 + r) & (my - 1), gx = (2 * ox0 + cc) & (mx - 1);
        return src[(int64_t)gy * mx + gx];
    });
    __syncthreads();
    // row pass
    const int nrg = (tx + ARB - 1) / ARB;
    for (int it = threadIdx.x; it < IH * nrg; it += blockDim.x) {
        const int r = it % IH, c0 = (it / IH) * ARB;
        const R* row = in + r * IWP + 2 * c0;
        R x[NX];
#pragma unroll
        for (int i = 0; i < NX; ++i) x[i] = (2 * c0 + i < IWP) ? row[i] : R(0);
#pragma unroll
        for (int o = 0; o < ARB; ++o) {
            R a = 0, d = 0;
#pragma unroll
            for (int j = 0; j < LF; ++j) { a += h[j] * x[2 * o + j]; d += g[j] * x[2 * o + j]; }
            if (c0 + o < tx) { ra[r * TP + c0 + o] = a; rd[r * TP + c0 + o] = d; }
        }
    }
    __syncthreads();
    // column pass: rows r0 .. r0 + ARB - 1 of column c
    const int ncg = (ty + ARB - 1) / ARB;
    for (int item = threadIdx.x; item < ncg * tx; item += blockDim.x) {
        const int c = item % tx, r0 = (item / tx) * ARB;
        const int ox = ox0 + c;
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            // half 0: the low-pass rows (LL, LH); half 1: the high-pass rows (HL, HH)
            const R* rr = half ? rd : ra;
            R sold[ARB][2];
            if (MODE == 1) {
#pragma unroll
                for (int o = 0; o < ARB; ++o) {
                    const int oy = oy0 + r0 + o;
                    if (r0 + o < ty) {
                        sold[o][0] = half ? out[boff + (int64_t)oy * nx + hx + ox]
                                          : (last ? out[boff + (int64_t)oy * nx + ox] : R(0));
                        sold[o][1] = out[boff + (int64_t)(hy + oy) * nx + (half ? hx : 0) + ox];
                    }
                }
            }
            R v[NX];
#pragma unroll
            for (int i = 0; i < NX; ++i) v[i] = 2 * r0 + i < IH ? rr[(2 * r0 + i) * TP + c] : R(0);
#pragma unroll
            for (int o = 0; o < ARB; ++o) {
                if (r0 + o >= ty) break;
                R lo = 0, hi = 0;
#pragma unroll
                for (int j = 0; j < LF; ++j) { lo += h[j] * v[2 * o + j]; hi += g[j] * v[2 * o + j]; }
                const int oy = oy0 + r0 + o;
                // low-pass along y: LL (half 0) or HL (half 1); high-pass along y: LH or HH
                const int64_t p_lo = boff + (int64_t)oy * nx + (half ? hx : 0) + ox;
                const int64_t p_hi = boff + (int64_t)(hy + oy) * nx + (half ? hx : 0) + ox;
                const bool store_lo = half || last;
                if (MODE == 0) {
                    if (store_lo) out[p_lo] = lo * scale;
                    out[p_hi] = hi * scale;
                } else {
                    // weighted prior: the threshold of each coefficient is alpha times its weight
                    if (store_lo) {
                        const R so = sold[o][0], sn = clip(so + lo * scale, wt ? alpha * wt[p_lo] : alpha);
                        out[p_lo] = sn; ds[p_lo] = sn - so;
                    }
                    const R so = sold[o][1], sn = clip(so + hi * scale, wt ? alpha * wt[p_hi] : alpha);
                    out[p_hi] = sn; ds[p_hi] = sn - so;
                }
                if (!half && !last) ll_out[ll_off + (int64_t)oy * hx + ox] = lo;
            }
        }
    }
}

// ---- FP32 levels on tiles of T x T per sub-band (both sides of the sub-bands multiples of T)
// The same filter bank as above, laid out for the FP32 pipes: every thread keeps the taps as
// pairs (h_j, g_j) and runs both filters in one packed multiply-add per value; rows are staged
// and filtered in 16-byte pieces (pitches of an odd number of pieces: eight threads of a
// quarter-warp on eight rows hit distinct banks), and in the column pass a warp's threads take
// consecutive columns. Bound by instruction issue (2 LF multiply-adds a pixel). The analysis of
// an iteration at 2048^2 (half of nine bases, four levels): 217 -> 124 us; at 256^2: 54 -> 25 us.
__device__ __forceinline__ float2 dup2(float x) { return make_float2(x, x); }

template <int LF, int T> struct Dwt32Shape {
    static constexpr int IH = 2 * T + LF - 2;             // staged rows
    static constexpr int IW4 = (2 * T + LF - 2 + 3) / 4;  // staged 16-byte pieces per row
    static constexpr int IP = 4 * (IW4 | 1), RP = T + 4;  // pitches: staged rows, row-pass results
    static constexpr int FLOATS = IH * (IP + 2 * RP);
};
template <int T> constexpr size_t dwt32_smem() { return (size_t)Dwt32Shape<MAX_FILTER, T>::FLOATS * sizeof(float); }
template <int T> constexpr int dwt32_threads() { return T == 32 ? 256 : 128; }

template <int MODE, int LF, int T>
__device__ __forceinline__ void dwt32_body(const float* __restrict__ src, float* __restrict__ ll_out,
                                           float* __restrict__ out, float* __restrict__ ds,
                                           const float* __restrict__ wt, const float* __restrict__ filt, int k, int my,
                                           int mx, int oy0, int ox0, bool last, int64_t boff, int nx, int64_t ll_off,
                                           float scale, float alpha, float* sm) {
    using S = Dwt32Shape<LF, T>;
    constexpr int NT = dwt32_threads<T>();
    const int hy = my >> 1, hx = mx >> 1;
    float* in = sm;                                   // [IH][IP]
    float* ra = in + S::IH * S::IP;                   // [IH][RP]
    float* rd = ra + S::IH * S::RP;                   // [IH][RP]
    // stage the tile and its halo (periodic), several rows' loads in flight
    {
        constexpr int N = S::IH * S::IW4, UB = 6;
#pragma unroll 1
        for (int base = threadIdx.x; base < N; base += UB * NT) {
            float4 v[UB];
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int i = base + u * NT, rr = i / S::IW4, q = i - rr * S::IW4;
                if (i < N)
                    v[u] = *reinterpret_cast<const float4*>(src + (int64_t)((2 * oy0 + rr) & (my - 1)) * mx +
                                                            ((2 * ox0 + 4 * q) & (mx - 1)));
            }
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int i = base + u * NT, rr = i / S::IW4, q = i - rr * S::IW4;
                if (i < N) *reinterpret_cast<float4*>(in + rr * S::IP + 4 * q) = v[u];
            }
        }
    }
    float2 hg[LF];
#pragma unroll
    for (int j = 0; j < LF; ++j)
        hg[j] = make_float2(filt[k * MAX_FILTER + j], ((j & 1) ? -1.f : 1.f) * filt[k * MAX_FILTER + LF - 1 - j]);
    __syncthreads();
    // row pass: four outputs of one row a thread, consecutive threads on consecutive rows
#pragma unroll 1
    for (int it = threadIdx.x; it < S::IH * (T / 4); it += NT) {
        const int gr = it / S::IH, rr = it - gr * S::IH;
        constexpr int NX4 = (LF + 6 + 3) / 4;
        float x[4 * NX4];
#pragma unroll
        for (int q = 0; q < NX4; ++q) {
            const float4 v = *reinterpret_cast<const float4*>(in + rr * S::IP + 8 * gr + 4 * q);
            x[4 * q] = v.x; x[4 * q + 1] = v.y; x[4 * q + 2] = v.z; x[4 * q + 3] = v.w;
        }
        float2 acc[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[o] = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < LF + 6; ++i) {
            const float2 xx = dup2(x[i]);
#pragma unroll
            for (int o = 0; o < 4; ++o)
                if (i - 2 * o >= 0 && i - 2 * o < LF) acc[o] = ffma2(hg[i - 2 * o], xx, acc[o]);
        }
        *reinterpret_cast<float4*>(ra + rr * S::RP + 4 * gr) = make_float4(acc[0].x, acc[1].x, acc[2].x, acc[3].x);
        *reinterpret_cast<float4*>(rd + rr * S::RP + 4 * gr) = make_float4(acc[0].y, acc[1].y, acc[2].y, acc[3].y);
    }
    __syncthreads();
    // column pass: RO output rows of one column of the low- (LL, LH) or high-pass (HL, HH) half
    constexpr int RO = T == 32 ? 8 : 4;
    static_assert(2 * T * (T / RO) <= 2 * NT, "at most two items a thread");
#pragma unroll 1
    for (int it = threadIdx.x; it < 2 * T * (T / RO); it += NT) {
        const int c = it % T, r0 = (it / T) % (T / RO) * RO, half = it / (T * (T / RO));
        const float* rr = half ? rd : ra;
        const bool store_lo = half || last;
        const int64_t p_lo = boff + (int64_t)(oy0 + r0) * nx + (half ? hx : 0) + ox0 + c;
        const int64_t p_hi = p_lo + (int64_t)hy * nx;
        float so[RO], th[RO];
        if (MODE == 1) {
#pragma unroll
            for (int o = 0; o < RO; ++o) {
                if (store_lo) so[o] = out[p_lo + (int64_t)o * nx];
                th[o] = out[p_hi + (int64_t)o * nx];
            }
        }
        float2 acc[RO];
#pragma unroll
        for (int o = 0; o < RO; ++o) acc[o] = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < LF + 2 * RO - 2; ++i) {
            const float2 xx = dup2(rr[(2 * r0 + i) * S::RP + c]);
#pragma unroll
            for (int o = 0; o < RO; ++o)
                if (i - 2 * o >= 0 && i - 2 * o < LF) acc[o] = ffma2(hg[i - 2 * o], xx, acc[o]);
        }
#pragma unroll
        for (int o = 0; o < RO; ++o) {
            const int64_t pl = p_lo + (int64_t)o * nx, ph = p_hi + (int64_t)o * nx;
            if (MODE == 0) {
                if (store_lo) out[pl] = acc[o].x * scale;
                out[ph] = acc[o].y * scale;
            } else {
                // weighted prior: the threshold of each coefficient is alpha times its weight
                if (store_lo) {
                    const float sn = clip(so[o] + acc[o].x * scale, wt ? alpha * wt[pl] : alpha);
                    out[pl] = sn;
                    ds[pl] = sn - so[o];
                }
                const float sn = clip(th[o] + acc[o].y * scale, wt ? alpha * wt[ph] : alpha);
                out[ph] = sn;
                ds[ph] = sn - th[o];
            }
            if (!half && !last) ll_out[ll_off + (int64_t)(oy0 + r0 + o) * hx + ox0 + c] = acc[o].x;
        }
    }
}

// One FP32 level for every basis in blockIdx.z; level 0 also treats the Dirac bases (the
// identity, elementwise on the tile's 2T x 2T pixels).
template <int MODE, int T>
__global__ void __launch_bounds__(dwt32_threads<T>(), T == 32 ? (MODE == 0 ? 3 : 2) : 6) k_dwt32_level(
    const float* __restrict__ x0, const float* __restrict__ ll_in, float* __restrict__ ll_out, float* __restrict__ out,
    float* __restrict__ ds, const float* __restrict__ wt, const float* __restrict__ filt,
    const int32_t* __restrict__ flen, const int32_t* __restrict__ active, int level, int L, int ny, int nx, float scale,
    float alpha) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int k = blockIdx.z;
    const int lf = flen[k];
    if (lf == 0 && level > 0) return;
    if (MODE == 1 && !active[k]) return;
    const int my = ny >> level, mx = nx >> level;
    const int oy0 = blockIdx.y * T, ox0 = blockIdx.x * T;
    const int64_t boff = (int64_t)k * ny * nx, ll_off = (int64_t)k * (ny / 2) * (nx / 2);
    if (lf == 0) {
        for (int i = threadIdx.x; i < 2 * T * (T / 2); i += dwt32_threads<T>()) {
            const int rr = i / (T / 2), q = i % (T / 2);
            const int64_t at = (int64_t)(2 * oy0 + rr) * nx + 2 * ox0 + 4 * q;
            const float4 x = *reinterpret_cast<const float4*>(x0 + at);
            float4* o = reinterpret_cast<float4*>(out + boff + at);
            if (MODE == 0) {
                *o = make_float4(x.x * scale, x.y * scale, x.z * scale, x.w * scale);
            } else {
                const float4 so = *o;
                float4 a = make_float4(alpha, alpha, alpha, alpha), sn;
                if (wt) {
                    const float4 w = *reinterpret_cast<const float4*>(wt + boff + at);
                    a = make_float4(alpha * w.x, alpha * w.y, alpha * w.z, alpha * w.w);
                }
                sn.x = clip(so.x + x.x * scale, a.x); sn.y = clip(so.y + x.y * scale, a.y);
                sn.z = clip(so.z + x.z * scale, a.z); sn.w = clip(so.w + x.w * scale, a.w);
                *o = sn;
                *reinterpret_cast<float4*>(ds + boff + at) =
                    make_float4(sn.x - so.x, sn.y - so.y, sn.z - so.z, sn.w - so.w);
            }
        }
        return;
    }
    const float* src = level == 0 ? x0 : ll_in + ll_off;
    float* sm = reinterpret_cast<float*>(smraw);
    PD_LF_DISPATCH(lf, (dwt32_body<MODE, LF, T>(src, ll_out, out, ds, wt, filt, k, my, mx, oy0, ox0, level == L - 1, boff,
                                                nx, ll_off, scale, alpha, sm)));
}

// One level for every basis in blockIdx.z. MODE 0: out = coefficient * scale.
// MODE 1: s/ds update of step 13 (wt: per-coefficient weights of the reweighted prior,
// same layout as s, or null). The last level also treats the approximation band.
template <typename R, int MODE>
__global__ void __launch_bounds__(NT_W, 3) k_dwt_level(const R* __restrict__ x0, const R* __restrict__ ll_in,
                                                    R* __restrict__ ll_out, R* __restrict__ out, R* __restrict__ ds,
                                                    const R* __restrict__ wt,
                                                    const R* __restrict__ filt, const int32_t* __restrict__ flen,
                                                    const int32_t* __restrict__ active, int level, int L, int ny,
                                                    int nx, R scale, R alpha) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int k = blockIdx.z;
    const int lf = flen[k];
    if (lf == 0) return;                               // Dirac basis: separate kernel
    if (MODE == 1 && !active[k]) return;
    const int my = ny >> level, mx = nx >> level;
    const int hy = my >> 1, hx = mx >> 1;
    const int ty = min(AT, hy), tx = min(AT, hx);
    const int oy0 = blockIdx.y * ty, ox0 = blockIdx.x * tx;
    if (oy0 >= hy || ox0 >= hx) return;
    const R* src = level == 0 ? x0 : ll_in + (int64_t)k * (ny / 2) * (nx / 2);
    const int64_t boff = (int64_t)k * ny * nx, ll_off = (int64_t)k * (ny / 2) * (nx / 2);
    const bool last = level == L - 1;
    R* sm = reinterpret_cast<R*>(smraw);
    PD_LF_DISPATCH(lf, (dwt_body<R, MODE, LF>(src, ll_out, out, ds, wt, filt, k, my, mx, oy0, ox0, ty, tx, last, boff,
                                              nx, ll_off, scale, alpha, sm)));
}

// Dirac basis (identity): MODE 0 copies x * scale, MODE 1 applies step 13 elementwise.
template <typename R, int MODE>
__global__ void k_dirac(const R* __restrict__ x, R* __restrict__ out, R* __restrict__ ds,
                        const R* __restrict__ wt, const int32_t* __restrict__ flen,
                        const int32_t* __restrict__ active, int b, int64_t n, R scale, R alpha) {
    for (int k = 0; k < b; ++k) {
        if (flen[k] != 0 || (MODE == 1 && !active[k])) continue;
        R* o = out + (int64_t)k * n;
        R* d = ds + (int64_t)k * n;
        const R* wk = wt ? wt + (int64_t)k * n : nullptr;
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
            if (MODE == 0) {
                o[i] = x[i] * scale;
            } else {
                const R so = o[i], sn = clip(so + x[i] * scale, wk ? alpha * wk[i] : alpha);
                o[i] = sn;
                d[i] = sn - so;
            }
        }
    }
}

// -------------------------------------------------------------------- synthesis
constexpr int SRP = 2;   // synthesis: output row pairs per thread (column pass), column pairs (row pass)

// Reconstruct a (ty x tx) tile of the level-`level` region (size my x mx) of basis k from
// its four sub-bands; the approximation band comes from ll_in (or from the packed
// coefficients at the coarsest level). Result left in `res` (shared, [ty][tx + 1]).
// Output rows 2m and 2m + 1 both read the sub-band rows m + off - i, i < LF/2 (even and
// odd taps): a thread computes SRP row pairs of one column from LF/2 + SRP - 1 staged
// values per band; the row pass likewise along the rows.
template <typename R, int LF>
__device__ __forceinline__ void synth_tile(const R* __restrict__ coef, const R* __restrict__ ll_in,
                                           const R* __restrict__ filt, int k, int level, int L, int ny, int nx,
                                           int oy0, int ox0, int ty, int tx, R* sm, R* res) {
    constexpr int NV = LF / 2 + SRP - 1, OFF = LF / 2 - 1;
    const int my = ny >> level, mx = nx >> level;
    const int hy = my >> 1, hx = mx >> 1;
    const int NKy = ty / 2 + LF / 2 - 1, NKx = tx / 2 + LF / 2 - 1;
    const int kby = oy0 / 2 - LF / 2 + 1, kbx = ox0 / 2 - LF / 2 + 1;
    R* LLs = sm;                      // [NKy][NKx] x4 sub-bands
    R* HLs = LLs + NKy * NKx;
    R* LHs = HLs + NKy * NKx;
    R* HHs = LHs + NKy * NKx;
    const int NKP = NKx | 1;          // odd pitch: threads walking down a column hit distinct banks
    R* lo = HHs + NKy * NKx;          // [ty][NKP] columns synthesised, low-x half
    R* hi = lo + ty * NKP;
    R h[LF], g[LF];
    load_filters<R, LF>(filt, k, h, g);
    const int64_t boff = (int64_t)k * ny * nx;
    const bool coarsest = level == L - 1;
    const R* llsrc = ll_in + (int64_t)k * (ny / 2) * (nx / 2);
    constexpr int UB = 2;                 // rows of the strided loop whose loads go out together
    for (int base = threadIdx.x; base < NKy * NKx; base += UB * (int)blockDim.x) {
        R v[UB][4];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int i = base + u * (int)blockDim.x;
            if (i < NKy * NKx) {
                const int r = i / NKx, c = i - r * NKx;
                const int gy = (kby + r) & (hy - 1), gx = (kbx + c) & (hx - 1);
                v[u][0] = coarsest ? coef[boff + (int64_t)gy * nx + gx] : llsrc[(int64_t)gy * hx + gx];
                v[u][1] = coef[boff + (int64_t)gy * nx + hx + gx];
                v[u][2] = coef[boff + (int64_t)(hy + gy) * nx + gx];
                v[u][3] = coef[boff + (int64_t)(hy + gy) * nx + hx + gx];
            }
        }
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int i = base + u * (int)blockDim.x;
            if (i < NKy * NKx) { LLs[i] = v[u][0]; HLs[i] = v[u][1]; LHs[i] = v[u][2]; HHs[i] = v[u][3]; }
        }
    }
    __syncthreads();
    // column pass: rows 2m .. 2m + 2 SRP - 1 of column c of lo and hi
    const int npr = (ty / 2 + SRP - 1) / SRP;
    for (int it = threadIdx.x; it < npr * NKx; it += blockDim.x) {
        const int c = it % NKx, m0 = (it / NKx) * SRP;
        R a[4][NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int kk = m0 + OFF - (LF / 2 - 1) + i;      // sub-band rows m0 + OFF - (LF/2 - 1) ...
            const bool ok = kk < NKy;
            a[0][i] = ok ? LLs[kk * NKx + c] : R(0);
            a[1][i] = ok ? LHs[kk * NKx + c] : R(0);
            a[2][i] = ok ? HLs[kk * NKx + c] : R(0);
            a[3][i] = ok ? HHs[kk * NKx + c] : R(0);
        }
#pragma unroll
        for (int pq = 0; pq < SRP; ++pq) {
            const int m = m0 + pq;
            if (2 * m >= ty) break;
#pragma unroll
            for (int par = 0; par < 2; ++par) {
                R l = 0, hh = 0;
#pragma unroll
                for (int i = 0; i < LF / 2; ++i) {
                    // tap j = 2 i + par reads sub-band row m + OFF - i = a[.][pq + LF/2 - 1 - i]
                    const int j = 2 * i + par, q = pq + LF / 2 - 1 - i;
                    l += h[j] * a[0][q] + g[j] * a[1][q];
                    hh += h[j] * a[2][q] + g[j] * a[3][q];
                }
                lo[(2 * m + par) * NKP + c] = l;
                hi[(2 * m + par) * NKP + c] = hh;
            }
        }
    }
    __syncthreads();
    // row pass: columns 2m .. 2m + 2 SRP - 1 of row r (consecutive threads take consecutive rows)
    const int npc = (tx / 2 + SRP - 1) / SRP;
    for (int it = threadIdx.x; it < ty * npc; it += blockDim.x) {
        const int r = it % ty, m0 = (it / ty) * SRP;
        R bl[NV], bh[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int kk = m0 + i;
            bl[i] = kk < NKx ? lo[r * NKP + kk] : R(0);
            bh[i] = kk < NKx ? hi[r * NKP + kk] : R(0);
        }
#pragma unroll
        for (int pq = 0; pq < SRP; ++pq) {
            const int m = m0 + pq;
            if (2 * m >= tx) break;
#pragma unroll
            for (int par = 0; par < 2; ++par) {
                R v = 0;
#pragma unroll
                for (int i = 0; i < LF / 2; ++i) {
                    const int j = 2 * i + par, q = pq + LF / 2 - 1 - i;
                    v += h[j] * bl[q] + g[j] * bh[q];
                }
                res[r * (tx + 1) + 2 * m + par] = v;
            }
        }
    }
    __syncthreads();
}

// FP32 tiles of 2P x 2P (P pairs of rows and columns, both sides of the sub-bands multiples of
// P): an output pair (2m, 2m + 1) takes the tap pairs (h_2i, h_2i+1) and (g_2i, g_2i+1), so
// each value is one packed multiply-add; bands are staged from a column that is a multiple of
// four (16-byte pieces) on. The synthesis of an iteration at 2048^2: 192 -> 111 us; at 256^2:
// 43 -> 27 us.
template <int LF, int P> struct Idwt32Shape {
    static constexpr int NK = P + LF / 2 - 1;             // staged rows of a band
    static constexpr int HA = (LF / 2 - 1 + 3) / 4 * 4;   // staged columns before the tile
    static constexpr int NC4 = (P + HA) / 4, BP = 4 * (NC4 | 1);
    static constexpr int FLOATS = 4 * NK * BP + 2 * (2 * P) * BP;
};
template <int P> constexpr size_t idwt32_smem() { return (size_t)Idwt32Shape<MAX_FILTER, P>::FLOATS * sizeof(float); }
template <int P> constexpr int idwt32_threads() { return P == 32 ? 256 : 128; }

template <int LF, int P>
__device__ __forceinline__ void idwt32_body(const float* __restrict__ coef, const float* __restrict__ ll_in,
                                            const float* __restrict__ filt, int k, int level, int L, int ny, int nx,
                                            int oy0, int ox0, float* __restrict__ dst, float* sm) {
    using S = Idwt32Shape<LF, P>;
    constexpr int NT = idwt32_threads<P>();
    const int mx = nx >> level, hy = (ny >> level) >> 1, hx = mx >> 1;
    float* band = sm;                                 // [4][NK][BP]: LL, LH, HL, HH
    float* col = sm + 4 * S::NK * S::BP;              // [2][2P][BP]: columns synthesised, low- and high-x half
    const int64_t boff = (int64_t)k * ny * nx;
    const bool coarsest = level == L - 1;
    const float* ll = coarsest ? coef + boff : ll_in + (int64_t)k * (ny / 2) * (nx / 2);
    const int llp = coarsest ? nx : hx;
    const int ky0 = oy0 / 2 - (LF / 2 - 1), kx0 = ox0 / 2 - S::HA;
    {
        constexpr int N = S::NK * S::NC4, UB = 2;
#pragma unroll 1
        for (int base = threadIdx.x; base < N; base += UB * NT) {
            float4 v[UB][4];
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int i = base + u * NT, rr = i / S::NC4, q = i - rr * S::NC4;
                if (i < N) {
                    const int gy = (ky0 + rr) & (hy - 1), gx = (kx0 + 4 * q) & (hx - 1);
                    const float* c = coef + boff + (int64_t)gy * nx + gx;
                    v[u][0] = *reinterpret_cast<const float4*>(ll + (int64_t)gy * llp + gx);
                    v[u][1] = *reinterpret_cast<const float4*>(c + (int64_t)hy * nx);
                    v[u][2] = *reinterpret_cast<const float4*>(c + hx);
                    v[u][3] = *reinterpret_cast<const float4*>(c + (int64_t)hy * nx + hx);
                }
            }
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int i = base + u * NT, rr = i / S::NC4, q = i - rr * S::NC4;
                if (i < N) {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        *reinterpret_cast<float4*>(band + (e * S::NK + rr) * S::BP + 4 * q) = v[u][e];
                }
            }
        }
    }
    float2 hp[LF / 2], gp[LF / 2];                    // tap pairs (even, odd)
#pragma unroll
    for (int i = 0; i < LF / 2; ++i) {
        hp[i] = make_float2(filt[k * MAX_FILTER + 2 * i], filt[k * MAX_FILTER + 2 * i + 1]);
        gp[i] = make_float2(filt[k * MAX_FILTER + LF - 1 - 2 * i], -filt[k * MAX_FILTER + LF - 2 - 2 * i]);
    }
    __syncthreads();
    // column pass: four row pairs of one column of the low- (LL, LH) or high-x (HL, HH) half
    constexpr int NC = P + S::HA;
#pragma unroll 1
    for (int it = threadIdx.x; it < 2 * NC * (P / 4); it += NT) {
        const int c = it % NC, q = it / NC, m0 = q % (P / 4) * 4, half = q / (P / 4);
        const float* b0 = band + 2 * half * S::NK * S::BP + c;
        const float* b1 = b0 + S::NK * S::BP;
        float2 acc[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[o] = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < LF / 2 + 3; ++i) {        // band row m0 + i meets tap pair o + LF/2 - 1 - i of pair o
            const float2 a = dup2(b0[(m0 + i) * S::BP]), e = dup2(b1[(m0 + i) * S::BP]);
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const int j = o + LF / 2 - 1 - i;
                if (j >= 0 && j < LF / 2) {
                    acc[o] = ffma2(hp[j], a, acc[o]);
                    acc[o] = ffma2(gp[j], e, acc[o]);
                }
            }
        }
        float* w = col + (half * 2 * P + 2 * m0) * S::BP + c;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            w[2 * o * S::BP] = acc[o].x;
            w[(2 * o + 1) * S::BP] = acc[o].y;
        }
    }
    __syncthreads();
    // row pass: four column pairs of one row, consecutive threads along the row
#pragma unroll 1
    for (int it = threadIdx.x; it < 2 * P * (P / 4); it += NT) {
        const int rr = it / (P / 4), m0 = it % (P / 4) * 4;
        constexpr int NV = S::HA + 4;
        float bl[NV], bh[NV];
#pragma unroll
        for (int q = 0; q < NV / 4; ++q) {
            const float4 a = *reinterpret_cast<const float4*>(col + rr * S::BP + m0 + 4 * q);
            const float4 e = *reinterpret_cast<const float4*>(col + (2 * P + rr) * S::BP + m0 + 4 * q);
            bl[4 * q] = a.x; bl[4 * q + 1] = a.y; bl[4 * q + 2] = a.z; bl[4 * q + 3] = a.w;
            bh[4 * q] = e.x; bh[4 * q + 1] = e.y; bh[4 * q + 2] = e.z; bh[4 * q + 3] = e.w;
        }
        float2 acc[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[o] = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < NV; ++i) {                // staged column m0 + i meets tap pair o + HA - i of pair o
            const float2 a = dup2(bl[i]), e = dup2(bh[i]);
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const int j = o + S::HA - i;
                if (j >= 0 && j < LF / 2) {
                    acc[o] = ffma2(hp[j], a, acc[o]);
                    acc[o] = ffma2(gp[j], e, acc[o]);
                }
            }
        }
        float4* o4 = reinterpret_cast<float4*>(dst + (int64_t)(oy0 + rr) * mx + ox0 + 2 * m0);
        o4[0] = make_float4(acc[0].x, acc[0].y, acc[1].x, acc[1].y);
        o4[1] = make_float4(acc[2].x, acc[2].y, acc[3].x, acc[3].y);
    }
}

template <int P>
__global__ void __launch_bounds__(idwt32_threads<P>(), P == 32 ? 3 : 6) k_idwt32_level(
    const float* __restrict__ coef, const float* __restrict__ ll_in, float* __restrict__ ll_out,
    const float* __restrict__ filt, const int32_t* __restrict__ flen, const int32_t* __restrict__ active, int level,
    int L, int ny, int nx, int64_t out_stride) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int k = blockIdx.z;
    const int lf = flen[k];
    if (lf == 0 || (active && !active[k])) return;
    PD_LF_DISPATCH(lf, (idwt32_body<LF, P>(coef, ll_in, filt, k, level, L, ny, nx, blockIdx.y * 2 * P, blockIdx.x * 2 * P,
                                           ll_out + (int64_t)k * out_stride, reinterpret_cast<float*>(smraw))));
}

// One level of one basis per blockIdx.z: reconstruct the (ny>>level) x (nx>>level)
// approximation of the next finer level into ll_out + basis * out_stride (at level 0:
// the basis's full-size synthesis).
template <typename R>
__global__ void __launch_bounds__(NT_W) k_idwt_level(const R* __restrict__ coef, const R* __restrict__ ll_in,
                                                     R* __restrict__ ll_out, const R* __restrict__ filt,
                                                     const int32_t* __restrict__ flen,
                                                     const int32_t* __restrict__ active, int level, int L, int ny,
                                                     int nx, int64_t out_stride) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int k = blockIdx.z;
    const int lf = flen[k];
    if (lf == 0) return;
    if (active && !active[k]) return;
    const int my = ny >> level, mx = nx >> level;
    const int ty = min(ST, my), tx = min(ST, mx);
    const int oy0 = blockIdx.y * ty, ox0 = blockIdx.x * tx;
    if (oy0 >= my || ox0 >= mx) return;
    R* sm = reinterpret_cast<R*>(smraw);
    R* res = sm + 4 * (ty / 2 + MAX_FILTER / 2) * (tx / 2 + MAX_FILTER / 2) + 2 * ty * ((tx / 2 + MAX_FILTER / 2) | 1);
    PD_LF_DISPATCH(lf, (synth_tile<R, LF>(coef, ll_in, filt, k, level, L, ny, nx, oy0, ox0, ty, tx, sm, res)));
    R* dst = ll_out + (int64_t)k * out_stride;
    for (int i = threadIdx.x; i < ty * tx; i += blockDim.x) {
        const int r = i / tx, c = i - r * tx;
        dst[(int64_t)(oy0 + r) * mx + ox0 + c] = res[r * (tx + 1) + c];
    }
}

// Sum of the bases' level-0 syntheses (the Dirac basis is its coefficients) over the
// active bases in basis order: MODE 0: out = acc * scale, MODE 1: out += acc * scale
// (the s~ update of step 14). Four consecutive pixels per thread.
template <typename R> struct Quad { R a, b, c, d; };
template <typename R, bool VEC> __device__ __forceinline__ Quad<R> ldq(const R* p) {
    if constexpr (!VEC) {
        return {p[0], p[1], p[2], p[3]};
    } else if constexpr (sizeof(R) == 4) {
        const float4 q = *reinterpret_cast<const float4*>(p);
        return {q.x, q.y, q.z, q.w};
    } else {
        const double2 q0 = *reinterpret_cast<const double2*>(p), q1 = *reinterpret_cast<const double2*>(p + 2);
        return {q0.x, q0.y, q1.x, q1.y};
    }
}
template <typename R, bool VEC> __device__ __forceinline__ void stq(R* p, const Quad<R>& v) {
    if constexpr (!VEC) {
        p[0] = v.a; p[1] = v.b; p[2] = v.c; p[3] = v.d;
    } else if constexpr (sizeof(R) == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(v.a, v.b, v.c, v.d);
    } else {
        *reinterpret_cast<double2*>(p) = make_double2(v.a, v.b);
        *reinterpret_cast<double2*>(p + 2) = make_double2(v.c, v.d);
    }
}

// VEC: both the coefficients and the output are 16-byte aligned (a caller's may start anywhere).
template <typename R, int MODE, bool VEC>
__global__ void __launch_bounds__(256) k_syn_sum(const R* __restrict__ coef, const R* __restrict__ part,
                                                 const int32_t* __restrict__ flen, const int32_t* __restrict__ active,
                                                 int b, int64_t n, R* __restrict__ out, R scale) {
    for (int64_t i4 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; 4 * i4 < n; i4 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = 4 * i4;
        Quad<R> acc{R(0), R(0), R(0), R(0)};
        for (int k = 0; k < b; ++k) {
            if (MODE == 1 && !active[k]) continue;
            const Quad<R> v = ldq<R, VEC>((flen[k] == 0 ? coef : part) + (int64_t)k * n + i);
            acc.a += v.a; acc.b += v.b; acc.c += v.c; acc.d += v.d;
        }
        Quad<R> o{acc.a * scale, acc.b * scale, acc.c * scale, acc.d * scale};
        if (MODE == 1) {
            const Quad<R> prev = ldq<R, VEC>(out + i);
            o.a += prev.a; o.b += prev.b; o.c += prev.c; o.d += prev.d;
        }
        stq<R, VEC>(out + i, o);
    }
}

// -------------------------------------------------------------------- launchers
template <typename R> static size_t ana_smem(int ty, int tx) {
    const int IH = 2 * ty + MAX_FILTER - 2, IWP = (2 * tx + MAX_FILTER - 2) | 1;
    return (size_t)(IH * IWP + 2 * IH * (tx + 1)) * sizeof(R);
}
template <typename R> static size_t syn_smem(int ty, int tx) {
    const int NKy = ty / 2 + MAX_FILTER / 2, NKx = tx / 2 + MAX_FILTER / 2;
    return (size_t)(4 * NKy * NKx + 2 * ty * (NKx | 1) + ty * (tx + 1)) * sizeof(R);
}

// FP32 tile edge of a level whose sub-bands are hy x hx: 32, or 16 where tiles of 32 would
// leave SMs without a CTA (at 256^2 the levels are one CTA's latency), 0 below 16 (the
// generic kernel).
static int dwt32_tile(int hy, int hx, int b, int sms) {
    if (hy < 16 || hx < 16) return 0;
    if (hy < 32 || hx < 32) return 16;
    return (int64_t)(hy / 32) * (hx / 32) * b >= 2 * (int64_t)sms ? 32 : 16;
}

// One analysis level of all bases (and, at level 0, the Dirac bases).
template <int MODE, typename R>
static cudaError_t analysis_level(const R* x, const R* llin, R* llout, R* out, R* ds, const R* wt, const R* filt,
                                  const int32_t* flen, const int32_t* active, int b, int lev, int L, int ny, int nx,
                                  R scale, R alpha, int sms, cudaStream_t s) {
    const int hy = (ny >> lev) / 2, hx = (nx >> lev) / 2;
    cudaError_t e;
    if constexpr (sizeof(R) == 4) {
        // 16-byte pieces: a caller's image, coefficients or weights may start anywhere
        const bool al = (((uintptr_t)x | (uintptr_t)out | (uintptr_t)ds | (uintptr_t)wt) & 15) == 0;
        const int T = al ? dwt32_tile(hy, hx, b, sms) : 0;
        if (T == 32) {
            if ((e = ensure_smem(k_dwt32_level<MODE, 32>, dwt32_smem<32>()))) return e;
            k_dwt32_level<MODE, 32><<<dim3(hx / 32, hy / 32, b), dwt32_threads<32>(), dwt32_smem<32>(), s>>>(
                x, llin, llout, out, ds, wt, filt, flen, active, lev, L, ny, nx, scale, alpha);
            return cudaGetLastError();
        }
        if (T == 16) {
            if ((e = ensure_smem(k_dwt32_level<MODE, 16>, dwt32_smem<16>()))) return e;
            k_dwt32_level<MODE, 16><<<dim3(hx / 16, hy / 16, b), dwt32_threads<16>(), dwt32_smem<16>(), s>>>(
                x, llin, llout, out, ds, wt, filt, flen, active, lev, L, ny, nx, scale, alpha);
            return cudaGetLastError();
        }
    }
    if (lev == 0) {
        const int64_t n = (int64_t)ny * nx;
        const int dgrid = (int)std::min<int64_t>((n + 255) / 256, (int64_t)sms * 4);
        k_dirac<R, MODE><<<dgrid, 256, 0, s>>>(x, out, MODE == 0 ? out : ds, wt, flen, active, b, n, scale, alpha);
        if ((e = cudaGetLastError())) return e;
    }
    const int ty = std::min(AT, hy), tx = std::min(AT, hx);
    const size_t sm = ana_smem<R>(ty, tx);
    if ((e = ensure_smem(k_dwt_level<R, MODE>, sm))) return e;
    k_dwt_level<R, MODE><<<dim3((hx + tx - 1) / tx, (hy + ty - 1) / ty, b), NT_W, sm, s>>>(
        x, llin, llout, out, ds, wt, filt, flen, active, lev, L, ny, nx, scale, alpha);
    return cudaGetLastError();
}

template <int MODE, typename R>
static cudaError_t analysis_t(const pd_plan* p, const R* x, R* out, R* ds, const int32_t* active, R alpha,
                              cudaStream_t s, const R* wt) {
    const int ny = p->g.ny, nx = p->g.nx, b = p->b, L = p->L;
    const R scale = R(1.0 / std::sqrt((double)b));
    if (p->n_wavelet == 0) {
        const int64_t n = (int64_t)ny * nx;
        const int dgrid = (int)std::min<int64_t>((n + 255) / 256, (int64_t)p->num_sms * 4);
        k_dirac<R, MODE><<<dgrid, 256, 0, s>>>(x, out, MODE == 0 ? out : ds, wt, p->filt_len, active, b, n, scale, alpha);
        return cudaGetLastError();
    }
    cudaError_t e = cudaSuccess;
    for (int lev = 0; lev < L && !e; ++lev)
        e = analysis_level<MODE, R>(x, (const R*)p->ll[(lev + 1) & 1], (R*)p->ll[lev & 1], out, ds, wt,
                                    (const R*)p->filt, p->filt_len, active, b, lev, L, ny, nx, scale, alpha, p->num_sms, s);
    return e;
}

template <typename R>
static cudaError_t analysis(const pd_plan* p, const R* x, R* out, R* ds, const int32_t* active, int mode, R alpha,
                            cudaStream_t s, const R* wt = nullptr) {
    return mode == 0 ? analysis_t<0, R>(p, x, out, ds, active, alpha, s, nullptr)
                     : analysis_t<1, R>(p, x, out, ds, active, alpha, s, wt);
}

template <typename R>
static cudaError_t synthesis(const pd_plan* p, const R* coef, R* out, const int32_t* active, int mode,
                             cudaStream_t s) {
    cudaError_t e;
    const int ny = p->g.ny, nx = p->g.nx, b = p->b, L = p->L;
    const R scale = R(1.0 / std::sqrt((double)b));
    const int64_t n = (int64_t)ny * nx;
    if (p->n_wavelet > 0) {
        for (int lev = L - 1; lev >= 0; --lev) {
            const int my = ny >> lev, mx = nx >> lev;
            const int ty = std::min(ST, my), tx = std::min(ST, mx);
            dim3 grid((mx + tx - 1) / tx, (my + ty - 1) / ty, b);
            if constexpr (sizeof(R) == 4) {
                const int P = ((uintptr_t)coef & 15) == 0 ? dwt32_tile(my / 2, mx / 2, b, p->num_sms) : 0;
                float* to = lev > 0 ? (float*)p->ll[lev & 1] : (float*)p->synpart;
                const int64_t st = lev > 0 ? (int64_t)(ny / 2) * (nx / 2) : n;
                const int32_t* act = mode == 1 ? active : nullptr;
                if (P == 32) {
                    if ((e = ensure_smem(k_idwt32_level<32>, idwt32_smem<32>()))) return e;
                    k_idwt32_level<32><<<dim3(mx / 64, my / 64, b), idwt32_threads<32>(), idwt32_smem<32>(), s>>>(
                        coef, (const float*)p->ll[(lev + 1) & 1], to, (const float*)p->filt, p->filt_len, act, lev, L, ny,
                        nx, st);
                } else if (P == 16) {
                    if ((e = ensure_smem(k_idwt32_level<16>, idwt32_smem<16>()))) return e;
                    k_idwt32_level<16><<<dim3(mx / 32, my / 32, b), idwt32_threads<16>(), idwt32_smem<16>(), s>>>(
                        coef, (const float*)p->ll[(lev + 1) & 1], to, (const float*)p->filt, p->filt_len, act, lev, L, ny,
                        nx, st);
                }
                if ((e = cudaGetLastError())) return e;
                if (P) continue;
            }
            if ((e = ensure_smem(k_idwt_level<R>, syn_smem<R>(ty, tx)))) return e;
            // levels L-1 .. 1 rebuild the approximations, level 0 each basis's full image
            R* dst = lev > 0 ? (R*)p->ll[lev & 1] : (R*)p->synpart;
            const int64_t stride = lev > 0 ? (int64_t)(ny / 2) * (nx / 2) : n;
            k_idwt_level<R><<<grid, NT_W, syn_smem<R>(ty, tx), s>>>(
                coef, (const R*)p->ll[(lev + 1) & 1], dst, (const R*)p->filt, p->filt_len,
                mode == 1 ? active : nullptr, lev, L, ny, nx, stride);
            if ((e = cudaGetLastError())) return e;
        }
    }
    const int ctas = (int)std::min<int64_t>((n / 4 + 255) / 256, (int64_t)p->num_sms * 8);
    const bool vec = (((uintptr_t)coef | (uintptr_t)out) & 15) == 0;
    auto sum = [&](auto kernel) {
        kernel<<<ctas, 256, 0, s>>>(coef, (const R*)p->synpart, p->filt_len, active, b, n, out, scale);
    };
    if (mode == 0) vec ? sum(k_syn_sum<R, 0, true>) : sum(k_syn_sum<R, 0, false>);
    else vec ? sum(k_syn_sum<R, 1, true>) : sum(k_syn_sum<R, 1, false>);
    return cudaGetLastError();
}

template <typename R>
cudaError_t psi_adj_plain(const pd_plan* p, const R* x, R* coeffs, cudaStream_t s) {
    return analysis<R>(p, x, coeffs, nullptr, p->ones_basis, 0, R(0), s);
}

template <typename R>
cudaError_t psi_plain(const pd_plan* p, const R* coeffs, R* x, cudaStream_t s) {
    return synthesis<R>(p, coeffs, x, p->ones_basis, 0, s);
}

// w = delta / (delta + |w|) in place (the reweighting rule of the weighted analysis prior)
template <typename R>
__global__ void k_sara_rule(R* __restrict__ w, int64_t n, R delta) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        w[i] = delta / (delta + fabs(w[i]));
}

template <typename R>
cudaError_t sara_weights(const pd_plan* p, const R* x, double delta, R* w, cudaStream_t s) {
    cudaError_t e = psi_adj_plain<R>(p, x, w, s);
    if (e) return e;
    const int64_t n = (int64_t)p->b * p->g.ny * p->g.nx;
    const int ctas = (int)std::min<int64_t>((n + 255) / 256, (int64_t)p->num_sms * 8);
    k_sara_rule<R><<<ctas, 256, 0, s>>>(w, n, (R)delta);
    return cudaGetLastError();
}

template <typename R>
cudaError_t sparsity_dual(const pd_plan* p, const R* xt, R* s, R* st, const int32_t* basis_active, double alpha,
                          cudaStream_t str, const R* wt) {
    prof_mark(PH_ANALYSIS, 0, str);
    cudaError_t e = analysis<R>(p, xt, s, (R*)p->ds, basis_active, 1, (R)alpha, str, wt);
    prof_mark(PH_ANALYSIS, 1, str);
    if (e) return e;
    prof_mark(PH_SYNTHESIS, 0, str);
    e = synthesis<R>(p, (const R*)p->ds, st, basis_active, 1, str);
    prof_mark(PH_SYNTHESIS, 1, str);
    return e;
}

// -------------------------------------------------------------------- allocation-free analysis
// pd_apply_psi_adj_noalloc runs the same analysis kernels as pd_apply_psi_adj, but
// without a plan: its scratch lives in this file-scope device array instead of memory
// allocated with cudaMalloc. Every GPU that loads the library holds the array until
// exit; every call shares it. Layout: the db1..db8 filter tables in FP64 and FP32
// (written once per device at set-up), then the per-call region: the filter table and
// flags of the call's bases (written by a kernel from its by-value arguments, so a call
// never copies from host memory) and the two approximation buffers of the level loop.
constexpr size_t PSI_STATIC_BYTES = size_t(16) << 20;
static __device__ __align__(256) unsigned char g_psi_static[PSI_STATIC_BYTES];

static size_t align256(size_t n) { return (n + 255) & ~size_t(255); }
constexpr size_t DB_TAB_D = 9 * MAX_FILTER * sizeof(double);   // [9][16], row 0 (Dirac) all zero
constexpr size_t DB_TAB_F = 9 * MAX_FILTER * sizeof(float);
static size_t psi_static_fixed() { return align256(DB_TAB_D) + align256(DB_TAB_F); }

static std::mutex g_psi_static_mu;
static void* g_psi_static_addr[64];       // device address of g_psi_static, per device
static int g_psi_static_sms[64];

// One-time set-up for device `dev` (current): the device address of the static array
// (host code may not use the symbol itself as a pointer), the SM count, and the
// Daubechies tables, written with a synchronous copy before the first call's kernels.
static pd_status psi_static_setup(int dev, void** addr, int* sms) {
    std::lock_guard<std::mutex> lock(g_psi_static_mu);
    if (dev < 0 || dev >= 64) return set_error(PD_ENOTSUP, "pd_apply_psi_adj_noalloc: device index above 63");
    if (!g_psi_static_addr[dev]) {
        void* ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_psi_static);
        if (e != cudaSuccess || ptr == nullptr)
            return set_error(PD_ECUDA, "pd_apply_psi_adj_noalloc: cudaGetSymbolAddress of the static scratch failed");
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return set_error(PD_ECUDA, "pd_apply_psi_adj_noalloc: cannot query the SM count");
        std::vector<unsigned char> tab(psi_static_fixed(), 0);
        double* td = (double*)tab.data();
        float* tf = (float*)(tab.data() + align256(DB_TAB_D));
        for (int k = 1; k <= 8; ++k) {
            const std::vector<double> h = daubechies(k);
            for (size_t j = 0; j < h.size(); ++j) { td[k * MAX_FILTER + j] = h[j]; tf[k * MAX_FILTER + j] = (float)h[j]; }
        }
        if (cudaMemcpy(ptr, tab.data(), tab.size(), cudaMemcpyHostToDevice) != cudaSuccess)
            return set_error(PD_ECUDA, "pd_apply_psi_adj_noalloc: writing the filter tables failed");
        g_psi_static_addr[dev] = ptr;
        g_psi_static_sms[dev] = n;
    }
    *addr = g_psi_static_addr[dev];
    *sms = g_psi_static_sms[dev];
    return PD_OK;
}

// The call's bases, passed by value as a kernel argument.
struct BasisList {
    int32_t id[MAX_BASES];
    int32_t b;
};

// Per-call filter table [b][MAX_FILTER], filter lengths and all-active flags of the
// call's bases, from the static db tables.
template <typename R>
__global__ void k_psi_call_tables(BasisList bl, const R* __restrict__ db, R* __restrict__ filt,
                                  int32_t* __restrict__ flen, int32_t* __restrict__ ones) {
    const int i = threadIdx.x;
    if (i >= bl.b * MAX_FILTER) return;
    const int k = i / MAX_FILTER, j = i - k * MAX_FILTER;
    const int id = bl.id[k];
    filt[i] = db[id * MAX_FILTER + j];
    if (j == 0) {
        flen[k] = id == 0 ? 0 : 2 * id;
        ones[k] = 1;
    }
}

template <typename R>
static pd_status psi_adj_static_t(const R* x, R* coeffs, int nx, int ny, int L, const int32_t* ids, int b,
                                  unsigned char* scratch, int sms, cudaStream_t s) {
    const R* db = (const R*)(scratch + (sizeof(R) == 8 ? 0 : align256(DB_TAB_D)));
    unsigned char* call = scratch + psi_static_fixed();
    const size_t filt_bytes = align256((size_t)b * MAX_FILTER * sizeof(R));
    const size_t flag_bytes = align256((size_t)b * sizeof(int32_t));
    const size_t ll_bytes = align256((size_t)b * (ny / 2) * (nx / 2) * sizeof(R));
    R* filt = (R*)call;
    int32_t* flen = (int32_t*)(call + filt_bytes);
    int32_t* ones = (int32_t*)(call + filt_bytes + flag_bytes);
    R* ll[2] = {(R*)(call + filt_bytes + 2 * flag_bytes), (R*)(call + filt_bytes + 2 * flag_bytes + ll_bytes)};
    BasisList bl{};
    bl.b = b;
    int nwav = 0;
    for (int k = 0; k < b; ++k) {
        bl.id[k] = ids[k];
        nwav += ids[k] > 0;
    }
    cudaError_t e;
    k_psi_call_tables<R><<<1, MAX_BASES * MAX_FILTER, 0, s>>>(bl, db, filt, flen, ones);
    if ((e = cudaGetLastError())) return set_error(PD_ECUDA, cudaGetErrorString(e));
    const R scale = R(1.0 / std::sqrt((double)b));
    if (nwav == 0) {
        const int64_t n = (int64_t)ny * nx;
        const int dgrid = (int)std::min<int64_t>((n + 255) / 256, (int64_t)sms * 4);
        k_dirac<R, 0><<<dgrid, 256, 0, s>>>(x, coeffs, coeffs, nullptr, flen, ones, b, n, scale, R(0));
        if ((e = cudaGetLastError())) return set_error(PD_ECUDA, cudaGetErrorString(e));
        return PD_OK;
    }
    for (int lev = 0; lev < L; ++lev)
        if ((e = analysis_level<0, R>(x, ll[(lev + 1) & 1], ll[lev & 1], coeffs, nullptr, nullptr, filt, flen, ones, b, lev,
                                      L, ny, nx, scale, R(0), sms, s)))
            return set_error(PD_ECUDA, cudaGetErrorString(e));
    return PD_OK;
}

}  // namespace pdgb

extern "C" pd_status pd_apply_psi_adj_noalloc(const void* x, void* coeffs, int32_t nx, int32_t ny, int32_t levels,
                                              const int32_t* basis_ids, int32_t nbases, int32_t precision,
                                              void* stream) {
    using namespace pdgb;
    auto pow2 = [](int v) { return v > 0 && (v & (v - 1)) == 0; };
    if (!x || !coeffs || !basis_ids) return set_error(PD_EINVAL, "pd_apply_psi_adj_noalloc: null pointer");
    if (!pow2(nx) || !pow2(ny) || nx < 16 || ny < 16 || nx > 8192 || ny > 8192)
        return set_error(PD_EINVAL, "pd_apply_psi_adj_noalloc: image sides must be powers of two in [16, 8192]");
    // bounded before the shift test (a shift by 32 or more is undefined)
    if (levels < 1 || levels > 13 || (nx >> levels) < 1 || (ny >> levels) < 1)
        return set_error(PD_EINVAL, "pd_apply_psi_adj_noalloc: levels must satisfy 1 <= L <= 13 and n >> L >= 1");
    if (nbases < 1 || nbases > MAX_BASES) return set_error(PD_EINVAL, "pd_apply_psi_adj_noalloc: nbases in [1, 16]");
    for (int k = 0; k < nbases; ++k)
        if (basis_ids[k] < 0 || basis_ids[k] > 8)
            return set_error(PD_EINVAL, "pd_apply_psi_adj_noalloc: basis ids must be 0 (Dirac) or 1..8");
    if (precision != PD_F32 && precision != PD_F64)
        return set_error(PD_EINVAL, "pd_apply_psi_adj_noalloc: precision must be PD_F32 or PD_F64");
    const size_t rsz = precision == PD_F64 ? 8 : 4;
    const size_t need = psi_static_fixed() + align256((size_t)nbases * MAX_FILTER * rsz) +
                        2 * align256((size_t)nbases * 4) + 2 * align256((size_t)nbases * (ny / 2) * (nx / 2) * rsz);
    if (need > PSI_STATIC_BYTES) {
        static thread_local char msg[160];
        snprintf(msg, sizeof msg,
                 "pd_apply_psi_adj_noalloc: needs %zu bytes of scratch, the static array holds %zu "
                 "(use pd_apply_psi_adj with a plan)", need, PSI_STATIC_BYTES);
        return set_error(PD_EINVAL, msg);
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return set_error(PD_ECUDA, "pd_apply_psi_adj_noalloc: no current device");
    cudaStream_t s = (cudaStream_t)stream;
    // the array's address is per device: the stream must belong to the current device
    if (s != nullptr) {
        int sdev = -1;
        if (cudaStreamGetDevice(s, &sdev) != cudaSuccess)
            return set_error(PD_EINVAL, "pd_apply_psi_adj_noalloc: cannot query the stream's device");
        if (sdev != dev)
            return set_error(PD_EINVAL, "pd_apply_psi_adj_noalloc: the stream belongs to another device than the current one");
    }
    void* addr = nullptr;
    int sms = 0;
    pd_status st = psi_static_setup(dev, &addr, &sms);
    if (st != PD_OK) return st;
    return precision == PD_F64
               ? psi_adj_static_t<double>((const double*)x, (double*)coeffs, nx, ny, levels, basis_ids, nbases,
                                          (unsigned char*)addr, sms, s)
               : psi_adj_static_t<float>((const float*)x, (float*)coeffs, nx, ny, levels, basis_ids, nbases,
                                         (unsigned char*)addr, sms, s);
}

namespace pdgb {

template cudaError_t psi_adj_plain<float>(const pd_plan*, const float*, float*, cudaStream_t);
template cudaError_t psi_adj_plain<double>(const pd_plan*, const double*, double*, cudaStream_t);
template cudaError_t psi_plain<float>(const pd_plan*, const float*, float*, cudaStream_t);
template cudaError_t psi_plain<double>(const pd_plan*, const double*, double*, cudaStream_t);
template cudaError_t sparsity_dual<float>(const pd_plan*, const float*, float*, float*, const int32_t*, double,
                                          cudaStream_t, const float*);
template cudaError_t sparsity_dual<double>(const pd_plan*, const double*, double*, double*, const int32_t*, double,
                                           cudaStream_t, const double*);
template cudaError_t sara_weights<float>(const pd_plan*, const float*, double, float*, cudaStream_t);
template cudaError_t sara_weights<double>(const pd_plan*, const double*, double, double*, cudaStream_t);

}  // namespace pdgb
