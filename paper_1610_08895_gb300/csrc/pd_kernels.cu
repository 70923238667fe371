// Small device-resident steps of Algorithm 1: the active-set draws (step 3) with
// the optional adaptive probabilities (Sec. 4, eq. prob-choice), the compaction of
// the active work lists for the persistent degridding/gridding launches, FP64
// reductions, and index permutations between user and internal visibility order.
#include <algorithm>

#include "common.cuh"
#include "plan.hpp"

namespace pdgb {

constexpr int SEL_NT = 1024;

// Tile t of the heaviest-first list: on if a block with points in it is active; its flag for
// the degridding and gridding launches, the parts that the gridding has to add for it, and
// the numbers of active segments and tiles.
__device__ __forceinline__ void flag_tile(int t, const int4* __restrict__ tile_info, const int32_t* __restrict__ seg_block,
                                          const int32_t* block_active, int32_t* __restrict__ tile_on,
                                          int32_t* __restrict__ pend, int& segs, int& tiles) {
    const int4 ti = tile_info[t];
    int n = 0;
    for (int k = 0; k < ti.y; ++k) n += block_active[seg_block[ti.x + k]];
    tile_on[t] = n > 0;
    pend[t] = n > 0 ? ti.z : 0;
    segs += n;
    tiles += n > 0;
}

// next_item: the gridding's work counter, set to the first item here.
// Step 3: Philox draws u(seed, t, stream, index) < p for blocks (stream 0) and
// bases (stream 1); with adaptive = 1 the block probabilities are first set by
// eq. (prob-choice) from the current residual norms. Then the tiles holding a
// visibility of an active block are flagged (here for up to SEL_TILES tiles, one or two a
// thread; more of them in k_flag_tiles, where every SM takes part).
constexpr int SEL_TILES = 2 * SEL_NT;
constexpr int SEL_D = 4096 / SEL_NT;      // blocks per thread at most
__global__ void __launch_bounds__(SEL_NT) k_select(
    uint64_t seed, int adaptive, double an, double pmin, double pmax, int64_t* __restrict__ tptr,
    double* __restrict__ p_block, const double* __restrict__ p_basis, const double* __restrict__ res_norm,
    const double* __restrict__ eps, int d, int b, int32_t* __restrict__ block_active,
    int32_t* __restrict__ basis_active, const int32_t* __restrict__ tile_order, const int4* __restrict__ tile_info,
    const int32_t* __restrict__ seg_block, int ntiles, int32_t* __restrict__ tile_on, int32_t* __restrict__ pend,
    int32_t* __restrict__ next_item, int32_t* __restrict__ counts) {
    __shared__ double shd[32];
    __shared__ int64_t t_sh;
    __shared__ int cnt_sh[2];
    const int tid = threadIdx.x;
    if (tid == 0) {
        const int64_t t = *tptr + 1;
        *tptr = t;
        t_sh = t;
        cnt_sh[0] = cnt_sh[1] = 0;
        *next_item = 0;
    }
    __syncthreads();
    if (adaptive) {
        // c_i = max(||r_i|| - eps_i, 0)^2 / eps_i^2; p_i = p_min + min(q_i + a, p_max - p_min)
        double c[SEL_D], csum = 0.0;
#pragma unroll
        for (int u = 0; u < SEL_D; ++u) {
            const int i = tid + u * SEL_NT;
            c[u] = 0.0;
            if (i < d) {
                const double e = eps[i], r = res_norm[i];
                c[u] = r > e ? (r - e) * (r - e) / (e * e) : 0.0;
            }
            csum += c[u];
        }
        auto all_sum = [&](double v) {
            v = block_sum(v, shd);
            if (tid == 0) shd[0] = v;
            __syncthreads();
            v = shd[0];
            __syncthreads();
            return v;
        };
        csum = all_sum(csum);
        const double cap = pmax - pmin, target = an - d * pmin;
        if (csum == 0.0) {
            for (int i = tid; i < d; i += SEL_NT) p_block[i] = an / d;
        } else {
            const double qs = target / csum;
            // a = 0 unless some q_i exceeds the cap (then some p_i saturates at p_max). f(a) =
            // sum min(q_i + a, cap) is concave, so Newton's steps from 0 stay left of the root and
            // each one passes a breakpoint or lands on it: a handful of steps instead of a bisection
            // to double precision (80 steps of one block-wide sum each)
            double a = 0.0;
            int sat = 0;
#pragma unroll
            for (int u = 0; u < SEL_D; ++u) sat |= qs * c[u] > cap;
            sat = __syncthreads_or(sat);
            for (int it = 0; sat && it <= d; ++it) {
                double f = 0.0, fr = 0.0;
#pragma unroll
                for (int u = 0; u < SEL_D; ++u) {
                    if (tid + u * SEL_NT >= d) break;
                    const double q = qs * c[u] + a;
                    f += fmin(q, cap);
                    fr += q < cap ? 1.0 : 0.0;
                }
                f = all_sum(f);
                fr = all_sum(fr);
                const double next = fr > 0.0 ? a + (target - f) / fr : a;
                if (!(next > a)) break;
                a = next;
            }
#pragma unroll
            for (int u = 0; u < SEL_D; ++u)
                if (tid + u * SEL_NT < d) p_block[tid + u * SEL_NT] = pmin + fmin(qs * c[u] + a, cap);
        }
    }
    __syncthreads();
    const int64_t t = t_sh;
    for (int i = tid; i < d; i += SEL_NT) block_active[i] = philox_uniform(seed, (uint64_t)t, 0, i) < p_block[i];
    for (int j = tid; j < b; j += SEL_NT) basis_active[j] = philox_uniform(seed, (uint64_t)t, 1, j) < p_basis[j];
    if (ntiles > SEL_TILES) {
        if (tid < 2) counts[tid] = 0;
        return;
    }
    __syncthreads();
    int segs = 0, tiles = 0;
    for (int k = tid; k < ntiles; k += SEL_NT)
        flag_tile(tile_order[k], tile_info, seg_block, block_active, tile_on, pend, segs, tiles);
    if (segs) { atomicAdd(&cnt_sh[0], segs); atomicAdd(&cnt_sh[1], tiles); }
    __syncthreads();
    if (tid < 2) counts[tid] = cnt_sh[tid];
}

__global__ void __launch_bounds__(256) k_flag_tiles(const int32_t* __restrict__ tile_order,
                                                    const int4* __restrict__ tile_info,
                                                    const int32_t* __restrict__ seg_block,
                                                    const int32_t* __restrict__ block_active, int ntiles,
                                                    int32_t* __restrict__ tile_on, int32_t* __restrict__ pend,
                                                    int32_t* __restrict__ counts) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    int segs = 0, tiles = 0;
    if (k < ntiles) flag_tile(tile_order[k], tile_info, seg_block, block_active, tile_on, pend, segs, tiles);
    segs = __reduce_add_sync(0xffffffffu, segs);
    tiles = __reduce_add_sync(0xffffffffu, tiles);
    if ((threadIdx.x & 31) == 0 && segs) { atomicAdd(counts, segs); atomicAdd(counts + 1, tiles); }
}

cudaError_t select_active(const pd_plan* p, pd_state* st, const SelectArgs& a, cudaStream_t s) {
    prof_mark(PH_SELECT, 0, s);
    const int nt = p->ntiles_nonempty;
    k_select<<<1, SEL_NT, 0, s>>>(a.seed, a.adaptive, a.n, a.p_min, a.p_max, st->t, st->p_block, st->p_basis,
                                 st->res_norm, st->eps, p->d, p->b, st->block_active, st->basis_active,
                                 p->tile_order, p->tile_info, p->seg_block, nt, st->tile_active, p->pend, p->sched + 8,
                                 st->counts);
    if (nt > SEL_TILES)
        k_flag_tiles<<<(nt + 255) / 256, 256, 0, s>>>(p->tile_order, p->tile_info, p->seg_block, st->block_active, nt,
                                                      st->tile_active, p->pend, st->counts);
    prof_mark(PH_SELECT, 1, s);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_grid_begin(const int4* __restrict__ tile_info, const int32_t* __restrict__ seg_block,
                                                    const int32_t* __restrict__ active, int ntiles,
                                                    int32_t* __restrict__ pend, int32_t* __restrict__ next_item,
                                                    float4* __restrict__ U, int64_t n4, int batch) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *next_item = 0;
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = i0; i < (int64_t)ntiles * batch; i += step) {
        const int4 ti = tile_info[i % ntiles];
        int on = active == nullptr && ti.y > 0;
        if (active)
            for (int k = 0; k < ti.y; ++k) on |= active[seg_block[ti.x + k]];
        pend[i] = on ? ti.z : 0;
    }
    for (int64_t i = i0; i < n4; i += step) U[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}
cudaError_t grid_begin(const pd_plan* p, const int32_t* active, int32_t* pend, float4* U, int64_t n4, int batch,
                       cudaStream_t s) {
    const int64_t n = std::max<int64_t>((int64_t)p->g.ntiles * batch, U ? n4 / 4 : 0);
    const int ctas = (int)std::min<int64_t>((n + 255) / 256, (int64_t)p->num_sms * 8);
    k_grid_begin<<<ctas, 256, 0, s>>>(p->tile_info, p->seg_block, active, p->g.ntiles, pend, p->sched + 8, U,
                                       U ? n4 : 0, batch);
    return cudaGetLastError();
}

// Fixed-order sum of per-CTA partials of the primal update: ||x^t - x^{t-1}||^2, ||x^t||^2.
__global__ void k_sum_pairs(const double* __restrict__ part, int n, double* __restrict__ out) {
    __shared__ double sh[32];
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) { a += part[2 * i]; b += part[2 * i + 1]; }
    a = block_sum(a, sh);
    b = block_sum(b, sh);
    if (threadIdx.x == 0) { out[0] = a; out[1] = b; }
}

cudaError_t primal_finish(const pd_plan* p, pd_state* st, cudaStream_t s) {
    prof_mark(PH_FINISH, 0, s);
    k_sum_pairs<<<1, 256, 0, s>>>(st->prim_part, inv_rows_ctas(p), st->diag);
    prof_mark(PH_FINISH, 1, s);
    return cudaGetLastError();
}

// Deterministic two-level FP64 sum of squares.
template <typename R>
__global__ void k_sq_part(const R* __restrict__ x, int64_t n, double* __restrict__ part) {
    __shared__ double sh[32];
    double a = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        a += (double)x[i] * (double)x[i];
    a = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = a;
}
__global__ void k_sum(const double* __restrict__ part, int n, double* __restrict__ out) {
    __shared__ double sh[32];
    double a = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) a += part[i];
    a = block_sum(a, sh);
    if (threadIdx.x == 0) *out = a;
}

template <typename R>
cudaError_t norm2(const pd_plan* p, const R* x, int64_t n, double* out, cudaStream_t s) {
    const int ctas = std::min<int64_t>(p->red_len, std::max<int64_t>(1, (n + 255) / 256));
    k_sq_part<R><<<ctas, 256, 0, s>>>(x, n, p->red);
    k_sum<<<1, 256, 0, s>>>(p->red, ctas, out);
    return cudaGetLastError();
}

template <typename R>
__global__ void k_scale_copy(const R* __restrict__ x, R* __restrict__ y, int64_t n, R scale) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = x[i] * scale;
}
template <typename R>
cudaError_t scale_copy(const R* x, R* y, int64_t n, double scale, cudaStream_t s) {
    const int ctas = (int)std::min<int64_t>(4096, (n + 255) / 256);
    k_scale_copy<R><<<ctas, 256, 0, s>>>(x, y, n, (R)scale);
    return cudaGetLastError();
}

template <typename C>
__global__ void k_gather(const C* __restrict__ user, C* __restrict__ internal, const int32_t* __restrict__ perm,
                         int64_t m) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        internal[i] = vis_conj(perm[i], user[vis_index(perm[i])]);
}
template <typename C>
__global__ void k_scatter(const C* __restrict__ internal, C* __restrict__ user, const int32_t* __restrict__ perm,
                          int64_t m) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        user[vis_index(perm[i])] = vis_conj(perm[i], internal[i]);
}
template <typename R>
cudaError_t gather_by(int64_t m, const int32_t* perm, const cplx_t<R>* src, cplx_t<R>* dst, cudaStream_t s) {
    const int ctas = (int)std::min<int64_t>(4096, (m + 255) / 256);
    k_gather<<<ctas, 256, 0, s>>>(src, dst, perm, m);
    return cudaGetLastError();
}
template <typename R>
cudaError_t scatter_by(int64_t m, const int32_t* perm, const cplx_t<R>* src, cplx_t<R>* dst, cudaStream_t s) {
    const int ctas = (int)std::min<int64_t>(4096, (m + 255) / 256);
    k_scatter<<<ctas, 256, 0, s>>>(src, dst, perm, m);
    return cudaGetLastError();
}
// The visibilities that are held as their conjugates (held = 1) or the others, in user order and
// convention, zeros in the place of the rest.
template <typename C>
__global__ void k_scatter_side(const C* __restrict__ internal, C* __restrict__ user, const int32_t* __restrict__ perm,
                               int64_t m, int held) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        C v = vis_conj(perm[i], internal[i]);
        if ((perm[i] < 0) != (held != 0)) v.x = v.y = 0;
        user[vis_index(perm[i])] = v;
    }
}
// U[k] += conj W[-k] over the whole grid.
template <typename C>
__global__ void k_add_mirrored(C* __restrict__ U, const C* __restrict__ W, int Ky, int Kx) {
    const int64_t n = (int64_t)Ky * Kx;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int ky = (int)(i / PW % Ky), kx = (int)(i / PW / Ky) * PW + (int)(i % PW);
        const C w = W[panel_off((Ky - ky) & (Ky - 1), (Kx - kx) & (Kx - 1), Ky)];
        C u = U[i];
        u.x += w.x;
        u.y -= w.y;
        U[i] = u;
    }
}
template <typename R>
cudaError_t unfolded_u(const pd_plan* p, const pd_state* st, cplx_t<R>* out, cudaStream_t s) {
    cplx_t<R>* user = (cplx_t<R>*)p->rbuf;
    cplx_t<R>* grid[2] = {out, (cplx_t<R>*)p->gridu};
    const int ctas = (int)std::min<int64_t>(4096, (p->M + 255) / 256);
    cudaError_t e;
    for (int held = 0; held < 2; ++held) {
        k_scatter_side<<<ctas, 256, 0, s>>>((const cplx_t<R>*)st->v, user, p->perm, p->M, held);
        if ((e = cudaGetLastError()) || (e = grid_plain<R>(p, user, grid[held], s, 1, nullptr, st->status))) return e;
    }
    k_add_mirrored<<<p->num_sms * 8, 256, 0, s>>>(out, (const cplx_t<R>*)grid[1], p->g.Ky, p->g.Kx);
    return cudaGetLastError();
}
template <typename R>
cudaError_t gather_internal(const pd_plan* p, const cplx_t<R>* user, cplx_t<R>* internal, cudaStream_t s) {
    return gather_by<R>(p->M, p->perm, user, internal, s);
}
template <typename R>
cudaError_t scatter_user(const pd_plan* p, const cplx_t<R>* internal, cplx_t<R>* user, cudaStream_t s) {
    return scatter_by<R>(p->M, p->perm, internal, user, s);
}

// ||y_i|| per block (= ||Phi_i x^(0) - y_i|| for x^(0) = 0): partial sums of every slot, one
// warp each, then a fixed-order sum per block, one warp each.
template <typename R>
__global__ void __launch_bounds__(256) k_slot_sq(const cplx_t<R>* __restrict__ y, const SegSlot* __restrict__ range,
                                                 int64_t nslot, double* __restrict__ part) {
    const int lane = threadIdx.x & 31;
    const int64_t step = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t k = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); k < nslot; k += step) {
        const SegSlot r = range[k];
        double a = 0.0;
        for (int m0 = r.start + lane; m0 < r.end; m0 += 4 * 32) {
            cplx_t<R> v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = m0 + 32 * u < r.end ? y[m0 + 32 * u] : mk<cplx_t<R>>(R(0), R(0));
#pragma unroll
            for (int u = 0; u < 4; ++u) a += (double)v[u].x * v[u].x + (double)v[u].y * v[u].y;
        }
        a = warp_sum(a);
        if (lane == 0) part[2 * k + 1] = a;
    }
}
__global__ void __launch_bounds__(128) k_block_sqrt(const double* __restrict__ part, const int32_t* __restrict__ bss,
                                                    const int32_t* __restrict__ bsl, int d, double* __restrict__ out) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= d) return;
    double a = 0.0;
    for (int k = bss[i] + lane; k < bss[i + 1]; k += 32) a += part[2 * (int64_t)bsl[k] + 1];
    a = warp_sum(a);
    if (lane == 0) out[i] = sqrt(a);
}
cudaError_t init_res_norm(const pd_plan* p, pd_state* st, cudaStream_t s) {
    const int ctas = (int)std::min<int64_t>((p->nslot + 7) / 8, (int64_t)p->num_sms * 16);
    if (p->prec == PD_F64)
        k_slot_sq<double><<<ctas, 256, 0, s>>>((const double2*)st->y, p->slot_range, p->nslot, p->seg_part);
    else
        k_slot_sq<float><<<ctas, 256, 0, s>>>((const float2*)st->y, p->slot_range, p->nslot, p->seg_part);
    k_block_sqrt<<<(p->d * 32 + 127) / 128, 128, 0, s>>>(p->seg_part, p->block_slot_start, p->block_slot_list, p->d,
                                                         st->res_norm);
    return cudaGetLastError();
}

// Synthesis form, dual of positivity and the image-domain term of the primal step:
// u <- min(u + x~, 0) (z - P_C(z)); back <- sigma u + varsigma back.
template <typename R>
__global__ void k_synth_dual(const R* __restrict__ xt, R* __restrict__ u, R* __restrict__ back, int64_t n, R sigma,
                             R varsigma) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const R z = u[i] + xt[i];
        const R un = z < R(0) ? z : R(0);
        u[i] = un;
        back[i] = sigma * un + varsigma * back[i];
    }
}

// Synthesis form, primal step on the coefficients: alpha_new = S_thr(alpha - tau w)
// (eq. prox-L1), alpha~ = 2 alpha_new - alpha, alpha = alpha_new.
template <typename R>
__global__ void k_synth_primal(R* __restrict__ alpha, R* __restrict__ alpha_t, const R* __restrict__ w, int64_t n,
                               R tau, R thr) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const R a = alpha[i];
        const R q = a - tau * w[i];
        const R an = q > thr ? q - thr : (q < -thr ? q + thr : R(0));
        alpha_t[i] = R(2) * an - a;
        alpha[i] = an;
    }
}

template <typename R>
cudaError_t synth_dual(const pd_plan* p, const R* xt, R* u, R* back, double sigma, double varsigma, cudaStream_t s) {
    const int64_t n = (int64_t)p->g.nx * p->g.ny;
    const int ctas = (int)std::min<int64_t>((n + 255) / 256, (int64_t)p->num_sms * 8);
    k_synth_dual<R><<<ctas, 256, 0, s>>>(xt, u, back, n, (R)sigma, (R)varsigma);
    return cudaGetLastError();
}

template <typename R>
cudaError_t synth_primal(const pd_plan* p, R* alpha, R* alpha_t, const R* w, double tau, double thr, cudaStream_t s) {
    const int64_t n = (int64_t)p->b * p->g.nx * p->g.ny;
    const int ctas = (int)std::min<int64_t>((n + 255) / 256, (int64_t)p->num_sms * 8);
    k_synth_primal<R><<<ctas, 256, 0, s>>>(alpha, alpha_t, w, n, (R)tau, (R)thr);
    return cudaGetLastError();
}

template cudaError_t synth_dual<float>(const pd_plan*, const float*, float*, float*, double, double, cudaStream_t);
template cudaError_t synth_dual<double>(const pd_plan*, const double*, double*, double*, double, double, cudaStream_t);
template cudaError_t synth_primal<float>(const pd_plan*, float*, float*, const float*, double, double, cudaStream_t);
template cudaError_t synth_primal<double>(const pd_plan*, double*, double*, const double*, double, double,
                                          cudaStream_t);
template cudaError_t norm2<float>(const pd_plan*, const float*, int64_t, double*, cudaStream_t);
template cudaError_t norm2<double>(const pd_plan*, const double*, int64_t, double*, cudaStream_t);
template cudaError_t scale_copy<float>(const float*, float*, int64_t, double, cudaStream_t);
template cudaError_t scale_copy<double>(const double*, double*, int64_t, double, cudaStream_t);
template cudaError_t gather_by<float>(int64_t, const int32_t*, const float2*, float2*, cudaStream_t);
template cudaError_t gather_by<double>(int64_t, const int32_t*, const double2*, double2*, cudaStream_t);
template cudaError_t scatter_by<float>(int64_t, const int32_t*, const float2*, float2*, cudaStream_t);
template cudaError_t scatter_by<double>(int64_t, const int32_t*, const double2*, double2*, cudaStream_t);
template cudaError_t unfolded_u<float>(const pd_plan*, const pd_state*, float2*, cudaStream_t);
template cudaError_t unfolded_u<double>(const pd_plan*, const pd_state*, double2*, cudaStream_t);
template cudaError_t gather_internal<float>(const pd_plan*, const float2*, float2*, cudaStream_t);
template cudaError_t gather_internal<double>(const pd_plan*, const double2*, double2*, cudaStream_t);
template cudaError_t scatter_user<float>(const pd_plan*, const float2*, float2*, cudaStream_t);
template cudaError_t scatter_user<double>(const pd_plan*, const double2*, double2*, cudaStream_t);

}  // namespace pdgb
