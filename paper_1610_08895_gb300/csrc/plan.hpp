// Internal plan/state layout of the PD-R CUDA library and the launcher interfaces
// between the host API (api.cu) and the kernel translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <string>
#include <vector>

#include "common.cuh"
#include "pd.h"

namespace pdgb {

constexpr int PW = 4;          // panel width (complex elements) of the column-panel grid layout
constexpr int MAX_FILTER = 16; // longest Daubechies filter (db8)
constexpr int MAX_BASES = 16;

// Device-side view of the plan, passed by value to kernels.
struct Geo {
    int nx, ny, Kx, Ky;
    int J;
    double beta;
    int tile, logT, ntx, nty, ntiles;
    int ext;        // T + J - 1: extended tile edge of the gridding accumulator
};

// Tile colour classes of the gridding: (tile row parity, tile column parity). Two tiles
// of one colour are at least two tiles apart, so for J - 1 <= T their windows (tile plus
// halo) are disjoint and one launch may update them in U without atomics. The grid has
// at least two tiles per side (an even number), so the four classes are equal in size.
__host__ __device__ __forceinline__ int tile_colour(int t, int ntx) { return (((t / ntx) & 1) << 1) | ((t % ntx) & 1); }

// Monomial coefficients (in x = 2 f - 1) of the per-tap Chebyshev interpolants of the
// Kaiser-Bessel weight phi(f + J/2 - 1 - a), used by the FP32 kernels.
constexpr int KB_DEG = 10;
// lo: what the constant terms' rounding to FP32 left.
struct KbPoly {
    float c[16][KB_DEG + 1];
    float lo[16];
};
// The same for the FP64 kernels; use = 0 where the fit is not exact to FP64 (a caller's own,
// larger kb_beta): those plans evaluate I0 itself.
constexpr int KB_DEG64 = 18;
// The outermost taps (kb_outer of them on either side) by a polynomial in s = 1 - (2 t / J)^2.
constexpr int KB_EDGE_MAX = 31;
__host__ __device__ constexpr int kb_outer(int J) { return J > 8 ? 2 : 1; }
__host__ __device__ constexpr int kb_edge_deg(int J) {
    return J > 8 ? KB_EDGE_MAX : J == 8 ? 19 : J == 6 ? 17 : J == 4 ? 15 : 11;
}
struct KbPoly64 {
    double c[8][KB_DEG64 + 1];
    double e[KB_EDGE_MAX + 1];
    int use;
};
template <typename R> struct KbPolyOf { using type = KbPoly; };
template <> struct KbPolyOf<double> { using type = KbPoly64; };
template <typename R> using kb_poly_t = typename KbPolyOf<R>::type;

// One degridding work item: a part of a tile's points. slot0: where the part's per-segment
// sums go in seg_part (one pair for each of the tile's segments).
struct TileItem {
    int32_t tile, part, parts, slot0;
    int32_t seg0, nseg, pad0, pad1;
};
// A slot of seg_part: the part's share of one segment's points.
struct SegSlot {
    int32_t start, end;
};

// Super-cells of SC x SC cells inside a tile: the visibilities of a segment are sorted by
// the super-cell of their footprint's first cell, then row-major by that cell.
constexpr int SC = 8;

// The image is real, so the visibility at -(u, v) is the conjugate of the one at (u, v):
// points with u < 0 are held at -(u, v) as conjugates (unless G is stored, or the point is
// on a grid line), which leaves norms, duals and Re(Phi^H .) as they are and halves the tiles that hold points. perm
// carries the flag in its sign bit; these read and write a value in the user's convention.
__host__ __device__ __forceinline__ int vis_index(int q) { return q & 0x7fffffff; }
template <typename C> __device__ __forceinline__ C vis_conj(int q, C v) {
    if (q < 0) v.y = -v.y;
    return v;
}

// Element offset of grid cell (ky, kx) in the column-panel layout [Kx/PW][K][PW].
__host__ __device__ __forceinline__ int64_t panel_off(int ky, int kx, int K) {
    return ((int64_t)(kx >> 2) * K + ky) * PW + (kx & 3);
}

}  // namespace pdgb

struct pd_plan {
    int prec;                  // PD_F32 / PD_F64
    size_t rsz, csz;           // sizeof real / complex
    pdgb::Geo g;
    int64_t M;
    int d, b, L;
    std::vector<int> basis_ids;
    int n_wavelet;             // bases with id > 0
    int64_t nseg;
    int ntiles_nonempty;
    int num_sms;
    int max_smem;              // opt-in shared memory per CTA (bytes)
    int device;

    // host copies of the static tables
    std::vector<int32_t> h_tile_seg_start, h_seg_block;

    // checkpoints keep the visibilities in the order of their base cells in tiles of ck_tile cells,
    // whatever the plan's internal order is: list of the internal index of each (sign bit: held as a
    // conjugate), made by the first save or load under the lock and only read after that; on the
    // device (outside of allocs, which only calls that are ordered on the plan may touch), or on the
    // host if there was no room
    int ck_tile = 0;
    std::mutex ck_mu;
    bool ck_ready = false;
    int32_t* ck_list = nullptr;
    std::vector<int32_t> ck_order;
    bool folded = false;           // some visibility is held as its conjugate

    // device: visibilities in internal (tile, block, row, column) order
    int32_t* cell = nullptr;       // (by << 16) | bx of the footprint's first cell, mod K
    void* fx = nullptr;            // real [M]: fractional part of g_x
    void* fy = nullptr;
    int32_t* perm = nullptr;       // internal -> user index; sign bit set: held as its conjugate (see vis_conj)
    int g_mode = PD_G_ON_THE_FLY;  // PD_G_CSR: G stored explicitly, below
    int kb_J = 0;                  // interpolation kernel width (g.J is the footprint: kb_J + dde - 1)
    int dde = 0;                   // DDE kernel width d (0: none)
    bool csr_cplx = false;         // CSR entries complex (DDE-aware G)
    std::vector<double> h_dde;     // DDE kernels, internal order (kept until G is built)
    int32_t* csr_col = nullptr;    // [J^2][M] grid cell (ky << 16 | kx) of each entry, internal order
    void* csr_val = nullptr;       // real [J^2][M] weight of each entry
    int32_t* seg_start = nullptr;  // [nseg + 1]
    int32_t* seg_block = nullptr;  // [nseg]
    int32_t* tile_seg_start = nullptr;  // [ntiles + 1]
    int nsc_side = 0;                      // super-cells per tile side (tile / SC)
    int32_t* seg_sc_start = nullptr;       // [nseg][nsc_side^2 + 1] super-cell starts inside each segment
    std::vector<int32_t> h_sc_start;       // (host, only during plan construction)
    int max_tile_segs = 0;                 // most (tile, block) segments in one tile
    pdgb::KbPoly kbpoly{};
    pdgb::KbPoly64 kbpoly64{};
    int32_t* block_slot_start = nullptr;   // [d + 1] into block_slot_list
    int32_t* block_slot_list = nullptr;    // [nslot] seg_part slots of each block, in a fixed order
    int32_t* tile_order = nullptr;         // [ntiles] tiles by decreasing visibility count
    int32_t* colour_tiles = nullptr;       // [4][ntiles/4] tiles of each colour, heaviest first
    int32_t* colour_counts = nullptr;      // [4] tiles of each colour that hold visibilities
    // FP32 gridding (k_grid_mma): a tile's points are cut into parts of about grid_part points,
    // and (tile, part) items are claimed tile colour by tile colour, heaviest tile first
    int grid_part = 0, grid_warps = 0, n_items = 0;
    size_t grid_smem = 0;                  // 0: the plan grids with the other kernels
    int4* tile_info = nullptr;             // [ntiles] {first segment, segments, parts, place in the order of items}
    int2* items = nullptr;                 // [nitems] {tile, part}
    int32_t* nitems = nullptr;             // device count
    int32_t* pend = nullptr;               // [ntiles] parts of the running launch not yet added to U
    int32_t* bpend = nullptr;              // the same for each image of a batch
    int32_t wait_polls = 1 << 22;          // polls (some seconds) after which a wait of the ordered adds gives up
    int32_t test_hold = 0;                 // tests only: launches start with one part too many pending
    pdgb::TileItem* ditems = nullptr;      // [n_ditems] degridding items, heaviest tile first
    int n_ditems = 0;
    int64_t nslot = 0;                     // slots of seg_part
    pdgb::SegSlot* slot_range = nullptr;   // [nslot] points of each slot (init_res_norm)
    std::vector<pdgb::TileItem> h_ditems;
    int32_t* counts_all = nullptr;         // {nseg, tiles that hold visibilities, n_ditems}
    int32_t* ones_block = nullptr;         // all blocks active
    int32_t* ones_basis = nullptr;

    // tables
    void* cx = nullptr;            // real [nx] deapodisation
    void* cy = nullptr;            // real [ny]
    void* cxl = nullptr;           // FP32: what rounding cx and cy to float left
    void* cyl = nullptr;
    void* twx = nullptr;           // complex [Kx]: exp(-2 pi i k / Kx)
    void* twy = nullptr;           // complex [Ky]
    void* filt = nullptr;          // real [b][MAX_FILTER] low-pass filters (0 for Dirac)
    int32_t* filt_len = nullptr;   // [b]
    std::vector<double> h_filt;    // host copy
    std::vector<int> h_filt_len;

    // scratch
    void* t1 = nullptr;            // complex [nx/PW + 1][ny][PW] half-spectrum row-pass intermediate
    void* gridb = nullptr;         // complex [nx/PW + 1][Ky][PW] b~ = F Z x~, columns 0 .. nx
    void* gridu = nullptr;         // complex grid for the plain adjoint
    int batch_cap = 0;             // images the batch scratch below holds (0: none yet)
    void* bt1 = nullptr;           // batch scratch of pd_apply_phi / pd_apply_phi_adj: t1, F Z x, U
    void* bgb = nullptr;
    void* bgu = nullptr;
    void* rbuf = nullptr;          // complex [M] residuals r = v + G b - y (internal order)
    double* seg_part = nullptr;    // [2 * nslot] FP64 partial norms of each segment's share of a part
    double* blk_norm = nullptr;    // [2 * d]: ||r_i||^2, ||G_i b - y_i||^2
    void* blk_scale = nullptr;     // real [d]: max(0, 1 - eps_i / ||r_i||)
    void* ll[2] = {nullptr, nullptr};  // real [b][ny/2][nx/2] wavelet approximation ping-pong
    void* ds = nullptr;            // real [b][ny][nx] change of the sparsity duals
    void* synpart = nullptr;       // real [b][ny][nx] level-0 synthesis of each basis
    double* red = nullptr;         // reduction scratch
    int32_t* sched = nullptr;      // [16] work counters of the dynamically scheduled launches: 0-3 gridding
                                   // colours (zeroed before each launch); 4-5 degridding (next item, CTAs done:
                                   // zeroed by the forward FFT and by every launch); 8 k_grid_mma (next item:
                                   // zeroed with pend); 10: a wait of a plain application gave up
    int red_len = 0;
    size_t device_bytes = 0;
    std::vector<void*> allocs;     // every device allocation of the plan
};

struct pd_state {
    pd_plan* plan = nullptr;
    void* x = nullptr;
    void* xt = nullptr;
    void* s = nullptr;             // [b][ny][nx]
    void* st = nullptr;            // s~ = Psi s
    void* syn_at = nullptr;        // synthesis form: alpha~ [b][ny][nx] (alpha lives in s)
    void* syn_u = nullptr;         // synthesis form: positivity dual u [ny][nx]
    void* v = nullptr;             // complex [M] internal order
    void* u = nullptr;             // complex grid G^T v (panel layout)
    void* y = nullptr;             // complex [M] internal order
    double* eps = nullptr;         // [d]
    double* res_norm = nullptr;    // [d]
    double* p_block = nullptr;     // [d]
    double* p_basis = nullptr;     // [b]
    int32_t* block_active = nullptr;   // [d]
    int32_t* basis_active = nullptr;   // [b]
    int32_t* tile_active = nullptr;    // [ntiles]: tile holds a visibility of an active block
    int32_t* counts = nullptr;         // {active segments, active tiles}
    int64_t* t = nullptr;              // iteration counter (device)
    double* diag = nullptr;            // [2]: ||dx||^2, ||x||^2
    void* u_out = nullptr;             // complex grid: G^T v itself, kept up to date once pd_state_u was called
    double* prim_part = nullptr;       // [2 * ny / rows-per-CTA]
    // staging of a checkpoint's visibilities (the state's own: other states of the plan may be
    // iterating on other streams meanwhile): ck_cap of them and their internal indices, one save
    // or load at a time
    std::mutex ck_mu;
    int64_t ck_cap = 0;
    void* ck_vis = nullptr;
    int32_t* ck_idx = nullptr;
    int32_t* status = nullptr;         // set: a wait of the gridding into this state's U gave up
    std::vector<void*> allocs;
    size_t device_bytes = 0;
    // CUDA graph of one iteration
    cudaGraphExec_t gexec = nullptr;
    std::vector<unsigned char> gkey;
    cudaStream_t gstream = nullptr;    // private stream the graph is captured on and replayed on
    cudaEvent_t ev_in = nullptr, ev_out = nullptr;
    // second stream for the sparsity-prior branch of an iteration (Alg. 1 steps 12-15
    // run concurrently with the data-fidelity steps 6-11), with its fork/join events
    cudaStream_t pstream = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    // plain per-block form (pd_params.per_block): one-hot activity flags, each block's tiles
    int32_t* pb_eye_blocks = nullptr;  // [d][d]
    int32_t* pb_eye_bases = nullptr;   // [b][b]
    pdgb::TileItem* pb_ditems = nullptr;   // degridding items of block i at pb_ditems[h_pb_off[i] ...]
    int32_t* pb_counts = nullptr;      // [d] number of them
    int32_t* pb_col = nullptr;         // tiles of block i and colour c at pb_col[h_pb_off[4 i + c] ...]
    int32_t* pb_ccounts = nullptr;     // [d][4] number of tiles of block i per colour
    int2* pb_items = nullptr;          // k_grid_mma's items of block i at pb_items[h_pb_item_off[i] ...]
    int32_t* pb_nitems = nullptr;      // [d]
    std::vector<int32_t> h_pb_item_off;
    std::vector<int32_t> h_pb_off;
    std::vector<int32_t> h_act, h_actb;
    int64_t h_t = 0;
    // per-phase timing (pd_params.profile)
    cudaEvent_t prof_ev[2 * 12] = {};
    double prof_ms[12] = {};
    int64_t prof_n[12] = {};
};

namespace pdgb {

template <typename R> inline const kb_poly_t<R>& kb_poly(const pd_plan* p) {
    if constexpr (sizeof(R) == 8) return p->kbpoly64;
    else return p->kbpoly;
}

// Kernel phases of one iteration, for optional per-phase CUDA-event timing.
enum Phase {
    PH_SELECT = 0, PH_FWD_ROWS, PH_FWD_COLS, PH_DEGRID, PH_NORMS, PH_GRID, PH_ANALYSIS,
    PH_SYNTHESIS, PH_INV_COLS, PH_INV_ROWS, PH_FINISH, PH_COUNT
};
// Record the start (end = 0) or end (end = 1) event of a phase on stream s when the
// calling thread has profiling switched on; otherwise a no-op.
void prof_mark(int phase, int end, cudaStream_t s);
// Record `msg` as the calling thread's last error (pd_last_error) and return `st`.
pd_status set_error(pd_status st, const char* msg);

// ---- fft.cu
// batch images at once (blockIdx.y); t1: the half-spectrum intermediate of the batch
// (nullptr = the plan's own, for batch 1)
template <typename R>
cudaError_t fwd_fft(const pd_plan* p, const R* x, cplx_t<R>* grid, cudaStream_t s, int batch = 1,
                    cplx_t<R>* t1 = nullptr);
struct PrimalArgs {
    double tau, sigma, varsigma;
    void* x;           // in/out
    void* xt;          // out
    const void* st;    // s~
    double* part;      // per-CTA partial sums
};
// mode 0: write Re(Z^T F^H grid) to out; mode 1: primal update (Alg. 1 steps 17-18)
template <typename R>
cudaError_t inv_fft(const pd_plan* p, const cplx_t<R>* grid, R* out, const PrimalArgs* pa, cudaStream_t s,
                    int batch = 1, cplx_t<R>* t1 = nullptr);
int inv_rows_ctas(const pd_plan* p);

// ---- gridding.cu
// decides whether the plan grids with k_grid_mma, with how many warps and which part size
void grid_setup(pd_plan* p);
struct DualArgs {
    const void* y;        // internal-order data (pd mode) or user-order input (plain mode)
    void* v;              // dual (pd mode)
    const int32_t* block_active;
    const double* eps;
    double* res_norm;     // updated for active blocks
    const int32_t* tile_on = nullptr;   // [ntiles] flags of the tiles to work on (nullptr: every listed one)
    const TileItem* ditems = nullptr;   // degridding items and their device count
    const int32_t* nditems = nullptr;
    const int2* items = nullptr;        // k_grid_mma's work items and their device count
    const int32_t* nitems = nullptr;
    int32_t* gave_up = nullptr;         // set if a wait of the ordered adds gives up
};
// plain degrid of `batch` half grids (stride: one image's half grid) into out (user order, stride M)
template <typename R>
cudaError_t degrid_plain(const pd_plan* p, const cplx_t<R>* grid, cplx_t<R>* out_user, cudaStream_t s, int batch = 1);
// ||G_i grid - y_i|| of every block into res_norm (the exact reading of Sec. 4's c_i)
template <typename R>
cudaError_t degrid_res_norms(const pd_plan* p, const cplx_t<R>* grid, const cplx_t<R>* y, double* res_norm,
                             cudaStream_t s);
// pd degrid over a's items: r = v + G b - y, segment partial norms, then block scales
template <typename R>
cudaError_t degrid_dual(const pd_plan* p, const cplx_t<R>* grid, const DualArgs& a, cudaStream_t s);
// G in CSR form (PD_G_CSR): the J^2 (cell, weight) entries of every visibility
cudaError_t build_csr(pd_plan* p, cudaStream_t s);
// plain grid: U = G^T y_user (U overwritten) for `batch` inputs (stride M) and grids (stride Kx Ky)
template <typename R>
cudaError_t grid_plain(const pd_plan* p, const cplx_t<R>* y_user, cplx_t<R>* U, cudaStream_t s, int batch = 1,
                       int32_t* pend = nullptr, int32_t* gave_up = nullptr);
// pd grid over the listed tiles, one launch per colour (tiles[c]: device list of colour c,
// counts4[c]: device count): v <- scale * r, U += G^T (v_new - v_old)
template <typename R>
cudaError_t grid_dual(const pd_plan* p, const DualArgs& a, const int32_t* const* tiles, const int32_t* counts4,
                      cplx_t<R>* U, cudaStream_t s);

// ---- wavelet.cu
// plain analysis: coeffs[b][ny][nx] = Psi^H x
template <typename R>
cudaError_t psi_adj_plain(const pd_plan* p, const R* x, R* coeffs, cudaStream_t s);
// plain synthesis: x = Psi coeffs
template <typename R>
cudaError_t psi_plain(const pd_plan* p, const R* coeffs, R* x, cudaStream_t s);
// pd: for active bases s <- clip(s + Psi_j^H x~ / sqrt(b), -alpha, alpha); s~ += Psi (s_new - s_old)
template <typename R>
cudaError_t sparsity_dual(const pd_plan* p, const R* xt, R* s, R* st, const int32_t* basis_active,
                          double alpha, cudaStream_t s_, const R* wt = nullptr);
// weights of the reweighted prior: w = delta / (delta + |Psi^H x|), w real [b][ny][nx]
template <typename R>
cudaError_t sara_weights(const pd_plan* p, const R* x, double delta, R* w, cudaStream_t s);

// ---- pd_kernels.cu
struct SelectArgs {
    uint64_t seed;
    int adaptive;
    double n, p_min, p_max;
};
cudaError_t select_active(const pd_plan* p, pd_state* st, const SelectArgs& a, cudaStream_t s);
// synthesis form: positivity dual and image-domain primal term; primal step on the coefficients
template <typename R>
cudaError_t synth_dual(const pd_plan* p, const R* xt, R* u, R* back, double sigma, double varsigma, cudaStream_t s);
template <typename R>
cudaError_t synth_primal(const pd_plan* p, R* alpha, R* alpha_t, const R* w, double tau, double thr, cudaStream_t s);
cudaError_t primal_finish(const pd_plan* p, pd_state* st, cudaStream_t s);
template <typename R>
cudaError_t norm2(const pd_plan* p, const R* x, int64_t n, double* out, cudaStream_t s);
template <typename R>
cudaError_t scale_copy(const R* x, R* y, int64_t n, double scale, cudaStream_t s);
template <typename R>
cudaError_t gather_internal(const pd_plan* p, const cplx_t<R>* user, cplx_t<R>* internal, cudaStream_t s);
// the same through another list of m places (checkpoints)
template <typename R>
cudaError_t gather_by(int64_t m, const int32_t* perm, const cplx_t<R>* src, cplx_t<R>* dst, cudaStream_t s);
template <typename R>
cudaError_t scatter_by(int64_t m, const int32_t* perm, const cplx_t<R>* src, cplx_t<R>* dst, cudaStream_t s);
// out = G^T v of a state, every visibility at its own (u, v): two plain griddings, of the
// visibilities held as conjugates and of the others (uses the plan's rbuf and gridu)
template <typename R>
cudaError_t unfolded_u(const pd_plan* p, const pd_state* st, cplx_t<R>* out, cudaStream_t s);
template <typename R>
cudaError_t scatter_user(const pd_plan* p, const cplx_t<R>* internal, cplx_t<R>* user, cudaStream_t s);
// pend[t] = parts of the tiles that hold a point of an active block (all of them: active null), else 0,
// the gridding's work counter = 0, and U = 0 where given (n4 float4 elements), for `batch` images
cudaError_t grid_begin(const pd_plan* p, const int32_t* active, int32_t* pend, float4* U, int64_t n4, int batch, cudaStream_t s);
cudaError_t init_res_norm(const pd_plan* p, pd_state* st, cudaStream_t s);

}  // namespace pdgb
