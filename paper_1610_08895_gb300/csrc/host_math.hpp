// Host-side FP64 tables of the plan (filters, deapodisation, twiddles).
#pragma once

#include <cstdint>
#include <cstdint>
#include <vector>

namespace pdgb {

// Low-pass filter of db_p, largest tap first, sum sqrt(2).
std::vector<double> daubechies(int p);
// pi sqrt((J/2)^2 (3/2)^2 - 0.8): Kaiser-Bessel shape for 2x oversampling.
double kb_beta_default(int J);
// c[i] = 1 / phi_hat((i - n/2) / K) for a J-wide Kaiser-Bessel kernel.
std::vector<double> deapodisation(int n, int K, int J, double beta);
// interleaved (cos, -sin)(2 pi k / K), k in [0, K)
std::vector<double> twiddles(int K);
// Monomial coefficients (in x = 2 f - 1, f in [0, 1)) of the degree-`deg` Chebyshev
// interpolant of tap a's weight phi(f + J/2 - 1 - a), for a = 0..J-1: [J][deg + 1].
std::vector<double> kb_tap_polynomials(int J, double beta, int deg);
// The weights for FP64, fitted in extended precision. Taps outer <= a < J/2: the same monomials,
// [J/2][deg + 1]. The `outer` outermost taps on either side, where the weight falls to 1 / I0(beta)
// of its largest value: one polynomial in s = 1 - (2 t / J)^2, [edge_deg + 1], exact to the weight
// itself there. *err: the larger of the first fit's deviation between the nodes relative to phi(0)
// and the second one's relative to the weight, before the coefficients are rounded to FP64 (1: not
// fitted, beta too large).
void kb_tap_polynomials_ext(int J, double beta, int deg, int outer, int edge_deg, std::vector<double>& inner,
                            std::vector<double>& edge, double* err);

// Tile edge (8, 16 or 32) for a stored G in FP32, from where the points' footprints start: cell as
// (y << 16) | x on a Kx x Ky grid. cplx: complex rows.
int stored_tile(const std::vector<int32_t>& cell, int Kx, int Ky, bool cplx, int num_sms);

// Points by (tile, block), then 8 x 8 super-cell, row, column and index. cell: (y << 16) | x, in
// tiles of 2^logT cells, ntx of them in a row. Segments are the runs of one (tile, block).
struct PointOrder {
    std::vector<int32_t> order;           // [n] indices of the points
    std::vector<int32_t> seg_start;       // [segments + 1]
    std::vector<int32_t> seg_block, seg_tile;
};
PointOrder order_points(const std::vector<int32_t>& cell, const int32_t* block, int nblocks, int logT, int ntx,
                        int ntiles);

}  // namespace pdgb
