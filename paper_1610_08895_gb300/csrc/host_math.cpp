// Host-side tables of the plan: Daubechies filters, Kaiser-Bessel deapodisation
// and FFT twiddles, all computed in FP64.
#include "host_math.hpp"

#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

namespace pdgb {

using cd = std::complex<double>;

// Roots of a polynomial with real coefficients a[0] x^n + ... + a[n] by the
// Weierstrass (Durand-Kerner) simultaneous iteration, polished by Newton steps.
static std::vector<cd> poly_roots(const std::vector<double>& a) {
    const int n = (int)a.size() - 1;
    std::vector<cd> z(n);
    if (n <= 0) return z;
    std::vector<double> m(a.size());
    for (size_t i = 0; i < a.size(); ++i) m[i] = a[i] / a[0];
    auto eval = [&](cd x) {
        cd v = 1.0;
        for (int i = 1; i <= n; ++i) v = v * x + m[i];
        return v;
    };
    auto deriv = [&](cd x) {
        cd v = (double)n;
        for (int i = 1; i < n; ++i) v = v * x + (double)(n - i) * m[i];
        return v;
    };
    const cd seed(0.4, 0.9);
    cd w = 1.0;
    for (int i = 0; i < n; ++i) { z[i] = w; w *= seed; }
    for (int it = 0; it < 2000; ++it) {
        double change = 0.0;
        for (int i = 0; i < n; ++i) {
            cd den = 1.0;
            for (int j = 0; j < n; ++j)
                if (j != i) den *= (z[i] - z[j]);
            const cd step = eval(z[i]) / den;
            z[i] -= step;
            change = std::max(change, std::abs(step));
        }
        if (change < 1e-15) break;
    }
    for (int i = 0; i < n; ++i)
        for (int k = 0; k < 3; ++k) {
            const cd d = deriv(z[i]);
            if (std::abs(d) > 0) z[i] -= eval(z[i]) / d;
        }
    return z;
}

static double binom(int n, int k) {
    double r = 1.0;
    for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
    return r;
}

// db_p low-pass filter: minimum-phase spectral factor of the maximally flat
// half-band polynomial P(y) = sum_{k<p} C(p-1+k, k) y^k (Daubechies 1988).
std::vector<double> daubechies(int p) {
    std::vector<cd> zeros;
    for (int i = 0; i < p; ++i) zeros.push_back(cd(-1.0, 0.0));
    if (p > 1) {
        std::vector<double> coef(p);   // decreasing powers of y
        for (int k = 0; k < p; ++k) coef[p - 1 - k] = binom(p - 1 + k, k);
        for (const cd& y : poly_roots(coef)) {
            // y = (2 - z - 1/z)/4  <=>  z^2 - (2 - 4y) z + 1 = 0; keep the root inside the unit circle
            const cd c = 1.0 - 2.0 * y;
            const cd s = std::sqrt(c * c - 1.0);
            const cd z1 = c + s, z2 = c - s;
            zeros.push_back(std::abs(z1) < 1.0 ? z1 : z2);
        }
    }
    // expand prod (z - zero) in decreasing powers
    std::vector<cd> poly(1, cd(1.0, 0.0));
    for (const cd& r : zeros) {
        std::vector<cd> nxt(poly.size() + 1, cd(0.0, 0.0));
        for (size_t i = 0; i < poly.size(); ++i) {
            nxt[i] += poly[i];
            nxt[i + 1] -= r * poly[i];
        }
        poly.swap(nxt);
    }
    std::vector<double> h(poly.size());
    double sum = 0.0;
    for (size_t i = 0; i < poly.size(); ++i) { h[i] = poly[i].real(); sum += h[i]; }
    for (double& v : h) v *= std::sqrt(2.0) / sum;
    return h;
}

double kb_beta_default(int J) {
    const double a = 2.0;
    return M_PI * std::sqrt((J / a) * (J / a) * (a - 0.5) * (a - 0.5) - 0.8);
}

// Fourier transform of the Kaiser-Bessel window of width J (cycles per cell).
static double kb_hat(double xi, int J, double beta) {
    const double z2 = beta * beta - (M_PI * J * xi) * (M_PI * J * xi);
    if (z2 > 0) { const double z = std::sqrt(z2); return J * std::sinh(z) / z; }
    if (z2 < 0) { const double z = std::sqrt(-z2); return J * std::sin(z) / z; }
    return J;
}

std::vector<double> deapodisation(int n, int K, int J, double beta) {
    std::vector<double> c(n);
    for (int i = 0; i < n; ++i) c[i] = 1.0 / kb_hat((i - n / 2) / (double)K, J, beta);
    return c;
}

std::vector<double> twiddles(int K) {
    std::vector<double> t(2 * K);
    for (int k = 0; k < K; ++k) {
        const double a = 2.0 * M_PI * (double)k / (double)K;
        t[2 * k] = std::cos(a);
        t[2 * k + 1] = -std::sin(a);
    }
    return t;
}

// Kaiser-Bessel weight I0(beta sqrt(1 - (2t/J)^2)), |t| <= J/2.
static double kb_phi(double t, int J, double beta) {
    const double u = 2.0 * t / J;
    const double arg = 1.0 - u * u;
    return arg >= 0 ? std::cyl_bessel_i(0.0, beta * std::sqrt(arg)) : 0.0;
}

// Chebyshev interpolation at the deg + 1 Chebyshev points of the first kind,
// then conversion of sum_j c_j T_j(x) to monomials with T_{j+1} = 2 x T_j - T_{j-1}.
std::vector<double> kb_tap_polynomials(int J, double beta, int deg) {
    const int n = deg + 1;
    std::vector<double> out((size_t)J * n, 0.0);
    for (int a = 0; a < J; ++a) {
        std::vector<double> fx(n), cheb(n, 0.0);
        for (int k = 0; k < n; ++k) {
            const double xk = std::cos(M_PI * (k + 0.5) / n);
            fx[k] = kb_phi((xk + 1.0) / 2.0 + J / 2 - 1 - a, J, beta);
        }
        for (int j = 0; j < n; ++j) {
            double acc = 0.0;
            for (int k = 0; k < n; ++k) acc += fx[k] * std::cos(M_PI * j * (k + 0.5) / n);
            cheb[j] = (j == 0 ? 1.0 : 2.0) * acc / n;
        }
        std::vector<double> tm1(n, 0.0), t0(n, 0.0), mono(n, 0.0);
        t0[0] = 1.0;                                   // T_0
        for (int j = 0; j < n; ++j) {
            for (int i = 0; i < n; ++i) mono[i] += cheb[j] * t0[i];
            std::vector<double> t1(n, 0.0);            // T_{j+1} = 2 x T_j - T_{j-1}
            for (int i = 0; i + 1 < n; ++i) t1[i + 1] += 2.0 * t0[i];
            if (j == 0) { t1.assign(n, 0.0); if (n > 1) t1[1] = 1.0; }
            else for (int i = 0; i < n; ++i) t1[i] -= tm1[i];
            tm1 = t0;
            t0 = t1;
        }
        for (int i = 0; i < n; ++i) out[(size_t)a * n + i] = mono[i];
    }
    return out;
}

// phi(t) = I0(beta sqrt(s)) with s = 1 - (2 t / J)^2 by its power series: positive terms
// (beta^2 / 4)^k s^k / (k!)^2, so that it is exact to its own rounding at every t.
void kb_tap_polynomials_ext(int J, double beta, int deg, int outer, int edge_deg, std::vector<double>& inner,
                            std::vector<double>& edge, double* err) {
    using ld = long double;
    const int n = deg + 1;
    const ld pi = 3.14159265358979323846264338327950288L;
    inner.assign((size_t)(J / 2) * n, 0.0);
    edge.assign(edge_deg + 1, 0.0);
    *err = 1.0;
    if (!(beta <= 64.0)) return;          // steeper than the degrees in use can follow
    std::vector<ld> c(1, 1.0L);
    for (int k = 1; c.back() > 1e-21L || k <= edge_deg; ++k) c.push_back(c.back() * ((ld)beta * beta / 4.0L) / ((ld)k * k));
    auto phi = [&](ld t) {
        const ld u = 2.0L * t / J, q = 1.0L - u * u;
        ld v = 0.0L;
        for (size_t k = c.size(); k-- > 0;) v = v * q + c[k];
        return v;
    };
    const ld phi0 = phi(0.0L);
    ld worst = 0.0L;
    // cos(pi i / (2 n)), for the nodes and the interpolation
    std::vector<ld> cs(4 * n);
    for (int i = 0; i < 4 * n; ++i) cs[i] = std::cos(pi * i / (2 * n));
    std::vector<ld> mono, prev, cur, next, fx(n), cheb(n);
    for (int a = outer; a < J / 2; ++a) {
        for (int k = 0; k < n; ++k) fx[k] = phi((cs[2 * k + 1] + 1.0L) / 2.0L + J / 2 - 1 - a);
        for (int j = 0; j < n; ++j) {
            ld acc = 0.0L;
            for (int k = 0; k < n; ++k) acc += fx[k] * cs[j * (2 * k + 1) % (4 * n)];
            cheb[j] = (j == 0 ? 1.0L : 2.0L) * acc / n;
        }
        // sum_j cheb_j T_j in monomials, T_{j+1} = 2 x T_j - T_{j-1}
        mono.assign(n, 0.0L);
        prev.assign(n, 0.0L);
        cur.assign(n, 0.0L);
        cur[0] = 1.0L;
        for (int j = 0; j < n; ++j) {
            for (int i = 0; i <= j; ++i) mono[i] += cheb[j] * cur[i];
            next.assign(n, 0.0L);
            for (int i = 0; i + 1 < n; ++i) next[i + 1] = (j == 0 ? 1.0L : 2.0L) * cur[i];
            if (j > 0)
                for (int i = 0; i < n; ++i) next[i] -= prev[i];
            prev.swap(cur);
            cur.swap(next);
        }
        for (int i = 0; i < n; ++i) inner[(size_t)a * n + i] = (double)mono[i];
        for (int k = 0; k <= n; ++k) {         // between the nodes, and the ends
            const ld x = cs[2 * k];
            ld v = 0.0L;
            for (int i = n - 1; i >= 0; --i) v = v * x + mono[i];
            worst = std::max(worst, std::abs(v - phi((x + 1.0L) / 2.0L + J / 2 - 1 - a)) / phi0);
        }
    }
    // the outer taps, s in [0, s1]: the series economised (Lanczos 1938): its highest term, replaced by
    // that term's best approximation of lower degree on [0, s1], again and again
    const ld q1 = (ld)(J / 2 - outer) / (J / 2), s1 = 1.0L - q1 * q1;
    const int K = (int)c.size() - 1;
    std::vector<ld> y(K + 1);
    ld pw = 1.0L, dropped = 0.0L;
    for (int k = 0; k <= K; ++k, pw *= s1) y[k] = c[k] * pw;
    // T_k(2 y - 1) / 2^(2 k - 1), leading coefficient 1; in FP64, since the terms they stand for are
    // below 1e-4 of the value
    std::vector<std::vector<double>> T(K + 1);
    for (int k = 0; k <= K; ++k) {
        T[k].assign(k + 1, 0.0);
        if (k == 0) T[0][0] = 1.0;
        else if (k == 1) { T[1][0] = -0.5; T[1][1] = 1.0; }
        else
            for (int i = 0; i <= k; ++i)       // T_k = (4 y - 2) T_{k-1} - T_{k-2}
                T[k][i] = (i > 0 ? T[k - 1][i - 1] : 0.0) - (i < k ? T[k - 1][i] / 2.0 : 0.0) -
                          (i < k - 1 ? T[k - 2][i] / (k == 2 ? 8.0 : 16.0) : 0.0);
    }
    for (int k = K; k > edge_deg; --k) {
        const ld top = y[k];
        for (int i = 0; i <= k; ++i) y[i] -= top * T[k][i];
        dropped += std::abs(std::ldexp(top, 1 - 2 * k));
    }
    pw = 1.0L;
    for (int k = 0; k <= edge_deg; ++k, pw *= s1) edge[k] = (double)(y[k] / pw);
    *err = (double)std::max(worst, dropped);   // phi >= 1 on the outer taps
}

// The gridding of a stored G (four launches by tile colour, one CTA a tile) takes about a + b n
// for a tile of n points, and a launch lasts as long as its heaviest tile or as the average over the
// resident CTAs, with some of the shorter of the two on top. Measured on GB300 (J = 8, real rows):
// a = 4.5, 5 and 7 us for tiles of 8, 16 and 32, b = 0.045, 0.025 and 0.025 us; four CTAs per SM for
// tiles of 8, two for the others and for complex rows. Larger tiles stage fewer window cells a point, in the
// degridding too, and win within 5%. Phi^H in tiles of 8 / 16 / 32: 262,144 points on 512^2 cells
// 154 / 294 / 839 us, 1.05M on 1024^2 239 / 211 / 541, 4.19M Gaussian on 2048^2 776 / 728 / 1340,
// 16.8M on 4096^2 3057 / 2794 / 2350, 1.05M there 1685 / 1100 / 554.
int stored_tile(const std::vector<int32_t>& cell, int Kx, int Ky, bool cplx, int num_sms) {
    std::vector<int32_t> n((size_t)(Kx / 8) * (Ky / 8), 0);
    for (int32_t c : cell) n[(size_t)(c >> 19) * (Kx / 8) + ((c & 0xFFFF) >> 3)]++;
    const double a[3] = {cplx ? 5.2 : 4.5, 5.0, 7.0};
    const double b[3] = {cplx ? 0.028 : 0.045, cplx ? 0.028 : 0.025, cplx ? 0.028 : 0.025};
    double best = 0.0;
    int tile = 8, w = Kx / 8, h = Ky / 8;
    for (int k = 0; k < 3; ++k) {
        if (k > 0) {                       // the counts of tiles twice as large
            if (w < 4 || h < 4) break;     // two tiles a side at least
            for (int y = 0; y < h / 2; ++y)
                for (int x = 0; x < w / 2; ++x) {
                    const size_t q = (size_t)2 * y * w + 2 * x;
                    n[(size_t)y * (w / 2) + x] = n[q] + n[q + 1] + n[q + w] + n[q + w + 1];
                }
            w /= 2;
            h /= 2;
        }
        int most = 0, used = 0;
        for (size_t i = 0; i < (size_t)w * h; ++i) {
            most = std::max(most, n[i]);
            used += n[i] > 0;
        }
        const double ctas = (double)num_sms * (k == 0 && !cplx ? 4 : 2);
        const double heavy = a[k] + b[k] * most, mean = (used * a[k] + b[k] * (double)cell.size()) / (4.0 * ctas);
        const double t = std::max(heavy, mean) + 0.4 * std::min(heavy, mean);
        if (k == 0 || t <= 1.05 * best) {
            best = k == 0 ? t : std::min(best, t);
            tile = 8 << k;
        }
    }
    return tile;
}

// Stable counting sort of `in` (or 0 .. n - 1) by key(i) in [0, nkeys).
template <typename Key>
static std::vector<int32_t> counting_sort(size_t n, const std::vector<int32_t>* in, int64_t nkeys, const Key& key) {
    std::vector<int32_t> at(nkeys + 1, 0), out(n);
    for (size_t i = 0; i < n; ++i) at[key((int32_t)i) + 1]++;
    for (int64_t k = 0; k < nkeys; ++k) at[k + 1] += at[k];
    for (size_t i = 0; i < n; ++i) {
        const int32_t m = in ? (*in)[i] : (int32_t)i;
        out[at[key(m)]++] = m;
    }
    return out;
}

PointOrder order_points(const std::vector<int32_t>& cell, const int32_t* block, int nblocks, int logT, int ntx,
                        int ntiles) {
    const size_t n = cell.size();
    const int T = 1 << logT, side = std::max(1, T / 8);
    auto tile_of = [&](int32_t m) { return (cell[m] >> (16 + logT)) * ntx + ((cell[m] & 0xFFFF) >> logT); };
    PointOrder o;
    // one pass over (tile, block) while its counters stay in reach of the caches, else one over the
    // blocks and one over the tiles
    if ((int64_t)ntiles * nblocks <= (int64_t)1 << 25) {
        o.order = counting_sort(n, nullptr, (int64_t)ntiles * nblocks,
                                [&](int32_t m) { return (int64_t)tile_of(m) * nblocks + block[m]; });
    } else {
        const std::vector<int32_t> by_block = counting_sort(n, nullptr, nblocks, [&](int32_t m) { return block[m]; });
        o.order = counting_sort(n, &by_block, ntiles, tile_of);
    }
    int ptile = -1, pblock = -1;
    for (size_t i = 0; i < n; ++i) {
        const int32_t m = o.order[i], t = tile_of(m);
        if (t != ptile || block[m] != pblock) {
            o.seg_start.push_back((int32_t)i);
            o.seg_tile.push_back(ptile = t);
            o.seg_block.push_back(pblock = block[m]);
        }
    }
    o.seg_start.push_back((int32_t)n);
    // within a segment: its points are in the order of their indices, so that a stable counting sort
    // over the tile's cells, or a sort of (cell, index) where the points are fewer, leaves ties so
    auto place = [&](int32_t m) {
        const int ly = (cell[m] >> 16) & (T - 1), lx = cell[m] & (T - 1);
        return ((uint64_t)((ly >> 3) * side + (lx >> 3)) << 6) | ((ly & 7) << 3) | (lx & 7);
    };
    const size_t places = (size_t)side * side << 6;
    std::vector<uint64_t> key;
    std::vector<int32_t> at, tmp;
    for (size_t sg = 0; sg + 1 < o.seg_start.size(); ++sg) {
        int32_t* p = o.order.data() + o.seg_start[sg];
        const size_t len = o.seg_start[sg + 1] - o.seg_start[sg];
        if (len > places / 4) {
            at.assign(places + 1, 0);
            tmp.assign(p, p + len);
            for (int32_t m : tmp) at[place(m) + 1]++;
            for (size_t k = 0; k < places; ++k) at[k + 1] += at[k];
            for (int32_t m : tmp) p[at[place(m)]++] = m;
        } else {
            key.resize(len);
            for (size_t i = 0; i < len; ++i) key[i] = place(p[i]) << 31 | (uint32_t)p[i];
            std::sort(key.begin(), key.end());
            for (size_t i = 0; i < len; ++i) p[i] = (int32_t)(key[i] & 0x7fffffffu);
        }
    }
    return o;
}

}  // namespace pdgb
