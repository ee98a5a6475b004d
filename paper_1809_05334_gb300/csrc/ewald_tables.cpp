// Host set-up of the Ewald series of one incidence (Sec. 2.2, Eq. (3)-(4)):
// the splitting parameter, the lattice images and Floquet orders inside the
// cut, and the Floquet-order rectangle and distinct decay constants of the
// FP32 tables.  Host code only (the library and the host-logic tests compile
// it).
#include <algorithm>
#include <array>
#include <cmath>
#include <complex>
#include <cstring>
#include <vector>

#include "../../include/vie.h"
#include "ewald_tables.h"

namespace vie {

// Ewald parameters and tables of one incidence (Sec. 2.2, Eq. (3)-(4)): the
// splitting parameter, the lattice images and Floquet modes inside the cut of
// the FP64 (fp64) or FP32 series, the limit of the regularised image term, the
// rectangle of Floquet orders and the distinct decay constants of the FP32
// tables (z_extent = the largest |dz| they must cover).  `orders` (may be null)
// receives the propagating orders [n][4] (k_tx, k_ty, k_z, 1 for (0,0)).  The
// solver and the allocation-free entry point both build their tables here.
// Returns VIE_OK, VIE_RAYLEIGH_ANOMALY (a Floquet order at grazing) or
// VIE_EINVAL (a table would overflow), with *why set.
int build_ewald_tables(double a, double b, double k0, double kx, double ky, double z_extent, bool fp64,
                       EwaldTables &E, std::vector<double> *orders, const char **why, double split_mult, bool pow2) {
    std::memset(&E, 0, sizeof(E));
    if (orders) orders->clear();
    E.E = ewald_split(a, b, k0, !fp64, kx == 0.0 && ky == 0.0, split_mult);
    E.bb = k0 / (2.0 * E.E);
    E.a = a;
    E.b = b;
    E.xcut64 = FP64_XCUT;
    E.xcut32 = FP32_XCUT;
    const double xc = fp64 ? FP64_XCUT : (double)FP32_XCUT;
    const int mm = (int)std::ceil(xc / (E.E * a)) + 2, nn = (int)std::ceil(xc / (E.E * b)) + 2;
    int ni = 0;
    for (int m = -mm; m <= mm; ++m)
        for (int n = -nn; n <= nn; ++n) {
            const double dmin = std::hypot(std::max(std::abs(m) - 1, 0) * a, std::max(std::abs(n) - 1, 0) * b);
            const bool nearimg = std::abs(m) <= 1 && std::abs(n) <= 1;
            if (dmin * E.E > xc && !nearimg) continue;
            if (ni >= MAX_IMG) { *why = "period too small for the image table"; return VIE_EINVAL; }
            const double phs = kx * m * a + ky * n * b, f = std::exp(E.bb * E.bb) / (4.0 * M_PI);
            const double v[4] = {m * a, n * b, f * std::cos(phs), f * std::sin(phs)};
            for (int q = 0; q < 4; ++q) { E.img64[ni][q] = v[q]; E.img32[ni][q] = (float)v[q]; }
            if (nearimg) E.near_img[(m + 1) * 3 + (n + 1)] = ni;
            ++ni;
        }
    E.n_img = ni;
    const int pm = (int)std::ceil((2.0 * E.E * xc + std::fabs(kx)) * a / (2 * M_PI)) + 1;
    const int qm = (int)std::ceil((2.0 * E.E * xc + std::fabs(ky)) * b / (2 * M_PI)) + 1;
    int nm = 0;
    for (int p = -pm; p <= pm; ++p)
        for (int q = -qm; q <= qm; ++q) {
            const double ktx = kx + 2 * M_PI * p / a, kty = ky + 2 * M_PI * q / b;
            const double kt2 = ktx * ktx + kty * kty, g2 = kt2 - k0 * k0;
            if (std::fabs(g2) * std::max(a, b) * std::max(a, b) < 1e-10) {
                *why = "a Floquet order is at grazing (Rayleigh anomaly)";
                return VIE_RAYLEIGH_ANOMALY;
            }
            if (g2 < 0 && orders) orders->insert(orders->end(), {ktx, kty, std::sqrt(-g2), (p == 0 && q == 0) ? 1.0 : 0.0});
            if (std::sqrt(kt2) > 2.0 * E.E * xc + k0) continue;
            if (nm >= MAX_MODE) { *why = "too many Floquet modes for the table"; return VIE_EINVAL; }
            // gamma = sqrt(g2) (evanescent) or j sqrt(-g2) (propagating); 1/(4 a b gamma)
            const double gr = g2 >= 0 ? std::sqrt(g2) : 0.0, gi = g2 >= 0 ? 0.0 : std::sqrt(-g2);
            const double ir = gr / (4.0 * a * b * (gr * gr + gi * gi)), ii = -gi / (4.0 * a * b * (gr * gr + gi * gi));
            const double w8[8] = {ktx, kty, gr, gi, std::exp(-g2 / (4 * E.E * E.E)), ir, ii, 0};
            for (int c = 0; c < 8; ++c) { E.mode64[nm][c] = w8[c]; E.mode32[nm][c] = (float)w8[c]; }
            ++nm;
        }
    E.n_mode = nm;
    {   // erfi(b) by its series, for the limit R -> 0 of the regularised image term
        double term = E.bb, sum = E.bb;
        for (int n = 1; n < 200; ++n) {
            term *= E.bb * E.bb / n;
            const double add = term / (2 * n + 1);
            sum += add;
            if (std::fabs(add) < 1e-18 * std::fabs(sum)) break;
        }
        const double erfi = 2.0 / std::sqrt(M_PI) * sum;
        E.reg0_re = (E.E / (4 * M_PI)) * (2 * E.bb * erfi - 2.0 / std::sqrt(M_PI) * std::exp(E.bb * E.bb));
    }
    // tabulated FP32 path: the truncation of the FP32 series
    const double xc32 = FP32_XCUT, zr = std::max(z_extent, 1e-6) * (1.0 + 1e-6);
    E.xs_max = (float)(xc32 + 0.5);
    // intervals per unit of x: such that E xs_inv_h, the table intervals per unit of
    // distance, is a power of two (distances scaled to table units stay exact) and
    // the cut falls in the table's upper half
    E.xs_inv_h = (float)(pow2 ? std::exp2(std::floor(std::log2(NSPAT * E.E / (xc32 + 0.5)))) / E.E : NSPAT / (xc32 + 0.5));
    // the interval itself in FP64: the kernels index with the exact power of two, and an
    // interval off by FP32 rounding would give the images another E than the orders have
    E.xs_h = pow2 ? E.E / std::exp2(std::floor(std::log2(NSPAT * E.E / (xc32 + 0.5)))) : (double)E.xs_max / NSPAT;
    E.z_max = (float)zr;
    E.z_inv_h = (float)(NZTAB / zr);
    E.e_mb2 = (float)std::exp(-E.bb * E.bb);
    E.Ef = (float)E.E;
    E.kx = (float)kx;
    E.ky = (float)ky;
    E.step_x = (float)(2 * M_PI / a);
    E.step_y = (float)(2 * M_PI / b);
    if (!mode_rect(kx, ky, a, b, 2.0 * E.E * xc32 + k0, E.p0, E.np, E.q0, E.nq)) {
        *why = "too many Floquet modes for the table";
        return VIE_EINVAL;
    }
    E.sym = (kx == 0.0 && ky == 0.0 && 2 * E.p0 + E.np == 1 && 2 * E.q0 + E.nq == 1) ? 1 : 0;
    int nt = 0;
    double g2s[MAX_MODE];
    for (int p = E.p0; p < E.p0 + E.np; ++p)
        for (int q = E.q0; q < E.q0 + E.nq; ++q) {
            const int idx = (p - E.p0) * E.nq + (q - E.q0);
            const double ktx = kx + 2 * M_PI * p / a, kty = ky + 2 * M_PI * q / b;
            const double kt2 = ktx * ktx + kty * kty;
            if (std::sqrt(kt2) > 2.0 * E.E * xc32 + k0) { E.rect_tab[idx] = -1; continue; }
            const double g2 = kt2 - k0 * k0;
            int found = -1;
            for (int j = 0; j < nt; ++j)
                if (std::fabs(g2s[j] - g2) <= 1e-12 * std::max(1e-6, std::fabs(g2))) { found = j; break; }
            if (found < 0) {
                found = nt++;
                g2s[found] = g2;
                const double gr = g2 >= 0 ? std::sqrt(g2) : 0.0, gi = g2 >= 0 ? 0.0 : std::sqrt(-g2);
                E.tab_gamma[found][0] = gr;
                E.tab_gamma[found][1] = gi;
                E.tab_ig[found][0] = gr / (4.0 * a * b * (gr * gr + gi * gi));
                E.tab_ig[found][1] = -gi / (4.0 * a * b * (gr * gr + gi * gi));
                E.tab_pre[found] = std::exp(-g2 / (4 * E.E * E.E));
            }
            // bit 16 marks a real decay constant (evanescent mode): its G is real
            E.rect_tab[idx] = found | (g2s[found] > 0 ? TAB_REAL : 0);
        }
    E.n_tab = nt;
    return VIE_OK;
}

// ---------------------------------------------------------------------------
// Polynomials of the spectral series
// ---------------------------------------------------------------------------
namespace {

using cd = std::complex<double>;

// w(j u) = erfcx(u), Re u >= 0, by Weideman's rational expansion with 40 terms
// (SIAM J. Numer. Anal. 31, 1994), FP64
cd erfcx_host(cd u) {
    constexpr int NT = 40;
    static const std::vector<double> a = [] {
        std::vector<double> c(NT + 1, 0.0);
        const double L = std::sqrt(NT / std::sqrt(2.0));
        const int M = 16 * NT;
        for (int k = 0; k < M; ++k) {
            const double th = -M_PI + (k + 0.5) * 2.0 * M_PI / M, t = L * std::tan(0.5 * th);
            const double F = std::exp(-t * t) * (L * L + t * t);
            for (int n = 0; n <= NT; ++n) c[n] += F * std::cos(n * th) / M;
        }
        return c;
    }();
    const double L = std::sqrt(NT / std::sqrt(2.0));
    const cd inv = 1.0 / (L + u), z = (L - u) * inv;
    cd p = a[NT];
    for (int n = NT - 1; n >= 1; --n) p = cd(p.real() * z.real() - p.imag() * z.imag() + a[n], p.real() * z.imag() + p.imag() * z.real());
    return inv * (2.0 * p * inv + 1.0 / std::sqrt(M_PI));
}

// G(z) of table tb: [e^{gz} erfc(g/2E + zE) + e^{-gz} erfc(g/2E - zE)] / (4ab g)
cd spectral_value(const EwaldTables &t, int tb, double z) {
    const double E = t.E, gr = t.tab_gamma[tb][0], gi = t.tab_gamma[tb][1];
    if (gi == 0.0) {
        const double u = gr / (2 * E);
        return (std::exp(gr * z) * std::erfc(u + z * E) + std::exp(-gr * z) * std::erfc(u - z * E)) * t.tab_ig[tb][0];
    }
    const cd e1 = erfcx_host(cd(z * E, gi / (2 * E)));
    const double pre = t.tab_pre[tb] * std::exp(-(z * E) * (z * E));
    const cd sum(2.0 * std::cos(gi * z), 2.0 * pre * e1.imag() - 2.0 * std::sin(gi * z));
    return sum * cd(t.tab_ig[tb][0], t.tab_ig[tb][1]);
}

}  // namespace

void build_far_poly(const EwaldTables &t, const EwaldF32 &f, FarPoly &fp, std::vector<float> &coef) {
    fp = FarPoly{};
    coef.clear();
    const int Q = (t.nq - 1) / 2;
    int rows = 0, nq = 0, mode = FAR_NONE;
    if (t.sym && f.sq_pq > 0) {
        mode = FAR_NORMAL;
        rows = (t.np - 1) / 2 + 1;
        nq = std::max(3, Q + 1);
    } else if (!t.sym && f.ob_nr > 0) {
        mode = f.ob_nq1 > 0 ? FAR_FOLD : FAR_FULL;
        rows = t.np;
        nq = f.ob_nq1 > 0 ? std::max(3, Q + 1) : (t.nq <= 4 ? 4 : (t.nq == 7 ? 8 : t.nq));
    }
    if (mode == FAR_NONE || rows > FP_ROWS) return;
    // table of entry (i, j) of the map, -1 outside the cut; whether it is propagating
    auto entry = [&](int i, int j, bool &prop) {
        prop = false;
        int off, im = -1;
        if (mode == FAR_NORMAL) {
            off = f.sq_off[i][j];
            prop = i == 0 && j == 0 && f.sq_im != t.n_tab * NZTAB;
        } else {
            off = f.ob_off[i][j];
            im = f.ob_im[i][j];
            prop = im >= 0;
        }
        const int tb = off / NZTAB;
        return tb == t.n_tab ? -1 : tb;
    };
    // Chebyshev coefficients of every table in use, in t on [-1, 1], from M nodes
    // (the degree grows as 3.5 + 3.8 E z_max; M leaves room for the tail to show)
    const double zm = t.z_max, Ez = t.E * zm;
    if (!(Ez < 9.0)) return;
    const int M = std::min(48, std::max(14, (int)std::ceil(13 + 4.6 * Ez)));
    std::vector<std::vector<double>> re(t.n_tab), im(t.n_tab);
    std::vector<double> cs((size_t)M * M);
    for (int k = 0; k < M; ++k)
        for (int n = 0; n < M; ++n) cs[(size_t)k * M + n] = std::cos(M_PI * n * (k + 0.5) / M);
    double gmax = 0;
    for (int i = 0; i < rows; ++i)
        for (int j = 0; j < nq; ++j) {
            bool prop;
            const int tb = entry(i, j, prop);
            if (tb < 0 || !re[tb].empty()) continue;
            std::vector<double> vr(M), vi(M);
            for (int k = 0; k < M; ++k) {
                const double tt = cs[(size_t)k * M + 1];
                const cd g = spectral_value(t, tb, zm * std::sqrt(0.5 * (tt + 1.0)));
                vr[k] = g.real();
                vi[k] = g.imag();
                gmax = std::max(gmax, std::fabs(vr[k]));
            }
            re[tb].assign(M, 0.0);
            im[tb].assign(M, 0.0);
            for (int n = 0; n < M; ++n) {
                double sr = 0, si = 0;
                for (int k = 0; k < M; ++k) {
                    sr += vr[k] * cs[(size_t)k * M + n];
                    si += vi[k] * cs[(size_t)k * M + n];
                }
                re[tb][n] = (n ? 2.0 : 1.0) / M * sr;
                im[tb][n] = (n ? 2.0 : 1.0) / M * si;
            }
        }
    if (!(gmax > 0) || !std::isfinite(gmax)) return;
    // a column keeps its terms until the rest is below 1e-9 of the largest order
    // (the FP32 rounding of the sum is 6e-8 of it)
    const double tol = 1e-9 * gmax;
    auto degree = [&](const std::vector<double> &c) {
        double rest = 0;
        int d = M - 1;
        while (d > 0 && rest + std::fabs(c[d]) <= tol) rest += std::fabs(c[d--]);
        return d;
    };
    // Chebyshev series up to degree d as a polynomial in t
    auto monomial = [](const std::vector<double> &c, int d) {
        std::vector<double> out(d + 1, 0.0), a(d + 1, 0.0), b(d + 1, 0.0), n(d + 1);
        a[0] = 1.0;   // T_0
        out[0] += c[0];
        if (d >= 1) { b[1] = 1.0; out[1] += c[1]; }
        for (int k = 2; k <= d; ++k) {
            for (int q = 0; q <= d; ++q) n[q] = (q ? 2.0 * b[q - 1] : 0.0) - a[q];
            for (int q = 0; q <= k; ++q) out[q] += c[k] * n[q];
            a.swap(b);
            b.swap(n);
        }
        return out;
    };
    fp.rows = rows;
    fp.nq = nq;
    for (int i = 0; i < rows; ++i)
        for (int part = 0; part < 2; ++part) {   // real, imaginary
            int deg = part ? -1 : 0;
            std::vector<std::vector<double>> col(nq);
            for (int j = 0; j < nq; ++j) {
                bool prop;
                const int tb = entry(i, j, prop);
                if (tb < 0 || (part && !prop)) continue;
                const std::vector<double> &c = part ? im[tb] : re[tb];
                const int d = degree(c);
                if (d > FP_MAX_DEG - 1) { fp = FarPoly{}; coef.clear(); return; }
                col[j] = monomial(c, d);
                deg = std::max(deg, d);
            }
            if (deg > 0) deg = (deg + 1) & ~1;   // even: the kernels take two powers per step
            (part ? fp.im_off : fp.off)[i] = (int)coef.size();
            (part ? fp.im_deg : fp.deg)[i] = deg;
            for (int n = deg; n >= 0; --n)
                for (int j = 0; j < ((nq + 1) & ~1); ++j)
                    coef.push_back(j < nq && n < (int)col[j].size() ? (float)col[j][n] : 0.f);
        }
    if ((int)coef.size() > FP_MAX_COEF) { fp = FarPoly{}; coef.clear(); return; }
    fp.n_coef = (int)coef.size();
    const double zs = zm * f.Eih;
    fp.t_scale = (float)(2.0 / (zs * zs));
    if (mode == FAR_NORMAL) {
        auto at_zero = [](const std::vector<double> &c) {   // t = -1
            double s = 0;
            for (int n = 0; n < (int)c.size(); ++n) s += n & 1 ? -c[n] : c[n];
            return s;
        };
        bool prop;
        const int tb = entry(0, 0, prop);
        if (tb >= 0) {
            fp.k_re = (float)at_zero(re[tb]);
            fp.k_im = prop ? (float)at_zero(im[tb]) : 0.f;
        }
    }
    fp.mode = mode;
}

// ---------------------------------------------------------------------------
// The FP64 form
// ---------------------------------------------------------------------------
namespace {

// Chebyshev coefficients of f on [-1, 1] from M nodes
using ld = long double;
using cld = std::complex<long double>;
const ld PI_L = 3.14159265358979323846264338327950288L;
// as erfcx_host, with 64 terms in extended precision
cld erfcx_ld(cld u) {
    constexpr int NT = 64;
    static const ld L = std::sqrt((ld)NT / std::sqrt((ld)2));
    static const std::vector<ld> a = [] {
        std::vector<ld> c(NT + 1, 0);
        const int M = 16 * NT;
        for (int k = 0; k < M; ++k) {
            const ld th = -PI_L + (k + 0.5L) * 2 * PI_L / M, t = L * std::tan(th / 2), F = std::exp(-t * t) * (L * L + t * t);
            for (int n = 0; n <= NT; ++n) c[n] += F * std::cos(n * th) / M;
        }
        return c;
    }();
    const cld inv = (ld)1 / (L + u), z = (L - u) * inv;
    cld p = a[NT];
    for (int n = NT - 1; n >= 1; --n) p = cld(p.real() * z.real() - p.imag() * z.imag() + a[n], p.real() * z.imag() + p.imag() * z.real());
    return inv * ((ld)2 * p * inv + (ld)1 / std::sqrt(PI_L));
}
template <typename F> std::vector<ld> cheb_fit(int M, F &&f) {
    std::vector<ld> v(M), c(M, 0);
    for (int k = 0; k < M; ++k) {
        const ld x = std::cos(PI_L * (k + 0.5L) / M), y = f(x);
        ld t0 = 1, t1 = x;
        for (int n = 0; n < M; ++n) {
            c[n] += (n ? 2 : 1) * y * t0 / M;
            const ld t2 = 2 * x * t1 - t0;
            t0 = t1;
            t1 = t2;
        }
    }
    return c;
}
// the series up to degree d as a polynomial, constant term first
std::vector<ld> cheb_poly(const std::vector<ld> &c, int d) {
    std::vector<ld> out(d + 1, 0), a(d + 1, 0), b(d + 1, 0), n(d + 1);
    a[0] = 1;
    out[0] += c[0];
    if (d >= 1) { b[1] = 1; out[1] += c[1]; }
    for (int k = 2; k <= d; ++k) {
        for (int q = 0; q <= d; ++q) n[q] = (q ? 2 * b[q - 1] : 0) - a[q];
        for (int q = 0; q <= k; ++q) out[q] += c[k] * n[q];
        a.swap(b);
        b.swap(n);
    }
    return out;
}

}  // namespace

void build_far64(const EwaldTables &t, double k0, double kx, double ky, Far64 &f, std::vector<double> &blob) {
    f = Far64{};
    blob.clear();
    const double a = t.a, b = t.b, E = t.E, bb = t.bb, xc = FP64_XCUT, kmax = 2.0 * E * xc + k0;
    const double zm = t.z_max, Ez = E * zm, ts = 2.0 / (zm * zm);
    if (!(Ez < 6.0)) return;
    int p0, np, q0, nq;
    if (!mode_rect(kx, ky, a, b, kmax, p0, np, q0, nq) || np == 0) return;
    const bool sym = kx == 0.0 && ky == 0.0 && 2 * p0 + np == 1 && 2 * q0 + nq == 1;
    if (p0 > 0 || q0 > 0 || p0 + np <= 0 || q0 + nq <= 0) return;   // (0, 0) is always inside the cut
    if (sym) { p0 = q0 = 0; np = (np + 1) / 2; nq = (nq + 1) / 2; }
    // spatial kernel: F on [i h, (i + 1) h] in v = x / h - i
    const double h = (xc + 0.5) / F64_SPAT;   // as the series: images up to the cut + 0.5
    for (int i = 0; i < F64_SPAT; ++i) {
        // F = Re y with y' = 2 j b y - (2 / sqrt pi) exp(-x^2): one value of y at the middle of
        // the interval and its Taylor terms by recurrence, then the Chebyshev terms of that
        // (13 values of y per interval, on a host whose extended precision is in software,
        // were 16 ms a request)
        constexpr int NT = 14;   // (h / 2)^15 < 1e-23
        const ld x = (i + 0.5L) * (ld)h, hh = (ld)h / 2, r = 2 / std::sqrt(PI_L);
        cld y = std::exp(-x * x) * erfcx_ld(cld(x, bb));
        ld g0 = 0, g1 = std::exp(-x * x);   // terms of exp(-x^2), n - 1 and n
        std::vector<ld> tay(NT + 1), c(NT + 1, 0);
        ld p = 1;
        for (int n = 0; n <= NT; ++n) {
            tay[n] = y.real() * p;   // in u: x = centre + u h / 2
            p *= hh;
            y = (cld(-2 * (ld)bb * y.imag(), 2 * (ld)bb * y.real()) - r * g1) / (ld)(n + 1);
            const ld g2 = -2 * (x * g1 + g0) / (n + 1);
            g0 = g1;
            g1 = g2;
        }
        // Chebyshev series by Horner in u: u T_k = (T_{k+1} + T_{k-1}) / 2
        std::vector<ld> w(NT + 2);
        for (int n = NT; n >= 0; --n) {
            std::fill(w.begin(), w.end(), (ld)0);
            for (int k = 0; k < NT - n; ++k) {   // degree so far
                if (k == 0) w[1] += c[0];
                else {
                    w[k + 1] += c[k] / 2;
                    w[k - 1] += c[k] / 2;
                }
            }
            w[0] += tay[n];
            c.assign(w.begin(), w.begin() + NT + 1);
        }
        // polynomial in u = 2 v - 1, shifted to v
        const std::vector<ld> pu = cheb_poly(c, F64_DEG);
        std::vector<ld> pv(F64_DEG + 1, 0);
        for (int n = F64_DEG; n >= 0; --n) {   // Horner in (2 v - 1)
            for (int q = F64_DEG; q >= 0; --q) pv[q] = (q ? 2 * pv[q - 1] : 0) - pv[q];
            pv[0] += pu[n];
        }
        blob.insert(blob.end(), pv.begin(), pv.end());
    }
    blob.resize((size_t)(F64_SPAT + 1) * (F64_DEG + 1), 0.0);
    f.img = (int)blob.size();
    for (int i = 0; i < t.n_img; ++i) blob.insert(blob.end(), t.img64[i], t.img64[i] + 4);
    if (blob.size() & 1) blob.push_back(0.0);   // the directory's entries are read as int4: 16-byte boundaries
    f.dir = (int)blob.size();
    blob.resize(blob.size() + 2 * (size_t)np * nq, 0.0);
    const int M = std::min(64, (int)std::ceil(24 + 7 * Ez));
    double g00 = 0;   // the size of the sum: the largest order at z = 0
    struct Fit { double g2; std::vector<ld> re, im; };
    std::vector<Fit> fits;   // per distinct decay constant
    std::vector<int> which((size_t)np * nq, -1);
    for (int i = 0; i < np; ++i)
        for (int j = 0; j < nq; ++j) {
            const double ktx = kx + 2 * M_PI * (p0 + i) / a, kty = ky + 2 * M_PI * (q0 + j) / b, kt2 = ktx * ktx + kty * kty;
            if (std::sqrt(kt2) > kmax) continue;
            const double g2 = kt2 - k0 * k0;
            int k = 0;
            while (k < (int)fits.size() && std::fabs(fits[k].g2 - g2) > 1e-12 * std::max(1e-6, std::fabs(g2))) ++k;
            which[(size_t)i * nq + j] = k;
            if (k < (int)fits.size()) continue;
            const ld kx_ = (ld)kx + 2 * PI_L * (p0 + i) / a, ky_ = (ld)ky + 2 * PI_L * (q0 + j) / b, g2l = kx_ * kx_ + ky_ * ky_ - (ld)k0 * k0;
            const ld gr = g2l >= 0 ? std::sqrt(g2l) : 0, gi = g2l >= 0 ? 0 : std::sqrt(-g2l), El = E;
            const ld pre0 = std::exp(-g2l / (4 * El * El)), zs = std::sqrt((ld)2 / (ld)ts);
            auto value = [&](ld u) {
                const ld z = zs * std::sqrt(std::max((ld)0, (u + 1) / 2));
                if (gi == 0) {
                    const ld w = gr / (2 * El);
                    return cld((std::exp(gr * z) * std::erfc(w + z * El) + std::exp(-gr * z) * std::erfc(w - z * El)) / (4 * (ld)a * b * gr), 0);
                }
                const cld e1 = erfcx_ld(cld(z * El, gi / (2 * El)));
                const ld pre = pre0 * std::exp(-(z * El) * (z * El));
                return cld(2 * std::cos(gi * z), 2 * pre * e1.imag() - 2 * std::sin(gi * z)) / cld(0, 4 * (ld)a * b * gi);
            };
            Fit fit{g2, cheb_fit(M, [&](ld u) { return value(u).real(); }), {}};
            if (gi > 0) fit.im = cheb_fit(M, [&](ld u) { return value(u).imag(); });
            g00 = std::max(g00, (double)std::abs(value(-1)));
            fits.push_back(std::move(fit));
        }
    if (!(g00 > 0) || !std::isfinite(g00)) { blob.clear(); return; }
    // up to the last term that stands out of the rounding of the fit (the level of its
    // last terms); M if it has not converged to 1e-13 of the largest order
    auto degree = [&](const std::vector<ld> &c) {
        ld rest = 0;
        int d = M - 1;
        while (d > 0 && rest + std::fabs(c[d]) <= 2e-17L * g00) rest += std::fabs(c[d--]);
        return d >= M - 1 ? M : d;
    };
    std::vector<std::array<int, 4>> at(fits.size());
    for (size_t k = 0; k < fits.size(); ++k) {
        at[k] = {0, -1, 0, -1};
        for (int part = 0; part < 2; ++part) {
            const std::vector<ld> &c = part ? fits[k].im : fits[k].re;
            if (c.empty()) continue;
            const int d = degree(c);
            if (d >= M) { blob.clear(); return; }
            const std::vector<ld> q = cheb_poly(c, d);
            at[k][2 * part] = (int)blob.size();
            at[k][2 * part + 1] = d;
            blob.insert(blob.end(), q.rbegin(), q.rend());
        }
    }
    for (size_t e = 0; e < which.size(); ++e) {
        const std::array<int, 4> v = which[e] >= 0 ? at[which[e]] : std::array<int, 4>{0, -1, 0, -1};
        std::memcpy(&blob[f.dir + 2 * e], v.data(), sizeof(v));
    }
    if (blob.size() > 4096) { blob.clear(); return; }   // 32 KB of shared memory
    f.sym = sym;
    f.rows = np;
    f.cols = nq;
    f.n_img = t.n_img;
    for (int k = 0; k < 9; ++k) f.near_img[k] = t.near_img[k];
    f.t_scale = ts;
    f.sx = 2 * M_PI / a;
    f.sy = 2 * M_PI / b;
    f.i0 = -p0;
    f.j0 = -q0;
    f.kx = kx;
    f.ky = ky;
    f.xs = E / h;
    f.e_mb2 = std::exp(-bb * bb);
    f.E = E;
    f.bb = bb;
    f.reg0 = 4.0 * M_PI * f.e_mb2 * t.reg0_re;
    f.n_blob = (int)blob.size();
}

}  // namespace vie
