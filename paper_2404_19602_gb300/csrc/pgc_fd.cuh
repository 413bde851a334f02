// pgc_fd.cuh -- the inverse of the Fermi-Dirac energy law (Sec. 2) from a table of Taylor
// polynomials, used where every particle needs it at every node (the initial sampling and its
// sensitivities).
//
// With w = eps / kT, m = mu / kT and G(w) = int_w^inf x / (1 + exp(x - m)) dx, the energy of a
// particle with uniform u at a node with band minimum eps0_q solves G(w) = (1 - u) G(w0_q).
// G is common to all nodes, so one table of Y = w^2 as a function of r = G / Gmax (Gmax the
// largest G(w0_q)) serves them: r = (1 - u) G(w0_q) / Gmax.  Y(r) is logarithmic at r = 0 and has
// a square-root branch at r = rs (w = 0, the smallest energy there is); between them it is smooth
// on the scale of the distance to the nearer of the two.  So the variable is v = r below
// rs / 2 and v = rs - r above, each octave of v is cut into 32 intervals (the leading bits of v are
// the interval number), and an interval of relative half-width 1/65 carries the Taylor
// polynomial about its centre, from the recurrences of w w' = -dG (1 + e^(w-m)): order 8, the
// last term folded into the lower ones by its Chebyshev expansion.  Truncation: 65^-8 / 128 of the
// singular part, below the rounding of the FP64 Horner evaluation.
//
// What it costs: one 64-byte row (L1-resident, ~50-100 KB in all) and ~25 FP64 operations per
// particle and node, where the iteration (fd_inverse) takes a 30-step FP32 bisection and about eight
// FP64 evaluations of G (each an exp, two log1p, a division and a 12-term series).  The FP64 pipe of
// this part issues two lanes per clock and SM, and bounds both.  Measured: the sampling of 500 000
// particles at 36 nodes 208 -> 1.6 ms (0.35 ms over the distinct band minima, k_init), of 1e6
// particles at 6 nodes 56.2 -> 0.44 ms, its
// sensitivities at 5e5 x 6 nodes 32.2 -> 0.5 ms; the table itself takes 26 us (a warp per
// block: latency of two FP64 Newton steps).  Error of eps against extended precision: rms
// 3.9e-16 (iteration: 4.1e-16) for eps0 in [0.05, 0.15] eV at eps_F = 0.4 eV, 300 K.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "pgc_device.cuh"

namespace pgc {

constexpr int kFdBits = 5;                       // 32 intervals per octave of v
constexpr int kFdMaxIntervals = 72 << kFdBits;   // the sampler falls back to fd_inverse beyond
constexpr size_t kFdTableBytes = (size_t)kFdMaxIntervals * 8 * sizeof(double);

struct FdInv {
    const double *tab = nullptr;  // [n][8] monomials in t in [-1, 1]; nullptr: no table (fd_inverse)
    double gmax = 0.0, rs = 0.0, split = 0.0, m = 0.0, wtop = 0.0;
    double gzero = 0.0, gmu = 0.0; // G(0) and G(max(m, 0))
    int32_t base0 = 0, base1 = 0; // leading-bit numbers subtracted below and above the split
    int32_t n0 = 0, n = 0;        // intervals below the split, in all
};

// G(w) and E = 1 + exp(w - m) at w >= 0 (Li2 by its Bernoulli series in log1p(exp(-|w - m|))).
__host__ __device__ inline double fd_G(double w, double m, double &E)
{
    const double b = w - m, x = exp(-fabs(b)), l = log1p(x);
    constexpr double c[12] = {(1.0 / 6.0) / 6.0, (-1.0 / 30.0) / 120.0, (1.0 / 42.0) / 5040.0,
                              (-1.0 / 30.0) / 362880.0, (5.0 / 66.0) / 39916800.0,
                              (-691.0 / 2730.0) / 6227020800.0, (7.0 / 6.0) / 1307674368000.0,
                              (-3617.0 / 510.0) / 355687428096000.0, (43867.0 / 798.0) / 121645100408832000.0,
                              (-174611.0 / 330.0) / 51090942171709440000.0,
                              (854513.0 / 138.0) / 25852016738884976640000.0,
                              (-236364091.0 / 2730.0) / 15511210043330985984000000.0};
    const double t2 = l * l, t4 = t2 * t2, t8 = t4 * t4;   // Estrin's scheme: a shorter chain than Horner's
    const double p0 = (c[3] * t2 + c[2]) * t4 + (c[1] * t2 + c[0]), p1 = (c[7] * t2 + c[6]) * t4 + (c[5] * t2 + c[4]),
                 p2 = (c[11] * t2 + c[10]) * t4 + (c[9] * t2 + c[8]), p = (p2 * t8 + p1) * t8 + p0;
    const double li = l + 0.25 * t2 + l * t2 * p;   // -Li2(-x)
    if (b >= 0.0) {
        E = 1.0 + 1.0 / x;
        return w * l + li;
    }
    E = 1.0 + x;
    return w * l - b * (m + 0.5 * b) + kPi * kPi / 6.0 - li;
}

// w with G(w) = g, safeguarded Newton on log G from the degenerate (w^2 / 2 = G(0) - g) or the
// Boltzmann limit, first in FP32 to a relative 1e-6, then in FP64 until a step's square is below
// rounding.
__host__ __device__ inline double fd_solve(double g, const FdInv &f)
{
    const double m = f.m;
    double E, lo = 0.0, hi = f.wtop;
    double w;
    if (m > 0.0 && g > f.gmu) w = sqrt(fmax(2.0 * (f.gzero - g), 0.0));
    else {
        const double L = g / (fmax(m, 0.0) + 1.0);
        w = m - (L < 30.0 ? log(expm1(L)) : L);
    }
    if (!(w > lo && w < hi)) w = 0.5 * (lo + hi);
    {   // the FP32 root: two iterations of the slow FP64 functions are left
        const float gf = (float)g, mf = (float)m;
        float x = (float)w;
        for (int it = 0; it < 7; ++it) {
            const float b = x - mf, ex = expf(-fabsf(b)), l = log1pf(ex), l2 = l * l;
            const float li = l + 0.25f * l2 + l * l2 * (0.027777778f + l2 * (-2.7777778e-4f + l2 * 4.7241118e-6f));
            const float G = b >= 0.0f ? x * l + li : x * l - b * (mf + 0.5f * b) + 1.6449341f - li;
            const float E = b >= 0.0f ? 1.0f + 1.0f / ex : 1.0f + ex;
            x = fmaxf(x + log1pf((G - gf) / gf) * G * E / x, 0.5f * x);
        }
        if (x > (float)lo && x < (float)hi) w = (double)x;   // (false for NaN)
    }
    for (int it = 0; it < 80; ++it) {
        const double G = fd_G(w, m, E), d = (G - g) / g;
        if (d == 0.0) break;
        if (d > 0.0) lo = w; else hi = w;
        double wn = w + log1p(d) * G * E / w;
        if (!(wn >= lo && wn <= hi)) wn = 0.5 * (lo + hi);
        const double step = fabs(wn - w);
        w = wn;
        if (step <= 1e-8 * fmin(w, 1.0)) break;   // the next one would be its square (exp(w) sets the scale above 1)
    }
    return w;
}

// The polynomial of interval j.
__host__ __device__ inline void fd_interval(const FdInv &f, int j, double out[8])
{
    const bool left = j < f.n0;
    const int64_t key = (int64_t)j + (left ? f.base0 : f.base1);
    const int64_t mid = (key << (52 - kFdBits)) | ((int64_t)1 << (51 - kFdBits));
    double vc;
    memcpy(&vc, &mid, 8);
    const double h = ldexp(1.0, (int)(key >> kFdBits) - 1023 - kFdBits - 1);
    const double r = left ? vc : f.rs - vc;
    const double D = (left ? h : -h) * f.gmax;   // dG / dt
    double E;
    double w[9], e[9], y[9];
    w[0] = fd_solve(r * f.gmax, f);
    fd_G(w[0], f.m, E);
    e[0] = E;
    y[0] = w[0] * w[0];
    for (int k = 0; k < 8; ++k) {
        double s = -D * e[k];
        y[k + 1] = 2.0 * s / (k + 1);
        for (int i = 1; i <= k; ++i) s -= w[i] * (k - i + 1) * w[k - i + 1];
        w[k + 1] = s / ((k + 1) * w[0]);
        double q = (e[0] - 1.0) * (k + 1) * w[k + 1];
        for (int i = 1; i <= k; ++i) q += e[i] * (k - i + 1) * w[k - i + 1];
        e[k + 1] = q / (k + 1);
    }
    // t^8 = 2 t^6 - 5/4 t^4 + 1/4 t^2 - 1/128 + T_8 / 128
    y[6] += 2.0 * y[8];
    y[4] -= 1.25 * y[8];
    y[2] += 0.25 * y[8];
    y[0] -= y[8] * 0.0078125;
    for (int k = 0; k < 8; ++k) out[k] = y[k];
}

// Y = (eps / kT)^2 at r in (0, 1]; with GRAD also E = 1 + exp((eps - mu) / kT), from dY/dG = -2 E.
template <bool GRAD>
__host__ __device__ __forceinline__ double fd_Y(const FdInv &f, double r, double *E)
{
    const bool left = r < f.split;
    const double v = left ? r : f.rs - r;
    int64_t bits;
    memcpy(&bits, &v, 8);
    const int hi = (int)(bits >> 32);
    int j = (hi >> (20 - kFdBits)) - (left ? f.base0 : f.base1);
    j = j < 0 ? 0 : (j >= f.n ? f.n - 1 : j);
    const int64_t cb = (int64_t)((hi & ~((1 << (20 - kFdBits)) - 1)) | (1 << (19 - kFdBits))) << 32;
    const int64_t sb = (int64_t)(((2046 + kFdBits + 1) << 20) - (hi & 0x7ff00000)) << 32;
    double vc, sc;
    memcpy(&vc, &cb, 8);
    memcpy(&sc, &sb, 8);
    const double t = (v - vc) * sc;
    const double2 *row = reinterpret_cast<const double2 *>(f.tab + (size_t)j * 8);
    const double2 a = row[0], b = row[1], c = row[2], d = row[3];
    if (GRAD) {
        const double dy = ((((((7.0 * d.y) * t + 6.0 * d.x) * t + 5.0 * c.y) * t + 4.0 * c.x) * t + 3.0 * b.y) * t + 2.0 * b.x) * t + a.y;
        *E = (left ? -0.5 : 0.5) * dy * sc / f.gmax;
    }
    return ((((((d.y * t + d.x) * t + c.y) * t + c.x) * t + b.y) * t + b.x) * t + a.y) * t + a.x;
}

// G(w) in extended precision on the host (the targets of the nodes are relative to it).
inline long double fd_G_host(long double w, long double m)
{
    const long double b = w - m, x = std::exp(-std::fabs(b)), l = std::log1p(x), t2 = l * l;
    constexpr long double c[12] = {(1.0L / 6.0L) / 6.0L, (-1.0L / 30.0L) / 120.0L, (1.0L / 42.0L) / 5040.0L,
                                   (-1.0L / 30.0L) / 362880.0L, (5.0L / 66.0L) / 39916800.0L,
                                   (-691.0L / 2730.0L) / 6227020800.0L, (7.0L / 6.0L) / 1307674368000.0L,
                                   (-3617.0L / 510.0L) / 355687428096000.0L, (43867.0L / 798.0L) / 121645100408832000.0L,
                                   (-174611.0L / 330.0L) / 51090942171709440000.0L,
                                   (854513.0L / 138.0L) / 25852016738884976640000.0L,
                                   (-236364091.0L / 2730.0L) / 15511210043330985984000000.0L};
    long double p = c[11];
    for (int k = 10; k >= 0; --k) p = p * t2 + c[k];
    const long double li = l + 0.25L * t2 + l * t2 * p, pi = 3.14159265358979323846264338327950288L;
    return b >= 0.0L ? w * l + li : w * l - b * (m + 0.5L * b) + pi * pi / 6.0L - li;
}

// Groups the nodes by band minimum: eg[0..ng) the distinct ones in order of first appearance, of[q] the
// group of node q, wg[g][h] the weights w[q][h] summed over the group's nodes.
inline int fd_groups(const double *eps0, int Q, const double *w, int P, double *eg, double *wg, int *of)
{
    int ng = 0;
    for (int q = 0; q < Q; ++q) {
        int g = 0;
        while (g < ng && eg[g] != eps0[q]) ++g;
        if (g == ng) {
            eg[ng++] = eps0[q];
            for (int h = 0; h < P; ++h) wg[g * P + h] = 0.0;
        }
        of[q] = g;
        for (int h = 0; h < P; ++h) wg[g * P + h] += w[q * P + h];
    }
    return ng;
}

// The table's layout for band minima eps0[0..Q); ratio[q] = G(w0_q) / Gmax.  Leaves tab null (no
// table) when the range of r over the nodes needs more intervals than there is room for.
inline FdInv fd_plan(const double *eps0, int Q, double mu, double kT, double *ratio)
{
    FdInv f;
    f.m = mu / kT;
    const long double m = (long double)mu / kT;
    std::vector<long double> g(Q);
    long double gmax = 0.0L, gmin = INFINITY;
    double w0max = 0.0;
    for (int q = 0; q < Q; ++q) {
        g[q] = fd_G_host((long double)eps0[q] / kT, m);
        gmax = std::max(gmax, g[q]);
        gmin = std::min(gmin, g[q]);
        w0max = std::max(w0max, eps0[q] / kT);
    }
    if (!(gmin > 1e-200L) || !std::isfinite((double)gmax)) return f;
    for (int q = 0; q < Q; ++q) ratio[q] = (double)(g[q] / gmax);
    f.gmax = (double)gmax;
    f.wtop = std::max(f.m, w0max) + 80.0;
    const long double gzero = fd_G_host(0.0L, m);
    f.gzero = (double)gzero;
    f.gmu = m > 0.0L ? (double)fd_G_host(m, m) : f.gzero;
    f.rs = (double)std::max(gzero / gmax, 1.0L);
    f.split = 0.5 * f.rs;
    auto key = [](double v) { int64_t b; memcpy(&b, &v, 8); return (int64_t)(b >> (52 - kFdBits)); };
    const double u0 = 0x1p-24;   // u is an odd multiple of 2^-24
    const int64_t a = key((double)(0.5 * u0 * gmin / gmax)), b = key(std::min(f.split, 1.0));
    f.base0 = (int32_t)a;
    f.n0 = (int32_t)(b - a + 1);
    f.n = f.n0;
    if (f.split < 1.0) {
        const int64_t c = key(f.rs - (1.0 - 0.5 * u0)), d = key(f.rs - f.split);
        f.base1 = (int32_t)(c - f.n0);
        f.n = (int32_t)(f.n0 + d - c + 1);
    }
    if (f.n > kFdMaxIntervals) f.n = 0;
    return f;
}

// One interval per thread, a warp per block: the solve is one chain of dependent FP64 operations.
static __global__ void __launch_bounds__(32) k_fd_table(const __grid_constant__ FdInv f, double *tab)
{
    const int j = blockIdx.x * 32 + threadIdx.x;
    if (j >= f.n) return;
    double c[8];
    fd_interval(f, j, c);
#pragma unroll
    for (int k = 0; k < 8; ++k) tab[(size_t)j * 8 + k] = c[k];
}

}  // namespace pgc
