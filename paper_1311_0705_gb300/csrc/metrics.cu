// Grid-quality metrics of Sect. 3.2 on the device: the true density rho_t
// of the analytic model at points, the true optical depth tau_t along paths
// by adaptive Gauss-Kronrod quadrature, and the two-pass FP64 statistics
// (mean, population standard deviation) of rho_t - rho_g and tau_t - tau_g.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "hg_internal.h"
#include "scratch.h"

namespace hg {
hg_status cuda_err(cudaError_t e, const char *what);
int sm_count();

struct DevModel {
    int32_t kind;
    int32_t n_table;
    double p[8];
    const double *table;
    double lo[3], hi[3];
};

__device__ double rho_true(const DevModel &m, double x, double y, double z) {
    switch (m.kind) {
    case HG_MODEL_CONST:
        return m.p[0];
    case HG_MODEL_DISK: {
        const double R = sqrt(x * x + y * y);
        return m.p[0] * exp(-(R / m.p[1]) - (fabs(z) / m.p[2]));
    }
    case HG_MODEL_TORUS: {
        const double s = sqrt(x * x + y * y) - m.p[0];
        double v = (s * s + z * z < m.p[1] * m.p[1]) ? m.p[2] : 0.0;
        const float xf = (float)x, yf = (float)y, zf = (float)z;
        for (int j = 0; j < m.n_table; j++) {
            const double *c = m.table + 5 * j;
            // single-precision pre-filter with a wide margin, exact test in FP64
            const float dxf = xf - (float)c[0], dyf = yf - (float)c[1], dzf = zf - (float)c[2];
            const float sf = (float)c[3];
            if (dxf * dxf + dyf * dyf + dzf * dzf > 25.5f * sf * sf + 1e-30f) continue;
            const double dx = x - c[0], dy = y - c[1], dz = z - c[2];
            const double r2 = dx * dx + dy * dy + dz * dz;
            const double s2 = c[3] * c[3];
            if (r2 < 25.0 * s2) v += c[4] * exp(-0.5 * (r2 / s2));
        }
        return v;
    }
    case HG_MODEL_DYADIC: {
        const int L = (int)m.p[0];
        const long long n = 1LL << L;
        const double pos[3] = {x, y, z};
        long long ix[3];
        for (int a = 0; a < 3; a++) {
            long long q = (long long)floor((pos[a] - m.lo[a]) / (m.hi[a] - m.lo[a]) * (double)n);
            ix[a] = q < 0 ? 0 : (q > n - 1 ? n - 1 : q);
        }
        return m.table[ix[0] + n * (ix[1] + n * ix[2])];
    }
    }
    return 0.0;
}

// ------------------------------------------------------------------ disk model
//
// One evaluation of the disk's density through the CUDA math library is two divisions, a square root and an
// exponential: about 50 instructions of the FP64 pipe, which issues one warp instruction per 19 cycles and SM and is
// what both kernels below wait for.  With reciprocals prepared per launch, and the two functions
// written for the arguments that occur (positive normal numbers), it is 24 in the quadrature.

constexpr double kExpLimit = 690.0;  // exp_neg's largest argument

// 2^(j/64), each to the nearest double.
__constant__ double c_exp2_64[64] = {
    0x1.0000000000000p+0, 0x1.02c9a3e778061p+0, 0x1.059b0d3158574p+0, 0x1.0874518759bc8p+0,
    0x1.0b5586cf9890fp+0, 0x1.0e3ec32d3d1a2p+0, 0x1.11301d0125b51p+0, 0x1.1429aaea92de0p+0,
    0x1.172b83c7d517bp+0, 0x1.1a35beb6fcb75p+0, 0x1.1d4873168b9aap+0, 0x1.2063b88628cd6p+0,
    0x1.2387a6e756238p+0, 0x1.26b4565e27cddp+0, 0x1.29e9df51fdee1p+0, 0x1.2d285a6e4030bp+0,
    0x1.306fe0a31b715p+0, 0x1.33c08b26416ffp+0, 0x1.371a7373aa9cbp+0, 0x1.3a7db34e59ff7p+0,
    0x1.3dea64c123422p+0, 0x1.4160a21f72e2ap+0, 0x1.44e086061892dp+0, 0x1.486a2b5c13cd0p+0,
    0x1.4bfdad5362a27p+0, 0x1.4f9b2769d2ca7p+0, 0x1.5342b569d4f82p+0, 0x1.56f4736b527dap+0,
    0x1.5ab07dd485429p+0, 0x1.5e76f15ad2148p+0, 0x1.6247eb03a5585p+0, 0x1.6623882552225p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6dfb23c651a2fp+0, 0x1.71f75e8ec5f74p+0, 0x1.75feb564267c9p+0,
    0x1.7a11473eb0187p+0, 0x1.7e2f336cf4e62p+0, 0x1.82589994cce13p+0, 0x1.868d99b4492edp+0,
    0x1.8ace5422aa0dbp+0, 0x1.8f1ae99157736p+0, 0x1.93737b0cdc5e5p+0, 0x1.97d829fde4e50p+0,
    0x1.9c49182a3f090p+0, 0x1.a0c667b5de565p+0, 0x1.a5503b23e255dp+0, 0x1.a9e6b5579fdbfp+0,
    0x1.ae89f995ad3adp+0, 0x1.b33a2b84f15fbp+0, 0x1.b7f76f2fb5e47p+0, 0x1.bcc1e904bc1d2p+0,
    0x1.c199bdd85529cp+0, 0x1.c67f12e57d14bp+0, 0x1.cb720dcef9069p+0, 0x1.d072d4a07897cp+0,
    0x1.d5818dcfba487p+0, 0x1.da9e603db3285p+0, 0x1.dfc97337b9b5fp+0, 0x1.e502ee78b3ff6p+0,
    0x1.ea4afa2a490dap+0, 0x1.efa1bee615a27p+0, 0x1.f50765b6e4540p+0, 0x1.fa7c1819e90d8p+0,
};
// exp(-s), 0 <= s <= kExpLimit: table-driven (P. T. P. Tang, ACM TOMS 15, 1989), s = -(64 m + j) ln2/64 - r,
// |r| <= ln2/128, the polynomial of exp(r) - 1 cut after r^5 (the next term is below 2^-54).  tab: c_exp2_64,
// in shared memory.
__device__ __forceinline__ double exp_neg(double s, const double *tab) {
    const double big = 6755399441055744.0;  // 1.5 * 2^52: the sum's low bits are the nearest whole number
    const double kd = fma(s, -0x1.71547652b82fep+6, big);
    const int k = __double2loint(kd);
    const double n = kd - big;
    double r = fma(n, -0x1.62e42fefa39efp-7, -s);
    r = fma(n, -0x1.abc9e3b39803fp-62, r);
    double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    p = fma(p, r, 1.0 / 6.0);
    p = fma(p, r, 0.5);
    p = fma(p, r * r, r);
    const double t = tab[k & 63];
    const double v = fma(t, p, t);
    return __hiloint2double(__double2hiint(v) + ((k >> 6) << 20), __double2loint(v));
}

// sqrt(x), x a normal number between 2^-120 and 2^120: a single-precision reciprocal root and Newton
// steps on x - s^2, which fused multiply-adds give without rounding error.  After two steps 7 of 1e6 roots are off by
// one unit in the last place, after three none of 4e7 is (on the host, the reciprocal root off by 2^-22.9 at most).
template <int STEPS>
__device__ __forceinline__ double sqrt_pos(double x) {
    const int hi = __double2hiint(x);
    float y;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(__int_as_float(__funnelshift_l(__double2loint(x), hi - 0x38000000, 3))));
    const int yb = __float_as_int(y);
    const double yd = __hiloint2double((yb >> 3) + 0x38000000, yb << 29);  // y, widened by integer operations
    const double yh = __hiloint2double(__double2hiint(yd) - (1 << 20), __double2loint(yd));
    double s = x * yd;
#pragma unroll
    for (int j = 0; j < STEPS; j++) s = fma(fma(-s, s, x), yh, s);
    return s;
}

// x / h with rh = 1 / h: the quotient's rounding error corrected once.
__device__ __forceinline__ double quotient(double x, double h, double rh) {
    const double q = x * rh;
    return fma(fma(-q, h, x), rh, q);
}

__device__ __forceinline__ void stage_exp_table(double *tab) {
    for (int i = threadIdx.x; i < 64; i += blockDim.x) tab[i] = c_exp2_64[i];
    __syncthreads();
}

// Scale lengths for which the functions above are made.
bool ordinary_disk(const DevModel &m) {
    auto ok = [](double v) { return v >= 0x1p-40 && v <= 0x1p40; };
    return m.kind == HG_MODEL_DISK && ok(m.p[1]) && ok(m.p[2]);
}

__global__ void model_density_kernel(const DevModel m, int64_t n, const double *__restrict__ pts, double *rho) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        rho[i] = rho_true(m, pts[3 * i], pts[3 * i + 1], pts[3 * i + 2]);
}

// The same for an ordinary disk, number for number: the root and the quotients are those of the library's functions, which
// they replace, and the exponential is the library's (exp_neg with the low parts of its table left a norm of errors of 9.2e-17
// against the formula in torch where this one's is 8.3e-17).  1e6 points with location and statistics: 180 us with
// the library's functions throughout, 152 so, 138 with exp_neg.  Points for which the root and the quotients are not made
// take rho_true.
__global__ void __launch_bounds__(256) disk_density_kernel(const DevModel m, double rhR, double rhz, int64_t n,
                                                           const double *__restrict__ pts, double *rho) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double x = pts[3 * i], y = pts[3 * i + 1], z = pts[3 * i + 2];
        const double R2 = x * x + y * y;
        const double s = quotient(sqrt_pos<3>(R2), m.p[1], rhR) + quotient(fabs(z), m.p[2], rhz);
        const bool fast = R2 >= 0x1p-120 && R2 <= 0x1p120 && s <= kExpLimit;
        rho[i] = fast ? m.p[0] * exp(-s) : rho_true(m, x, y, z);
    }
}

// 15-point Kronrod abscissae/weights and the embedded 7-point Gauss weights on [-1, 1].
__constant__ double c_xgk[8] = {0.991455371120812639206854697526329, 0.949107912342758524526189684047851,
                                0.864864423359769072789712788640926, 0.741531185599394439863864773280788,
                                0.586087235467691130294144845693013, 0.405845151377397166906606412076961,
                                0.207784955007898467600689403773245, 0.0};
__constant__ double c_wgk[8] = {0.022935322010529224963732008058970, 0.063092092629978553290700663189204,
                                0.104790010322250183839876322541518, 0.140653259715525918745189590510238,
                                0.169004726639267902826583426598550, 0.190350578064785409913256402421014,
                                0.204432940075298892414161999234649, 0.209482141084727828012999174891714};
__constant__ double c_wg[4] = {0.129484966168869693270611432679082, 0.279705391489276667901467771423780,
                               0.381830050505118944950369775488975, 0.417959183673469387755102040816327};

__device__ __forceinline__ double ray_rho(const DevModel &m, const double *o, const double *k, double t) {
    return rho_true(m, o[0] + k[0] * t, o[1] + k[1] * t, o[2] + k[2] * t);
}

__device__ void gk15(const DevModel &m, const double *o, const double *k, double a, double b, double *res,
                     double *err) {
    const double c = 0.5 * (a + b), h = 0.5 * (b - a);
    const double fc = ray_rho(m, o, k, c);
    double rk = fc * c_wgk[7], rg = fc * c_wg[3];
#pragma unroll
    for (int j = 0; j < 7; j++) {
        const double x = h * c_xgk[j];
        const double f1 = ray_rho(m, o, k, c - x), f2 = ray_rho(m, o, k, c + x);
        rk += c_wgk[j] * (f1 + f2);
        if (j & 1) rg += c_wg[j / 2] * (f1 + f2);
    }
    *res = rk * h;
    *err = fabs((rk - rg) * h);
}

// Adaptive bisection with an explicit stack, left half first (the order of
// a recursive depth-first integrator).
__device__ double adapt(const DevModel &m, const double *o, const double *k, double a, double b, double rtol) {
    constexpr int kStack = 64;
    double sa[kStack], sb[kStack];
    int sd[kStack];
    int top = 0;
    sa[0] = a;
    sb[0] = b;
    sd[0] = 0;
    top = 1;
    double total = 0.0;
    while (top > 0) {
        top--;
        const double x0 = sa[top], x1 = sb[top];
        const int dep = sd[top];
        double r, e;
        gk15(m, o, k, x0, x1, &r, &e);
        if (dep >= 60 || e <= rtol * fabs(r) || e < 1e-300 || !(x1 > x0) || top + 2 > kStack) {
            total += r;
            continue;
        }
        const double xm = 0.5 * (x0 + x1);
        sa[top] = xm;
        sb[top] = x1;
        sd[top] = dep + 1;
        sa[top + 1] = x0;
        sb[top + 1] = xm;
        sd[top + 1] = dep + 1;
        top += 2;
    }
    return total;
}

__device__ __forceinline__ double horner(const double *c, int deg, double t) {
    double v = c[deg];
    for (int j = deg - 1; j >= 0; j--) v = v * t + c[j];
    return v;
}

// Real roots in (a, b) of a polynomial of degree <= 4, from the roots of its
// successive derivatives (each splits the interval into monotone pieces
// that are bisected).
__device__ int poly_roots4(const double *c4, double a, double b, double *roots) {
    double der[5][5];
    for (int j = 0; j <= 4; j++) der[0][j] = c4[j];
    for (int d = 1; d <= 4; d++)
        for (int j = 0; j <= 4 - d; j++) der[d][j] = (j + 1) * der[d - 1][j + 1];
    double crit[6];
    int nc = 0;
    for (int d = 3; d >= 0; d--) {
        const double *c = der[d];
        int deg = 4 - d;
        while (deg > 0 && c[deg] == 0.0) deg--;
        double edges[6];
        int ne = 0;
        edges[ne++] = a;
        for (int j = 0; j < nc; j++) edges[ne++] = crit[j];
        edges[ne++] = b;
        double out[5];
        int nr = 0;
        if (deg >= 1) {
            for (int j = 0; j + 1 < ne; j++) {
                double lo = edges[j], hi = edges[j + 1];
                double flo = horner(c, deg, lo);
                const double fhi = horner(c, deg, hi);
                if (flo == 0.0) {
                    if (lo > a) out[nr++] = lo;
                    continue;
                }
                if ((flo < 0.0) == (fhi < 0.0)) continue;
                for (int it = 0; it < 200; it++) {
                    const double mid = 0.5 * (lo + hi);
                    if (mid <= lo || mid >= hi) break;
                    const double fm = horner(c, deg, mid);
                    if ((fm < 0.0) == (flo < 0.0)) {
                        lo = mid;
                        flo = fm;
                    } else {
                        hi = mid;
                    }
                }
                out[nr++] = 0.5 * (lo + hi);
            }
        }
        nc = nr;
        for (int j = 0; j < nr; j++) crit[j] = out[j];
    }
    for (int j = 0; j < nc; j++) roots[j] = crit[j];
    return nc;
}

constexpr int kMaxBreak = 160;

__device__ __forceinline__ void add_bp(double *bp, int &nb, double t, double L) {
    if (t > 0.0 && t < L && nb < kMaxBreak - 1) bp[nb++] = t;
}

// Integral of the density along one path, piece by piece between its breakpoints.
__device__ double path_integral(const DevModel &m, const double *o, const double *k, double L, double rtol) {
    {
        double bp[kMaxBreak];
        int nb = 0;
        bp[nb++] = 0.0;
        if (m.kind == HG_MODEL_DISK) {
            if (k[2] != 0.0) add_bp(bp, nb, -o[2] / k[2], L);
            const double kk = k[0] * k[0] + k[1] * k[1];
            if (kk > 0.0) add_bp(bp, nb, -(o[0] * k[0] + o[1] * k[1]) / kk, L);
        } else if (m.kind == HG_MODEL_TORUS) {
            const double R = m.p[0], r = m.p[1];
            const double A = k[0] * k[0] + k[1] * k[1] + k[2] * k[2];
            const double B = 2.0 * (o[0] * k[0] + o[1] * k[1] + o[2] * k[2]);
            const double C = o[0] * o[0] + o[1] * o[1] + o[2] * o[2] + R * R - r * r;
            const double D = k[0] * k[0] + k[1] * k[1];
            const double E = 2.0 * (o[0] * k[0] + o[1] * k[1]);
            const double F = o[0] * o[0] + o[1] * o[1];
            const double c4[5] = {C * C - 4.0 * R * R * F, 2.0 * B * C - 4.0 * R * R * E,
                                  B * B + 2.0 * A * C - 4.0 * R * R * D, 2.0 * A * B, A * A};
            double roots[5];
            const int nr = poly_roots4(c4, 0.0, L, roots);
            for (int j = 0; j < nr; j++) add_bp(bp, nb, roots[j], L);
            for (int j = 0; j < m.n_table; j++) {
                const double *cl = m.table + 5 * j;
                const double w0 = o[0] - cl[0], w1 = o[1] - cl[1], w2 = o[2] - cl[2];
                const double b2 = w0 * k[0] + w1 * k[1] + w2 * k[2];
                const double cc = w0 * w0 + w1 * w1 + w2 * w2 - 25.0 * cl[3] * cl[3];
                const double disc = b2 * b2 - A * cc;
                if (disc <= 0.0) continue;
                const double sq = sqrt(disc);
                add_bp(bp, nb, (-b2 - sq) / A, L);
                add_bp(bp, nb, (-b2 + sq) / A, L);
                add_bp(bp, nb, -b2 / A, L);
            }
        } else if (m.kind == HG_MODEL_DYADIC) {
            const long long nn = 1LL << (int)m.p[0];
            for (int a = 0; a < 3; a++) {
                if (k[a] == 0.0) continue;
                for (long long j = 1; j < nn; j++) {
                    const double pl = m.lo[a] + (m.hi[a] - m.lo[a]) * ((double)j / (double)nn);
                    add_bp(bp, nb, (pl - o[a]) / k[a], L);
                }
            }
        }
        bp[nb++] = L;
        // insertion sort (short lists)
        for (int a = 1; a < nb; a++) {
            const double v = bp[a];
            int b = a - 1;
            while (b >= 0 && bp[b] > v) {
                bp[b + 1] = bp[b];
                b--;
            }
            bp[b + 1] = v;
        }
        double tot = 0.0;
        for (int j = 0; j + 1 < nb; j++)
            if (bp[j + 1] > bp[j]) tot += adapt(m, o, k, bp[j], bp[j + 1], rtol);
        return tot;
    }
}

__global__ void model_tau_kernel(const DevModel m, int64_t n, const double *__restrict__ O,
                                 const double *__restrict__ K, const double *__restrict__ len, double kappa,
                                 double rtol, double *tau) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double o[3] = {O[3 * i], O[3 * i + 1], O[3 * i + 2]};
        const double k[3] = {K[3 * i], K[3 * i + 1], K[3 * i + 2]};
        tau[i] = kappa * path_integral(m, o, k, len[i], rtol);
    }
}

// Optical depths through an ordinary disk: the same rule, tolerance and bisection as path_integral, with the
// intervals of a warp's paths in one pool of which every lane takes one at a time.
//
// The bound is the FP64 pipe, which a warp instruction holds for 19 cycles whatever its active lanes.  With a
// path per thread a warp lasted as long as its longest path (17.6 rule evaluations per path on average, 45
// for the longest of 32: the pipe did 2.5 times the work), and an evaluation cost ~100 FP64 instructions.
// A density is evaluated at the point o + k t, with the functions above 24 FP64 instructions and 28 with the rule's sums.
// Roundings that are the same all along the path do not average out over its ~260 densities as the others do: hence the
// reciprocals as sums (two instructions), and not the exponent in units of the scale lengths from the closest approach to the
// axis, sqrt(A u^2 + D2) + |oz + kz t| (four fewer; A and D2 also lose their digits where the square of a nearly vertical
// path's horizontal part underflows).  Mean relative error of 3000 depths against 113-bit arithmetic, h_R 0.25, h_z 0.03:
// 4.33e-16, as with divisions and the host's exp (in those units 6.8e-16; 0.1, 0.3: 1.21, 1.30 and 3.5e-16).  The
// exponential's own rounding does average out.
//
// A pool that is nearly full is worked down one interval at a time, depth first (an interval needs at most
// kMaxDepth entries beyond its own).  The terms of a path are those of path_integral, added in another order: in each
// round pairwise those of the lanes that hold some, in lane order, then to the path's sum.  Which paths a warp takes, and
// so what its pool holds in each round, depends on the path numbers alone: a call repeats itself bit for bit.  (The warps of
// a block took paths from one counter and added with shared-memory atomics before: 1e5 paths, call 1835 us, now 1774; with
// a path per thread and the library's functions 12.5 ms.)
constexpr int kTauWarps = 8, kPool = 256, kSlots = 64, kMaxDepth = 60;
// The scale lengths as the kernel uses them.
struct DiskScale {
    double unit;                  // power of two: h_R unit is between 1 and 2
    double rR, rz, rR_lo, rz_lo;  // 1 / (h_R unit) and 1 / h_z, each as a sum
};
DiskScale disk_scale(const DevModel &m) {
    DiskScale q;
    int e;
    frexp(m.p[1], &e);
    q.unit = ldexp(1.0, 1 - e);
    const double h = m.p[1] * q.unit;
    q.rR = 1.0 / h;
    q.rR_lo = std::fma(-q.rR, h, 1.0) / h;
    q.rz = 1.0 / m.p[2];
    q.rz_lo = std::fma(-q.rz, m.p[2], 1.0) / m.p[2];
    return q;
}
// A path, its horizontal part times DiskScale's unit (exact).
struct DiskPath {
    double o[3], k[3];
    bool ordinary;  // something to integrate, the exponent in exp_neg's range all along
    __device__ __forceinline__ DiskPath(const DiskScale &q, const double *oo, const double *kk, double L) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
            o[a] = a < 2 ? oo[a] * q.unit : oo[a];
            k[a] = a < 2 ? kk[a] * q.unit : kk[a];
        }
        auto s = [&](double t) {
            const double x = fma(k[0], t, o[0]), y = fma(k[1], t, o[1]), z = fma(k[2], t, o[2]);
            return sqrt(x * x + y * y) * q.rR + fabs(z) * q.rz;
        };
        ordinary = L > 0.0 && s(0.0) <= kExpLimit && s(L) <= kExpLimit;  // the exponent is convex: largest at an end
    }
};
struct TauWarp {
    double a[kPool], b[kPool];                       // intervals
    double o[3][kSlots], k[3][kSlots];               // paths under way (DiskPath)
    double acc[kSlots];
    long long path[kSlots];
    int left[kSlots];                                // intervals of the path not yet added (0: the slot is free)
    int meta[kPool];                                 // slot | depth << 8
};

__global__ void __launch_bounds__(32 * kTauWarps, 2) disk_tau_kernel(const DevModel m, const DiskScale q, int64_t n, int64_t share,
                                                                  const double *__restrict__ O,
                                                                  const double *__restrict__ K,
                                                                  const double *__restrict__ len, double kappa,
                                                                  double rtol, double *tau) {
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ double tab[64];
    __shared__ int s_other;  // some of the block's paths are not ordinary
    TauWarp &W = reinterpret_cast<TauWarp *>(raw)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t first = (int64_t)blockIdx.x * share;
    const unsigned count = (unsigned)(first >= n ? 0 : (n - first < share ? n - first : share));
    if (threadIdx.x == 0) s_other = 0;
    for (int i = lane; i < kSlots; i += 32) W.left[i] = 0;
    stage_exp_table(tab);
    int size = 0;         // entries in the pool
    unsigned turn = 0;    // paths this warp has taken (their slots go round): every kTauWarps-th of the block's share
    const unsigned warp = threadIdx.x >> 5;
    const unsigned mine_all = count > warp ? (count - warp + kTauWarps - 1) / kTauWarps : 0;
    for (;;) {
        // ---- paths to fill the pool with
        if (turn < mine_all && size < 32) {
            const int want = __popc(__ballot_sync(0xffffffffu, W.left[(turn + lane) % kSlots] == 0 && lane < 32 - size));
            // slots are reused in turn: only the free ones next in line count
            const unsigned busy = __ballot_sync(0xffffffffu, W.left[(turn + lane) % kSlots] != 0);
            const int free_run = busy ? __ffs(busy) - 1 : 32;
            int take = want < free_run ? want : free_run;
            if ((unsigned)take > mine_all - turn) take = (int)(mine_all - turn);
            const bool mine = lane < take;
            int pieces = 0;
            double cut[4];
            const int slot = (int)((turn + lane) % kSlots);
            if (mine) {
                const int64_t i = first + warp + (int64_t)(turn + lane) * kTauWarps;
                const double o[3] = {O[3 * i], O[3 * i + 1], O[3 * i + 2]};
                const double k[3] = {K[3 * i], K[3 * i + 1], K[3 * i + 2]};
                const double L = len[i];
                const DiskPath P(q, o, k, L);
                if (!P.ordinary) {
                    s_other = 1;
                } else {
                    // pieces between the closest approach to the axis and the midplane
                    const double kk = k[0] * k[0] + k[1] * k[1];
                    double c1 = kk > 0.0 ? -(o[0] * k[0] + o[1] * k[1]) / kk : 0.0, c2 = k[2] != 0.0 ? -o[2] / k[2] : 0.0;
                    if (c2 < c1) {
                        const double c = c1;
                        c1 = c2;
                        c2 = c;
                    }
                    cut[0] = 0.0;
                    if (c1 > 0.0 && c1 < L) cut[++pieces] = c1;
                    if (c2 > 0.0 && c2 < L && c2 > cut[pieces]) cut[++pieces] = c2;
                    cut[++pieces] = L;
#pragma unroll
                    for (int a = 0; a < 3; a++) {
                        W.o[a][slot] = P.o[a];
                        W.k[a][slot] = P.k[a];
                    }
                    W.acc[slot] = 0.0;
                    W.path[slot] = i;
                    W.left[slot] = pieces;
                }
            }
            turn += (unsigned)take;
            int incl = pieces;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += v;
            }
            const int at = size + incl - pieces;
            for (int j = 0; j < pieces; j++) {
                W.a[at + j] = cut[j];
                W.b[at + j] = cut[j + 1];
                W.meta[at + j] = slot;
            }
            size += __shfl_sync(0xffffffffu, incl, 31);
            __syncwarp();
        }
        if (size == 0) {
            if (turn == mine_all) break;
            continue;
        }
        // ---- one interval per lane
        const int pop = size <= kPool - kMaxDepth - 36 ? (size < 32 ? size : 32) : 1;
        const bool on = lane < pop;
        const int at = size - 1 - (on ? lane : 0);
        const double x0 = W.a[at], x1 = W.b[at];
        const int slot = W.meta[at] & 255, depth = W.meta[at] >> 8;
        const double ox = W.o[0][slot], oy = W.o[1][slot], oz = W.o[2][slot];
        const double kx = W.k[0][slot], ky = W.k[1][slot], kz = W.k[2][slot];
        auto f = [&](double t) {
            const double x = fma(kx, t, ox), y = fma(ky, t, oy), z = fabs(fma(kz, t, oz));
            const double R = sqrt_pos<2>(fma(x, x, fma(y, y, 0x1p-118)));  // (on the axis: a normal argument)
            return exp_neg(fma(R, q.rR, fma(z, q.rz, fma(z, q.rz_lo, R * q.rR_lo))), tab);
        };
        const double c = 0.5 * (x0 + x1), h = 0.5 * (x1 - x0);
        const double fc = f(c);
        double rk = fc * c_wgk[7], rg = fc * c_wg[3];
#pragma unroll 1
        for (int j = 0; j < 7; j++) {
            const double x = h * c_xgk[j];
            const double v = f(c - x) + f(c + x);
            rk = fma(c_wgk[j], v, rk);
            if (j & 1) rg = fma(c_wg[j >> 1], v, rg);
        }
        const double r = rk * h, err = fabs((rk - rg) * h);
        const bool halve = on && depth < kMaxDepth && err > rtol * fabs(r) && !(err * fabs(m.p[0]) < 1e-300) && x1 > x0;
        __syncwarp();
        size -= pop;
        const unsigned halves = __ballot_sync(0xffffffffu, halve);
        if (halve) {
            const int p = size + 2 * __popc(halves & ((1u << lane) - 1u));
            W.a[p] = c;
            W.b[p] = x1;
            W.a[p + 1] = x0;
            W.b[p + 1] = c;
            W.meta[p] = W.meta[p + 1] = slot | (depth + 1) << 8;
            atomicAdd(&W.left[slot], 1);
        }
        // the lanes of one path that have a term: sums of pairs until the first of them holds all
        const bool term = on && !halve;
        const unsigned group = __match_any_sync(0xffffffffu, term ? slot : kSlots);
        const bool leads = term && lane == __ffs(group) - 1;
        unsigned later = group & ~((2u << lane) - 1u);  // lanes of the group after this one, that still hold a sum
        int rank = __popc(group & ((1u << lane) - 1u));
        double sum = r;
        while (__any_sync(0xffffffffu, term && later != 0u)) {
            const int next = __ffs(later);
            const double v = __shfl_sync(0xffffffffu, sum, (next - 1) & 31);
            if (term && next) sum += v;
            later &= __ballot_sync(0xffffffffu, (rank & 1) == 0);
            rank >>= 1;
        }
        if (leads) W.acc[slot] += sum;
        size += 2 * __popc(halves);
        __syncwarp();
        if (on && !halve && atomicSub(&W.left[slot], 1) == 1) tau[W.path[slot]] = kappa * (m.p[0] * W.acc[slot]);
        __syncwarp();
    }
    __syncthreads();
    if (!s_other) return;
    for (unsigned j = threadIdx.x; j < count; j += blockDim.x) {
        const int64_t i = first + j;
        const double o[3] = {O[3 * i], O[3 * i + 1], O[3 * i + 2]};
        const double k[3] = {K[3 * i], K[3 * i + 1], K[3 * i + 2]};
        if (!DiskPath(q, o, k, len[i]).ordinary) tau[i] = kappa * path_integral(m, o, k, len[i], rtol);
    }
}

// Deterministic two-pass statistics in three launches: per-block sums of x = a - b; per-block sums of
// (x - mean)^2, every block adding up the first pass's sums for itself; one block for the results.
// 1e6 values: 40 us with a launch of one block after each pass and one chain of additions per thread, now
// 27 (see the FP64 instructions: a serial sum of 8 by every thread of 977 blocks alone took 4 us).
constexpr int kStatBlock = 256;
__device__ __forceinline__ double block_sum(double v, double *sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    if (wid == 0) {
        double s = lane < kStatBlock / 32 ? sh[lane] : 0.0;
        for (int o = kStatBlock / 64; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) sh[kStatBlock / 32] = s;
    }
    __syncthreads();
    return sh[kStatBlock / 32];
}
__device__ __forceinline__ double sum_parts(int nparts, const double *part, double *sh) {
    double s = 0.0;
    for (int i = threadIdx.x; i < nparts; i += kStatBlock) s += part[i];
    return block_sum(s, sh);
}

template <bool SECOND>
__global__ void __launch_bounds__(kStatBlock) diff_partial(int64_t n, const double *__restrict__ a,
                                                           const double *__restrict__ b, int nparts,
                                                           const double *__restrict__ sums, double *part) {
    __shared__ double sh[kStatBlock / 32 + 1];
    const double mu = SECOND ? sum_parts(nparts, sums, sh) / (double)n : 0.0;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    const int64_t step = (int64_t)gridDim.x * kStatBlock;
    for (int64_t i = (int64_t)blockIdx.x * kStatBlock + threadIdx.x; i < n; i += 4 * step) {
        double x[4];
#pragma unroll
        for (int j = 0; j < 4; j++) x[j] = i + j * step < n ? a[i + j * step] - b[i + j * step] : 0.0;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            // (past the end: nothing, whatever the mean is)
            const double y = !SECOND || i + j * step < n ? x[j] - mu : 0.0;
            s[j] = SECOND ? fma(y, y, s[j]) : s[j] + x[j];
        }
    }
    const double t = block_sum((s[0] + s[1]) + (s[2] + s[3]), sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

__global__ void __launch_bounds__(kStatBlock) diff_final(int64_t n, int nparts, const double *sums,
                                                         const double *squares, double *out) {
    __shared__ double sh[kStatBlock / 32 + 1];
    const double s = sum_parts(nparts, sums, sh), q = sum_parts(nparts, squares, sh);
    if (threadIdx.x == 0) {
        out[0] = (double)n;
        out[1] = n ? s / (double)n : 0.0;
        out[2] = n ? sqrt(q / (double)n) : 0.0;
    }
}

}  // namespace hg

struct hg_dmodel {
    hg::DevModel m;
    void *d_table = nullptr;
};

using namespace hg;

extern "C" hg_status hg_load_model(const hg_model *model, hg_dmodel **out) {
    if (!model || !out) { set_error("hg_load_model: null argument"); return HG_EINVAL; }
    *out = nullptr;
    if (model->kind < HG_MODEL_CONST || model->kind > HG_MODEL_DYADIC || model->n_table < 0 ||
        (model->n_table > 0 && !model->table)) {
        set_error("hg_load_model: bad model");
        return HG_EINVAL;
    }
    hg_dmodel *dm = new hg_dmodel();
    dm->m.kind = model->kind;
    dm->m.n_table = model->n_table;
    for (int j = 0; j < 8; j++) dm->m.p[j] = model->p[j];
    for (int a = 0; a < 3; a++) {
        dm->m.lo[a] = model->lo[a];
        dm->m.hi[a] = model->hi[a];
    }
    const size_t per = (model->kind == HG_MODEL_TORUS) ? 5 : 1;
    const size_t bytes = std::max<size_t>(8, (size_t)model->n_table * per * sizeof(double));
    cudaError_t e = device_malloc(&dm->d_table, bytes);
    if (e == cudaSuccess && model->n_table > 0)
        e = cudaMemcpy(dm->d_table, model->table, (size_t)model->n_table * per * sizeof(double),
                       cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        hg_free_model(dm);
        return cuda_err(e, "hg_load_model");
    }
    dm->m.table = static_cast<const double *>(dm->d_table);
    *out = dm;
    return HG_OK;
}

extern "C" void hg_free_model(hg_dmodel *m) {
    if (!m) return;
    if (m->d_table) cudaFree(m->d_table);
    delete m;
}

extern "C" hg_status hg_model_density(const hg_dmodel *m, int64_t n, const double *pts, double *rho,
                                      hg_stream stream) {
    if (!m || n < 0 || (n > 0 && (!pts || !rho))) { set_error("hg_model_density: bad arguments"); return HG_EINVAL; }
    if (n == 0) return HG_OK;
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)sm_count() * 8);
    if (ordinary_disk(m->m))
        disk_density_kernel<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(m->m, 1.0 / m->m.p[1], 1.0 / m->m.p[2],
                                                                               n, pts, rho);
    else
        model_density_kernel<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(m->m, n, pts, rho);
    note_launches(1);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? HG_OK : cuda_err(e, "model density launch");
}

extern "C" hg_status hg_model_tau(const hg_dmodel *m, int64_t n, const double *o, const double *d,
                                  const double *len, double kappa, double rtol, double *tau, hg_stream stream) {
    if (!m || n < 0 || (n > 0 && (!o || !d || !len || !tau)) || !(rtol > 0.0)) {
        set_error("hg_model_tau: bad arguments");
        return HG_EINVAL;
    }
    if (n == 0) return HG_OK;
    if (ordinary_disk(m->m)) {
        // two blocks per SM; each block shares its paths out among its warps
        constexpr size_t smem = kTauWarps * sizeof(TauWarp);
        cudaError_t e = cudaFuncSetAttribute(disk_tau_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return cuda_err(e, "model tau shared memory");
        const int64_t blocks = std::min<int64_t>((n + kTauWarps - 1) / kTauWarps, (int64_t)sm_count() * 2);
        const int64_t share = (n + blocks - 1) / blocks;
        disk_tau_kernel<<<(unsigned)blocks, 32 * kTauWarps, smem, (cudaStream_t)stream>>>(m->m, disk_scale(m->m), n, share, o, d, len,
                                                                                       kappa, rtol, tau);
    } else {
        const int block = 128;
        const int64_t blocks = std::min<int64_t>((n + block - 1) / block, (int64_t)sm_count() * 16);
        model_tau_kernel<<<(unsigned)blocks, block, 0, (cudaStream_t)stream>>>(m->m, n, o, d, len, kappa, rtol, tau);
    }
    note_launches(1);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? HG_OK : cuda_err(e, "model tau launch");
}

extern "C" hg_status hg_diff_stats(int64_t n, const double *a, const double *b, double *out, hg_stream stream) {
    if (n < 0 || !out || (n > 0 && (!a || !b))) { set_error("hg_diff_stats: bad arguments"); return HG_EINVAL; }
    cudaStream_t s = (cudaStream_t)stream;
    const int parts = (int)std::max<int64_t>(
        1, std::min<int64_t>((n + 4 * kStatBlock - 1) / (4 * kStatBlock), (int64_t)sm_count() * 2));
    Scratch scratch;
    cudaError_t e = scratch_get(scratch, 2 * (size_t)parts * sizeof(double), s);
    if (e != cudaSuccess) return cuda_err(e, "diff stats scratch");
    double *part = static_cast<double *>(scratch.p);
    diff_partial<false><<<parts, kStatBlock, 0, s>>>(n, a, b, parts, nullptr, part);
    diff_partial<true><<<parts, kStatBlock, 0, s>>>(n, a, b, parts, part, part + parts);
    diff_final<<<1, kStatBlock, 0, s>>>(n, parts, part, part + parts, out);
    note_launches(3);
    e = cudaGetLastError();
    scratch_put(scratch, s);
    return e == cudaSuccess ? HG_OK : cuda_err(e, "diff stats launch");
}
