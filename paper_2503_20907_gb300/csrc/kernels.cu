// Kernels of the spline x-ray projector: line setup, footprint tables,
// forward projection, adjoint, visited-set listing, line expansion and a
// footprint probe.  The method is that of "Generalized Ray Tracing with Basis
// Functions for Tomographic Projections" (arXiv 2503.20907); see common.cuh
// for the geometry and the table layout.
#include <cfloat>
#include <cmath>

#include "common.cuh"

namespace spx {
namespace {

// Left-anchored B-spline beta^n on [0, n+1] (Sec. III.C, centred beta^n
// shifted by (n+1)/2), piece l on x = l + tau, tau in [0, 1): coefficients of
// tau^0..tau^n, from beta^n(x) = 1/n! sum_k (-1)^k C(n+1,k) (x-k)_+^n.
// Read with lane-dependent l, so it sits in global memory (L1), not in the
// constant bank.
__device__ const float kBPiece[4][4][4] = {
    {{1.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}},
    {{0.f, 1.f, 0.f, 0.f}, {1.f, -1.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}},
    {{0.f, 0.f, 0.5f, 0.f}, {0.5f, 1.f, -1.f, 0.f}, {0.5f, -1.f, 0.5f, 0.f}, {0.f, 0.f, 0.f, 0.f}},
    {{0.f, 0.f, 0.f, 1.f / 6.f}, {1.f / 6.f, 0.5f, 0.5f, -0.5f}, {2.f / 3.f, 0.f, -1.f, 0.5f},
     {1.f / 6.f, -0.5f, 0.5f, -1.f / 6.f}},
};

// Binomial coefficient C(n, k) (exact in float for n < 25); folded to a
// constant wherever its arguments are.
__host__ __device__ constexpr float binomf(int n, int k)
{
    if (k < 0 || k > n) return 0.f;
    float r = 1.f;
    for (int i = 1; i <= k; ++i) r = r * (float)(n - k + i) / (float)i;
    return r;
}

__device__ __forceinline__ float factf(int n)
{
    float r = 1.f;
    for (int i = 2; i <= n; ++i) r *= (float)i;
    return r;
}

// Unit direction (dx, dy) and a point (px, py) of line r, in double.
__device__ void line_geometry(const LinesDev &L, int64_t r, double &dx, double &dy, double &px,
                              double &py)
{
    switch (L.kind) {
    case SP_LINES_THETA_Y: {
        double th = (double)L.theta[r], yy = (double)L.y[r], s, c;
        sincos(th, &s, &c);
        dx = c; dy = s; px = yy * s; py = -yy * c;
        break;
    }
    case SP_LINES_POINTS: {
        double sx = L.src[2 * r], sy = L.src[2 * r + 1];
        double vx = (double)L.dst[2 * r] - sx, vy = (double)L.dst[2 * r + 1] - sy;
        double inv = 1.0 / sqrt(vx * vx + vy * vy);
        dx = vx * inv; dy = vy * inv; px = sx; py = sy;
        break;
    }
    case SP_LINES_PARALLEL: {
        int64_t v = r / L.n_det, j = r - v * L.n_det;
        double s, c;
        sincos((double)L.view[v], &s, &c);
        double yy = (double)L.det0 + (double)j * (double)L.ddet;
        dx = c; dy = s; px = yy * s; py = -yy * c;
        break;
    }
    default: {  // SP_LINES_FAN
        int64_t v = r / L.n_det, j = r - v * L.n_det;
        double sb, cb;
        sincos((double)L.view[v], &sb, &cb);
        double sx = (double)L.dso * cb, sy = (double)L.dso * sb;
        double off = (double)L.det0 + (double)j * (double)L.ddet;
        double ex = -(double)L.dod * cb - off * sb, ey = -(double)L.dod * sb + off * cb;
        double vx = ex - sx, vy = ey - sy;
        double inv = 1.0 / sqrt(vx * vx + vy * vy);
        dx = vx * inv; dy = vy * inv; px = sx; py = sy;
        break;
    }
    }
}

// The footprint parameters a, b as the table uses them.  For degree >= 1 a
// b below kBMin changes phi by less than about 2 kBMin and is taken as the
// Dirac of Prop. 1; degree 0 keeps any representable b (its ramps have slope
// 1/(a b), so dropping b would move mass by O(1) near cell edges).
__device__ __forceinline__ void footprint_ab(int degree, double dx, double dy, float &af, float &bf)
{
    af = (float)fmax(fabs(dx), fabs(dy));
    bf = (float)fmin(fabs(dx), fabs(dy));
    if (bf < (degree == 0 ? 1e-30f : kBMin)) bf = 0.f;
}

__device__ __forceinline__ float two_w_of(int m, float af, float bf)
{
    return (float)((double)m * ((double)af + (double)bf));
}

__device__ __forceinline__ int slots_of(int m, float af, float bf, float two_w)
{
    if (bf == 0.f) return m;
    int K = (int)floorf(two_w / af) + 1;
    return K < 2 * m ? K : 2 * m;
}

// Support of phi_theta in u = y~ + w: its length 2w (float, as the kernels
// compare it), w (double), and the candidate slots K of a row.  B-splines:
// 2w = (n+1)(a+b).  Box-spline: the three box widths b, a, a -+ b add up to
// 2a (sin and cos of equal sign) or 2(a+b) (opposite signs).
__device__ __forceinline__ void support_params(int kdeg, float af, float bf, int mode, float &two_w, double &w,
                                               int &K)
{
    if (mode == kModeBspline) {
        const int m = kdeg + 1;
        two_w = two_w_of(m, af, bf);
        w = 0.5 * m * ((double)af + (double)bf);
        K = slots_of(m, af, bf, two_w);
    } else {
        const double W = (mode == kModeBoxSame) ? 2.0 * (double)af : 2.0 * ((double)af + (double)bf);
        two_w = (float)W;
        w = 0.5 * W;
        const int k = (int)floorf(two_w / af) + 1;
        K = k < 2 * (kdeg + 1) ? k : 2 * (kdeg + 1);
    }
}

__device__ __forceinline__ int footprint_mode(int basis, double dx, double dy)
{
    if (basis != SP_BASIS_BOX3) return kModeBspline;
    return (dx * dy >= 0.0) ? kModeBoxSame : kModeBoxOpp;
}

// Split x into hi + lo with hi carrying `bits` significant bits (1..23).
__device__ __forceinline__ void split_hi_lo(double x, int bits, float &hi, float &lo)
{
    const unsigned unit = 1u << (24 - bits);
    hi = __uint_as_float((__float_as_uint((float)x) + unit / 2) & ~(unit - 1));
    lo = (float)(x - (double)hi);
}

// ------------------------------------------------------------------ setup
// Bound by the FP64 units (2 FMAs per clock and SM): what the records do not
// need in FP64 (the row range, the quotients, integer parts) is not, the row
// range with margins far above FP32's error, and what the lines of a view share
// is computed once per view.  2.2 M parallel lines take 258 us (718 us with the
// range and its five divisions in FP64).
constexpr int kSetupThreads = 128;

// What the lines of one view share, relative to the grid's centre (fan beams:
// the source and the detector's foot point as seen from it).
struct ViewGeo {
    double s, c, px, py, vx, vy;
};

__device__ void view_geometry(const GridDev &g, const LinesDev &L, int64_t v, ViewGeo &V)
{
    sincos((double)L.view[v], &V.s, &V.c);
    if (L.kind == SP_LINES_FAN) {
        const double dist = (double)L.dso + (double)L.dod;
        V.px = (double)L.dso * V.c - (double)g.cx;
        V.py = (double)L.dso * V.s - (double)g.cy;
        V.vx = -dist * V.c;
        V.vy = -dist * V.s;
    } else {
        V.px = (double)g.cy * V.c - (double)g.cx * V.s;   // the offset of the centre's line
    }
}

// Line setup of line r: its record hdr[r] (see LineHdr) and the footprint's
// a, b and kind.  V (parallel and fan beams, else NULL): its view; j: its bin;
// tab: the index of its table.
__device__ __forceinline__ void setup_line(const GridDev &g, const LinesDev &L, int64_t r, LineHdr *hdr, const ViewGeo *V,
                                           int j, int tab, float &af, float &bf, int &mode)
{
    double dx, dy, Yhat;   // direction; ((p - centre) x direction), then over h
    if (L.kind == SP_LINES_PARALLEL) {
        dx = V->c;
        dy = V->s;
        Yhat = (double)L.det0 + (double)j * (double)L.ddet + V->px;
    } else if (L.kind == SP_LINES_FAN) {
        const double off = (double)L.det0 + (double)j * (double)L.ddet;
        const double vx = V->vx - off * V->s, vy = V->vy + off * V->c;
        const double inv = rsqrt(vx * vx + vy * vy);
        dx = vx * inv;
        dy = vy * inv;
        Yhat = V->px * dy - V->py * dx;
    } else {
        double px, py;
        line_geometry(L, r, dx, dy, px, py);
        Yhat = (px - (double)g.cx) * dy - (py - (double)g.cy) * dx;
    }
    if (g.h != 1.f) Yhat /= (double)g.h;
    LineHdr H;
    H.U0_lo = 0.f;
    H.a_corr = 0.f;
    H.tab = tab;
    footprint_ab(g.kdeg, dx, dy, af, bf);
    mode = footprint_mode(g.basis, dx, dy);
    double w;
    support_params(g.kdeg, af, bf, mode, H.two_w, w, H.K);
    const bool vert = fabs(dy) >= fabs(dx);
    const float ic = 0.5f * (float)(g.nx - 1), jc = 0.5f * (float)(g.ny - 1);
    double kap, rho;
    float rc, qc;
    int Nr, Nq;
    if (vert) { kap = -dy; rho = dx; rc = jc; qc = ic; Nr = g.ny; Nq = g.nx; }
    else { kap = dx; rho = -dy; rc = ic; qc = jc; Nr = g.nx; Nq = g.ny; }
    // a line and its reverse are one line, and phi is even: take the direction
    // in which u grows with the column
    if (kap < 0.0) { kap = -kap; rho = -rho; Yhat = -Yhat; }
    const double A = kap;
    // w as the table sees it (support_params, with the table's a and b)
    int flags = vert ? kVert : 0;
    if (g.degree == 0 && (vert ? dx : dy) == 0.0) flags |= kDeg0Axis;

    // Rows whose support run meets the columns [0, Nq): the column of the
    // support centre (u = w) moves linearly with the row.  In FP32: at 16384
    // columns it is off by less than 0.01 column, against a margin of two.
    const float kapf = (float)kap, rhof = (float)rho, wa = (float)w / kapf + 2.f;
    const float lo = -wa, hi = (float)(Nq - 1) + wa;
    const float c0 = qc - ((float)Yhat - rc * rhof) / kapf;   // centre column at row 0
    const float gam = -rhof / kapf;
    int rb = 0, re = 0;
    if (fabsf(gam) < 1e-30f) {
        if (c0 >= lo && c0 <= hi) { rb = 0; re = Nr; }
    } else {
        float t0 = (lo - c0) / gam, t1 = (hi - c0) / gam;
        if (t0 > t1) { const float t = t0; t0 = t1; t1 = t; }
        t0 = fmaxf(floorf(t0) - 1.f, 0.f);
        t1 = fminf(ceilf(t1) + 2.f, (float)Nr);
        if (t1 > t0) { rb = (int)t0; re = (int)t1; }
    }
    if (rb >= re || !(Yhat == Yhat)) {
        H.flags = flags | kEmpty;
        H.U0 = H.rho_hi = H.rho_lo = H.a_hi = H.a_lo = 0.f;
        H.a = af;
        H.r_ref = H.q_ref = H.r_begin = H.r_end = 0;
        hdr[r] = H;
        return;
    }
    const int r_ref = (rb + re) / 2;
    // u at (r_ref, q = 0), then the reference column with U0 in (0, a].
    const double Ur = Yhat + w + (double)((float)r_ref - rc) * rho - (double)qc * kap;
    int qr = (int)floorf(-(float)Ur / kapf) + 1;   // off by one at most
    double U0 = Ur + (double)qr * kap;
    if (U0 <= 0.0) { ++qr; U0 = Ur + (double)qr * kap; }
    else if (U0 > A) { --qr; U0 = Ur + (double)qr * kap; }
    // hi parts exact against |row offset| and |step count|, both < maxc
    const int maxc = (re - rb) + 8;
    const int bits = 23 - (32 - __clz(maxc));
    H.U0 = (float)U0;
    H.U0_lo = (float)(U0 - (double)H.U0);
    split_hi_lo(rho, bits, H.rho_hi, H.rho_lo);
    split_hi_lo(A, bits, H.a_hi, H.a_lo);
    H.a = af;
    H.a_corr = (float)(A - (double)af);
    H.r_ref = r_ref;
    H.q_ref = qr;
    H.r_begin = rb;
    H.r_end = re;
    H.flags = flags;
    hdr[r] = H;
}

// ------------------------------------------------------------------ centre records
// e-th derivative of the centred B-spline beta^n at x2 / 2 (right limit).
__host__ __device__ constexpr double bspline_deriv(int n, int x2, int e)
{
    const int m = n + 1, t2 = x2 + m;   // twice the distance from the support's start
    if (e > n || t2 < 0 || t2 / 2 >= m) return 0.0;
    double sum = 0.0, binom = 1.0;
    for (int k = 0; k <= t2 / 2; ++k) {
        double pw = 1.0;
        for (int i = 1; i <= n - e; ++i) pw = pw * (0.5 * (t2 - 2 * k)) / i;
        sum += ((k & 1) ? -binom : binom) * pw;
        binom = binom * (m - k) / (k + 1);
    }
    return sum;
}

__host__ __device__ constexpr double factorial(int n)
{
    double r = 1.0;
    for (int i = 2; i <= n; ++i) r *= i;
    return r;
}

// The constants of build_center, folded into its code.
template <int N>
struct CenterConst {
    // piece[x2][e][k]: coefficient of (x - x2/2)^k of the e-th derivative of
    // beta^N in the piece around x2/2 (x2 = 0..3)
    float piece[4][N + 1][N + 1] = {};
    // low[j][e][k][r]: weight of the moment mu[k][r] in the e-th derivative at
    // (j + c) a, both signs of k together
    float low[4][N + 1][3][N + 1] = {};
    float rest[4][3][N + 1] = {};   // what its rounding took off low[j][0]
    constexpr CenterConst()
    {
        constexpr int m = N + 1;
        for (int x2 = 0; x2 < 4; ++x2)
            for (int e = 0; e <= N; ++e)
                for (int k = 0; k <= N - e; ++k) piece[x2][e][k] = (float)(bspline_deriv(N, x2, e + k) / factorial(k));
        for (int j = 0; j < 4; ++j)
            for (int e = 0; e <= N; ++e)
                for (int k = 0; k < 3; ++k)
                    for (int r = 0; r <= N - e; ++r) {
                        // beta^(e)(j - k + c - d) = sum_r D d^r, and d -> -d for -k
                        const int c2 = m % 2 == 0 ? 1 : 0;
                        const double sg = (r & 1) ? -1.0 : 1.0;
                        const double up = bspline_deriv(N, 2 * (j - k) + c2, e + r) / factorial(r) * sg;
                        const double dn = bspline_deriv(N, 2 * (j + k) + c2, e + r) / factorial(r);
                        low[j][e][k][r] = (float)(up + dn);
                        if (e == 0) rest[j][k][r] = (float)(up + dn - (double)low[j][e][k][r]);
                    }
    }
};

// e-th derivative of beta^n at x in its polynomial piece around x2 / 2.
template <int N>
__device__ __forceinline__ float bspline_piece(const CenterConst<N> &T, int x2, int e, float x)
{
    const float d = x - 0.5f * (float)x2;
    float r = 0.f;
#pragma unroll
    for (int k = N; k >= 0; --k)
        if (k <= N - e) r = __fmaf_rn(r, d, T.piece[x2][e][k]);
    return r;
}

// Gauss-Legendre rule of N + 1 points on [-1, 1] (exact to degree 2N + 1).
template <int N>
__device__ __forceinline__ void gauss(int i, float &x, float &w)
{
    if constexpr (N == 1) {
        x = i ? 0.577350269189626f : -0.577350269189626f;
        w = 1.f;
    } else if constexpr (N == 2) {
        x = i == 0 ? -0.774596669241483f : i == 1 ? 0.f : 0.774596669241483f;
        w = i == 1 ? 8.f / 9.f : 5.f / 9.f;
    } else {
        x = i == 0 ? -0.861136311594053f : i == 1 ? -0.339981043584856f : i == 2 ? 0.339981043584856f : 0.861136311594053f;
        w = (i == 0 || i == 3) ? 0.347854845137454f : 0.652145154862546f;
    }
}

// The centre record (common.cuh) of a direction with parameters a >= b, degree
// N, m = N + 1, by one thread.  With y the offset from the footprint's centre,
//   phi(y) = 1/a int beta(s) beta((y - b s)/a) ds,
// so at y = (j + c) a, c = 1/2 (m even) or 0 (m odd), the second factor and its
// first n derivatives are polynomials in d = b s/a - k on the pieces
// |d| < 1/2, the same pieces for every j: the derivatives 0..n are sums of the
// moments mu[k][r] = int beta(s) d^r ds with rational weights (all terms of one
// size: no cancellation).  The derivatives n + e + 1 are
//   a^-m sum_p (-1)^p C(m, p) (d/dy)^e beta_b((j + c + m/2 - p) a),
// beta_b the B-spline of knot spacing b, at most two of whose arguments,
// +- a/2 and +- 3a/2, lie in its support.  The knots follow the same comparisons
// as the pieces taken there.
template <int N>
__device__ void build_center(float a, float b, float *__restrict__ out)
{
    constexpr int m = N + 1;
    constexpr CenterConst<N> T;
    const float ia = 1.0f / a, tau = b * ia;
    const float t1 = 0.5f / tau, t2 = 1.5f / tau;   // where b s/a passes 1/2 and 3/2 (infinite at b = 0)
    float mu[3][N + 1];   // s >= 0
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int r = 0; r <= N; ++r) mu[k][r] = 0.f;
    // pieces of beta^N(s), s >= 0: around x2 / 2, [lo, hi]
    constexpr int kPieces = (m + 1) / 2;
#pragma unroll
    for (int p = 0; p < kPieces; ++p) {
        const int x2 = (m % 2 == 0) ? 2 * p + 1 : 2 * p;
        const float lo = fmaxf(0.5f * (float)(x2 - 1), 0.f), hi = 0.5f * (float)(x2 + 1);
        const int k0 = (lo >= t1) + (lo >= t2);
        const float cut = fminf(fmaxf(k0 == 0 ? t1 : k0 == 1 ? t2 : hi, lo), hi);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float l0 = h ? cut : lo, l1 = h ? hi : cut;
            const float hw = 0.5f * (l1 - l0), mid = 0.5f * (l1 + l0);
            const int k = k0 + h;
#pragma unroll
            for (int i = 0; i <= N; ++i) {
                float x, w;
                gauss<N>(i, x, w);
                const float s = __fmaf_rn(hw, x, mid);
                float g = w * hw * bspline_piece<N>(T, x2, 0, s);
                const float d = __fmaf_rn(tau, s, -(float)k);
#pragma unroll
                for (int r = 0; r <= N; ++r) {
#pragma unroll
                    for (int kk = 0; kk < 3; ++kk)
                        if (k == kk) mu[kk][r] += g;
                    g *= d;
                }
            }
        }
    }
    // The rounding of constants, and of moments that are the same for many
    // directions, shifts all footprints alike: 5e-8 of every line at degree 2 and
    // 3e-8 at degree 3, which a backprojection of small residuals sums up over the
    // views.  The values at (j + c) a (e = 0 below) therefore take what the moments
    // lack of their sum 1/2, and what the weights lost, in a second term, and the
    // terms that are alike last: mean of the mass over directions off by less than
    // 1e-9.
    const float lack = ((0.5f - mu[0][0]) - mu[1][0]) - mu[2][0];
    // beta_b's derivatives (times b^(1+e)) at a/2 and 3a/2, in the pieces that
    // the comparisons choose
    float H0[N + 1], H1[N + 1];
    {
        const bool in0 = N == 2 ? 3.f * b >= a : 2.f * b >= a;
        const bool in1 = N == 3 && 4.f * b >= a;   // one piece further out
        const float x = 0.5f * a / b;
#pragma unroll
        for (int e = 0; e <= N; ++e) {
            float v = 0.f;
            if (in0) v = bspline_piece<N>(T, N == 2 ? 2 : 1, e, x);
            else if (in1) v = bspline_piece<N>(T, 3, e, x);
            H0[e] = v;
            H1[e] = (N == 3 && 4.f * b >= 3.f * a) ? bspline_piece<N>(T, 3, e, 3.f * x) : 0.f;
        }
    }
    const float ib = b > 0.f ? 1.0f / b : 0.f;
    float iam = ia;
#pragma unroll
    for (int k = 1; k < m; ++k) iam *= ia;
    float4 *o4 = reinterpret_cast<float4 *>(out);
    constexpr int J = N == 1 ? 2 : 4;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float c[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) c[k] = 0.f;
        if (j < J) {
            float sc = ia;   // a^-(1+e)
#pragma unroll
            for (int e = 0; e <= N; ++e) {
                float acc = 0.f, rest = e == 0 ? T.low[j][0][0][0] * lack : 0.f;
#pragma unroll
                for (int k = 2; k >= 0; --k)
#pragma unroll
                    for (int r = N; r >= 0; --r)
                        if (e == 0 && T.rest[j][k][r] != 0.f) rest = __fmaf_rn(T.rest[j][k][r], mu[k][r], rest);
#pragma unroll
                for (int k = 2; k >= 0; --k)
#pragma unroll
                    for (int r = N; r >= 0; --r)
                        if (T.low[j][e][k][r] != 0.f) acc = __fmaf_rn(T.low[j][e][k][r], mu[k][r], acc);
                constexpr float kInvFact[4] = {1.f, 1.f, 0.5f, 1.f / 6.f};
                c[e] = e == 0 ? __fmaf_rn(acc, sc, rest * sc) : acc * sc * kInvFact[e];
                sc *= ia;
            }
            float sb = iam * ib;   // a^-m b^-(1+e)
#pragma unroll
            for (int e = 0; e <= N; ++e) {
                float acc = 0.f;
#pragma unroll
                for (int p = 0; p <= m; ++p) {
                    const int i2 = 2 * j + (m % 2 == 0 ? 1 : 0) + m - 2 * p;   // twice the argument over a
                    const float w = binomf(m, p) * ((p & 1) ? -1.f : 1.f) * ((i2 < 0 && (e & 1)) ? -1.f : 1.f);
                    if (i2 == 1 || i2 == -1) acc = __fmaf_rn(w, H0[e], acc);
                    if (N == 3 && (i2 == 3 || i2 == -3)) acc = __fmaf_rn(w, H1[e], acc);
                }
                constexpr float kInvFact[8] = {1.f, 1.f, 1.f / 2.f, 1.f / 6.f, 1.f / 24.f, 1.f / 120.f, 1.f / 720.f, 1.f / 5040.f};
                c[m + e] = acc * sb * kInvFact[m + e];
                sb *= ib;
            }
        }
        o4[2 * j] = make_float4(c[0], c[1], c[2], c[3]);
        o4[2 * j + 1] = make_float4(c[4], c[5], c[6], c[7]);
    }
    // knots: 1 / ((2n+1)! (a b)^(n+1)), none at b = 0 (the Dirac of Prop. 1)
    float ab = a * b, kap = ab;
#pragma unroll
    for (int k = 1; k < m; ++k) kap *= ab;
    constexpr float kInvFact = N == 3 ? 1.f / 5040.f : N == 2 ? 1.f / 120.f : 1.f / 6.f;
    kap = b > 0.f ? kInvFact / kap : 0.f;
    // knot q, at +beta of the candidates kk = p - off, p = 0..m
    auto knot = [&](int slot, int q, int off, float beta) {
        out[kCenterBeta + slot] = beta;
        const float kq = kap * binomf(m, q) * ((q & 1) ? -1.f : 1.f);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int pp = j + off, pm = (m % 2 == 0 ? -j - 1 : -j) + off;
            const float jp = binomf(m, pp) * ((pp & 1) ? -0.5f : 0.5f), jm = binomf(m, pm) * ((pm & 1) ? -0.5f : 0.5f);
            out[kCenterJump + 8 * slot + 2 * j] = (jp + jm) * kq;
            out[kCenterJump + 8 * slot + 2 * j + 1] = (jp - jm) * kq;
        }
    };
    if constexpr (N == 3) {
        if (2.f * b >= a) knot(0, 3, 2, b - 0.5f * a);
        else knot(0, 1, 3, 0.5f * a - b);
        if (2.f * b < a) {
            if (4.f * b >= a) knot(1, 4, 2, 2.f * b - 0.5f * a);
            else knot(1, 0, 3, 0.5f * a - 2.f * b);
        } else {
            if (4.f * b >= 3.f * a) knot(1, 4, 1, 2.f * b - 1.5f * a);
            else knot(1, 0, 4, 1.5f * a - 2.f * b);
        }
    } else if constexpr (N == 2) {
        knot(0, 1, 2, 0.5f * (a - b));
        if (3.f * b <= 2.f * a) {
            if (3.f * b >= a) knot(1, 3, 1, 1.5f * b - 0.5f * a);
            else knot(1, 0, 2, 0.5f * a - 1.5f * b);
        } else {
            knot(1, 0, 3, 1.5f * (a - b));
        }
    } else {
        if (2.f * b >= a) knot(0, 2, 1, b - 0.5f * a);
        else knot(0, 0, 2, 0.5f * a - b);
        kap = 0.f;
        knot(1, 0, 0, a);   // none
    }
    out[kCenterA] = a;
    out[kCenterB] = b;
}

// Line records, and per table (one per line, one per view for parallel beams):
// with tabs its head (a, b and the footprint's kind, from which tables_kernel
// builds the rest), with rec (degree 1..3 B-splines) its centre record.
template <int DEG>
__global__ void __launch_bounds__(kSetupThreads) setup_kernel(GridDev g, LinesDev L, LineHdr *hdr, float *tabs, float *rec,
                                                              int64_t M)
{
    chain_begin();
    const int64_t r0 = (int64_t)blockIdx.x * kSetupThreads, r = r0 + threadIdx.x;
    // parallel and fan beams: the views of the block's lines (at most one per thread)
    __shared__ ViewGeo geo[kSetupThreads];
    const bool views = (L.kind == SP_LINES_PARALLEL || L.kind == SP_LINES_FAN);
    int64_t v0 = 0;
    int k = 0, j = 0;   // this line's view, from v0 on, and bin
    if (views) {
        v0 = r0 / L.n_det;
        const unsigned b0 = (unsigned)(r0 - v0 * L.n_det), n = (unsigned)L.n_det;   // the first line's bin
        const unsigned last = b0 + (unsigned)(min((int64_t)kSetupThreads, M - r0) - 1);
        if (threadIdx.x <= last / n) view_geometry(g, L, v0 + threadIdx.x, geo[threadIdx.x]);
        k = (int)((b0 + threadIdx.x) / n);
        j = (int)((b0 + threadIdx.x) - (unsigned)k * n);
        __syncthreads();
    }
    if (r >= M) return;
    float af, bf;
    int mode;
    const int64_t tab = (L.kind == SP_LINES_PARALLEL) ? v0 + k : r;
    setup_line(g, L, r, hdr, views ? geo + k : nullptr, j, (int)tab, af, bf, mode);
    if (L.kind != SP_LINES_PARALLEL || j == 0) {
        if (tabs) {
            tabs[tab * kTabFloats + kTabA] = af;
            tabs[tab * kTabFloats + kTabB] = bf;
            tabs[tab * kTabFloats + kTabMode] = (float)mode;
        }
        if constexpr (DEG >= 1)
            if (rec) build_center<DEG>(af, bf, rec + tab * kCenterFloats);
    }
}

// ------------------------------------------------------------------ tables
// Derivatives e = 0..N of B-spline piece l at tau, times b^-(1+e).
template <int N>
__device__ __forceinline__ void bspline_piece_derivs(int l, float tau, float binv, float *D)
{
    float sc = binv;
#pragma unroll
    for (int e = 0; e <= N; ++e) {
        float acc = 0.f;
#pragma unroll
        for (int k = N; k >= e; --k) {
            float ff = 1.f;   // k!/(k-e)!
#pragma unroll
            for (int t = 0; t < e; ++t) ff *= (float)(k - t);
            acc = acc * tau + kBPiece[N][l][k] * ff;
        }
        D[e] = acc * sc;
        sc *= binv;
    }
}

// Sign of (pa + qb) - (p2 a + q2 b) + extra, formed from the integer
// differences so that it is accurate whatever the size of a and b.
__device__ __forceinline__ float sym_diff(int dp, int dq, float a, float b, float extra)
{
    return __fmaf_rn((float)dp, a, __fmaf_rn((float)dq, b, extra));
}

// Slot l of a B-spline table's head, s its interval end: what the line setup left
// there for the builder stays, so that a table can be built again from its head.
__device__ __forceinline__ float head_slot(int l, float a, float b, float s)
{
    return l == kTabA ? a : l == kTabB ? b : l == kTabMode ? (float)kModeBspline : s;
}

// Build the footprint table of one direction (see common.cuh), degree N, on
// one half-warp: l is the lane within the half (0..15) and gmask the half's
// lanes.  sm is the half's shared scratch of kBuildScratch floats; the table
// is assembled there and then written to out (if out is not NULL).  Every
// phase fits 16 lanes (at most 15 pieces start before the centre of the
// support; 25 breakpoints are ranked two per lane), so a warp builds two
// tables at once.
constexpr int kBuildScratch = kTabFloats + 32 + 32 + 25 * 8 + 8 + 8 + 8;
constexpr int kTabWarps = 8;

template <int N>
__device__ void build_table_half(float a, float b, float *out, float *sm, int l, unsigned gmask)
{
    constexpr int n = N, m = N + 1, nc = 2 * N + 2;
    constexpr int G = 16;
    float *tab = sm;
    float *bv = tab + kTabFloats;                       // sorted breakpoint values
    int *bpq = reinterpret_cast<int *>(bv + 32);        // and their (p, q), p | q << 8
    float *P = reinterpret_cast<float *>(bpq + 32);     // piece polynomials [25][8]
    float *sv = P + 25 * 8;                             // sorted u_0 interval ends
    int *sq = reinterpret_cast<int *>(sv + 8);
    int *sf = sq + 8;
    for (int k = l; k < kTabFloats / 4; k += G) reinterpret_cast<float4 *>(tab)[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp(gmask);
    const float two_w = two_w_of(m, a, b);
    const float ainv = 1.0f / a;
    if (b == 0.f) {
        // Dirac factor (Prop. 1): phi(u) = beta^n(u/a)/a on the a-knots.
        if (l < kTabHead) tab[l] = head_slot(l, a, 0.f, l < m ? a : FLT_MAX);
        if (l < m * (n + 1)) {
            const int i = l / (n + 1), e = l - i * (n + 1);
            float sc = ainv;
            for (int k = 0; k < e; ++k) sc *= ainv;
            tab[tab_poly(0, i) + e] = kBPiece[n][i][e] * sc;
        }
    } else {
        // breakpoints p a + q b, ranked (ties by p, then q) by their exact values in
        // units of 2^-47 (a and b >= kBMin > 2^-24 are multiples): rounded values of
        // breakpoints less than an ulp apart, as at b/a = 1/2, came in the wrong
        // order, and the piece that then stood last lacked a derivative's jump
        constexpr int NB = (m + 1) * (m + 1);
        constexpr int NI = (NB + G - 1) / G;   // breakpoints per lane: l and l + 16
        constexpr float kUnit = 140737488355328.f;   // 2^47
        const long long A = __float2ll_rn(a * kUnit), B = __float2ll_rn(b * kUnit);
        // all values in the scratch of the pieces (filled later), read back
        // two at a time; ties go by index, which orders (p, q) lexicographically
        long long *vr = reinterpret_cast<long long *>(P);
        int p[NI], q[NI];
        long long v[NI];
#pragma unroll
        for (int it = 0; it < NI; ++it) {
            const int idx = l + G * it;
            p[it] = 0; q[it] = 0; v[it] = 0;
            if (idx < NB) {
                p[it] = idx / (m + 1);
                q[it] = idx - p[it] * (m + 1);
                v[it] = p[it] * A + q[it] * B;
                vr[idx] = v[it];
            }
        }
        __syncwarp(gmask);
        int rank[NI];
#pragma unroll
        for (int it = 0; it < NI; ++it) rank[it] = 0;
#pragma unroll
        for (int j2 = 0; j2 < (NB + 1) / 2; ++j2) {
            const longlong2 w2 = reinterpret_cast<const longlong2 *>(vr)[j2];
            const long long vj[2] = {w2.x, w2.y};
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int j = 2 * j2 + u;
                if (j < NB)
#pragma unroll
                    for (int it = 0; it < NI; ++it)
                        rank[it] += (vj[u] < v[it]) || (vj[u] == v[it] && j < l + G * it);
            }
        }
        __syncwarp(gmask);
#pragma unroll
        for (int it = 0; it < NI; ++it)
            if (l + G * it < NB) bpq[rank[it]] = p[it] | (q[it] << 8);
        __syncwarp(gmask);
        // pieces that start at or before the centre w: the leading sorted run
        // (the last breakpoint, at 2w, is always beyond it)
        int mp = 0, mq = 0;
        unsigned outside = 0u;
#pragma unroll
        for (int it = 0; it < NI; ++it) {
            const int idx = l + G * it;
            int ip = 0, iq = 0;
            if (idx < NB) { ip = bpq[idx] & 255; iq = bpq[idx] >> 8; }
            if (it == 0) { mp = ip; mq = iq; }
            const unsigned bal = __ballot_sync(gmask, idx >= NB || sym_diff(2 * ip - m, 2 * iq - m, a, b, 0.f) > 0.f);
            outside |= ((bal >> (threadIdx.x & 16)) & 0xFFFFu) << (G * it);
        }
        int nh = __ffs(outside) - 1;
        if (nh < 1) nh = 1;
        // derivatives n+1..2n+1 of every piece directly (right-sided at its start)
        const float binv = 1.0f / b;
        float am = 1.f;
#pragma unroll
        for (int k = 0; k < m; ++k) am *= ainv;
        if (l < nh) {
            const int p0 = mp, q0 = mq;
            float hi[n + 1];
#pragma unroll
            for (int e = 0; e <= n; ++e) hi[e] = 0.f;
#pragma unroll
            for (int pp = 0; pp <= m; ++pp) {
                int piece;
                float tau;
                if (pp == p0) {
                    if (q0 >= m) continue;
                    piece = q0; tau = 0.f;
                } else {
                    // the piece of the B-spline of b that starts at or before this
                    // breakpoint, by the exact values as in the ranking
                    long long left = (p0 - pp) * A + q0 * B;
                    if (left < 0) continue;
                    piece = 0;
#pragma unroll
                    for (int k = 0; k < m; ++k)
                        if (left >= B) { left -= B; ++piece; }
                    if (piece >= m) continue;
                    tau = __fdiv_rn((float)left, (float)B);
                }
                float D[n + 1];
                bspline_piece_derivs<n>(piece, tau, binv, D);
                const float wp = binomf(m, pp) * ((pp & 1) ? -1.f : 1.f);
#pragma unroll
                for (int e = 0; e <= n; ++e) hi[e] = __fmaf_rn(wp, D[e], hi[e]);
            }
#pragma unroll
            for (int e = 0; e <= n; ++e) P[l * 8 + n + 1 + e] = hi[e] * am / factf(n + 1 + e);
            if (l == 0)
#pragma unroll
                for (int d = 0; d <= n; ++d) P[d] = 0.f;
        }
        __syncwarp(gmask);
        // derivatives 0..n carried from piece to piece (lane d computes coefficient d);
        // C(k, l) held in registers (a lane-dependent index into a constant
        // table would serialise the warp's constant loads)
        float cb[nc];
#pragma unroll
        for (int k = 0; k < nc; ++k) {
            float c = 0.f;
#pragma unroll
            for (int d = 0; d <= n; ++d)
                if (l == d) c = binomf(k, d);
            cb[k] = c;
        }
        // lane pi holds the length of piece pi - 1 (the step to piece pi); the
        // low coefficients of the previous piece travel in registers (lane d
        // holds coefficient d), the top ones come from the scratch
        float dlv = 0.f;
        if (l >= 1 && l < nh) {
            const int cur = bpq[l], prev = bpq[l - 1];
            dlv = sym_diff((cur & 255) - (prev & 255), (cur >> 8) - (prev >> 8), a, b, 0.f);
        }
        float low = 0.f;   // piece 0 starts the support: its coefficients 0..n vanish
        for (int pi = 1; pi < nh; ++pi) {
            const float dl = __shfl_sync(gmask, dlv, pi, G);
            float c[nc];
#pragma unroll
            for (int k = 0; k <= n; ++k) c[k] = __shfl_sync(gmask, low, k, G);
#pragma unroll
            for (int k = n + 1; k < nc; ++k) c[k] = P[(pi - 1) * 8 + k];
            float sacc = 0.f;
#pragma unroll
            for (int k = nc - 1; k >= 0; --k)
                if (k >= l) sacc = __fmaf_rn(sacc, dl, cb[k] * c[k]);
            low = sacc;
            if (l <= n) P[pi * 8 + l] = sacc;
        }
        __syncwarp(gmask);
        // u_0 interval ends s_q = (q b) mod a in (0, a], sorted (stable in q)
        float rq = 0.f;
        int fq = 0;
        if (l >= 1 && l <= m) {
            fq = (int)floorf((float)l * b * ainv);
            rq = __fmaf_rn((float)(-fq), a, (float)l * b);
            if (rq <= 0.f) { fq -= 1; rq = __fmaf_rn((float)(-fq), a, (float)l * b); }
            else if (rq > a) { fq += 1; rq = __fmaf_rn((float)(-fq), a, (float)l * b); }
        }
        int srank = 1;
#pragma unroll
        for (int j = 1; j <= m; ++j) {
            const float rj = __shfl_sync(gmask, rq, j, G);
            srank += (j < l) ? (rj <= rq) : (j > l ? (rj < rq) : 0);
        }
        if (l >= 1 && l <= m) { sv[srank] = rq; sq[srank] = l; sf[srank] = fq; }
        if (l == 0) { sv[0] = 0.f; sq[0] = 0; sf[0] = 0; }
        __syncwarp(gmask);
        if (l < kTabHead) tab[l] = head_slot(l, a, b, l < m ? sv[l + 1] : FLT_MAX);
        const int K = slots_of(m, a, b, two_w);
        // entry e = (sigma, candidate) = (e / 8, e % 8), two sigmas per pass
#pragma unroll
        for (int pass = 0; pass < ((m + 1) * 8 + G - 1) / G; ++pass) {
            const int e = l + G * pass;
            const int sg = e >> 3, i = e & 7;
            if (sg > m || i >= K) continue;
            const float hw = 0.5f * (((sg < m) ? sv[sg + 1] : a) - sv[sg]);
            // interval start u_lo = (i - f) a + q b; midpoint u_lo + hw
            const int pl = i - sf[sg], ql = sq[sg];
            if (sym_diff(pl - m, ql - m, a, b, hw) >= 0.f) continue;          // beyond 2w
            const bool mirror = sym_diff(2 * pl - m, 2 * ql - m, a, b, 2.f * hw) > 0.f;
            // last piece (of the nh sorted ones) starting at or before the
            // midpoint of the entry (mirrored into the left half if needed):
            // binary search, the predicate being monotone in the piece index
            const int pq = mirror ? m - pl : pl, qq = mirror ? m - ql : ql;
            const float hs = mirror ? -hw : hw;
            int pi = 0;
#pragma unroll
            for (int st = 16; st > 0; st >>= 1) {
                const int c = pi + st;
                if (c < nh && sym_diff(pq - (bpq[c] & 255), qq - (bpq[c] >> 8), a, b, hs) >= 0.f) pi = c;
            }
            const int bp = bpq[pi] & 255, bq = bpq[pi] >> 8;
            const float X = mirror ? sym_diff(m - pl - bp, m - ql - bq, a, b, 0.f) : sym_diff(pl - bp, ql - bq, a, b, 0.f);
            float *T = tab + tab_poly(sg, i);
            float c[8];
            {
                const float4 c0 = reinterpret_cast<const float4 *>(P + pi * 8)[0];
                const float4 c1 = reinterpret_cast<const float4 *>(P + pi * 8)[1];
                c[0] = c0.x; c[1] = c0.y; c[2] = c0.z; c[3] = c0.w;
                c[4] = c1.x; c[5] = c1.y; c[6] = c1.z; c[7] = c1.w;
            }
            float r[8];
#pragma unroll
            for (int d = 0; d < 8; ++d) r[d] = 0.f;   // slots beyond nc stay zero
            if (X != 0.f) {
                // Taylor shift of the piece to the interval start
#pragma unroll
                for (int d = 0; d < nc; ++d) {
                    float sacc = 0.f;
#pragma unroll
                    for (int k = nc - 1; k >= d; --k) sacc = __fmaf_rn(sacc, X, binomf(k, d) * c[k]);
                    r[d] = (mirror && (d & 1)) ? -sacc : sacc;
                }
            } else {
#pragma unroll
                for (int d = 0; d < nc; ++d) r[d] = (mirror && (d & 1)) ? -c[d] : c[d];
            }
            reinterpret_cast<float4 *>(T)[0] = make_float4(r[0], r[1], r[2], r[3]);
            reinterpret_cast<float4 *>(T)[1] = make_float4(r[4], r[5], r[6], r[7]);
        }
    }
    __syncwarp(gmask);
    if (out)
        for (int k = l; k < kTabFloats / 4; k += G)
            reinterpret_cast<float4 *>(out)[k] = reinterpret_cast<const float4 *>(tab)[k];
    __syncwarp(gmask);
}

// Table of the 3-direction box-spline (Sec. III.D), same layout as the
// B-spline tables of kernel degree 2 (polynomials of degree <= 2 in t).
// phi_theta is the convolution of the boxes of widths b, a and a -+ b
// (Prop. 1 with D = 3): piecewise quadratic, C^1, with breakpoints at the
// sums of subsets of the widths, each carrying the sign (-1)^(subset size);
// phi'' = (sum of the signs passed) / (product of the widths).  Built
// stably like the B-spline tables: phi and phi' are carried from piece to
// piece with piece lengths formed from the integer coordinates (p, q) of the
// breakpoints p a + q b, so a narrow box never divides a large sum.  A width
// below kBMin (b near an axis, a - b near a diagonal) is a Dirac: the
// remaining two boxes give a piecewise-linear phi.
__device__ void build_table_box(float a, float b, int mode, float *out, float *sm, int lane)
{
    constexpr int K2 = 2, NSMAX = 3;          // kernel degree 2: up to 3 interval ends in the head
    float *tab = sm;
    float *pc = tab + kTabFloats;             // pieces: [8][3] (phi, phi', top derivative)
    int *bp = reinterpret_cast<int *>(pc + 24);   // sorted breakpoints p | q << 8 (q biased by 4)
    float *sv = reinterpret_cast<float *>(bp + 8);
    int *sq = reinterpret_cast<int *>(sv + 4);
    int *sf = sq + 4;
    int *nbp = sf + 4;
    for (int k = lane; k < kTabFloats; k += 32) tab[k] = 0.f;
    __syncwarp();
    if (lane == 0) {
        // box widths with their coordinates: b = (0,1), a = (1,0), a -+ b = (1,-+1)
        const int q3 = (mode == kModeBoxSame) ? -1 : 1;
        float wv[3] = {b, a, (mode == kModeBoxSame) ? a - b : (float)((double)a + (double)b)};
        int wp[3] = {0, 1, 1}, wq[3] = {1, 0, q3};
        int used[3], nu = 0;
        for (int d = 0; d < 3; ++d)
            if (wv[d] >= kBMin) used[nu++] = d;
        float prod = 1.f;
        for (int u = 0; u < nu; ++u) prod *= wv[used[u]];
        // all subset sums, sorted by value (ties by p, then q)
        const int nb = 1 << nu;
        int P[8], Q[8], S[8];
        float V[8];
        for (int e = 0; e < nb; ++e) {
            int pp = 0, qq = 0, c = 0;
            for (int u = 0; u < nu; ++u)
                if ((e >> u) & 1) { pp += wp[used[u]]; qq += wq[used[u]]; ++c; }
            int k = e;
            const float v = __fmaf_rn((float)pp, a, (float)qq * b);
            while (k > 0 && (V[k - 1] > v || (V[k - 1] == v && (P[k - 1] > pp || (P[k - 1] == pp && Q[k - 1] > qq))))) {
                V[k] = V[k - 1]; P[k] = P[k - 1]; Q[k] = Q[k - 1]; S[k] = S[k - 1];
                --k;
            }
            V[k] = v; P[k] = pp; Q[k] = qq; S[k] = (c & 1) ? -1 : 1;
        }
        // walk the pieces: phi, phi' and the top derivative (phi'' for three
        // boxes, phi' for two) on each
        float f0 = 0.f, f1 = 0.f;
        int acc = 0;
        for (int j = 0; j < nb; ++j) {
            acc += S[j];
            const float D = (float)acc / prod;
            bp[j] = P[j] | ((Q[j] + 4) << 8);
            pc[3 * j] = f0;
            pc[3 * j + 1] = (nu == 3) ? f1 : D;
            pc[3 * j + 2] = (nu == 3) ? 0.5f * D : 0.f;
            if (j + 1 < nb) {
                const float dl = sym_diff(P[j + 1] - P[j], Q[j + 1] - Q[j], a, b, 0.f);
                if (nu == 3) {
                    f0 = __fmaf_rn(__fmaf_rn(0.5f * D, dl, f1), dl, f0);
                    f1 = __fmaf_rn(D, dl, f1);
                } else {
                    f0 = __fmaf_rn(D, dl, f0);
                }
            }
        }
        *nbp = nb;
        // interval ends s = (q b) mod a in (0, a] for the q of the widths used
        int qs[2], nq = 0;
        for (int u = 0; u < nu; ++u) {
            const int qq = wq[used[u]];
            if (qq != 0 && (nq == 0 || qs[0] != qq)) qs[nq++] = qq;
        }
        if (mode == kModeBoxOpp && nu == 3) qs[nq++] = 2;   // b + (a + b) = a + 2b
        const float ainv = 1.0f / a;
        float rs[3];
        int fs[3], qv[3];
        for (int t = 0; t < nq; ++t) {
            const int qq = qs[t];
            int fq = (int)floorf((float)qq * b * ainv);
            float rq = __fmaf_rn((float)(-fq), a, (float)qq * b);
            if (rq <= 0.f) { fq -= 1; rq = __fmaf_rn((float)(-fq), a, (float)qq * b); }
            else if (rq > a) { fq += 1; rq = __fmaf_rn((float)(-fq), a, (float)qq * b); }
            int k = t;
            while (k > 0 && rs[k - 1] > rq) { rs[k] = rs[k - 1]; fs[k] = fs[k - 1]; qv[k] = qv[k - 1]; --k; }
            rs[k] = rq; fs[k] = fq; qv[k] = qq;
        }
        sv[0] = 0.f; sq[0] = 0; sf[0] = 0;
        for (int t = 0; t < nq; ++t) { sv[t + 1] = rs[t]; sq[t + 1] = qv[t]; sf[t + 1] = fs[t]; }
        for (int t = nq + 1; t <= NSMAX; ++t) { sv[t] = a; sq[t] = 0; sf[t] = -1; }
        for (int t = 0; t < kTabHead; ++t) tab[t] = FLT_MAX;
        for (int t = 0; t < nq; ++t) tab[t] = rs[t];
        tab[kTabMode] = (float)mode;
        tab[kTabA] = a;
        tab[kTabB] = b;
    }
    __syncwarp();
    // entries: lane = (interval sg, candidate i)
    const int nb = *nbp;
    const int sg = lane >> 3, i = lane & 7;
    const int nsg = NSMAX;   // intervals (s_sg, s_sg+1], sg = 0..2
    if (sg < nsg && i < 2 * (K2 + 1)) {
        const float hw = 0.5f * (sv[sg + 1] - sv[sg]);
        const int pl = i - sf[sg], ql = sq[sg];
        const int top = bp[nb - 1];
        const int ptop = top & 255, qtop = (top >> 8) - 4;
        // entry inside the support: its midpoint below the last breakpoint.
        // Empty intervals (hw = 0) are filled too, with the expansion just
        // right of their start: rows step by the exact |kappa|, which can
        // exceed the table's float a by an ulp, and a u_0 in that gap lands
        // in an empty last interval.
        if (sym_diff(pl - ptop, ql - qtop, a, b, hw) < 0.f) {
            int pi = 0;
#pragma unroll
            for (int st = 4; st > 0; st >>= 1) {
                const int c = pi + st;
                if (c < nb - 1) {
                    const int bc = bp[c];
                    if (sym_diff(pl - (bc & 255), ql - ((bc >> 8) - 4), a, b, hw) >= 0.f) pi = c;
                }
            }
            const int bc = bp[pi];
            const float X = sym_diff(pl - (bc & 255), ql - ((bc >> 8) - 4), a, b, 0.f);
            const float c0 = pc[3 * pi], c1 = pc[3 * pi + 1], c2 = pc[3 * pi + 2];
            float *T = tab + tab_poly(sg, i);
            T[0] = __fmaf_rn(__fmaf_rn(c2, X, c1), X, c0);
            T[1] = __fmaf_rn(2.f * c2, X, c1);
            T[2] = c2;
        }
    }
    __syncwarp();
    if (out)
        for (int k = lane; k < kTabFloats / 4; k += 32)
            reinterpret_cast<float4 *>(out)[k] = reinterpret_cast<const float4 *>(tab)[k];
    __syncwarp();
}

// Two tables per warp, one per half-warp (box-spline tables: one after the
// other on the full warp).  a, b and the footprint kind were written into the
// table head by the line setup (FP64 geometry stays there, once per line).
template <int DEG>
__global__ void __launch_bounds__(kTabWarps * 32) tables_kernel(float *tabs, int64_t n_tab)
{
    __shared__ __align__(16) float scratch[2 * kTabWarps][kBuildScratch];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, half = lane >> 4;
    const int64_t t0 = ((int64_t)blockIdx.x * kTabWarps + warp) * 2;
    if (t0 >= n_tab) return;
    const int nt = (t0 + 1 < n_tab) ? 2 : 1;
    const int mode0 = (int)tabs[t0 * kTabFloats + kTabMode];
    __syncwarp();
    if (DEG == 2 && mode0 != kModeBspline) {
        // box-spline tables (one basis per grid, so both are): full warp each
        for (int k = 0; k < nt; ++k) {
            float *out = tabs + (t0 + k) * (int64_t)kTabFloats;
            const float af = out[kTabA], bf = out[kTabB];
            const int mode = (int)out[kTabMode];
            __syncwarp();
            if (mode != kModeBspline) build_table_box(af, bf, mode, out, scratch[2 * warp], lane);
            else if (half == 0) build_table_half<DEG>(af, bf, out, scratch[2 * warp], lane, 0x0000FFFFu);
            __syncwarp();
        }
        return;
    }
    if (half >= nt) return;
    float *out = tabs + (t0 + half) * (int64_t)kTabFloats;
    const float af = out[kTabA], bf = out[kTabB];
    build_table_half<DEG>(af, bf, out, scratch[2 * warp + half], lane & 15, half ? 0xFFFF0000u : 0x0000FFFFu);
}

// ------------------------------------------------------------------ evaluation
// Visit every candidate of every row of one line; `op(node, phi)` is called
// for in-grid candidates (phi may be 0 beyond the support).
template <int DEG, typename Op>
__device__ __forceinline__ void walk_line(const LineHdr &H, const float *tab, const GridDev &g,
                                          int lane, Op op)
{
    const bool vert = H.flags & kVert;
    const int Nq = vert ? g.nx : g.ny;
    const float inv_a = 1.0f / H.a;
    float s[DEG + 1];
#pragma unroll
    for (int q = 0; q <= DEG; ++q) s[q] = tab[q];
    for (int r = H.r_begin + lane; r < H.r_end; r += 32) {
        const RowEval e = row_eval<DEG>(H, s, inv_a, r);
        for (int i = 0; i < H.K; ++i) {
            int q = e.q0 + i;
            if ((unsigned)q < (unsigned)Nq) {
                float ti = (DEG == 0) ? __fmaf_rn((float)i, H.a_corr, e.t) : e.t;
                float phi = horner<DEG>(tab + tab_poly(e.sg, i), ti);
                if (DEG == 0 && e.tie) phi = 0.5f * phi;
                int node = vert ? r * g.nx + q : q * g.nx + r;
                op(node, phi);
            }
        }
        if (DEG == 0 && e.tie) {
            // the run also starts at u = 0: midpoint value on that edge too
            int q = e.q0 - 1;
            if ((unsigned)q < (unsigned)Nq) {
                int node = vert ? r * g.nx + q : q * g.nx + r;
                op(node, 0.5f * inv_a);
            }
        }
    }
}

// At degree 0, whose automatic path these kernels are for few or sparse lines,
// candidates beyond the support are left out, so that coefficients and values
// that are not finite do not reach across it.  (The forward still loads them:
// with loads that wait for phi 512 x 512 pixels and 300 lines took 24 us instead
// of 21; the adjoint saves the additions, 770 -> 615 us at 256 x 256 pixels and
// 552,960 lines.)
template <int DEG>
__device__ __forceinline__ bool in_support(float phi) { return DEG > 0 || phi != 0.f; }

// Is candidate i of a row in the support (u_0 + i a < 2w; <= for ties)?
template <int DEG>
__device__ __forceinline__ bool candidate_in(const LineHdr &H, const float *s, const RowEval &e, int i,
                                             float bf)
{
    if constexpr (DEG == 0) {
        // u_0 + i|kappa| - (a + b) with u_0 = uhi + ulo and |kappa| = a + a_corr:
        // (uhi - (1-i) a) is exact when it is small, the rest are small terms.
        float d = __fadd_rn(__fsub_rn(e.uhi, (float)(1 - i) * H.a),
                            __fsub_rn(__fmaf_rn((float)i, H.a_corr, e.ulo), bf));
        return (H.flags & kDeg0Axis) ? d <= 0.f : d < 0.f;
    } else {
        float u0 = (e.sg ? s[e.sg - 1] : 0.f) + e.t;
        return __fmaf_rn((float)i, H.a, u0) < H.two_w;
    }
}

template <int DEG>
__global__ void __launch_bounds__(256) fwd_kernel(GridDev g, const LineHdr *__restrict__ hdr,
                                                  const float *__restrict__ tabs, int64_t M,
                                                  const float *__restrict__ coef,
                                                  float *__restrict__ sino)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t line = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); line < M;
         line += nw) {
        const LineHdr H = hdr[line];
        float acc = 0.f;
        if (!(H.flags & kEmpty)) {
            const float *tab = tabs + (int64_t)H.tab * kTabFloats;
            walk_line<DEG>(H, tab, g, lane, [&](int node, float phi) {
                const float c = __ldg(coef + node);
                acc = __fmaf_rn(in_support<DEG>(phi) ? c : 0.f, phi, acc);
            });
        }
        acc = warp_sum(acc);
        if (lane == 0) sino[line] = g.h * acc;
    }
}

template <int DEG>
__global__ void __launch_bounds__(256) adj_kernel(GridDev g, const LineHdr *__restrict__ hdr,
                                                  const float *__restrict__ tabs, int64_t M,
                                                  const float *__restrict__ sino,
                                                  float *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t line = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); line < M;
         line += nw) {
        const LineHdr H = hdr[line];
        if (H.flags & kEmpty) continue;
        const float hp = g.h * __ldg(sino + line);
        if (hp == 0.f) continue;
        const float *tab = tabs + (int64_t)H.tab * kTabFloats;
        walk_line<DEG>(H, tab, g, lane, [&](int node, float phi) {
            if (in_support<DEG>(phi)) atomicAdd(out + node, hp * phi);
        });
    }
}

template <int DEG>
__global__ void visited_kernel(GridDev g, const LineHdr *__restrict__ hdr,
                               const float *__restrict__ tabs, int64_t M, int32_t *counts,
                               const int64_t *offsets, int32_t *nodes)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t line = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); line < M;
         line += nw) {
        const LineHdr H = hdr[line];
        int total = 0;
        if (!(H.flags & kEmpty)) {
            const float *tab = tabs + (int64_t)H.tab * kTabFloats;
            const bool vert = H.flags & kVert;
                    const int Nq = vert ? g.nx : g.ny;
            const float inv_a = 1.0f / H.a;
            // b of the table: 2w = m (a + b)
            const float bf = tab[kTabB];   // b the table was built with
            float s[DEG + 1];
#pragma unroll
            for (int q = 0; q <= DEG; ++q) s[q] = tab[q];
            const int64_t base = offsets ? offsets[line] : 0;
            // rows in rounds of 32 so that every lane's writes have a place
            for (int r0 = H.r_begin; r0 < H.r_end; r0 += 32) {
                const int r = r0 + lane;
                int cnt = 0;
                RowEval e{0, 0, 0.f, false, 0.f, 0.f};
                if (r < H.r_end) {
                    e = row_eval<DEG>(H, s, inv_a, r);
                    for (int i = 0; i < H.K; ++i) {
                        int q = e.q0 + i;
                        if ((unsigned)q < (unsigned)Nq && candidate_in<DEG>(H, s, e, i, bf)) ++cnt;
                    }
                    if (e.tie && (unsigned)(e.q0 - 1) < (unsigned)Nq) ++cnt;
                }
                int incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    int v = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += v;
                }
                const int excl = incl - cnt;
                const int round_total = __shfl_sync(0xffffffffu, incl, 31);
                if (nodes && offsets && cnt > 0) {
                    int64_t pos = base + total + excl;
                    for (int i = 0; i < H.K; ++i) {
                        int q = e.q0 + i;
                        if ((unsigned)q < (unsigned)Nq && candidate_in<DEG>(H, s, e, i, bf))
                            nodes[pos++] = vert ? r * g.nx + q : q * g.nx + r;
                    }
                    if (e.tie && (unsigned)(e.q0 - 1) < (unsigned)Nq) {
                        int q = e.q0 - 1;
                        nodes[pos++] = vert ? r * g.nx + q : q * g.nx + r;
                    }
                }
                total += round_total;
            }
        }
        if (lane == 0) counts[line] = total;
    }
}

__global__ void expand_kernel(LinesDev L, int64_t M, float *theta_out, float *y_out)
{
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= M) return;
    if (L.kind == SP_LINES_THETA_Y) {
        if (theta_out) theta_out[r] = L.theta[r];
        if (y_out) y_out[r] = L.y[r];
        return;
    }
    double dx, dy, px, py;
    line_geometry(L, r, dx, dy, px, py);
    if (theta_out) theta_out[r] = (float)atan2(dy, dx);
    if (y_out) y_out[r] = (float)(px * dy - py * dx);
}

template <int DEG>
__device__ float footprint_from_table(const float *tab, float a, float b, int mode, float yt)
{
    // The offset is split in double so that the probe measures the table only.
    float two_w;
    double w;
    int K;
    support_params(DEG, a, b, mode, two_w, w, K);
    const double u = (double)yt + w;
    const bool ties = (DEG == 0) && (b == 0.f);
    const double tw = 2.0 * w;
    if (ties) {
        if (u < 0.0 || u > tw) return 0.f;
        if (u == 0.0 || u == tw) return 0.5f / a;
    } else if (u <= 0.0 || u >= tw) {
        return 0.f;
    }
    int i = (int)ceil(u / (double)a) - 1;
    double u0d = u - (double)i * (double)a;
    if (u0d <= 0.0) { i -= 1; u0d += (double)a; }
    else if (u0d > (double)a) { i += 1; u0d -= (double)a; }
    if (i < 0 || i >= K) return 0.f;
    float s_lo;
    const float u0 = (float)u0d;
    int sg = sigma_of<DEG>(tab, u0, s_lo);
    return horner<DEG>(tab + tab_poly(sg, i), (float)(u0d - (double)s_lo));
}

template <int DEG>
__global__ void footprint_eval_kernel(int64_t count, const float *theta, const float *yt, float *out, int basis)
{
    __shared__ __align__(16) float scratch[kTabWarps][kBuildScratch];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * kTabWarps + warp;
    if (r >= count) return;
    double s, c;
    sincos((double)theta[r], &s, &c);
    float af, bf;
    footprint_ab(DEG, c, s, af, bf);
    const int mode = footprint_mode(basis, c, s);
    if (DEG == 2 && mode != kModeBspline) build_table_box(af, bf, mode, nullptr, scratch[warp], lane);
    else if (lane < 16) build_table_half<DEG>(af, bf, nullptr, scratch[warp], lane, 0x0000FFFFu);
    __syncwarp();
    if (lane == 0) out[r] = footprint_from_table<DEG>(scratch[warp], af, bf, mode, yt[r]);
}

inline unsigned blocks_for(int64_t n, int per)
{
    int64_t b = (n + per - 1) / per;
    return (unsigned)(b < 1 ? 1 : b);
}

inline unsigned warp_blocks(int64_t lines)
{
    // 8 warps per block, grid-stride; enough blocks for several waves on 152 SMs
    int64_t b = (lines + 7) / 8;
    if (b > 152 * 64) b = 152 * 64;
    return (unsigned)(b < 1 ? 1 : b);
}

}  // namespace

#define SPX_DISPATCH(DEGVAR, KERNEL, GRID, BLOCK, STREAM, ...)                          \
    switch (DEGVAR) {                                                                     \
    case 0: KERNEL<0><<<GRID, BLOCK, 0, STREAM>>>(__VA_ARGS__); break;                    \
    case 1: KERNEL<1><<<GRID, BLOCK, 0, STREAM>>>(__VA_ARGS__); break;                    \
    case 2: KERNEL<2><<<GRID, BLOCK, 0, STREAM>>>(__VA_ARGS__); break;                    \
    default: KERNEL<3><<<GRID, BLOCK, 0, STREAM>>>(__VA_ARGS__); break;                   \
    }

cudaError_t launch_setup(const GridDev &g, const LinesDev &L, LineHdr *hdr, float *tabs, float *rec, cudaStream_t s)
{
    if (L.m <= 0) return cudaSuccess;
    if (!center_records(g)) rec = nullptr;
    switch (g.kdeg) {
    case 0: launch_chained(setup_kernel<0>, blocks_for(L.m, kSetupThreads), kSetupThreads, 0, s, g, L, hdr, tabs, rec, L.m); break;
    case 1: launch_chained(setup_kernel<1>, blocks_for(L.m, kSetupThreads), kSetupThreads, 0, s, g, L, hdr, tabs, rec, L.m); break;
    case 2: launch_chained(setup_kernel<2>, blocks_for(L.m, kSetupThreads), kSetupThreads, 0, s, g, L, hdr, tabs, rec, L.m); break;
    default: launch_chained(setup_kernel<3>, blocks_for(L.m, kSetupThreads), kSetupThreads, 0, s, g, L, hdr, tabs, rec, L.m); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_tables(const GridDev &g, const LinesDev &L, float *tabs, int64_t n_tab,
                          cudaStream_t s)
{
    (void)L;
    if (n_tab <= 0) return cudaSuccess;
    SPX_DISPATCH(g.kdeg, tables_kernel, blocks_for(n_tab, 2 * kTabWarps), kTabWarps * 32, s, tabs, n_tab);
    return cudaGetLastError();
}

cudaError_t launch_fwd(const GridDev &g, const LineHdr *hdr, const float *tabs, int64_t m,
                       const float *coef, float *sino, cudaStream_t s)
{
    if (m <= 0) return cudaSuccess;
    SPX_DISPATCH(g.kdeg, fwd_kernel, warp_blocks(m), 256, s, g, hdr, tabs, m, coef, sino);
    return cudaGetLastError();
}

cudaError_t launch_adj(const GridDev &g, const LineHdr *hdr, const float *tabs, int64_t m,
                       const float *sino, float *coef_out, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(coef_out, 0, sizeof(float) * (size_t)g.nx * (size_t)g.ny, s);
    if (e != cudaSuccess || m <= 0) return e;
    SPX_DISPATCH(g.kdeg, adj_kernel, warp_blocks(m), 256, s, g, hdr, tabs, m, sino, coef_out);
    return cudaGetLastError();
}

cudaError_t launch_visited(const GridDev &g, const LineHdr *hdr, const float *tabs, int64_t m,
                           int32_t *counts, const int64_t *offsets, int32_t *nodes,
                           cudaStream_t s)
{
    if (m <= 0) return cudaSuccess;
    SPX_DISPATCH(g.kdeg, visited_kernel, warp_blocks(m), 256, s, g, hdr, tabs, m, counts,
                 offsets, nodes);
    return cudaGetLastError();
}

cudaError_t launch_expand(const LinesDev &L, float *theta_out, float *y_out, cudaStream_t s)
{
    if (L.m <= 0) return cudaSuccess;
    expand_kernel<<<blocks_for(L.m, 256), 256, 0, s>>>(L, L.m, theta_out, y_out);
    return cudaGetLastError();
}

cudaError_t launch_footprint_eval(const GridDev &g, int64_t count, const float *theta, const float *yt,
                                  float *out, float *scratch, cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    (void)scratch;
    SPX_DISPATCH(g.kdeg, footprint_eval_kernel, blocks_for(count, kTabWarps), kTabWarps * 32, s, count, theta, yt,
                 out, g.basis);
    return cudaGetLastError();
}

}  // namespace spx
