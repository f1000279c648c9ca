// Forward projection and adjoint with coefficient strips in shared memory,
// for parallel and fan beams and for free line lists sorted into the same
// kind of chunks (order.cu).
//
// One CTA takes a chunk of up to kChunk neighbouring lines of one view
// (consecutive detector bins, or consecutive lines of a sorted free list).
// Such lines are nearly parallel and adjacent, so in every major-axis row
// their runs of nonzero nodes fall inside a short window; the CTA keeps those
// windows (a skewed strip, one row per major-axis row) in shared memory:
// staged from the coefficients for the forward projection, accumulated and
// then added to the output for the adjoint.  Lines whose major axis is x1 use
// transposed images so that strip rows stay contiguous in global memory.
//
// Lane = line, and the lanes of a warp walk the rows together.  Which
// polynomial a candidate takes depends on where the row's u_0 lies among the
// breakpoints s_q of the line's direction, which differs from lane to lane
// and row to row.  So the kernels do not select polynomials at all.  The
// footprint of degree n is a spline of degree 2n+1 with simple knots: across
// the knot p a + q b only its (2n+1)-th derivative jumps, by
// (-1)^(p+q) C(n+1,p) C(n+1,q) / (a b)^(n+1).  With the polynomials B_i of one
// base interval of u_0, every candidate i is, for any u_0 in (0, a],
//
//   phi(u_0 + i a) = B_i(u_0 - s_base) + sum_q J_{p q} z_q,   p = i - floor(q b / a),
//   J_{p q} = (-1)^(p+q) C(n+1,p) C(n+1,q) / ((2n+1)! (a b)^(n+1)),
//   z_q = |u_0 - s_q|^(2n+1) beyond s_q as seen from the base interval, else 0.
//
// The sum over q depends on the candidate only through p, so breakpoints with
// the same floor(q b / a) share one number Z_f = sum_q g_{qf} z_q, and a
// candidate adds C(n+1, i - f) (-1)^(i - f) Z_f for each of the D = 1 + max f
// values of f: integer weights known at compile time.  A lane holds its
// line's B_i in registers (two candidates per packed FMA, fma.rn.f32x2) for
// the whole strip: no table look-ups, no sorting and no branches per row.
// The base interval is the one that leaves u_0 the shortest way to go
// (its distance to the ends of (0, a]); the terms J z then stay below a few
// tenths, and the FP32 evaluation of phi is about as accurate as one from
// the interval's own polynomial (rms over random directions 1.4e-8 against
// 1.2e-8 at degree 3).
//
// u_0 is stepped from row to row in 64-bit fixed point: with W(r) =
// 2^32 u(r)/a - 1 (u(r) the line's offset in row r at its reference column)
// the high word of W is the row's step count and the low word its u_0.
//
// Sums.  Rows are taken in blocks of kRowBlock whose bounds are fixed in the
// image.  A block's sum is one FP32 chain; block sums are added as float pairs
// (two-sum), so that a line's value does not depend on how its blocks were
// spread over warps and lanes, i.e. on the lines it shares a chunk with.
//
// What bounds it: the FMA pipe.  A row of a line with N = n + 1 + D candidates
// takes N (2n+1) Horner FMAs, about (n + 2) D for the knots, 7 (n + 1) for the
// z_q and N to accumulate (87 at n = 3, D = 2), and N shared-memory accesses;
// the lanes' accesses of one row fall on neighbouring columns, in distinct
// banks.
//
// The adjoint accumulates its strip in 32-bit fixed point: a shared-memory
// integer reduction costs about what a plain shared store does on this GPU,
// a float one four to six times more.  Each chunk takes the power of two S
// that puts its largest contribution h |p| phi (phi <= sqrt(2) < 1.5 for
// every basis here) at 2^21 or less; a pair then adds round(S h p phi) to its
// node, at most 2^26 in magnitude after 32 lines, and the flush adds the
// sums times 1/S (exact) to the image.  Adding M = 1.5 2^23 does the rounding:
// the result lies in [2^23, 2^24) where floats are the integers, and its bits
// minus M's bits are round(S h p phi).  Per pair that is an error of about
// half a unit, 1/S <= 1.5 h max|p| 2^-21 = 7e-7 h max|p|.
#include <climits>
#include <cfloat>

#include "common.cuh"

namespace spx {
namespace {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kChunk = 32;          // lines per chunk (lanes of a warp)
constexpr int kRowBlock = 4;        // rows summed in one FP32 chain
constexpr int kSlopeBits = 15;      // fractional bits of the window's slope
constexpr int kMaxWidth = 192;      // widest strip row (floats)
constexpr int kStripFloats = 25280; // strip rows held at once times their width
constexpr int kBasePitch = kSigStride + kTabHead + 4;   // a line's base polynomials and table head, spaced so that
                                                        // 16-byte reads of 8 lanes meet 32 banks

constexpr size_t kStripBytes = sizeof(float) * kStripFloats;
constexpr size_t kBaseBytes = sizeof(float) * kBasePitch * kChunk;
constexpr size_t kHdrBytes = sizeof(LineHdr) * kChunk;
constexpr size_t kPartBytes = 2 * sizeof(float) * kWarps * kChunk;
constexpr size_t kSmemBytes = kStripBytes + kBaseBytes + kHdrBytes + kPartBytes;
static_assert(kStripBytes % 16 == 0 && kBaseBytes % 16 == 0 && kHdrBytes % 16 == 0, "16-byte alignment of the regions");
static_assert(kSmemBytes <= 115712, "two CTAs per SM");
static_assert(kStripFloats / kMaxWidth >= 8 * kRowBlock, "the widest strip holds a row block per warp");
static_assert(kBasePitch % 8 == 4, "conflict-free 16-byte reads");

// What the kernels are instantiated for: the B-spline degrees, and the
// 3-direction box-spline (whose footprint is piecewise quadratic with knots
// in its first two derivatives).
constexpr int kKindBox = 4;
inline int strip_kind(const GridDev &g) { return g.basis == SP_BASIS_BOX3 ? kKindBox : g.kdeg; }

// ------------------------------------------------------------------ packed FP32
typedef unsigned long long f2;

__device__ __forceinline__ f2 f2pack(float a, float b)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ void f2unpack(f2 v, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}

__device__ __forceinline__ f2 f2fma(f2 a, f2 b, f2 c)
{
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ f2 f2mul(f2 a, f2 b)
{
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ f2 f2add(f2 a, f2 b)
{
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// (hi, lo) += x, hi + lo kept to about 48 bits (two-sum).
__device__ __forceinline__ void pair_add(float &hi, float &lo, float x)
{
    const float s = __fadd_rn(hi, x);
    const float bb = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb)));
    hi = s;
}

__device__ __forceinline__ void red_shared(float *p, float v)
{
    asm volatile("red.shared.add.f32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(p)), "f"(v)
                 : "memory");
}

// No "memory" clobber: the strip is read only after the block's barrier
// before its flush, so the reductions need not order any other access.
__device__ __forceinline__ void red_shared_u32(int *p, int v)
{
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(p)), "r"(v));
}

// Fixed-point rounding constant M = 1.5 * 2^23 (see the top of the file).
constexpr float kFixMagic = 12582912.0f;
constexpr int kFixMagicBits = 0x4B400000;
// Largest contribution of a chunk after scaling, and the bound on phi used
// to choose the scale.
constexpr float kFixMax = 2097152.0f;   // 2^21
constexpr float kPhiBound = 1.5f;

// Which chunks an adjoint call runs (strip_chunk's FM).
enum FixMode { kFmAll = 0, kFmFixed = 1, kFmFloat = 2 };

__device__ __forceinline__ void cp_async16(unsigned dst, const void *src, bool in = true)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}
// 4 bytes, or zeros where in is false (src is then not read).
__device__ __forceinline__ void cp_async4(unsigned dst, const void *src, bool in)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(in ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// (xh + xl) / a in fixed point with F fractional bits, a = H.a_hi + H.a_lo:
// the float quotient and one correction step.
template <int F>
__device__ __forceinline__ long long fix_quot(const LineHdr &H, float inv_a, float xh, float xl)
{
    constexpr float kOne = F == 32 ? 4294967296.f : 281474976710656.f;
    const float q1 = xh * inv_a;
    const float r = __fmaf_rn(-q1, H.a_lo, __fmaf_rn(-q1, H.a_hi, xh) + xl);
    return __float2ll_rn(q1 * kOne) + __float2ll_rn(r * inv_a * kOne);
}

// W of row 0 and its step per row.
template <int F>
__device__ __forceinline__ void row_stepping(const LineHdr &H, long long &W, long long &step)
{
    const float inv_a = 1.0f / H.a;
    step = fix_quot<F>(H, inv_a, H.rho_hi, H.rho_lo);
    W = fix_quot<F>(H, inv_a, H.U0, H.U0_lo) - 1 - H.r_ref * step;
}

// The row records a plan keeps: every line's W of row 0 and its step, from
// which all its rows follow (degree >= 1).
__global__ void row_record_kernel(const LineHdr *__restrict__ hdr, int64_t m, longlong2 *__restrict__ rec)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const LineHdr H = hdr[i];
    long long W = 0, step = 0;
    if (!(H.flags & kEmpty)) row_stepping<32>(H, W, step);
    rec[i] = make_longlong2(W, step);
}

// ------------------------------------------------------------------ one line on a strip
// A lane's line on a strip: W of strip row 0 and the step per row; a run
// starts in column q_ref minus W's high part.
struct LaneLine {
    long long W0, Wstep;
    int q_ref;
    float a, ua;               // a, and a / 2^F
    float hp;                  // adjoint: h p (times the chunk's scale S for fixed-point strips)
    // 1 at run time: multiplied by it the polynomials settle in register pairs;
    // left as loaded, the compiler packs them anew in every row (48 moves a row
    // at degree 3, 1.39 against 1.19 ms at the 512 x 512 cubic fan)
    float one;
    const float *base;         // B_i [8][8], then the table head
    float s_base;              // the base interval's start
    // the rows whose run reaches the line's last candidate slot (x up to the
    // end of the support): slot N - 1 of lines with the warp's most slots N,
    // slot N - 2 of the others
    bool has_last;
    unsigned x_end;
};

// The strip in shared memory: `rows` rows of `pitch` floats, row rr starting
// at the column c0 + slope rr 2^-kSlopeBits rounded down to a multiple of 4.
struct Strip {
    float *p;
    int pitch, rows, c0, slope;
    __device__ __forceinline__ int first(int rr) const { return (c0 + ((slope * rr) >> kSlopeBits)) & ~3; }
};

// Candidate pair (2p, 2p+1)'s weights for the knots with floor(q b / a) = f:
// (-1)^k C(m, k) at k = 2p - f and 2p + 1 - f.
__host__ __device__ constexpr float knot_weight(int m, int k)
{
    if (k < 0 || k > m) return 0.f;
    float r = 1.f;
    for (int i = 1; i <= k; ++i) r = r * (float)(m - k + i) / (float)i;
    return (k & 1) ? -r : r;
}

// The values of f = floor(q b / a) that knot q can have in a warp whose lines
// have D or D - 1 of them (b / a in (max(D - 2, 0) / m, D / m)).
__host__ __device__ constexpr int knot_f_lo(int m, int D, int q) { return D >= 2 ? q * (D - 2) / m : 0; }
__host__ __device__ constexpr int knot_f_hi(int m, int D, int q) { return (q * D + m - 1) / m - 1; }

// Rows [r0, r1) of a block for one B-spline line of degree DEG, m = DEG + 1,
// N = m + D candidates: the polynomials and knots in registers.
template <int DEG, int D, bool ADJ, bool FIX>
struct SplineRows {
    static constexpr int F = 32;
    static constexpr int m = DEG + 1, NC = 2 * DEG + 2, N = m + D, NP = N / 2;
    static constexpr int NQ = (m + 1) / 2;   // knots, two per packed operation
    f2 C[NP][NC];      // candidates 2p, 2p + 1
    float cl[NC];      // the last one of an odd N
    f2 zs[NQ], zb[NQ]; // distance to knot q: zs u + zb, positive beyond it
    float g[m][D];     // Z_f = sum_q g[q][f] z_q
    float ua, ub;      // t = ua x + ub
    float hp;          // float adjoint: the factor of phi
    unsigned x_last, x_prev;   // rows that have candidates N - 1 and N - 2: x up to these
    bool has_last;

    __device__ __forceinline__ void load(const LaneLine &ln)
    {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            float c[8];
#pragma unroll
            for (int d4 = 0; d4 < (NC + 3) / 4; ++d4) {
                const float4 w = *reinterpret_cast<const float4 *>(ln.base + i * kNC + 4 * d4);
                c[4 * d4] = w.x; c[4 * d4 + 1] = w.y; c[4 * d4 + 2] = w.z; c[4 * d4 + 3] = w.w;
            }
#pragma unroll
            for (int d = 0; d < NC; ++d) {
                const float v = c[d] * (FIX ? ln.hp : ln.one);
                if (i == 2 * NP) {
                    cl[d] = v;
                } else if (i & 1) {
                    float lo, hi;
                    f2unpack(C[i / 2][d], lo, hi);
                    C[i / 2][d] = f2pack(lo, v);
                } else {
                    C[i / 2][d] = f2pack(v, 0.f);
                }
            }
        }
        const float a = ln.a, b = ln.base[kSigStride + kTabB], inv_a = 1.0f / a;
        // 1 / ((2n+1)! (a b)^(n+1)); no knots in b = 0 (the Dirac of Prop. 1)
        float ab = a * b, kap = ab;
#pragma unroll
        for (int k = 1; k < m; ++k) kap *= ab;
        constexpr float kFact = DEG == 3 ? 5040.f : DEG == 2 ? 120.f : 6.f;
        kap = b > 0.f ? 1.0f / (kFact * kap) : 0.f;
        if constexpr (FIX) kap *= ln.hp;
        float zsv[2 * NQ], zbv[2 * NQ];
#pragma unroll
        for (int k = 0; k < 2 * NQ; ++k) { zsv[k] = 0.f; zbv[k] = 0.f; }
#pragma unroll
        for (int q = 1; q <= m; ++q) {
            // s_q = q b - f a in (0, a], as the table builder takes it
            int f = (int)floorf((float)q * b * inv_a);
            float s = __fmaf_rn((float)(-f), a, (float)q * b);
            if (s <= 0.f) { f -= 1; s = __fmaf_rn((float)(-f), a, (float)q * b); }
            else if (s > a) { f += 1; s = __fmaf_rn((float)(-f), a, (float)q * b); }
            const float sg = s <= ln.s_base ? -1.f : 1.f;   // knots below the base interval look down
            zsv[q - 1] = sg * ln.ua;
            zbv[q - 1] = sg * (ln.ua - s);
            // (a value of f outside the range only arises at s_q = 0 or a to
            // rounding, where z_q vanishes)
#pragma unroll
            for (int k = 0; k < D; ++k) {
                const bool can = k >= knot_f_lo(m, D, q) && k <= knot_f_hi(m, D, q);
                g[q - 1][k] = (can && f == k) ? kap * knot_weight(m, q) : 0.f;
            }
        }
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            zs[k] = f2pack(zsv[2 * k], zsv[2 * k + 1]);
            zb[k] = f2pack(zbv[2 * k], zbv[2 * k + 1]);
        }
        ua = ln.ua;
        ub = ln.ua - ln.s_base;
        hp = ln.hp;
        has_last = ln.has_last;
        x_last = ln.x_end;
        x_prev = has_last ? 0xffffffffu : ln.x_end;
    }

    // One row at strip address sp (the run's first column).
    __device__ __forceinline__ void row(long long W, float *sp, f2 &acc) const
    {
        const float xf = (float)(unsigned)W;
                const bool on_last = has_last && (unsigned)W <= x_last, on_prev = (unsigned)W <= x_prev;
        const float t = __fmaf_rn(xf, ua, ub);
        const f2 tt = f2pack(t, t), xx = f2pack(xf, xf);
        float z[2 * NQ];
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            float d0, d1;
            f2unpack(f2fma(xx, zs[k], zb[k]), d0, d1);
            const f2 d = f2pack(fmaxf(d0, 0.f), fmaxf(d1, 0.f));
            const f2 d2 = f2mul(d, d);
            f2 w = f2mul(d2, d);                     // d^3
            if constexpr (DEG == 2) w = f2mul(w, d2);                  // d^5
            if constexpr (DEG == 3) w = f2mul(w, f2mul(d2, d2));       // d^7
            f2unpack(w, z[2 * k], z[2 * k + 1]);
        }
        float Z[D];
#pragma unroll
        for (int f = 0; f < D; ++f) {
            bool any = false;
            Z[f] = 0.f;
#pragma unroll
            for (int q = 1; q <= m; ++q)
                if (f >= knot_f_lo(m, D, q) && f <= knot_f_hi(m, D, q)) {
                    Z[f] = any ? __fmaf_rn(g[q - 1][f], z[q - 1], Z[f]) : g[q - 1][f] * z[q - 1];
                    any = true;
                }
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            f2 e = C[p][0], phi = C[p][NC - 1];
#pragma unroll
            for (int f = 0; f < D; ++f)
                if (2 * p + 1 - f >= 0 && 2 * p - f <= m) {
                    // (scalar FMAs with immediate weights: packed ones need
                    // two moves per weight pair and row, 4 % slower)
                    float e0, e1;
                    f2unpack(e, e0, e1);
                    if (2 * p - f >= 0 && 2 * p - f <= m) e0 = __fmaf_rn(Z[f], knot_weight(m, 2 * p - f), e0);
                    if (2 * p + 1 - f >= 0 && 2 * p + 1 - f <= m) e1 = __fmaf_rn(Z[f], knot_weight(m, 2 * p + 1 - f), e1);
                    e = f2pack(e0, e1);
                }
#pragma unroll
            for (int d = NC - 2; d >= 1; --d) phi = f2fma(phi, tt, C[p][d]);
            phi = f2fma(phi, tt, e);
            const bool on0 = 2 * p == N - 2 ? on_prev : true;
            const bool on1 = 2 * p + 1 == N - 1 ? on_last : 2 * p + 1 == N - 2 ? on_prev : true;
            if constexpr (ADJ) {
                float v0, v1;
                if constexpr (FIX) {
                    int *ip = reinterpret_cast<int *>(sp);
                    f2unpack(f2add(phi, f2pack(kFixMagic, kFixMagic)), v0, v1);
                    // (adding zero instead of branching)
                    red_shared_u32(ip + 2 * p, on0 ? __float_as_int(v0) - kFixMagicBits : 0);
                    red_shared_u32(ip + 2 * p + 1, on1 ? __float_as_int(v1) - kFixMagicBits : 0);
                } else {
                    f2unpack(phi, v0, v1);
                    if (on0) red_shared(sp + 2 * p, hp * v0);
                    if (on1) red_shared(sp + 2 * p + 1, hp * v1);
                }
            } else {
                float c0 = 0.f, c1 = 0.f;
                if (on0) c0 = sp[2 * p];
                if (on1) c1 = sp[2 * p + 1];
                acc = f2fma(f2pack(c0, c1), phi, acc);
            }
        }
        if constexpr (N & 1) {
            float e = cl[0], phi = cl[NC - 1];
#pragma unroll
            for (int f = 0; f < D; ++f)
                if (N - 1 - f <= m) e = __fmaf_rn(Z[f], knot_weight(m, N - 1 - f), e);
#pragma unroll
            for (int d = NC - 2; d >= 1; --d) phi = __fmaf_rn(phi, t, cl[d]);
            phi = __fmaf_rn(phi, t, e);
            if constexpr (ADJ) {
                if constexpr (FIX) {
                    red_shared_u32(reinterpret_cast<int *>(sp) + N - 1,
                                   on_last ? __float_as_int(phi + kFixMagic) - kFixMagicBits : 0);
                } else {
                    if (on_last) red_shared(sp + N - 1, hp * phi);
                }
            } else {
                float c = 0.f, a0, a1;
                if (on_last) c = sp[N - 1];
                f2unpack(acc, a0, a1);
                acc = f2pack(__fmaf_rn(c, phi, a0), a1);
            }
        }
    }
};

// The same for the 3-direction box-spline: at most three breakpoints, across
// which the first two derivatives jump (the first one where a box is as
// narrow as a Dirac), per candidate as the table's polynomials differ.
template <int N, bool ADJ, bool FIX>
struct BoxRows {
    static constexpr int F = 32, NB = 3;
    float c[N][3], j1[NB][N], j2[NB][N];
    float zs[NB], zb[NB];
    float ua, ub, hp;
    unsigned x_last, x_prev;
    bool has_last;

    __device__ __forceinline__ void load(const LaneLine &ln, const float *tab)
    {
        float s[NB + 1];
        s[0] = 0.f;
#pragma unroll
        for (int k = 0; k < NB; ++k) s[k + 1] = fminf(tab[k], ln.a);
        const float sc = FIX ? ln.hp : 1.f;
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int d = 0; d < 3; ++d) c[i][d] = ln.base[i * kNC + d] * sc;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            // breakpoint s[k + 1] between the intervals k and k + 1
            const float L = s[k + 1] - s[k];
            const float sg = s[k + 1] <= ln.s_base ? -1.f : 1.f;
            zs[k] = sg * ln.ua;
            zb[k] = sg * (ln.ua - s[k + 1]);
            const bool real = s[k + 1] < ln.a;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const float *lo = tab + tab_poly(k, i), *hi = tab + tab_poly(k + 1, i);
                const float d1 = hi[1] - __fmaf_rn(2.f * lo[2], L, lo[1]), d2 = hi[2] - lo[2];
                j1[k][i] = real ? d1 * sc : 0.f;
                j2[k][i] = real ? sg * d2 * sc : 0.f;
            }
        }
        ua = ln.ua;
        ub = ln.ua - ln.s_base;
        hp = ln.hp;
        has_last = ln.has_last;
        x_last = ln.x_end;
        x_prev = has_last ? 0xffffffffu : ln.x_end;
    }

    __device__ __forceinline__ void row(long long W, float *sp, f2 &acc) const
    {
        const float xf = (float)(unsigned)W;
        const bool on_last = has_last && (unsigned)W <= x_last, on_prev = (unsigned)W <= x_prev;
        const float t = __fmaf_rn(xf, ua, ub);
        float d[NB], dd[NB], a0, a1;
        f2unpack(acc, a0, a1);
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            d[k] = fmaxf(__fmaf_rn(xf, zs[k], zb[k]), 0.f);
            dd[k] = d[k] * d[k];
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            float phi = __fmaf_rn(__fmaf_rn(c[i][2], t, c[i][1]), t, c[i][0]);
#pragma unroll
            for (int k = 0; k < NB; ++k) phi = __fmaf_rn(j1[k][i], d[k], __fmaf_rn(j2[k][i], dd[k], phi));
            const bool on = i == N - 1 ? on_last : i == N - 2 ? on_prev : true;
            if constexpr (ADJ) {
                if constexpr (FIX) {
                    if (on) red_shared_u32(reinterpret_cast<int *>(sp) + i, __float_as_int(phi + kFixMagic) - kFixMagicBits);
                } else {
                    if (on) red_shared(sp + i, hp * phi);
                }
            } else {
                float v = 0.f;
                if (on) v = sp[i];
                if (i & 1) a1 = __fmaf_rn(v, phi, a1);
                else a0 = __fmaf_rn(v, phi, a0);
            }
        }
        acc = f2pack(a0, a1);
    }
};

// The strip's row blocks [b0, b1) of this lane's line.  Forward: adds their
// sums to (hi, lo).
template <typename Rows>
__device__ __forceinline__ void walk_blocks(const Rows &R, const LaneLine &ln, const Strip &st, int b0, int b1, bool adj,
                                            float &hi, float &lo)
{
    long long W = ln.W0 + (long long)(b0 * kRowBlock) * ln.Wstep;
    for (int b = b0; b < b1; ++b) {
        f2 acc = 0ull;
        int rr = b * kRowBlock;
#pragma unroll
        for (int k = 0; k < kRowBlock; ++k, ++rr) {
            float *sp = st.p + (rr * st.pitch + (ln.q_ref - (int)(W >> Rows::F) - st.first(rr)));
            R.row(W, sp, acc);
            W += ln.Wstep;
        }
        if (!adj) {
            float a0, a1;
            f2unpack(acc, a0, a1);
            pair_add(hi, lo, a0 + a1);
        }
    }
}

// ------------------------------------------------------------------ degree 0
// Degree 0 has at most two candidates per row and two intervals; its lanes
// select the (linear) polynomials.  Its footprint can have ramps far narrower
// than one float ulp of u, so W carries 48 fractional bits.
constexpr int kFrac0 = 48;

// One row of a degree-0 line exactly along an axis (kDeg0Axis), whose
// footprint is a rectangle with edges on nodes, each taking the midpoint value
// on both sides (so a row has one more candidate): straight from or to global
// memory.  Such lines occur only at views exactly along an axis.
__device__ __noinline__ float axis_row0(const LineHdr &H, const float *tab, int r, const float *__restrict__ src,
                                        float *dst, int Nq, float hp, bool adj)
{
    const float inv_a = 1.0f / H.a;
    float s0[1] = {tab[0]};
    float acc = 0.f;
    const RowEval e = row_eval<0>(H, s0, inv_a, r);
    for (int i = -1; i < H.K; ++i) {
        const int q = e.q0 + i;
        if ((unsigned)q >= (unsigned)Nq) continue;
        float phi;
        if (i < 0) {
            if (!e.tie) continue;
            phi = 0.5f * inv_a;   // the run also starts at u = 0
        } else {
            phi = horner<0>(tab + tab_poly(e.sg, i), __fmaf_rn((float)i, H.a_corr, e.t));
            if (e.tie) phi = 0.5f * phi;
        }
        if (adj) atomicAdd(dst + (size_t)r * Nq + q, hp * phi);
        else acc = __fmaf_rn(__ldg(src + (size_t)r * Nq + q), phi, acc);
    }
    return acc;
}

template <bool ADJ, bool FIX>
struct PixelRows {
    static constexpr int F = kFrac0;
    // c0 + c1 t of candidates 0 and 1 in the intervals 0 and 1 (candidate 1
    // with its argument shift |kappa| - a folded in)
    float c0[2][2], c1[2][2];
    unsigned long long S1;   // the interval's boundary
    float ua, hp;
    bool has_last;

    __device__ __forceinline__ void load(const LaneLine &ln, const float *tab, float a_corr)
    {
#pragma unroll
        for (int sg = 0; sg < 2; ++sg)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float *T = tab + tab_poly(sg, i);
                c1[sg][i] = T[1];
                c0[sg][i] = i ? __fmaf_rn(T[1], a_corr, T[0]) : T[0];
                if constexpr (FIX) {
                    c0[sg][i] = __fmaf_rn(c0[sg][i], ln.hp, kFixMagic);
                    c1[sg][i] *= ln.hp;
                }
            }
        const float s = tab[0], a = ln.a, inv_a = 1.0f / a;
        const float q1 = fminf(s * inv_a, 2.f);
        const float r = fminf(__fmaf_rn(-q1, a, s) * inv_a, 1.f);
        S1 = (unsigned long long)max(__float2ll_rn(q1 * 281474976710656.f) + __float2ll_rn(r * 281474976710656.f), 0ll);
        ua = ln.ua;
        hp = ln.hp;
        has_last = ln.has_last;
    }

    __device__ __forceinline__ void row(long long W, float *sp, f2 &acc) const
    {
        const unsigned long long x = (unsigned long long)W & ((1ull << kFrac0) - 1ull);
        const bool up = x >= S1, on_last = has_last && !up;   // candidate 1 ends with interval 0
        const float t = (float)(x - (up ? S1 : 0ull) + 1ull) * ua;
        const float p0 = __fmaf_rn(up ? c1[1][0] : c1[0][0], t, up ? c0[1][0] : c0[0][0]);
        const float p1 = __fmaf_rn(up ? c1[1][1] : c1[0][1], t, up ? c0[1][1] : c0[0][1]);
        if constexpr (FIX) {
            red_shared_u32(reinterpret_cast<int *>(sp), __float_as_int(p0) - kFixMagicBits);
            if (on_last) red_shared_u32(reinterpret_cast<int *>(sp) + 1, __float_as_int(p1) - kFixMagicBits);
        } else if constexpr (ADJ) {
            red_shared(sp, hp * p0);
            if (on_last) red_shared(sp + 1, hp * p1);
        } else {
            float v = 0.f;
            if (on_last) v = sp[1];
            acc = f2fma(f2pack(sp[0], v), f2pack(p0, p1), acc);
        }
    }
};

// ------------------------------------------------------------------ chunks
// The rows of this lane's line on a strip, blocks [b0, b1) (none where the
// lane has no line): loads the line's polynomials and walks.  n: the
// candidates of the warp's lines (the most).
template <int KIND, bool ADJ, bool FIX>
__device__ __forceinline__ void strip_line(int n, const LaneLine &ln, const LineHdr &H, const float *tab, const Strip &st,
                                           int S0, int b0, int b1, const float *__restrict__ src, float *dst, int Nq,
                                           float hp_raw, float &hi, float &lo)
{
    if constexpr (KIND == 0) {
        if (H.flags & kDeg0Axis) {
            for (int b = b0; b < b1; ++b) {
                float acc = 0.f;
                for (int r = max(S0 + b * kRowBlock, H.r_begin); r < min(S0 + (b + 1) * kRowBlock, H.r_end); ++r)
                    acc += axis_row0(H, tab, r, src, dst, Nq, hp_raw, ADJ);
                pair_add(hi, lo, acc);
            }
            return;
        }
        PixelRows<ADJ, FIX> R;
        R.load(ln, tab, H.a_corr);
        walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo);
    } else if constexpr (KIND == kKindBox) {
        switch (n) {
        case 6: { BoxRows<6, ADJ, FIX> R; R.load(ln, tab); walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo); break; }
        case 5: { BoxRows<5, ADJ, FIX> R; R.load(ln, tab); walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo); break; }
        case 4: { BoxRows<4, ADJ, FIX> R; R.load(ln, tab); walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo); break; }
        default: { BoxRows<3, ADJ, FIX> R; R.load(ln, tab); walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo); break; }
        }
    } else {
        constexpr int m = KIND + 1;
        switch (n - m) {
        case 4: if constexpr (m >= 4) { SplineRows<KIND, m >= 4 ? 4 : 1, ADJ, FIX> R; R.load(ln); walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo); } break;
        case 3: if constexpr (m >= 3) { SplineRows<KIND, m >= 3 ? 3 : 1, ADJ, FIX> R; R.load(ln); walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo); } break;
        case 2: { SplineRows<KIND, 2, ADJ, FIX> R; R.load(ln); walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo); break; }
        default: { SplineRows<KIND, 1, ADJ, FIX> R; R.load(ln); walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo); break; }
        }
    }
}

// The fewest candidates that strip_line is instantiated for.
template <int KIND>
__device__ __forceinline__ int fewest_slots() { return KIND == 0 ? 2 : KIND == kKindBox ? 3 : KIND + 2; }

// Adds the accumulated strip into the image: 16-byte reductions where the
// image rows allow it.
__device__ __forceinline__ void strip_flush(const Strip &st, int S0, int Nr, int Nq, float *dst, bool fixed, float finv,
                                            int vec)
{
    if (vec) {
        const int nch = st.pitch / 4;
        const unsigned inv = 0xffffffffu / (unsigned)nch + 1u;   // i / nch = umulhi(i, inv) for every strip index
        for (int i = threadIdx.x; i < st.rows * nch; i += kThreads) {
            const int rr = (int)__umulhi((unsigned)i, inv), q = st.first(rr) + 4 * (i - rr * nch);
            const int4 n4 = reinterpret_cast<const int4 *>(st.p)[i];
            float4 v = make_float4(__int_as_float(n4.x), __int_as_float(n4.y), __int_as_float(n4.z), __int_as_float(n4.w));
            if (fixed)
                v = make_float4((float)n4.x * finv, (float)n4.y * finv, (float)n4.z * finv, (float)n4.w * finv);
            if ((unsigned)q < (unsigned)Nq && S0 + rr < Nr && (v.x != 0.f || v.y != 0.f || v.z != 0.f || v.w != 0.f))
                asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst + (size_t)(S0 + rr) * Nq + q),
                             "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                             : "memory");
        }
    } else {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        for (int rr = warp; rr < st.rows && S0 + rr < Nr; rr += kWarps)
            for (int c = lane; c < st.pitch; c += 32) {
                const int w = reinterpret_cast<const int *>(st.p)[rr * st.pitch + c], q = st.first(rr) + c;
                const float v = fixed ? (float)w * finv : __int_as_float(w);
                if ((unsigned)q < (unsigned)Nq && v != 0.f) atomicAdd(dst + (size_t)(S0 + rr) * Nq + q, v);
            }
    }
}

// Stages the strip's coefficients, zeros outside the grid.
__device__ __forceinline__ void strip_stage(const Strip &st, int S0, int Nr, int Nq, const float *__restrict__ src, int vec)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(st.p);
    if (vec) {
        // asynchronous 16-byte copies; chunks are wholly inside or outside the
        // grid (Nq and chunk starts are multiples of 4)
        const int nch = st.pitch / 4;
        const unsigned inv = 0xffffffffu / (unsigned)nch + 1u;
        for (int i = threadIdx.x; i < st.rows * nch; i += kThreads) {
            const int rr = (int)__umulhi((unsigned)i, inv), q = st.first(rr) + 4 * (i - rr * nch);
            const bool in = (unsigned)q < (unsigned)Nq && S0 + rr < Nr;
            cp_async16(sa + 16 * i, in ? src + (size_t)(S0 + rr) * Nq + q : src, in);
        }
    } else {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        for (int rr = warp; rr < st.rows; rr += kWarps)
            for (int c = lane; c < st.pitch; c += 32) {
                const int q = st.first(rr) + c;
                const bool in = (unsigned)q < (unsigned)Nq && S0 + rr < Nr;
                cp_async4(sa + 4 * (rr * st.pitch + c), in ? src + (size_t)(S0 + rr) * Nq + q : src, in);
            }
    }
}

// floor(a / b) for b > 0.
__device__ __forceinline__ int floor_div(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// Forward (ADJ false): sino[line] = h sum c phi.  Adjoint (ADJ true): adds
// h sino[line] phi to out (vertical lines) or outT (horizontal lines, the
// transposed image).
// One chunk (view v, bins j0..j0+31) of one instance; smem is the CTA's
// dynamic shared memory (kSmemBytes).
// FM (adjoint only) picks the chunks a call runs: kFmFixed only those that
// accumulate in fixed point, kFmFloat only the others (non-finite values, or
// a scale outside the safe range; see the top of the file), with float
// strips; returns whether the chunk was one of them.  The forward takes
// kFmAll.
template <int KIND, bool ADJ, int FM = kFmAll>
__device__ __forceinline__ bool strip_chunk(unsigned char *smem, const GridDev g, const LinesDev L,
                                            const LineHdr *__restrict__ hdr, const float *__restrict__ tabs,
                                            const float *__restrict__ coef, const float *__restrict__ coefT,
                                            float *__restrict__ sino, float *__restrict__ out,
                                            float *__restrict__ outT, int chunks_per_view, int vec, int chunk,
                                            const longlong2 *__restrict__ rec)
{
    static_assert(!ADJ || FM != kFmAll, "the adjoint runs as fixed-point and float launches");
    constexpr bool FIX = ADJ && FM == kFmFixed;
    constexpr int F = KIND == 0 ? kFrac0 : 32;
    float *strip = reinterpret_cast<float *>(smem);
    float *base_s = reinterpret_cast<float *>(smem + kStripBytes);
    LineHdr *hdr_s = reinterpret_cast<LineHdr *>(smem + kStripBytes + kBaseBytes);
    float2 *part_s = reinterpret_cast<float2 *>(smem + kStripBytes + kBaseBytes + kHdrBytes);   // [warp][line]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int v = chunk / chunks_per_view, cb = chunk - v * chunks_per_view;
    const int j0 = cb * kChunk;
    const int64_t nd = chunk_bins(L);
    const int nl = (int)min((int64_t)kChunk, nd - j0);
    // position of the chunk's first line (in the sorted order for free lists),
    // and lane l's line and table index in every warp (one table per view for
    // parallel beams, else table = line)
    const int64_t line0 = (int64_t)v * nd + j0;
    const int my_line = lane < nl ? (L.order ? __ldg(L.order + line0 + lane) : (int)(line0 + lane)) : 0;
    const bool shared_tab = L.kind == SP_LINES_PARALLEL;
    const float *my_tab = tabs + (shared_tab ? (int64_t)v : (int64_t)my_line) * kTabFloats;

    // The adjoint's values, and the chunk's fixed-point scale (a power of two;
    // see the top of the file).  Non-finite values, or values so large or
    // small that it leaves a safe exponent range, keep the float reductions.
    float pv = 0.f, fscale = 1.f, finv = 1.f;
    if constexpr (ADJ) {
        if (lane < nl) pv = sino[my_line];
        // (bits of non-negative floats order like the floats; non-finite ones on top)
        const unsigned pm = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(pv)));
        const float top = kPhiBound * g.h * __uint_as_float(pm);   // largest |h p phi| of the chunk
        // (an all-zero chunk counts as fixed point: its lines are skipped)
        const bool fix = pm < 0x7f800000u && (top == 0.f || (top >= 1e-20f && top <= 1e20f));
        if (fix != FIX) return false;   // left to the other launch
        if (FIX && top > 0.f) {
            int e;
            frexpf(kFixMax / top, &e);   // kFixMax / top in [2^(e-1), 2^e)
            e -= 1;                      // S = 2^e <= kFixMax / top
            fscale = ldexpf(1.f, e);
            finv = ldexpf(1.f, -e);
        }
    }

    // the chunk's line records into shared memory, and every line's base
    // interval: the one that leaves u_0 the shortest way to the ends of (0, a]
    static_assert(kChunk * 4 <= kThreads && sizeof(LineHdr) == 64, "one pass over the chunk's line records");
    {
        const int src = __shfl_sync(0xffffffffu, my_line, (threadIdx.x >> 2) & 31);
        if ((int)threadIdx.x < nl * 4)
            reinterpret_cast<int4 *>(hdr_s)[threadIdx.x] =
                __ldg(reinterpret_cast<const int4 *>(hdr + src) + (threadIdx.x & 3));
    }
    int sg_base = 0;
    float s_base = 0.f;
    if constexpr (KIND != 0) {
        const float4 h0 = __ldg(reinterpret_cast<const float4 *>(my_tab));
        const float a = __ldg(my_tab + kTabA);
        const float s[5] = {h0.x, h0.y, h0.z, h0.w, a};
        constexpr int NI = KIND == kKindBox ? 4 : KIND + 2;   // intervals
        float lo = 0.f, best = FLT_MAX;
#pragma unroll
        for (int k = 0; k < NI; ++k) {
            const float end = k < NI - 1 ? fminf(s[k], a) : a;
            const float far = fmaxf(lo, a - end);
            if (far < best && end > lo) { best = far; sg_base = k; s_base = lo; }
            lo = end;
        }
        // the base polynomials and the table head
        const int nt = shared_tab ? 1 : nl;
        constexpr int kCh = (kSigStride + kTabHead) / 4;
        const unsigned ba = (unsigned)__cvta_generic_to_shared(base_s);
        for (int i0 = warp * 32; i0 < nt * kCh; i0 += kThreads) {
            const int i = i0 + lane, li = min(i / kCh, kChunk - 1), c = i - li * kCh;
            const int sg = __shfl_sync(0xffffffffu, sg_base, li);
            const int ti = shared_tab ? v : __shfl_sync(0xffffffffu, my_line, li);
            const float *t = tabs + (int64_t)ti * kTabFloats;
            if (i < nt * kCh)
                cp_async16(ba + 4 * (li * kBasePitch + 4 * c),
                           c < kSigStride / 4 ? t + tab_poly(sg, 0) + 4 * c : t + 4 * (c - kSigStride / 4));
        }
    }
    if (!ADJ) part_s[warp * kChunk + lane] = make_float2(0.f, 0.f);
    __syncthreads();

    // this lane's line: W at its reference row, and the step per row
    bool mine = false, mine_vert = false;
    long long my_W = 0, my_step = 0;
    int my_K = 0;
    if (lane < nl) {
        const LineHdr &H = hdr_s[lane];
        mine = !(H.flags & kEmpty) && H.r_end > H.r_begin && (!ADJ || pv != 0.f);
        mine_vert = (H.flags & kVert) != 0;
        if (mine) {
            if (rec) {
                const longlong2 t = __ldg(rec + my_line);
                my_W = t.x;
                my_step = t.y;
            } else {
                row_stepping<F>(H, my_W, my_step);
            }
            my_K = max(H.K, fewest_slots<KIND>() - 1);
        }
    }
    for (int axis = 0; axis < 2; ++axis) {
        const bool vert = axis == 0;
        const unsigned mask = __ballot_sync(0xffffffffu, mine && mine_vert == vert);
        const int Nq = vert ? g.nx : g.ny, Nr = vert ? g.ny : g.nx;
        const float *src = vert ? coef : coefT;
        float *dst = vert ? out : outT;
        // Groups: aligned spans of lines [ga, ga + len), len a power of two,
        // whose runs fit a strip row and whose candidate slots differ by at
        // most one; others are halved.  Every warp finds the same ones.
        for (int ga = 0, len = kChunk; ga < kChunk; ga += len, len = ga & -ga) {
            auto in_span = [&](int a, int n) { return mask & ((n >= 32 ? 0xffffffffu : (1u << n) - 1u) << a); };
            if (in_span(ga, len) == 0u) continue;
            int R0, R1, la, lb, n, width;
            for (;;) {
                // a half without lines is left out
                while (len > 1 && in_span(ga + (len >> 1), len >> 1) == 0u) len >>= 1;
                const bool in = (in_span(ga, len) >> lane) & 1u;
                // row range of the group in whole blocks, and the lowest and
                // highest run start of its lines in the first and the last
                // row.  A run starts within one column above its line, and
                // lines are straight, so between the two rows the starts stay
                // within a column of the chords through the extremes.
                R0 = __reduce_min_sync(0xffffffffu, in ? hdr_s[lane].r_begin : INT_MAX) & -kRowBlock;
                R1 = (__reduce_max_sync(0xffffffffu, in ? hdr_s[lane].r_end : INT_MIN) + kRowBlock - 1) & -kRowBlock;
                const int qa = in ? hdr_s[lane].q_ref - (int)((my_W + R0 * my_step) >> F) : 0;
                const int qb = in ? hdr_s[lane].q_ref - (int)((my_W + (R1 - 1) * my_step) >> F) : 0;
                la = __reduce_min_sync(0xffffffffu, in ? qa : INT_MAX);
                lb = __reduce_min_sync(0xffffffffu, in ? qb : INT_MAX);
                const int ha = __reduce_max_sync(0xffffffffu, in ? qa : INT_MIN);
                const int hb = __reduce_max_sync(0xffffffffu, in ? qb : INT_MIN);
                n = max(__reduce_max_sync(0xffffffffu, in ? my_K : 0), fewest_slots<KIND>());
                const int nmin = __reduce_min_sync(0xffffffffu, in ? my_K : INT_MAX);
                // 3 columns below the lowest start, 3 beyond the highest run,
                // 3 for the start rounded down to a multiple of 4
                width = (max(ha - la, hb - lb) + n + 9 + 3) & ~3;
                if (len == 1 || (width <= kMaxWidth && n - nmin <= 1)) break;
                len >>= 1;
                if (in_span(ga, len) == 0u) ga += len;
            }

            // this lane's line of the group (groups of fewer than 32 lines:
            // several lanes per line, on consecutive rows)
            const int li = ga + (lane & (len - 1)), parts = kChunk / len;
            const bool on = in_span(li, 1) != 0u;
            const int lj = on ? li : __ffs(in_span(ga, len)) - 1;   // (a lane without one looks at another's)
            const LineHdr &H = hdr_s[lj];
            LaneLine ln;
            ln.Wstep = __shfl_sync(0xffffffffu, my_step, lj);
            const long long W_row0 = __shfl_sync(0xffffffffu, my_W, lj);
            ln.q_ref = H.q_ref;
            ln.one = __uint_as_float(0x3f800000u + (unsigned)(nd >> 62));
            ln.a = H.a;
            ln.ua = H.a * (F == 32 ? 2.3283064365386963e-10f : 3.5527136788005009e-15f);
            const float hp_raw = ADJ ? g.h * __shfl_sync(0xffffffffu, pv, lj) : 0.f;
            ln.hp = hp_raw * fscale;
            ln.base = base_s + (shared_tab ? 0 : lj) * kBasePitch;
            ln.s_base = __shfl_sync(0xffffffffu, s_base, lj);
            ln.has_last = __shfl_sync(0xffffffffu, my_K, lj) >= n;
            {
                // 2w - (K - 1) a in units of a 2^-32
                const float end = H.two_w / H.a - (float)(H.K - 1);
                ln.x_end = end >= 1.f ? 0xffffffffu : (unsigned)(fmaxf(end, 0.f) * 4294967296.f);
            }
            const float *tab = tabs + (shared_tab ? (int64_t)v : (int64_t)__shfl_sync(0xffffffffu, my_line, lj)) * kTabFloats;

            Strip st;
            st.p = strip;
            st.pitch = width;
            const int span = max(R1 - 1 - R0, 1);
            st.slope = floor_div((lb - la) * (1 << kSlopeBits), span);
            // slabs of equal height that the strip can hold
            const int most = (kStripFloats / width) & -kRowBlock;
            const int slabs = (R1 - R0 + most - 1) / most;
            const int per = ((R1 - R0 + slabs - 1) / slabs + kRowBlock - 1) & -kRowBlock;
            float hi = 0.f, lo = 0.f;
            for (int S0 = R0; S0 < R1; S0 += per) {
                st.rows = min(per, R1 - S0);
                st.c0 = la + floor_div((lb - la) * (S0 - R0), span) - 3;
                __syncthreads();   // the strip's last readers are done
                if constexpr (ADJ) {
                    float4 *s4 = reinterpret_cast<float4 *>(strip);
                    for (int i = threadIdx.x; i < st.rows * width / 4; i += kThreads) s4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                } else {
                    strip_stage(st, S0, Nr, Nq, src, vec);
                }
                cp_async_wait_all();   // the strip's copies, and the base polynomials'
                __syncthreads();
                const int nb = st.rows / kRowBlock, unit = warp * parts + lane / len, units = kWarps * parts;
                const int b0 = nb * unit / units, b1 = on ? nb * (unit + 1) / units : b0;
                ln.W0 = W_row0 + S0 * ln.Wstep;
                strip_line<KIND, ADJ, FIX>(n, ln, H, tab, st, S0, b0, b1, src, dst, Nq, hp_raw, hi, lo);
                if constexpr (ADJ) {
                    __syncthreads();
                    strip_flush(st, S0, Nr, Nq, dst, FIX, finv, vec);
                }
            }
            if constexpr (!ADJ) {
                for (int o = len; o < 32; o <<= 1) {
                    const float h2 = __shfl_xor_sync(0xffffffffu, hi, o), l2 = __shfl_xor_sync(0xffffffffu, lo, o);
                    pair_add(hi, lo, h2);
                    lo += l2;
                }
                if (on && lane < len) {
                    float2 t = part_s[warp * kChunk + li];
                    pair_add(t.x, t.y, hi);
                    part_s[warp * kChunk + li] = make_float2(t.x, t.y + lo);
                }
            }
        }
    }
    cp_async_wait_all();   // (a chunk without lines still has its copies in flight)
    if constexpr (!ADJ) {
        __syncthreads();
        if ((int)threadIdx.x < nl) {   // warp 0: lane = line
            float hi = 0.f, lo = 0.f;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const float2 t = part_s[w * kChunk + lane];
                pair_add(hi, lo, t.x);
                lo += t.y;
            }
            sino[my_line] = g.h * (hi + lo);
        }
    }
    return true;
}

// One CTA per chunk.  The adjoint runs the fixed-point chunks (FM kFmFixed:
// nearly all) and appends the others to defer[2..] (count defer[0]) for
// strip_float_kernel.
template <int KIND, bool ADJ, int FM = kFmAll>
__global__ void __launch_bounds__(kThreads, 2)
strip_kernel(GridDev g, LinesDev L, const LineHdr *__restrict__ hdr, const float *__restrict__ tabs,
             const float *__restrict__ coef, const float *__restrict__ coefT, float *__restrict__ sino,
             float *__restrict__ out, float *__restrict__ outT, int chunks_per_view, int vec, unsigned *defer,
             const longlong2 *__restrict__ rec)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const bool ran = strip_chunk<KIND, ADJ, FM>(smem, g, L, hdr, tabs, coef, coefT, sino, out, outT, chunks_per_view,
                                                vec, (int)blockIdx.x, rec);
    if (FM == kFmFixed && !ran && threadIdx.x == 0) defer[2 + atomicAdd(defer, 1u)] = blockIdx.x;
}

// The deferred adjoint chunks (float strip accumulators): a small persistent
// grid over defer[2 .. 2 + defer[0]), defer[1] its counter.
template <int KIND>
__global__ void __launch_bounds__(kThreads, 2)
strip_float_kernel(GridDev g, LinesDev L, const LineHdr *__restrict__ hdr, const float *__restrict__ tabs,
                   float *__restrict__ sino, float *__restrict__ out, float *__restrict__ outT, int chunks_per_view,
                   int vec, unsigned *defer, const longlong2 *__restrict__ rec)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned cur;
    const unsigned n = defer[0];
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) cur = atomicAdd(defer + 1, 1u);
        __syncthreads();
        if (cur >= n) break;
        strip_chunk<KIND, true, kFmFloat>(smem, g, L, hdr, tabs, nullptr, nullptr, sino, out, outT, chunks_per_view,
                                          vec, (int)defer[2 + cur], rec);
    }
}

// Persistent kernel over the chunks of several instances of one kind (B-spline
// degree, or box-spline): each
// CTA takes the next chunk from one counter (atomicAdd; no CTA waits on
// another) and runs it with its instance's parameters, until every chunk is
// taken.  Instance k owns chunks [jobs[k].chunk0, jobs[k + 1].chunk0).  The
// adjoint runs the fixed-point chunks and appends the others to defer[]
// (count *defer_n) for strip_queue_float_kernel, as the per-instance adjoint
// does with its second launch.  (One kernel per degree: a kernel holding all
// three degrees spilled over a hundred bytes per thread.)
__device__ __forceinline__ const StripJob *queue_job(const StripJob *__restrict__ jobs, int njobs, long long c)
{
    int lo = 0, hi = njobs - 1;   // last job whose first chunk is <= c
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].chunk0 <= c) lo = mid;
        else hi = mid - 1;
    }
    return jobs + lo;
}

template <int KIND, bool ADJ>
__global__ void __launch_bounds__(kThreads, 2)
strip_queue_kernel(const StripJob *__restrict__ jobs, int njobs, long long total, unsigned long long *counter,
                   long long *defer, unsigned long long *defer_n)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long cur;
    for (;;) {
        __syncthreads();   // the previous chunk's last readers of shared memory are done
        if (threadIdx.x == 0) cur = (long long)atomicAdd(counter, 1ull);
        __syncthreads();
        const long long c = cur;
        if (c >= total) break;
        const StripJob *J = queue_job(jobs, njobs, c);
        const bool ran = strip_chunk<KIND, ADJ, ADJ ? kFmFixed : kFmAll>(
            smem, J->g, J->L, J->hdr, J->tabs, J->coef, J->coefT, J->sino, J->out, J->outT, J->cpv, J->vec,
            (int)(c - J->chunk0), nullptr);
        if (ADJ && !ran && threadIdx.x == 0) defer[atomicAdd(defer_n, 1ull)] = c;
    }
}

// The deferred adjoint chunks (float strip accumulators), persistent likewise.
template <int KIND>
__global__ void __launch_bounds__(kThreads, 2)
strip_queue_float_kernel(const StripJob *__restrict__ jobs, int njobs, const long long *__restrict__ defer,
                         const unsigned long long *__restrict__ defer_n, unsigned long long *counter)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long cur;
    const unsigned long long n = *defer_n;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) cur = (long long)atomicAdd(counter, 1ull);
        __syncthreads();
        const long long k = cur;
        if (k >= (long long)n) break;
        const long long c = defer[k];
        const StripJob *J = queue_job(jobs, njobs, c);
        strip_chunk<KIND, true, kFmFloat>(smem, J->g, J->L, J->hdr, J->tabs, J->coef, J->coefT, J->sino,
                                                   J->out, J->outT, J->cpv, J->vec, (int)(c - J->chunk0),
                                         nullptr);
    }
}

// 16-byte staging and flushing: image rows (nx and ny floats) and bases aligned.
inline int strip_vec(const GridDev &g, const void *img, const void *imgT)
{
    return (g.nx % 4 == 0) && (g.ny % 4 == 0) && ((reinterpret_cast<uintptr_t>(img) & 15) == 0) &&
           ((reinterpret_cast<uintptr_t>(imgT) & 15) == 0);
}

template <int KIND>
cudaError_t launch_queue_t(bool adj, const StripJob *jobs, int njobs, int64_t total, unsigned long long *counter,
                           long long *defer, int64_t grid, int sms, cudaStream_t s)
{
    cudaError_t e;
    if (adj) {
        e = cudaFuncSetAttribute(strip_queue_kernel<KIND, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kSmemBytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(strip_queue_float_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSmemBytes);
        if (e != cudaSuccess) return e;
        strip_queue_kernel<KIND, true><<<(unsigned)grid, kThreads, kSmemBytes, s>>>(jobs, njobs, (long long)total,
                                                                                  counter, defer, counter + 1);
        e = cudaGetLastError();
        // the deferred chunks are few (non-finite or extreme sinogram values): a small grid
        if (e == cudaSuccess)
            strip_queue_float_kernel<KIND><<<(unsigned)(grid < sms ? grid : sms), kThreads, kSmemBytes, s>>>(
                jobs, njobs, defer, counter + 1, counter + 2);
        return e == cudaSuccess ? cudaGetLastError() : e;
    }
    e = cudaFuncSetAttribute(strip_queue_kernel<KIND, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kSmemBytes);
    if (e != cudaSuccess) return e;
    strip_queue_kernel<KIND, false><<<(unsigned)grid, kThreads, kSmemBytes, s>>>(jobs, njobs, (long long)total, counter,
                                                                               nullptr, nullptr);
    return cudaGetLastError();
}

__global__ void transpose_kernel(const float *__restrict__ in, float *__restrict__ out, int nx, int ny)
{
    __shared__ float tile[32][33];
    const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
    for (int y = threadIdx.y; y < 32; y += 8) {
        const int i = bx + threadIdx.x, j = by + y;
        if (i < nx && j < ny) tile[y][threadIdx.x] = in[(size_t)j * nx + i];
    }
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += 8) {
        const int j = by + threadIdx.x, i = bx + y;
        if (i < nx && j < ny) out[(size_t)i * ny + j] = tile[threadIdx.x][y];
    }
}

// out[j][i] += inT[i][j]
__global__ void add_transposed_kernel(const float *__restrict__ inT, float *__restrict__ out, int nx, int ny)
{
    __shared__ float tile[32][33];
    const int bi = blockIdx.x * 32, bj = blockIdx.y * 32;
    for (int y = threadIdx.y; y < 32; y += 8) {
        const int i = bi + y, j = bj + threadIdx.x;
        if (i < nx && j < ny) tile[y][threadIdx.x] = inT[(size_t)i * ny + j];
    }
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += 8) {
        const int j = bj + y, i = bi + threadIdx.x;
        if (i < nx && j < ny) out[(size_t)j * nx + i] += tile[threadIdx.x][y];
    }
}

template <int KIND, bool ADJ>
cudaError_t launch_strip_t(const GridDev &g, const LinesDev &L, const LineHdr *hdr, const float *tabs,
                           const float *coef, float *imgT, float *sino, float *out, cudaStream_t s, const longlong2 *rec,
                           unsigned *defer = nullptr)
{
    const dim3 tb(32, 8), tg((g.nx + 31) / 32, (g.ny + 31) / 32);
    cudaError_t e;
    if (ADJ && !defer) return cudaErrorInvalidValue;
    if (!ADJ) {
        transpose_kernel<<<tg, tb, 0, s>>>(coef, imgT, g.nx, g.ny);
    } else {
        e = cudaMemsetAsync(out, 0, sizeof(float) * (size_t)g.nx * g.ny, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(imgT, 0, sizeof(float) * (size_t)g.nx * g.ny, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(defer, 0, 2 * sizeof(unsigned), s);
        if (e != cudaSuccess) return e;
    }
    // the adjoint: fixed-point chunks, then (a small second launch) the
    // chunks they deferred to float strips
    constexpr int FM1 = ADJ ? kFmFixed : kFmAll;
    auto kern = strip_kernel<KIND, ADJ, FM1>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    if (e == cudaSuccess && ADJ)
        e = cudaFuncSetAttribute(strip_float_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    if (e != cudaSuccess) return e;
    if (strip_needs_order(L) && !L.order) return cudaErrorInvalidValue;   // free lists need their order
    const int cpv = (int)((chunk_bins(L) + kChunk - 1) / kChunk);
    const unsigned grid = (unsigned)(chunk_views(L) * cpv);
    const int vec = strip_vec(g, ADJ ? out : coef, imgT);
    kern<<<grid, kThreads, kSmemBytes, s>>>(g, L, hdr, tabs, coef, imgT, const_cast<float *>(sino), out, imgT, cpv,
                                            vec, defer, rec);
    e = cudaGetLastError();
    if (e == cudaSuccess && ADJ) {
        int dev = 0, sms = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const unsigned g2 = grid < (unsigned)sms ? grid : (unsigned)sms;
        if (e == cudaSuccess)
            strip_float_kernel<KIND><<<g2, kThreads, kSmemBytes, s>>>(g, L, hdr, tabs, const_cast<float *>(sino), out,
                                                                     imgT, cpv, vec, defer, rec);
        if (e == cudaSuccess) e = cudaGetLastError();
    }
    if (e == cudaSuccess && ADJ) {
        add_transposed_kernel<<<tg, tb, 0, s>>>(imgT, out, g.nx, g.ny);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace

int strip_queue_kind(const GridDev &g) { return strip_kind(g); }

StripJob make_strip_job(const GridDev &g, const LinesDev &L, const LineHdr *hdr, const float *tabs, bool adj,
                        const float *img_in, float *sino, float *img_out, void *scratch)
{
    StripJob J;
    J.g = g;
    J.L = L;
    J.hdr = hdr;
    J.tabs = tabs;
    J.coef = adj ? nullptr : img_in;
    J.coefT = static_cast<float *>(scratch);
    J.sino = sino;
    J.out = adj ? img_out : nullptr;
    J.outT = static_cast<float *>(scratch);
    J.cpv = (int)((chunk_bins(L) + kChunk - 1) / kChunk);
    J.vec = strip_vec(g, adj ? img_out : img_in, scratch);
    J.chunk0 = 0;
    return J;
}

int64_t strip_job_chunks(const StripJob &J) { return chunk_views(J.L) * J.cpv; }

cudaError_t launch_strip_pre(const StripJob &J, bool adj, cudaStream_t s)
{
    const dim3 tb(32, 8), tg((J.g.nx + 31) / 32, (J.g.ny + 31) / 32);
    if (!adj) {
        transpose_kernel<<<tg, tb, 0, s>>>(J.coef, J.coefT, J.g.nx, J.g.ny);
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(J.out, 0, sizeof(float) * (size_t)J.g.nx * J.g.ny, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(J.outT, 0, sizeof(float) * (size_t)J.g.nx * J.g.ny, s);
    return e;
}

cudaError_t launch_strip_post(const StripJob &J, bool adj, cudaStream_t s)
{
    if (!adj) return cudaSuccess;
    const dim3 tb(32, 8), tg((J.g.nx + 31) / 32, (J.g.ny + 31) / 32);
    add_transposed_kernel<<<tg, tb, 0, s>>>(J.outT, J.out, J.g.nx, J.g.ny);
    return cudaGetLastError();
}

cudaError_t launch_strip_queue(int kind, bool adj, const StripJob *jobs, int njobs, int64_t total,
                               unsigned long long *counter, long long *defer, cudaStream_t s)
{
    if (njobs <= 0 || total <= 0) return cudaSuccess;
    if (kind < 0 || kind > kKindBox || (adj && !defer)) return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaMemsetAsync(counter, 0, 3 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    int64_t grid = 2 * (int64_t)sms;   // two CTAs per SM, resident at once
    if (grid > total) grid = total;
    switch (kind) {
    case 0: return launch_queue_t<0>(adj, jobs, njobs, total, counter, defer, grid, sms, s);
    case 1: return launch_queue_t<1>(adj, jobs, njobs, total, counter, defer, grid, sms, s);
    case 2: return launch_queue_t<2>(adj, jobs, njobs, total, counter, defer, grid, sms, s);
    case 3: return launch_queue_t<3>(adj, jobs, njobs, total, counter, defer, grid, sms, s);
    default: return launch_queue_t<kKindBox>(adj, jobs, njobs, total, counter, defer, grid, sms, s);
    }
}

bool strip_supported(const GridDev &g, const LinesDev &L)
{
    return (L.kind == SP_LINES_PARALLEL || L.kind == SP_LINES_FAN || strip_needs_order(L)) && g.kdeg >= 0;
}

size_t strip_scratch_bytes(const GridDev &g) { return sizeof(float) * (size_t)g.nx * g.ny + 256; }

cudaError_t launch_fwd_strip(const GridDev &g, const LinesDev &L, const LineHdr *hdr, const float *tabs,
                             const float *coef, void *scratch, float *sino, cudaStream_t s, const longlong2 *rec)
{
    float *coefT = static_cast<float *>(scratch);
    switch (strip_kind(g)) {
    case 0: return launch_strip_t<0, false>(g, L, hdr, tabs, coef, coefT, sino, nullptr, s, rec);
    case 1: return launch_strip_t<1, false>(g, L, hdr, tabs, coef, coefT, sino, nullptr, s, rec);
    case 2: return launch_strip_t<2, false>(g, L, hdr, tabs, coef, coefT, sino, nullptr, s, rec);
    case 3: return launch_strip_t<3, false>(g, L, hdr, tabs, coef, coefT, sino, nullptr, s, rec);
    default: return launch_strip_t<kKindBox, false>(g, L, hdr, tabs, coef, coefT, sino, nullptr, s, rec);
    }
}

cudaError_t launch_row_records(const LineHdr *hdr, int64_t m, longlong2 *rec, cudaStream_t s)
{
    if (m <= 0) return cudaSuccess;
    row_record_kernel<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(hdr, m, rec);
    return cudaGetLastError();
}

int64_t strip_chunk_count(const LinesDev &L) { return chunk_views(L) * ((chunk_bins(L) + kChunk - 1) / kChunk); }

cudaError_t launch_adj_strip(const GridDev &g, const LinesDev &L, const LineHdr *hdr, const float *tabs,
                             const float *sino, void *scratch, float *coef_out, cudaStream_t s, const longlong2 *rec,
                             unsigned *defer)
{
    float *outT = static_cast<float *>(scratch);
    float *p = const_cast<float *>(sino);
    switch (strip_kind(g)) {
    case 0: return launch_strip_t<0, true>(g, L, hdr, tabs, nullptr, outT, p, coef_out, s, rec, defer);
    case 1: return launch_strip_t<1, true>(g, L, hdr, tabs, nullptr, outT, p, coef_out, s, rec, defer);
    case 2: return launch_strip_t<2, true>(g, L, hdr, tabs, nullptr, outT, p, coef_out, s, rec, defer);
    case 3: return launch_strip_t<3, true>(g, L, hdr, tabs, nullptr, outT, p, coef_out, s, rec, defer);
    default: return launch_strip_t<kKindBox, true>(g, L, hdr, tabs, nullptr, outT, p, coef_out, s, rec, defer);
    }
}

}  // namespace spx
