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
// polynomial a candidate takes depends on where the row lies among the
// footprint's knots, which differs from lane to lane and row to row, so the
// kernels do not select polynomials.  The footprint of degree n is a spline
// of degree 2n+1 with simple knots: across the knot p a + q b only its
// (2n+1)-th derivative jumps, by (-1)^(p+q) C(n+1,p) C(n+1,q) / (a b)^(n+1).
// Take the offsets of a row's candidates from the footprint's centre as
// (kk + c) a + v with v in [-a/2, a/2) common to the row (c = 1/2 or 0 as n + 1
// is even or odd).  In v the knots lie symmetrically around 0, in two pairs
// +-beta (one at degree 1); a third kind, at v = +-a/2, is where the candidates
// change.  So with the polynomials P_j of the interval around v = 0, w = |v|
// and z = max(w - beta, 0)^(2n+1),
//
//   phi((j + c) a + w) = P_j(w) + J_j z + J'_j z',
//
// and, as phi is even, the candidate on the other side is P_j(-w) with jumps
// of its own.  One chain in v^2 gives the even and the odd part of P_j and
// with them both candidates; half the sum of their jumps joins the even part,
// half the difference, with the sign of v, the odd one.  A lane holds its line's P_j and J in registers
// for the whole strip (the centre records of common.cuh): no table look-ups,
// no sorting and no branches per row.  The jump terms stay below 1e-2 (w goes
// at most min(b, a - b) or min(2b, a - 2b) beyond a knot), so phi keeps the
// accuracy of its polynomials.
//
// v is stepped from row to row in 64-bit fixed point: with Y(r) =
// 2^32 (y(r)/a + 1/2 - c), y(r) the offset from the centre in row r at the
// line's reference column, the high word of Y is the row's step count and the
// low word is v / a + 1/2.
//
// Sums.  Rows are taken in blocks of kRowBlock whose bounds are fixed in the
// image.  A block's sum is one FP32 chain; block sums are added as float pairs
// (two-sum), so that a line's value does not depend on how its blocks were
// spread over warps and lanes, i.e. on the lines it shares a chunk with.
//
// What bounds it: the issue slots (about 75 instructions per row and warp
// forward and 80 in the adjoint at n = 3, 64 % of the slots filled) and the FMA
// pipe (54 and 52 % busy).  A pair of
// candidates takes 3 packed FMAs (n = 3) for the even and odd parts, one
// multiply and two additions to join them, 2 packed FMAs for the jumps and one
// to accumulate; a row adds about 25 instructions (step, v, z, addresses).  The
// lanes' strip accesses of one row fall on neighbouring columns, in distinct
// banks.  Measured at the 512 x 512 cubic fan (552,960 lines), forward and
// adjoint: 0.83 and 0.86 ms (the forward 0.80 without the tests of its outermost
// candidates); one polynomial of 7 FMAs per candidate of a base
// interval plus truncated powers with integer weights 1.19 and 1.28 ms; rows
// sorted by interval, a lane per candidate and row, 2.18 and 2.35 ms.
// Four CTAs of four warps per SM: while one CTA waits for its line records,
// its strip or its flush, three others compute; two CTAs of eight warps with
// strips of twice the height took 0.91 and 0.99 ms, three CTAs of eight warps
// (80 registers) 0.95 and 0.98 ms, five of four warps (96 registers) 0.93 and
// 0.92 ms, against 0.80 and 0.86.
//
// The adjoint of degree >= 1 accumulates its strip in 32-bit fixed point: a
// shared-memory integer reduction costs about what a plain shared store does on
// this GPU, a float one four to six times more.  Each chunk takes the power of two S
// that puts its largest contribution h |p| phi (phi <= sqrt(2) < 1.5 for
// every basis here) at 2^22 or less; a pair then adds round(S h p phi) to its
// node, at most 2^27 in magnitude after 32 lines, and the flush adds the
// sums times 1/S (exact) to the image.  Adding M = 1.5 2^23 does the rounding:
// the result lies in [2^23, 2^24) where floats are the integers, and its bits
// minus M's bits are round(S h p phi).  Per pair that is an error of about
// half a unit, 1/S <= 1.5 h max|p| 2^-21 = 7e-7 h max|p|.  Degree 0 adds floats.
#include <climits>
#include <cfloat>

#include "common.cuh"

namespace spx {
namespace {

constexpr int kWarps = 4;            // four CTAs of four warps per SM (see below)
constexpr int kThreads = kWarps * 32;
constexpr int kCtas = 4;             // CTAs per SM
constexpr int kChunk = 32;          // lines per chunk (lanes of a warp)
constexpr int kRowBlock = 4;        // rows summed in one FP32 chain
constexpr int kSlopeBits = 15;      // fractional bits of the window's slope
constexpr int kMaxWidth = 192;      // widest strip row (floats)
constexpr int kStripFloats = 11264; // strip rows held at once times their width
constexpr int kSlabRows = 512;      // strip rows held at once, at most
constexpr size_t kStripBytes = sizeof(float) * kStripFloats;
constexpr size_t kRecBytes = sizeof(float) * kCenterFloats * kChunk;
constexpr size_t kHdrBytes = sizeof(LineHdr) * kChunk;
constexpr size_t kPartBytes = 2 * sizeof(float) * kWarps * kChunk;
constexpr size_t kOffBytes = sizeof(int) * kSlabRows;
constexpr size_t kSmemBytes = kStripBytes + kRecBytes + kHdrBytes + kPartBytes + kOffBytes;
static_assert(kStripBytes % 16 == 0 && kRecBytes % 16 == 0 && kHdrBytes % 16 == 0, "16-byte alignment of the regions");
static_assert(kSmemBytes <= 57344, "four CTAs per SM");
static_assert(kStripFloats / kMaxWidth >= kWarps * kRowBlock, "the widest strip holds a row block per warp");
static_assert(kPartBytes % 16 == 0 && kRowBlock == 4, "row offsets are read four at a time");
static_assert(kCenterFloats % 8 == 4, "16-byte reads of 8 lanes meet 32 banks");

// What the kernels are instantiated for: the B-spline degrees, and the
// 3-direction box-spline (whose footprint is piecewise quadratic with knots
// in its first two derivatives).
constexpr int kKindBox = 4;
__host__ __device__ constexpr int image_ld(int cols) { return (cols + 3) & ~3; }
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
constexpr float kFixMax = 4194304.0f;   // 2^22
constexpr float kPhiBound = 1.5f;

// Which chunks an adjoint call runs (strip_chunk's FM).  Degree 0 has float
// strips only: its pixels belong to few lines, and where those are far below the
// chunk's largest, fixed point would leave them fewer bits than FP32 sums have.
// (Parallel beams, 501 x 501 pixels, 367 x 751 lines: 332 us, in fixed point 274,
// with the general kernel's global additions 488.)
enum FixMode { kFmAll = 0, kFmFixed = 1, kFmFloat = 2 };
template <int KIND>
__host__ __device__ constexpr int adj_mode() { return KIND == 0 ? kFmFloat : kFmFixed; }

__device__ __forceinline__ void cp_async16(unsigned dst, const void *src, bool in = true)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Degree 0 (see PixelRows) carries more fractional bits.
constexpr int kFrac0 = 48;

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

// Fixed-point position of a line's rows: the value in row 0 and the step per
// row.  KIND 1..3: Y (see the top), b the line's b; others: W = 2^F u/a - 1,
// whose high part is the step count of the run's first candidate and whose low
// part is u_0 (F fractional bits).
template <int KIND>
__device__ __forceinline__ void row_stepping(const LineHdr &H, float b, long long &W, long long &step)
{
    constexpr int F = KIND == 0 ? kFrac0 : 32;
    const float inv_a = 1.0f / H.a;
    step = fix_quot<F>(H, inv_a, H.rho_hi, H.rho_lo);
    W = fix_quot<F>(H, inv_a, H.U0, H.U0_lo) - H.r_ref * step;
    if constexpr (KIND >= 1 && KIND <= 3) {
        // y = u - w, w = m (a + b) / 2; a + b as a float pair
        constexpr int m = KIND + 1;
        const float s = __fadd_rn(H.a, b), e = __fsub_rn(b, __fsub_rn(s, H.a));
        W -= (m * fix_quot<F>(H, inv_a, s, e)) >> 1;
        if (m & 1) W += 1ll << 31;
    } else {
        W -= 1;
    }
}

// The row records a plan keeps: every line's position in row 0 and its step,
// from which all its rows follow (degree >= 1).
template <int KIND>
__global__ void row_record_kernel(const LineHdr *hdr, const float *center, int per_table,
                                  int64_t m, longlong2 *out)
{
    chain_begin();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const LineHdr H = hdr[i];
    long long W = 0, step = 0;
    if (!(H.flags & kEmpty)) {
        const float b = KIND <= 3 ? center[(i / per_table) * kCenterFloats + kCenterB] : 0.f;
        row_stepping<KIND>(H, b, W, step);
    }
    out[i] = make_longlong2(W, step);
}

// ------------------------------------------------------------------ one line on a strip
// A lane's line on a strip: the fixed-point position of strip row 0 and the
// step per row; the run starts in column q_first minus the position's high
// part.
struct LaneLine {
    long long W0, Wstep;
    int q_first;
    float a, ua;               // a, and a / 2^F
    float w_sup;               // half-width of the support
    float hp;                  // adjoint: h p (times the chunk's scale S for fixed-point strips)
    const float *rec;          // centre record (shared memory; KIND 1..3)
    bool has_last;             // box-spline and degree 0: the line has the warp's last candidate,
    unsigned x_end;            // ... and the rows that reach its own last one (low part up to this)
};

// The strip in shared memory: `rows` rows of `pitch` floats, row rr starting
// at the column c0 + slope rr 2^-kSlopeBits rounded down to a multiple of 4.
struct Strip {
    float *p;
    int *off;   // per row: its start in p less its first column
    int pitch, rows, c0, slope;
    __device__ __forceinline__ int first(int rr) const { return (c0 + ((slope * rr) >> kSlopeBits)) & ~3; }
};

// One B-spline line of degree DEG in registers: J pairs of candidates around
// v = 0 (and for odd m = DEG + 1 the one in the middle), N columns from the
// run's first.
template <int DEG, int J, bool ADJ, bool FIX>
struct SplineRows {
    static constexpr int F = 32;
    static constexpr int m = DEG + 1, NC = 2 * DEG + 2, NH = NC / 2;
    static constexpr bool kMid = m % 2 == 1;       // a candidate at v itself
    static constexpr int kKnots = DEG == 1 ? 1 : 2;
    // the inner knots leave the fourth pair (degree 2: counting the middle one) alone
    static constexpr __device__ int first_knot(int j) { return j + (kMid ? 1 : 0) == 3 ? 1 : 0; }
    f2 C[J][NH];            // (even, odd) coefficients, by powers of v^2
    f2 K[J][kKnots];        // jumps: half their sum and half their difference
    float cm[NH], km[kKnots];   // the middle candidate
    float beta[2], ua, ha;
    float hp;                   // float adjoint: factor
    // The candidates of pair j lie in the support where v < end[j] and -v <
    // end[j], w - (j + c) a.  Only the outermost pair can leave it, and in lines
    // that share a warp with wider ones the one before.
    float end[J];
    static constexpr int kTail = DEG == 1 || J == DEG ? J - 1 : J - 2;

    __device__ __forceinline__ void load(const LaneLine &ln)
    {
        const float sc = FIX ? ln.hp : 1.f;
        const f2 sc2 = f2pack(sc, sc);
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const float *T = ln.rec + 8 * (j + (kMid ? 1 : 0));
#pragma unroll
            for (int k = 0; k < NH; k += 2) {
                const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(T + 2 * k);
                C[j][k] = FIX ? f2mul(t.x, sc2) : t.x;
                if (k + 1 < NH) C[j][k + 1] = FIX ? f2mul(t.y, sc2) : t.y;
            }
#pragma unroll
            for (int q = first_knot(j); q < kKnots; ++q) {
                const f2 t = *reinterpret_cast<const f2 *>(ln.rec + kCenterJump + 8 * q + 2 * (j + (kMid ? 1 : 0)));
                K[j][q] = FIX ? f2mul(t, sc2) : t;
            }
            end[j] = ln.w_sup - ((float)j + (kMid ? 1.f : 0.5f)) * ln.a;
        }
        if constexpr (kMid) {
#pragma unroll
            for (int k = 0; k < NH; ++k) cm[k] = ln.rec[2 * k] * sc;
#pragma unroll
            for (int q = 0; q < kKnots; ++q) km[q] = ln.rec[kCenterJump + 8 * q] * sc;
        }
        beta[0] = ln.rec[kCenterBeta];
        beta[1] = ln.rec[kCenterBeta + 1];
        ua = ln.ua;
        ha = 0.5f * ln.a;
        hp = ln.hp;
    }

    // One row at strip address sp (the run's first column).
    __device__ __forceinline__ void row(long long Y, float *sp, f2 &acc) const
    {
        const float v = __fmaf_rn((float)(unsigned)Y, ua, -ha);
        const float w = fabsf(v), s = v * v;
        const f2 ss = f2pack(s, s);
        float z[2] = {0.f, 0.f};
        if constexpr (kKnots == 2) {
            const f2 d = f2pack(fmaxf(w - beta[0], 0.f), fmaxf(w - beta[1], 0.f));
            const f2 d2 = f2mul(d, d);
            f2 t = f2mul(d2, d);                                       // d^3
            if constexpr (DEG == 2) t = f2mul(t, d2);                  // d^5
            if constexpr (DEG == 3) t = f2mul(t, f2mul(d2, d2));       // d^7
            f2unpack(t, z[0], z[1]);
        } else {
            const float d = fmaxf(w - beta[0], 0.f);
            z[0] = d * d * d;
        }
        f2 zz[kKnots];   // (z, z sign(v))
#pragma unroll
        for (int q = 0; q < kKnots; ++q) zz[q] = f2pack(z[q], copysignf(z[q], v));
#pragma unroll
        for (int j = 0; j < J; ++j) {
            f2 h = C[j][NH - 1];
#pragma unroll
            for (int k = NH - 2; k >= 0; --k) h = f2fma(h, ss, C[j][k]);
            float e, o;
            f2unpack(h, e, o);
            // even and odd part with the jumps: the candidate on the side of
            // larger columns takes their sum, its mirror image the difference
            f2 eo = f2pack(e, v * o);
#pragma unroll
            for (int q = first_knot(j); q < kKnots; ++q) eo = f2fma(zz[q], K[j][q], eo);
            f2unpack(eo, e, o);
            put(sp, J + (kMid ? 1 : 0) + j, J - 1 - j, __fadd_rn(e, o), __fsub_rn(e, o), j, v, acc);
        }
        if constexpr (kMid) {
            float e = cm[NH - 1];
#pragma unroll
            for (int k = NH - 2; k >= 0; --k) e = __fmaf_rn(e, s, cm[k]);
#pragma unroll
            for (int q = 0; q < kKnots; ++q) e = __fmaf_rn(z[q], km[q], e);
            if constexpr (ADJ) {
                if constexpr (FIX) red_shared_u32(reinterpret_cast<int *>(sp) + J, __float_as_int(e + kFixMagic) - kFixMagicBits);
                else red_shared(sp + J, hp * e);
            } else {
                float a0, a1;
                f2unpack(acc, a0, a1);
                acc = f2pack(__fmaf_rn(sp[J], e, a0), a1);
            }
        }
    }

    // Adds the pair j: p at column ip and q at column im.  Beyond the support
    // the polynomials leave their rounding (up to 2e-8) where phi is 0: the
    // forward does not read nodes there, so that a line does not see what it does
    // not meet (whatever the size of the coefficient), and the fixed-point strip
    // rounds such values to 0.
    __device__ __forceinline__ void put(float *sp, int ip, int im, float p, float q, int j, float v, f2 &acc) const
    {
        if constexpr (ADJ && FIX) {
            f2unpack(f2add(f2pack(p, q), f2pack(kFixMagic, kFixMagic)), p, q);
            red_shared_u32(reinterpret_cast<int *>(sp) + ip, __float_as_int(p) - kFixMagicBits);
            red_shared_u32(reinterpret_cast<int *>(sp) + im, __float_as_int(q) - kFixMagicBits);
        } else if constexpr (ADJ) {
            if (v < end[j]) red_shared(sp + ip, hp * p);
            if (-v < end[j]) red_shared(sp + im, hp * q);
        } else {
            float x = 0.f, y = 0.f;
            if (j < kTail || v < end[j]) x = sp[ip];
            if (j < kTail || -v < end[j]) y = sp[im];
            acc = f2fma(f2pack(x, y), f2pack(p, q), acc);
        }
    }
};

// A line of the 3-direction box-spline: the polynomials of one base interval of
// u_0 in (0, a], the one that leaves u_0 the shortest way to the ends, and for
// each of at most three breakpoints what the table's polynomials change there
// (the first two derivatives, the first one where a box is as narrow as a
// Dirac).
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
        float s[NB + 2];
        s[0] = 0.f;
        s[NB + 1] = ln.a;
#pragma unroll
        for (int k = 0; k < NB; ++k) s[k + 1] = fminf(tab[k], ln.a);
        int sg_base = 0;
        float s_base = 0.f, best = FLT_MAX;
#pragma unroll
        for (int k = 0; k <= NB; ++k) {
            const float far = fmaxf(s[k], ln.a - s[k + 1]);
            if (far < best && s[k + 1] > s[k]) { best = far; sg_base = k; s_base = s[k]; }
        }
        const float sc = FIX ? ln.hp : 1.f;
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int d = 0; d < 3; ++d) c[i][d] = tab[tab_poly(sg_base, i) + d] * sc;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            // breakpoint s[k + 1] between the intervals k and k + 1
            const float L = s[k + 1] - s[k];
            const float sg = s[k + 1] <= s_base ? -1.f : 1.f;
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
        ub = ln.ua - s_base;
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
        const int4 off4 = reinterpret_cast<const int4 *>(st.off)[b];
        const int off[kRowBlock] = {off4.x, off4.y, off4.z, off4.w};
#pragma unroll
        for (int k = 0; k < kRowBlock; ++k) {
            float *sp = st.p + (off[k] + ln.q_first - (int)(W >> Rows::F));
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
template <bool ADJ>
struct PixelRows {
    static constexpr int F = kFrac0;
    // c0 + c1 t of candidates 0 and 1 in the intervals 0 and 1 (candidate 1
    // with its argument shift |kappa| - a folded in)
    float c0[2][2], c1[2][2];
    unsigned long long S1;   // the interval's boundary
    float ua, hp;
    bool has_last;

    // b: |sin| or |cos|, the shorter; a_corr = |kappa| - a
    __device__ __forceinline__ void load(const LaneLine &ln, float b, float a_corr)
    {
        // the trapezoid of height 1/a: a ramp of width b up in interval 0
        // (candidate 0) and down (candidate 1), its top in interval 1
        const float a = ln.a, top = 1.0f / a, slope = b > 0.f ? top / b : 0.f;
        c0[0][0] = b > 0.f ? 0.f : top;
        c1[0][0] = slope;
        c0[0][1] = __fmaf_rn(-slope, a_corr, top);
        c1[0][1] = -slope;
        c0[1][0] = top;
        c1[1][0] = c0[1][1] = c1[1][1] = 0.f;
        const float s = b > 0.f ? b : a;
        const float q1 = s * top;
        const float r = __fmaf_rn(-q1, a, s) * top;
        S1 = (unsigned long long)max(__float2ll_rn(q1 * 281474976710656.f) + __float2ll_rn(r * 281474976710656.f), 0ll);
        ua = ln.ua;
        hp = ln.hp;
        has_last = ln.has_last;
    }

    // A line exactly along an axis (kDeg0Axis): all rows alike, the footprint a
    // rectangle; where its edges fall on two nodes (tie), the midpoint value on
    // both.  (4 views of 512 x 512 pixels, one of them along an axis: forward 27
    // us; with such rows walked one by one in global memory 87.)
    __device__ __forceinline__ void load_axis(const LaneLine &ln, bool tie)
    {
        const float top = 1.0f / ln.a;
        c0[0][0] = c0[0][1] = tie ? 0.5f * top : top;
        c0[1][0] = c0[1][1] = c1[0][0] = c1[0][1] = c1[1][0] = c1[1][1] = 0.f;
        S1 = 1ull << kFrac0;   // interval 0 throughout
        ua = ln.ua;
        hp = ln.hp;
        has_last = tie;
    }

    __device__ __forceinline__ void row(long long W, float *sp, f2 &acc) const
    {
        const unsigned long long x = (unsigned long long)W & ((1ull << kFrac0) - 1ull);
        const bool up = x >= S1, on_last = has_last && !up;   // candidate 1 ends with interval 0
        const float t = (float)(x - (up ? S1 : 0ull) + 1ull) * ua;
        const float p0 = __fmaf_rn(up ? c1[1][0] : c1[0][0], t, up ? c0[1][0] : c0[0][0]);
        const float p1 = __fmaf_rn(up ? c1[1][1] : c1[0][1], t, up ? c0[1][1] : c0[0][1]);
        if constexpr (ADJ) {
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
// One of the two images the strips are cut from: nodes [row][column] with the
// lines' major axis along the rows; rows of ld floats, a multiple of 4, the
// columns from Nq on zero (forward) or ignored (adjoint).
struct Image {
    const float *src;
    float *dst;
    int Nr, Nq, ld;
};

// The rows of this lane's line on a strip, blocks [b0, b1) (none where the
// lane has no line): loads the line's polynomials and walks.  n: the columns of
// the warp's runs.
template <int KIND, bool ADJ, bool FIX>
__device__ __forceinline__ void strip_line(int n, const LaneLine &ln, const LineHdr &H, const float *tab, const Strip &st,
                                           int b0, int b1, float &hi, float &lo)
{
    if constexpr (KIND == 0) {
        PixelRows<ADJ> R;
        LaneLine l = ln;
        if (H.flags & kDeg0Axis) {
            const float s0[1] = {H.a};   // b = 0: one interval
            const RowEval e = row_eval<0>(H, s0, 1.0f / H.a, H.r_begin);
            R.load_axis(ln, e.tie);
            l.q_first = (e.tie ? e.q0 - 1 : e.q0) + (int)(ln.W0 >> kFrac0);
        } else {
            const float b = fabsf(H.rho_hi + H.rho_lo);
            R.load(ln, b < 1e-30f ? 0.f : b, H.a_corr);
        }
        walk_blocks(R, l, st, b0, b1, ADJ, hi, lo);
    } else if constexpr (KIND == kKindBox) {
        switch (n) {
        case 6: { BoxRows<6, ADJ, FIX> R; R.load(ln, tab); walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo); break; }
        case 5: { BoxRows<5, ADJ, FIX> R; R.load(ln, tab); walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo); break; }
        case 4: { BoxRows<4, ADJ, FIX> R; R.load(ln, tab); walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo); break; }
        default: { BoxRows<3, ADJ, FIX> R; R.load(ln, tab); walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo); break; }
        }
    } else if constexpr (KIND == 1) {
        SplineRows<1, 2, ADJ, FIX> R;
        R.load(ln);
        walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo);
    } else {
        if (n > 2 * KIND + 1) {
            SplineRows<KIND, KIND + 1, ADJ, FIX> R;
            R.load(ln);
            walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo);
        } else {
            SplineRows<KIND, KIND, ADJ, FIX> R;
            R.load(ln);
            walk_blocks(R, ln, st, b0, b1, ADJ, hi, lo);
        }
    }
}

// Columns of a line's runs as strip_line takes them, and how many of them lie
// before the column of the position's high part.  B-splines of degree >= 1:
// every (j + c) a +- v that can lie in the support, (j + c) a - a/2 < w, on both
// sides; degree 0 and the box-spline: the slots K of u_0 + i a.
template <int KIND>
__device__ __forceinline__ int run_columns(const LineHdr &H, float b)
{
    if constexpr (KIND == 1) return 4;
    else if constexpr (KIND == 2) return 3.f * b <= 2.f * H.a ? 5 : 7;
    else if constexpr (KIND == 3) return 2.f * b <= H.a ? 6 : 8;
    else return max(H.K, KIND == 0 ? 2 : 3);
}
template <int KIND>
__device__ __forceinline__ int run_lead(int n) { return KIND >= 1 && KIND <= 3 ? n / 2 : 0; }

// Adds the accumulated strip into the image by 16-byte reductions.
__device__ __forceinline__ void strip_flush(const Strip &st, int S0, const Image &im, bool fixed, float finv)
{
    const int nch = st.pitch / 4;
    const unsigned inv = 0xffffffffu / (unsigned)nch + 1u;   // i / nch = umulhi(i, inv) for every strip index
    for (int i = threadIdx.x; i < st.rows * nch; i += kThreads) {
        const int rr = (int)__umulhi((unsigned)i, inv), q = st.first(rr) + 4 * (i - rr * nch);
        const int4 n4 = reinterpret_cast<const int4 *>(st.p)[i];
        float4 v = make_float4(__int_as_float(n4.x), __int_as_float(n4.y), __int_as_float(n4.z), __int_as_float(n4.w));
        if (fixed) v = make_float4((float)n4.x * finv, (float)n4.y * finv, (float)n4.z * finv, (float)n4.w * finv);
        if ((unsigned)q < (unsigned)im.ld && S0 + rr < im.Nr && (v.x != 0.f || v.y != 0.f || v.z != 0.f || v.w != 0.f))
            asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(im.dst + (size_t)(S0 + rr) * im.ld + q),
                         "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                         : "memory");
    }
}

// Stages the strip's coefficients with asynchronous 16-byte copies, zeros
// outside the image (chunks are wholly inside or outside: ld and chunk starts
// are multiples of 4).
__device__ __forceinline__ void strip_stage(const Strip &st, int S0, const Image &im)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(st.p);
    const int nch = st.pitch / 4;
    const unsigned inv = 0xffffffffu / (unsigned)nch + 1u;
    for (int i = threadIdx.x; i < st.rows * nch; i += kThreads) {
        const int rr = (int)__umulhi((unsigned)i, inv), q = st.first(rr) + 4 * (i - rr * nch);
        const bool in = (unsigned)q < (unsigned)im.ld && S0 + rr < im.Nr;
        cp_async16(sa + 16 * i, in ? im.src + (size_t)(S0 + rr) * im.ld + q : im.src, in);
    }
}

// floor(a / b) for b > 0.
__device__ __forceinline__ int floor_div(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// The arguments of one strip projection.  img: the image (forward, read) and
// the scratch images the adjoint adds to, as stored (0) and transposed (1).
struct StripArgs {
    GridDev g;
    LinesDev L;
    const LineHdr *hdr;
    const float *center;       // centre records (B-splines of degree 1..3)
    const float *tabs;         // footprint tables (box-spline)
    const float *src[2];
    float *dst[2];
    float *sino;
    const longlong2 *rec;      // row records, or NULL
    int cpv;                   // chunks per view
};

// Forward (ADJ false): sino[line] = h sum c phi.  Adjoint (ADJ true): adds
// h sino[line] phi to dst[0] (vertical lines) or dst[1] (horizontal lines, the
// transposed image).
// One chunk (view v, bins j0..j0+31) of one instance; smem is the CTA's
// dynamic shared memory (kSmemBytes).
// FM (adjoint only) picks the chunks a call runs: kFmFixed only those that
// accumulate in fixed point, kFmFloat only the others (non-finite values, or
// a scale outside the safe range; see the top of the file), with float
// strips; returns whether the chunk was one of them.  The forward takes
// kFmAll.
template <int KIND, bool ADJ, int FM = kFmAll>
__device__ __forceinline__ bool strip_chunk(unsigned char *smem, const StripArgs &A, int chunk)
{
    static_assert(!ADJ || FM != kFmAll, "the adjoint runs as fixed-point and float launches");
    constexpr bool FIX = ADJ && FM == kFmFixed;
    constexpr int F = KIND == 0 ? kFrac0 : 32;
    constexpr bool kCenter = KIND >= 1 && KIND <= 3;
    const GridDev &g = A.g;
    const LinesDev &L = A.L;
    float *strip = reinterpret_cast<float *>(smem);
    float *rec_s = reinterpret_cast<float *>(smem + kStripBytes);
    LineHdr *hdr_s = reinterpret_cast<LineHdr *>(smem + kStripBytes + kRecBytes);
    float2 *part_s = reinterpret_cast<float2 *>(smem + kStripBytes + kRecBytes + kHdrBytes);   // [warp][line]
    int *off_s = reinterpret_cast<int *>(smem + kStripBytes + kRecBytes + kHdrBytes + kPartBytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int v = chunk / A.cpv, cb = chunk - v * A.cpv;
    const int j0 = cb * kChunk;
    const int64_t nd = chunk_bins(L);
    const int nl = (int)min((int64_t)kChunk, nd - j0);
    // position of the chunk's first line (in the sorted order for free lists),
    // and lane l's line in every warp (directions: one per view for parallel
    // beams, else one per line)
    const int64_t line0 = (int64_t)v * nd + j0;
    const int my_line = lane < nl ? (L.order ? L.order[line0 + lane] : (int)(line0 + lane)) : 0;
    const bool shared_dir = L.kind == SP_LINES_PARALLEL;

    // The adjoint's values, and the chunk's fixed-point scale (a power of two;
    // see the top of the file).  Non-finite values, or values so large or
    // small that it leaves a safe exponent range, keep the float reductions.
    float pv = 0.f, fscale = 1.f, finv = 1.f;
    if constexpr (ADJ) {
        if (lane < nl) pv = A.sino[my_line];
        if constexpr (adj_mode<KIND>() == kFmFixed) {
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
    }

    // the chunk's line records and centre records into shared memory
    static_assert(kChunk * 4 <= kThreads && sizeof(LineHdr) == 64, "one pass over the chunk's line records");
    {
        const int src = __shfl_sync(0xffffffffu, my_line, (threadIdx.x >> 2) & 31);
        if ((int)threadIdx.x < nl * 4)
            reinterpret_cast<int4 *>(hdr_s)[threadIdx.x] =
                reinterpret_cast<const int4 *>(A.hdr + src)[threadIdx.x & 3];
    }
    float my_b = 0.f;
    if constexpr (kCenter) {
        my_b = A.center[(shared_dir ? (int64_t)v : (int64_t)my_line) * kCenterFloats + kCenterB];
        const int nt = shared_dir ? 1 : nl;
        constexpr int kCh = kCenterFloats / 4;
        const unsigned ba = (unsigned)__cvta_generic_to_shared(rec_s);
        for (int i0 = warp * 32; i0 < nt * kCh; i0 += kThreads) {
            const int i = i0 + lane, li = min(i / kCh, kChunk - 1);
            const int ti = shared_dir ? v : __shfl_sync(0xffffffffu, my_line, li);
            if (i < nt * kCh) cp_async16(ba + 16 * i, A.center + (int64_t)ti * kCenterFloats + 4 * (i - li * kCh));
        }
    }
    if (!ADJ) part_s[warp * kChunk + lane] = make_float2(0.f, 0.f);
    __syncthreads();

    // this lane's line: its position in row 0, and the step per row
    bool mine = false, mine_vert = false;
    long long my_W = 0, my_step = 0;
    int my_n = 0;
    if (lane < nl) {
        const LineHdr &H = hdr_s[lane];
        mine = !(H.flags & kEmpty) && H.r_end > H.r_begin && (!ADJ || pv != 0.f);
        mine_vert = (H.flags & kVert) != 0;
        if (mine) {
            if (A.rec) {
                const longlong2 t = A.rec[my_line];
                my_W = t.x;
                my_step = t.y;
            } else {
                row_stepping<KIND>(H, my_b, my_W, my_step);
            }
            my_n = run_columns<KIND>(H, my_b);
        }
    }
    for (int axis = 0; axis < 2; ++axis) {
        const bool vert = axis == 0;
        const unsigned mask = __ballot_sync(0xffffffffu, mine && mine_vert == vert);
        if (mask == 0u) continue;
        Image im;
        im.src = A.src[axis];
        im.dst = A.dst[axis];
        im.Nr = vert ? g.ny : g.nx;
        im.Nq = vert ? g.nx : g.ny;
        im.ld = image_ld(im.Nq);
        // Groups: aligned spans of lines [ga, ga + len), len a power of two,
        // whose runs fit a strip row (and, where the run is the line's slots,
        // differ by at most one); others are halved.  Every warp finds the
        // same ones.
        for (int ga = 0, len = kChunk; ga < kChunk; ga += len, len = ga & -ga) {
            auto in_span = [&](int a, int n) { return mask & ((n >= 32 ? 0xffffffffu : (1u << n) - 1u) << a); };
            if (in_span(ga, len) == 0u) continue;
            int R0, R1, la, lb, n, width;
            for (;;) {
                // a half without lines is left out
                while (len > 1 && in_span(ga + (len >> 1), len >> 1) == 0u) len >>= 1;
                const bool in = (in_span(ga, len) >> lane) & 1u;
                // row range of the group in whole blocks, and the lowest and
                // highest column of its lines in the first and the last row.
                // The position's column lies within one above the line's, and
                // lines are straight, so between the two rows the columns stay
                // within one of the chords through the extremes.
                R0 = __reduce_min_sync(0xffffffffu, in ? hdr_s[lane].r_begin : INT_MAX) & -kRowBlock;
                R1 = (__reduce_max_sync(0xffffffffu, in ? hdr_s[lane].r_end : INT_MIN) + kRowBlock - 1) & -kRowBlock;
                const int qa = in ? hdr_s[lane].q_ref - (int)((my_W + R0 * my_step) >> F) : 0;
                const int qb = in ? hdr_s[lane].q_ref - (int)((my_W + (R1 - 1) * my_step) >> F) : 0;
                la = __reduce_min_sync(0xffffffffu, in ? qa : INT_MAX);
                lb = __reduce_min_sync(0xffffffffu, in ? qb : INT_MAX);
                const int ha = __reduce_max_sync(0xffffffffu, in ? qa : INT_MIN);
                const int hb = __reduce_max_sync(0xffffffffu, in ? qb : INT_MIN);
                n = __reduce_max_sync(0xffffffffu, in ? my_n : 0);
                const int nmin = __reduce_min_sync(0xffffffffu, in ? my_n : INT_MAX);
                // 3 columns below the lowest run, 3 beyond the highest, 3 for
                // the start rounded down to a multiple of 4
                width = (max(ha - la, hb - lb) + n + 9 + 3) & ~3;
                if (len == 1 || (width <= kMaxWidth && (kCenter || n - nmin <= 1))) break;
                len >>= 1;
                if (in_span(ga, len) == 0u) ga += len;
            }

            // this lane's line of the group (groups of fewer than 32 lines:
            // several lanes per line, on consecutive rows)
            const int li = ga + (lane & (len - 1)), parts = kChunk / len, lead = run_lead<KIND>(n);
            const bool on = in_span(li, 1) != 0u;
            const int lj = on ? li : __ffs(in_span(ga, len)) - 1;   // (a lane without one looks at another's)
            const LineHdr &H = hdr_s[lj];
            LaneLine ln;
            ln.Wstep = __shfl_sync(0xffffffffu, my_step, lj);
            const long long W_row0 = __shfl_sync(0xffffffffu, my_W, lj);
            ln.q_first = H.q_ref - lead;
            ln.a = H.a;
            ln.ua = H.a * (F == 32 ? 2.3283064365386963e-10f : 3.5527136788005009e-15f);
            ln.w_sup = 0.5f * H.two_w;
            ln.hp = ADJ ? g.h * __shfl_sync(0xffffffffu, pv, lj) * fscale : 0.f;
            ln.rec = rec_s + (shared_dir ? 0 : lj) * kCenterFloats;
            ln.has_last = __shfl_sync(0xffffffffu, my_n, lj) >= n && H.K >= n;
            {
                // 2w - (K - 1) a in units of a 2^-32
                const float end = H.two_w / H.a - (float)(H.K - 1);
                ln.x_end = end >= 1.f ? 0xffffffffu : (unsigned)(fmaxf(end, 0.f) * 4294967296.f);
            }
            const float *tab = nullptr;
            if constexpr (KIND == kKindBox)
                tab = A.tabs + (shared_dir ? (int64_t)v : (int64_t)__shfl_sync(0xffffffffu, my_line, lj)) * kTabFloats;

            Strip st;
            st.p = strip;
            st.off = off_s;
            st.pitch = width;
            const int span = max(R1 - 1 - R0, 1);
            st.slope = floor_div((lb - la) * (1 << kSlopeBits), span);
            // slabs of equal height that the strip can hold
            const int most = min(kStripFloats / width, kSlabRows) & -kRowBlock;
            const int slabs = (R1 - R0 + most - 1) / most;
            const int per = ((R1 - R0 + slabs - 1) / slabs + kRowBlock - 1) & -kRowBlock;
            float hi = 0.f, lo = 0.f;
            for (int S0 = R0; S0 < R1; S0 += per) {
                st.rows = min(per, R1 - S0);
                st.c0 = la - lead + floor_div((lb - la) * (S0 - R0), span) - 3;
                __syncthreads();   // the strip's last readers are done
                for (int rr = threadIdx.x; rr < st.rows; rr += kThreads) st.off[rr] = rr * width - st.first(rr);
                if constexpr (ADJ) {
                    float4 *s4 = reinterpret_cast<float4 *>(strip);
                    for (int i = threadIdx.x; i < st.rows * width / 4; i += kThreads) s4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                } else {
                    strip_stage(st, S0, im);
                }
                cp_async_wait_all();   // the strip's copies, and the centre records'
                __syncthreads();
                const int nb = st.rows / kRowBlock, unit = warp * parts + lane / len, units = kWarps * parts;
                const int b0 = nb * unit / units, b1 = on ? nb * (unit + 1) / units : b0;
                ln.W0 = W_row0 + S0 * ln.Wstep;
                strip_line<KIND, ADJ, FIX>(n, ln, H, tab, st, b0, b1, hi, lo);
                if constexpr (ADJ) {
                    __syncthreads();
                    strip_flush(st, S0, im, FIX, finv);
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
            // (an infinite sum leaves no finite remainder)
            A.sino[my_line] = g.h * (isfinite(lo) ? hi + lo : hi);
        }
    }
    return true;
}

// One CTA per chunk.  The adjoint runs the fixed-point chunks (FM kFmFixed:
// nearly all) and appends the others to defer[2..] (count defer[0]) for
// strip_float_kernel.
template <int KIND, bool ADJ, int FM = kFmAll>
__global__ void __launch_bounds__(kThreads, kCtas) strip_kernel(const __grid_constant__ StripArgs A, unsigned *defer)
{
    chain_begin();
    extern __shared__ __align__(16) unsigned char smem[];
    const bool ran = strip_chunk<KIND, ADJ, FM>(smem, A, (int)blockIdx.x);
    if (FM == kFmFixed && !ran && threadIdx.x == 0) defer[2 + atomicAdd(defer, 1u)] = blockIdx.x;
}

// The deferred adjoint chunks (float strip accumulators): a small persistent
// grid over defer[2 .. 2 + defer[0]), defer[1] its counter.
template <int KIND>
__global__ void __launch_bounds__(kThreads, kCtas) strip_float_kernel(const __grid_constant__ StripArgs A, unsigned *defer)
{
    chain_begin();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned cur;
    const unsigned n = defer[0];
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) cur = atomicAdd(defer + 1, 1u);
        __syncthreads();
        if (cur >= n) break;
        strip_chunk<KIND, true, kFmFloat>(smem, A, (int)defer[2 + cur]);
    }
}

// One instance of the persistent kernel's work queue.
struct StripJob {
    StripArgs A;
    long long chunk0;   // its first chunk in the queue
};

// Persistent kernel over the chunks of several instances of one kind (B-spline
// degree, or box-spline): each
// CTA takes the next chunk from one counter (atomicAdd; no CTA waits on
// another) and runs it with its instance's parameters, until every chunk is
// taken.  Instance k owns chunks [jobs[k].chunk0, jobs[k + 1].chunk0).  The
// adjoint runs the fixed-point chunks and appends the others to defer[]
// (count *defer_n) for strip_queue_float_kernel, as the per-instance adjoint
// does with its second launch.  (One kernel per degree: a kernel holding all
// three degrees spilled over a hundred bytes per thread.)
__device__ __forceinline__ const StripJob *queue_job(const StripJob *jobs, int njobs, long long c)
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
__global__ void __launch_bounds__(kThreads, kCtas)
strip_queue_kernel(const StripJob *jobs, int njobs, long long total, unsigned long long *counter,
                   long long *defer, unsigned long long *defer_n)
{
    chain_begin();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long cur;
    for (;;) {
        __syncthreads();   // the previous chunk's last readers of shared memory are done
        if (threadIdx.x == 0) cur = (long long)atomicAdd(counter, 1ull);
        __syncthreads();
        const long long c = cur;
        if (c >= total) break;
        const StripJob *J = queue_job(jobs, njobs, c);
        constexpr int FM = ADJ ? adj_mode<KIND>() : kFmAll;
        const bool ran = strip_chunk<KIND, ADJ, FM>(smem, J->A, (int)(c - J->chunk0));
        if (FM == kFmFixed && !ran && threadIdx.x == 0) defer[atomicAdd(defer_n, 1ull)] = c;
    }
}

// The deferred adjoint chunks (float strip accumulators), persistent likewise.
template <int KIND>
__global__ void __launch_bounds__(kThreads, kCtas)
strip_queue_float_kernel(const StripJob *jobs, int njobs, const long long *defer,
                         const unsigned long long *defer_n, unsigned long long *counter)
{
    chain_begin();
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
        strip_chunk<KIND, true, kFmFloat>(smem, J->A, (int)(c - J->chunk0));
    }
}

template <int KIND>
cudaError_t launch_queue_t(bool adj, const StripJob *jobs, int njobs, int64_t total, unsigned long long *counter,
                           long long *defer, int64_t grid, int sms, cudaStream_t s)
{
    cudaError_t e;
    if (adj) {
        e = cudaFuncSetAttribute(strip_queue_kernel<KIND, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kSmemBytes);
        if (e != cudaSuccess) return e;
        launch_chained(strip_queue_kernel<KIND, true>, (unsigned)grid, kThreads, kSmemBytes, s, jobs, njobs,
                       (long long)total, counter, defer, counter + 1);
        e = cudaGetLastError();
        if constexpr (adj_mode<KIND>() == kFmFixed) {
            // the deferred chunks are few (non-finite or extreme sinogram values): a small grid
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(strip_queue_float_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kSmemBytes);
            if (e != cudaSuccess) return e;
            launch_chained(strip_queue_float_kernel<KIND>, (unsigned)(grid < sms ? grid : sms), kThreads, kSmemBytes, s,
                           jobs, njobs, defer, counter + 1, counter + 2);
            e = cudaGetLastError();
        }
        return e;
    }
    e = cudaFuncSetAttribute(strip_queue_kernel<KIND, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kSmemBytes);
    if (e != cudaSuccess) return e;
    launch_chained(strip_queue_kernel<KIND, false>, (unsigned)grid, kThreads, kSmemBytes, s, jobs, njobs, (long long)total,
                   counter, nullptr, nullptr);
    return cudaGetLastError();
}

// The forward's images: the coefficients transposed, and (plain not NULL) as
// stored, with rows padded by zeros to a multiple of 4.
__global__ void stage_images_kernel(const float *in, float *plain, float *trans,
                                    int nx, int ny)
{
    chain_begin();
    __shared__ float tile[32][33];
    const int bx = blockIdx.x * 32, by = blockIdx.y * 32, ldx = image_ld(nx), ldy = image_ld(ny);
    for (int y = threadIdx.y; y < 32; y += 8) {
        const int i = bx + threadIdx.x, j = by + y;
        const float v = (i < nx && j < ny) ? in[(size_t)j * nx + i] : 0.f;
        tile[y][threadIdx.x] = v;
        if (plain && i < ldx && j < ny) plain[(size_t)j * ldx + i] = v;
    }
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += 8) {
        const int j = by + threadIdx.x, i = bx + y;
        if (i < nx && j < ldy) trans[(size_t)i * ldy + j] = tile[threadIdx.x][y];
    }
}

// out[j][i] = plain[j][i] + trans[i][j] (padded rows in, plain rows out)
__global__ void join_images_kernel(const float *plain, const float *trans, float *out,
                                   int nx, int ny)
{
    chain_begin();
    __shared__ float tile[32][33];
    const int bi = blockIdx.x * 32, bj = blockIdx.y * 32, ldx = image_ld(nx), ldy = image_ld(ny);
    for (int y = threadIdx.y; y < 32; y += 8) {
        const int i = bi + y, j = bj + threadIdx.x;
        if (i < nx && j < ny) tile[y][threadIdx.x] = trans[(size_t)i * ldy + j];
    }
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += 8) {
        const int j = bj + y, i = bi + threadIdx.x;
        if (i < nx && j < ny) out[(size_t)j * nx + i] = plain[(size_t)j * ldx + i] + tile[threadIdx.x][y];
    }
}

size_t image_bytes(int rows, int cols) { return (sizeof(float) * (size_t)rows * image_ld(cols) + 255) & ~(size_t)255; }

// The arguments of a strip projection.  Forward: img is read, as it is where its
// rows are whole 16-byte chunks.  scratch: strip_scratch_bytes.
StripArgs make_args(const GridDev &g, const LinesDev &L, const LineHdr *hdr, const float *center, const float *tabs,
                    const float *img, void *scratch, float *sino, const longlong2 *rec)
{
    StripArgs A;
    A.g = g;
    A.L = L;
    A.hdr = hdr;
    A.center = center;
    A.tabs = tabs;
    float *plain = static_cast<float *>(scratch);
    float *trans = reinterpret_cast<float *>(static_cast<char *>(scratch) + image_bytes(g.ny, g.nx));
    A.dst[0] = plain;
    A.dst[1] = trans;
    const bool direct = img && g.nx % 4 == 0 && (reinterpret_cast<uintptr_t>(img) & 15) == 0;
    A.src[0] = direct ? img : plain;
    A.src[1] = trans;
    A.sino = sino;
    A.rec = rec;
    A.cpv = (int)((chunk_bins(L) + kChunk - 1) / kChunk);
    return A;
}

// Before a projection: the forward's images, or the adjoint's cleared ones (and
// the `words` words behind them); after the adjoint: its result.
cudaError_t launch_images(const StripArgs &A, const float *img, cudaStream_t s)
{
    const dim3 tb(32, 8), tg((A.g.nx + 31) / 32, (image_ld(A.g.ny) + 31) / 32);
    launch_chained(stage_images_kernel, tg, tb, 0, s, img, A.src[0] == img ? nullptr : A.dst[0], A.dst[1], A.g.nx, A.g.ny);
    return cudaGetLastError();
}

cudaError_t launch_join(const StripArgs &A, float *out, cudaStream_t s)
{
    const dim3 tb(32, 8), tg((A.g.nx + 31) / 32, (A.g.ny + 31) / 32);
    launch_chained(join_images_kernel, tg, tb, 0, s, A.dst[0], A.dst[1], out, A.g.nx, A.g.ny);
    return cudaGetLastError();
}

template <int KIND>
cudaError_t launch_strip_t(const StripArgs &A, bool adj, unsigned *defer, cudaStream_t s)
{
    const unsigned grid = (unsigned)(chunk_views(A.L) * A.cpv);
    cudaError_t e;
    if (!adj) {
        e = cudaFuncSetAttribute(strip_kernel<KIND, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
        if (e != cudaSuccess) return e;
        launch_chained(strip_kernel<KIND, false>, grid, kThreads, kSmemBytes, s, A, nullptr);
        return cudaGetLastError();
    }
    constexpr int FM = adj_mode<KIND>();
    e = cudaFuncSetAttribute(strip_kernel<KIND, true, FM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    if (e != cudaSuccess) return e;
    launch_chained(strip_kernel<KIND, true, FM>, grid, kThreads, kSmemBytes, s, A, defer);
    e = cudaGetLastError();
    if constexpr (FM == kFmFixed) {
        // a small second launch for the chunks deferred to float strips
        int dev = 0, sms = 0;
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(strip_float_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        launch_chained(strip_float_kernel<KIND>, grid < (unsigned)sms ? grid : (unsigned)sms, kThreads, kSmemBytes, s, A, defer);
        e = cudaGetLastError();
    }
    return e;
}

cudaError_t launch_strip(const StripArgs &A, bool adj, unsigned *defer, cudaStream_t s)
{
    if (strip_needs_order(A.L) && !A.L.order) return cudaErrorInvalidValue;   // free lists need their order
    switch (strip_kind(A.g)) {
    case 0: return launch_strip_t<0>(A, adj, defer, s);
    case 1: return launch_strip_t<1>(A, adj, defer, s);
    case 2: return launch_strip_t<2>(A, adj, defer, s);
    case 3: return launch_strip_t<3>(A, adj, defer, s);
    default: return launch_strip_t<kKindBox>(A, adj, defer, s);
    }
}

}  // namespace

int strip_queue_kind(const GridDev &g) { return strip_kind(g); }

int64_t strip_chunk_count(const LinesDev &L) { return chunk_views(L) * ((chunk_bins(L) + kChunk - 1) / kChunk); }

size_t strip_job_bytes(int count) { return sizeof(StripJob) * (size_t)count; }

void make_strip_job(void *jobs, int k, const GridDev &g, const LinesDev &L, const LineHdr *hdr, const float *center,
                    const float *tabs, const float *img, float *sino, void *scratch, long long chunk0)
{
    StripJob *J = static_cast<StripJob *>(jobs) + k;
    J->A = make_args(g, L, hdr, center, tabs, img, scratch, sino, nullptr);
    J->chunk0 = chunk0;
}

cudaError_t launch_strip_pre(const void *jobs, int k, const float *img, cudaStream_t s)
{
    const StripArgs &A = static_cast<const StripJob *>(jobs)[k].A;
    if (img) return launch_images(A, img, s);
    return cudaMemsetAsync(A.dst[0], 0, strip_scratch_bytes(A.g), s);
}

cudaError_t launch_strip_post(const void *jobs, int k, float *out, cudaStream_t s)
{
    return launch_join(static_cast<const StripJob *>(jobs)[k].A, out, s);
}

cudaError_t launch_strip_queue(int kind, bool adj, const void *jobs_dev, int job0, int njobs, int64_t total,
                               unsigned long long *counter, long long *defer, cudaStream_t s)
{
    if (njobs <= 0 || total <= 0) return cudaSuccess;
    const StripJob *jobs = static_cast<const StripJob *>(jobs_dev) + job0;
    if (kind < 0 || kind > kKindBox || (adj && !defer)) return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaMemsetAsync(counter, 0, 3 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    int64_t grid = kCtas * (int64_t)sms;   // resident at once
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

size_t strip_scratch_bytes(const GridDev &g) { return image_bytes(g.ny, g.nx) + image_bytes(g.nx, g.ny); }

cudaError_t launch_fwd_strip(const GridDev &g, const LinesDev &L, const LineHdr *hdr, const float *center,
                             const float *tabs, const float *coef, void *scratch, float *sino, cudaStream_t s,
                             const longlong2 *rec)
{
    const StripArgs A = make_args(g, L, hdr, center, tabs, coef, scratch, sino, rec);
    cudaError_t e = launch_images(A, coef, s);
    return e == cudaSuccess ? launch_strip(A, false, nullptr, s) : e;
}

cudaError_t launch_adj_strip(const GridDev &g, const LinesDev &L, const LineHdr *hdr, const float *center,
                             const float *tabs, const float *sino, void *scratch, float *coef_out, cudaStream_t s,
                             const longlong2 *rec)
{
    const StripArgs A = make_args(g, L, hdr, center, tabs, nullptr, scratch, const_cast<float *>(sino), rec);
    // the images and, right behind them, the deferred list's count and counter
    unsigned *defer = reinterpret_cast<unsigned *>(static_cast<char *>(scratch) + strip_scratch_bytes(g));
    cudaError_t e = cudaMemsetAsync(scratch, 0, strip_scratch_bytes(g) + 2 * sizeof(unsigned), s);
    if (e == cudaSuccess) e = launch_strip(A, true, defer, s);
    return e == cudaSuccess ? launch_join(A, coef_out, s) : e;
}

cudaError_t launch_row_records(const GridDev &g, const LinesDev &L, const LineHdr *hdr, const float *center,
                               longlong2 *rec, cudaStream_t s)
{
    if (L.m <= 0) return cudaSuccess;
    const unsigned nb = (unsigned)((L.m + 255) / 256);
    const int per = L.kind == SP_LINES_PARALLEL ? L.n_det : 1;
    switch (strip_kind(g)) {
    case 1: launch_chained(row_record_kernel<1>, nb, 256, 0, s, hdr, center, per, L.m, rec); break;
    case 2: launch_chained(row_record_kernel<2>, nb, 256, 0, s, hdr, center, per, L.m, rec); break;
    case 3: launch_chained(row_record_kernel<3>, nb, 256, 0, s, hdr, center, per, L.m, rec); break;
    case kKindBox: launch_chained(row_record_kernel<kKindBox>, nb, 256, 0, s, hdr, center, per, L.m, rec); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace spx
