// FP32 spectral kernels for the acoustic correlation A and its transpose
// (Sec. 2.3.3, Eq. acoustic-full-forward), with the switching map P and its
// transpose folded in.
//
// A correlates every state image with a k x k kernel per (depth, sample).  On
// a zero-padded periodic grid of Ly x Lx >= (Y + r) x (X + r) points the
// lateral sums become one small product per lateral frequency f,
//   u^_m[t](f) = sum_j K^[j][t](f) b^_m[j](f),   b^_m = sum_p S[m][p] c^_p,
// exact in real arithmetic.  The direct sums of the largest workload are 741
// GFLOP (31 x 31 taps); here they are 4 GFLOP of products and 1 GFLOP of
// transforms, in FP32 throughout (error 1e-7 to 2e-7 against 64 bits where the
// direct FP32 sums, chains of 10^4 products, have 4e-7 to 5e-6).  H^T H of that
// workload: 0.60 ms; the direct sums took 130 + 130 ms on the CUDA cores and, in
// BF16 on the tensor cores at 98% of their peak over the padded band, 2.2 + 2.4 ms.
//
// Structure used:
//  * Two neighbouring channels (depths or samples) are the real and imaginary
//    part of one complex image, which is how a float2 of the channel-fastest
//    layout reads: no packing pass and no real-transform post-processing.  The
//    product unpacks them from Z(f) and conj Z(-f), which it needs anyway, and
//    so runs on half of the frequency plane.
//  * The arrival time grows with depth: over all taps a depth reaches a run of
//    16 to 50% of the samples.  K^ is stored per group of 8 output channels
//    with the hull of contracted channels that reach it (43% of the dense
//    size on the largest workload), in the order in which a warp reads it.
//  * P and P^T do not depend on the lateral position, so they commute with the
//    transform: P images are transformed, not Q state images (P^T likewise),
//    except where the operands are rounded to BF16 per state first.
//  * A length L = R1 R2 transform is two passes of register DFTs of radix up
//    to 16 with one exchange through shared memory; lanes run over channel
//    pairs, so that global and shared accesses are contiguous in both axes.
//  * Scans wider than the largest transform are cut into overlapping tiles
//    (L - 2 r outputs each).
//
// A transform would spread an infinity, a NaN or a huge value (a mask of the
// type's lowest one) of the input over the whole image.  The first pass of A and
// of A^T therefore takes every value that is not below 2^64 out, as a zero, and
// marks its scan position; the last pass adds such values' own terms to the
// outputs within the support of a marked position.  So they reach the outputs
// whose sums contain them and no others.  Without marks that costs a comparison per
// value; one iteration of the largest workload (k = 31, 128^2 x 96, 0.89 ms) takes
// 1.5 ms with NaNs or infinities at one pixel of the measurements and 2.6 ms with
// nothing else in them.  Finite values from 2^64 cost the direct sums over what they
// reach, and a solve spreads them: 1.2 s where one pixel holds 1e30.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <limits>

#include "swopt_internal.cuh"

namespace swopt {
namespace {

constexpr int kFB = 8;           // frequencies per block of the spectral product
constexpr int kOG = 8;           // output channels per group of the banded kernel
constexpr int kMaxFftThreads = 256;
constexpr int kSpecThreads = 256;
constexpr size_t kSpecSmem = 220 * 1024;  // most dynamic shared memory of the product

// ---------------------------------------------------------------------------
// Register DFTs
// ---------------------------------------------------------------------------
constexpr double kPi = 3.14159265358979323846;

constexpr double taylor_cos(double x)  // |x| <= pi
{
    double term = 1.0, s = 1.0;
    for (int i = 1; i < 16; ++i) {
        term *= -x * x / ((2.0 * i - 1.0) * (2.0 * i));
        s += term;
    }
    return s;
}

constexpr double taylor_sin(double x)
{
    double term = x, s = x;
    for (int i = 1; i < 16; ++i) {
        term *= -x * x / ((2.0 * i) * (2.0 * i + 1.0));
        s += term;
    }
    return s;
}

// exp(-2 pi i n / N), n < N
template <int N>
struct Roots {
    float re[N], im[N];
    constexpr Roots() : re(), im()
    {
        for (int n = 0; n < N; ++n) {
            const double a = 2.0 * kPi * (2 * n > N ? n - N : n) / N;
            re[n] = (float)taylor_cos(a);
            im[n] = (float)-taylor_sin(a);
        }
    }
};

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float re, float im)
{
    return make_float2(fmaf(a.x, re, -a.y * im), fmaf(a.x, im, a.y * re));
}

// S = -1: forward (exp(-...)), +1: inverse; unnormalised.
template <int R, int S>
struct Dft;

template <int S>
struct Dft<2, S> {
    static __device__ __forceinline__ void run(float2 (&v)[2])
    {
        const float2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    }
};

template <int S>
struct Dft<3, S> {
    static __device__ __forceinline__ void run(float2 (&v)[3])
    {
        constexpr float h = 0.866025403784438646763723170752936f;
        const float2 t = cadd(v[1], v[2]), d = csub(v[1], v[2]);
        const float2 m = make_float2(fmaf(-0.5f, t.x, v[0].x), fmaf(-0.5f, t.y, v[0].y));
        const float sx = -(float)S * h * d.y, sy = (float)S * h * d.x;  // S i h d
        v[0] = cadd(v[0], t);
        v[1] = make_float2(m.x + sx, m.y + sy);
        v[2] = make_float2(m.x - sx, m.y - sy);
    }
};

template <int S>
struct Dft<4, S> {
    static __device__ __forceinline__ void run(float2 (&v)[4])
    {
        const float2 a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
        const float2 c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
        const float2 e = make_float2(-(float)S * d.y, (float)S * d.x);  // S i d
        v[0] = cadd(a, c);
        v[2] = csub(a, c);
        v[1] = cadd(b, e);
        v[3] = csub(b, e);
    }
};

template <int S>
struct Dft<5, S> {
    static __device__ __forceinline__ void run(float2 (&v)[5])
    {
        constexpr float c1 = 0.309016994374947424102293417182819f;
        constexpr float c2 = -0.809016994374947424102293417182819f;
        constexpr float s1 = 0.951056516295153572116439333379382f;
        constexpr float s2 = 0.587785252292473129168705954639073f;
        const float2 t1 = cadd(v[1], v[4]), d1 = csub(v[1], v[4]);
        const float2 t2 = cadd(v[2], v[3]), d2 = csub(v[2], v[3]);
        const float2 a = make_float2(fmaf(c1, t1.x, fmaf(c2, t2.x, v[0].x)),
                                     fmaf(c1, t1.y, fmaf(c2, t2.y, v[0].y)));
        const float2 b = make_float2(fmaf(c2, t1.x, fmaf(c1, t2.x, v[0].x)),
                                     fmaf(c2, t1.y, fmaf(c1, t2.y, v[0].y)));
        const float2 p = make_float2(fmaf(s1, d1.x, s2 * d2.x), fmaf(s1, d1.y, s2 * d2.y));
        const float2 q = make_float2(fmaf(s2, d1.x, -s1 * d2.x), fmaf(s2, d1.y, -s1 * d2.y));
        const float2 ip = make_float2(-(float)S * p.y, (float)S * p.x);
        const float2 iq = make_float2(-(float)S * q.y, (float)S * q.x);
        v[0] = cadd(v[0], cadd(t1, t2));
        v[1] = cadd(a, ip);
        v[4] = csub(a, ip);
        v[2] = cadd(b, iq);
        v[3] = csub(b, iq);
    }
};

// R = A B by Cooley-Tukey: input n = n1 B + n2, output k = k1 + A k2.
template <int A, int B, int S>
__device__ __forceinline__ void dft_pair(float2 (&v)[A * B])
{
    constexpr Roots<A * B> w{};
    float2 t[B][A];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) {
#pragma unroll
        for (int n1 = 0; n1 < A; ++n1) t[n2][n1] = v[n1 * B + n2];
        Dft<A, S>::run(t[n2]);
#pragma unroll
        for (int k1 = 1; k1 < A; ++k1)
            if (n2 > 0)
                t[n2][k1] = cmul(t[n2][k1], w.re[n2 * k1], (S < 0 ? 1.f : -1.f) * w.im[n2 * k1]);
    }
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
        float2 x[B];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) x[n2] = t[n2][k1];
        Dft<B, S>::run(x);
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = x[k2];
    }
}

#define SW_DFT(R, A, B)                                                           \
    template <int S>                                                              \
    struct Dft<R, S> {                                                            \
        static __device__ __forceinline__ void run(float2 (&v)[R]) { dft_pair<A, B, S>(v); } \
    };
SW_DFT(6, 2, 3)
SW_DFT(8, 2, 4)
SW_DFT(9, 3, 3)
SW_DFT(10, 2, 5)
SW_DFT(12, 3, 4)
SW_DFT(16, 4, 4)
#undef SW_DFT

// Calls F<R> for the runtime radix (the ones that choose_length uses).
#define SW_RADIX(r, CALL)            \
    switch (r) {                     \
    case 2: { CALL(2); } break;      \
    case 3: { CALL(3); } break;      \
    case 4: { CALL(4); } break;      \
    case 5: { CALL(5); } break;      \
    case 6: { CALL(6); } break;      \
    case 8: { CALL(8); } break;      \
    case 9: { CALL(9); } break;      \
    case 10: { CALL(10); } break;    \
    case 12: { CALL(12); } break;    \
    default: { CALL(16); } break;    \
    }

// One axis of the periodic grid: length L = R1 R2, tiles of `out` positions
// (all of them in one tile when L >= n + r), input origin tile * out - pad.
struct FftAxis {
    int L, R1, R2, tiles, out, pad;
    const float2* tw;  // exp(-2 pi i n / L), n < L
};

// First pass of a transform: the radix-R1 DFTs over n1 of x[n1 R2 + n2],
// twiddled, into shared memory [k1 R2 + n2][lane].  load(v, n2, R2) fills
// v[n1] (all loads of a DFT are issued together).
template <int R, int S, class Load>
__device__ __forceinline__ void fft_pass1(const float2* __restrict__ tw, int R2, int n2,
                                          float2* sm, int lane, Load& load)
{
    float2 v[R];
    load(v, n2, R2);
    Dft<R, S>::run(v);
    sm[n2 * 32 + lane] = v[0];
#pragma unroll
    for (int k1 = 1; k1 < R; ++k1) {
        const float2 w = __ldg(tw + n2 * k1);
        sm[(k1 * R2 + n2) * 32 + lane] = cmul(v[k1], w.x, S < 0 ? w.y : -w.y);
    }
}

// Second pass: the radix-R2 DFTs over n2; store(v, k1, R1) takes the entries
// k = k1 + R1 k2.
template <int R, int S, class Store>
__device__ __forceinline__ void fft_pass2(int R1, int k1, const float2* sm, int lane, Store& store)
{
    float2 v[R];
#pragma unroll
    for (int n2 = 0; n2 < R; ++n2) v[n2] = sm[(k1 * R + n2) * 32 + lane];
    Dft<R, S>::run(v);
    store(v, k1, R1);
}

template <int S, class Load, class Store>
__device__ __forceinline__ void fft_line(const FftAxis& ax, float2* sm, Load load, Store store)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#define SW_P1(R)                                  \
    for (int n2 = warp; n2 < ax.R2; n2 += nw)     \
        fft_pass1<R, S>(ax.tw, ax.R2, n2, sm, lane, load)
    SW_RADIX(ax.R1, SW_P1)
#undef SW_P1
    if (S > 0) asm volatile("cp.async.wait_all;" ::: "memory");  // see fetch_marks
    __syncthreads();
#define SW_P2(R)                                  \
    for (int k1 = warp; k1 < ax.R1; k1 += nw)     \
        fft_pass2<R, S>(ax.R1, k1, sm, lane, store)
    SW_RADIX(ax.R2, SW_P2)
#undef SW_P2
}

// Values that the transforms do not take: infinities, NaNs and magnitudes from 2^64.
// (What is below leaves 2^64 of FP32's range to the sums of the transforms.)
constexpr float kHuge = 1.8446744e19f;

__device__ __forceinline__ bool huge(float v) { return !(fabsf(v) < kHuge); }

// True if any of the values is one.
template <int R>
__device__ __forceinline__ bool any_huge(const float2 (&v)[R])
{
    float top = 0.f;  // the largest magnitude, or a NaN
#pragma unroll
    for (int i = 0; i < R; ++i)
        asm("max.NaN.abs.f32 %0, %0, %1, %2;" : "+f"(top) : "f"(v[i].x), "f"(v[i].y));
    return huge(top);
}

// ---------------------------------------------------------------------------
// Shared arguments
// ---------------------------------------------------------------------------
struct FftShape {
    FftAxis y, x;
    int Y, X, Z, T, N, P, Q, ncyc, Twp, t0, k, r;
    int tiles;      // y.tiles * x.tiles
    int rows_in;    // rows of a tile that hold data before the y transform
    int rows_out;   // rows of a tile that hold results after the inverse y transform
    // Launches that serve a decision taken on the device (the refined solve's
    // increment or exact gradient): *sel != 0 takes the arguments marked 2.
    const int* sel;  // null: no second variant
    int round;      // operands rounded to BF16 (per state)
    int round2;
    const float* Sm;  // [Q][P][Z]
    const float* Kf;  // [Z][k][k][Twp] FP32 kernel (terms of the marked positions)
    const int4* ftab; // banded groups of the kernel: depths per eight samples,
    const int4* atab; // samples per eight depths (see Spec)
    // Marked positions of A's and of A^T's input.  A mark is the tag of the call, one
    // more than its predecessor's, so that nothing has to be cleared:
    // marks[0] the call's tag, marks[1 + which] the last one with a marked position,
    // then (from 4) [which][Y] the same per row and [which][Y][X] per position.
    unsigned* marks;
    const int* gate;
    int want;
};

// True if the launch takes its second variant (after grid_dependency()).
__device__ __forceinline__ bool second_variant(const FftShape& s)
{
    return s.sel != nullptr && *(volatile const int*)s.sel != 0;
}

__device__ __forceinline__ float round_if(float v, int round)
{
    return round ? __bfloat162float(__float2bfloat16_rn(v)) : v;
}

// b[m][pos][j] = sum_p S[m][p][j] c[p][pos][j] (the order of states_kernel)
__device__ __forceinline__ float state_value(const FftShape& s, const float* __restrict__ c, int m,
                                             size_t pos, int j)
{
    const size_t SZ = (size_t)s.Y * s.X * s.Z;
    float acc = 0.f;
    for (int p = 0; p < s.P; ++p)
        acc = fmaf(__ldg(s.Sm + ((size_t)m * s.P + p) * s.Z + j), c[p * SZ + pos * s.Z + j], acc);
    return acc;
}

// Measurements of state m folded over its pulses, window sample w (as fold_kernel).
__device__ __forceinline__ float folded(const FftShape& s, const float* __restrict__ y, int m,
                                        size_t pos, int w)
{
    const int t = s.t0 + w;
    float acc = 0.f;
    if (t < s.T)
        for (int n = m; n < s.N; n += s.ncyc) acc += y[((size_t)n * s.Y * s.X + pos) * s.T + t];
    return acc;
}

enum { MARK_A = 0, MARK_AT = 1 };

__device__ __forceinline__ unsigned* row_marks(const FftShape& s, int which)
{
    return s.marks + 4 + which * s.Y;
}

__device__ __forceinline__ unsigned* pos_marks(const FftShape& s, int which)
{
    return s.marks + 4 + 2 * s.Y + (size_t)which * s.Y * s.X;
}

// The call's tag: before its second launch has counted it (the first one marks
// with it), and from then on.
__device__ __forceinline__ unsigned next_tag(const FftShape& s) { return *(volatile unsigned*)s.marks + 1u; }
__device__ __forceinline__ unsigned this_tag(const FftShape& s) { return *(volatile unsigned*)s.marks; }

// The words marks[0 .. 2] into shared memory by the first thread: on their way during
// the first pass, waited for before its barrier, and in no register until they are read.
__device__ __forceinline__ void fetch_marks(const FftShape& s, uint4* words)
{
    if (threadIdx.x == 0)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         (unsigned)__cvta_generic_to_shared(words)),
                     "l"(s.marks)
                     : "memory");
}

// True if the input of A or A^T has marked positions in this call.
__device__ __forceinline__ bool any_mark(const uint4& words, int which)
{
    return words.x == (which == MARK_A ? words.y : words.z);
}

// The values of a thread's line entries, through shared-memory slots that only it
// uses, around `f`: a call on values in registers would have the compiler spill them
// on every path.
template <int R, class F>
__device__ __forceinline__ void through_slots(float2 (&v)[R], float2* slot, int stride, F f)
{
#pragma unroll
    for (int i = 0; i < R; ++i) slot[i * stride] = v[i];
    f();
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = slot[i * stride];
}

// Takes the huge values among line entries out, marking their positions (row y,
// columns x0 + i step).
__device__ __noinline__ void take_out(const FftShape& s, int which, unsigned tag, float2* slot, int stride,
                                      int R, int y, int x0, int step)
{
    for (int i = 0; i < R; ++i) {
        const float2 v = slot[i * stride];
        if (!huge(v.x) && !huge(v.y)) continue;
        pos_marks(s, which)[(size_t)y * s.X + x0 + i * step] = tag;
        row_marks(s, which)[y] = tag;
        s.marks[1 + which] = tag;
        slot[i * stride] = make_float2(huge(v.x) ? 0.f : v.x, huge(v.y) ? 0.f : v.y);
    }
}

// Calls f(dy, dx, position) for the marked positions that output (y, x) sums over
// (SIGN 1: A, at (y + dy - r, x + dx - r); -1: A^T, at (y - dy + r, x - dx + r)).
// f returns false to end.
template <int SIGN, class F>
__device__ __forceinline__ void marked_taps(const FftShape& s, int which, int y, int x, F f)
{
    const unsigned tag = this_tag(s);
    const unsigned *rows = row_marks(s, which), *cells = pos_marks(s, which);
    for (int dy = 0; dy < s.k; ++dy) {
        const int yy = y + SIGN * (dy - s.r);
        if (yy < 0 || yy >= s.Y || rows[yy] != tag) continue;
        for (int dx = 0; dx < s.k; ++dx) {
            const int xx = x + SIGN * (dx - s.r);
            if (xx < 0 || xx >= s.X || cells[(size_t)yy * s.X + xx] != tag) continue;
            if (!f(dy, dx, (size_t)yy * s.X + xx)) return;
        }
    }
}

// True if a row within the support of row y is marked.
__device__ __forceinline__ bool marked_near(const FftShape& s, int which, int y)
{
    const unsigned tag = this_tag(s);
    for (int yy = max(0, y - s.r); yy <= min(s.Y - 1, y + s.r); ++yy)
        if (row_marks(s, which)[yy] == tag) return true;
    return false;
}

// acc += value * kernel.  A value that is not finite also counts against a zero entry
// of a block of eight that is not all zero, as in the direct kernels; block(i) is
// entry i of that block.
template <class Block>
__device__ __forceinline__ void add_term(float& acc, float value, float kernel, int round, Block block)
{
    if (kernel == 0.f) {
        if (isfinite(value)) return;
        bool any = false;
        for (int i = 0; i < 8; ++i) any |= block(i) != 0.f;
        if (!any) return;
    }
    acc = fmaf(round_if(value, round), round_if(kernel, round), acc);
}

// The terms of the marked positions in one output of A (state m, sample w).  A sum
// that is NaN stays so: it ends there, and the cost of NaNs with it.
__device__ float marked_forward(const FftShape& s, int round, const float* c, int m, int y, int x, int w)
{
    const int4 band = s.ftab[w / kOG];
    const size_t SZ = (size_t)s.Y * s.X * s.Z;
    float acc = 0.f;
    marked_taps<1>(s, MARK_A, y, x, [&](int dy, int dx, size_t pos) {
        for (int j = band.y; j < band.y + band.z; ++j) {
            float b = 0.f;  // what the first pass took out
            if (round) {
                b = state_value(s, c, m, pos, j);
                if (!huge(b)) continue;
            } else {
                bool any = false;
                for (int p = 0; p < s.P; ++p) {
                    const float v = c[p * SZ + pos * s.Z + j];
                    if (!huge(v)) continue;
                    any = true;
                    b = fmaf(__ldg(s.Sm + ((size_t)m * s.P + p) * s.Z + j), v, b);
                }
                if (!any) continue;
            }
            const float* kp = s.Kf + (((size_t)j * s.k + dy) * s.k + dx) * s.Twp;
            add_term(acc, b, kp[w], round, [&](int i) { return kp[(w & ~7) + i]; });
            if (isnan(acc)) return false;
        }
        return true;
    });
    return acc;
}

// The same of A^T (depth j), for state m or, with m < 0, for species p (P^T over
// the states); r is either the residual [Q][Y][X][Twp] or (from_y) the measurements.
__device__ float marked_adjoint(const FftShape& s, int round, const float* r, int from_y, int m, int p,
                                int y, int x, int j)
{
    const int4 band = s.atab[j / kOG];
    const int j8 = j & ~7;
    const size_t kk = (size_t)s.k * s.k * s.Twp;
    float acc = 0.f;
    marked_taps<-1>(s, MARK_AT, y, x, [&](int dy, int dx, size_t pos) {
        const float* kt = s.Kf + ((size_t)dy * s.k + dx) * s.Twp;
        for (int q = m < 0 ? 0 : m; q < (m < 0 ? s.Q : m + 1); ++q) {
            float sum = 0.f;
            for (int w = band.y; w < band.y + band.z && !isnan(sum); ++w) {
                const float v = from_y ? folded(s, r, q, pos, w)
                                       : r[((size_t)q * s.Y * s.X + pos) * s.Twp + w];
                if (!huge(v)) continue;
                add_term(sum, v, kt[(size_t)j * kk + w], round, [&](int i) {
                    return j8 + i < s.Z ? kt[(size_t)(j8 + i) * kk + w] : 0.f;
                });
            }
            if (sum == 0.f) continue;
            acc = m < 0 ? fmaf(s.Sm[((size_t)q * s.P + p) * s.Z + j], sum, acc) : acc + sum;
            if (isnan(acc)) return false;
        }
        return true;
    });
    return acc;
}

// ---------------------------------------------------------------------------
// Transforms along x and y.  A block takes 32 lines, one per lane: neighbouring
// lanes are neighbouring channel pairs (then rows, or x frequencies).  A pass
// reads and writes every value once and is bound by memory and its latency: at
// three blocks per SM (80 registers; with two 10 to 20% slower) the y pass moves
// 10 x 144^2 x 56 pairs, 186 MB, in 29 us, 6.4 TB/s (mostly L2), and the x passes,
// whose sources are strided, 160 MB in 49 to 54 us.
// ---------------------------------------------------------------------------
// SRC_GATED: SRC_STATES, or SRC_C as the second variant
enum { SRC_C = 0, SRC_STATES = 1, SRC_U = 2, SRC_Y = 3, SRC_GATED = 4 };

struct XForward {
    FftShape s;
    const float* src;
    float2* out;    // [plane][tile][rows_in][Lx][C2]
    int C2;         // channel pairs
    int vec;        // pairs may be read as one float2
    unsigned items; // planes * tiles * rows_in * C2
    const float* src2;
    unsigned items2;
};

template <int SRC>
__global__ void __launch_bounds__(kMaxFftThreads, 3) fft_x_forward_kernel(const XForward a)
{
    extern __shared__ float2 sm[];
    const FftShape& s = a.s;
    grid_dependency();
    if (gated_off(s.gate, s.want)) return;
    const int lane = threadIdx.x & 31;
    const unsigned item = blockIdx.x * 32u + lane;
    const bool alt = second_variant(s);
    const float* src = alt ? a.src2 : a.src;
    const int round = alt ? s.round2 : s.round;
    constexpr bool kStates = SRC == SRC_STATES || SRC == SRC_GATED;
    const bool ok = item < (alt ? a.items2 : a.items);
    const unsigned q = item % (unsigned)a.C2, line = item / (unsigned)a.C2;
    const unsigned row = line % (unsigned)s.rows_in, pt = line / (unsigned)s.rows_in;
    const int tile = (int)(pt % (unsigned)s.tiles), plane = (int)(pt / (unsigned)s.tiles);
    const int gy = tile / s.x.tiles * s.y.out - s.y.pad + (int)row;
    const int gx0 = tile % s.x.tiles * s.x.out - s.x.pad;
    const bool row_ok = ok && gy >= 0 && gy < s.Y;
    const int ch = 2 * (int)q;
    const size_t YX = (size_t)s.Y * s.X;
    const size_t row0 = (size_t)(row_ok ? gy : 0) * s.X;
    const bool two = ch + 1 < s.Z;
    constexpr int kWhich = SRC == SRC_U || SRC == SRC_Y ? MARK_AT : MARK_A;
    // SRC_STATES: this thread's switching weights (its state and depths)
    float2 wt[kStates ? 8 : 1];
    if (kStates) {
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            wt[p] = make_float2(0.f, 0.f);
            if (!ok || p >= s.P || (SRC == SRC_GATED && alt)) continue;
            const float* sp = s.Sm + ((size_t)plane * s.P + p) * s.Z + ch;
            wt[p].x = __ldg(sp);
            if (two) wt[p].y = __ldg(sp + 1);
        }
    }
    auto load = [&](auto& v, int n2, int R2) {
        constexpr int R = sizeof(v) / sizeof(v[0]);
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = make_float2(0.f, 0.f);
        if (!row_ok) return;
        const int first = gx0 + n2;
        auto inside = [&](int i) {
            const int gx = first + i * R2;
            return gx >= 0 && gx < s.X;
        };
        // v += w * (the channel pair at p + i * stride), w the SRC_STATES weight;
        // all loads before the sums
        auto add = [&](const float* p, size_t stride, bool second, float2 w) {
            float2 t[R];
            if (a.vec) {
#pragma unroll
                for (int i = 0; i < R; ++i)
                    t[i] = inside(i) ? load_produced(reinterpret_cast<const float2*>(p + i * stride))
                                     : make_float2(0.f, 0.f);
            } else {
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    t[i].x = inside(i) ? load_produced(p + i * stride) : 0.f;
                    t[i].y = inside(i) && second ? load_produced(p + i * stride + 1) : 0.f;
                }
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
                v[i] = kStates
                           ? make_float2(fmaf(w.x, t[i].x, v[i].x), fmaf(w.y, t[i].y, v[i].y))
                           : cadd(v[i], t[i]);
        };
        const ptrdiff_t at = (ptrdiff_t)row0 + first;  // may lie outside; guarded by inside()
        const float2 none = make_float2(0.f, 0.f);
        if (SRC == SRC_C) {
            add(src + ((ptrdiff_t)(plane * YX) + at) * s.Z + ch, (size_t)R2 * s.Z, two, none);
        } else if (SRC == SRC_GATED && alt) {
            add(src + ((ptrdiff_t)(plane * YX) + at) * s.Z + ch, (size_t)R2 * s.Z, two,
                make_float2(1.f, 1.f));
        } else if (kStates) {
#pragma unroll
            for (int p = 0; p < 8; ++p)
                if (p < s.P)
                    add(src + ((ptrdiff_t)(p * YX) + at) * s.Z + ch, (size_t)R2 * s.Z, two, wt[p]);
        } else if (SRC == SRC_U) {
            add(src + ((ptrdiff_t)(plane * YX) + at) * s.Twp + ch, (size_t)R2 * s.Twp, true, none);
        } else {
            const int t = s.t0 + ch;
            if (t < s.T)
                for (int n = plane; n < s.N; n += s.ncyc)
                    add(src + ((ptrdiff_t)(n * YX) + at) * s.T + t, (size_t)R2 * s.T, t + 1 < s.T,
                        none);
        }
        if (any_huge(v)) {
            float2* slot = sm + n2 * 32 + lane;
            through_slots(v, slot, 32 * R2,
                          [&] { take_out(s, kWhich, next_tag(s), slot, 32 * R2, R, gy, first, R2); });
        }
        if (SRC != SRC_C && round) {
#pragma unroll
            for (int i = 0; i < R; ++i) v[i] = make_float2(round_if(v[i].x, 1), round_if(v[i].y, 1));
        }
    };
    float2* out = a.out + (size_t)line * s.x.L * a.C2 + q;
    fft_line<-1>(s.x, sm, load, [&](auto& v, int k1, int R1) {
        constexpr int R = sizeof(v) / sizeof(v[0]);
        if (!ok) return;
#pragma unroll
        for (int i = 0; i < R; ++i) out[(size_t)(k1 + R1 * i) * a.C2] = v[i];
    });
}

struct YPass {
    FftShape s;
    const float2* in;   // forward: [plane tile][rows_in][Lx][C2]; inverse: [..][Ly][Lx][C2]
    float2* out;        // forward: [plane tile][Ly][Lx][C2]; inverse: [..][rows_out][Lx][C2]
    unsigned width;     // Lx * C2
    unsigned items;     // plane-tiles * width
    unsigned items2;
    int count;          // the second launch of a call: counts its tag
};

template <int S>
__global__ void __launch_bounds__(kMaxFftThreads, 3) fft_y_kernel(const YPass a)
{
    extern __shared__ float2 sm[];
    const FftShape& s = a.s;
    grid_dependency();
    if (gated_off(s.gate, s.want)) return;
    if (a.count && blockIdx.x == 0 && threadIdx.x == 0)
        asm volatile("red.global.add.u32 [%0], 1;" ::"l"(s.marks) : "memory");
    const unsigned item = blockIdx.x * 32u + (threadIdx.x & 31);
    const bool ok = item < (second_variant(s) ? a.items2 : a.items);
    const unsigned col = item % a.width, pt = item / a.width;
    const int rows = S < 0 ? s.rows_in : s.y.L;
    const float2* in = a.in + (size_t)pt * rows * a.width + col;
    const int rows_w = S < 0 ? s.y.L : s.rows_out;
    const int first = S < 0 ? 0 : s.y.pad;
    float2* out = a.out + (size_t)pt * rows_w * a.width + col;
    fft_line<S>(
        s.y, sm,
        [&](auto& v, int n2, int R2) {
            constexpr int R = sizeof(v) / sizeof(v[0]);
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int n = n2 + i * R2;
                v[i] = ok && n < rows ? load_produced(in + (size_t)n * a.width) : make_float2(0.f, 0.f);
            }
        },
        [&](auto& v, int k1, int R1) {
            constexpr int R = sizeof(v) / sizeof(v[0]);
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int w = k1 + R1 * i - first;
                if (ok && w >= 0 && w < rows_w) out[(size_t)w * a.width] = v[i];
            }
        });
}

enum { IMG_STORE = 0, IMG_REFINE = 1 };

struct XInverse {
    FftShape s;
    const float2* in;   // [plane][tile][rows_out][Lx][C2]
    int C2;
    int q_end;          // pairs written per position (u: Twp / 2, zero past C2)
    unsigned items;     // planes * tiles * rows_out * q_end
    int vec;
    float* out;
    // u: out = (scale ? Cm : 1) v - ytil
    const float* ytil;
    const float* Cmf;   // null: no scale
    const float* c;     // input of A (terms of its marked positions)
    // images: IMG_STORE out = v; IMG_REFINE as pt_refine_kernel
    int add, add2;
    float alpha;
    const float* xi;
    float* G;
    const double* scal;
    const float* r;     // input of A^T (the same): residual or measurements
    int from_y;
    int per_state;      // planes are states (else species, summed over the states)
};

// The terms of marked positions in the image line that a thread has written, added
// to what it wrote (the line of row gy, tile columns from gx0, channels ch and
// ch + 1).  At the end of the kernel, where no value of the transform is live.
template <int MODE>
__device__ __noinline__ void add_marked_image(const XInverse& a, int gx0, int gy, int plane, int ch)
{
    const FftShape& s = a.s;
    if (!marked_near(s, MARK_AT, gy)) return;
    const int round = second_variant(s) ? s.round2 : s.round;
    const float beta = MODE == IMG_REFINE ? (float)a.scal[1] : 0.f;
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int k1 = warp; k1 < s.x.R1; k1 += nw)
        for (int i = 0; i < s.x.R2; ++i) {
            const int o = k1 + s.x.R1 * i - s.x.pad, gx = gx0 + o;
            if (o < 0 || o >= s.x.out || gx >= s.X) continue;
            for (int h = 0; h < 2 && ch + h < s.Z; ++h) {
                const float t = marked_adjoint(s, round, a.r, a.from_y, a.per_state ? plane : -1, plane,
                                               gy, gx, ch + h);
                const size_t at = (((size_t)plane * s.Y + gy) * s.X + gx) * s.Z + ch + h;
                if (MODE == IMG_REFINE) a.G[at] += t;
                a.out[at] = MODE == IMG_STORE ? a.out[at] + t : fmaf(-a.alpha, fmaf(beta, t, t), a.out[at]);
            }
        }
}

// The same for a line of u (state m, samples w and w + 1): u += factor * terms, or with
// `from` u = from + factor * terms (null: of zero).
__device__ __noinline__ void add_marked_u(const FftShape& s, int round, const float* c, float factor,
                                          const float* from, bool in_place, float* u, int gx0, int gy,
                                          int m, int w)
{
    const bool near = marked_near(s, MARK_A, gy);
    if (in_place && !near) return;
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int k1 = warp; k1 < s.x.R1; k1 += nw)
        for (int i = 0; i < s.x.R2; ++i) {
            const int o = k1 + s.x.R1 * i - s.x.pad, gx = gx0 + o;
            if (o < 0 || o >= s.x.out || gx >= s.X) continue;
            const size_t at = (((size_t)m * s.Y + gy) * s.X + gx) * s.Twp + w;
            for (int h = 0; h < 2; ++h) {
                const float t = near ? marked_forward(s, round, c, m, gy, gx, w + h) : 0.f;
                u[at + h] = fmaf(factor, t, in_place ? u[at + h] : from ? from[at + h] : 0.f);
            }
        }
}

// A^T's inverse along x: images [plane][Y][X][Z].
template <int MODE>
__global__ void __launch_bounds__(kMaxFftThreads, 3) fft_x_image_kernel(const XInverse a)
{
    extern __shared__ float2 sm[];
    const FftShape& s = a.s;
    grid_dependency();
    if (gated_off(s.gate, s.want)) return;
    const unsigned item = blockIdx.x * 32u + (threadIdx.x & 31);
    const bool ok = item < a.items;
    const unsigned q = item % (unsigned)a.C2, line = item / (unsigned)a.C2;
    const unsigned row = line % (unsigned)s.rows_out, pt = line / (unsigned)s.rows_out;
    const int tile = (int)(pt % (unsigned)s.tiles), plane = (int)(pt / (unsigned)s.tiles);
    const int gy = tile / s.x.tiles * s.y.out + (int)row;
    const int gx0 = tile % s.x.tiles * s.x.out;
    const bool row_ok = ok && gy < s.Y;
    const int ch = 2 * (int)q;
    const size_t YX = (size_t)s.Y * s.X;
    const float2* in = a.in + (size_t)line * s.x.L * a.C2 + q;
    const float beta = MODE == IMG_REFINE ? (float)a.scal[1] : 0.f;
    const bool alt = second_variant(s);
    const int add = alt ? a.add2 : a.add;
    __shared__ uint4 words;
    fetch_marks(s, &words);
    const bool two = ch + 1 < s.Z;
    fft_line<1>(
        s.x, sm,
        [&](auto& v, int n2, int R2) {
            constexpr int R = sizeof(v) / sizeof(v[0]);
#pragma unroll
            for (int i = 0; i < R; ++i)
                v[i] = ok ? load_produced(in + (size_t)(n2 + i * R2) * a.C2) : make_float2(0.f, 0.f);
        },
        [&](auto& v, int k1, int R1) {
            constexpr int R = sizeof(v) / sizeof(v[0]);
            if (!row_ok) return;
            auto out_x = [&](int i) {  // scan column of entry i, or -1
                const int o = k1 + R1 * i - s.x.pad, gx = gx0 + o;
                return o >= 0 && o < s.x.out && gx < s.X ? gx : -1;
            };
            const size_t base = ((size_t)plane * YX + (size_t)gy * s.X) * s.Z + ch;
            auto at = [&](int gx) { return base + (size_t)gx * s.Z; };
            auto get = [&](const float* p) {
                return a.vec ? *reinterpret_cast<const float2*>(p)
                             : make_float2(p[0], two ? p[1] : 0.f);
            };
            auto put = [&](float* p, float2 w) {
                if (a.vec) {
                    *reinterpret_cast<float2*>(p) = w;
                } else {
                    p[0] = w.x;
                    if (two) p[1] = w.y;
                }
            };
            // a few entries at a time, every read of them before the first write
            constexpr int CH = 6;
#pragma unroll
            for (int b = 0; b < R; b += CH) {
                float2 go[CH], xi[CH];
#pragma unroll
                for (int i = 0; i < CH; ++i) {
                    const int gx = b + i < R ? out_x(b + i) : -1;
                    go[i] = xi[i] = make_float2(0.f, 0.f);
                    if (MODE == IMG_REFINE && gx >= 0) go[i] = get(a.G + at(gx));
                    if (MODE == IMG_REFINE && gx >= 0) xi[i] = get(a.xi + at(gx));
                }
#pragma unroll
                for (int i = 0; i < CH; ++i) {
                    const int gx = b + i < R ? out_x(b + i) : -1;
                    if (gx < 0) continue;
                    float2 g = v[b + i];
                    if (MODE == IMG_REFINE) {
                        if (add) g = cadd(go[i], g);
                        put(a.G + at(gx), g);
                        g = make_float2(fmaf(beta, g.x - go[i].x, g.x),
                                        fmaf(beta, g.y - go[i].y, g.y));
                        g = make_float2(fmaf(-a.alpha, g.x, xi[i].x),
                                        fmaf(-a.alpha, g.y, xi[i].y));
                    }
                    put(a.out + at(gx), g);
                }
            }
        });
    if (row_ok && any_mark(words, MARK_AT)) add_marked_image<MODE>(a, gx0, gy, plane, ch);
}

// A's inverse along x: u [Q][Y][X][Twp], the scaled folded residual, zero past
// the window.
__global__ void __launch_bounds__(kMaxFftThreads, 3) fft_x_u_kernel(const XInverse a)
{
    extern __shared__ float2 sm[];
    const FftShape& s = a.s;
    grid_dependency();
    if (gated_off(s.gate, s.want)) return;
    const unsigned item = blockIdx.x * 32u + (threadIdx.x & 31);
    const bool ok = item < a.items;
    const unsigned q = item % (unsigned)a.q_end, line = item / (unsigned)a.q_end;
    const unsigned row = line % (unsigned)s.rows_out, pt = line / (unsigned)s.rows_out;
    const int tile = (int)(pt % (unsigned)s.tiles), m = (int)(pt / (unsigned)s.tiles);
    const int gy = tile / s.x.tiles * s.y.out + (int)row;
    const int gx0 = tile % s.x.tiles * s.x.out;
    const bool row_ok = ok && gy < s.Y, in_ok = ok && (int)q < a.C2;
    const int w = 2 * (int)q;
    const float2* in = a.in + (size_t)line * s.x.L * a.C2 + q;
    const float cm = ok && a.Cmf ? a.Cmf[m] : 1.f;
    __shared__ uint4 words;
    fetch_marks(s, &words);
    fft_line<1>(
        s.x, sm,
        [&](auto& v, int n2, int R2) {
            constexpr int R = sizeof(v) / sizeof(v[0]);
#pragma unroll
            for (int i = 0; i < R; ++i)
                v[i] = in_ok ? load_produced(in + (size_t)(n2 + i * R2) * a.C2) : make_float2(0.f, 0.f);
        },
        [&](auto& v, int k1, int R1) {
            constexpr int R = sizeof(v) / sizeof(v[0]);
            if (!row_ok) return;
            auto out_x = [&](int i) {  // scan column of entry i, or -1
                const int o = k1 + R1 * i - s.x.pad, gx = gx0 + o;
                return o >= 0 && o < s.x.out && gx < s.X ? gx : -1;
            };
            const size_t base = (((size_t)m * s.Y + gy) * s.X) * s.Twp + w;
            float2 yt[R];
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int gx = out_x(i);
                yt[i] = a.ytil && gx >= 0 ? load_produced(reinterpret_cast<const float2*>(
                                                a.ytil + base + (size_t)gx * s.Twp))
                                          : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
                if (const int gx = out_x(i); gx >= 0)
                    *reinterpret_cast<float2*>(a.out + base + (size_t)gx * s.Twp) =
                        make_float2(fmaf(cm, v[i].x, -yt[i].x), fmaf(cm, v[i].y, -yt[i].y));
        });
    if (row_ok && in_ok && any_mark(words, MARK_A))
        add_marked_u(s, s.round, a.c, cm, nullptr, true, a.out, gx0, gy, m, w);
}

// A's inverse along x, the scaled folded residual, and A^T's forward along x in
// one pass (one tile): u stays in registers.  The inverse's second DFTs leave
// x = k1 + R1 k2 in the thread that needs exactly these for a first DFT of the
// transform taken as L = R2 R1, so the two transforms share that step.  Against the
// two kernels it replaces it saves a write and a read of u.  u is written too, and
// its huge values taken out, where they can come from the input: A's has marked
// positions, or the measurements hold values from 2^48 (by the sum of their squares).
struct XResidual {
    FftShape s;
    const float2* in;   // [state][Y][Lx][C2]
    float2* out;        // [state][Y][Lx][C2]
    int C2;
    unsigned items;     // states * Y * C2
    const float* ytil;
    const float* Cmf;
    const float* c;
    float* u;
    int keep;           // u is written in any case
    const double* ysq;  // sum of squares of the measurements behind ytil
    const float* ytil2;
    const float* c2;
};

constexpr double kHugeYsq = 7.9228162514264338e28;  // 2^96

// 96 registers, three blocks of 6 warps per SM (at 80 the spills cost more than the
// fourth block gave); 48 bytes are spilled.
__global__ void __launch_bounds__(288, 2) fft_x_residual_kernel(const XResidual a)
{
    extern __shared__ float2 sm[];
    const FftShape& s = a.s;
    grid_dependency();
    if (gated_off(s.gate, s.want)) return;
    const FftAxis& ax = s.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned item = blockIdx.x * 32u + lane;
    const bool ok = item < a.items;
    const unsigned q = item % (unsigned)a.C2, line = item / (unsigned)a.C2;
    const int row = (int)(line % (unsigned)s.Y), m = (int)(line / (unsigned)s.Y);
    const int w = 2 * (int)q;
    const float2* in = a.in + (size_t)line * ax.L * a.C2 + q;
    float2* out = a.out + (size_t)line * ax.L * a.C2 + q;
    const float cm = ok ? a.Cmf[m] : 1.f;
    const bool alt = second_variant(s);
    const float* ytil = alt ? a.ytil2 : a.ytil;
    const int round = alt ? s.round2 : s.round;
    __shared__ uint4 words;
    __shared__ int s_keep;
    fetch_marks(s, &words);
    if (threadIdx.x == 0) s_keep = a.keep || (ytil && !(*a.ysq < kHugeYsq));
    const size_t base = (((size_t)m * s.Y + row) * s.X) * s.Twp + w;
    auto load = [&](auto& v, int n2, int R2) {
        constexpr int R = sizeof(v) / sizeof(v[0]);
#pragma unroll
        for (int i = 0; i < R; ++i)
            v[i] = ok ? load_produced(in + (size_t)(n2 + i * R2) * a.C2) : make_float2(0.f, 0.f);
    };
#define SW_P1(R)                                  \
    for (int n2 = warp; n2 < ax.R2; n2 += nw)     \
        fft_pass1<R, 1>(ax.tw, ax.R2, n2, sm, lane, load)
    SW_RADIX(ax.R1, SW_P1)
#undef SW_P1
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const bool marked = any_mark(words, MARK_A);
    // the marked positions' terms join ytil, in the place of u
    if (ok && marked) {
        add_marked_u(s, round, alt ? a.c2 : a.c, -cm, ytil, false, a.u, 0, row, m, w);
        ytil = a.u;
    }
    auto middle = [&](auto& v, int k1, int R1) {
        constexpr int R = sizeof(v) / sizeof(v[0]);
        const bool keep = marked || s_keep;
        float2 yt[R];
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int gx = k1 + R1 * i;
            yt[i] = ytil && ok && gx < s.X ? load_produced(reinterpret_cast<const float2*>(
                                                   ytil + base + (size_t)gx * s.Twp))
                                             : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int gx = k1 + R1 * i;
            v[i] = make_float2(fmaf(cm, v[i].x, -yt[i].x), fmaf(cm, v[i].y, -yt[i].y));
            if (keep && ok && gx < s.X)
                *reinterpret_cast<float2*>(a.u + base + (size_t)gx * s.Twp) = v[i];
            if (gx >= s.X) v[i] = make_float2(0.f, 0.f);
        }
        if (keep && ok && any_huge(v)) {
            float2* slot = sm + k1 * R * 32 + lane;
            through_slots(v, slot, 32,
                          [&] { take_out(s, MARK_AT, this_tag(s), slot, 32, R, row, k1, R1); });
        }
        if (round) {
#pragma unroll
            for (int i = 0; i < R; ++i) v[i] = make_float2(round_if(v[i].x, 1), round_if(v[i].y, 1));
        }
        Dft<R, -1>::run(v);
        // into the entries that this thread has read
        float2* slot = sm + k1 * R * 32 + lane;
        slot[0] = v[0];
#pragma unroll
        for (int i = 1; i < R; ++i) {
            const float2 t = __ldg(ax.tw + k1 * i);
            slot[i * 32] = cmul(v[i], t.x, t.y);
        }
    };
#define SW_P2(R)                                  \
    for (int k1 = warp; k1 < ax.R1; k1 += nw)     \
        fft_pass2<R, 1>(ax.R1, k1, sm, lane, middle)
    SW_RADIX(ax.R2, SW_P2)
#undef SW_P2
    __syncthreads();
    // last pass of the forward transform: its first pass left entry (n2, k1) at n2 R2 + k1
    auto last = [&](auto& v, int k1) {
        constexpr int R = sizeof(v) / sizeof(v[0]);
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = sm[(i * ax.R2 + k1) * 32 + lane];
        Dft<R, -1>::run(v);
        if (!ok) return;
#pragma unroll
        for (int i = 0; i < R; ++i) out[(size_t)(k1 + ax.R2 * i) * a.C2] = v[i];
    };
#define SW_P3(R)                                    \
    float2 v[R];                                    \
    for (int k1 = warp; k1 < ax.R2; k1 += nw) last(v, k1)
    SW_RADIX(ax.R1, SW_P3)
#undef SW_P3
}

// ---------------------------------------------------------------------------
// The spectral product.  A block takes kFB frequencies of the half plane and
// one chunk of MC states; the unpacked (and P-mapped) inputs of all contracted
// channels are staged in shared memory [channel][frequency][state].  A warp
// takes groups of kOG output channels: lane = (frequency, channel pair), each
// thread MC states x 2 channels; every K^ entry feeds 4 MC FMAs.  The products
// run as packed FP32 pairs (fma.rn.f32x2):
//   acc += (K.re, K.re) (b.re, b.im) + (-K.im, K.im) (b.im, b.re),
// the signs of K.im exchanged for the adjoint's conj(K).
// K^ (512 contiguous bytes per warp and contracted channel) streams through a
// ring of asynchronous copies that runs ahead across the warp's groups and
// starts before the inputs are staged; a thread reads back only what it copied
// itself, so the ring needs no barrier.
// Bound by latency at 12 to 14 warps per SM (the inputs of 10 states take 61 KB per
// block): 145 us per product of the largest workload (k = 31, 10 states), where the K^
// stream alone is 56 us of HBM time and the FMAs 48 us.  The schedulers issue in 0.46
// to 0.55 of the cycles; the first stalls are loads in flight and the FMA pipe.  One register accumulator per value with K^ read by the thread itself:
// 200 us (164 to 255 registers, one block per SM).
// ---------------------------------------------------------------------------
struct Spec {
    FftShape s;
    const float2* in;      // [plane][tile][Ly][Lx][in_C2]
    float2* out;           // [plane][tile][Ly][Lx][out_C2]
    const float4* K;       // [freq block][row][kFB][kOG / 2] (two channels each)
    const float4* K2;
    const int4* tab;       // per group: first row, first contracted channel, their count
    const float4* S4;      // [Z][Q][species in fours]
    int groups;
    long long rows;        // rows per frequency block
    int in_C2, out_C2;
    int chunks;
    int hx;                // Lx / 2 + 1
};

__device__ __forceinline__ uint64_t pack2(float a, float b)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ float2 unpack2(uint64_t v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// Contracted channels per ring slot, and slots (two in flight while one is consumed).
// 2 x 4 gave 1% on 128^2 planes, but 53 for 44 us on 45 x 37, where a block has its
// SM to itself and the waits per row count; 2 x 6, 1 x 8 and 8 x 2 are slower on all.
constexpr int kRingRows = 4;
constexpr int kRingSlots = 3;

// float2 slots per (channel, frequency) of the staged inputs: MC, padded so
// that 8 frequencies start in 8 different 16-byte bank groups
__host__ __device__ constexpr int spec_stride(int MC) { return MC % 4 == 0 ? MC + 2 : MC; }

// Dynamic shared memory: staged inputs, then the warps' rings.
__host__ __device__ constexpr size_t spec_smem(int MC, int pairs, int warps)
{
    return (size_t)2 * pairs * kFB * spec_stride(MC) * sizeof(float2) +
           (size_t)warps * kRingSlots * kRingRows * 512;
}

// MAP: how P (or P^T) takes part.  MAP_NONE: the planes are states; MAP_SPECIES:
// they are species; MAP_GATED: states, or species as the second variant (A).
enum { MAP_NONE = 0, MAP_SPECIES = 1, MAP_GATED = 2 };

template <int MC, bool ADJ, int MAP>
__global__ void __launch_bounds__(kSpecThreads, 2) spec_kernel(const Spec a)
{
    extern __shared__ float4 sm4[];
    const FftShape& s = a.s;
    grid_dependency();
    if (gated_off(s.gate, s.want)) return;
    constexpr int MS2 = spec_stride(MC) / 2;  // float4 per (channel, frequency)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int Lx = s.x.L, Ly = s.y.L;
    const size_t area = (size_t)Ly * Lx;
    const bool alt = second_variant(s);
    const bool species = MAP == MAP_GATED ? alt : MAP == MAP_SPECIES;
    constexpr bool kFuseT = ADJ && MAP == MAP_SPECIES;
    const int loops = kFuseT ? a.chunks : 1;
    const int tile = kFuseT ? (int)blockIdx.y : (int)blockIdx.y / a.chunks;
    const int chunk0 = kFuseT ? 0 : (int)blockIdx.y % a.chunks;
    const int P4 = (s.P + 3) / 4;
    float4* ring = sm4 + (size_t)2 * a.in_C2 * kFB * MS2 + warp * (kRingSlots * kRingRows * 32) + lane;
    const float4* kblk = (alt ? a.K2 : a.K) + (size_t)blockIdx.x * a.rows * (kFB * kOG / 2) + lane;

    auto locate = [&](int f, size_t* at, size_t* mirror) -> bool {
        const int id = (int)blockIdx.x * kFB + f;
        const int ky = id / a.hx, kx = id - ky * a.hx;
        if (ky >= Ly) return false;
        // both halves of the self-mirrored columns hold the same pairs: one is taken
        if ((kx == 0 || 2 * kx == Lx) && 2 * ky > Ly) return false;
        *at = (size_t)ky * Lx + kx;
        *mirror = (size_t)(ky ? Ly - ky : 0) * Lx + (kx ? Lx - kx : 0);
        return true;
    };

    for (int it = 0; it < loops; ++it) {
        const int m0 = (chunk0 + it) * MC;
        if (it > 0) __syncthreads();

        // the ring's producer: the next kRingRows rows of this warp's groups
        int pg = warp, pi = 0, pslot = 0;
        int4 pt = pg < a.groups ? __ldg(a.tab + pg) : make_int4(0, 0, 0, 0);
        auto produce = [&]() {
            while (pg < a.groups && pi >= pt.z) {
                pg += nw;
                pi = 0;
                pt = pg < a.groups ? __ldg(a.tab + pg) : make_int4(0, 0, 0, 0);
            }
            if (pg < a.groups) {
                const float4* src = kblk + (size_t)(pt.x + pi) * 32;
                const unsigned dst =
                    (unsigned)__cvta_generic_to_shared(ring + pslot * (kRingRows * 32));
#pragma unroll
                for (int u = 0; u < kRingRows; ++u)
                    if (pi + u < pt.z)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + u * 512),
                                     "l"(src + u * 32)
                                     : "memory");
                pi += kRingRows;
            }
            pslot = pslot + 1 == kRingSlots ? 0 : pslot + 1;
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
#pragma unroll
        for (int i = 0; i < kRingSlots - 1; ++i) produce();

        {
            const int f = lane & 7;
            size_t at = 0, mi = 0;
            const bool f_ok = locate(f, &at, &mi);
            for (int q0 = warp * 4; q0 < a.in_C2; q0 += nw * 4) {
                const int q = q0 + (lane >> 3);
                if (q >= a.in_C2) continue;
                float4* d0 = sm4 + ((size_t)(2 * q) * kFB + f) * MS2;
                float4* d1 = d0 + kFB * MS2;
                auto unpacked = [&](int plane, bool use, float2& x0, float2& x1) {
                    const float2* p = a.in + ((size_t)plane * s.tiles + tile) * area * a.in_C2 + q;
                    const float2 none = make_float2(0.f, 0.f);
                    const float2 z = use ? load_produced(p + at * a.in_C2) : none;
                    const float2 zm = use ? load_produced(p + mi * a.in_C2) : none;
                    x0 = make_float2(z.x + zm.x, z.y - zm.y);
                    x1 = make_float2(z.y + zm.y, zm.x - z.x);
                };
                if (!ADJ && MAP != MAP_NONE && species) {
                    for (int p4 = 0; p4 < P4; ++p4) {
                        float2 x0[4], x1[4];
#pragma unroll
                        for (int p = 0; p < 4; ++p)
                            unpacked(4 * p4 + p, f_ok && 4 * p4 + p < s.P, x0[p], x1[p]);
                        const float4* w0 = a.S4 + (size_t)(2 * q) * s.Q * P4 + p4;
                        const float4* w1 = 2 * q + 1 < s.Z ? w0 + (size_t)s.Q * P4 : w0;
                        auto mapped = [](float4 w, const float2* x, float2 b) -> float2 {
                            b.x = fmaf(w.x, x[0].x, b.x);
                            b.y = fmaf(w.x, x[0].y, b.y);
                            b.x = fmaf(w.y, x[1].x, b.x);
                            b.y = fmaf(w.y, x[1].y, b.y);
                            b.x = fmaf(w.z, x[2].x, b.x);
                            b.y = fmaf(w.z, x[2].y, b.y);
                            b.x = fmaf(w.w, x[3].x, b.x);
                            b.y = fmaf(w.w, x[3].y, b.y);
                            return b;
                        };
#pragma unroll
                        for (int i = 0; i < MC / 2; ++i) {
                            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
                            const int m = m0 + 2 * i;
                            const bool ma = m < s.Q, mb = m + 1 < s.Q;
                            const float4 a0 = ma ? __ldg(w0 + (size_t)m * P4) : zero;
                            const float4 a1 = ma ? __ldg(w1 + (size_t)m * P4) : zero;
                            const float4 b0 = mb ? __ldg(w0 + (size_t)(m + 1) * P4) : zero;
                            const float4 b1 = mb ? __ldg(w1 + (size_t)(m + 1) * P4) : zero;
                            const float4 o0 = p4 ? d0[i] : zero, o1 = p4 ? d1[i] : zero;
                            const float2 r00 = mapped(a0, x0, make_float2(o0.x, o0.y));
                            const float2 r01 = mapped(b0, x0, make_float2(o0.z, o0.w));
                            const float2 r10 = mapped(a1, x1, make_float2(o1.x, o1.y));
                            const float2 r11 = mapped(b1, x1, make_float2(o1.z, o1.w));
                            d0[i] = make_float4(r00.x, r00.y, r01.x, r01.y);
                            d1[i] = make_float4(r10.x, r10.y, r11.x, r11.y);
                        }
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < MC / 2; ++i) {
                        const int m = m0 + 2 * i;
                        float2 a0, a1, b0, b1;
                        unpacked(m, f_ok && m < s.Q, a0, a1);
                        unpacked(m + 1, f_ok && m + 1 < s.Q, b0, b1);
                        d0[i] = make_float4(a0.x, a0.y, b0.x, b0.y);
                        d1[i] = make_float4(a1.x, a1.y, b1.x, b1.y);
                    }
                }
            }
        }
        __syncthreads();

        const int f = lane >> 2, pl = lane & 3;
        size_t at = 0, mi = 0;
        const bool f_ok = locate(f, &at, &mi);
        int cslot = 0;
        for (int g = warp; g < a.groups; g += nw) {
            const int4 t = __ldg(a.tab + g);
            uint64_t A0[MC], A1[MC];
#pragma unroll
            for (int m = 0; m < MC; ++m) A0[m] = A1[m] = 0ull;
            const float4* bp = sm4 + ((size_t)t.y * kFB + f) * MS2;
            auto row = [&](const float4 k, const float4* b) {
                const uint64_t k0r = pack2(k.x, k.x), k1r = pack2(k.z, k.z);
                const uint64_t k0i = ADJ ? pack2(k.y, -k.y) : pack2(-k.y, k.y);
                const uint64_t k1i = ADJ ? pack2(k.w, -k.w) : pack2(-k.w, k.w);
#pragma unroll
                for (int h = 0; h < MC / 2; ++h) {
                    const float4 v = b[h];
                    const uint64_t x = pack2(v.x, v.y), xs = pack2(v.y, v.x);
                    const uint64_t y = pack2(v.z, v.w), ys = pack2(v.w, v.z);
                    fma2(A0[2 * h], k0r, x);
                    fma2(A1[2 * h], k1r, x);
                    fma2(A0[2 * h + 1], k0r, y);
                    fma2(A1[2 * h + 1], k1r, y);
                    fma2(A0[2 * h], k0i, xs);
                    fma2(A1[2 * h], k1i, xs);
                    fma2(A0[2 * h + 1], k0i, ys);
                    fma2(A1[2 * h + 1], k1i, ys);
                }
            };
            for (int i = 0; i < t.z; i += kRingRows) {
                asm volatile("cp.async.wait_group %0;" ::"n"(kRingSlots - 2) : "memory");
                const float4* src = ring + cslot * (kRingRows * 32);
                cslot = cslot + 1 == kRingSlots ? 0 : cslot + 1;
                if (i + kRingRows <= t.z) {
                    float4 k[kRingRows];
#pragma unroll
                    for (int u = 0; u < kRingRows; ++u) k[u] = src[u * 32];
                    produce();  // into the slot whose rows were consumed last
#pragma unroll
                    for (int u = 0; u < kRingRows; ++u) row(k[u], bp + (size_t)(i + u) * (kFB * MS2));
                } else {
                    produce();
                    for (int u = 0; i + u < t.z; ++u)
                        row(src[u * 32], bp + (size_t)(i + u) * (kFB * MS2));
                }
            }

            const int oq = g * (kOG / 2) + pl;
            if (!f_ok || oq >= a.out_C2) continue;
            auto put = [&](int plane, float2 u0, float2 u1, bool add) {
                // channels 2 oq and 2 oq + 1 as one complex image: U0 + i U1 at f, and
                // conj(U0) + i conj(U1) at -f
                float2* o = a.out + ((size_t)plane * s.tiles + tile) * area * a.out_C2 + oq;
                float2 w = make_float2(u0.x - u1.y, u0.y + u1.x);
                float2 wm = make_float2(u0.x + u1.y, u1.x - u0.y);
                if (add) {
                    w = cadd(w, o[at * a.out_C2]);
                    if (mi != at) wm = cadd(wm, o[mi * a.out_C2]);
                }
                o[at * a.out_C2] = w;
                if (mi != at) o[mi * a.out_C2] = wm;
            };
            if (kFuseT) {
                for (int p4 = 0; p4 < P4; ++p4) {
                    const float4* w0 = a.S4 + ((size_t)(2 * oq) * s.Q + m0) * P4 + p4;
                    const float4* w1 = 2 * oq + 1 < s.Z ? w0 + (size_t)s.Q * P4 : w0;
                    float2 u0[4], u1[4];
#pragma unroll
                    for (int p = 0; p < 4; ++p) u0[p] = u1[p] = make_float2(0.f, 0.f);
#pragma unroll
                    for (int m = 0; m < MC; ++m) {
                        if (m0 + m >= s.Q) break;
                        const float4 v0 = __ldg(w0 + (size_t)m * P4), v1 = __ldg(w1 + (size_t)m * P4);
                        const float2 g0 = unpack2(A0[m]), g1 = unpack2(A1[m]);
                        const float s0[4] = {v0.x, v0.y, v0.z, v0.w};
                        const float s1[4] = {v1.x, v1.y, v1.z, v1.w};
#pragma unroll
                        for (int p = 0; p < 4; ++p) {
                            u0[p].x = fmaf(s0[p], g0.x, u0[p].x);
                            u0[p].y = fmaf(s0[p], g0.y, u0[p].y);
                            u1[p].x = fmaf(s1[p], g1.x, u1[p].x);
                            u1[p].y = fmaf(s1[p], g1.y, u1[p].y);
                        }
                    }
#pragma unroll
                    for (int p = 0; p < 4; ++p)
                        if (4 * p4 + p < s.P) put(4 * p4 + p, u0[p], u1[p], it > 0);
                }
            } else {
#pragma unroll
                for (int m = 0; m < MC; ++m)
                    if (m0 + m < s.Q) put(m0 + m, unpack2(A0[m]), unpack2(A1[m]), false);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
}

// ---------------------------------------------------------------------------
// Set-up of K^ (FP64 sums of the FP32 kernel, or of its BF16 rounding), one
// pass per lateral axis; frequencies of u[y] = sum_d b[y + d] K[d], so with
// exp(+2 pi i k d / L), scaled by 1 / (2 Ly Lx) (the 2 of the unpacking).
// ---------------------------------------------------------------------------
struct BandEntry {
    int j, w;
};

// part[entry][dy][kx] = sum_dx K[j][dy][dx][w] exp(2 pi i kx (dx - r) / Lx)
__global__ void spectrum_x_kernel(const float* __restrict__ Kf, const BandEntry* __restrict__ band,
                                  int first, int count, double2* __restrict__ part, int k, int Twp,
                                  int Lx, int hx, int round)
{
    extern __shared__ double2 root[];
    for (int i = threadIdx.x; i < Lx; i += blockDim.x) {
        double sn, cs;
        sincospi(2.0 * i / Lx, &sn, &cs);
        root[i] = make_double2(cs, sn);
    }
    __syncthreads();
    const size_t n = (size_t)count * k * hx;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n;
         e += (size_t)gridDim.x * blockDim.x) {
        const int kx = (int)(e % hx);
        const int dy = (int)((e / hx) % k);
        const BandEntry b = band[first + e / ((size_t)hx * k)];
        const float* kp = Kf + (((size_t)b.j * k + dy) * k) * Twp + b.w;
        double re = 0.0, im = 0.0;
        int ph = (int)(((long long)kx * (Lx - k / 2 % Lx)) % Lx);
        for (int dx = 0; dx < k; ++dx) {
            const double v = round_if(kp[(size_t)dx * Twp], round);
            re = fma(v, root[ph].x, re);
            im = fma(v, root[ph].y, im);
            ph += kx;
            if (ph >= Lx) ph -= Lx;
        }
        part[e] = make_double2(re, im);
    }
}

struct SpectrumOut {
    float2* F;          // forward layout (contracted depths)
    float2* A;          // adjoint layout (contracted samples)
    const int4* ftab;
    const int4* atab;
    long long frows, arows;
};

// K^[entry](ky, kx) = sum_dy part[entry][dy][kx] exp(2 pi i ky (dy - r) / Ly)
__global__ void spectrum_y_kernel(const double2* __restrict__ part,
                                  const BandEntry* __restrict__ band, int first, int count, int k,
                                  int Ly, int Lx, int hx, SpectrumOut o)
{
    extern __shared__ double2 sh[];
    double2* root = sh;          // [Ly]
    double2* col = sh + Ly;      // [k][32]
    for (int i = threadIdx.x; i < Ly; i += blockDim.x) {
        double sn, cs;
        sincospi(2.0 * i / Ly, &sn, &cs);
        root[i] = make_double2(cs, sn);
    }
    const int kx = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    const int e = blockIdx.x * 32 + lane;
    const bool ok = e < count;
    for (int dy = warp; dy < k; dy += nw)
        col[dy * 32 + lane] = ok ? part[((size_t)e * k + dy) * hx + kx] : make_double2(0.0, 0.0);
    __syncthreads();
    if (!ok) return;
    const BandEntry b = band[first + e];
    const double scale = 0.5 / ((double)Ly * Lx);
    const int4 ft = o.ftab[b.w / kOG], at = o.atab[b.j / kOG];
    for (int ky = warp; ky < Ly; ky += nw) {
        double re = 0.0, im = 0.0;
        int ph = (int)(((long long)ky * (Ly - k / 2 % Ly)) % Ly);
        for (int dy = 0; dy < k; ++dy) {
            const double2 v = col[dy * 32 + lane], w = root[ph];
            re = fma(v.x, w.x, fma(-v.y, w.y, re));
            im = fma(v.x, w.y, fma(v.y, w.x, im));
            ph += ky;
            if (ph >= Ly) ph -= Ly;
        }
        const float2 val = make_float2((float)(re * scale), (float)(im * scale));
        const long long id = (long long)ky * hx + kx;
        const long long blk = id / kFB, f = id % kFB;
        o.F[((blk * o.frows + ft.x + (b.j - ft.y)) * kFB + f) * kOG + b.w % kOG] = val;
        o.A[((blk * o.arows + at.x + (b.w - at.y)) * kFB + f) * kOG + b.j % kOG] = val;
    }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
// Transform lengths: products of two of the radices above, close to square.
struct Length {
    int L, R1, R2;
};
const Length kLengths[] = {
    {4, 2, 2},    {6, 2, 3},    {8, 2, 4},    {9, 3, 3},    {10, 2, 5},   {12, 3, 4},
    {15, 3, 5},   {16, 4, 4},   {18, 3, 6},   {20, 4, 5},   {24, 4, 6},   {25, 5, 5},
    {30, 5, 6},   {32, 4, 8},   {36, 6, 6},   {40, 5, 8},   {45, 5, 9},   {48, 6, 8},
    {50, 5, 10},  {54, 6, 9},   {60, 6, 10},  {64, 8, 8},   {72, 8, 9},   {80, 8, 10},
    {90, 9, 10},  {96, 8, 12},  {100, 10, 10}, {108, 9, 12}, {120, 10, 12}, {128, 8, 16},
    {144, 12, 12}, {160, 10, 16}, {192, 12, 16}, {256, 16, 16}};

// The axis of n positions under support radius r with transform length `len`;
// false if the length leaves no output.
bool make_axis(const Length& len, int n, int r, FftAxis* a)
{
    a->L = len.L;
    a->R1 = len.R1;
    a->R2 = len.R2;
    a->tw = nullptr;
    if (len.L >= n + r) {
        a->tiles = 1;
        a->out = n;
        a->pad = 0;
        return true;
    }
    a->out = len.L - 2 * r;
    if (a->out < 1) return false;
    a->pad = r;
    a->tiles = (n + a->out - 1) / a->out;
    return true;
}

template <typename T>
bool try_alloc(T** p, size_t count)
{
    *p = nullptr;
    if (cudaMalloc((void**)p, std::max<size_t>(count, 1) * sizeof(T)) == cudaSuccess) return true;
    cudaGetLastError();  // an operator that does not fit falls back to the direct kernels
    *p = nullptr;
    return false;
}

int fft_warps(const FftAxis& a)
{
    const int r = std::max(a.R1, a.R2);
    return r <= 8 ? r : (r + 1) / 2;
}

}  // namespace

struct FftOperator {
    FftAxis y, x;
    int tiles = 1, rows_in = 0, rows_out = 0;
    int hx = 0;              // x frequencies of the half plane
    long long blocks = 0;    // blocks of kFB frequencies
    int Cz2 = 0, Ct2 = 0;    // channel pairs: depths, window samples
    int fgroups = 0, agroups = 0;
    long long frows = 0, arows = 0;
    int4* ftab = nullptr;
    int4* atab = nullptr;
    float4* S4 = nullptr;    // switching weights as the products read them
    float2* twx = nullptr;
    float2* twy = nullptr;
    float2* KF[2] = {nullptr, nullptr};  // K^ of the FP32 kernel, and of its BF16 rounding
    float2* KA[2] = {nullptr, nullptr};
    BandEntry* band = nullptr;
    int nband = 0;
    unsigned* marks = nullptr;  // see FftShape
    float2* w0 = nullptr;    // workspaces, the spectra before and after a pass
    float2* w1 = nullptr;
    int fchunk = 2, achunk = 2;  // states per block of the two products
};

namespace {

// Banded groups of kOG output channels: the hull of the contracted channels
// that reach any of them (an empty group keeps no rows).
long long band_table(const std::vector<int>& lo, const std::vector<int>& hi, int outs,
                     std::vector<int4>* tab)
{
    tab->clear();
    long long rows = 0;
    for (int g = 0; g * kOG < outs; ++g) {
        int a = std::numeric_limits<int>::max(), b = -1;
        for (int o = g * kOG; o < std::min(outs, (g + 1) * kOG); ++o) {
            a = std::min(a, lo[o]);
            b = std::max(b, hi[o]);
        }
        const int n = b >= a ? b - a + 1 : 0;
        tab->push_back(make_int4((int)rows, n ? a : 0, n, 0));
        rows += n;
    }
    return rows;
}

// Warps of a block: the fewest rounds of up to 8 over the groups, evenly filled
// (9 groups on 7 warps took two rounds of which one held 2 groups).
int spec_warps(int groups)
{
    const int rounds = (groups + kSpecThreads / 32 - 1) / (kSpecThreads / 32);
    return std::max(1, (groups + rounds - 1) / std::max(1, rounds));
}

// States per block: an even count up to 10, the fewest reads of K^ first, then
// the fewest padding states; blocks that leave room for two per SM where
// possible (0: none fits).
int pick_chunk(int Q, int pairs, int warps)
{
    for (size_t cap : {(size_t)112 * 1024, kSpecSmem}) {
        int best = 0, least = 1 << 30;
        for (int mc = 10; mc >= 2; mc -= 2) {
            if (spec_smem(mc, pairs, warps) > cap) continue;
            const int blocks = (Q + mc - 1) / mc, cost = blocks * (64 + mc);
            if (cost < least) {
                least = cost;
                best = mc;
            }
        }
        if (best) return best;
    }
    return 0;
}

}  // namespace

void fft_release(swopt_handle* h)
{
    FftOperator* f = h->fft;
    if (!f) return;
    cudaFree(f->ftab);
    cudaFree(f->atab);
    cudaFree(f->S4);
    cudaFree(f->twx);
    cudaFree(f->twy);
    for (int i = 0; i < 2; ++i) {
        cudaFree(f->KF[i]);
        cudaFree(f->KA[i]);
    }
    cudaFree(f->band);
    cudaFree(f->marks);
    cudaFree(f->w0);
    cudaFree(f->w1);
    delete f;
    h->fft = nullptr;
}

// K^ of the FP32 kernel (which 0) or of its BF16 rounding (which 1).
static bool build_spectrum(swopt_handle* h, int which)
{
    FftOperator* f = h->fft;
    if (f->KF[which]) return true;
    const size_t nf = (size_t)f->blocks * f->frows * kFB * kOG;
    const size_t na = (size_t)f->blocks * f->arows * kFB * kOG;
    // band entries per pass, so that the partial sums stay within 256 MB
    const size_t per = (size_t)h->k * f->hx;
    const int step = (int)std::max<size_t>(32, std::min<size_t>(f->nband, (256u << 20) / (per * 16)));
    double2* part = nullptr;
    bool ok = try_alloc(&f->KF[which], nf) && try_alloc(&f->KA[which], na) &&
              try_alloc(&part, per * step);
    ok = ok && cudaMemset(f->KF[which], 0, nf * sizeof(float2)) == cudaSuccess &&
         cudaMemset(f->KA[which], 0, na * sizeof(float2)) == cudaSuccess;
    const SpectrumOut o{f->KF[which], f->KA[which], f->ftab, f->atab, f->frows, f->arows};
    for (int first = 0; ok && first < f->nband; first += step) {
        const int n = std::min(step, f->nband - first);
        const int g = (int)std::min<size_t>((per * n + 255) / 256, 152 * 16);
        spectrum_x_kernel<<<g, 256, f->x.L * sizeof(double2)>>>(h->Kf, f->band, first, n, part, h->k,
                                                                 h->Twp, f->x.L, f->hx, which);
        spectrum_y_kernel<<<dim3((n + 31) / 32, f->hx), 256,
                            (f->y.L + (size_t)h->k * 32) * sizeof(double2)>>>(
            part, f->band, first, n, h->k, f->y.L, f->x.L, f->hx, o);
        ok = cudaGetLastError() == cudaSuccess;
    }
    ok = ok && cudaDeviceSynchronize() == cudaSuccess;
    cudaFree(part);
    if (!ok) {
        cudaFree(f->KF[which]);
        cudaFree(f->KA[which]);
        f->KF[which] = f->KA[which] = nullptr;
    }
    return ok;
}

// S in the order the products read it: [j][m][species in fours], zero padded.
swopt_status fft_weights(swopt_handle* h)
{
    if (!h->fft) return SWOPT_OK;
    const int P4 = (h->P + 3) / 4;
    std::vector<float> w((size_t)h->Z * h->Q * P4 * 4, 0.f);
    for (int m = 0; m < h->Q; ++m)
        for (int p = 0; p < h->P; ++p)
            for (int j = 0; j < h->Z; ++j)
                w[((size_t)j * h->Q + m) * P4 * 4 + p] =
                    (float)h->Sm64[((size_t)m * h->P + p) * h->Z + j];
    SW_CUDA(cudaMemcpy(h->fft->S4, w.data(), w.size() * sizeof(float), cudaMemcpyHostToDevice));
    return SWOPT_OK;
}

// Plans the transforms for the handle's geometry and builds K^.  No error: a
// geometry that does not fit keeps the direct kernels (h->fft null).
void fft_prepare(swopt_handle* h)
{
    // band of the kernel over all taps: samples reached per depth, and depths per sample
    const int tw = h->tw, kk = h->k * h->k;
    std::vector<int> jlo(h->Z, std::numeric_limits<int>::max()), jhi(h->Z, -1);
    std::vector<int> wlo(tw, std::numeric_limits<int>::max()), whi(tw, -1);
    for (int j = 0; j < h->Z; ++j)
        for (int d = 0; d < kk; ++d) {
            const double* kp = h->K64.data() + ((size_t)j * kk + d) * h->T + h->t0;
            int a = 0, b = tw - 1;
            // outside the run found so far
            for (; a < std::min(tw, jlo[j]) && kp[a] == 0.0; ++a) {}
            for (; b > jhi[j] && b >= a && kp[b] == 0.0; --b) {}
            if (a <= b && kp[a] != 0.0) jlo[j] = std::min(jlo[j], a);
            if (a <= b && kp[b] != 0.0) jhi[j] = std::max(jhi[j], b);
        }
    std::vector<BandEntry> band;
    for (int j = 0; j < h->Z; ++j)
        for (int w = jlo[j]; w <= jhi[j]; ++w) {
            band.push_back({j, w});
            wlo[w] = std::min(wlo[w], j);
            whi[w] = std::max(whi[w], j);
        }
    if (band.empty()) return;
    std::vector<int4> ft, at;
    const long long frows = band_table(wlo, whi, tw, &ft);
    const long long arows = band_table(jlo, jhi, h->Z, &at);
    const int Cz2 = (h->Z + 1) / 2, Ct2 = (tw + 1) / 2;
    const int fchunk = pick_chunk(h->Q, Cz2, spec_warps((int)ft.size()));
    const int achunk = pick_chunk(h->Q, Ct2, spec_warps((int)at.size()));
    if (!fchunk || !achunk) return;

    // lengths: the least estimated time over all pairs (K^ and the spectra through
    // memory at 5 TB/s, the products at 40 TFLOP/s), for a nominal number of
    // states: shards of one problem take the same lengths, hence the same bits.
    // The tiles of a k = 1 kernel do not overlap, so that small ones cost the same in
    // this estimate: few are preferred (one H^T H at 128^2 x 96 in 4 x 4 tiles 717 us,
    // in one 417; 64^2 x 64 139 and 92)
    const double states = 8.0;
    // channel pairs of all planes, on the side where they are most: samples of the
    // states, or depths of the states or species
    const size_t planes = std::max((size_t)h->Q * Ct2, (size_t)std::max(h->Q, h->P) * Cz2);
    double best = 1e300;
    FftAxis by{}, bx{};
    for (const Length& ly : kLengths)
        for (const Length& lx : kLengths) {
            FftAxis y, x;
            if (!make_axis(ly, h->Y, h->r, &y) || !make_axis(lx, h->X, h->r, &x)) continue;
            const double tiles = (double)y.tiles * x.tiles, area = (double)ly.L * lx.L;
            const double kbytes = 0.5 * area * (frows + arows) * kOG * 8.0;
            const double sbytes = tiles * area * 8.0 * 8.0 * (h->P * Cz2 + states * Ct2);
            const double flops = tiles * 0.5 * area * (frows + arows) * kOG * 8.0 * states;
            const double work = 8.0 * tiles * area * h->Q * (double)std::max(Ct2, Cz2);
            // memory limits: 24 GB of K^ (twice with the BF16 one), 8 GB of a workspace for
            // the states' planes (with more species than states it takes up to P / Q of that)
            if (kbytes > 24e9 || work > 8e9) continue;
            double t = std::max(kbytes / 5e12, flops / 40e12) + sbytes / 5e12;
            if (h->r == 0) t *= 1.0 + 0.02 * tiles;
            if (t < best) {
                best = t;
                by = y;
                bx = x;
            }
        }
    if (best > 1e299) return;
    // 32-bit line counts of the transform kernels
    const double lines = (double)by.tiles * bx.tiles * std::max(by.L, bx.L) *
                         std::max(h->Q, h->P) * std::max(std::max(Cz2, Ct2), h->Twp / 2) *
                         (double)std::max(by.L, bx.L);
    if (lines > 2e9) return;

    FftOperator* f = new FftOperator();
    h->fft = f;
    f->y = by;
    f->x = bx;
    f->tiles = by.tiles * bx.tiles;
    f->rows_in = by.tiles == 1 ? h->Y : by.L;
    f->rows_out = by.out;
    f->hx = bx.L / 2 + 1;
    f->blocks = ((long long)by.L * f->hx + kFB - 1) / kFB;
    f->Cz2 = Cz2;
    f->Ct2 = Ct2;
    f->fgroups = (int)ft.size();
    f->agroups = (int)at.size();
    f->frows = frows;
    f->arows = arows;
    f->nband = (int)band.size();
    f->fchunk = fchunk;
    f->achunk = achunk;
    auto upload = [](auto** dst, const auto& v) {
        return try_alloc(dst, v.size()) &&
               cudaMemcpy(*dst, v.data(), v.size() * sizeof(v[0]), cudaMemcpyHostToDevice) ==
                   cudaSuccess;
    };
    auto roots = [](int L) {
        std::vector<float2> w(L);
        for (int n = 0; n < L; ++n) {
            const double a = 2.0 * kPi * n / L;
            w[n] = make_float2((float)std::cos(a), (float)-std::sin(a));
        }
        return w;
    };
    const size_t area = (size_t)by.L * bx.L;
    const size_t marks = 4 + 2 * (size_t)h->Y * (1 + h->X);
    const size_t ws = (size_t)f->tiles * area * planes;
    const bool ok = upload(&f->ftab, ft) && upload(&f->atab, at) && upload(&f->band, band) &&
                    upload(&f->twy, roots(by.L)) && upload(&f->twx, roots(bx.L)) &&
                    try_alloc(&f->w0, ws) && try_alloc(&f->w1, ws) &&
                    try_alloc(&f->marks, marks) &&
                    cudaMemset(f->marks, 0, marks * sizeof(unsigned)) == cudaSuccess &&
                    try_alloc(&f->S4, (size_t)h->Z * h->Q * ((h->P + 3) / 4)) &&
                    fft_weights(h) == SWOPT_OK && build_spectrum(h, 0);
    f->y.tw = f->twy;
    f->x.tw = f->twx;
    if (!ok) fft_release(h);
}

double fft_issued_macs(const swopt_handle* h, int kernel)
{
    const FftOperator* f = h->fft;
    return 4.0 * h->Q * f->tiles * (double)f->blocks * kFB * kOG *
           (double)(kernel == 0 ? f->frows : f->arows);
}

bool fft_prepare_bf16(swopt_handle* h) { return h->fft && build_spectrum(h, 1); }

namespace {

FftShape shape_of(const swopt_handle* h, bool round)
{
    const FftOperator* f = h->fft;
    FftShape s;
    s.y = f->y; s.x = f->x;
    s.Y = h->Y; s.X = h->X; s.Z = h->Z; s.T = h->T; s.N = h->N; s.P = h->P; s.Q = h->Q;
    s.ncyc = h->ncyc; s.Twp = h->Twp; s.t0 = h->t0; s.k = h->k; s.r = h->r;
    s.tiles = f->tiles; s.rows_in = f->rows_in; s.rows_out = f->rows_out;
    s.sel = nullptr;
    s.round = s.round2 = round ? 1 : 0;
    s.Sm = h->Sm; s.Kf = h->Kf;
    s.ftab = f->ftab; s.atab = f->atab; s.marks = f->marks;
    s.gate = h->gate; s.want = h->gate_want;
    return s;
}

bool aligned8(const void* p) { return ((uintptr_t)p & 7u) == 0; }

// Launches a line-transform kernel over `items` lines along axis `ax` (the larger
// count where the device picks between two variants).
template <class Args>
swopt_status launch_lines(swopt_handle* h, void (*kernel)(const Args), const Args& a, unsigned items,
                          const FftAxis& ax, cudaStream_t st)
{
    const size_t smem = (size_t)ax.L * 32 * sizeof(float2);
    if (smem > 48 * 1024)
        SW_CUDA(cudaFuncSetAttribute((const void*)kernel,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024));
    SW_CUDA(launch_pdl(kernel, (items + 31) / 32, 32 * fft_warps(ax), smem, st, a));
    SW_LAUNCHED(h);
    return SWOPT_OK;
}

swopt_status launch_y(swopt_handle* h, const FftShape& s, bool inverse, int planes, int planes2, int C2,
                      const float2* in, float2* out, bool count, cudaStream_t st)
{
    YPass a{};
    a.s = s;
    a.in = in;
    a.out = out;
    a.width = (unsigned)(s.x.L * C2);
    a.items = (unsigned)(planes * s.tiles) * a.width;
    a.items2 = (unsigned)(planes2 * s.tiles) * a.width;
    a.count = count ? 1 : 0;
    return launch_lines(h, inverse ? fft_y_kernel<1> : fft_y_kernel<-1>, a,
                        std::max(a.items, a.items2), s.y, st);
}

template <int MC, bool ADJ, int MAP>
swopt_status launch_spec_mc(swopt_handle* h, const Spec& a, cudaStream_t st)
{
    auto kernel = spec_kernel<MC, ADJ, MAP>;
    const int warps = spec_warps(a.groups);
    const size_t smem = spec_smem(MC, a.in_C2, warps);
    if (smem > 48 * 1024)
        SW_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSpecSmem));
    const dim3 grid((unsigned)h->fft->blocks,
                    (unsigned)(a.s.tiles * (ADJ && MAP == MAP_SPECIES ? 1 : a.chunks)));
    SW_CUDA(launch_pdl(kernel, grid, 32 * warps, smem, st, a));
    SW_LAUNCHED(h);
    return SWOPT_OK;
}

template <bool ADJ, int MAP>
swopt_status launch_spec(swopt_handle* h, const FftShape& s, const float2* in, float2* out,
                         cudaStream_t st)
{
    const FftOperator* f = h->fft;
    const int mc = ADJ ? f->achunk : f->fchunk;
    Spec a{};
    a.s = s;
    a.in = in;
    a.out = out;
    a.K = reinterpret_cast<const float4*>(ADJ ? f->KA[s.round] : f->KF[s.round]);
    a.K2 = reinterpret_cast<const float4*>(ADJ ? f->KA[s.round2] : f->KF[s.round2]);
    if (!a.K || !a.K2) {
        set_error("internal: no spectrum of the kernel for the selected precision");
        return SWOPT_ERR_DEVICE_CHECK;
    }
    a.tab = ADJ ? f->atab : f->ftab;
    a.groups = ADJ ? f->agroups : f->fgroups;
    a.rows = ADJ ? f->arows : f->frows;
    a.in_C2 = ADJ ? f->Ct2 : f->Cz2;
    a.out_C2 = ADJ ? f->Cz2 : f->Ct2;
    a.chunks = (s.Q + mc - 1) / mc;
    a.hx = f->hx;
    a.S4 = f->S4;
    switch (mc) {
    case 2: return launch_spec_mc<2, ADJ, MAP>(h, a, st);
    case 4: return launch_spec_mc<4, ADJ, MAP>(h, a, st);
    case 6: return launch_spec_mc<6, ADJ, MAP>(h, a, st);
    case 8: return launch_spec_mc<8, ADJ, MAP>(h, a, st);
    default: return launch_spec_mc<10, ADJ, MAP>(h, a, st);
    }
}

}  // namespace

namespace {

// c (c2 in the second variant) -> the spectra of the state images' A, transformed
// back along y, in f->w1.
swopt_status forward_to_lines(swopt_handle* h, const FftShape& s, const float* c, const float* c2,
                              cudaStream_t st)
{
    FftOperator* f = h->fft;
    const int planes = s.round ? h->Q : h->P, planes2 = s.round2 ? h->Q : h->P;
    const unsigned per = (unsigned)(f->tiles * f->rows_in * f->Cz2);
    XForward a{};
    a.s = s;
    a.src = c;
    a.src2 = c2;
    a.out = f->w0;
    a.C2 = f->Cz2;
    a.vec = (h->Z % 2) == 0 && aligned8(c) && aligned8(c2);
    a.items = (unsigned)planes * per;
    a.items2 = (unsigned)planes2 * per;
    const bool gated = s.round != s.round2;  // states first, species second
    SW_TRY(launch_lines(h,
                        gated     ? fft_x_forward_kernel<SRC_GATED>
                        : s.round ? fft_x_forward_kernel<SRC_STATES>
                                  : fft_x_forward_kernel<SRC_C>,
                        a, std::max(a.items, a.items2), f->x, st));
    SW_TRY(launch_y(h, s, false, planes, planes2, f->Cz2, f->w0, f->w1, true, st));
    if (gated) SW_TRY((launch_spec<false, MAP_GATED>(h, s, f->w1, f->w0, st)));
    else if (s.round) SW_TRY((launch_spec<false, MAP_NONE>(h, s, f->w1, f->w0, st)));
    else SW_TRY((launch_spec<false, MAP_SPECIES>(h, s, f->w1, f->w0, st)));
    return launch_y(h, s, true, h->Q, h->Q, f->Ct2, f->w0, f->w1, false, st);
}

// The lines of A^T's input, transformed along x in f->w0 -> the image outputs.
// first: the launch before this was the call's first one.
swopt_status adjoint_from_lines(swopt_handle* h, const FftShape& s, const float* r, bool from_y,
                                bool first, const FftImage& img, cudaStream_t st)
{
    FftOperator* f = h->fft;
    SW_TRY(launch_y(h, s, false, h->Q, h->Q, f->Ct2, f->w0, f->w1, first, st));
    if (img.per_state) SW_TRY((launch_spec<true, MAP_NONE>(h, s, f->w1, f->w0, st)));
    else SW_TRY((launch_spec<true, MAP_SPECIES>(h, s, f->w1, f->w0, st)));
    const int planes = img.per_state ? h->Q : h->P;
    SW_TRY(launch_y(h, s, true, planes, planes, f->Cz2, f->w0, f->w1, false, st));
    XInverse v{};
    v.s = s;
    v.in = f->w1;
    v.C2 = f->Cz2;
    v.items = (unsigned)(planes * f->tiles * f->rows_out * f->Cz2);
    v.out = img.out;
    v.add = img.add;
    v.add2 = img.add2;
    v.alpha = img.alpha;
    v.xi = img.xi;
    v.G = img.G;
    v.scal = h->scal;
    v.r = r;
    v.from_y = from_y ? 1 : 0;
    v.per_state = img.per_state ? 1 : 0;
    v.vec = (h->Z % 2) == 0 && aligned8(img.out) && aligned8(img.xi) && aligned8(img.G);
    return launch_lines(h,
                        img.refine ? fft_x_image_kernel<IMG_REFINE> : fft_x_image_kernel<IMG_STORE>, v,
                        v.items, f->x, st);
}

}  // namespace

swopt_status fft_forward(swopt_handle* h, const float* c, const float* ytil, int scale, bool round,
                         cudaStream_t st)
{
    FftOperator* f = h->fft;
    const FftShape s = shape_of(h, round);
    ProfileRec rec;
    prof_begin(h, 0, st, &rec);
    SW_TRY(forward_to_lines(h, s, c, c, st));
    XInverse v{};
    v.s = s;
    v.in = f->w1;
    v.C2 = f->Ct2;
    v.q_end = h->Twp / 2;
    v.items = (unsigned)(h->Q * f->tiles * f->rows_out * v.q_end);
    v.out = h->u;
    v.ytil = ytil;
    v.Cmf = scale ? h->Cmf : nullptr;
    v.c = c;
    SW_TRY(launch_lines(h, fft_x_u_kernel, v, v.items, f->x, st));
    prof_end(h, &rec, st);
    return SWOPT_OK;
}

swopt_status fft_adjoint(swopt_handle* h, const float* src, bool from_y, bool round,
                         const FftImage& img, cudaStream_t st)
{
    FftOperator* f = h->fft;
    const FftShape s = shape_of(h, round);
    XForward a{};
    a.s = s;
    a.src = src;
    a.out = f->w0;
    a.C2 = f->Ct2;
    a.vec = !from_y || ((h->T % 2) == 0 && aligned8(src));
    a.items = (unsigned)(h->Q * f->tiles * f->rows_in * f->Ct2);
    ProfileRec rec;
    prof_begin(h, 1, st, &rec);
    SW_TRY(launch_lines(h, from_y ? fft_x_forward_kernel<SRC_Y> : fft_x_forward_kernel<SRC_U>, a,
                        a.items, f->x, st));
    SW_TRY(adjoint_from_lines(h, s, src, from_y, true, img, st));
    prof_end(h, &rec, st);
    return SWOPT_OK;
}

namespace {

// From the lines of A in f->w1 through the residual to A^T's output.
swopt_status residual_to_image(swopt_handle* h, const FftShape& s, const XResidual& args,
                               const FftImage& img, cudaStream_t st)
{
    FftOperator* f = h->fft;
    XResidual v = args;
    v.s = s;
    v.in = f->w1;
    v.out = f->w0;
    v.C2 = f->Ct2;
    v.items = (unsigned)(h->Q * h->Y * f->Ct2);
    v.Cmf = h->Cmf;
    v.u = h->u;
    v.ysq = h->scal + kScalYsq;
    const size_t smem = (size_t)f->x.L * 32 * sizeof(float2);
    if (smem > 48 * 1024)
        SW_CUDA(cudaFuncSetAttribute(fft_x_residual_kernel,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024));
    // nine sub-transforms a pass: one round of nine warps
    const int warps = std::max(f->x.R1, f->x.R2) == 9 ? 9 : fft_warps(f->x);
    SW_CUDA(launch_pdl(fft_x_residual_kernel, (v.items + 31) / 32, 32 * warps, smem, st, v));
    SW_LAUNCHED(h);
    return adjoint_from_lines(h, s, h->u, false, false, img, st);
}

}  // namespace

swopt_status fft_normal(swopt_handle* h, const float* c, const float* ytil, bool round, bool keep_u,
                        const FftImage& img, cudaStream_t st)
{
    if (h->fft->tiles > 1) {
        SW_TRY(fft_forward(h, c, ytil, 1, round, st));
        return fft_adjoint(h, h->u, false, round, img, st);
    }
    const FftShape s = shape_of(h, round);
    ProfileRec rec;
    prof_begin(h, 0, st, &rec);
    SW_TRY(forward_to_lines(h, s, c, c, st));
    prof_end(h, &rec, st);
    prof_begin(h, 1, st, &rec);
    XResidual v{};
    v.ytil = v.ytil2 = ytil;
    v.c = v.c2 = c;
    v.keep = keep_u ? 1 : 0;
    SW_TRY(residual_to_image(h, s, v, img, st));
    prof_end(h, &rec, st);
    return SWOPT_OK;
}

bool fft_refine_gated(const swopt_handle* h) { return h->fft->tiles == 1; }

swopt_status fft_refine(swopt_handle* h, const float* delta, const float* c, const float* ytil,
                        bool round, bool round2, const FftImage& image, cudaStream_t st)
{
    FftShape s = shape_of(h, round);
    s.sel = h->sched;
    s.round2 = round2 ? 1 : 0;
    FftImage img = image;
    img.add = 1;
    img.add2 = 0;
    // the launches count as the increment's or the exact gradient's, as decided
    ProfileRec r0, r2;
    auto gated = [&](auto f) {
        const int* g = h->gate;
        h->gate = h->sched;
        f();
        h->gate = g;
    };
    auto begin = [&](int kernel) {
        gated([&] {
            prof_begin(h, kernel, st, &r0);
            h->in_ref = true;
            prof_begin(h, kernel, st, &r2);
            h->in_ref = false;
        });
    };
    auto end = [&] {
        gated([&] {
            prof_end(h, &r0, st);
            prof_end(h, &r2, st);
        });
    };
    begin(0);
    SW_TRY(forward_to_lines(h, s, delta, c, st));
    end();
    begin(1);
    XResidual v{};
    v.ytil2 = ytil;
    v.c = delta;
    v.c2 = c;
    SW_TRY(residual_to_image(h, s, v, img, st));
    end();
    return SWOPT_OK;
}

}  // namespace swopt
