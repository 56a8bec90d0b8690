// zm_fft.cu -- low-order velocity by FFT Riesz transforms (paper Sec. 2: the low-order Z-Model
// approximates the Birkhoff-Rott integral with FFTs; Sec. 3.1 ZModel Order::Low; periodic only):
//     s = R1 w1 + R2 w2,  R_l^(k) = -i k_l / |k|,  k_l = 2 pi m_l / L_l,
//     multiplier zero at k = 0 and on the Nyquist row and column;  u = -1/2 s N,
//     Phi = q + 1/2 |u|^2.
// The two real fields are packed as c = w1 + i w2 and one complex transform suffices, because
// s = Re IFFT[(m1 - i m2) FFT(c)] with m_l = -i k_l/|k| (the imaginary part of that inverse is R1 w2
// - R2 w1 and is dropped).  Three passes, each reading and writing the n1 x n2 complex field once:
//   pass A: rows (along alpha2) forward, transposed write          [n1][n2] -> [n2][n1]
//   pass B: rows of the transpose (along alpha1) forward, multiply by -(k2 + i k1)/|k|,
//           inverse along alpha1, transposed write                  [n2][n1] -> [n1][n2]
//   pass C: rows inverse along alpha2, real part / (n1 n2), epilogue u = -s/2 N, Phi.
//
// Arithmetic: 60-bit integers (zm_fix.cuh), because the FP64 pipe bound the passes (216 FP64
// instructions per point at 4096^2, 7.0 ms per evaluation at 85 % of that pipe).  A CTA holds complete
// rows in shared memory with one power-of-two unit for all of them.  The log2 L radix-2 stages run in
// chunks of K <= 4 stages on groups of 2^K values in registers (radix-2^2 butterflies, bit-reversed
// order out for decimation in frequency, in for decimation in time); before each chunk the values
// are shifted to leave room for its growth of 2^K, by what the OR of all magnitudes after the last
// chunk says, so that a spectrum of a few modes keeps its precision in both directions.  The rounding
// noise, about one unit per chunk against row maxima of 2^55 to 2^60, is below that of FP64
// butterflies.  Each CTA leaves the exponent of its unit beside its output, and the largest one
// in a word that the next pass aligns its input to.  A value that is not finite sets that word
// beyond every exponent, and all results are NaN, as they would be in FP64.
// ms per evaluation, FP64 butterflies / integers: 1024^2 0.452 / 0.102, 4096^2 6.85 / 1.44, 4864^2 13.18 /
// 2.88, 512^2 0.115 / 0.052, 152 x 304 0.138 / 0.064, 128^2 0.031 / 0.029 (latency).  Relative error of u
// against a long double transform: 128^2 3.8e-16 / 3.2e-16, 256^2 4.7e-16 / 4.3e-16, 512^2 5.6e-16 /
// 5.2e-16, 152 x 304 5.5e-16 / 5.3e-16, 608 x 152 5.5e-16 / 5.6e-16.  What bounds it now: latency at 16
// warps per SM (128 registers for 16 values), the schedulers issuing in 34 to 47 % of cycles.
//
// Sides L = R M with M = 2^a (a >= 3) and R odd (3 .. 19; 4864 = 19 x 256 is the paper's
// low-order mesh, Sec. 5.1) add one radix-R stage: before the length-M transforms in decimation
// in frequency, after them in decimation in time.  Frequency R k1 + k2 then sits at position
// k2 M + bitrev(k1) of a row.
//
// The multipliers k2/|k|, k1/|k| come from a table over a quarter of the spectrum (4 bytes per
// mesh point): forming them took 16 FP64 instructions per point, as much time as all of the
// integer transforms.
#include <algorithm>
#include <type_traits>

#include "zm_fix.cuh"

namespace zm {
namespace {

constexpr int kElems = 4096;          // complex values per CTA (or one row)
constexpr int kMaxSide = 8192;        // 2^13
constexpr int kNotFinite = 1 << 20;   // "exponent" of a field with a NaN or an infinity
constexpr int kAllZero = -kNotFinite;  // of a field of zeros (whose integers may hold rounding constants)

__device__ __forceinline__ int bitrev(int j, int logL) { return (int)(__brev((unsigned)j) >> (32 - logL)); }
__device__ __forceinline__ int phys(int i) { return i + (i >> 4); }  // one pad entry per 16

// ---- butterflies on register groups ----------------------------------------------------------------

// Decimation in frequency on v[m], v[m+Q], v[m+2Q], v[m+3Q]; e1 = exponent of W_{4S}^p on W_L (a
// compile-time zero drops the products).
template <int Q>
__device__ __forceinline__ void bfly_dif(Z *v, int m, int e1, bool unit, const int4 *__restrict__ tw, int sgn)
{
    const Z a0 = v[m], a1 = v[m + Q], a2 = v[m + 2 * Q], a3 = v[m + 3 * Q];
    const Z s02 = zadd(a0, a2), d02 = zsub(a0, a2), s13 = zadd(a1, a3), d13 = zsub(a1, a3);
    v[m] = zadd(s02, s13);
    const Z x2 = zsub(s02, s13), x1 = zadd_i(d02, d13, sgn), x3 = zadd_i(d02, d13, -sgn);
    if (unit) {
        v[m + Q] = x2;
        v[m + 2 * Q] = x1;
        v[m + 3 * Q] = x3;
    } else {
        v[m + Q] = zmul(x2, __ldg(tw + 2 * e1), -sgn);
        v[m + 2 * Q] = zmul(x1, __ldg(tw + e1), -sgn);
        v[m + 3 * Q] = zmul(x3, __ldg(tw + 3 * e1), -sgn);
    }
}

template <int Q>
__device__ __forceinline__ void bfly_dit(Z *v, int m, int e1, bool unit, const int4 *__restrict__ tw, int sgn)
{
    const Z a0 = v[m];
    Z c1 = v[m + Q], c2 = v[m + 2 * Q], c3 = v[m + 3 * Q];
    if (!unit) {
        c1 = zmul(c1, __ldg(tw + 2 * e1), -sgn);
        c2 = zmul(c2, __ldg(tw + e1), -sgn);
        c3 = zmul(c3, __ldg(tw + 3 * e1), -sgn);
    }
    const Z s01 = zadd(a0, c1), d01 = zsub(a0, c1), s23 = zadd(c2, c3), d23 = zsub(c2, c3);
    v[m] = zadd(s01, s23);
    v[m + 2 * Q] = zsub(s01, s23);
    v[m + Q] = zadd_i(d01, d23, sgn);
    v[m + 3 * Q] = zadd_i(d01, d23, -sgn);
}

// The K stages of one chunk on a register group: v[m] is the value at position base + m h of its
// row (h = 2^LH, pos = base mod h).  Table tw: W_L^k = exp(-2 pi i k / L), k < 3L/4.
template <int K, int LH, int L>
__device__ __forceinline__ void dif_chunk(Z *v, int pos, const int4 *__restrict__ tw, int sgn)
{
    constexpr int R = 1 << K;
    if (K & 1) {  // one radix-2 stage at the top span
#pragma unroll
        for (int m = 0; m < R / 2; ++m) {
            const Z a = v[m], b = v[m + R / 2];
            v[m] = zadd(a, b);
            const Z d = zsub(a, b);
            const int e = (pos + (m << LH)) << (L - LH - K);
            v[m + R / 2] = (LH == 0 && m == 0) ? d : zmul(d, __ldg(tw + e), -sgn);
        }
    }
#pragma unroll
    for (int jj = (K & 1) ? K - 3 : K - 2; jj >= 0; jj -= 2) {
#pragma unroll
        for (int m = 0; m < R; ++m) {
            if ((m & ((4 << jj) - 1)) >= (1 << jj)) continue;  // quadruple leaders only
            const int r = m & ((1 << jj) - 1);
            const int e1 = (pos + (r << LH)) << (L - LH - jj - 2);
            if (jj == 0) bfly_dif<1>(v, m, e1, LH == 0 && r == 0, tw, sgn);
            else bfly_dif<4>(v, m, e1, LH == 0 && r == 0, tw, sgn);
        }
    }
}

template <int K, int LH, int L>
__device__ __forceinline__ void dit_chunk(Z *v, int pos, const int4 *__restrict__ tw, int sgn)
{
    constexpr int R = 1 << K;
#pragma unroll
    for (int jj = 0; jj + 2 <= K; jj += 2) {
#pragma unroll
        for (int m = 0; m < R; ++m) {
            if ((m & ((4 << jj) - 1)) >= (1 << jj)) continue;
            const int r = m & ((1 << jj) - 1);
            const int e1 = (pos + (r << LH)) << (L - LH - jj - 2);
            if (jj == 0) bfly_dit<1>(v, m, e1, LH == 0 && r == 0, tw, sgn);
            else bfly_dit<4>(v, m, e1, LH == 0 && r == 0, tw, sgn);
        }
    }
    if (K & 1) {
#pragma unroll
        for (int m = 0; m < R / 2; ++m) {
            const Z a = v[m];
            Z b = v[m + R / 2];
            const int e = (pos + (m << LH)) << (L - LH - K);
            if (!(LH == 0 && m == 0)) b = zmul(b, __ldg(tw + e), -sgn);
            v[m] = zadd(a, b);
            v[m + R / 2] = zsub(a, b);
        }
    }
}

// Chunk plan per row length 2^l: ceil(l / 4) chunks of near-equal size, the larger ones last.
constexpr int nc_of(int l) { return (l + 3) / 4; }
constexpr int k_of(int l, int c) { return l / nc_of(l) + (c >= nc_of(l) - l % nc_of(l) ? 1 : 0); }
constexpr int lh_of(int l, int c) { return c < 0 ? l : lh_of(l, c - 1) - k_of(l, c); }

struct Grp {
    int row, pos, base;
};
__device__ __forceinline__ Grp group_of(int g, int K, int lh, int l)
{
    const int gi = g & ((1 << (l - K)) - 1);
    const int pos = gi & ((1 << lh) - 1);
    return Grp{g >> (l - K), pos, ((gi >> lh) << (lh + K)) + pos};
}

// ---- the CTA's unit -----------------------------------------------------------------------------------
// Shared words: one OR of magnitudes per chunk, in the order in which the chunks run, and two norms.
constexpr int kSlots = 14, kNorm = 12;

__device__ __forceinline__ void publish_or(unsigned *word, unsigned o)
{
    o = __reduce_or_sync(0xffffffffu, o);
    if ((threadIdx.x & 31) == 0 && o) atomicOr(word, o);
}

// State carried through a pass: the shift that the next chunk applies on load, the exponent of the
// unit (value = integer 2^e), and the next shared word.
struct Unit {
    int e;
    unsigned *word;
    Shift sh;  // for the next load
};
// After a barrier that follows publish_or(u.word, ..): the shift that leaves room for 2^k.
template <bool kLeft>
__device__ __forceinline__ void next_room(Unit &u, int k)
{
    int s = room_shift(*u.word, k);
    if (!kLeft) s = max(s, 0);
    u.sh = make_shift(s);
    u.e += s;
    ++u.word;
}

// One chunk over all rows in shared memory: load (shifted), K stages, store; the magnitudes' OR goes to
// u.word.  post(v, group): applied to each group before the store.
struct NoPost {
    __device__ __forceinline__ void operator()(Z *, const Grp &) const {}
};
template <int K, bool kDif, int L, int LH, bool kLeft, class Post = NoPost>
__device__ __forceinline__ void chunk_pass(ulonglong2 *sx, int rows, const int4 *__restrict__ tw, int sgn,
                                           const Unit &u, Post post = Post())
{
    constexpr int R = 1 << K;
    const int ngroups = rows << (L - K);
    unsigned o = 0;
    for (int g = threadIdx.x; g < ngroups; g += blockDim.x) {
        const Grp q = group_of(g, K, LH, L);
        Z v[R];
#pragma unroll
        for (int m = 0; m < R; ++m) {
            const Z a = ldz(sx[phys((q.row << L) + q.base + (m << LH))]);
            v[m] = kLeft ? zshift(a, u.sh) : zshift_right(a, u.sh);
        }
        if (kDif) dif_chunk<K, LH, L>(v, q.pos, tw, sgn);
        else dit_chunk<K, LH, L>(v, q.pos, tw, sgn);
        post(v, q);
#pragma unroll
        for (int m = 0; m < R; ++m) {
            or_mag(o, v[m]);
            sx[phys((q.row << L) + q.base + (m << LH))] = stz(v[m]);
        }
    }
    __syncwarp();
    publish_or(u.word, o);
}

// Forward chunks C .. CEnd; kLeft: chunk C may shift to the left (the first one of a pass).
template <int L, int C, int CEnd, bool kLeft>
__device__ __forceinline__ void dif_seq(ulonglong2 *sx, const int4 *__restrict__ tw, int rows, int sgn, Unit &u)
{
    if constexpr (C <= CEnd) {
        constexpr int K = k_of(L, C);
        next_room<kLeft>(u, K);
        chunk_pass<K, true, L, lh_of(L, C), kLeft>(sx, rows, tw, sgn, u);
        __syncthreads();
        dif_seq<L, C + 1, CEnd, false>(sx, tw, rows, sgn, u);
    }
}

// Inverse chunks C, C - 1, .., 0.
template <int L, int C>
__device__ __forceinline__ void dit_seq(ulonglong2 *sx, const int4 *__restrict__ tw, int rows, int sgn, Unit &u)
{
    if constexpr (C >= 0) {
        constexpr int K = k_of(L, C);
        next_room<false>(u, K);
        chunk_pass<K, false, L, lh_of(L, C), false>(sx, rows, tw, sgn, u);
        __syncthreads();
        dit_seq<L, C - 1>(sx, tw, rows, sgn, u);
    }
}

// ---- the radix-R stage ------------------------------------------------------------------------------
// DFT of length R (odd), v[t] -> sum_t v[t] W_R^(t k) (conjugate roots for sgn > 0); output k goes to
// out(k, X_k).  With the sums s_n = v_n + v_{R-n} and differences d_n = v_n - v_{R-n}, outputs k and R - k
// share A_k = v0 + sum_n s_n Re W^(nk) and B_k = sum_n d_n Im W^(nk).  Roots (table rt) in units of 2^-59:
// the cross products of a sum then stay below 2^63 for column sums below 2^60.  The dropped products of
// the low limbs, xl wl / 2^59, have a mean (xl is uniform) that the table holds summed per k.
__device__ __forceinline__ void acc_real(long long &h, long long &c, long long x, int wh, int wl)
{
    const int xh = (int)(x >> kLimb), xl = (int)x & kLow;
    h = mad_w(xh, wh, h);
    c = mad_w(xh, wl, c);
    c = mad_w(xl, wh, c);
}
__device__ __forceinline__ long long acc_value(long long h, long long c) { return (h << 1) + (c >> (kLimb - 1)); }

template <int R, class Out>
__device__ __forceinline__ void dft_fix(Z (&v)[R], const int4 *__restrict__ rt, int sgn, Out out)
{
    constexpr int H = (R - 1) / 2;
    Z x0 = v[0];
#pragma unroll
    for (int n = 1; n <= H; ++n) {
        const Z a = v[n], b = v[R - n];
        v[n] = zadd(a, b);
        v[R - n] = zsub(a, b);
        x0 = zadd(x0, v[n]);
    }
    out(0, x0);
#pragma unroll 1
    for (int k = 1; k <= H; ++k) {
        const longlong2 mean = __ldg(reinterpret_cast<const longlong2 *>(rt) + R + k);
        long long har = 0, hai = 0, hbr = 0, hbi = 0, car = mean.x, cai = mean.x, cbr = mean.y, cbi = mean.y;
#pragma unroll
        for (int n = 1; n <= H; ++n) {
            const int4 w = __ldg(rt + (n * k) % R);
            acc_real(har, car, v[n].re, w.x, w.y);
            acc_real(hai, cai, v[n].im, w.x, w.y);
            acc_real(hbr, cbr, v[R - n].re, w.z, w.w);
            acc_real(hbi, cbi, v[R - n].im, w.z, w.w);
        }
        const Z A{v[0].re + acc_value(har, car), v[0].im + acc_value(hai, cai)};
        const Z B{acc_value(hbr, cbr), acc_value(hbi, cbi)};
        out(k, zadd_i(A, B, -sgn));      // the table holds W = exp(-2 pi i / R): sgn < 0 adds i B
        out(R - k, zadd_i(A, B, sgn));
    }
}

// Decimation in frequency: column n1 of each row of length L = R M, in place; twl: W_L^k, k < L; the roots
// W_R follow at twl + L.  Not inlined: each radix is compiled once per pass kernel.
template <int R>
__device__ __noinline__ void radix_dif(ulonglong2 *sx, int rows, int lM, const int4 *__restrict__ twl, int sgn,
                                       const Unit u)
{
    const int M = 1 << lM, L = R * M;
    unsigned o = 0;
    for (int b = threadIdx.x; b < rows * M; b += blockDim.x) {
        const int row = b >> lM, n1 = b & (M - 1);
        if (!ZM_IDX_OK(row, rows)) continue;
        const int base = row * L + n1;
        Z v[R];
#pragma unroll
        for (int t = 0; t < R; ++t) v[t] = zshift(ldz(sx[phys(base + M * t)]), u.sh);
        dft_fix<R>(v, twl + L, sgn, [&](int k, Z x) {
            if (k) x = zmul(x, __ldg(twl + n1 * k), -sgn);
            or_mag(o, x);
            sx[phys(base + M * k)] = stz(x);
        });
    }
    __syncwarp();
    publish_or(u.word, o);
}

template <int R>
__device__ __noinline__ void radix_dit(ulonglong2 *sx, int rows, int lM, const int4 *__restrict__ twl, int sgn,
                                       const Unit u)
{
    const int M = 1 << lM, L = R * M;
    unsigned o = 0;
    for (int b = threadIdx.x; b < rows * M; b += blockDim.x) {
        const int row = b >> lM, n1 = b & (M - 1);
        if (!ZM_IDX_OK(row, rows)) continue;
        const int base = row * L + n1;
        Z v[R];
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const Z x = zshift_right(ldz(sx[phys(base + M * k)]), u.sh);
            v[k] = k ? zmul(x, __ldg(twl + n1 * k), -sgn) : x;
        }
        dft_fix<R>(v, twl + L, sgn, [&](int t, Z x) {
            or_mag(o, x);
            sx[phys(base + M * t)] = stz(x);
        });
    }
    __syncwarp();
    publish_or(u.word, o);
}

#define ZM_FOR_RADICES(X) X(3) X(5) X(7) X(9) X(11) X(13) X(15) X(17) X(19)

// The stage's shift comes from the largest column sum of |re| + |im|, which bounds every output and
// partial sum: R times the largest value would leave a spectrum of a few modes four bits short
// (relative error of u at 152 x 304: 1.4e-15 with that bound).  `norm`: a cleared shared word.
template <bool kDif, bool kLeft>
__device__ __forceinline__ void radix_stage(ulonglong2 *sx, int rows, int R, int lM, const int4 *__restrict__ twl,
                                            int sgn, Unit &u, unsigned *norm)
{
    const int M = 1 << lM;
    unsigned top = 0;
    for (int b = threadIdx.x; b < rows * M; b += blockDim.x) {
        const int base = (b >> lM) * R * M + (b & (M - 1));
        unsigned long long sum = 0;  // in units of 2^5: at most 38 terms below 2^58
        for (int t = 0; t < R; ++t) {
            const Z a = ldz(sx[phys(base + M * t)]);
            sum += (unsigned long long)(llabs(a.re) >> 5) + (unsigned long long)(llabs(a.im) >> 5);
        }
        top = max(top, (unsigned)(sum >> 32));
    }
    __syncwarp();
    top = __reduce_max_sync(0xffffffffu, top);
    if ((threadIdx.x & 31) == 0) atomicMax(norm, top);
    __syncthreads();
    int s = 32 - __clz((int)*norm) + 37 - 60;
    if (!kLeft) s = max(s, 0);
    u.sh = make_shift(s);
    u.e += s;
    ++u.word;
    switch (R) {
#define ZM_CASE(r)                                                     \
    case r:                                                            \
        if (kDif) radix_dif<r>(sx, rows, lM, twl, sgn, u);             \
        else radix_dit<r>(sx, rows, lM, twl, sgn, u);                  \
        break;
        ZM_FOR_RADICES(ZM_CASE)
#undef ZM_CASE
    default: break;
    }
    __syncthreads();
}

// ---- passes -----------------------------------------------------------------------------------------
// One side: L = R 2^A; tables W_{2^A} (k < 3/4 2^A) and, for R > 1, W_L and W_R.
struct Side {
    int L, R, A;
    const int4 *tw, *twl;
};

// Exponent words of the two passes that hand data on: per CTA of the writing pass, and their maximum.
struct Exps {
    int *e;    // [CTAs]
    int *max;
    int lr;    // log2 of the rows per writing CTA
};

// Position in a row after decimation in frequency of the output with index f.
template <int A, bool kMix>
__device__ __forceinline__ int dif_pos(int f, int R)
{
    if (!kMix) return bitrev(f, A);
    const int k1 = f / R;
    return (f - k1 * R) * (1 << A) + bitrev(k1, A);
}

// Whole rows forward (sgn < 0) or inverse (sgn > 0) by decimation in frequency, data staged in sx and
// its OR published.
template <int A, bool kMix>
__device__ __forceinline__ void rows_dif(ulonglong2 *sx, int rows, const Side &s, int sgn, Unit &u,
                                         unsigned *norm)
{
    if (kMix) {
        radix_stage<true, true>(sx, rows, s.R, A, s.twl, sgn, u, norm);
        dif_seq<A, 0, nc_of(A) - 1, false>(sx, s.tw, rows * s.R, sgn, u);
    } else {
        dif_seq<A, 0, nc_of(A) - 1, true>(sx, s.tw, rows, sgn, u);
    }
}

constexpr int threads_for(int A, bool mix) { return mix ? 256 : ((1 << A) > kElems ? (1 << A) : kElems) / 16; }
constexpr int minb_for(int A, bool mix) { return mix || A <= 12 ? 2 : 1; }

// Elements a thread has in flight when a pass reads or writes its rows (one at a time left the passes
// waiting for HBM: 4096 x 4096 FFT 1.75 ms per evaluation).
constexpr int kBatch = 8;

// The field handed on by the last pass, rows row0 .. of length `len`, aligned to the largest exponent,
// into shared memory.  Element (row, k) was written by CTA k >> in.lr of the last pass.
__device__ __forceinline__ void stage_rows(ulonglong2 *sx, int rows, int len, const ulonglong2 *__restrict__ src,
                                           const Exps &in, int emax, unsigned *word)
{
    unsigned o = 0;
    const int total = rows * len;
    int k = threadIdx.x % len;
    const int step = blockDim.x % len;
    for (int e0 = threadIdx.x; e0 < total; e0 += kBatch * blockDim.x) {
        ulonglong2 v[kBatch];
        int d[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int e = e0 + b * blockDim.x;
            if (e < total) {
                v[b] = __ldcs(src + e);
                d[b] = __ldg(in.e + (k >> in.lr));
            }
            k += step;
            if (k >= len) k -= len;
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int e = e0 + b * blockDim.x;
            if (e < total) {
                const Z a = zshift_right(ldz(v[b]), make_shift(min(emax - d[b], 62)));
                or_mag(o, a);
                sx[phys(e)] = stz(a);
            }
        }
    }
    __syncwarp();
    publish_or(word, o);
}

__device__ __forceinline__ void clear_words(unsigned *words, int count)
{
    if (threadIdx.x < count) words[threadIdx.x] = 0u;
    __syncthreads();
}

// The leading word of |v|, at least 1 where v is not zero (denormal numbers have theirs in the other).
__device__ __forceinline__ unsigned size_bits(double v)
{
    return ((unsigned)__double2hiint(v) & 0x7fffffffu) | (__double2loint(v) != 0 ? 1u : 0u);
}

// pass A: rows i of length n2 from w1 + i w2; forward; write out[j][i] (transposed).
template <int A, bool kMix>
__global__ void __launch_bounds__(threads_for(A, kMix), minb_for(A, kMix))
    pass_a(int n1, Side s2, int lr, const double *__restrict__ w, ulonglong2 *__restrict__ out, Exps ea, int *reset)
{
    extern __shared__ ulonglong2 sx[];
    __shared__ unsigned words[kSlots];
    clear_words(words, kSlots);
    const int L = s2.L, rows = 1 << lr, i0 = blockIdx.x * rows;
    if (!ZM_IDX_OK(i0 + rows - 1, n1)) return;  // checked build: the CTA's rows exist
    const size_t N = (size_t)n1 * L;
    const double *w1 = w + (size_t)i0 * L, *w2 = w1 + N;
    unsigned mx = 0;
    const int total = rows * L;
    for (int e0 = threadIdx.x; e0 < total; e0 += kBatch * blockDim.x) {
        double a[kBatch], b[kBatch];
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int e = e0 + k * blockDim.x;
            if (e < total) {
                a[k] = __ldcs(w1 + e);
                b[k] = __ldcs(w2 + e);
            }
        }
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int e = e0 + k * blockDim.x;
            if (e < total) {
                mx = max(mx, max(size_bits(a[k]), size_bits(b[k])));
                sx[phys(e)] = make_ulonglong2((unsigned long long)__double_as_longlong(a[k]),
                                              (unsigned long long)__double_as_longlong(b[k]));
            }
        }
    }
    __syncwarp();
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(&words[0], mx);
    __syncthreads();
    mx = words[0];
    // |w| < 2^eb (denormal numbers: the least exponent); to integers below 2^54
    const int eb = max((int)(mx >> 20) - 1022, -1021);
    unsigned o = 0;
    for (int e = threadIdx.x; e < rows * L; e += blockDim.x) {  // the thread's own elements
        const ulonglong2 v = sx[phys(e)];
        const Z a{fix_of(v.x, eb), fix_of(v.y, eb)};
        or_mag(o, a);
        sx[phys(e)] = stz(a);
    }
    __syncwarp();
    publish_or(&words[1], o);
    __syncthreads();
    Unit u{eb - 54, &words[1], make_shift(0)};
    rows_dif<A, kMix>(sx, rows, s2, -1, u, &words[kNorm]);
    // in storage order: each output row j gets `rows` adjacent values wherever j lies, and reading in
    // the order of j would take one shared-memory bank in eight
#pragma unroll 4
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int pos = e >> lr, r = e & (rows - 1);
        const int j = kMix ? s2.R * bitrev(pos & ((1 << A) - 1), A) + (pos >> A) : bitrev(pos, A);
        const size_t dst = (size_t)j * n1 + i0 + r;
        if (ZM_IDX_OK(dst, N)) out[dst] = sx[phys(r * L + pos)];
    }
    if (threadIdx.x == 0) {
        const int e = mx >= 0x7ff00000u ? kNotFinite : (mx ? u.e : kAllZero);
        ea.e[blockIdx.x] = e;
        atomicMax(ea.max, e);
        if (blockIdx.x == 0) *reset = kAllZero;  // pass B's maximum: not in use now
    }
}

// The multiplier on a group of 2^K consecutive (bit-reversed) positions after the last forward chunk:
// applied before the store, so that the product costs no pass of its own.  The rows are the R sub-rows
// of each column.
template <int A, int K, bool kMix>
struct Multiply {
    int j0, n1, n2, R;
    const int4 *__restrict__ mult;
    __device__ __forceinline__ void operator()(Z *v, const Grp &q) const
    {
        const int ib = bitrev(q.base, A);
        int col = j0 + q.row, k2 = 0;
        if (kMix) {
            const int r = q.row / R;
            col = j0 + r;
            k2 = q.row - r * R;
        }
        const int m2 = 2 * col < n2 ? col : col - n2;
        const int4 *mc = mult + (size_t)abs(m2) * (n1 / 2 + 1);
#pragma unroll
        for (int m = 0; m < (1 << K); ++m) {
            const int k1 = ib | (bitrev(m, K) << (A - K));
            const int i = kMix ? R * k1 + k2 : k1;  // frequency index of position base + m
            const int m1 = 2 * i < n1 ? i : i - n1;
            int4 t = __ldg(mc + abs(m1));  // k2/|k|, k1/|k|, both >= 0: the product with -(k2 + i k1)/|k|
            if (m2 > 0) {
                t.x = -t.x;
                t.y = -t.y;
            }
            v[m] = zmul(v[m], t, m1 > 0 ? -1 : 1);
        }
    }
};

// pass B: rows j (length n1) of the transpose; forward; multiply; inverse; write out[i][j].
template <int A, bool kMix>
__global__ void __launch_bounds__(threads_for(A, kMix), minb_for(A, kMix))
    pass_b(int n2, Side s1, int lr, const ulonglong2 *__restrict__ in, const int4 *__restrict__ mult,
           ulonglong2 *__restrict__ out, Exps ea, Exps eb)
{
    extern __shared__ ulonglong2 sx[];
    __shared__ unsigned words[kSlots];
    clear_words(words, kSlots);
    const int n1 = s1.L, rows = 1 << lr, j0 = blockIdx.x * rows;
    if (!ZM_IDX_OK(j0 + rows - 1, n2)) return;  // checked build: the CTA's columns exist
    const int emax = *ea.max;
    if (emax >= kNotFinite || emax == kAllZero) {
        if (threadIdx.x == 0) {
            eb.e[blockIdx.x] = emax;
            atomicMax(eb.max, emax);
        }
        return;
    }
    stage_rows(sx, rows, n1, in + (size_t)j0 * n1, ea, emax, &words[0]);
    __syncthreads();
    Unit u{emax, &words[0], make_shift(0)};
    constexpr int C = nc_of(A) - 1;
    if (kMix) {
        radix_stage<true, true>(sx, rows, s1.R, A, s1.twl, -1, u, &words[kNorm]);
        dif_seq<A, 0, C - 1, false>(sx, s1.tw, rows * s1.R, -1, u);
    } else {
        dif_seq<A, 0, C - 1, true>(sx, s1.tw, rows, -1, u);
    }
    constexpr int K = k_of(A, C);
    const int sub_rows = kMix ? rows * s1.R : rows;
    next_room<C == 0 && !kMix>(u, K);
    chunk_pass<K, true, A, 0, C == 0 && !kMix>(sx, sub_rows, s1.tw, -1, u,
                                               Multiply<A, K, kMix>{j0, n1, n2, s1.R, mult});
    __syncthreads();
    dit_seq<A, C>(sx, s1.tw, sub_rows, +1, u);
    if (kMix) radix_stage<false, false>(sx, rows, s1.R, A, s1.twl, +1, u, &words[kNorm + 1]);
#pragma unroll 4
    for (int e = threadIdx.x; e < rows * n1; e += blockDim.x) {
        const int i = e >> lr, r = e & (rows - 1);
        if (ZM_IDX_OK((size_t)i * n2 + j0 + r, (size_t)n1 * n2)) out[(size_t)i * n2 + j0 + r] = sx[phys(r * n1 + i)];
    }
    if (threadIdx.x == 0) {
        eb.e[blockIdx.x] = u.e;
        atomicMax(eb.max, u.e);
    }
}

// pass C: rows i (length n2); inverse; s = Re / (n1 n2); u = -s/2 N; Phi = q + |u|^2 / 2.
template <int A, bool kMix>
__global__ void __launch_bounds__(threads_for(A, kMix), minb_for(A, kMix))
    pass_c(int n1, Side s2, int lr, double inv, const ulonglong2 *__restrict__ in, const double *__restrict__ nrm,
           const double *__restrict__ q, double *__restrict__ u, double *__restrict__ phi, Exps eb, int *reset)
{
    extern __shared__ ulonglong2 sx[];
    __shared__ unsigned words[kSlots];
    clear_words(words, kSlots);
    const int L = s2.L, rows = 1 << lr, i0 = blockIdx.x * rows;
    if (!ZM_IDX_OK(i0 + rows - 1, n1)) return;  // checked build: the CTA's rows exist
    const size_t N = (size_t)n1 * L, o0 = (size_t)i0 * L;
    const int emax = *eb.max;
    const bool finite = emax < kNotFinite, data = finite && emax != kAllZero;
    Unit un{emax, &words[0], make_shift(0)};
    if (data) {
        stage_rows(sx, rows, L, in + o0, eb, emax, &words[0]);
        __syncthreads();
        rows_dif<A, kMix>(sx, rows, s2, +1, un, &words[kNorm]);
    }
    // -s/2 per unit as 2^e1 in the conversion and a factor (the exponent may lie outside the range of one)
    const int e1 = data ? min(max(un.e, -800), 800) : 0, e2 = data ? un.e - e1 : 0;
    const double f2 = finite ? -0.5 * inv * __hiloint2double((1023 + e2) << 20, 0) : __longlong_as_double(0x7ff8000000000000ll);
    const int total = rows * L, step = blockDim.x % L, rstep = blockDim.x / L;
    int r = threadIdx.x / L, j = threadIdx.x % L;
    constexpr int kB = kBatch / 2;
    for (int e0 = threadIdx.x; e0 < total; e0 += kB * blockDim.x) {
        double n0[kB], n1v[kB], n2v[kB], qv[kB], s[kB];
#pragma unroll
        for (int b = 0; b < kB; ++b) {
            const int e = e0 + b * blockDim.x;
            const size_t p = o0 + e;
            const int k = r * L + dif_pos<A, kMix>(j, s2.R);
            if (e < total && ZM_IDX_OK(p, N) && ZM_IDX_OK(k, total)) {
                n0[b] = __ldcs(nrm + p);
                n1v[b] = __ldcs(nrm + N + p);
                n2v[b] = __ldcs(nrm + 2 * N + p);
                qv[b] = __ldcs(q + p);
                s[b] = fp64_of(data ? ldz(sx[phys(k)]).re : 0ll, e1) * f2;
            }
            r += rstep;
            j += step;
            if (j >= L) {
                j -= L;
                ++r;
            }
        }
#pragma unroll
        for (int b = 0; b < kB; ++b) {
            const int e = e0 + b * blockDim.x;
            const size_t p = o0 + e;
            if (e < total && ZM_IDX_OK(p, N)) {
                const double ux = s[b] * n0[b], uy = s[b] * n1v[b], uz = s[b] * n2v[b];
                u[p] = ux;
                u[N + p] = uy;
                u[2 * N + p] = uz;
                phi[p] = qv[b] + 0.5 * (ux * ux + uy * uy + uz * uz);
            }
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *reset = kAllZero;  // pass A's maximum: not in use now
}

// ---- tables --------------------------------------------------------------------------------------------
// W_L^k = exp(-2 pi i k / L), k < count, in units of 2^-60
__global__ void twiddle_kernel(int L, int count, int4 *tw)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= count) return;
    double s, c;
    sincospi(-2.0 * (double)k / (double)L, &s, &c);
    int4 w;
    limbs60(c, w.x, w.y);
    limbs60(s, w.z, w.w);
    tw[k] = w;
}

// W_R^k, k < R, in units of 2^-59; after them per k the constants that the sums of dft_fix start from:
// the rounding half of their shift and half of the roots' low limbs.
__global__ void root_kernel(int R, int4 *rt)
{
    const int k = threadIdx.x;
    if (k >= R) return;
    longlong2 mean = make_longlong2(1ll << (kLimb - 2), 1ll << (kLimb - 2));
    for (int n = 0; n <= (R - 1) / 2; ++n) {  // n = 0: the root itself, k / R
        double s, c;
        const int e = n ? (n * k) % R : k;
        sincospi(-2.0 * (double)e / (double)R, &s, &c);
        int4 w;
        limbs60(0.5 * c, w.x, w.y);
        limbs60(0.5 * s, w.z, w.w);
        if (n) {
            mean.x += w.y / 2;
            mean.y += w.w / 2;
        } else {
            rt[k] = w;
        }
    }
    reinterpret_cast<longlong2 *>(rt)[R + k] = mean;
}

// k2/|k| and k1/|k| at |m1| <= n1/2, |m2| <= n2/2 (t_l = m_l / L_l: the 2 pi cancels), zero at k = 0 and
// on the Nyquist row and column.
__global__ void multiplier_kernel(int n1, int n2, double invL1, double invL2, int4 *mult)
{
    const int h1 = n1 / 2 + 1;
    const size_t count = (size_t)h1 * (n2 / 2 + 1);
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
        const int m2 = (int)(e / h1), m1 = (int)(e - (size_t)m2 * h1);
        int4 w = make_int4(0, 0, 0, 0);
        if ((m1 || m2) && 2 * m1 != n1 && 2 * m2 != n2) {
            const double t1 = m1 * invL1, t2 = m2 * invL2;
            const double big = fmax(t1, t2), a = t1 / big, b = t2 / big, h = sqrt(a * a + b * b);
            limbs60(b / h, w.x, w.y);
            limbs60(a / h, w.z, w.w);
        }
        mult[e] = w;
    }
}

int ilog2(int n)
{
    int l = 0;
    while ((1 << l) < n) ++l;
    return l;
}

Side make_side(int L, const void *tw, const void *twl)
{
    Side s;
    s.L = L;
    s.A = ilog2(L & -L);
    s.R = L >> s.A;
    s.tw = static_cast<const int4 *>(tw);
    s.twl = static_cast<const int4 *>(twl);
    return s;
}

// log2 of the rows per CTA: a power of two dividing the number of rows the pass has (`avail`), within
// kElems values, halved (down to one) while the pass would have fewer than two CTAs per SM.
int log_rows(int L, int avail)
{
    const int cap = std::max(1, std::min(kElems / L, avail & -avail));
    int r = 0;
    while ((2 << r) <= cap) ++r;
    while (r > 0 && (avail >> r) < 304) --r;
    return r;
}

size_t smem_for(int L, int lr)
{
    const size_t e = (size_t)L << lr;
    return (e + e / 16) * sizeof(ulonglong2);
}

template <class F>
int with_log2(int l, F &&f)
{
    switch (l) {
#define ZM_CASE(n) \
    case n: return f(std::integral_constant<int, n>{});
        ZM_CASE(3) ZM_CASE(4) ZM_CASE(5) ZM_CASE(6) ZM_CASE(7) ZM_CASE(8) ZM_CASE(9) ZM_CASE(10) ZM_CASE(11)
        ZM_CASE(12) ZM_CASE(13)
#undef ZM_CASE
    default: return set_error(ZM_ERR_UNSUPPORTED, "Riesz pass: side must be R 2^a, 3 <= a <= 13");
    }
}

// Threads per CTA: one per group of 16 values, at least a warp.
int threads_launch(int A, bool mix, int L, int lr)
{
    if (mix) return 256;
    return std::max(32, std::min(threads_for(A, false), (L << lr) / 16));
}

template <class Kernel, class... Args>
int launch_pass(Kernel kernel, int grid, int threads, size_t smem, cudaStream_t s, Args... args)
{
    int rc = cuda_check(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                        "Riesz pass shared-memory attribute");
    if (rc) return rc;
    kernel<<<grid, threads, smem, s>>>(args...);
    return cuda_check(cudaGetLastError(), "Riesz FFT launch");
}

// Calls f(std::integral_constant<int, A>, std::bool_constant<mixed>) for a side.
template <class F>
int with_side(const Side &s, F &&f)
{
    return with_log2(s.A, [&](auto a) {
        return s.R > 1 ? f(a, std::true_type{}) : f(a, std::false_type{});
    });
}

}  // namespace

bool fft_side_ok(int L)
{
    if (L < 8 || L > kMaxSide) return false;
    const int M = L & -L, R = L / M;
    if (M < 8) return false;
    switch (R) {
    case 1:
#define ZM_CASE(r) case r:
        ZM_FOR_RADICES(ZM_CASE)
#undef ZM_CASE
        return true;
    default: return false;
    }
}

int fft_setup(zm_ctx *c)
{
    const Geom &g = c->geom;
    const size_t N = g.N;
    const Side s1 = make_side(g.n1, nullptr, nullptr), s2 = make_side(g.n2, nullptr, nullptr);
    const size_t nm = (size_t)(g.n1 / 2 + 1) * (g.n2 / 2 + 1);
    const int q1 = 3 << (s1.A - 2), q2 = 3 << (s2.A - 2);
    if (cudaMalloc(&c->fa, N * sizeof(ulonglong2)) != cudaSuccess ||
        cudaMalloc(&c->fb, N * sizeof(ulonglong2)) != cudaSuccess ||
        cudaMalloc(&c->tw1, q1 * sizeof(int4)) != cudaSuccess || cudaMalloc(&c->tw2, q2 * sizeof(int4)) != cudaSuccess ||
        (s1.R > 1 && cudaMalloc(&c->twl1, (g.n1 + 2 * s1.R) * sizeof(int4)) != cudaSuccess) ||
        (s2.R > 1 && cudaMalloc(&c->twl2, (g.n2 + 2 * s2.R) * sizeof(int4)) != cudaSuccess) ||
        cudaMalloc(&c->fmult, nm * sizeof(int4)) != cudaSuccess ||
        cudaMalloc(&c->fexp, (g.n1 + g.n2 + 2) * sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        return set_error(ZM_ERR_NOMEM, "fft_setup: device allocation failed");
    }
    auto tw = [](double2 *p) { return reinterpret_cast<int4 *>(p); };
    twiddle_kernel<<<(q1 + 255) / 256, 256>>>(1 << s1.A, q1, tw(c->tw1));
    twiddle_kernel<<<(q2 + 255) / 256, 256>>>(1 << s2.A, q2, tw(c->tw2));
    if (c->twl1) {
        twiddle_kernel<<<(g.n1 + 255) / 256, 256>>>(g.n1, g.n1, tw(c->twl1));
        root_kernel<<<1, 32>>>(s1.R, tw(c->twl1) + g.n1);
    }
    if (c->twl2) {
        twiddle_kernel<<<(g.n2 + 255) / 256, 256>>>(g.n2, g.n2, tw(c->twl2));
        root_kernel<<<1, 32>>>(s2.R, tw(c->twl2) + g.n2);
    }
    multiplier_kernel<<<608, 256>>>(g.n1, g.n2, 1.0 / g.L1, 1.0 / g.L2, static_cast<int4 *>(c->fmult));
    int rc = cuda_check(cudaGetLastError(), "twiddle kernel");
    const int none[2] = {kAllZero, kAllZero};  // the two passes' largest exponents
    if (!rc) rc = cuda_check(cudaMemcpy(c->fexp, none, sizeof(none), cudaMemcpyHostToDevice), "fft_setup");
    return rc;
}

int launch_riesz(zm_ctx *c, const double *y)
{
    if (!y || !c->fa || !c->fb || !c->tw1 || !c->tw2 || !c->fmult || !c->fexp || !c->nrm || !c->q || !c->u || !c->phi)
        return set_error(ZM_ERR_INVALID, "Riesz pass: missing buffer");
    const Geom &g = c->geom;
    const Side s1 = make_side(g.n1, c->tw1, c->twl1), s2 = make_side(g.n2, c->tw2, c->twl2);
    if ((s1.R > 1 && !c->twl1) || (s2.R > 1 && !c->twl2))
        return set_error(ZM_ERR_INVALID, "Riesz pass: missing twiddle table");
    const int ra = log_rows(g.n2, g.n1), rb = log_rows(g.n1, g.n2);
    if (g.n1 % (1 << ra) || g.n2 % (1 << rb))
        return set_error(ZM_ERR_INVALID, "Riesz pass: rows per CTA do not divide the side");
    const Exps ea{c->fexp + 2, c->fexp, ra}, eb{c->fexp + 2 + g.n1, c->fexp + 1, rb};
    ulonglong2 *fa = reinterpret_cast<ulonglong2 *>(c->fa), *fb = reinterpret_cast<ulonglong2 *>(c->fb);
    const int4 *mult = static_cast<const int4 *>(c->fmult);
    cudaEvent_t ev = nullptr;
    prof_begin(c, ZM_K_FFT, &ev);
    int rc = with_side(s2, [&](auto a, auto m) {
        constexpr int A = decltype(a)::value;
        constexpr bool M = decltype(m)::value;
        return launch_pass(pass_a<A, M>, g.n1 >> ra, threads_launch(A, M, g.n2, ra), smem_for(g.n2, ra), c->stream,
                           g.n1, s2, ra, y + 3 * (size_t)g.N, fa, ea, eb.max);
    });
    if (!rc) rc = with_side(s1, [&](auto a, auto m) {
        constexpr int A = decltype(a)::value;
        constexpr bool M = decltype(m)::value;
        return launch_pass(pass_b<A, M>, g.n2 >> rb, threads_launch(A, M, g.n1, rb), smem_for(g.n1, rb), c->stream,
                           g.n2, s1, rb, (const ulonglong2 *)fa, mult, fb, ea, eb);
    });
    if (!rc) rc = with_side(s2, [&](auto a, auto m) {
        constexpr int A = decltype(a)::value;
        constexpr bool M = decltype(m)::value;
        return launch_pass(pass_c<A, M>, g.n1 >> ra, threads_launch(A, M, g.n2, ra), smem_for(g.n2, ra), c->stream,
                           g.n1, s2, ra, 1.0 / ((double)g.n1 * (double)g.n2), (const ulonglong2 *)fb,
                           (const double *)c->nrm, (const double *)c->q, c->u, c->phi, eb, ea.max);
    });
    prof_end(c, ZM_K_FFT, ev);
    if (!rc) c->prof.acc.launches[ZM_K_FFT] += 2;  // three kernels per Riesz evaluation
    return rc;
}

ZM_BOUNDS_READER(bounds_fft)

}  // namespace zm
