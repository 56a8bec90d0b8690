// zm_brdw.cu -- the FP64 all-pairs Birkhoff-Rott sum (paper Sec. 2 BRSolver, Sec. 3.2.1
// ExactBRSolver) on meshes of at least kDwMinN nodes, with the FP64 pipe kept for the pairs whose
// rounding decides the result:
//     u_i = sum_j (z_j - z_i) x gamma'_j / (|z_j - z_i|^2 + delta^2)^(3/2).
//
// What bounds it.  GB300 executes 2 FP64 instructions per clock and SM, so the 21 FP64 instructions of
// a pair (zm_br.cu) cost 10.5 clocks of an SM whose other pipes idle (measured: the pipe 90 % busy, 190 ms
// per 256 x 256 evaluation).  A pair far apart compared with its source tile is evaluated here in 64-bit
// integers instead, to the same precision: 29 integer multiply-adds 32 x 32 + 64 bits (60 per clock and
// SM), some 50 other integer operations, 9 in FP32, one reciprocal square root, 108 instructions with the
// rest: 1.6 clocks, the multiply and ALU pipes 61 and 53 % busy, the FP64 pipe 19 %, the schedulers issuing
// in 54 % of cycles.
// 190.3 -> 21.4 ms at 256 x 256, 13.0 -> 1.63 at 128 x 128, 7.5 -> 0.93 at 90 x 131, 0.81 -> 0.23 at
// 64 x 64 (one evaluation).  (q and K as FP32 pairs take 12.5 ms at 256 x 256 but hold a far pair to 2^-46
// only: u is then 2e-14 off, relative, where all strength lies further away than the near tiles.)
//
// Tiles.  8 x 8 mesh patches (64 nodes) serve as target tiles (one CTA of 64 threads, one target
// per thread) and as source tiles, staged by 1D bulk TMA.  Small tiles keep the near region, whose
// pairs cost 7 times as much, small; where a source tile is not far from the target tile, its
// four quarters (4 x 4 nodes) are classified against each warp's 32 targets.  By bounding spheres:
//   far   (centres at least kappa source radii plus the targets' radius apart): the form below;
//   near  FP64 throughout, as in zm_br.cu, on the untouched positions and strengths.
// A tile's near neighbours spread over the source splits (the splits take the tiles in turn).
//
// Far pairs.  Everything is relative to the source tile's centre c: s_j = z_j - c, t_i = z_i - c, FP64
// differences, so that the origin of the coordinates does not matter.  Per target and tile, in units 2^m in
// which the least q of the tile has 58 bits:
//   q = (|t|^2 + delta^2) + |s|^2 - 2 s . t   in 64 bits, the products of the leading 31-bit limbs exact, those
//       of the remainders, 2^-30 of them, in FP32;
//   K = q^(-3/2) from the special-function estimate Y of q^(-1/2), taken as an integer: e = 1 - q Y^2 to
//       2^-52 from the products of the 32-bit limbs, K = Y^3 (1 + 3/2 e + 15/8 e^2) to 2^-57 (the square in FP32);
//   sums G = sum K g, M = sum K (s x g), and u_tile = M - t x G.  K has a leading limb below 2^30 and a
//       trailing one of 28 bits (in a far tile K varies by less than 26), g 26 and 28 bits; the products of the
//       leading limbs and the mixed ones accumulate exactly in 64-bit integers.
// Shifts that round down have the mean of what they drop made up for by a constant, since the error of
// a tile's pairs would not average out.  Tiles whose radius or strength does not fit (or is not finite) have an
// infinite radius, that is, are near to all.
//
// Accuracy.  One source node's contribution, relative, rms over random positions: 2.3e-16 (4.5e-16 at the
// edge of the far region; the FP64 pair 1.5e-16); 64 random strengths in a tile 3.7e-16 (5.1e-16), 64 alike
// 1.2e-16 (2.2e-16).  u against long double sums (multi-mode interface, relative L2 over sampled
// targets; zm_br.cu's plain FP64 sum / here): 56 x 56 7.5e-16 / 2.0e-16, 80 x 80 4.7e-16 / 2.6e-16, 96 x 96
// 8.2e-16 / 2.8e-16, 90 x 131 1.2e-15 / 2.4e-16, 128 x 128 1.5e-15 / 2.6e-16, 200 x 150 1.8e-15 / 2.7e-16,
// 256 x 256 5.7e-15 / 5.1e-16: the plain sums are longer.
#include <algorithm>
#include <cmath>

#include "zm_fix.cuh"
#include "zm_stencil.cuh"

namespace zm {
namespace {

constexpr int kT = 8;         // tile side
constexpr int kTs = kT * kT;  // nodes per tile, threads per CTA
constexpr int kSub = 4;       // a tile's quarters: 4 x 4 nodes
constexpr int kNearRows = 6;  // FP64: position, scaled strength
// Far record of a node, 24 words side by side: s as integers (3), as FP32 (3) and the integers' remainders
// (3), |s|^2 (2), leading (6) and trailing (6) limbs of g and s x g, one word of padding.
constexpr int kNodeWords = 24;
constexpr int kFarWords = kNodeWords * kTs;  // the far record of a tile, or of its four quarters
// the near block of a tile: its quarters' far records (quarter k from node 16 k on) and the FP64 record
constexpr int kNearWords = kFarWords + 2 * kNearRows * kTs;
constexpr int kGBits = 26, kGLow = 28;  // g and s x g: n 2^-26 + l 2^-54, |l| <= 2^27

constexpr float kInf = __builtin_huge_valf();
constexpr float kMaxLength = 1048576.0f;  // 2^20: distances and radii of far tiles, scaled

// Classification: 2 source radii, and a sixteenth so that the bounds of far_tile's integers hold with
// the rounding of the radii (3 radii: 27.7 against 27.0 ms at 256 x 256 with an earlier form, 2.10 against 1.96
// at 128 x 128).
constexpr float kKappa = 2.0625f;

// One tile as the pair kernel sees it.
struct __align__(16) DwTile {
    double c[3];   // centre, scaled
    double gs[2];  // 2^(strength exponent) x 2^(-2 length exponent); the same times sqrt 2
    float rho;     // radius, scaled (infinite: near to all)
    int es;        // |s| <= rho < 2^es
};

// A tile and its quarters.
struct DwInfo {
    DwTile tile, quarter[4];
};

struct DwMesh {
    int n1, n2, nt1, nt2;
};

// Nodes of tile `tile`: its corner, its extents (edge tiles are smaller) and their number.
struct Patch {
    int i0, j0, h1, h2, count;
};
__device__ __forceinline__ Patch patch_of(int tile, const DwMesh &m)
{
    Patch p;
    p.i0 = (tile / m.nt2) * kT;
    p.j0 = (tile - (tile / m.nt2) * m.nt2) * kT;
    p.h1 = min(kT, m.n1 - p.i0);
    p.h2 = min(kT, m.n2 - p.j0);
    p.count = p.h1 * p.h2;
    return p;
}
// Mesh node of slot `s` < count (row-major in the patch, no holes in edge tiles).
__device__ __forceinline__ int node_of(const Patch &p, int s, int n2)
{
    const int a = s / p.h2;
    return (p.i0 + a) * n2 + p.j0 + (s - a * p.h2);
}
// Quarter `k` of a patch (possibly empty in edge tiles).
__device__ __forceinline__ Patch quarter_of(const Patch &p, int k)
{
    Patch q;
    const int a = (k >> 1) * kSub, b = (k & 1) * kSub;
    q.i0 = p.i0 + a;
    q.j0 = p.j0 + b;
    q.h1 = max(0, min(kSub, p.h1 - a));
    q.h2 = max(0, min(kSub, p.h2 - b));
    q.count = q.h1 * q.h2;
    return q;
}

__device__ __forceinline__ unsigned hi_abs(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// Exponent e with rho < 2^e <= 2 rho.
__device__ __forceinline__ int exp_above(float rho) { return (int)(__float_as_uint(rho) >> 23) - 126; }
__device__ __forceinline__ double pow2d(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// ---- the far form --------------------------------------------------------------------------------------

// c + a b; unsigned factors
__device__ __forceinline__ unsigned long long mad_wu(unsigned a, unsigned b, unsigned long long c)
{
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
    return c;
}
__device__ __forceinline__ unsigned hi32(unsigned long long v) { return (unsigned)(v >> 32); }

// round(v 2^b), |v 2^b| < 2^61, from the bits of v (no FP64 instructions); ties away from zero.
__device__ __forceinline__ long long fixed(double v, int b)
{
    const int hi = __double2hiint(v);
    const unsigned long long m = ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(v))
                                 << 8;
    const int n = min(1083 - ((hi >> 20) & 0x7ff) - b, 63);  // v = m 2^(e - 1083)
    const long long r = (long long)((m + ((1ull << n) >> 1)) >> n);
    return hi < 0 ? -r : r;
}
// |v| as FP32, truncated (0 below 2^-126); |v| < 2^127.
__device__ __forceinline__ float abs_f32(double v)
{
    const unsigned h = (unsigned)__double2hiint(v) & 0x7fffffffu;
    return h < (897u << 20) ? 0.0f
                            : __uint_as_float(((h << 3) | ((unsigned)__double2loint(v) >> 29)) - (896u << 23));
}

// Writes one node's far record: s = position relative to the centre (|s| < 2^es), gg = strength
// below 1; s x g in units of 2^es.
__device__ __forceinline__ void put_far(float *__restrict__ fr, const double s[3], const double gg[3], int es)
{
    const double iu = pow2d(-es);
    const double t[3] = {s[0] * iu, s[1] * iu, s[2] * iu};
    const double g6[6] = {gg[0], gg[1], gg[2], t[1] * gg[2] - t[2] * gg[1], t[2] * gg[0] - t[0] * gg[2],
                          t[0] * gg[1] - t[1] * gg[0]};
    int *w = reinterpret_cast<int *>(fr);
    double a2 = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        a2 = fma(t[k], t[k], a2);
        const double v = t[k] * 1073741824.0, n = rint(v);  // 2^30
        w[k] = __double2int_rn(n);
        fr[3 + k] = __double2float_rn(v);
        fr[6 + k] = __double2float_rn(v - n);
    }
    const long long A = __double2ll_rn(a2 * 4611686018427387904.0);  // 2^62
    w[9] = (int)(unsigned)A;
    w[10] = (int)(A >> 32);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const double v = g6[k] * (double)(1 << kGBits), n = rint(v);
        w[11 + k] = __double2int_rn(n);
        w[17 + k] = __double2int_rn((v - n) * (double)(1 << kGLow));
    }
}

// The far pairs of one target and one source tile (records of `count` nodes in shared memory): adds
// sum_j K (s - t) x g to u.  td: the target, scaled; d2: delta^2, scaled.
__device__ __forceinline__ void far_tile(const float *__restrict__ rec, int count, const double td[3],
                                         const DwTile &T, double d2, float d2f, double u[3])
{
    const double e[3] = {td[0] - T.c[0], td[1] - T.c[1], td[2] - T.c[2]};
    // the unit 2^m of q: its least value in the tile, (|t| - rho)^2 + delta^2, lies in [2^57, 2^58)
    const float fx = abs_f32(e[0]), fy = abs_f32(e[1]), fz = abs_f32(e[2]);
    const float t2 = fmaf(fx, fx, fmaf(fy, fy, fz * fz));
    const float tm = fmaf(t2, dev::rsqrt_approx(t2), -T.rho);
    const int m = (int)(__float_as_uint(fmaf(tm, tm, d2f) * 0.9999f) >> 23) - (127 + 57);
    // t in units 2^-b with 2 b + m = 62 - odd, and its square in units of q, from limbs of 31 bits
    const int b = (62 - m) >> 1, odd = m & 1;
    long long t[3], hi = 0, mid = 0, lo = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        t[k] = fixed(e[k], b);
        const int h = (int)((t[k] + (1 << 30)) >> 31), l = (int)(t[k] - ((long long)h << 31));
        hi = mad_w(h, h, hi);
        mid = mad_w(h, l, mid);
        lo = mad_w(l, l, lo);
    }
    const long long B = (hi << odd) + ((mid + (lo >> 32) + (1 << (29 - odd))) >> (30 - odd)) + fixed(d2, -m);
    // -2 t in units 2^(m - es + 30), whose products with s (units 2^(es - 30)) are in units of q
    const int rt = min(b + m - T.es - 1, 63), ra = min(m - 2 * T.es + 62, 63);
    const long long half = (long long)((1ull << rt) >> 1);
    int th[3];
    float tf[3], tl[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const long long v = -((t[k] + half) >> rt);
        th[k] = (int)((v + (1 << 29)) >> 30);
        tf[k] = (float)th[k];
        tl[k] = (float)(int)(v - ((long long)th[k] << 30)) * 9.313225746154785e-10f;  // 2^-30
    }

    long long I[6] = {0, 0, 0, 0, 0, 0}, J[6] = {0, 0, 0, 0, 0, 0};
    const int4 *r = reinterpret_cast<const int4 *>(rec);
#pragma unroll 2
    for (int j = 0; j < count; ++j, r += kNodeWords / 4) {
        const int4 w0 = r[0], w1 = r[1], w2 = r[2], w3 = r[3], w4 = r[4], w5 = r[5];
        // q = |t|^2 + delta^2 - 2 t . s + |s|^2: the remainders' products, 2^-30 of the terms, in FP32
        const long long h = mad_w(w0.z, th[2], mad_w(w0.y, th[1], mad_w(w0.x, th[0], B)));
        const float s0 = __int_as_float(w0.w), s1 = __int_as_float(w1.x), s2 = __int_as_float(w1.y);
        const float l0 = __int_as_float(w1.z), l1 = __int_as_float(w1.w), l2 = __int_as_float(w2.x);
        float c = fmaf(s2, tl[2], fmaf(s1, tl[1], s0 * tl[0]));
        c = fmaf(l2, tf[2], fmaf(l1, tf[1], fmaf(l0, tf[0], c)));
        const long long a = (long long)((unsigned long long)(unsigned)w2.z << 32 | (unsigned)w2.y);
        const unsigned long long q = (unsigned long long)(h + __float2int_rn(c) + (a >> ra));
        // Y = 2^60 q^(-1/2) (1 - e/2 ..) and W = Y^2; e = 1 - q W 2^-120, in units 2^-56, then 2^-52 (8: to
        // round; -1: the mean of what the limbs' products drop)
        const unsigned qh = hi32(q), ql = (unsigned)q;
        const unsigned Y = __float2uint_rn(dev::rsqrt_approx(__uint2float_rn(qh)) * 17592186044416.0f);  // 2^44
        const unsigned long long W = mad_wu(Y, Y, 0);
        const unsigned wh = hi32(W), wl = (unsigned)W;
        const unsigned long long x = mad_wu(ql, wh, mad_wu(qh, wl, 0));
        const int e1 = (int)(((long long)((1ull << 56) + 8 - 1 - mad_wu(qh, wh, 0)) - hi32(x)) >> 4);
        // e + 1.25 e^2, the square in FP32, as integer by the constant 1.5 2^23
        const float ef = __int2float_rn(e1);
        const int ec = e1 + (int)(__float_as_uint(fmaf(ef * 2.7755575615628914e-16f, ef, 12582912.0f)) - 0x4b400000u);
        // K = Y^3 2^-33 (1 + 3/2 (e + 1.25 e^2)) = 2^147 q^(-3/2) (Y is even, having 24 leading bits; 9: the means of
        // what the shifts drop)
        const unsigned long long K0 = mad_wu(Y >> 1, wh, 9) + hi32(mad_wu(Y >> 1, wl, 0));
        const long long X = mad_w((int)hi32(K0), ec, mul_w((int)((unsigned)K0 >> 1), ec) >> 31);
        const unsigned long long K = K0 + (unsigned long long)((X + (X << 1)) >> 21);
        const int kh = (int)hi32(K), kl = (int)((unsigned)K >> 4);
        const int gh[6] = {w2.w, w3.x, w3.y, w3.z, w3.w, w4.x}, gl[6] = {w4.y, w4.z, w4.w, w5.x, w5.y, w5.z};
#pragma unroll
        for (int y = 0; y < 6; ++y) {
            I[y] = mad_w(kh, gh[y], I[y]);
            J[y] = mad_w(kl, gh[y], mad_w(kh, gl[y], J[y]));
        }
    }
    double v[6];
#pragma unroll
    for (int x = 0; x < 6; ++x) v[x] = fp64_of(I[x] + ((J[x] + (1 << (kGLow - 1))) >> kGLow), 0);
    // K 2^(-3/2 m), the limbs and the strength's scale
    const double gs = odd ? T.gs[1] : T.gs[0];
    const double sd = __hiloint2double(__double2hiint(gs) + ((((-3 * m) >> 1) + 32 - 147 - kGBits) << 20),
                                       __double2loint(gs));
    const double rs = pow2d(T.es);
    u[0] = fma(fma(rs, v[3], fma(e[2], v[1], -e[1] * v[2])), sd, u[0]);
    u[1] = fma(fma(rs, v[4], fma(e[0], v[2], -e[2] * v[0])), sd, u[1]);
    u[2] = fma(fma(rs, v[5], fma(e[1], v[0], -e[0] * v[1])), sd, u[2]);
}

// ---- geometry ------------------------------------------------------------------------------------------

__device__ __forceinline__ DwTile make_tile(const double c[3], float rho, double gs)
{
    DwTile t;
#pragma unroll
    for (int k = 0; k < 3; ++k) t.c[k] = c[k];
    t.gs[0] = gs;
    t.gs[1] = gs * 1.4142135623730950488;
    t.rho = rho;
    t.es = exp_above(rho);
    return t;
}

// Geometry pass of one tile per CTA: q, the far record and the near block.  One thread per node;
// the radii and the largest strength come from a CTA reduction, so the far records can be written
// already scaled.  Bound by the FP64 instructions of the stencils; 64-thread CTAs spread small
// meshes over the SMs (with 256-thread CTAs 64 x 64 runs on 16 of them).
__global__ void __launch_bounds__(kTs)
    geometry_dw_kernel(Geom g, DwMesh m, const double *__restrict__ y, double pref, double grav, double pscale,
                       double gscale, float *__restrict__ near_rec, float *__restrict__ far_rec,
                       DwInfo *__restrict__ info, double *__restrict__ q)
{
    __shared__ unsigned rmax[5], gmax;  // the tile's radius, the quarters'; the largest strength
    const int tile = blockIdx.x, tid = threadIdx.x;
    if (!ZM_IDX_OK(tile, m.nt1 * m.nt2)) return;
    if (tid < 5) rmax[tid] = 0u;
    if (tid == 5) gmax = 0u;
    const Patch pt = patch_of(tile, m);
    const bool valid = tid < pt.count;
    const int p = node_of(pt, valid ? tid : 0, m.n2);
    if (!ZM_IDX_OK(p, g.N)) return;
    const int li = p / m.n2 - pt.i0, lj = p - (p / m.n2) * m.n2 - pt.j0;  // within the tile
    const int qk = (li / kSub) * 2 + lj / kSub;
    const Patch pq = quarter_of(pt, qk);
    const size_t N = g.N;
    const double zc[3] = {y[p], y[N + p], y[2 * N + p]};
    double gm[3];
    const double qn = geometry_strength(g, p, y, pref, grav, gm);
    if (valid) q[p] = qn;

    // the centres are nodes
    const int pc = (pt.i0 + pt.h1 / 2) * m.n2 + pt.j0 + pt.h2 / 2;
    const int pcq = (pq.i0 + pq.h1 / 2) * m.n2 + pq.j0 + pq.h2 / 2;
    if (!ZM_IDX_OK(pc, g.N) || !ZM_IDX_OK(pcq, g.N)) return;
    double c[3], cq[3], s[3], sq[3];
    double r2 = 0.0, r2q = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        c[k] = y[k * N + pc] * pscale;
        cq[k] = y[k * N + pcq] * pscale;
        const double a = zc[k] * pscale;
        s[k] = a - c[k];
        sq[k] = a - cq[k];
        r2 = fma(s[k], s[k], r2);
        r2q = fma(sq[k], sq[k], r2q);
    }
    __syncthreads();
    if (valid) {
        // not less than kMaxLength (also for NaN): infinite
        const float rn = sqrtf(__double2float_ru(r2)) * 1.000001f, rq = sqrtf(__double2float_ru(r2q)) * 1.000001f;
        atomicMax(&rmax[0], __float_as_uint(rn < kMaxLength ? rn : kInf));
        atomicMax(&rmax[1 + qk], __float_as_uint(rq < kMaxLength ? rq : kInf));
        atomicMax(&gmax, max(hi_abs(gm[0]), max(hi_abs(gm[1]), hi_abs(gm[2]))));
    }
    __syncthreads();
    const int eg = gmax ? (int)(gmax >> 20) - 1022 : 0;  // |strength components| < 2^eg
    const bool fit = eg >= -400 && eg <= 400 && __uint_as_float(rmax[0]) < kInf;
    const double gs = pow2d(fit ? eg : 0) * gscale;

    float *fr = far_rec + (size_t)tile * kFarWords;
    float *nf = near_rec + (size_t)tile * kNearWords;
    double *nd = reinterpret_cast<double *>(nf + kFarWords);
    if (valid) {
        const int slot = qk * 16 + (li - (qk >> 1) * kSub) * pq.h2 + (lj - (qk & 1) * kSub);
        if (!ZM_IDX_OK(slot, kTs)) return;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            nd[k * kTs + slot] = zc[k];
            nd[(3 + k) * kTs + slot] = gm[k];
        }
        if (fit) {
            const double gi = pow2d(-eg);
            const double gg[3] = {gm[0] * gi, gm[1] * gi, gm[2] * gi};
            put_far(fr + tid * kNodeWords, s, gg, exp_above(__uint_as_float(rmax[0])));
            put_far(nf + slot * kNodeWords, sq, gg, exp_above(__uint_as_float(rmax[1 + qk])));
        }
    }
    if (tid == 0) info[tile].tile = make_tile(c, fit ? __uint_as_float(rmax[0]) : kInf, gs);
    if (valid && p == pcq) info[tile].quarter[qk] = make_tile(cq, fit ? __uint_as_float(rmax[1 + qk]) : kInf, gs);
}

struct DwArgs {
    DwMesh m;
    int N, ntiles, nsplit;
    double d2;       // delta^2
    double d2s;      // delta^2 scaled
    float kappa;     // far: centres at least kappa source radii + a target radius apart
    double pscale;
    const double *z;
    const float *near_rec, *far_rec;
    const DwInfo *info;
    double *part;
    int *err;
};

// Distance between a tile's centre and a point, less the point's own radius.
__device__ __forceinline__ float gap(const DwTile &s, const double *p, float rho)
{
    const float dx = (float)(s.c[0] - p[0]), dy = (float)(s.c[1] - p[1]), dz = (float)(s.c[2] - p[2]);
    return sqrtf(dx * dx + dy * dy + dz * dz) * 0.9999f - rho;
}
// 2^-20 and 2^20 keep K and the scale factors in range; an infinite radius is never far.
__device__ __forceinline__ bool is_far(float gap, float kappa, float rho)
{
    return gap >= kappa * rho && gap >= 1.0f / kMaxLength && gap <= kMaxLength;
}

__global__ void __launch_bounds__(kTs, 7) brdw_kernel(const DwArgs a)
{
    constexpr uint32_t kFarBytes = kFarWords * sizeof(float), kNearBytes = kNearWords * sizeof(float);
    __shared__ __align__(128) float stage[2][kNearWords];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ uint32_t farmask[2];
    const int tid = threadIdx.x, tt = blockIdx.x;
    if (!ZM_IDX_OK(tt, a.ntiles)) return;
    const Patch pt = patch_of(tt, a.m);
    const bool valid = tid < pt.count;
    const int p = node_of(pt, valid ? tid : 0, a.m.n2);
    const size_t N = a.N;
    if (!ZM_IDX_OK(p, N)) return;
    const double tx = a.z[p], ty = a.z[N + p], tz = a.z[2 * N + p];
    const double td[3] = {tx * a.pscale, ty * a.pscale, tz * a.pscale};
    // the target tile's sphere, and the sphere of this warp's 32 targets around one of them
    const DwTile me = a.info[tt].tile;
    double cw[3];
    float wr = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        cw[k] = __shfl_sync(0xffffffffu, td[k], 20);
        const float d = (float)(td[k] - cw[k]);
        wr = fmaf(d, d, wr);
    }
    wr = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(sqrtf(wr) * 1.0001f)));
    if (!(me.rho < kInf)) wr = kInf;
    double u[3] = {0.0, 0.0, 0.0};

    if (tid == 0) {
        dev::mbar_init(&bar[0], 1);
        dev::mbar_init(&bar[1], 1);
        dev::fence_mbar_init();
    }
    // the source tiles of this split: blockIdx.y, blockIdx.y + nsplit, .. (a tile's near
    // neighbours, whose FP64 pairs cost most, spread over the splits)
    const int total = (a.ntiles - (int)blockIdx.y + a.nsplit - 1) / a.nsplit;
    int unit = 0;
    for (int base = 0; base < total; base += kTs) {
        // classify up to 64 source tiles at once
        const int n = min(kTs, total - base);
        auto tile_of = [&](int k) { return (int)blockIdx.y + (base + k) * a.nsplit; };
        bool far = false;
        if (tid < n && ZM_IDX_OK(tile_of(tid), a.ntiles)) {
            const DwTile &s = a.info[tile_of(tid)].tile;
            far = is_far(gap(s, me.c, me.rho), a.kappa, s.rho);
        }
        const uint32_t mk = __ballot_sync(0xffffffffu, far);
        if ((tid & 31) == 0) farmask[tid >> 5] = mk;
        __syncthreads();
        const uint64_t mask = farmask[0] | ((uint64_t)farmask[1] << 32);
        auto issue = [&](int k, int b) {
            const size_t s = tile_of(k);
            if ((mask >> k) & 1) dev::tma_load_1d(stage[b], a.far_rec + s * kFarWords, kFarBytes, &bar[b]);
            else dev::tma_load_1d(stage[b], a.near_rec + s * kNearWords, kNearBytes, &bar[b]);
        };
        if (tid == 0) {
            // both stages were read by the last 64 tiles: order those reads (ended by the barrier
            // above) before the copies that overwrite them
            dev::fence_proxy_async();
            for (int k = 0; k < 2 && k < n; ++k) issue(k, (unit + k) & 1);
        }
        for (int k = 0; k < n; ++k, ++unit) {
            const int b = unit & 1;
            const bool ok = dev::mbar_wait_bounded(&bar[b], (unit >> 1) & 1);
            if (ok) {
                const Patch ps = patch_of(tile_of(k), a.m);
                const DwInfo &I = a.info[tile_of(k)];
                const bool whole = (mask >> k) & 1;
#pragma unroll 1
                for (int q = 0; q < (whole ? 1 : 4); ++q) {
                    const int count = whole ? ps.count : quarter_of(ps, q).count;
                    if (count == 0) continue;
                    const DwTile s = whole ? I.tile : I.quarter[q];
                    if (whole || is_far(gap(s, cw, wr), a.kappa, s.rho)) {
                        far_tile(stage[b] + 16 * kNodeWords * q, count, td, s, a.d2s, (float)a.d2s, u);
                        continue;
                    }
                    const double *r = reinterpret_cast<const double *>(stage[b] + kFarWords) + 16 * q;
                    double px = 0.0, py = 0.0, pz = 0.0;  // per quarter: short sums round less
#pragma unroll 2
                    for (int j = 0; j < count; ++j) {
                        const double rx = r[j] - tx, ry = r[kTs + j] - ty, rz = r[2 * kTs + j] - tz;
                        const double gx = r[3 * kTs + j], gy = r[4 * kTs + j], gz = r[5 * kTs + j];
                        const double qq = fma(rx, rx, fma(ry, ry, fma(rz, rz, a.d2)));
                        const double kk = dev::rsqrt_cube(qq);
                        px = fma(kk, ry * gz - rz * gy, px);
                        py = fma(kk, rz * gx - rx * gz, py);
                        pz = fma(kk, rx * gy - ry * gx, pz);
                    }
                    u[0] += px;
                    u[1] += py;
                    u[2] += pz;
                }
            }
            const int bad = __syncthreads_or(!ok);
            if (bad) {
                if (tid == 0) {
                    int flags = kErrTimeout;
                    // let the copies still in flight land before shared memory is released
                    for (int w = 0; w < 2 && k + w < n; ++w)
                        if (!dev::mbar_wait_bounded(&bar[(unit + w) & 1], ((unit + w) >> 1) & 1)) flags |= kErrDrain;
                    atomicOr(a.err, flags);
                }
                return;
            }
            if (tid == 0 && k + 2 < n) {
                dev::fence_proxy_async();
                issue(k + 2, b);
            }
        }
    }
    if (valid) {
        double *o = a.part + (size_t)blockIdx.y * 3 * N;
        o[p] = u[0];
        o[N + p] = u[1];
        o[2 * N + p] = u[2];
    }
}

int length_exponent(const Geom &g) { return std::ilogb(std::max(g.L1, g.L2)); }

// Factor of the far classification.  Lengths or a core size outside the range of the integers' scales
// leave every pair near.
float kappa_of(const zm_ctx *c)
{
    const Geom &g = c->geom;
    const int e = length_exponent(g);
    const double d = std::ldexp(c->delta, -e);
    if (e < -100 || e > 100 || !(d < 16.0) || !(std::min(g.L1, g.L2) > 0)) return kInf;
    return kKappa;
}

DwMesh dw_mesh(const Geom &g)
{
    return DwMesh{g.n1, g.n2, (g.n1 + kT - 1) / kT, (g.n2 + kT - 1) / kT};
}

}  // namespace

// Meshes below 56^2 keep the plain FP64 kernel.  One evaluation, plain / here, and the errors of u: 32 x 32
// 0.090 / 0.106 ms, 2.0e-16 / 2.4e-16; 40 x 40 0.190 / 0.132 ms, 3.2e-16 / 2.6e-16; 48 x 48 0.305 / 0.196 ms,
// 3.5e-16 / 2.2e-16; 56 x 56 0.610 / 0.227 ms, 5.1e-16 / 2.0e-16.  (The line lies where a less accurate far form,
// FP32 pairs, began to be the better one; the present form would be from 40^2 on.)
constexpr int kDwMinN = 56 * 56;

bool brdw_mesh(const Geom &g) { return g.N >= kDwMinN; }

BrPlan plan_brdw(const Geom &g, int sm_count)
{
    const DwMesh m = dw_mesh(g);
    BrPlan p;
    p.tpb = kTs;
    p.r = 1;
    p.qsplit = 1;
    p.ntb = m.nt1 * m.nt2;
    // four waves of seven resident CTAs per SM, so that the last wave is short
    const int want = 4 * 7 * sm_count;
    const int ns = std::max(1, std::min((want + p.ntb - 1) / p.ntb, p.ntb));
    p.tiles_per_split = (p.ntb + ns - 1) / ns;
    p.nsplit = (p.ntb + p.tiles_per_split - 1) / p.tiles_per_split;
    return p;
}

size_t brdw_near_bytes(const Geom &g)
{
    const DwMesh m = dw_mesh(g);
    return (size_t)m.nt1 * m.nt2 * kNearWords * sizeof(float);
}

size_t brdw_far_bytes(const Geom &g)
{
    const DwMesh m = dw_mesh(g);
    return (size_t)m.nt1 * m.nt2 * (kFarWords * sizeof(float) + sizeof(DwInfo));
}

int launch_geometry_dw(zm_ctx *c, const double *y, double pref)
{
    if (!c->src || !c->src_far || !c->q) return set_error(ZM_ERR_INVALID, "geometry pass: missing buffer");
    const DwMesh m = dw_mesh(c->geom);
    const int e = std::max(-100, std::min(100, length_exponent(c->geom)));
    DwInfo *info = reinterpret_cast<DwInfo *>(c->src_far);
    float *far_rec = reinterpret_cast<float *>(info + (size_t)m.nt1 * m.nt2);
    geometry_dw_kernel<<<m.nt1 * m.nt2, kTs, 0, c->stream>>>(c->geom, m, y, pref, c->g, std::ldexp(1.0, -e),
                                                            std::ldexp(1.0, -2 * e), static_cast<float *>(c->src),
                                                            far_rec, info, c->q);
    return cuda_check(cudaGetLastError(), "geometry kernel launch");
}

int launch_brdw(zm_ctx *c, const double *y)
{
    if (!y || !c->src || !c->src_far || !c->part) return set_error(ZM_ERR_INVALID, "Birkhoff-Rott pass: missing buffer");
    const Geom &g = c->geom;
    const int e = std::max(-100, std::min(100, length_exponent(g)));
    DwArgs a;
    a.m = dw_mesh(g);
    a.N = g.N;
    a.ntiles = a.m.nt1 * a.m.nt2;
    a.nsplit = c->plan.nsplit;
    a.d2 = c->delta * c->delta;
    const double d2s = std::ldexp(a.d2, -2 * e);
    a.d2s = d2s;
    a.kappa = kappa_of(c);
    a.pscale = std::ldexp(1.0, -e);
    a.z = y;
    a.near_rec = static_cast<const float *>(c->src);
    a.info = reinterpret_cast<const DwInfo *>(c->src_far);
    a.far_rec = reinterpret_cast<const float *>(a.info + a.ntiles);
    a.part = c->part;
    a.err = c->err;
    cudaEvent_t ev = nullptr;
    prof_begin(c, ZM_K_BR, &ev);
    brdw_kernel<<<dim3(c->plan.ntb, c->plan.nsplit), kTs, 0, c->stream>>>(a);
    prof_end(c, ZM_K_BR, ev);
    c->prof.acc.pairs += (int64_t)g.N * (int64_t)g.N;
    return cuda_check(cudaGetLastError(), "Birkhoff-Rott kernel launch");
}

ZM_BOUNDS_READER(bounds_brdw)

}  // namespace zm
