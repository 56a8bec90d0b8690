// zm_brdw.cu -- the FP64 all-pairs Birkhoff-Rott sum (paper Sec. 2 BRSolver, Sec. 3.2.1
// ExactBRSolver) on meshes of at least kDwMinN nodes, with the FP64 pipe kept for the pairs whose
// rounding decides the result:
//     u_i = sum_j (z_j - z_i) x gamma'_j / (|z_j - z_i|^2 + delta^2)^(3/2).
//
// What bounds it.  GB300 executes 2 FP64 instructions per clock and SM against 128 FP32 ones, so
// the 21 FP64 instructions of a pair (zm_br.cu) cost 10.5 clocks of an SM whose other pipes idle
// (measured: the pipe 90 % busy, 190 ms per 256 x 256 evaluation).  A pair far apart compared with
// its source tile is evaluated here in FP32 pairs and integers instead: 53 FP32 lane
// operations (two lanes per packed instruction), 6 integer multiply-adds 32 x 32 + 64 bits, one
// reciprocal square root and one conversion, about half a clock of the FMA pipe, which bounds it.
// 190.3 -> 12.5 ms at 256 x 256, 13.0 -> 1.2 at 128 x 128, 7.5 -> 0.70 at 90 x 131, 0.81 -> 0.27 at
// 64 x 64 (one evaluation).
//
// Tiles.  8 x 8 mesh patches (64 nodes) serve as target tiles (one CTA of 64 threads, one target
// per thread) and as source tiles, staged by 1D bulk TMA.  Small tiles keep the near region, whose
// pairs cost 20 times as much, small; where a source tile is not far from the target tile, its
// four quarters (4 x 4 nodes) are classified against each warp's 32 targets.  Measured at 256 x
// 256 / 128 x 128: without the quarters 17.4 / 1.94 ms, with them 15.6 / 1.27.  By bounding spheres:
//   far   (centres at least kappa source radii plus the targets' radius apart): the form below;
//   near  FP64 throughout, as in zm_br.cu, on the untouched positions and strengths.
// A tile's near neighbours spread over the source splits (the splits take the tiles in turn).
// Near pairs carry most of the sum's rounding error: a sheet's pair terms fall off as 1/r^2,
// so the root sum square of all terms beyond R is 0.14 dx / R of the strength, and an independent
// relative error of 1e-14 in them is lost in the FP64 rounding of the near terms and of the sum
// itself.  What a target and a source tile have in common (t, |t|^2, the final products) is kept
// in FP64 or exact, since its error would not average out over the tile.
//
// Far pairs.  Everything is relative to the source tile's centre c: s_j = z_j - c, t_i = z_i - c
// (exact differences of fixed-point words, below), |s| <= |t| / 2, and
//   q = (|t|^2 + delta^2) + |s|^2 - 2 s . t   as an FP32 pair: a power of two C above the first term is
//       added to the running sum, so that no partial sum falls below half of the one before it, the
//       difference of two of them is exact and one FMA returns the rounding error of the product added;
//   K = q^(-3/2) from the special-function estimate y: e = 1 - q y^2 with y^2 exact,
//       y^3 (1 + 3e/2 + 15e^2/8), as FP32 pair (kh, kl);
//   sums G = sum K g, M = sum K (s x g), and u_tile = M - t x G.  K's leading part is
//       scaled to an integer below 2^30 (in a far tile K varies by less than 27, so all of its
//       24 bits are integer bits), g to 27 bits, and K g accumulates exactly in 64-bit integers;
//       the remainders' products, 2^-26 of the terms, accumulate in FP32.  (FP32-pair sums lost
//       up to 2e-14: their low words grow with the number of terms.)
// Positions enter as three words on grids 2^-20, 2^-44 and below (scaled by the mesh's length), so
// that t = z - c has exact word differences.  Tiles whose coordinates, radius or strength do not
// fit these ranges (or are not finite) have an infinite radius, that is, are near to all.
//
// Accuracy of u against long double sums (multi-mode interface, relative L2 over sampled targets;
// zm_br.cu's plain FP64 sum / here): 56 x 56 7.5e-16 / 5.1e-16, 80 x 80 4.7e-16 / 5.6e-16, 96 x 96
// 8.2e-16 / 6.3e-16, 90 x 131 1.2e-15 / 7.5e-16, 128 x 128 1.5e-15 / 7.1e-16, 256 x 256 5.7e-15 /
// 6.9e-16: the long FP64 sums rounded more than the far pairs lose.
#include <algorithm>
#include <cmath>

#include "zm_df64.cuh"
#include "zm_stencil.cuh"

namespace zm {
namespace {

using namespace dw;

constexpr int kT = 8;         // tile side
constexpr int kTs = kT * kT;  // nodes per tile, threads per CTA
constexpr int kSub = 4;       // a tile's quarters: 4 x 4 nodes
constexpr int kNearRows = 6;  // FP64: position, scaled strength
// far rows (32-bit words): s hi (3), s lo (3), |s|^2 hi, lo, g and s x g as integers (6), their
// remainders (6), both as FP32 (6)
constexpr int kFarRows = 26;
constexpr int kRowA = 6, kRowI = 8, kRowR = 14, kRowF = 20;
constexpr int kFarWords = kFarRows * kTs;  // the far record of a tile, or of its four quarters
// the near block of a tile: its quarters' far records (quarter k in columns 16 k ..) and the FP64 record
constexpr int kNearWords = kFarWords + 2 * kNearRows * kTs;
constexpr int kGBits = 26;  // g and s x g: integers below 2^26 in magnitude
constexpr double kGrid1 = 1048576.0, kGrid2 = 17592186044416.0;  // 2^20, 2^44

constexpr float kInf = __builtin_huge_valf();

// One tile as the pair kernel sees it.
struct __align__(16) DwTile {
    float c1[3], c2[3], c3[3];  // centre, scaled, as fixed-point words
    float rho;                  // radius, scaled (infinite: near to all)
    int es;                     // |s| <= rho < 2^es
    float pad;
    double gs;                  // 2^(strength exponent) x 2^(-2 length exponent)
    double c[3];                // centre, scaled
    double pad2[2];
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

// a = w1 + w2 + w3 exactly up to 2^-69: multiples of 2^-20 and 2^-44, and the rest.
__device__ __forceinline__ void words3(double a, float &w1, float &w2, float &w3)
{
    const double g1 = rint(a * kGrid1) * (1.0 / kGrid1);
    const double r1 = a - g1;
    const double g2 = rint(r1 * kGrid2) * (1.0 / kGrid2);
    w1 = __double2float_rn(g1);
    w2 = __double2float_rn(g2);
    w3 = __double2float_rn(r1 - g2);
}

__device__ __forceinline__ unsigned hi_abs(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// Exponent e with rho < 2^e <= 2 rho.
__device__ __forceinline__ int exp_above(float rho) { return (int)(__float_as_uint(rho) >> 23) - 126; }
__device__ __forceinline__ double pow2d(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// Writes one node's far-record column: s = position relative to the centre (|s| < 2^es), gg =
// strength below 1; s x g in units of 2^es.
__device__ __forceinline__ void put_far(float *__restrict__ fr, const double s[3], const double gg[3], int es)
{
    const double iu = pow2d(-es);
    const double t[3] = {s[0] * iu, s[1] * iu, s[2] * iu};
    const double g6[6] = {gg[0], gg[1], gg[2], t[1] * gg[2] - t[2] * gg[1], t[2] * gg[0] - t[0] * gg[2],
                          t[0] * gg[1] - t[1] * gg[0]};
    double a2 = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        a2 = fma(s[k], s[k], a2);
        const float sh = __double2float_rn(s[k]);
        fr[k * kTs] = sh;
        fr[(3 + k) * kTs] = __double2float_rn(s[k] - (double)sh);
    }
    const float ah = __double2float_rn(a2);
    fr[kRowA * kTs] = ah;
    fr[(kRowA + 1) * kTs] = __double2float_rn(a2 - (double)ah);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const double n = rint(g6[k] * (1 << kGBits));
        fr[(kRowI + k) * kTs] = __int_as_float(__double2int_rn(n));
        fr[(kRowR + k) * kTs] = __double2float_rn(g6[k] - n * (1.0 / (1 << kGBits)));
        fr[(kRowF + k) * kTs] = __double2float_rn(g6[k]);
    }
}

__device__ __forceinline__ DwTile make_tile(const double c[3], float rho, double gs)
{
    DwTile t;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        t.c[k] = c[k];
        if (rho < kInf) words3(c[k], t.c1[k], t.c2[k], t.c3[k]);
        else t.c1[k] = t.c2[k] = t.c3[k] = 0.0f;
    }
    t.rho = rho;
    t.es = exp_above(rho);
    t.pad = 0.0f;
    t.gs = gs;
    t.pad2[0] = t.pad2[1] = 0.0;
    return t;
}

// Geometry pass of one tile per CTA: q, the far record and the near block.  One thread per node;
// the radii and the largest strength come from a CTA reduction, so the far records can be written
// already scaled.  Bound by the FP64 instructions of the stencils; 64-thread CTAs spread small
// meshes over the SMs (before, 256-thread CTAs: 48 x 48 ran on 9 SMs).
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
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        c[k] = y[k * N + pc] * pscale;
        cq[k] = y[k * N + pcq] * pscale;
        const double a = zc[k] * pscale;
        ok = ok && fabs(a) < 7.0;  // false for NaN
        s[k] = a - c[k];
        sq[k] = a - cq[k];
        r2 = fma(s[k], s[k], r2);
        r2q = fma(sq[k], sq[k], r2q);
    }
    __syncthreads();
    if (valid) {
        atomicMax(&rmax[0], __float_as_uint(ok ? sqrtf(__double2float_ru(r2)) * 1.000001f : kInf));
        atomicMax(&rmax[1 + qk], __float_as_uint(ok ? sqrtf(__double2float_ru(r2q)) * 1.000001f : kInf));
        atomicMax(&gmax, max(hi_abs(gm[0]), max(hi_abs(gm[1]), hi_abs(gm[2]))));
    }
    __syncthreads();
    const int eg = gmax ? (int)(gmax >> 20) - 1022 : 0;  // |strength components| < 2^eg
    const bool fit = eg >= -400 && eg <= 400 && __uint_as_float(rmax[0]) < 1e30f;
    const double gs = pow2d(fit ? eg : 0) * gscale;

    float *fr = far_rec + (size_t)tile * kFarWords;
    float *nf = near_rec + (size_t)tile * kNearWords;
    double *nd = reinterpret_cast<double *>(nf + kFarWords);
    // zero every column that no node fills
    if (pt.count < kTs) {
        for (int e = tid; e < kFarWords; e += kTs)
            if ((e & (kTs - 1)) >= pt.count) fr[e] = 0.0f;
        for (int e = tid; e < kFarWords; e += kTs) {
            const int col = e & (kTs - 1);
            if ((col & 15) >= quarter_of(pt, col >> 4).count) nf[e] = 0.0f;
        }
    }
    if (valid) {
        const int slot = qk * 16 + (li - (qk >> 1) * kSub) * pq.h2 + (lj - (qk & 1) * kSub);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            nd[k * kTs + slot] = zc[k];
            nd[(3 + k) * kTs + slot] = gm[k];
        }
        if (fit) {
            const double gi = pow2d(-eg);
            const double gg[3] = {gm[0] * gi, gm[1] * gi, gm[2] * gi};
            put_far(fr + tid, s, gg, exp_above(__uint_as_float(rmax[0])));
            put_far(nf + slot, sq, gg, exp_above(__uint_as_float(rmax[1 + qk])));
        }
    }
    if (tid == 0) info[tile].tile = make_tile(c, fit ? __uint_as_float(rmax[0]) : kInf, gs);
    if (valid && p == pcq) info[tile].quarter[qk] = make_tile(cq, fit ? __uint_as_float(rmax[1 + qk]) : kInf, gs);
}

__device__ __forceinline__ u64 dup2(float x) { return pk(x, x); }
__device__ __forceinline__ u64 rsq2(u64 v) { return pk(dev::rsqrt_approx(lane0(v)), dev::rsqrt_approx(lane1(v))); }

// acc += a b, 64-bit; as PTX because the C expression compiles to three instructions (counted: 13
// instead of 4 integer multiplies for 4 products)
__device__ __forceinline__ void mad_wide(long long &acc, int a, int b)
{
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// The far pairs of one target and one source tile (record in shared memory): adds sum_j K (s - t) x g
// to u.  td: the target, scaled, in FP64; tw: its words.
__device__ __forceinline__ void far_tile(const float *__restrict__ rec, int groups, const double td[3],
                                           const float *tw, const DwTile &T, double d2, float d2f, double u[3])
{
    df t[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        // exact word differences; the leading one is zero or larger than the second
        const df h = fast_two_sum(__fsub_rn(tw[k], T.c1[k]), __fsub_rn(tw[3 + k], T.c2[k]));
        t[k] = fast_two_sum(h.hi, __fadd_rn(h.lo, __fsub_rn(tw[6 + k], T.c3[k])));
    }
    const double ex = td[0] - T.c[0], ey = td[1] - T.c[1], ez = td[2] - T.c[2];
    const double t2d = fma(ex, ex, fma(ey, ey, ez * ez)), B = t2d + d2;
    // B + C with the power of two C above B: the leading part, rounded to C's grid, from B's leading 23
    // mantissa bits, and the signed rest from its last 30 (no FP64 instructions)
    const int bhi = __double2hiint(B), eq = (bhi >> 20) - 1022;
    const unsigned blo = (unsigned)__double2loint(B);
    const u64 CC = dup2(__int_as_float((127 + eq) << 23));
    const u64 F0 = dup2(__int_as_float(((127 + eq) << 23) + (1 << 22) + (((bhi & 0xfffff) << 2) | (blo >> 30)) +
                                       ((blo >> 29) & 1)));
    const u64 BL = dup2(__fmul_rn(__int2float_rn((int)(blo << 2) >> 2), __int_as_float((127 + eq - 53) << 23)));
    u64 mh[3], ml[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        mh[k] = dup2(-2.0f * t[k].hi);
        ml[k] = dup2(-2.0f * t[k].lo);
    }
    // the largest K of the tile gives the scale: K 2^S < 2^30
    const float t2 = fmaf(t[0].hi, t[0].hi, fmaf(t[1].hi, t[1].hi, t[2].hi * t[2].hi));
    const float tm = __fsub_rn(__fmul_rn(t2, dev::rsqrt_approx(t2)), T.rho);
    const float ym = dev::rsqrt_approx(__fmaf_rn(tm, tm, d2f));
    const float km = __fmul_rn(__fmul_rn(__fmul_rn(ym, ym), ym), 1.001f);
    const int S = 29 - ((int)(__float_as_uint(km) >> 23) - 127);
    const u64 sc = dup2(__uint_as_float((unsigned)(127 + S) << 23));

    const u64 kOne = dup2(1.0f), kC1 = dup2(1.5f), kC2 = dup2(1.875f);
    const u64 kMagic = dup2(12582912.0f);
    long long I[6] = {0, 0, 0, 0, 0, 0};
    u64 al[6] = {0, 0, 0, 0, 0, 0};
    const ulonglong2 *r4 = reinterpret_cast<const ulonglong2 *>(rec);  // four sources of row k: r4[k * 16 + g]
    constexpr int H = kTs / 4;
#pragma unroll 1
    for (int gq = 0; gq < groups; ++gq) {
        const ulonglong2 *r = r4 + gq;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            auto row = [&](int k) {
                const ulonglong2 v = r[k * H];
                return h ? v.y : v.x;
            };
            const u64 ah = row(kRowA), alo = row(kRowA + 1);
            u64 f = add2(F0, ah);
            u64 l = add2(add2(BL, alo), sub2(ah, sub2(f, F0)));
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const u64 sh = row(k), sl = row(3 + k);
                const u64 f1 = fma2(mh[k], sh, f);
                const u64 er = fma2(mh[k], sh, sub2(f, f1));  // m s - (f1 - f), exact
                l = add2(l, er);
                l = fma2(mh[k], sl, l);
                l = fma2(ml[k], sh, l);
                f = f1;
            }
            const u64 qh = sub2(f, CC), nq = sub2(CC, f);
            const u64 y = rsq2(qh);
            const u64 w = mul2(y, y), nw = neg2(w);
            const u64 wl = fma2(y, y, nw);
            u64 e = fma2(nq, w, kOne);
            e = fma2(nq, wl, e);
            e = fma2(l, nw, e);
            const u64 ys = mul2(y, sc);
            const u64 kh = mul2(w, ys);
            u64 kl = fma2(wl, ys, fma2(w, ys, neg2(kh)));
            const u64 c = mul2(fma2(e, kC2, kC1), e);
            kl = fma2(kl, c, kl);
            kl = fma2(kh, c, kl);
            // integer part of kl into the integer K, the rest below half a unit
            const u64 km2 = add2(kl, kMagic);
            kl = sub2(kl, sub2(km2, kMagic));
            const int ka = __float2int_rn(lane0(kh)) + ((int)(unsigned)km2 - 0x4b400000);
            const int kb = __float2int_rn(lane1(kh)) + ((int)(unsigned)(km2 >> 32) - 0x4b400000);
#pragma unroll
            for (int x = 0; x < 6; ++x) {
                const u64 gi = row(kRowI + x);
                mad_wide(I[x], ka, (int)(unsigned)gi);
                mad_wide(I[x], kb, (int)(unsigned)(gi >> 32));
                al[x] = fma2(kh, row(kRowR + x), al[x]);
                al[x] = fma2(kl, row(kRowF + x), al[x]);
            }
        }
    }
    // the remainders into the integers (below 2^10 K units, to 2^-20), then the tile's sums in FP64
    double v[6];
#pragma unroll
    for (int x = 0; x < 6; ++x) {
        const int rest = __float2int_rn(__fmul_rn(__fadd_rn(lane0(al[x]), lane1(al[x])), 1048576.0f));
        v[x] = (double)(I[x] + ((long long)rest << (kGBits - 20)));
    }
    const double sd = __hiloint2double(__double2hiint(T.gs) - ((S + kGBits) << 20), __double2loint(T.gs));
    const double rs = pow2d(T.es);
    u[0] = fma(fma(rs, v[3], fma(ez, v[1], -ey * v[2])), sd, u[0]);
    u[1] = fma(fma(rs, v[4], fma(ex, v[2], -ez * v[0])), sd, u[1]);
    u[2] = fma(fma(rs, v[5], fma(ey, v[0], -ex * v[1])), sd, u[2]);
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

// Distance between the centre words of a tile and a point's, less the point's own radius.
__device__ __forceinline__ float gap(const DwTile &s, const float *w, float rho)
{
    const float dx = (s.c1[0] - w[0]) + (s.c2[0] - w[3]);
    const float dy = (s.c1[1] - w[1]) + (s.c2[1] - w[4]);
    const float dz = (s.c1[2] - w[2]) + (s.c2[2] - w[5]);
    return sqrtf(dx * dx + dy * dy + dz * dz) * 0.9999f - rho;
}
// 2^-20 keeps K in range; an infinite radius is never far.
__device__ __forceinline__ bool is_far(float gap, float kappa, float rho)
{
    return gap >= kappa * rho && gap >= 9.5367431640625e-7f;
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
    float tw[9];
    words3(td[0], tw[0], tw[3], tw[6]);
    words3(td[1], tw[1], tw[4], tw[7]);
    words3(td[2], tw[2], tw[5], tw[8]);
    // the target tile's sphere, and the sphere of this warp's 32 targets around one of them
    float cw[6], ct[6];
    const DwTile me = a.info[tt].tile;
    float wr = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        ct[k] = me.c1[k];
        ct[3 + k] = me.c2[k];
        cw[k] = __shfl_sync(0xffffffffu, tw[k], 20);
        cw[3 + k] = __shfl_sync(0xffffffffu, tw[3 + k], 20);
        const float d = (tw[k] - cw[k]) + (tw[3 + k] - cw[3 + k]);
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
            far = is_far(gap(s, ct, me.rho), a.kappa, s.rho);
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
                        far_tile(stage[b] + 16 * q, (count + 3) >> 2, td, tw, s, a.d2s, (float)a.d2s, u);
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

// Factor of the far classification: 2 source radii, or 3 on small meshes, whose plain FP64 sums are
// short and round little (u at 64 x 64 against long double: 5.2e-16 with 3, 7.3e-16 with 2, 7.5e-16
// for the plain sum; 0.27 and 0.24 ms).  Lengths or a core size outside the FP32-pair range leave
// every pair near.
float kappa_of(const zm_ctx *c)
{
    const Geom &g = c->geom;
    const int e = length_exponent(g);
    const double d = std::ldexp(c->delta, -e);
    if (e < -100 || e > 100 || !(d < 16.0) || !(std::min(g.L1, g.L2) > 0)) return kInf;
    return g.N >= 96 * 96 ? 2.0f : 3.0f;
}

DwMesh dw_mesh(const Geom &g)
{
    return DwMesh{g.n1, g.n2, (g.n1 + kT - 1) / kT, (g.n2 + kT - 1) / kT};
}

}  // namespace

// Meshes below 56^2 keep the plain FP64 kernel: most of their tiles are near each other, and its short
// sums are the more accurate ones (48 x 48: 0.31 against 0.25 ms, 3.5e-16 against 4.5e-16).
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
