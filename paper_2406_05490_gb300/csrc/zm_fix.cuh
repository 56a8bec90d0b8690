// zm_fix.cuh -- complex 64-bit integer arithmetic for the FFT Riesz passes (zm_fft.cu): block
// floating point, one power-of-two unit per CTA and pass.
//
// Why integers.  GB300 runs 2 FP64 instructions per clock and SM, and 64 integer adds or 32 x 32 + 64
// bit multiply-adds.  A complex sum is 4 integer adds (a thirtieth of its two FP64 adds' time), a
// complex product 12 multiply-adds and 14 other operations (a sixth of its four FP64 instructions'
// time), and a 60-bit product rounds less than a 53-bit one.
//
// Numbers are integers below 2^60 in magnitude.  In a product the factor x is cut into x = xh 2^30 + xl
// (0 <= xl < 2^30) and the constant w = wh 2^30 + wl (in units of 2^-60) is stored cut:
//     x w = xh wh + (xh wl + xl wh) / 2^30      (xl wl / 2^60, below one unit, dropped),
// each 64-bit sum of four cross products below 2^62.
#pragma once

#include "zm_internal.cuh"

namespace zm {
namespace {

struct Z {
    long long re, im;
};

__device__ __forceinline__ Z ldz(ulonglong2 v) { return Z{(long long)v.x, (long long)v.y}; }
__device__ __forceinline__ ulonglong2 stz(Z a)
{
    return make_ulonglong2((unsigned long long)a.re, (unsigned long long)a.im);
}
__device__ __forceinline__ Z zadd(Z a, Z b) { return Z{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ Z zsub(Z a, Z b) { return Z{a.re - b.re, a.im - b.im}; }
// a + i b for s > 0, a - i b for s < 0
__device__ __forceinline__ Z zadd_i(Z a, Z b, int s)
{
    return s > 0 ? Z{a.re - b.im, a.im + b.re} : Z{a.re + b.im, a.im - b.re};
}

// As PTX: the C expression of a widening multiply-add compiles to three instructions.
__device__ __forceinline__ long long mul_w(int a, int b)
{
    long long r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ long long mad_w(int a, int b, long long c)
{
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
    return c;
}

constexpr int kLimb = 30;
constexpr int kLow = (1 << kLimb) - 1;

// x (w.x 2^30 + w.y + s i (w.z 2^30 + w.w)) 2^-60
__device__ __forceinline__ Z zmul(Z x, int4 w, int s)
{
    const int ih = s > 0 ? w.z : -w.z, il = s > 0 ? w.w : -w.w;
    const int nh = s > 0 ? -w.z : w.z, nl = s > 0 ? -w.w : w.w;
    const int ah = (int)(x.re >> kLimb), al = (int)x.re & kLow;
    const int bh = (int)(x.im >> kLimb), bl = (int)x.im & kLow;
    const long long hr = mad_w(bh, nh, mul_w(ah, w.x));
    const long long hi = mad_w(bh, w.x, mul_w(ah, ih));
    long long cr = 1ll << (kLimb - 1), ci = 1ll << (kLimb - 1);
    cr = mad_w(ah, w.y, cr);
    cr = mad_w(al, w.x, cr);
    cr = mad_w(bh, nl, cr);
    cr = mad_w(bl, nh, cr);
    ci = mad_w(ah, il, ci);
    ci = mad_w(al, ih, ci);
    ci = mad_w(bh, w.y, ci);
    ci = mad_w(bl, w.x, ci);
    return Z{hr + (cr >> kLimb), hi + (ci >> kLimb)};
}

// Rounded right shift (half = 2^(s - 1), 0 for s = 0), after a left shift where s < 0.
struct Shift {
    int l, r;
    long long half;
};
__device__ __forceinline__ Shift make_shift(int s)
{
    return Shift{s < 0 ? -s : 0, s > 0 ? s : 0, s > 0 ? 1ll << (s - 1) : 0ll};
}
// Between FP64 words and fixed point without the FP64 pipe, which the conversions and their scale factors
// would hold longer than the first and last pass can hide (1024 x 1024: pass A 30.8 -> 25.8 us, pass C 42.0 ->
// 37.7; 4096 x 4096: 403 -> 395 and 429 -> 431).
// round(v 2^(54 - eb)) of an FP64 number below 2^eb (eb >= -1021), from its bits; ties away from zero.
__device__ __forceinline__ long long fix_of(unsigned long long v, int eb)
{
    const int e = (int)(v >> 52) & 0x7ff;
    const unsigned long long f = v & ((1ull << 52) - 1);
    // v = m 2^(max(e, 1) - 1076), m < 2^54
    const unsigned long long m = (e ? f | (1ull << 52) : f) << 1;
    const int n = min(1022 + eb - max(e, 1), 63);
    const long long r = (long long)((m + ((1ull << n) >> 1)) >> n);
    return (long long)v < 0 ? -r : r;
}
// v 2^e rounded to FP64 (ties away from zero); |e| <= 900.
__device__ __forceinline__ double fp64_of(long long v, int e)
{
    const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
    const int z = __clzll((long long)a);
    const unsigned long long m = a << (z & 63);
    const unsigned long long r = (m >> 11) + ((m >> 10) & 1);  // 2^52 <= r <= 2^53: the leading bit is added below
    const unsigned long long b = ((unsigned long long)(unsigned)(1023 + 63 - 1 - z + e) << 52) + r;
    return a ? __longlong_as_double((long long)(b | ((unsigned long long)v & 0x8000000000000000ull))) : 0.0;
}
__device__ __forceinline__ Z zshift(Z a, const Shift &s)
{
    return Z{((a.re << s.l) + s.half) >> s.r, ((a.im << s.l) + s.half) >> s.r};
}
__device__ __forceinline__ Z zshift_right(Z a, const Shift &s)
{
    return Z{(a.re + s.half) >> s.r, (a.im + s.half) >> s.r};
}

// OR of the leading words of |re| and |im| (up to one unit) into o: its top bit bounds them.
__device__ __forceinline__ void or_mag(unsigned &o, Z a)
{
    const int h = (int)(a.re >> 32), k = (int)(a.im >> 32);
    o |= (unsigned)(h ^ (h >> 31)) | (unsigned)(k ^ (k >> 31));
}
// Values with OR word o are below 2^(32 + bits); the shift that leaves room for a growth of 2^k
// (and sqrt 2) below 2^60.
__device__ __forceinline__ int room_shift(unsigned o, int k) { return 32 - __clz((int)o) + 32 - (59 - k); }

// x = round(v 2^60) cut into limbs, |v| <= 1
__device__ __forceinline__ void limbs60(double v, int &h, int &l)
{
    const long long x = __double2ll_rn(v * 1152921504606846976.0);
    h = (int)(x >> kLimb);
    l = (int)x & kLow;
}

}  // namespace
}  // namespace zm
