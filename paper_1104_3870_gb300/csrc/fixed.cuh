// Two-limb fixed-point arithmetic on the integer pipe, for FP64-accurate products of bounded numbers on
// a GPU with two FP64 multiply-adds per cycle and SM.  A real is x = h 2^-28 + l 2^-58 with |l| <= 2^29;
// a product sum keeps sum h h' and sum (h l' + l h') in 64-bit registers (three IMAD.WIDE per real
// product).  l l' is left out: below 2^-58 for two such limbs, below 2^-57 where one comes from limbs58 (a low
// limb in [0, 2^30)), with an rms of 2^-57.3 for the six of a row times a vector.
#pragma once
#include "common.cuh"

namespace laph {

struct FX {
    int h, l;
};
struct CX {
    FX re, im;
};
__device__ __forceinline__ FX neg(FX a) { return {-a.h, -a.l}; }
__device__ __forceinline__ CX conj(CX a) { return {a.re, neg(a.im)}; }

// mantissa of x with its leading bit at bit 63 (garbage of the same size for zeros and subnormals)
__device__ __forceinline__ uint64_t fx_mantissa(uint32_t hi, uint32_t lo) {
    return (uint64_t)(__funnelshift_l(lo, hi, 11) | 0x80000000u) << 32 | (lo << 11);
}
// logical right shift, zero for 64 and more
__device__ __forceinline__ uint64_t fx_shr(uint64_t m, int sh) {
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(sh));
    return m;
}
// round(x 2^58) as limbs, |x| < 2
__device__ __forceinline__ FX to_fx(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint64_t m = fx_shr(fx_mantissa(hi, lo), 1027 - (int)((hi >> 20) & 0x7FFu));
    long long f = (long long)((m + 1) >> 1);
    if (hi >> 31) f = -f;
    const int h = (int)((f + (1ll << 29)) >> 30);
    return {h, (int)(f - ((long long)h << 30))};
}
// a real of the result: sum of products in units 2^-56
struct Acc {
    long long hh = 0, cr = 0;
    __device__ __forceinline__ void mad(FX a, FX b) {
        hh += (long long)a.h * b.h;
        cr += (long long)a.h * b.l;
        cr += (long long)a.l * b.h;
    }
    __device__ __forceinline__ long long value() const { return hh + ((cr + (1ll << 29)) >> 30); }
};

constexpr int EXP_NONE = -2000;   // a spinor of zeros
constexpr int EXP_MIN = -1021;    // every FP64 number below 2^EXP_MIN is subnormal

// x 2^(58 - E) cut towards zero, |x| < 2^E, E >= EXP_MIN
__device__ __forceinline__ long long cut(double x, int E) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int ex = (int)((hi >> 20) & 0x7FFu);
    const uint32_t top = __funnelshift_l(lo, hi, 11) | (ex ? 0x80000000u : 0u);   // zeros and subnormals have no leading one
    const uint64_t m = fx_shr((uint64_t)top << 32 | (lo << 11), 1028 + E - max(ex, 1));
    const uint64_t s = (uint64_t)(int64_t)((int32_t)hi >> 31);
    return (long long)((m ^ s) - s);
}
// t 2^-58 as limbs, |t| < 2^59, the low one in [0, 2^30)
__device__ __forceinline__ FX limbs58(long long t) { return {(int)(t >> 30), (int)((uint32_t)t & 0x3FFFFFFFu)}; }
// sum of a product in units 2^-56
__device__ __forceinline__ long long floor_value(const Acc &a) { return a.hh + (a.cr >> 30); }
__device__ __forceinline__ long long shr_near(long long t, int s) { return s > 0 ? (t + (1ll << (s - 1))) >> s : t; }
// the double nearest to t 2^q
__device__ __forceinline__ double to_double(long long t, int q) {
    if (t == 0) return 0.0;
    const long long s = t >> 63;
    const uint64_t a = (uint64_t)((t ^ s) - s);
    const int lz = __clzll((long long)a);
    const uint64_t top = a << lz;
    const uint64_t m = (top >> 11) + ((top >> 10) & 1);   // [2^52, 2^53]
    const int ex = q + 11 - lz + 1075;
    if (ex < 1 || ex > 2045) return ldexp((double)t, q);
    const uint64_t bits = ((uint64_t)ex << 52) + (m - (1ull << 52));
    return __longlong_as_double((long long)(bits | (uint64_t)s << 63));
}

}  // namespace laph
