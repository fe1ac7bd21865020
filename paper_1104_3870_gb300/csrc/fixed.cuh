// Two-limb fixed-point arithmetic on the integer pipe, for FP64-accurate products of bounded numbers on
// a GPU with two FP64 multiply-adds per cycle and SM.  A real is x = h 2^-28 + l 2^-58 with |l| <= 2^29;
// a product sum keeps sum h h' and sum (h l' + l h') in 64-bit registers (three IMAD.WIDE per real
// product; l l' is below 2^-58).
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

}  // namespace laph
