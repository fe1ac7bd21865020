// FP64-accurate batched complex GEMM on the tensor cores from exact integer slices:
//   C[z][n][c] = sum_{k < K} conj(A(z, n, k)) B(z, c, k)
// for operands that a loader functor reads in any layout.  Users: the sink coefficients
// (sinks_tc.cu), the momentum and displaced overlaps and the meson functions (mesonfn_tc.cu).
//
// Exact slices (the error-free splitting of Ozaki, Ogita, Oishi and Rump, 2012).  Over the reals
// (k2 = 2k + part) row (n, re) of A holds (Re a, Im a), row (n, im) holds (-Im a, Re a), column c of
// B holds (Re b, Im b).  Every row and column is scaled by a power of two 2^-E with E from its
// largest entry, so the scaled entries x lie in (-1, 1), and rounded to F = round(x 2^55), an
// integer of eight balanced base-128 digits:
//   F = sum_{j=1..8} d_j 128^(8-j),   d_1 in [-64, 64], d_j in [-64, 63] else
// (add 64 to every digit, cut the sum into 7-bit fields, subtract 64 again).  FP16 holds each
// digit exactly, a digit product is at most 2^12 and a diagonal j + l = D has at most eight pairs,
// so the sums of one diagonal over 512 real k stay within 8 * 512 * 2^12 = 2^24 and the tensor
// cores' FP32 accumulation is exact.  The eight diagonals D = 2..9 (36 digit pairs) are read from
// TMEM every 512 real k and added as integers into one 96-bit sum per output (units of 2^-61), which
// stays exact too; splitting K over CTAs adds such sums, so a result does not depend on the split.  What is lost: the rounding of the entries
// (2^-56 of the largest entry of the row or column, so an entry below an eighth of that keeps fewer than 53
// bits, and a result is accurate to the rows' largest entries, not to its own size) and the pairs j + l >= 10 (seven products of
// at most 2^-56 each at D = 10).  With x of typical size 1/20 of the row's largest entry that is
// below the rounding of an FP64 sum.
//
// Kernel: one CTA per 64 rows n (128 real rows) x 64 columns x K range.  Sixteen warps
// cut the digits of a sub-chunk of 32 real k into shared memory (K-major core matrices without
// swizzle), warps 0-7 those of A, 8-15 those of B; every thread owns one row or column (four complex
// k), whose operands it loads one sub-chunk ahead, and the 96-bit sums of 16 outputs.  Eight lanes
// take two rows x four k: their loads are two 64-byte segments, and the slabs' 32-byte offset keeps
// their 16-byte stores on different banks (eight rows x one k took 32 instead of 8 wavefronts a load,
// and the shared-memory pipe, which feeds the tensor cores too, was 88 % busy).  One more thread issues tcgen05.mma kind::f16 (M = 128, N = 128, K = 16).
// N = 128 takes two neighbouring digit planes of B at once and writes the accumulators of two
// neighbouring diagonals, so an A plane is read from shared memory half as often as with N = 64
// (at N = 64 the operand reads, 6 KB per 32 cycles, would be the limit); with D paired as (2,3),
// (4,5), (6,7), (8,9) an even j starts at l = 0, a plane of zeros in front of B, and all MMAs on an
// accumulator have one shape, which orders them.  20 MMAs per 16 real k carry 40 plane products for
// the 36 needed.  Two buffers of 100 KB, 512 columns of TMEM: one CTA per SM.
//
// Bounds: 40 * 128 * 64 * 16 FP16 multiply-adds per 16 real k and CTA = 1280 tensor cycles, and
// about as long for the integer instructions that cut 2 * 2048 digits; the FP64 pipe (2 FMA per
// cycle and SM on this GPU) is not used at all.
//
// Every wait is bounded (about a second); a wait that gives up sets a host-visible flag, the CTA
// stops issuing, waits for its issued MMAs (bounded) and frees its TMEM.
#pragma once
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include <cuda_fp16.h>

#include "common.cuh"

namespace laph {
namespace xg {

constexpr int TN = 64;             // rows n (complex) and columns per CTA
constexpr int KS = 32;             // real k per sub-chunk (16 complex)
constexpr int DRAIN = 16;          // sub-chunks per drain (512 real k)
constexpr int PLANES = 8;
// A buffer holds, for each of the four 16-byte k groups of a sub-chunk, a slab of core matrices (8 rows
// x 16 B): the eight planes of A, then a zero plane and the eight planes of B.
constexpr int A_PLANE = 2 * TN * 16, B_PLANE = TN * 16;   // bytes of a plane in a slab (128 and 64 real rows)
constexpr int A_SLAB = PLANES * A_PLANE + 32, B_SLAB = (PLANES + 1) * B_PLANE + 32;   // + 32: the k groups on other banks
constexpr int A_BYTES = 4 * A_SLAB;
constexpr int BUF = A_BYTES + 4 * B_SLAB;
constexpr size_t SMEM = 2 * (size_t)BUF + 1024 + 128;
constexpr int WARPS = 20;           // 16 that cut digits and hold the sums, a warpgroup that issues the MMAs
constexpr long long WAIT = 1LL << 31;               // about one second at the maximum SM clock
constexpr int E_MIN = -958;                         // least exponent: subnormals stay more than 63 bits below it
constexpr int DIRECT = 4096;      // exponent of a row / column that has to be summed in FP64: entries at an end of the range
constexpr int NONFINITE = 8192;   // the same with NaN or inf

__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    for (;;) {
        uint32_t ok;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(ok)
                     : "r"(bar), "r"(parity)
                     : "memory");
        if (ok) return true;
        if (clock64() - t0 > WAIT) return false;
    }
}
__device__ __forceinline__ void bar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint64_t desc(uint32_t saddr, int slab) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)(slab >> 4) << 16;              // K-adjacent core matrices a slab apart
    d |= (uint64_t)(128 >> 4) << 32;               // 8-row groups 128 B apart
    d |= (uint64_t)1 << 46;
    return d;
}

// g = 2 (F + bias) + a rounding bit, F = round(a 2^(55 - E)), bias = 64 in every digit: digit j (plane
// j, weight 128^(8-j)) plus 64 sits in bits 7 (8 - j) + 1 up (eight bits for j = 1).
// rbase = E + 1022, |a| < 2^E, E >= E_MIN (so that zeros and subnormals shift out to zero).
struct Fix {
    uint32_t g0, g1;
};
__device__ __forceinline__ Fix fixed_point(double a, int rbase) {
    const uint32_t h = (uint32_t)__double2hiint(a), l = (uint32_t)__double2loint(a);
    const int sh = 8 + rbase - (int)((h >> 20) & 0x7FFu);   // >= 8
    uint64_t m = (uint64_t)(__funnelshift_l(l, h, 11) | 0x80000000u) << 32 | (l << 11);
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(sh));         // 2 |F| before rounding; 0 past 63
    const uint64_t s = (uint64_t)((int64_t)((int32_t)h >> 31));
    // m ^ s is the floor of the signed value
    const uint64_t g = (m ^ s) + ((((1ull << 56) - 1) / 127 * 64) * 2 + 1);
    return {(uint32_t)g, (uint32_t)(g >> 32)};
}
// FP16 pair (digit of re, digit of im) of plane q + 1.  The byte pair that holds the digit at bits
// off .. off + 6 (off <= 3) becomes the mantissa of 1024 + 2^off u; one multiply-add takes it to u - 64.
template <int q>
__device__ __forceinline__ uint32_t digit_pair(const Fix &re, const Fix &im) {
    constexpr int bit = 7 * (7 - q) + 1;                   // in g
    constexpr bool useh = (bit & 7) > 3;                   // in g >> 4 instead, at bit - 4
    constexpr int pos = useh ? bit - 4 : bit, off = pos & 7, byte = (pos >> 3) & 3;
    constexpr int nxt = byte < 3 ? byte + 1 : byte;        // the digit does not reach past byte 3 of its word
    constexpr uint32_t sel = byte | (nxt << 4) | ((4 + byte) << 8) | ((4 + nxt) << 12);
    constexpr uint32_t mask = ((q == 0 ? 0xFFu : 0x7Fu) << off) * 0x10001u;
    auto word = [](const Fix &f) {
        return useh ? (pos >= 32 ? f.g1 >> 4 : __funnelshift_r(f.g0, f.g1, 4)) : (pos >= 32 ? f.g1 : f.g0);
    };
    const uint32_t a = word(re), b = word(im);
    const uint32_t v = (__byte_perm(a, b, sel) & mask) | 0x64006400u;
    constexpr float sc = 1.0f / (1 << off);
    const __half2 w = __hfma2(*reinterpret_cast<const __half2 *>(&v), __float2half2_rn(sc),
                              __float2half2_rn(-(1024.0f * sc + 64.0f)));
    return *reinterpret_cast<const uint32_t *>(&w);
}

// Op provides (all const __device__):
//   struct RawA / RawB;  rows(), cols(), expA, expB, direct, store;
//   ItemA itemA(z, n), ItemB itemB(z, c)  (fixed for a CTA's life; .rbase the exponent base)
//   load(ItemA, k0, RawA&), value(ItemA, RawA, j) and the same for B: element j is k0 + 4 j (zero past K),
//   so the four lanes of a row read 64 contiguous bytes (the order of k is free as long as A and B share it)
template <class Op>
__global__ void __launch_bounds__(WARPS * 32, 1)
    gemm_kernel(const Op op, int ctiles, int rtiles, int splits, int nsub, int tile0, longlong2 *__restrict__ part, int *flag) {
    extern __shared__ unsigned char xsm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char *base = (unsigned char *)(((uintptr_t)xsm + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = (uint64_t *)(base + 2 * BUF);    // full[2], empty[2], drained
    uint32_t *tslot = (uint32_t *)(bars + 5);
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(base);
    const uint32_t full0 = (uint32_t)__cvta_generic_to_shared(bars), empty0 = full0 + 16, drained = full0 + 32;

    // unit: column tile fastest, then row tile, K split, batch (the CTAs of a batch share its operands in L2);
    // a pass from tile tile0 on has one split unless it is the only one
    int u = tile0 + blockIdx.x;
    const int ct = u % ctiles;
    u /= ctiles;
    const int rt = u % rtiles;
    u /= rtiles;
    const int split = u % splits, z = u / splits;
    const int per = (nsub + splits - 1) / splits;
    const int sub0 = split * per, nloc = min(nsub, sub0 + per) - sub0;   // >= 1 by the choice of splits

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(tslot)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 32) {
        for (int b = 0; b < 2; ++b) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 16;" ::"r"(full0 + 8 * b));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(empty0 + 8 * b));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 16;" ::"r"(drained));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (tid < 512)   // the zero planes
        *(uint4 *)(base + (tid >> 8) * BUF + A_BYTES + ((tid >> 6) & 3) * B_SLAB + (tid & 63) * 16) = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tslot;

    // One thread of the last warpgroup issues the MMAs (a thread that also cut digits was held by the
    // queue of the tensor pipe for most of its 2560 cycles per sub-chunk, and every warp waited for it).
    // 640 threads start with 96 registers each; the four warpgroups that hold the sums take 112 and
    // this one gives up all but 24: 512 * 112 + 128 * 24 = 60416 <= 640 * 96.
    auto issue = [&]() {
        // FP32 accumulate, FP16 A and B, both K-major, M = 128, N = 128
        const uint32_t idesc = (1u << 4) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
        int issued = 0;
        bool ok = true;
        for (int i = 0; i < nloc; ++i) {
            const int b = i & 1;
            if (i % DRAIN == 0 && i > 0) ok = bar_wait(drained, (uint32_t)((i / DRAIN - 1) & 1));
            ok = ok && bar_wait(full0 + 8 * b, (uint32_t)((i >> 1) & 1));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint64_t a0 = desc(sbase + b * BUF, A_SLAB), b0 = desc(sbase + b * BUF + A_BYTES, B_SLAB);
#pragma unroll 1
            for (int ks = 0; ks < KS / 16; ++ks)
#pragma unroll
                for (int j = 1; j <= PLANES; ++j)
#pragma unroll
                    for (int l = j & 1; j + l <= PLANES; l += 2) {   // diagonals j + l and j + l + 1
                        const uint64_t ad = a0 + (uint64_t)(((j - 1) * A_PLANE + ks * 2 * A_SLAB) >> 4);
                        const uint64_t bd = b0 + (uint64_t)((l * B_PLANE + ks * 2 * B_SLAB) >> 4);
                        const uint32_t acc = (j == 1 && ks == 0 && i % DRAIN == 0) ? 0u : 1u;
                        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
                                         tmem + (uint32_t)((j + l - 2) * TN)),
                                     "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
                    }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                empty0 + 8 * b));
            issued = i + 1;
        }
        if (!ok) {
            *(volatile int *)flag = 1;
            // no MMA of this CTA may outlive its TMEM
            if (issued) (void)bar_wait(empty0 + 8 * ((issued - 1) & 1), (uint32_t)(((issued - 1) >> 1) & 1));
        }
    };

    // The loop of one warp; ROWS: it cuts the rows of A (warps 0-7), else the columns of B (warps 8-15).
    auto work = [&](auto rows_tag) {
        constexpr bool ROWS = decltype(rows_tag)::value;
        const int w8 = warp & 7, kg = lane & 3;
        const int item = 8 * w8 + (lane >> 2);   // this thread's row or column of the tile
        const auto it = [&] {
            if constexpr (ROWS)
                return op.itemA(z, rt * TN + item);
            else
                return op.itemB(z, ct * TN + item);
        }();
        std::conditional_t<ROWS, typename Op::RawA, typename Op::RawB> raw;
        uint32_t w0[16], w1[16], w2[16];   // 96-bit sums of 16 columns
#pragma unroll
        for (int c = 0; c < 16; ++c) w0[c] = w1[c] = w2[c] = 0;
        const uint32_t off = (uint32_t)(kg * (ROWS ? A_SLAB : B_SLAB) + (ROWS ? 0 : B_PLANE) + item * 16);
        long k0 = (long)sub0 * (KS / 2) + kg;
        op.load(it, k0, raw);
        auto drain = [&](int i) -> bool {   // diagonals after the MMAs of sub-chunk i
            if (!__all_sync(0xffffffffu, bar_wait(empty0 + 8 * (i & 1), (uint32_t)((i >> 1) & 1)))) return false;
            asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
            for (int d = 0; d < 8; ++d) {
                uint32_t r[16];
                const uint32_t ta = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(d * TN + (warp >> 2) * 16);
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                    : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                      "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                    : "r"(ta));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const int sft = 7 * (7 - d);   // units of 2^-61
                    const long long v = (long long)__float2int_rn(__uint_as_float(r[c])) * (1 << (sft & 31));
                    const uint32_t vl = (uint32_t)v, vh = (uint32_t)(v >> 32);
                    if (sft >= 32)
                        asm("add.cc.u32 %0, %0, %2;\n addc.u32 %1, %1, %3;" : "+r"(w1[c]), "+r"(w2[c]) : "r"(vl), "r"(vh));
                    else
                        asm("add.cc.u32 %0, %0, %3;\n addc.cc.u32 %1, %1, %4;\n addc.u32 %2, %2, %5;"
                            : "+r"(w0[c]), "+r"(w1[c]), "+r"(w2[c])
                            : "r"(vl), "r"(vh), "r"((uint32_t)((int32_t)vh >> 31)));
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            return true;
        };
        bool ok = true;
        for (int i = 0; i < nloc; ++i) {
            const int b = i & 1;
            Fix re[4], im[4];   // the loaded entries in fixed point, before the buffer is free
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const c64 v = op.value(it, raw, j);
                re[j] = fixed_point(v.re, it.rbase);
                im[j] = fixed_point(v.im, it.rbase);
            }
            k0 += KS / 2;
            if (i + 1 < nloc) op.load(it, k0, raw);
            if (i >= 2 && !__all_sync(0xffffffffu, bar_wait(empty0 + 8 * b, (uint32_t)(((i >> 1) - 1) & 1)))) {
                ok = false;
                break;
            }
            unsigned char *buf = base + b * BUF + (ROWS ? 0 : A_BYTES) + off;
            auto plane = [&](auto qtag) {
                constexpr int q = decltype(qtag)::value;
                uint32_t w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) w[j] = digit_pair<q>(re[j], im[j]);
                *(uint4 *)(buf + q * (ROWS ? A_PLANE : B_PLANE)) = make_uint4(w[0], w[1], w[2], w[3]);
                if (ROWS) {   // the row (-im, re)
                    uint32_t x[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t t = __byte_perm(w[j], 0, 0x1032);
                        const __half2 y = __hmul2(*reinterpret_cast<const __half2 *>(&t), __floats2half2_rn(-1.0f, 1.0f));
                        x[j] = *reinterpret_cast<const uint32_t *>(&y);
                    }
                    *(uint4 *)(buf + q * A_PLANE + A_PLANE / 2) = make_uint4(x[0], x[1], x[2], x[3]);
                }
            };
            plane(std::integral_constant<int, 0>{});
            plane(std::integral_constant<int, 1>{});
            plane(std::integral_constant<int, 2>{});
            plane(std::integral_constant<int, 3>{});
            plane(std::integral_constant<int, 4>{});
            plane(std::integral_constant<int, 5>{});
            plane(std::integral_constant<int, 6>{});
            plane(std::integral_constant<int, 7>{});
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) bar_arrive(full0 + 8 * b);
            if (i % DRAIN == 0 && i > 0) {
                ok = drain(i - 1);
                __syncwarp();
                if (!ok) break;
                if (lane == 0) bar_arrive(drained);
            }
        }
        ok = ok && drain(nloc - 1);
        if (!ok) {
            if (lane == 0) *(volatile int *)flag = 1;
        } else {
            // part[split][tile][column 64][real row 128]; the lane is the real row
            const long tile = ((long)z * rtiles + rt) * ctiles + ct - tile0;
            const long tiles = (long)(gridDim.x / splits);
            longlong2 *dst = part + ((split * tiles + tile) * TN + (warp >> 2) * 16) * (2 * TN) + (warp & 3) * 32 + lane;
#pragma unroll
            for (int c = 0; c < 16; ++c)
                if (ct * TN + (warp >> 2) * 16 + c < op.cols())
                    dst[(long)c * 2 * TN] = make_longlong2((long long)((uint64_t)w2[c] << 32 | w1[c]), (long long)w0[c]);
        }
    };
    if (warp >= 16) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 24;");
        if (tid == 512) issue();
        __syncwarp();
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
        if (warp < 8)
            work(std::true_type{});
        else
            work(std::false_type{});
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// The double nearest to (x 2^32 + y) 2^e, y >= 0, in integer arithmetic (four conversions, a multiply-add
// and ldexp on the FP64 pipe made the finish of a small problem 20 us instead of 6).
__device__ __forceinline__ double from_fixed(long long x, long long y, int e) {
    x += y >> 32;
    uint32_t lo = (uint32_t)y;
    const bool neg = x < 0;
    uint64_t hi = (uint64_t)x;
    if (neg) {
        lo = 0u - lo;
        hi = ~hi + (lo == 0 ? 1 : 0);
    }
    if (hi == 0) {
        hi = lo;
        lo = 0;
        e -= 32;
    }
    if (hi == 0) return 0.0;
    const int lz = __clzll((long long)hi);
    const uint64_t w = (uint64_t)lo << 32;
    const uint64_t top = lz ? (hi << lz) | (w >> (64 - lz)) : hi;
    const bool rest = (w << lz) != 0;
    uint64_t m = top >> 11;
    const uint32_t r = (uint32_t)top & 0x7FFu;
    if (r > 0x400u || (r == 0x400u && (rest || (m & 1)))) ++m;   // nearest, ties to even
    const int p = e + 43 - lz;                                    // |value| = m 2^p, m in [2^52, 2^53]
    double v;
    if (p + 1075 < 1 || p + 1075 > 2045)
        v = ldexp((double)m, p);
    else
        v = __longlong_as_double((long long)(((uint64_t)(p + 1075) << 52) + (m - (1ull << 52))));
    return neg ? -v : v;
}

// Adds the K splits and hands C[z][n][c] to Op::store; a row or column with NaN, inf or entries at an end of
// the FP64 range goes through Op::direct (the plain FP64 sum, or NaN where the entry point documents that).
template <class Op>
__global__ void finish_kernel(const Op op, int ctiles, int rtiles, int splits, int tile0, long tiles,
                              const longlong2 *__restrict__ part) {
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const int row = (int)(idx % TN), c = (int)((idx / TN) % TN);
    const long tile = idx / (TN * TN), of = tile0 + tile;   // in the pass, of all
    if (tile >= tiles) return;
    const int ct = (int)(of % ctiles), rt = (int)((of / ctiles) % rtiles);
    const int z = (int)(of / ((long)ctiles * rtiles)), n = rt * TN + row, col = ct * TN + c;
    if (n >= op.rows() || col >= op.cols()) return;
    const int En = op.expA(z, n), Ec = op.expB(z, col);
    if (En >= DIRECT || Ec >= DIRECT) {
        op.store(z, n, col, op.direct(z, n, col));
        return;
    }
    long long rh = 0, rl = 0, ih = 0, il = 0;
    for (int s = 0; s < splits; ++s) {
        const longlong2 *p = part + (((long)s * tiles + tile) * TN + c) * (2 * TN) + row;
        const longlong2 a = p[0], b = p[TN];
        rh += a.x;
        rl += a.y;
        ih += b.x;
        il += b.y;
    }
    op.store(z, n, col, c64{from_fixed(rh, rl, En + Ec - 61), from_fixed(ih, il, En + Ec - 61)});
}

// E of a row from the largest high word of its entries (sign cleared): every entry is below 2^E; 0
// for rows of zeros, NONFINITE where an entry is not finite, DIRECT where the largest is below 2^E_MIN (it
// would be cut short) or at least 2^1023 (a loader's product may overflow).
__device__ __forceinline__ int exp_of_hi(uint32_t h) {
    const int ex = (int)(h >> 20);
    return ex == 0x7FF ? NONFINITE : h == 0 ? 0 : ex - 1022 < E_MIN || ex == 0x7FE ? DIRECT : ex - 1022;
}
__device__ __forceinline__ uint32_t hi_abs(const double2 v) {
    return max((uint32_t)__double2hiint(v.x) & 0x7FFFFFFFu, (uint32_t)__double2hiint(v.y) & 0x7FFFFFFFu);
}

// E of rows of `len` contiguous complex entries, a warp per row (short rows) or a block per row
static __global__ void rows_exp_kernel(const c64 *__restrict__ x, long nrows, int len, int per_warp, int *__restrict__ E) {
    const double2 *src = reinterpret_cast<const double2 *>(x);
    __shared__ uint32_t sm[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long row = per_warp ? (long)blockIdx.x * 8 + warp : blockIdx.x;
    const int first = per_warp ? lane : (int)threadIdx.x, step = per_warp ? 32 : 256;
    uint32_t m = 0;
    if (row < nrows) {
        const double2 *p = src + row * len;
        int k = first;
        for (; k + 7 * step < len; k += 8 * step) {
            double2 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = __ldg(p + k + q * step);
#pragma unroll
            for (int q = 0; q < 8; ++q) m = max(m, hi_abs(v[q]));
        }
        for (; k < len; k += step) m = max(m, hi_abs(__ldg(p + k)));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (per_warp) {
        if (lane == 0 && row < nrows) E[row] = exp_of_hi(m);
        return;
    }
    if (lane == 0) sm[warp] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) m = max(m, sm[w]);
        E[row] = exp_of_hi(m);
    }
}
inline void rows_exp(const c64 *x, long nrows, long len, int *E, cudaStream_t s) {
    const int per_warp = len <= 1024;
    rows_exp_kernel<<<(unsigned)(per_warp ? (nrows + 7) / 8 : nrows), 256, 0, s>>>(x, nrows, (int)len, per_warp, E);
    LAPH_LAUNCH_CHECK();
}

// K splits: the fewest sub-chunk times on the busiest SM, a CTA costing its sub-chunks plus about
// four more (start, drain, partial sums)
inline int choose_splits(long tiles, int nsub, int sms) {
    int best = 1;
    double bt = 1e300;
    for (int s = 1; s <= 32 && s <= nsub; ++s) {
        const int per = (nsub + s - 1) / s;
        if ((nsub + per - 1) / per != s) continue;   // every split gets at least one sub-chunk
        const double t = (double)((tiles * s + sms - 1) / sms) * (per + 4.0) + 0.02 * s;
        if (t < bt * 0.995) {
            bt = t;
            best = s;
        }
    }
    return best;
}

// Host-visible flag of the context that a CTA raises when a wait gives up (checked after the stream drained).
int *host_flag(laph_ctx *ctx);
void check_host_flag(laph_ctx *ctx);

// Tiles whose partial sums are kept at a time: 512 MB, 27 waves of CTAs; down to 32 MB where device memory is short
constexpr long PASS = 4096, PASS_MIN = 256;

template <class Op>
void run(laph_ctx *ctx, const Op &op, long K, int nbatch, int rows, int cols, cudaStream_t s) {
    static bool attr[64] = {false};
    if (!attr[ctx->device & 63]) {
        LAPH_CUDA(cudaFuncSetAttribute(gemm_kernel<Op>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM));
        attr[ctx->device & 63] = true;
    }
    const int ctiles = (cols + TN - 1) / TN, rtiles = (rows + TN - 1) / TN;
    const int nsub = (int)((2 * K + KS - 1) / KS);
    const long tiles = (long)nbatch * ctiles * rtiles;
    LAPH_REQUIRE(tiles < (1L << 31), "problem too large");
    int splits = choose_splits(tiles, nsub, ctx->sm_count > 0 ? ctx->sm_count : 152);
    const size_t unit = sizeof(longlong2) * 2 * TN * TN;
    long pass = std::min(tiles * splits, PASS);
    longlong2 *part = nullptr;
    while (pass > PASS_MIN && !(part = (longlong2 *)ws_spare(ctx, "xgemm:part", unit * (size_t)pass))) pass = std::max(pass / 2, PASS_MIN);
    if (!part) part = (longlong2 *)ws_get(ctx, "xgemm:part", unit * (size_t)pass);
    if (pass < tiles * splits) splits = 1;
    for (long t0 = 0; t0 < tiles; t0 += pass) {
        const long n = std::min(tiles - t0, pass);
        gemm_kernel<Op><<<(unsigned)(n * splits), WARPS * 32, SMEM, s>>>(op, ctiles, rtiles, splits, nsub, (int)t0, part,
                                                                         host_flag(ctx));
        LAPH_LAUNCH_CHECK();
        finish_kernel<Op><<<(unsigned)(n * (TN * TN / 256)), 256, 0, s>>>(op, ctiles, rtiles, splits, (int)t0, n, part);
        LAPH_LAUNCH_CHECK();
    }
}

}  // namespace xg
}  // namespace laph
