// The FP64 even-odd hop in two-limb fixed point (fixed.cuh).
//
// The FP64 kernel (dslash.cu) is at the limit of its pipe (89 % busy): 1128 FP64 instructions per site and
// right-hand side at two lanes per cycle and SM, 18000 cycles a warp.  Here a thread (site, right-hand
// side) takes the operand as 58-bit integers over a power of two per spinor (made by a pass over it),
// shifts its eight neighbours to their largest exponent E, and does the spin projection, the link products
// (links with their hop weight, as limbs) and the clover block (limbs over a power of two per block) in
// integers: 2520 IMAD.WIDE in all and more shifts and additions, on pipes of 32 and 64 lanes.  Only the
// difference with z is FP64.  24^3 x 8, 32 right-hand sides: 1.59 ms and 0.09 ms to cut the operand,
// against 4.86 ms (3.00 ms with the eight directions unrolled, which missed the instruction cache).
//
// Accuracy: an entry is cut at 2^-58 of the power of two above the largest neighbour entry and a product sum
// rounded at 2^-57 of it, and the products of low limbs that are left out come to an rms of 2^-57.3 a sum,
// against the 2^-53 of every FP64 operation.  All of it goes by that largest entry: an entry below 2^-5 of it
// has fewer than 53 bits.
//
// Operands and clover blocks with NaN or infinities, links not bounded by one, links or hop weights that are
// small against the limbs' unit (clover.cu; ordinary links up to xi = 16 are not) and hop weights >= 1 (xi <= 1/2)
// take the FP64 kernel, which is launched behind this one and returns at once otherwise.
#include "dirac.cuh"
#include "fixed.cuh"

namespace laph {

namespace {

// fix[cb][12][r] = the entries cut at 2^(e - 58), exps[cb][r] = e with all 24 reals below 2^e;
// flag[1] set where one is not finite
__global__ void __launch_bounds__(256) cut_kernel(long n, int nr, const c64 *__restrict__ in, longlong2 *__restrict__ fix,
                                                  short *__restrict__ exps, int *flag) {
    const long i = (long)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const long o = (i / nr) * 12 * nr + i % nr;
    const double2 *f = reinterpret_cast<const double2 *>(in) + o;
    double2 v[12];
    uint32_t m = 0, low = 0;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        v[k] = __ldg(f + (long)k * nr);
        m = max(m, max((uint32_t)__double2hiint(v[k].x) & 0x7FFFFFFFu, (uint32_t)__double2hiint(v[k].y) & 0x7FFFFFFFu));
        low |= (uint32_t)__double2loint(v[k].x) | (uint32_t)__double2loint(v[k].y);
    }
    const int ex = (int)(m >> 20);
    if (ex == 0x7FF) flag[1] = 1;
    const int E = max(ex - 1022, EXP_MIN);
    exps[i] = (short)((m | low) == 0 ? EXP_NONE : E);
#pragma unroll
    for (int k = 0; k < 12; ++k) fix[o + (long)k * nr] = make_longlong2(cut(v[k].x, E), cut(v[k].y, E));
}

struct C6 {   // int64 complex
    long long re, im;
};
__device__ __forceinline__ C6 operator+(C6 a, C6 b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ C6 operator-(C6 a, C6 b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ C6 c6i(C6 a) { return {-a.im, a.re}; }    // i a
__device__ __forceinline__ C6 c6mi(C6 a) { return {a.im, -a.re}; }   // -i a

__device__ __forceinline__ C6 c6neg(C6 a) { return {-a.re, -a.im}; }

// h = u -+ G d of direction dir = 2 mu + (0 forward, 1 backward) and colour c
template <int DIR>
__device__ __forceinline__ void project(const C6 v[4], C6 &a, C6 &b) {
    constexpr int MU = DIR >> 1;
    constexpr bool FWD = !(DIR & 1);
    // G d with G_1 = -i s1, G_2 = -i s2, G_3 = -i s3, G_4 = 1
    const C6 g0 = MU == 0 ? c6mi(v[3]) : MU == 1 ? c6neg(v[3]) : MU == 2 ? c6mi(v[2]) : v[2];
    const C6 g1 = MU == 0 ? c6mi(v[2]) : MU == 1 ? v[2] : MU == 2 ? c6i(v[3]) : v[3];
    a = FWD ? v[0] - g0 : v[0] + g0;
    b = FWD ? v[1] - g1 : v[1] + g1;
}
// lower components -+ G^dag k
template <int DIR>
__device__ __forceinline__ void lower(C6 &a, C6 &b, C6 k0, C6 k1) {
    constexpr int MU = DIR >> 1;
    constexpr bool FWD = !(DIR & 1);
    const C6 l0 = MU == 0 ? c6i(k1) : MU == 1 ? k1 : MU == 2 ? c6i(k0) : k0;
    const C6 l1 = MU == 0 ? c6i(k0) : MU == 1 ? c6neg(k0) : MU == 2 ? c6mi(k1) : k1;
    a = FWD ? a - l0 : a + l0;
    b = FWD ? b - l1 : b + l1;
}
#define FIX_CASES(F)                                                                                       \
    switch (dir) {                                                                                         \
        case 0: F(0) break;                                                                                \
        case 1: F(1) break;                                                                                \
        case 2: F(2) break;                                                                                \
        case 3: F(3) break;                                                                                \
        case 4: F(4) break;                                                                                \
        case 5: F(5) break;                                                                                \
        case 6: F(6) break;                                                                                \
        default: F(7) break;                                                                               \
    }

// acc += hw (1 -+ gamma_mu) U psi in units 2^-56 2^E, psi cut at 2^(E - sh - 58).  One copy of the code
// for the eight directions (eight copies missed the instruction cache half of the time): a backward hop
// is the conjugate of the forward product with the conjugate spinor and the transposed link.
__device__ __forceinline__ void dir_fix(int dir, C6 acc[12], const longlong2 *__restrict__ f, int nr, const int4 *__restrict__ u,
                                        int sh, bool flip) {
    const bool bwd = dir & 1;
    C6 v[12], h0[3], h1[3];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const longlong2 z = __ldg(f + (long)k * nr);
        v[k] = {z.x >> sh, z.y >> sh};
    }
#define FIX_PROJ(D)                                                  \
    _Pragma("unroll") for (int c = 0; c < 3; ++c) {                  \
        const C6 w[4] = {v[c], v[3 + c], v[6 + c], v[9 + c]};        \
        project<D>(w, h0[c], h1[c]);                                 \
    }
    FIX_CASES(FIX_PROJ)
#undef FIX_PROJ
    if (bwd) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            h0[c].im = -h0[c].im;
            h1[c].im = -h1[c].im;
        }
    }
    CX h[2][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        h[0][c] = {limbs58(h0[c].re), limbs58(h0[c].im)};
        h[1][c] = {limbs58(h1[c].re), limbs58(h1[c].im)};
    }
    const int sa = bwd ? 1 : 3, sb = bwd ? 3 : 1;
    C6 k0[3], k1[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        Acc re[2], im[2];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int4 e = __ldg(u + a * sa + b * sb);
            const FX ur{e.x, e.y}, ui{e.z, e.w}, un = neg(ui);
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                re[s].mad(ur, h[s][b].re);
                im[s].mad(ur, h[s][b].im);
                re[s].mad(un, h[s][b].im);
                im[s].mad(ui, h[s][b].re);
            }
        }
        k0[a] = {floor_value(re[0]), floor_value(im[0])};
        k1[a] = {floor_value(re[1]), floor_value(im[1])};
    }
    if (bwd) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            k0[a].im = -k0[a].im;
            k1[a].im = -k1[a].im;
        }
    }
    if (flip) {   // a hop across the time boundary
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            k0[a] = c6neg(k0[a]);
            k1[a] = c6neg(k1[a]);
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        acc[a] = acc[a] + k0[a];
        acc[3 + a] = acc[3 + a] + k1[a];
    }
#define FIX_LOWER(D) \
    _Pragma("unroll") for (int a = 0; a < 3; ++a) lower<D>(acc[6 + a], acc[9 + a], k0[a], k1[a]);
    FIX_CASES(FIX_LOWER)
#undef FIX_LOWER
}

// row i of a packed Hermitian block times x (sum in units 2^-28 of the limbs' units of x)
__device__ __forceinline__ C6 herm_row(const int2 *__restrict__ blk, int i, const CX x[6]) {
    Acc re, im;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        if (j == i) {
            const int2 d = __ldg(blk + i);
            re.mad(FX{d.x, d.y}, x[j].re);
            im.mad(FX{d.x, d.y}, x[j].im);
        } else {
            const int o = 6 + 2 * (i > j ? i * (i - 1) / 2 + j : j * (j - 1) / 2 + i);
            const int4 e = __ldg(reinterpret_cast<const int4 *>(blk + o));
            const FX lr{e.x, e.y}, li{i > j ? e.z : -e.z, i > j ? e.w : -e.w};
            re.mad(lr, x[j].re);
            re.mad(neg(li), x[j].im);
            im.mad(lr, x[j].im);
            im.mad(li, x[j].re);
        }
    }
    return {floor_value(re), floor_value(im)};
}

// y = A x in FP64 for operands that are not finite
__device__ __noinline__ void herm12_fp64(const double *__restrict__ b, const c64 *__restrict__ x, int nr, c64 *y) {
    for (int h = 0; h < 2; ++h)
        for (int i = 0; i < 6; ++i) {
            c64 s{0, 0};
            for (int j = 0; j < 6; ++j) {
                const c64 v = x[(long)(6 * h + j) * nr];
                const double *q = b + h * 36;
                if (i == j) {
                    s += q[i] * v;
                } else {
                    const int o = 6 + 2 * (i > j ? i * (i - 1) / 2 + j : j * (j - 1) / 2 + i);
                    const c64 l{q[o], q[o + 1]};
                    s += i > j ? l * v : cmul_conj(l, v);
                }
            }
            y[6 * h + i] = s;
        }
}

template <int MODE>
__global__ void __launch_bounds__(128) hop_fix_kernel(const DiracOp op, int p, c64 *__restrict__ out,
                                                      const longlong2 *__restrict__ in, const c64 *__restrict__ z,
                                                      const c64 *__restrict__ xp, int nr, const short *__restrict__ exps) {
    if (op.general[0] || op.general[1]) return;
    const long tid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long Vh = op.g.Vh;
    if (tid >= Vh * nr) return;
    const int cb = (int)(tid / nr), r = (int)(tid - (long)cb * nr);
    const int *nb8 = op.nbr + ((long)p * Vh + cb) * 8;
    int E = EXP_MIN;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int j = __ldg(nb8 + k);
        E = max(E, (int)exps[(long)(j < 0 ? ~j : j) * nr + r]);
    }
    C6 acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = {0, 0};
#pragma unroll 1
    for (int dir = 0; dir < 8; ++dir) {
        const int mu = dir >> 1, e = __ldg(nb8 + (dir & 1 ? 4 + mu : mu)), j = e < 0 ? ~e : e;
        const int sh = min(E - max((int)exps[(long)j * nr + r], EXP_MIN), 63);
        const int4 *u = op.Lfix + (dir & 1 ? ((long)(1 - p) * 4 + mu) * Vh + j : ((long)p * 4 + mu) * Vh + cb) * 9;
        dir_fix(dir, acc, in + (long)j * 12 * nr + r, nr, u, sh, e < 0);
    }
    const long site = (long)p * Vh + cb;
    c64 *dst = out + (long)cb * 12 * nr + r;
    const c64 *zz = z + (long)cb * 12 * nr + r;
    constexpr bool inv = MODE == HOP_CLOVINV || MODE == HOP_CLOVINV_XPAY;
    constexpr bool subz = MODE == HOP_CLOVINV_XPAY || MODE == HOP_RESID;
    if (inv) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            // the sums over the power of two just above them: t 2^-56 2^E = (t 2^up) 2^-58 2^(E + 2 - up)
            uint64_t any = 0;
#pragma unroll
            for (int k = 0; k < 6; ++k)
                any |= (uint64_t)(acc[6 * h + k].re ^ (acc[6 * h + k].re >> 63)) | (uint64_t)(acc[6 * h + k].im ^ (acc[6 * h + k].im >> 63));
            const int up = __clzll((long long)any) - 6;   // leading bit to 2^57 (63 - 6)
            CX x[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const C6 t = acc[6 * h + k];
                x[k] = up >= 0 ? CX{limbs58(t.re << up), limbs58(t.im << up)}
                               : CX{limbs58(shr_near(t.re, -up)), limbs58(shr_near(t.im, -up))};
            }
            const int q = E + 2 - up + __ldg(op.cinvexp + site * 2 + h) - 56;
            const int2 *blk = op.cinvfix + (site * 2 + h) * CLOV_BLOCK;
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                const C6 y = herm_row(blk, i, x);
                c64 v{to_double(y.re, q), to_double(y.im, q)};
                if (subz) v = zz[(long)(6 * h + i) * nr] - v;
                dst[(long)(6 * h + i) * nr] = v;
            }
        }
        return;
    }
    // A xp + hop [or z - that]: the block product at its own exponent, both shifted to the larger one
    const c64 *xx = xp + (long)cb * 12 * nr + r;
    uint32_t m = 0;
    double2 xv[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        xv[k] = __ldg(reinterpret_cast<const double2 *>(xx) + (long)k * nr);
        m = max(m, max((uint32_t)__double2hiint(xv[k].x) & 0x7FFFFFFFu, (uint32_t)__double2hiint(xv[k].y) & 0x7FFFFFFFu));
    }
    if ((m >> 20) == 0x7FF) {
        c64 y[12];
        herm12_fp64(op.clov64 + site * 2 * CLOV_BLOCK, xx, nr, y);
        for (int k = 0; k < 12; ++k) {
            c64 v = y[k] + c64{to_double(acc[k].re, E - 56), to_double(acc[k].im, E - 56)};
            if (subz) v = zz[(long)k * nr] - v;
            dst[(long)k * nr] = v;
        }
        return;
    }
    const int Ex = max((int)(m >> 20) - 1022, EXP_MIN);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        CX x[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) x[k] = {limbs58(cut(xv[6 * h + k].x, Ex)), limbs58(cut(xv[6 * h + k].y, Ex))};
        // at the larger exponent: |block product| < 12 2^Ey, |acc| < 40 2^E in units 2^-56, no overflow
        const int Ey = Ex + __ldg(op.clovexp + site * 2 + h), Em = max(E, Ey);
        const int sa = min(Em - E, 62), sy = min(Em - Ey, 62);
        const int2 *blk = op.clovfix + (site * 2 + h) * CLOV_BLOCK;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const C6 y = herm_row(blk, i, x), a = acc[6 * h + i];
            c64 v{to_double(shr_near(y.re, sy) + shr_near(a.re, sa), Em - 56),
                  to_double(shr_near(y.im, sy) + shr_near(a.im, sa), Em - 56)};
            if (subz) v = zz[(long)(6 * h + i) * nr] - v;
            dst[(long)(6 * h + i) * nr] = v;
        }
    }
}

}  // namespace

// The fixed-point hop where the operator allows it; false if the FP64 kernel has to do the launch.  The
// FP64 kernel still follows (guarded by op.general) for operands that turn out not to be finite.
bool hop_fix(const DiracOp &op, int p, HopMode mode, c64 *out, const c64 *in, const c64 *z, const c64 *xp, int nr, int block,
             cudaStream_t s) {
    const long n = op.g.Vh * nr;
    if (!op.weights_bounded || !op.Lfix) return false;
    longlong2 *fix = (longlong2 *)ws_spare(op.ctx, "hop:fix", sizeof(longlong2) * 12 * n);
    if (!fix) return false;
    short *exps = (short *)ws_get(op.ctx, "hop:exps", sizeof(short) * n);
    LAPH_CUDA(cudaMemsetAsync(op.general + 1, 0, sizeof(int), s));
    cut_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, nr, in, fix, exps, op.general);
    LAPH_LAUNCH_CHECK();
    const unsigned grid = grid_for(n, block);
    switch (mode) {
        case HOP_CLOVINV: hop_fix_kernel<HOP_CLOVINV><<<grid, block, 0, s>>>(op, p, out, fix, z, xp, nr, exps); break;
        case HOP_CLOVINV_XPAY: hop_fix_kernel<HOP_CLOVINV_XPAY><<<grid, block, 0, s>>>(op, p, out, fix, z, xp, nr, exps); break;
        case HOP_APPLY: hop_fix_kernel<HOP_APPLY><<<grid, block, 0, s>>>(op, p, out, fix, z, xp, nr, exps); break;
        case HOP_RESID: hop_fix_kernel<HOP_RESID><<<grid, block, 0, s>>>(op, p, out, fix, z, xp, nr, exps); break;
    }
    LAPH_LAUNCH_CHECK();
    return true;
}

}  // namespace laph
