// Operand preparation of the Wilson-clover operator: links in the even-odd layouts, the clover field
// strength, the chiral 6x6 blocks A and their inverses (Sec. IV, the improved anisotropic action; the
// formula is in include/laph.h).
//
// This GPU has two FP64 multiply-adds per cycle and SM, and a site's field strength takes sixty 3x3
// complex products (6500 of them): in FP64, with the blocks in local memory, it took 14 ms on
// 24^3 x 32.  Link matrices have entries of modulus <= 1, so the products are formed here in fixed
// point on the integer pipe (64 multiply-adds per cycle and SM): a real is two limbs,
//   x = h 2^-28 + l 2^-58,  |l| <= 2^29,
// a product sum keeps sum h h' and sum (h l' + l h') in 64-bit registers (three IMAD.WIDE per real
// product; l l', below 2^-58, is left out), and the result is rounded to 2^-56, finer than the FP64 rounding of
// entries near 1/2 that it replaces.  Links that are not bounded this way (a row of norm above 1.001,
// or not finite) or small against the limbs' unit raise a flag, and the FP64 kernels do the lattice instead.
//
//   1. pack_kernel: coalesced through shared memory; L64, L32w, the limbs by site, the flag.
//   2. field_kernel: one thread per site, plane and pair of leaves that share their outer link (five
//      products, six leaf by leaf); its part of F as nine reals by site.
//   3. blocks_kernel: one thread per site and chirality; A and its inverse (L D L^dag in registers),
//      stored through shared memory in FP64 and in the FP32 form of the stencil.
// Times at prepare_dirac.
#include <algorithm>
#include <cmath>

#include "dirac.cuh"
#include "fixed.cuh"
#include "su3.cuh"

namespace laph {

namespace {

// ------------------------------------------------------------------ fixed point
struct MX {
    CX m[3][3];
};
__device__ __forceinline__ FX split(long long t) {   // 2^-56 units to limbs
    const int h = (int)((t + (1ll << 27)) >> 28);
    return {h, (int)((t - ((long long)h << 28)) << 2)};
}
// element (i, j) of op(a) op(b), op = conjugate transpose where the flag is set
template <bool DA, bool DB>
__device__ __forceinline__ void mx_elem(const MX &a, const MX &b, int i, int j, long long &re, long long &im) {
    Acc r, s;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const CX x = DA ? a.m[k][i] : a.m[i][k], y = DB ? b.m[j][k] : b.m[k][j];
        const FX xi = DA ? neg(x.im) : x.im, yi = DB ? neg(y.im) : y.im;
        r.mad(x.re, y.re);
        r.mad(neg(xi), yi);
        s.mad(x.re, yi);
        s.mad(xi, y.re);
    }
    re = r.value();
    im = s.value();
}
template <bool DA, bool DB>
__device__ __forceinline__ MX mx_mul(const MX &a, const MX &b) {
    MX c;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            long long re, im;
            mx_elem<DA, DB>(a, b, i, j, re, im);
            c.m[i][j] = {split(re), split(im)};
        }
    return c;
}
// op(a) op(b) - c
template <bool DA, bool DB>
__device__ __forceinline__ MX mx_mul_sub(const MX &a, const MX &b, const MX &c) {
    MX d;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            long long re, im;
            mx_elem<DA, DB>(a, b, i, j, re, im);
            const CX x = c.m[i][j];
            re -= ((long long)x.re.h << 28) + (x.re.l >> 2);
            im -= ((long long)x.im.h << 28) + (x.im.l >> 2);
            d.m[i][j] = {split(re), split(im)};
        }
    return d;
}

// ------------------------------------------------------------------ packing
constexpr int PK_SITES = 64;

// cb site (p, cb) of the block's 64 consecutive lexicographic sites: local index of the site
__device__ __forceinline__ int local_site(const Geom &g, long s0, int p, int icb) {
    int c[4];
    cb_coords(g, p, (s0 >> 1) + icb, c);
    return 2 * icb + (c[0] & 1);
}

__global__ void __launch_bounds__(256) pack_kernel(Geom g, const c64 *__restrict__ U, double hws, double hwt,
                                                   c64 *__restrict__ L64, float4 *__restrict__ L32w,
                                                   int4 *__restrict__ Lfix, int4 *__restrict__ fix, int *flag) {
    __shared__ double2 sm[PK_SITES * 36];
    __shared__ unsigned char loc[2][PK_SITES / 2];
    const long s0 = (long)blockIdx.x * PK_SITES;
    const int ns = (int)min((long)PK_SITES, g.V - s0);   // even
    const double2 *src = reinterpret_cast<const double2 *>(U) + s0 * 36;
    for (int e = threadIdx.x; e < ns * 36; e += 256) sm[e] = __ldg(src + e);
    if (threadIdx.x < PK_SITES && (int)(threadIdx.x & 31) < ns / 2)
        loc[threadIdx.x >> 5][threadIdx.x & 31] = (unsigned char)local_site(g, s0, threadIdx.x >> 5, threadIdx.x & 31);
    __syncthreads();
    const int nh = ns / 2;
    for (int e = threadIdx.x; e < 8 * nh * 9; e += 256) {   // [p][mu][cb][9]
        const int k = e % 9, icb = (e / 9) % nh, pm = e / (9 * nh);
        const double2 v = sm[loc[pm >> 2][icb] * 36 + (pm & 3) * 9 + k];
        const long o = ((long)pm * g.Vh + (s0 >> 1) + icb) * 9 + k;
        L64[o] = c64{v.x, v.y};
        const float re = (float)v.x, im = (float)v.y;
        L32w[o] = make_float4(re, re, im, im);
        if (Lfix) {
            const double w = (pm & 3) == 3 ? hwt : hws;
            const FX a = to_fx(w * v.x), b = to_fx(w * v.y);
            Lfix[o] = make_int4(a.h, a.l, b.h, b.l);
        }
    }
    for (int e = threadIdx.x; e < 36 * ns; e += 256) {      // [mu][k][site]
        const int is = e % ns, mk = e / ns;
        const double2 v = sm[is * 36 + mk];
        const FX a = to_fx(v.x), b = to_fx(v.y);
        fix[(long)mk * g.V + s0 + is] = make_int4(a.h, a.l, b.h, b.l);
    }
    // Rows of norm up to one; hop weight times row or column zero or at least 2^-5: the limbs' rounding, 2^-59
    // an entry, is then below that of an FP64 sum over it (links of size 1e-6 lost five digits).
    // One conversion of an entry serves its row and its column (16^3 x 32: 73 us, 82 with one for each).
    float *nrm = reinterpret_cast<float *>(sm);   // |entry|^2 in the entry's place, zero for zeros alone
    __syncthreads();
    for (int e = threadIdx.x; e < 36 * ns; e += 256) {
        const double2 v = sm[e];
        const float re = (float)v.x, im = (float)v.y, n = fmaf(re, re, im * im);
        const uint32_t any = ((uint32_t)__double2hiint(v.x) << 1) | (uint32_t)__double2loint(v.x) |
                             ((uint32_t)__double2hiint(v.y) << 1) | (uint32_t)__double2loint(v.y);
        nrm[4 * e] = any ? (n < 1e-30f ? 1e-30f : n) : 0.f;
    }
    __syncthreads();
    bool ok = true;
    const float wt2 = (float)(hwt * hwt), ws2 = (float)(hws * hws);
    for (int e = threadIdx.x; e < 24 * ns; e += 256) {
        const int is = e % 12, step = e % 24 < 12 ? 1 : 3;   // a row or a column
        const float *q = nrm + 4 * ((e / 24) * 36 + (step == 1 ? is * 3 : (is / 3) * 9 + is % 3));
        const float n = q[0] + q[4 * step] + q[8 * step];
        ok &= (step == 3 || n <= 1.001f) && (n == 0.f || (is >= 9 ? wt2 : ws2) * n >= 0.99f / 1024);   // false for NaN
    }
    if (!ok) *flag = 1;
}

// ------------------------------------------------------------------ field strength
__device__ __forceinline__ MX load_fix(const int4 *__restrict__ fix, long V, int mu, int s) {
    MX r;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int4 v = __ldg(fix + (long)(mu * 9 + k) * V + s);
        r.m[k / 3][k % 3] = {{v.x, v.y}, {v.z, v.w}};
    }
    return r;
}

// F[plane][pair][9][V]: the pair's part of (f00, f11, f22, f10, f20, f21) of the Hermitian traceless F_{mu nu}(x).
// The two pairs run the same code on other links: with both in one thread the code (ten products) missed
// the instruction cache for a third of the time.
__global__ void __launch_bounds__(128) field_kernel(Geom g, const int4 *__restrict__ fix, const int *flag,
                                                    double *__restrict__ F) {
    if (*flag) return;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    const int pl = blockIdx.y >> 1, pair = blockIdx.y & 1;
    const int mu = pl < 3 ? 0 : pl < 5 ? 1 : 2, nu = pl < 3 ? pl + 1 : pl < 5 ? pl - 1 : 3;
    const int ns = g.ns, nt = g.nt;
    int c[4], r = s;
    c[0] = r % ns;
    r /= ns;
    c[1] = r % ns;
    r /= ns;
    c[2] = r % ns;
    c[3] = r / ns;
    const int dim[4] = {ns, ns, ns, nt}, str[4] = {1, ns, ns * ns, ns * ns * ns};
    const int mf = c[mu] + 1 == dim[mu] ? -(dim[mu] - 1) * str[mu] : str[mu];
    const int mb = c[mu] == 0 ? (dim[mu] - 1) * str[mu] : -str[mu];
    const int nf = c[nu] + 1 == dim[nu] ? -(dim[nu] - 1) * str[nu] : str[nu];
    const int nb = c[nu] == 0 ? (dim[nu] - 1) * str[nu] : -str[nu];
    auto U = [&](int d, int off) { return load_fix(fix, g.V, d, s + off); };
    // pair 0: leaf 1 - leaf 4^dag = U_mu(x) X,
    //   X = U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag - U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu)
    // pair 1: leaf 2 - leaf 3^dag = X U_mu(x-mu),
    //   X = U_nu(x) U_mu(x-mu+nu)^dag U_nu(x-mu)^dag - U_nu(x-nu)^dag U_mu(x-mu-nu)^dag U_nu(x-mu-nu)
    const int a = pair ? 0 : mf, b = pair ? mb : 0;
    MX x = mx_mul<true, true>(U(nu, a + nb), U(mu, b + nb));
    x = mx_mul<false, false>(x, U(nu, b + nb));
    const MX y = mx_mul<false, true>(U(nu, a), U(mu, b + nf));
    x = mx_mul_sub<false, true>(y, U(nu, b), x);
    const MX o = U(mu, b), l = pair ? x : o, m = pair ? o : x;
    long long wr[3][3], wi[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) mx_elem<false, false>(l, m, i, j, wr[i][j], wi[i][j]);
    // F = (W - W^dag) / (8 i), traceless; W in units 2^-56
    const double u = 1.7347234759768071e-18;   // 2^-59
    double d[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) d[i] = (double)(2 * wi[i][i]) * u;
    const double tr = (double)(2 * (wi[0][0] + wi[1][1] + wi[2][2])) * u * (1.0 / 3.0);
    double *f = F + (long)blockIdx.y * 9 * g.V + s;
#pragma unroll
    for (int i = 0; i < 3; ++i) f[i * g.V] = d[i] - tr;
    int k = 3;
#pragma unroll
    for (int i = 1; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < i; ++j) {
            f[k++ * g.V] = (double)(wi[i][j] + wi[j][i]) * u;
            f[k++ * g.V] = (double)(wr[j][i] - wr[i][j]) * u;
        }
}

// ------------------------------------------------------------------ chiral blocks
__device__ __forceinline__ constexpr int lw(int i, int j) { return i * (i - 1) / 2 + j; }   // strictly lower, i > j

// Packed form of a Hermitian 6x6 block: d[6], then the 15 strictly lower entries row by row.
struct Herm6 {
    double d[6];
    c64 l[15];
};

// Gauss-Jordan inverse with partial pivoting of a packed Hermitian block (for blocks that are not definite)
__device__ __noinline__ void herm6_inverse_pivoted(const double *a_in, double *out) {
    c64 a[6][6], inv[6][6];
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) {
            const double *p = a_in + 6 + 2 * (i > j ? lw(i, j) : i < j ? lw(j, i) : 0);
            a[i][j] = i == j ? c64{a_in[i], 0.0} : i > j ? c64{p[0], p[1]} : c64{p[0], -p[1]};
            inv[i][j] = c64{i == j ? 1.0 : 0.0, 0.0};
        }
    for (int col = 0; col < 6; ++col) {
        int piv = col;
        double best = norm2(a[col][col]);
        for (int r = col + 1; r < 6; ++r)
            if (norm2(a[r][col]) > best) {
                best = norm2(a[r][col]);
                piv = r;
            }
        if (piv != col)
            for (int j = 0; j < 6; ++j) {
                c64 t = a[col][j];
                a[col][j] = a[piv][j];
                a[piv][j] = t;
                t = inv[col][j];
                inv[col][j] = inv[piv][j];
                inv[piv][j] = t;
            }
        const c64 d = a[col][col];
        const double dn = norm2(d);
        const c64 di{d.re / dn, -d.im / dn};
        for (int j = 0; j < 6; ++j) {
            a[col][j] = a[col][j] * di;
            inv[col][j] = inv[col][j] * di;
        }
        for (int r = 0; r < 6; ++r) {
            if (r == col) continue;
            const c64 f = a[r][col];
            for (int j = 0; j < 6; ++j) {
                a[r][j] -= f * a[col][j];
                inv[r][j] -= f * inv[col][j];
            }
        }
    }
    for (int i = 0; i < 6; ++i) out[i] = inv[i][i].re;
    for (int i = 1; i < 6; ++i)
        for (int j = 0; j < i; ++j) {
            const c64 v = 0.5 * (inv[i][j] + conj(inv[j][i]));
            out[6 + 2 * lw(i, j)] = v.re;
            out[6 + 2 * lw(i, j) + 1] = v.im;
        }
}

// a <- a^{-1} by L D L^dag for definite blocks; false for others (a is then spoilt).  With pivots of one sign
// no entry exceeds the largest of the diagonal and the elimination needs no pivoting; without that, a
// diagonal of 1e-9 beside entries of 0.2 passed a bound on the pivots and cost the inverse nine digits.
__device__ __forceinline__ bool herm6_inverse(Herm6 &a) {
    double amax = 0.0;
#pragma unroll
    for (int i = 0; i < 6; ++i) amax = fmax(amax, fabs(a.d[i]));
    const bool neg = a.d[0] < 0.0;
    double di[6];   // 1 / D
    bool ok = true;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        double dj = a.d[j];
#pragma unroll
        for (int k = 0; k < j; ++k) dj = fma(-norm2(a.l[lw(j, k)]), a.d[k], dj);
        ok &= (neg ? -dj : dj) > 0.02 * amax;   // false for NaN
        a.d[j] = dj;
        di[j] = 1.0 / dj;
        c64 v[6];   // d_k conj(l_jk)
#pragma unroll
        for (int k = 0; k < j; ++k) v[k] = a.d[k] * conj(a.l[lw(j, k)]);
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            c64 s = a.l[lw(i, j)];
#pragma unroll
            for (int k = 0; k < j; ++k) s -= a.l[lw(i, k)] * v[k];
            a.l[lw(i, j)] = di[j] * s;
        }
    }
    // L <- L^{-1} (unit lower triangular), column by column
#pragma unroll
    for (int j = 0; j < 6; ++j)
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            c64 s = -a.l[lw(i, j)];
            // M_ij = -(L_ij + sum_{j<k<i} L_ik M_kj): column j is M above row i, the columns k > j are still L
#pragma unroll
            for (int k = j + 1; k < i; ++k) s -= a.l[lw(i, k)] * a.l[lw(k, j)];
            a.l[lw(i, j)] = s;
        }
    // A^{-1} = M^dag D^{-1} M: entries (i, j) = sum_{k >= i} conj(M_ki) M_kj / D_k, M_ii = 1
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        double s = di[i];
#pragma unroll
        for (int k = i + 1; k < 6; ++k) s = fma(norm2(a.l[lw(k, i)]), di[k], s);
        a.d[i] = s;
    }
#pragma unroll
    for (int i = 1; i < 6; ++i)
#pragma unroll
        for (int j = 0; j < i; ++j) {
            c64 s = di[i] * a.l[lw(i, j)];
#pragma unroll
            for (int k = i + 1; k < 6; ++k) s += di[k] * cmul_conj(a.l[lw(k, i)], a.l[lw(k, j)]);
            a.l[lw(i, j)] = s;   // only rows > i of M are read from here on
        }
    return ok;
}


// x 2^n for x of exponent near -n (integer arithmetic; zeros and subnormals give zero)
__device__ __forceinline__ double scale_pow2(double x, int n) {
    const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7FF;
    if (ex == 0 || ex + n <= 0) return 0.0;
    return __hiloint2double(hi + (n << 20), __double2loint(x));
}

// smem [site][2][36] doubles -> fixed-point limbs with exponents, FP64 array and FP32 stencil form of the block's sites
template <int BK_SITES>
__device__ __forceinline__ void store_blocks(const Geom &g, const double *sm, const short *ex, const unsigned char (*loc)[BK_SITES / 2], long s0,
                                             int ns, double *__restrict__ a64, float *__restrict__ a32, int2 *__restrict__ afix,
                                             int *__restrict__ aexp) {
    const int nh = ns / 2;
    // limbs of a block's entries over a power of two above them
    for (int e = threadIdx.x; afix && e < 2 * nh * 72; e += blockDim.x) {
        const int k = e % 72, icb = (e / 72) % nh, p = e / (72 * nh);
        const int l = loc[p][icb], E = ex[l * 2 + k / 36];
        const FX f = to_fx(scale_pow2(sm[l * 73 + k], -E));
        const long o = (long)p * g.Vh + (s0 >> 1) + icb;
        afix[o * 72 + k] = make_int2(f.h, f.l);
        if (k % 36 == 0) aexp[o * 2 + k / 36] = E;
    }
    for (int e = threadIdx.x; e < 2 * nh * 72; e += blockDim.x) {   // [p][cb][2][36]
        const int k = e % 72, icb = (e / 72) % nh, p = e / (72 * nh);
        a64[((long)p * g.Vh + (s0 >> 1) + icb) * 72 + k] = sm[loc[p][icb] * 73 + k];
    }
    // per block 6 (d, d) then 15 (re, re, im, im): 72 floats
    for (int e = threadIdx.x; e < 2 * nh * 72; e += blockDim.x) {   // float2 index
        const int k = e % 72, icb = (e / 72) % nh, p = e / (72 * nh);
        const float v = (float)sm[loc[p][icb] * 73 + k];
        reinterpret_cast<float2 *>(a32)[((long)p * g.Vh + (s0 >> 1) + icb) * 72 + k] = make_float2(v, v);
    }
}

// Coefficients -csw w / 2 of the planes (0,1), (0,2), (0,3), (1,2), (1,3), (2,3).  In the chiral basis
// sigma_{mu nu} restricted to chirality h is a Pauli matrix: planes (0,1) and (2,3): -s3 and +-s3,
// (0,2) and (1,3): s2 and +-s2, (0,3) and (1,2): +-s1 and -s1 (upper sign h = 0), so
//   A_h = diag + s1 x G1 + s2 x G2 + s3 x G3 with three Hermitian colour matrices.
template <int BK_SITES>
__global__ void __launch_bounds__(2 * BK_SITES) blocks_kernel(Geom g, const double *__restrict__ F, double diag,
                                                              double cs, double ct,
                                                              double *__restrict__ clov64, double *__restrict__ cinv64,
                                                              float *__restrict__ C32wA, float *__restrict__ C32w,
                                                              int2 *__restrict__ clovfix, int2 *__restrict__ cinvfix,
                                                              int *__restrict__ clovexp, int *__restrict__ cinvexp,
                                                              int *general) {
    __shared__ double sm[BK_SITES * 73];
    __shared__ short ex[BK_SITES * 2];     // every entry of the block is below 2^ex
    __shared__ unsigned char loc[2][BK_SITES / 2];
    const long s0 = (long)blockIdx.x * BK_SITES;
    const int ns = (int)min((long)BK_SITES, g.V - s0);
    const int is = threadIdx.x % BK_SITES, h = threadIdx.x / BK_SITES;
    if (is < ns / 2) {
        int c[4];
        cb_coords(g, h, (s0 >> 1) + is, c);
        loc[h][is] = (unsigned char)(2 * is + (c[0] & 1));
    }
    Herm6 a;
    bool ok = true;
    if (is < ns) {
        const double *f = F + s0 + is;
        const double sg = h ? -1.0 : 1.0;
        // G1 = +-c03 F03 - c12 F12, G2 = c02 F02 +- c13 F13, G3 = -c01 F01 +- c23 F23
        auto comb = [&](int pa, double ca, int pb, double cb, double *G) {
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const double *a = f + (long)(2 * pa * 9 + k) * g.V, *b = f + (long)(2 * pb * 9 + k) * g.V;
                G[k] = fma(cb, __ldg(b) + __ldg(b + 9 * g.V), ca * (__ldg(a) + __ldg(a + 9 * g.V)));
            }
        };
        double G1[9], G2[9], G3[9];
        comb(2, sg * ct, 3, -cs, G1);
        comb(1, cs, 4, sg * ct, G2);
        comb(0, -cs, 5, sg * ct, G3);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            a.d[i] = diag + G3[i];
            a.d[3 + i] = diag - G3[i];
        }
        int k = 3;
#pragma unroll
        for (int i = 1; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < i; ++j, k += 2) {
                a.l[lw(i, j)] = c64{G3[k], G3[k + 1]};
                a.l[lw(3 + i, 3 + j)] = c64{-G3[k], -G3[k + 1]};
                // G1 + i G2 at (i, j) and (j, i)
                a.l[lw(3 + i, j)] = c64{G1[k] - G2[k + 1], G1[k + 1] + G2[k]};
                a.l[lw(3 + j, i)] = c64{G1[k] + G2[k + 1], G2[k] - G1[k + 1]};
            }
#pragma unroll
        for (int i = 0; i < 3; ++i) a.l[lw(3 + i, i)] = c64{G1[i], G2[i]};
    }
    double *o = sm + is * 73 + h * 36;
    auto put = [&] {
#pragma unroll
        for (int i = 0; i < 6; ++i) o[i] = a.d[i];
#pragma unroll
        for (int i = 0; i < 15; ++i) {
            o[6 + 2 * i] = a.l[i].re;
            o[6 + 2 * i + 1] = a.l[i].im;
        }
        uint32_t m = 0;
#pragma unroll 4
        for (int i = 0; i < 36; ++i) m = max(m, (uint32_t)__double2hiint(o[i]) & 0x7FFFFFFFu);
        // limbs hold neither a block with NaN or infinities (a singular block's inverse, a mass that is not finite)
        // nor one at the lower end of the FP64 range
        if ((m >> 20) == 0x7FF || (m != 0 && (m >> 20) < 100)) *general = 1;
        ex[is * 2 + h] = (short)max((int)(m >> 20) - 1022, -958);
    };
    if (is < ns) put();
    __syncthreads();
    store_blocks<BK_SITES>(g, sm, ex, loc, s0, ns, clov64, C32wA, clovfix, clovexp);
    if (is < ns) ok = herm6_inverse(a);
    double piv[36];
    if (!ok) herm6_inverse_pivoted(o, piv);
    __syncthreads();
    if (is < ns) {
        if (!ok) {
            for (int i = 0; i < 6; ++i) a.d[i] = piv[i];
            for (int i = 0; i < 15; ++i) a.l[i] = c64{piv[6 + 2 * i], piv[7 + 2 * i]};
        }
        put();
    }
    __syncthreads();
    store_blocks<BK_SITES>(g, sm, ex, loc, s0, ns, cinv64, C32w, cinvfix, cinvexp);
}

// ------------------------------------------------------------------ general links (FP64)
__global__ void __launch_bounds__(64) field_general_kernel(Geom g, const c64 *__restrict__ U, int *flag, double *__restrict__ F) {
    if (!*flag) return;
    for (long s = (long)blockIdx.x * 64 + threadIdx.x; s < g.V; s += 64l * gridDim.x) {
        const int pl = blockIdx.y;
        const int mu = pl < 3 ? 0 : pl < 5 ? 1 : 2, nu = pl < 3 ? pl + 1 : pl < 5 ? pl - 1 : 3;
        int c[4];
        site_coords(g, s, c);
        const int dims[4] = {g.ns, g.ns, g.ns, g.nt};
        auto sh = [&](const int *cc, int d, int step, int *o) {
            o[0] = cc[0];
            o[1] = cc[1];
            o[2] = cc[2];
            o[3] = cc[3];
            o[d] = (cc[d] + step + dims[d]) % dims[d];
        };
        auto link = [&](const int *cc, int d) { return m3_load(U + (site_of(g, cc) * 4 + d) * 9); };
        int xpm[4], xpn[4], xmm[4], xmn[4], xmm_pn[4], xmm_mn[4], xmn_pm[4];
        sh(c, mu, 1, xpm);
        sh(c, nu, 1, xpn);
        sh(c, mu, -1, xmm);
        sh(c, nu, -1, xmn);
        sh(xmm, nu, 1, xmm_pn);
        sh(xmm, nu, -1, xmm_mn);
        sh(xmn, mu, 1, xmn_pm);
        M3 umu = link(c, mu), unu = link(c, nu);
        // leaf 1: U_mu(x) U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
        M3 q = m3_mul_nd(m3_mul_nd(m3_mul(umu, link(xpm, nu)), link(xpn, mu)), unu);
        // leaf 2: U_nu(x) U_mu(x-mu+nu)^dag U_nu(x-mu)^dag U_mu(x-mu)
        M3 umu_m = link(xmm, mu);
        m3_add(q, m3_mul(m3_mul_nd(m3_mul_nd(unu, link(xmm_pn, mu)), link(xmm, nu)), umu_m));
        // leaf 3: U_mu(x-mu)^dag U_nu(x-mu-nu)^dag U_mu(x-mu-nu) U_nu(x-nu)
        M3 unu_n = link(xmn, nu);
        m3_add(q, m3_mul(m3_mul_dn(m3_mul(link(xmm_mn, nu), umu_m), link(xmm_mn, mu)), unu_n));
        // leaf 4: U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu) U_mu(x)^dag
        m3_add(q, m3_mul_nd(m3_mul(m3_mul_dn(unu_n, link(xmn, mu)), link(xmn_pm, nu)), umu));
        // F = (Q - Q^dag)/(8i), traceless
        double d[3];
        for (int i = 0; i < 3; ++i) d[i] = 2.0 * q.m[i][i].im / 8.0;
        const double tr = (d[0] + d[1] + d[2]) / 3.0;
        double *o = F + (long)pl * 18 * g.V + s;   // all of it as pair 0
        for (int k = 9; k < 18; ++k) o[k * g.V] = 0.0;
        for (int i = 0; i < 3; ++i) o[i * g.V] = d[i] - tr;
        int k = 3;
        for (int i = 1; i < 3; ++i)
            for (int j = 0; j < i; ++j) {
                const c64 w = q.m[i][j] - conj(q.m[j][i]);
                o[k++ * g.V] = w.im / 8.0;
                o[k++ * g.V] = -w.re / 8.0;
            }
    }
}

}  // namespace

// On 24^3 x 32 3.6 ms in all, for a call of laph_dslash_eo of 4.2 ms; FP64 in one kernel with the blocks
// in local memory, and four more to convert layouts, took 15.1 of 15.7 ms.
DiracOp prepare_dirac(laph_ctx *ctx, const Geom &g, const c64 *links, double m0, double csw, double xi, cudaStream_t s) {
    LAPH_REQUIRE(xi > 0.0, "xi must be positive");
    LAPH_REQUIRE(g.V < (1L << 30), "lattice too large for 32-bit site indices");
    DiracOp op;
    op.g = g;
    op.m0 = m0;
    op.csw = csw;
    op.xi = xi;
    const double w[4] = {1.0 / xi, 1.0 / xi, 1.0 / xi, 1.0};
    for (int mu = 0; mu < 4; ++mu) op.hw[mu] = -0.5 * w[mu];
    op.L64 = (c64 *)ws_get(ctx, "dirac:L64", sizeof(c64) * 9 * 8 * g.Vh);
    op.L32w = (float4 *)ws_get(ctx, "dirac:L32w", sizeof(float4) * 9 * 8 * g.Vh);
    op.clov64 = (double *)ws_get(ctx, "dirac:clov64", sizeof(double) * CLOV_BLOCK * 4 * g.Vh);
    op.cinv64 = (double *)ws_get(ctx, "dirac:cinv64", sizeof(double) * CLOV_BLOCK * 4 * g.Vh);
    op.C32w = (float *)ws_get(ctx, "dirac:C32w", sizeof(float) * 144 * 2 * g.Vh);
    op.C32wA = (float *)ws_get(ctx, "dirac:C32wA", sizeof(float) * 144 * 2 * g.Vh);
    op.Lfix = (int4 *)ws_spare(ctx, "dirac:limbs", (sizeof(int4) * 9 * 8 + 2 * sizeof(int2) * CLOV_BLOCK * 4) * g.Vh);
    op.clovfix = op.Lfix ? (int2 *)(op.Lfix + 9 * 8 * g.Vh) : nullptr;
    op.cinvfix = op.Lfix ? op.clovfix + CLOV_BLOCK * 4 * g.Vh : nullptr;
    op.clovexp = (int *)ws_get(ctx, "dirac:clovexp", sizeof(int) * 4 * g.Vh);
    op.cinvexp = (int *)ws_get(ctx, "dirac:cinvexp", sizeof(int) * 4 * g.Vh);
    op.ctx = ctx;
    int4 *fix = (int4 *)op.C32w;   // the site limbs, 576 bytes a site as C32w, which blocks_kernel writes behind their last use
    double *F = (double *)ws_get(ctx, "dirac:F", sizeof(double) * 108 * g.V);
    int *flag = (int *)ws_get(ctx, "dirac:flag", 2 * sizeof(int));
    op.general = flag;
    const double diag = m0 + w[0] + w[1] + w[2] + w[3];
    LAPH_CUDA(cudaMemsetAsync(flag, 0, 2 * sizeof(int), s));
    op.weights_bounded = 0.5 * std::max(w[0], w[3]) < 1.0;
    pack_kernel<<<grid_for(g.V, PK_SITES), 256, 0, s>>>(g, links, op.hw[0], op.hw[3], op.L64, op.L32w, op.Lfix, fix, flag);
    LAPH_LAUNCH_CHECK();
    // small lattices: short blocks, so that the work reaches more SMs
    const bool few = g.V < 32 * 2 * 152;
    const int fb = few ? 32 : 128;
    field_kernel<<<dim3(grid_for(g.V, fb), 12), fb, 0, s>>>(g, fix, flag, F);
    LAPH_LAUNCH_CHECK();
    field_general_kernel<<<dim3(grid_for(g.V, 64, 512), 6), 64, 0, s>>>(g, links, flag, F);
    LAPH_LAUNCH_CHECK();
    const double cs = -0.5 * csw / xi, ct = -0.25 * csw * (1.0 + 1.0 / xi);
    if (few)
        blocks_kernel<8><<<grid_for(g.V, 8), 16, 0, s>>>(g, F, diag, cs, ct, op.clov64, op.cinv64, op.C32wA, op.C32w,
                                                            op.clovfix, op.cinvfix, op.clovexp, op.cinvexp, flag);
    else
        blocks_kernel<32><<<grid_for(g.V, 32), 64, 0, s>>>(g, F, diag, cs, ct, op.clov64, op.cinv64, op.C32wA, op.C32w,
                                                              op.clovfix, op.cinvfix, op.clovexp, op.cinvexp, flag);
    LAPH_LAUNCH_CHECK();
    prepare_f32_operands(ctx, op, s);
    return op;
}

}  // namespace laph
