// LapH-space contractions on the tensor cores (exact_gemm.cuh): momentum / displaced overlaps and
// meson functions.  Both are small-batch complex GEMMs that the FP64 pipe of this GPU (two FMA per
// cycle and SM) bounded.  Four momenta at N_v = 32 on 16^3 x 32: 0.91 ms (21.9 ms in FP64); the four
// meson functions of 32 x 32 projectors of a pi pi correlator at N_v = 64 on 128 slices, one GEMM with
// the sources as one more slice: 47 us (8 x 256 us).
#include "exact_gemm.cuh"
#include "gamma_host.cuh"

namespace laph {

namespace {

// Phi[p][t][n][m] = scale sum_k conj(A[t][n][k]) ph[p][k / 3] B[t][m][k]: rows n, columns (p, m), batch t.
// The phase is multiplied in FP64 before the digits are cut; a part of ph b is below sqrt 2 max|part of b|,
// so the column's exponent is B's plus one.
struct OverlapOp {
    const c64 *A, *B, *ph;
    const int *EA, *EB;   // [nt][nv]
    int nv, nt, nmom;
    long K, V3;
    c64 scale;
    c64 *phi;
    struct ItemA {
        const c64 *p;
        int rbase;
    };
    struct ItemB {
        const c64 *p, *f;
        int rbase;
    };
    struct RawA {
        double2 v[4];
    };
    struct RawB {
        double2 v[4], f[4];
    };
    __device__ int rows() const { return nv; }
    __device__ int cols() const { return nmom * nv; }
    __device__ int expA(int t, int n) const { return EA[t * nv + n]; }
    __device__ int expB(int t, int c) const { return EB[t * nv + c % nv] + 1; }
    __device__ ItemA itemA(int t, int n) const {
        if (n >= nv) return {nullptr, 1022};
        return {A + ((long)t * nv + n) * K, 1022 + expA(t, n)};
    }
    __device__ ItemB itemB(int t, int c) const {
        if (c >= cols()) return {nullptr, nullptr, 1022};
        return {B + ((long)t * nv + c % nv) * K, ph + (long)(c / nv) * V3, 1022 + expB(t, c)};
    }
    __device__ void load(const ItemA &it, long k0, RawA &r) const {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            r.v[j] = (it.p && k0 + 4 * j < K) ? __ldg(reinterpret_cast<const double2 *>(it.p) + k0 + 4 * j)
                                              : make_double2(0., 0.);
    }
    __device__ void load(const ItemB &it, long k0, RawB &r) const {
        int x = (int)((unsigned)k0 / 3u), c = (int)k0 - 3 * x;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool in = it.p && k0 + 4 * j < K;
            r.v[j] = in ? __ldg(reinterpret_cast<const double2 *>(it.p) + k0 + 4 * j) : make_double2(0., 0.);
            r.f[j] = in ? __ldg(reinterpret_cast<const double2 *>(it.f) + x) : make_double2(0., 0.);
            ++x;   // k + 4: the next site's next colour
            if (++c == 3) {
                c = 0;
                ++x;
            }
        }
    }
    __device__ c64 value(const ItemA &, const RawA &r, int j) const { return {r.v[j].x, r.v[j].y}; }
    __device__ c64 value(const ItemB &, const RawB &r, int j) const {
        return c64{r.f[j].x, r.f[j].y} * c64{r.v[j].x, r.v[j].y};
    }
    __device__ c64 direct(int t, int n, int c) const {
        const c64 *a = A + ((long)t * nv + n) * K, *b = B + ((long)t * nv + c % nv) * K, *f = ph + (long)(c / nv) * V3;
        c64 s{0, 0};
        for (long k = 0; k < K; ++k) s += conj(a[k]) * (f[k / 3] * b[k]);
        return s;
    }
    __device__ void store(int t, int n, int c, c64 v) const {
        phi[(((long)(c / nv) * nt + t) * nv + n) * nv + c % nv] = scale * v;
    }
};

// M[z][r][c] = sum_{al be n} conj(a_r(z, al, n)) W[al][be] b_c(z, be, n) over rows r = (line, b1) and
// columns c = (line, b2); z < nt are the slices of the coefficients [nb][nt][4][nv], z = nt the
// source operands [nb][4][nv].  W has one unit entry (a power of i) per column be, so row r of A is
// a_r(perm[be], n) times the conjugate of that entry.
struct MesonOp {
    const c64 *a[2], *b[2], *ra[2], *rb[2];
    const int *E;   // per array (a0, a1, b0, b1: [nb][nt]; then ra, rb: [nb] each)
    int nl, nb, nt, nv;
    int perm[4], code[4];   // column be: row perm[be], conj(W) = i^code[be]
    c64 *M;
    struct Item {
        const c64 *p;
        int rbase;
    };
    struct ItemB : Item {};
    struct RawA {
        double2 v[4];
        int pc;
    };
    struct RawB {
        double2 v[4];
    };
    __device__ int rows() const { return nl * nb; }
    __device__ int cols() const { return nl * nb; }
    __device__ int exp_at(int side, int z, int r) const {
        const int l = r / nb, i = r % nb, arr = 2 * side + l;
        return z < nt ? E[((long)arr * nb + i) * nt + z] : E[(long)4 * nb * nt + arr * nb + i];
    }
    __device__ const c64 *ptr(int side, int z, int r) const {
        const int l = r / nb, i = r % nb;
        if (z < nt) return (side ? b[l] : a[l]) + ((long)i * nt + z) * 4 * nv;
        return (side ? rb[l] : ra[l]) + (long)i * 4 * nv;
    }
    __device__ int expA(int z, int n) const { return exp_at(0, z, n); }
    __device__ int expB(int z, int c) const { return exp_at(1, z, c); }
    __device__ Item itemA(int z, int n) const {
        if (n >= rows()) return {nullptr, 1022};
        return {ptr(0, z, n), 1022 + expA(z, n)};
    }
    __device__ ItemB itemB(int z, int c) const {
        ItemB r;
        r.p = c < cols() ? ptr(1, z, c) : nullptr;
        r.rbase = c < cols() ? 1022 + expB(z, c) : 1022;
        return r;
    }
    __device__ void load(const Item &it, long k0, RawA &r) const {
        int be = (int)k0 / nv, n = (int)k0 - be * nv;
        r.pc = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool in = it.p && be < 4;
            const int q = be < 4 ? be : 0;
            r.v[j] = in ? __ldg(reinterpret_cast<const double2 *>(it.p) + perm[q] * nv + n) : make_double2(0., 0.);
            r.pc |= code[q] << (2 * j);
            for (n += 4; n >= nv && be < 4; n -= nv) ++be;
        }
    }
    __device__ void load(const ItemB &it, long k0, RawB &r) const {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            r.v[j] = (it.p && k0 + 4 * j < 4 * nv) ? __ldg(reinterpret_cast<const double2 *>(it.p) + k0 + 4 * j)
                                                   : make_double2(0., 0.);
    }
    __device__ static c64 turn(int code, c64 v) {
        return code == 0 ? v : code == 1 ? times_i(v) : code == 2 ? -v : c64{v.im, -v.re};
    }
    __device__ c64 value(const Item &, const RawA &r, int j) const {
        return turn((r.pc >> (2 * j)) & 3, c64{r.v[j].x, r.v[j].y});
    }
    __device__ c64 value(const ItemB &, const RawB &r, int j) const { return {r.v[j].x, r.v[j].y}; }
    __device__ c64 direct(int z, int n, int c) const {
        const c64 *pa = ptr(0, z, n), *pb = ptr(1, z, c);
        c64 s{0, 0};
        for (int be = 0; be < 4; ++be)
            for (int m = 0; m < nv; ++m) s += conj(turn(code[be], pa[perm[be] * nv + m])) * pb[be * nv + m];
        return s;
    }
    __device__ void store(int z, int n, int c, c64 v) const { M[((long)z * rows() + n) * cols() + c] = v; }
};

struct RowSets {
    const c64 *p[8];
    int rows[8];
    int *E[8];
};
// E of the rows of up to eight arrays, a warp per row, blockIdx.y the array
__global__ void __launch_bounds__(256) row_sets_exp_kernel(const RowSets rs, int len) {
    const long row = (long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= rs.rows[blockIdx.y]) return;
    const double2 *p = reinterpret_cast<const double2 *>(rs.p[blockIdx.y]) + row * len;
    uint32_t m = 0;
    for (int k = threadIdx.x & 31; k < len; k += 32) m = max(m, xg::hi_abs(__ldg(p + k)));
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) rs.E[blockIdx.y][row] = xg::exp_of_hi(m);
}

}  // namespace

void overlaps_tc(laph_ctx *ctx, const Geom &g, int nv, int nmom, const c64 *A, const c64 *B, const c64 *ph, c64 scale,
                 c64 *phi, cudaStream_t s) {
    const long K = 3 * g.V3, rows = (long)g.nt * nv;
    LAPH_REQUIRE(K < (1L << 30) && (long)nmom * nv < (1L << 30), "overlap problem too large");
    int *E = (int *)ws_get(ctx, "ov:exp", sizeof(int) * 2 * rows);
    xg::rows_exp(A, rows, K, E, s);
    if (B != A) xg::rows_exp(B, rows, K, E + rows, s);
    OverlapOp op;
    op.A = A;
    op.B = B;
    op.ph = ph;
    op.EA = E;
    op.EB = B == A ? E : E + rows;
    op.nv = nv;
    op.nt = g.nt;
    op.nmom = nmom;
    op.K = K;
    op.V3 = g.V3;
    op.scale = scale;
    op.phi = phi;
    xg::run(ctx, op, K, g.nt, nv, nmom * nv, s);
}

void meson_fns_tc(laph_ctx *ctx, int nt, int nv, int nb, const MesonLines &ln, const Mat4 &W, bool new_lines, c64 *M,
                  cudaStream_t s) {
    MesonOp op;
    op.nl = ln.nl;
    op.nb = nb;
    op.nt = nt;
    op.nv = nv;
    op.M = M;
    for (int be = 0; be < 4; ++be) {
        int found = 0;
        for (int al = 0; al < 4; ++al) {
            const c64 w = W.m[al][be];
            if (w.re == 0.0 && w.im == 0.0) continue;
            ++found;
            op.perm[be] = al;
            op.code[be] = w.re == 1.0 ? 0 : w.im == -1.0 ? 1 : w.re == -1.0 ? 2 : 3;   // conj(w) = i^code
            LAPH_REQUIRE(norm2(w) == 1.0, "the spin weight of a meson function is a product of Dirac matrices");
        }
        LAPH_REQUIRE(found == 1, "the spin weight of a meson function is a product of Dirac matrices");
    }
    int *E = (int *)ws_get(ctx, "mfn:exp", sizeof(int) * 4 * (size_t)nb * (nt + 1));
    op.E = E;
    RowSets rs{};
    int sets = 0;
    for (int side = 0; side < 2; ++side)
        for (int l = 0; l < 2; ++l) {
            const int use = l < ln.nl ? l : 0;
            (side ? op.b : op.a)[l] = side ? ln.b[use] : ln.a[use];
            (side ? op.rb : op.ra)[l] = side ? ln.rb[use] : ln.ra[use];
            if (l >= ln.nl) continue;
            const int arr = 2 * side + l;
            rs.p[sets] = side ? ln.b[l] : ln.a[l];
            rs.rows[sets] = nb * nt;
            rs.E[sets++] = E + (size_t)arr * nb * nt;
            rs.p[sets] = side ? ln.rb[l] : ln.ra[l];
            rs.rows[sets] = nb;
            rs.E[sets++] = E + (size_t)4 * nb * nt + arr * nb;
        }
    if (new_lines) {
        row_sets_exp_kernel<<<dim3((unsigned)((nb * nt + 7) / 8), (unsigned)sets), 256, 0, s>>>(rs, 4 * nv);
        LAPH_LAUNCH_CHECK();
    }
    xg::run(ctx, op, 4L * nv, nt + 1, ln.nl * nb, ln.nl * nb, s);
}

}  // namespace laph
