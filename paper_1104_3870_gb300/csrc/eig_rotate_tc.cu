// The restart GEMM of the eigensolver, Out[t][c] = sum_{j < m} V[t][j] Y[t][j][c] for c < k, on the
// exact-slice tensor-core GEMM (exact_gemm.cuh): rows are the entries of the vectors, K the m basis vectors.
// Bound by the FP64 pipe in FP64 (four multiply-adds per term at two per cycle and SM); here by the start and
// drain of short CTAs (m = 80: five sub-chunks) and the partial sums.
// 10^3 x 12, m = 56: about 70 us (1290); N_v = 32 on 16^3 x 32, the whole call, 526 ms (648).
#include "exact_gemm.cuh"

namespace laph {

namespace {

struct RotateOp {
    const c64 *V, *Y;
    const int *EA, *EB;   // [t][n], [t][k]
    long n, ldv;
    int m, k;
    c64 *out;
    struct Item {
        const c64 *p;
        int rbase;
    };
    struct ItemB : Item {};
    struct RawA {
        double2 v[4];
    };
    struct RawB : RawA {};
    __device__ int rows() const { return (int)n; }
    __device__ int cols() const { return k; }
    __device__ int expA(int t, int r) const { return EA[(long)t * n + r]; }
    __device__ int expB(int t, int c) const { return EB[(long)t * k + c]; }
    __device__ Item itemA(int t, int r) const {
        if (r >= n) return {nullptr, 1022};
        return {V + (long)t * ldv * n + r, 1022 + expA(t, r)};
    }
    __device__ ItemB itemB(int t, int c) const {
        ItemB i;
        i.p = c < k ? Y + (long)t * m * m + c : nullptr;
        i.rbase = c < k ? 1022 + expB(t, c) : 1022;
        return i;
    }
    __device__ void load(const Item &it, long k0, RawA &r) const {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            r.v[j] = (it.p && k0 + 4 * j < m) ? __ldg(reinterpret_cast<const double2 *>(it.p) + (k0 + 4 * j) * n)
                                              : make_double2(0., 0.);
    }
    __device__ void load(const ItemB &it, long k0, RawB &r) const {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            r.v[j] = (it.p && k0 + 4 * j < m) ? __ldg(reinterpret_cast<const double2 *>(it.p) + (k0 + 4 * j) * m)
                                              : make_double2(0., 0.);
    }
    // the GEMM conjugates A
    __device__ c64 value(const Item &, const RawA &r, int j) const { return {r.v[j].x, -r.v[j].y}; }
    __device__ c64 value(const ItemB &, const RawB &r, int j) const { return {r.v[j].x, r.v[j].y}; }
    __device__ c64 direct(int t, int r, int c) const {
        c64 s{0, 0};
        for (int j = 0; j < m; ++j) s += V[((long)t * ldv + j) * n + r] * Y[((long)t * m + j) * m + c];
        return s;
    }
    __device__ void store(int t, int r, int c, c64 v) const { out[((long)t * k + c) * n + r] = v; }
};

// E[t][r] of the entries x[t * tstride + j * jstride + r], j < m, for r < rows
__global__ void __launch_bounds__(128) strided_exp_kernel(long rows, int m, long jstride, long tstride, const c64 *__restrict__ x,
                                                          int *__restrict__ E) {
    const long r = (long)blockIdx.x * 128 + threadIdx.x;
    if (r >= rows) return;
    const double2 *p = reinterpret_cast<const double2 *>(x) + blockIdx.y * tstride + r;
    uint32_t h = 0;
#pragma unroll 8
    for (int j = 0; j < m; ++j) h = max(h, xg::hi_abs(__ldg(p + j * jstride)));
    E[blockIdx.y * rows + r] = xg::exp_of_hi(h);
}

}  // namespace

void rotate_tc(laph_ctx *ctx, long n, int nt, int ldv, int m, int k, const c64 *V, const c64 *Y, c64 *out, cudaStream_t s) {
    int *EA = (int *)ws_get(ctx, "eig:expV", sizeof(int) * nt * (size_t)n);
    int *EB = (int *)ws_get(ctx, "eig:expY", sizeof(int) * nt * (size_t)k);
    strided_exp_kernel<<<dim3(grid_for(n, 128), nt), 128, 0, s>>>(n, m, n, (long)ldv * n, V, EA);
    LAPH_LAUNCH_CHECK();
    strided_exp_kernel<<<dim3(grid_for(k, 128), nt), 128, 0, s>>>(k, m, m, (long)m * m, Y, EB);
    LAPH_LAUNCH_CHECK();
    RotateOp op{V, Y, EA, EB, n, ldv, m, k, out};
    xg::run(ctx, op, m, nt, (int)n, k, s);
}

}  // namespace laph
