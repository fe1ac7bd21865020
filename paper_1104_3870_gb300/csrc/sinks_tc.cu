// Sink coefficients on the tensor cores (Sec. IV: the quark-propagation coefficients
// V_s^dag x of every slice), FP64-accurate through exact integer slices (exact_gemm.cuh):
//
//   coef[i][t][alpha][n] = sum_{x,c} conj(V[t][n][x][c]) X[i][t][x][alpha][c]
//
// Per slice t this is C = V^H X with K = 3 V3, rows n and columns (i, alpha).  At 24^3 x 128, N_v = 64 and
// 32 solutions: 11.6 ms (8.9 ms of GEMM, 62 % of the tensor pipe, and 2.6 ms to read both operands for
// their exponents), 184 ms with one CTA of four warps per 128 x 32 tile and 6-bit digits; its error
// against a 64-bit sum fell from 2.6e-14 to 2.3e-15.  6^3 x 12, N_v = 10, 5 solutions: 50 us (500 us).
#include "exact_gemm.cuh"

namespace laph {

namespace xg {

int *host_flag(laph_ctx *ctx) {
    if (!ctx->xg_flag) {
        LAPH_CUDA(cudaHostAlloc(&ctx->xg_flag, sizeof(int), cudaHostAllocMapped | cudaHostAllocPortable));
        *ctx->xg_flag = 0;
    }
    return ctx->xg_flag;   // host memory is addressed by the same pointer on the device
}

void check_host_flag(laph_ctx *ctx) {
    if (ctx->xg_flag && *(volatile int *)ctx->xg_flag) {
        *ctx->xg_flag = 0;
        throw Error(LAPH_ERR_TIMEOUT, "a tensor-core GEMM wait gave up (device wait cap)");
    }
}

}  // namespace xg

namespace {

struct SinkOp {
    const c64 *V, *X;
    const int *Erow, *Ecol;   // [nt][nv], [nrhs][nt][4]
    int nv, nrhs, nt;
    long K;                   // 3 V3
    c64 *coef;
    struct Item {
        const c64 *p;   // null for a row or column outside the problem
        int rbase;
    };
    struct Raw {
        double2 v[4];
    };
    using RawA = Raw;
    struct RawB : Raw {};
    struct ItemB : Item {};
    __device__ int rows() const { return nv; }
    __device__ int cols() const { return 4 * nrhs; }
    __device__ int expA(int t, int n) const { return Erow[t * nv + n]; }
    __device__ int expB(int t, int c) const { return Ecol[((long)(c >> 2) * nt + t) * 4 + (c & 3)]; }
    __device__ Item itemA(int t, int n) const {
        if (n >= nv) return {nullptr, 1022};
        return {V + ((long)t * nv + n) * K, 1022 + expA(t, n)};
    }
    __device__ ItemB itemB(int t, int c) const {
        ItemB r;
        r.p = c < 4 * nrhs ? X + ((long)(c >> 2) * nt + t) * K * 4 + (c & 3) * 3 : nullptr;
        r.rbase = c < 4 * nrhs ? 1022 + expB(t, c) : 1022;
        return r;
    }
    __device__ void load(const Item &it, long k0, RawA &r) const {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            r.v[j] = (it.p && k0 + 4 * j < K) ? __ldg(reinterpret_cast<const double2 *>(it.p) + k0 + 4 * j)
                                              : make_double2(0., 0.);
    }
    __device__ void load(const ItemB &it, long k0, RawB &r) const {
        const int x0 = (int)((unsigned)k0 / 3u);
        int c = (int)k0 - 3 * x0;
        long o = k0 + 9l * x0;   // x 12 + c
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            r.v[j] = (it.p && k0 + 4 * j < K) ? __ldg(reinterpret_cast<const double2 *>(it.p) + o) : make_double2(0., 0.);
            o += 13;   // k + 4: the next site's next colour
            if (++c == 3) {
                c = 0;
                o += 9;
            }
        }
    }
    __device__ c64 value(const Item &, const Raw &r, int j) const { return {r.v[j].x, r.v[j].y}; }
    // a non-finite input row or column gives a non-finite coefficient
    __device__ c64 direct(int t, int n, int c) const {
        if (expA(t, n) >= xg::NONFINITE || expB(t, c) >= xg::NONFINITE) {
            const double q = __longlong_as_double(0x7FF8000000000000ll);
            return {q, q};
        }
        const c64 *a = itemA(t, n).p, *b = itemB(t, c).p;
        c64 s{0, 0};
        for (long k = 0; k < K; ++k) s += conj(a[k]) * b[k + 9 * (k / 3)];   // x 12 + c
        return s;
    }
    __device__ void store(int t, int n, int c, c64 v) const { coef[(((long)(c >> 2) * nt + t) * 4 + (c & 3)) * nv + n] = v; }
};

// Ecol[i][t][alpha] over X[i][t][x][alpha][c], one block of 192 threads per (i, t): a thread's
// elements all belong to one alpha (192 is a multiple of 12), and only the high words are compared
// (the FP64 pipe, at 2 operations per cycle and SM, held the FP64 comparison to 2.1 TB/s).
__global__ void __launch_bounds__(192) col_exp_kernel(const c64 *__restrict__ X, long V3, int nt, int *Ecol) {
    __shared__ uint32_t sm[4];
    const int i = blockIdx.x, t = blockIdx.y;
    const double2 *x = reinterpret_cast<const double2 *>(X) + ((long)i * nt + t) * V3 * 12;
    const long len = V3 * 12;
    if (threadIdx.x < 4) sm[threadIdx.x] = 0;
    __syncthreads();
    uint32_t m = 0;
    long e = threadIdx.x;
    for (; e + 7 * 192 < len; e += 8 * 192) {
        double2 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = __ldg(x + e + q * 192);
#pragma unroll
        for (int q = 0; q < 8; ++q) m = max(m, xg::hi_abs(v[q]));
    }
    for (; e < len; e += 192) m = max(m, xg::hi_abs(__ldg(x + e)));
    atomicMax(&sm[(threadIdx.x % 12) / 3], m);
    __syncthreads();
    if (threadIdx.x < 4) Ecol[((long)i * nt + t) * 4 + threadIdx.x] = xg::exp_of_hi(sm[threadIdx.x]);
}

}  // namespace

// coef[i][t][alpha][n] for nrhs solutions (device arrays; layouts as laph_sinks).
void sinks_tensor_core(laph_ctx *ctx, const Geom &g, const c64 *V, int nv, const c64 *X, int nrhs, c64 *coef,
                       cudaStream_t s) {
    const long K = 3 * g.V3;
    LAPH_REQUIRE(K < (1L << 30), "slice too large");
    int *Erow = (int *)ws_get(ctx, "sinks_tc:erow", sizeof(int) * g.nt * (size_t)nv);
    int *Ecol = (int *)ws_get(ctx, "sinks_tc:ecol", sizeof(int) * 4 * g.nt * (size_t)nrhs);
    prof_begin("sinks", s);
    xg::rows_exp(V, (long)g.nt * nv, K, Erow, s);
    col_exp_kernel<<<dim3(nrhs, g.nt), 192, 0, s>>>(X, g.V3, g.nt, Ecol);
    LAPH_LAUNCH_CHECK();
    SinkOp op;
    op.V = V;
    op.X = X;
    op.Erow = Erow;
    op.Ecol = Ecol;
    op.nv = nv;
    op.nrhs = nrhs;
    op.nt = g.nt;
    op.K = K;
    op.coef = coef;
    xg::run(ctx, op, K, g.nt, nv, 4 * nrhs, s);
    // algorithmic bytes: solutions and eigenvectors once, the coefficients written; flops: the digit-plane
    // products the tensor cores execute, padding included
    const double tiles = (double)g.nt * ((nv + xg::TN - 1) / xg::TN) * ((4 * nrhs + xg::TN - 1) / xg::TN);
    prof_end("sinks", s, 16.0 * (double)g.V * 12 * nrhs + 16.0 * (double)g.nt * nv * K + 16.0 * (double)nrhs * g.nt * 4 * nv,
             40.0 * 2.0 * 128.0 * 64.0 * 2.0 * (double)K * tiles);
}

}  // namespace laph
