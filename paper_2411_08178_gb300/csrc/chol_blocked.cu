// Float64 Cholesky factorisation of the ell x ell matrices of Algorithm 1 (the
// shifted core, steps 4-5) and of the preconditioner set-up (I + Ubar^T Ubar),
// and the inverse of the triangular factor.
//
// GB300's float64 pipe issues about two FMAs per clock per SM, so the work is
// spread over all SMs in panels of 32 columns, two launches a panel: every
// CTA of chol_panel factors the 32 x 32 diagonal block for itself (one warp, a
// row per lane, no square root on the dependent chain) and solves
// for 32 rows of the panel; chol_update subtracts the panel's product from the
// trailing matrix, one CTA per 16 x 16 tile.  A 16-CTA cluster kernel
// (chol_cluster.cu) factored n = 400 in 1.00 ms, most of it latency (31 us a
// 13-column panel); this takes 0.47 ms.  n = 200: 0.38 ms there, 0.25 ms here.
#include "internal.cuh"

namespace nys {
namespace {

constexpr int PB = 32;

// A = sym(Omega^T Y) + v Omega^T Omega (lower triangle) from the Gram G2 of
// [Omega | Y] (ld 2n), v = eps sqrt(trace Omega^T Omega); info = {0, v, 0}
__global__ void __launch_bounds__(256) core_form_kernel(const double* __restrict__ G2, int n, double eps,
                                                        double* __restrict__ A, double* __restrict__ info) {
    pdl_enter();
    __shared__ double sh[32];
    const int ld = 2 * n;
    double tr = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) tr += G2[(size_t)i * ld + i];
    const double v = eps * sqrt(block_sum(tr, sh));
    if (blockIdx.x == 0 && threadIdx.x == 0) info[0] = 0.0, info[1] = v, info[2] = 0.0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n * n; t += gridDim.x * blockDim.x) {
        const int i = t / n, j = t - i * n;
        if (j > i) continue;
        const double oy = 0.5 * (G2[(size_t)i * ld + n + j] + G2[(size_t)j * ld + n + i]);
        A[t] = oy + v * G2[(size_t)i * ld + j];
    }
}

// panel of columns p0 .. p0 + 31: CTA b eliminates the diagonal block (a row per
// lane) and, for b > 0, the 32 rows p0 + 32 b .. with it.  A float64 operation
// of one warp takes its scheduler 64 cycles, so the columns are dealt to four
// warps (column j to warp j mod 4); the owner of the next column updates it
// first and publishes it with the reciprocal of its pivot while the others
// finish the step (51 us a panel with one warp, 30 us so).  The lower triangle
// of A is read, L's panel written (block 0: the diagonal block, zeros above it).
// info[slot] = 1 on a pivot that is not positive and finite.
__global__ void __launch_bounds__(128) chol_panel_kernel(const double* __restrict__ A, double* __restrict__ L, int n,
                                                         int p0, double* __restrict__ info, int slot) {
    pdl_enter();
    __shared__ double sd[PB][PB + 1], sp[PB][PB + 1];     // diagonal block, this CTA's rows
    __shared__ double cd[2][PB], cp[2][PB];               // the published column
    __shared__ double piv[PB], inv[PB];
    if (p0 > 0 && info[slot] != 0.0) return;              // an earlier panel failed
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nb = min(PB, n - p0);
    const int i0 = p0 + PB * blockIdx.x, rows = blockIdx.x ? min(PB, n - i0) : 0;
    for (int r = w; r < PB; r += 4) {
        sd[r][lane] = (r < nb && lane <= r) ? A[(size_t)(p0 + r) * n + p0 + lane] : (r == lane ? 1.0 : 0.0);
        sp[r][lane] = r < rows ? A[(size_t)(i0 + r) * n + p0 + lane] : 0.0;    // rows below: nb = 32
    }
    __syncthreads();
    // L D L^T: column k stays l_ik d_k (a row per lane, diagonal block and rows below)
    double ad[8], ap[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) ad[c] = sd[lane][4 * c + w], ap[c] = sp[lane][4 * c + w];
    auto publish = [&](int k, double d, double p) {
        cd[k & 1][lane] = d;
        cp[k & 1][lane] = p;
        const double pk = __shfl_sync(0xffffffffu, d, k), ik = 1.0 / pk;
        if (lane == 0) piv[k] = pk, inv[k] = ik;
    };
    if (w == 0) publish(0, ad[0], ap[0]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PB - 1; ++k) {
        const double xd = cd[k & 1][lane], xp = cp[k & 1][lane];
        const double m = xd * inv[k];                     // l_jk of j = lane
        constexpr unsigned ALL = 0xffffffffu;
        if (((k + 1) & 3) == w) {
            const int c = (k + 1) >> 2;
            const double mj = __shfl_sync(ALL, m, k + 1);
            ad[c] = fma(-xd, mj, ad[c]);
            ap[c] = fma(-xp, mj, ap[c]);
            publish(k + 1, ad[c], ap[c]);
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            if (4 * c + 3 <= k + 1) continue;             // no column of this group is left
            const int j = 4 * c + w;
            const double mj = __shfl_sync(ALL, m, j);
            if (j > k + 1) {
                ad[c] = fma(-xd, mj, ad[c]);
                if (rows) ap[c] = fma(-xp, mj, ap[c]);
            }
        }
        __syncthreads();
    }
    const double d = piv[lane], iv = inv[lane];
    if (!__all_sync(0xffffffffu, d > 0.0 && isfinite(d) && iv > 0.0 && isfinite(iv))) {   // the same in every warp and CTA
        if (blockIdx.x == 0 && threadIdx.x == 0) info[slot] = 1.0;
        return;
    }
    const double root = sqrt(d), rs = root * iv;          // L_kk and 1 / L_kk of k = lane
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int j = 4 * c + w;
        const double rj = __shfl_sync(0xffffffffu, rs, j);
        if (rows) sp[lane][j] = ap[c] * rj;
        else sd[lane][j] = lane > j ? ad[c] * rj : (lane == j ? root : 0.0);
    }
    __syncthreads();
    if (rows) {
        for (int r = w; r < rows; r += 4) L[(size_t)(i0 + r) * n + p0 + lane] = sp[r][lane];
        return;
    }
    for (int r = w; r < nb; r += 4) {
        if (lane < nb) L[(size_t)(p0 + r) * n + p0 + lane] = sd[r][lane];
        // zeros to the right of the diagonal block
        for (int j = p0 + nb + lane; j < n; j += 32) L[(size_t)(p0 + r) * n + j] = 0.0;
    }
}

// A_ij -= sum_k L_ik L_jk over the panel's 32 columns, lower triangle from row
// and column p0 + 32 on
__global__ void __launch_bounds__(256) chol_update_kernel(double* __restrict__ A, const double* __restrict__ L, int n,
                                                          int p0, const double* __restrict__ info, int slot) {
    pdl_enter();
    if (blockIdx.x > blockIdx.y || info[slot] != 0.0) return;
    __shared__ double si[16][PB + 1], sj[16][PB + 1];
    const int i0 = p0 + PB + 16 * blockIdx.y, j0 = p0 + PB + 16 * blockIdx.x;
    for (int t = threadIdx.x; t < 16 * PB; t += 256) {
        const int r = t / PB, k = t % PB;
        si[r][k] = i0 + r < n ? L[(size_t)(i0 + r) * n + p0 + k] : 0.0;
        sj[r][k] = j0 + r < n ? L[(size_t)(j0 + r) * n + p0 + k] : 0.0;
    }
    __syncthreads();
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15, i = i0 + ty, j = j0 + tx;
    if (i >= n || j > i) return;
    double s = A[(size_t)i * n + j];
#pragma unroll
    for (int k = 0; k < PB; ++k) s = fma(-si[ty][k], sj[tx][k], s);
    A[(size_t)i * n + j] = s;
}

// X = L^{-1}, row by row: x L = e_r from the diagonal back, one CTA of four
// warps per row r, the row's remaining entries in registers (entry j with
// thread j mod 128); x_k known, row k of L times x_k is subtracted from the
// entries left of k.  The warp that holds entry k - 1 updates it first and
// publishes x_{k-1} while the others finish the step: one product, one
// subtraction and a barrier on the dependent chain.  n = 400: 96 us
// (forward substitution by columns with a warp reduction and a division per
// entry: 581 us; one warp per row: 143 us).
template <int RPL>   // entries per thread, n <= 128 RPL
__global__ void __launch_bounds__(128) tri_inv_kernel(const double* __restrict__ L, double* __restrict__ X, int n) {
    pdl_enter();
    __shared__ double xs[2];
    const int r = n - 1 - blockIdx.x, t = threadIdx.x;      // the longest rows first
    double s[RPL], inv[RPL], row[RPL];
#pragma unroll
    for (int c = 0; c < RPL; ++c) {
        const int j = 128 * c + t;
        s[c] = j == r ? 1.0 : 0.0;
        inv[c] = j <= r ? 1.0 / L[(size_t)j * n + j] : 0.0;
        row[c] = j < r ? L[(size_t)r * n + j] : 0.0;
    }
    // entry k becomes x_k
#pragma unroll
    for (int c = 0; c < RPL; ++c)
        if (128 * c + t == r) xs[r & 1] = s[c] = inv[c];
    __syncthreads();
#pragma unroll
    for (int cb = RPL - 1; cb >= 0; --cb) {
        for (int k = min(r, 128 * cb + 127); k >= max(1, 128 * cb); --k) {
            const double x = xs[k & 1];
            double next[RPL];
#pragma unroll
            for (int c = 0; c <= cb; ++c) next[c] = 128 * c + t < k - 1 ? L[(size_t)(k - 1) * n + 128 * c + t] : 0.0;
            // the group of four warps that holds entry k - 1: this block, or at its
            // lower end the one below
            const bool below = k == 128 * cb;
            const int m = k - 1;
            if (((m >> 5) & 3) == (t >> 5)) {
                if (!below) {
                    s[cb] = fma(-x, row[cb], s[cb]);
                    const double y = s[cb] * inv[cb];
                    if ((m & 127) == t) xs[m & 1] = s[cb] = y;
                } else if (cb > 0) {
                    s[cb > 0 ? cb - 1 : 0] = fma(-x, row[cb > 0 ? cb - 1 : 0], s[cb > 0 ? cb - 1 : 0]);
                    const double y = s[cb > 0 ? cb - 1 : 0] * inv[cb > 0 ? cb - 1 : 0];
                    if ((m & 127) == t) xs[m & 1] = s[cb > 0 ? cb - 1 : 0] = y;
                }
            } else {
                if (!below) s[cb] = fma(-x, row[cb], s[cb]);
                else if (cb > 0) s[cb > 0 ? cb - 1 : 0] = fma(-x, row[cb > 0 ? cb - 1 : 0], s[cb > 0 ? cb - 1 : 0]);
            }
#pragma unroll
            for (int c = 0; c < cb; ++c)
                if (!(below && c == cb - 1)) s[c] = fma(-x, row[c], s[c]);
#pragma unroll
            for (int c = 0; c <= cb; ++c) row[c] = next[c];
            __syncthreads();
        }
    }
#pragma unroll
    for (int c = 0; c < RPL; ++c) {
        const int j = 128 * c + t;
        if (j < n) X[(size_t)r * n + j] = j <= r ? s[c] : 0.0;
    }
}

}  // namespace

// L = chol(A), L and the lower triangle of A n x n row-major in different
// buffers, A overwritten; info[slot] (zero before) = 1 if A is not positive
// definite
int chol_blocked(nys_ctx* ctx, double* A, int n, double* L, double* info, int slot) {
    cudaStream_t s = ctx->stream;
    for (int p0 = 0; p0 < n; p0 += PB) {
        NYS_CK(ctx, launch_pdl(chol_panel_kernel, (n - p0 + PB - 1) / PB, 128, 0, s, (const double*)A, L, n, p0, info,
                               slot));
        NYS_LAUNCH_CK(ctx);
        const int rest = n - p0 - PB, t = (rest + 15) / 16;
        if (rest <= 0) break;
        NYS_CK(ctx, launch_pdl(chol_update_kernel, dim3(t, t), 256, 0, s, A, (const double*)L, n, p0,
                               (const double*)info, slot));
        NYS_LAUNCH_CK(ctx);
    }
    return NYS_OK;
}

// the shifted core's factor (no retries: info[0] = 1 asks for them), work n x n
int chol_core(nys_ctx* ctx, const double* G2, int n, double eps, double* work, double* L, double* info) {
    NYS_CK(ctx, launch_pdl(core_form_kernel, 64, 256, 0, ctx->stream, G2, n, eps, work, info));
    NYS_LAUNCH_CK(ctx);
    return chol_blocked(ctx, work, n, L, info, 0);
}

// X = L^{-1} for lower-triangular L (n x n, n <= 1024)
int tri_inv(nys_ctx* ctx, const double* L, double* X, int n) {
    auto go = [&](auto kernel) { return launch_pdl(kernel, n, 128, 0, ctx->stream, L, X, n); };
    NYS_CK(ctx, n <= 128 ? go(tri_inv_kernel<1>) : n <= 256 ? go(tri_inv_kernel<2>) : n <= 512 ? go(tri_inv_kernel<4>)
                                                                                              : go(tri_inv_kernel<8>));
    NYS_LAUNCH_CK(ctx);
    return NYS_OK;
}

}  // namespace nys
