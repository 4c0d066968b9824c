// Interleaved lanes of the ray transforms (radon.cu, fanbeam.cu).  Positions and
// weights cost as much as the arithmetic on the data, so the projectors carry
// IB values per position, interleaved in memory (one 16-byte load feeds four
// float32 lanes).  A lane is an image of a batch, or one of V copies of the
// same image moved by a symmetry of the geometry (mirrored, transposed,
// turned): the angle that sees the image as base angle k sees the copy shares
// every position and weight with angle k.
#pragma once

#include "internal.cuh"

#include <algorithm>

namespace nys {
namespace {

constexpr int PAD = 3;    // zeros of an interleaved line: one before, two after

// symmetries of a lane: source pixel of the copy's pixel (i, j) is (i, j), with
// i and j exchanged (T, square images), then mirrored (FJ, FI); REV: the bins
// of the lane's angle run backwards
enum : unsigned { LANE_FJ = 1, LANE_FI = 2, LANE_T = 4, LANE_REV = 8 };

// the angles of a launch: lane v of base entry kb holds angle ang[kb V + v] or,
// when negative, nothing; the positions are those of angle ang[kb V]
struct LaneSet {
    const int* ang;
    int V, n_base;
    unsigned tf;          // four bits per lane
    __host__ __device__ unsigned sym(int v) const { return (tf >> (4 * v)) & 15u; }
};

template <class TC, int IB>
struct alignas(sizeof(TC) * IB >= 16 ? 16 : sizeof(TC) * IB) Lanes {
    TC v[IB];
};

__device__ __forceinline__ void lane_src(unsigned tf, int& i, int& j, int n1, int n2) {
    if (tf & LANE_T) {
        const int t = i;
        i = j;
        j = t;
    }
    if (tf & LANE_FJ) j = n2 - 1 - j;
    if (tf & LANE_FI) i = n1 - 1 - i;
}

// 32 x 32 tiles of nl lines of na positions
__host__ __device__ __forceinline__ int lane_tiles(int nl, int na) { return (nl + 31) / 32 * ((na + PAD + 31) / 32); }

// interleaved lines: rows[g][i][1 + j] and, when the set has column-step base
// angles (cols), cols[g][j][1 + i]; lane q of group g is copy q % V
// of image g IB / V + q / V.  One CTA (the tiles of the rows, then those of the
// columns; a grid over the square of the longer side spent 129 us on 8000 x
// 100 pixels, this 11) writes 32 lines x 32 positions: every lane
// is read with its image's rows along the threads, through shared memory.
template <class TI, class TC, int IB>
__global__ void __launch_bounds__(256) lane_prep_kernel(const TI* __restrict__ x, Lanes<TC, IB>* __restrict__ rows,
                                                        Lanes<TC, IB>* __restrict__ cols, int n1, int n2, LaneSet set,
                                                        int batch) {
    pdl_enter();
    __shared__ TC tile[IB][32][33];
    const int nr = lane_tiles(n1, n2), o = (int)blockIdx.x >= nr, g = blockIdx.y;
    const int nl = o ? n2 : n1, na = o ? n1 : n2;
    const int bt = (int)blockIdx.x - (o ? nr : 0), nt = (na + PAD + 31) / 32;
    const int l0 = bt / nt * 32, p0 = bt % nt * 32 - 1;
    const int R = IB / set.V;
    const size_t N = (size_t)n1 * n2;
#pragma unroll
    for (int q = 0; q < IB; ++q) {
        const int b = g * R + q / set.V;
        const unsigned tf = set.sym(q % set.V);
        const bool along = (o == 0) == !(tf & LANE_T);      // the source's j runs along the line's positions
        for (int r = threadIdx.y; r < 32; r += 8) {
            const int dl = along ? r : threadIdx.x, dp = along ? threadIdx.x : r;
            const int l = l0 + dl, p = p0 + dp;
            TC val = TC(0);
            if (b < batch && l < nl && p >= 0 && p < na) {
                int i = o ? p : l, j = o ? l : p;
                lane_src(tf, i, j, n1, n2);
                val = (TC)ldf(x + (size_t)b * N + (size_t)i * n2 + j);
            }
            tile[q][dl][dp] = val;
        }
    }
    __syncthreads();
    Lanes<TC, IB>* dst = (o ? cols : rows) + (size_t)g * nl * (na + PAD);
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int l = l0 + r, e = p0 + 1 + threadIdx.x;
        if (l < nl && e < na + PAD) {
            Lanes<TC, IB> w;
#pragma unroll
            for (int q = 0; q < IB; ++q) w.v[q] = tile[q][r][threadIdx.x];
            dst[(size_t)l * (na + PAD) + e] = w;
        }
    }
}

// planar sinogram (images x angles x bins) to the interleaved lanes [g][kb][m]
template <class TI, class TC, int IB>
__global__ void __launch_bounds__(256) lane_bins_kernel(const TI* __restrict__ s, Lanes<TC, IB>* __restrict__ out,
                                                          int n_angles, int n_bins, int batch, LaneSet set) {
    pdl_enter();
    const int kb = blockIdx.x, g = blockIdx.y;
    const int* ang = set.ang + kb * set.V;
    for (int m = threadIdx.x; m < n_bins; m += blockDim.x) {
        Lanes<TC, IB> w;
#pragma unroll
        for (int q = 0; q < IB; ++q) {
            const int b = g * (IB / set.V) + q / set.V, a = ang[q % set.V];
            const int mq = set.sym(q % set.V) & LANE_REV ? n_bins - 1 - m : m;
            w.v[q] = b < batch && a >= 0 ? (TC)ldf(s + ((size_t)b * n_angles + a) * n_bins + mq) : TC(0);
        }
        out[((size_t)g * set.n_base + kb) * n_bins + m] = w;
    }
}

__device__ __forceinline__ void cp_async_zfill(void* dst, const void* src, int bytes, bool ok) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = ok ? bytes : 0;
    if (bytes == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n));
    else if (bytes == 8) asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(n));
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(n));
}

// x[b] = the sum of image b's planes: ns angle ranges x V lanes (V a power of
// two), eight loads in flight (20 planes of 81 x 70: 10.2 to 5.7 us)
template <class TC, class TO, int IB>
__global__ void __launch_bounds__(256) lane_sum_kernel(const TC* __restrict__ planes, TO* __restrict__ x, int64_t N,
                                                        int V, int ns) {
    pdl_enter();
    const int b = blockIdx.y, R = IB / V, g = b / R, q0 = (b - g * R) * V, n = ns * V, lv = V >> 1;   // log2 of 1, 2, 4
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < N; t += (int64_t)gridDim.x * blockDim.x) {
        TC v = TC(0);
        const TC* p = planes + ((size_t)g * ns * IB + q0) * N + t;
#pragma unroll 8
        for (int e = 0; e < n; ++e) v += p[(size_t)((e >> lv) * IB + (e & (V - 1))) * N];
        stf(x + (size_t)b * N + t, v);
    }
}

// position of a ray on its line, stepped line by line: an integer part and a
// binary fraction f of 40 (float) or 64 (double) bits, so that the rounding of
// the step stays below the weights' over thousands of lines; weights() are those
// of the positions index() and index() + 1, 1 - f and f.  In float f is its top
// 32 bits converted (rounded to 2^-25; 23 bits put into a float between 1 and 2
// leave 2^-24 with rounding and twice that without)
template <class TC>
struct RayPos;
template <>
struct RayPos<float> {
    long long p;
    __device__ __forceinline__ void set40(long long u) { p = u; }
    __device__ __forceinline__ void step(const RayPos& d) { p += d.p; }
    __device__ __forceinline__ int index() const { return (int)(p >> 40); }
    __device__ __forceinline__ void weights(float& w0, float& w1) const {
        const float F = __uint2float_rn((unsigned)(p >> 8));
        w1 = F * 0x1p-32f;
        w0 = fmaf(F, -0x1p-32f, 1.0f);
    }
};
template <>
struct RayPos<double> {
    int i;
    unsigned long long f;
    __device__ __forceinline__ void set(double u) {
        const double fl = floor(u);
        i = (int)fl;
        f = (unsigned long long)((u - fl) * 18446744073709551616.0);   // 2^64; saturates below it
    }
    __device__ __forceinline__ void step(const RayPos& d) {
        const unsigned long long s = f + d.f;
        i += d.i + (s < f ? 1 : 0);
        f = s;
    }
    __device__ __forceinline__ int index() const { return i; }
    __device__ __forceinline__ void weights(double& w0, double& w1) const {
        const double F = __longlong_as_double((long long)((f >> 12) | 0x3ff0000000000000ull));   // 1 + f
        w1 = F - 1.0;
        w0 = 2.0 - F;
    }
};

// Lanes and mirror lanes for a part of a batch: fours of images while there
// are four; a rest of one to three takes four mirror lanes an image where the
// angles allow it (a quarter of the angles each), else two (two images to a
// launch group), else plain lanes.  Images for which scratch is short
// (ray_chunk) go one group at a time, the largest by themselves.
struct Part {
    int nb, IB, V;
};
constexpr int RAY_CHUNK = 32;
inline Part next_part(const nys_op* op, int left) {
    if (op->chunk == 1) return {1, 1, 1};
    if (left >= 4) return {left / 4 * 4, 4, 1};
    const bool one = op->chunk < RAY_CHUNK;
    if (op->lane_sets & 4) return {one ? 1 : left, 4, 4};
    if (op->lane_sets & 2) return left == 1 ? Part{1, 2, 2} : Part{one ? 2 : left, 4, 2};
    return {left, left == 3 ? 4 : left, 1};
}

// images to a chunk: 32 while their lines (two copies each) stay within 2 GB
// (2048 x 2048 in float64), then as many as do, at least a group (eight in
// float32: the bf16 forward); one, in plain lanes, where a group with its planes
// would take more than 64 GB.  32 throughout took 8.6 GB for an operator of 4096
// x 4096 pixels in float64, whatever it was used on; this 2.7 GB.  (A^T A of 32
// float32 images of 4096 x 4096, 90 angles: within 4 GB 37.1, 2 GB 38.3, 1 GB
// 41.6 ms.)
inline int ray_chunk(const nys_op* op) {
    const int64_t image = op->N * (op->dtype == NYS_F64 ? 8 : 4), unit = op->dtype == NYS_F64 ? 4 : 8;
    if ((2 * unit + 4) * image > (int64_t(64) << 30)) return 1;
    return (int)std::max(unit, std::min<int64_t>(RAY_CHUNK, (int64_t(2) << 30) / (2 * image) / unit * unit));
}

template <class TI, class TC, int IB>
int lane_prep(nys_op* op, const TI* x, int nb, const LaneSet& set, bool with_cols) {
    const int R = IB / set.V, groups = (nb + R - 1) / R;
    auto* rows = (Lanes<TC, IB>*)op->lines;
    auto* cols = with_cols ? rows + (size_t)groups * op->n1 * (op->n2 + PAD) : nullptr;
    const int tiles = lane_tiles(op->n1, op->n2) + (cols ? lane_tiles(op->n2, op->n1) : 0);
    NYS_CK(op->ctx, launch_pdl(lane_prep_kernel<TI, TC, IB>, dim3(tiles, groups), dim3(32, 8), 0,
                               op->ctx->stream, x, rows, cols, op->n1, op->n2, set, nb));
    NYS_LAUNCH_CK(op->ctx);
    return NYS_OK;
}

template <class TI, class TC, int IB>
int lane_bins(nys_op* op, const TI* s, int nb, const LaneSet& set) {
    const int R = IB / set.V, groups = (nb + R - 1) / R;
    NYS_CK(op->ctx, launch_pdl(lane_bins_kernel<TI, TC, IB>, dim3(set.n_base, groups), 256, 0,
                               op->ctx->stream, s, (Lanes<TC, IB>*)op->inter, op->n_angles, op->n_bins, nb, set));
    NYS_LAUNCH_CK(op->ctx);
    return NYS_OK;
}

template <class TC, class TO, int IB>
int lane_sum(nys_op* op, TO* x, int nb, int V, int ns) {
    NYS_CK(op->ctx, launch_pdl(lane_sum_kernel<TC, TO, IB>, dim3((unsigned)std::min<int64_t>((op->N + 255) / 256, 1024),
                                                                 nb), 256, 0, op->ctx->stream, (const TC*)op->planes, x,
                               op->N, V, ns));
    NYS_LAUNCH_CK(op->ctx);
    return NYS_OK;
}

}  // namespace
}  // namespace nys
