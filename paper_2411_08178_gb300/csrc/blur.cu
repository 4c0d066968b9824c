// Periodic blur H, its adjoint H^T and the normal operator H^T H (Sec. IV-A),
// plus blur + decimation D H (super-resolution).
//
// Definition (correlation form, periodic boundary, odd kh x kw kernel h):
//     (Hx)[i,j] = sum_{a,b} h[a,b] x[(i + a - ch) mod n1, (j + b - cw) mod n2]
// with ch = (kh-1)/2, cw = (kw-1)/2.  H^T is the same correlation with the
// flipped kernel.  When h is rank one (every Gaussian blur), h = u v^T and
// H = H_col(u) H_row(v), so each apply is two 1-D passes, and
// H^T H = H_col(u * u) H_row(v * v) (autocorrelations of length 2k-1,
// centred at k-1): the normal operator is ONE fused separable pass.
//
// Kernel design (sm_103a): batches of bf16 images stream down strips of
// columns in persistent CTAs (sepstream_kernel below); everything else takes
// one CTA per output tile, its side chosen by size (pick_tile).  The input
// tile and its periodic halo are staged once in shared memory; the row pass
// writes an intermediate tile to shared memory; the column pass writes the
// output.  Each thread computes 8 consecutive outputs of a row (or column)
// with a sliding register window, so every shared-memory load feeds 8 FMAs and
// the tile kernel is bound by the FP32 FMA pipe rather than by shared-memory
// bandwidth.  Row pitches are odd so that lanes reading consecutive rows hit distinct banks.
#include "internal.cuh"

#include <cmath>
#include <type_traits>

namespace nys {
namespace {

constexpr int RB = 8;  // register block (outputs per thread along a pass)

// Stage rows x cols input values starting at (r0, c0) (periodic) into a
// shared-memory tile of pitch `pitch`: one warp per row, lanes along the row.
// The wrap is one conditional step when the staged extent fits in the image
// (no integer division per element); small images take the modulo.
template <class TI, class TC>
__device__ __forceinline__ void stage_tile(const TI* __restrict__ xb, int n1, int n2, int r0, int c0, int rows,
                                           int cols, TC* __restrict__ s, int pitch) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const bool step = r0 >= -n1 && r0 + rows <= 2 * n1 && c0 >= -n2 && c0 + cols <= 2 * n2;
    constexpr int MQ = 4;   // rows of up to 128 columns: every load of two rows issued before any store
    if (step && cols <= 32 * MQ) {
        for (int ra = warp; ra < rows; ra += 2 * nw) {
            TC v[2][MQ];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = ra + h * nw;
                int gi = r0 + r;
                gi = gi < 0 ? gi + n1 : (gi >= n1 ? gi - n1 : gi);
                const TI* xr = xb + (size_t)gi * n2;
#pragma unroll
                for (int q = 0; q < MQ; ++q) {
                    const int c = lane + 32 * q;
                    int gj = c0 + c;
                    gj = gj < 0 ? gj + n2 : (gj >= n2 ? gj - n2 : gj);
                    v[h][q] = (r < rows && c < cols) ? (TC)ldf(xr + gj) : TC(0);
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = ra + h * nw;
#pragma unroll
                for (int q = 0; q < MQ; ++q) {
                    const int c = lane + 32 * q;
                    if (r < rows && c < cols) s[(size_t)r * pitch + c] = v[h][q];
                }
            }
        }
        return;
    }
    for (int r = warp; r < rows; r += nw) {
        int gi = r0 + r;
        gi = step ? (gi < 0 ? gi + n1 : (gi >= n1 ? gi - n1 : gi)) : pmod(gi, n1);
        const TI* xr = xb + (size_t)gi * n2;
        TC* sr = s + (size_t)r * pitch;
        for (int c = lane; c < cols; c += 32) {
            int gj = c0 + c;
            gj = step ? (gj < 0 ? gj + n2 : (gj >= n2 ? gj - n2 : gj)) : pmod(gj, n2);
            sr[c] = (TC)ldf(xr + gj);
        }
    }
}

__host__ __device__ inline int round8(int x) { return (x + 7) & ~7; }
__host__ __device__ inline int odd_pitch(int x) { return x | 1; }

// Sliding-window 1-D correlation of 8 consecutive outputs:
//   acc[r] += sum_{t < Lp} g[t] * src[(r + t) * stride]
template <class TC>
__device__ __forceinline__ void window8(const TC* __restrict__ src, int stride, const TC* __restrict__ g,
                                        int Lp, TC acc[RB]) {
    TC win[RB], nxt[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) win[r] = src[r * stride];
    for (int t0 = 0; t0 < Lp; t0 += RB) {
#pragma unroll
        for (int r = 0; r < RB; ++r) nxt[r] = src[(t0 + RB + r) * stride];
#pragma unroll
        for (int dt = 0; dt < RB; ++dt) {
            const TC gv = g[t0 + dt];
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                const TC v = (r + dt < RB) ? win[r + dt] : nxt[r + dt - RB];
                acc[r] = fma(gv, v, acc[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < RB; ++r) win[r] = nxt[r];
    }
}

// The same window over two independent lines (rows or columns) a and b at
// once: the two lines' values sit in the halves of a float2, so one packed
// FMA (FFMA2, sm_100 and later) does the tap for both, with the same
// rounding as two scalar FMAs; half the FMA instructions of two window8
// calls, and the taps loaded once for both lines.
__device__ __forceinline__ void window8x2(const float* __restrict__ sa, const float* __restrict__ sb, int stride,
                                         const float* __restrict__ g, int Lp, float2 acc[RB]) {
    float2 win[RB], nxt[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) win[r] = make_float2(sa[r * stride], sb[r * stride]);
    for (int t0 = 0; t0 < Lp; t0 += RB) {
#pragma unroll
        for (int r = 0; r < RB; ++r) nxt[r] = make_float2(sa[(t0 + RB + r) * stride], sb[(t0 + RB + r) * stride]);
#pragma unroll
        for (int dt = 0; dt < RB; ++dt) {
            const float gv = g[t0 + dt];
            const float2 g2 = make_float2(gv, gv);
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                const float2 v = (r + dt < RB) ? win[r + dt] : nxt[r + dt - RB];
                acc[r] = __ffma2_rn(g2, v, acc[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < RB; ++r) win[r] = nxt[r];
    }
}

template <class TC> struct PairWindow { static constexpr bool on = false; };
template <> struct PairWindow<float> { static constexpr bool on = true; };

// y = H_col(gc) H_row(gr) x, separable periodic correlation.
// taps: gc (Lcp entries, zero padded) followed by gr (Lrp entries).
template <class TI, class TO, class TC, int TY, int TX>
__global__ void __launch_bounds__(256) sepcorr_kernel(const TI* __restrict__ x, TO* __restrict__ y, int n1,
                                                      int n2, const TC* __restrict__ taps, int Lcp, int Lrp,
                                                      int cc, int cr) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TC* s_tap = reinterpret_cast<TC*>(smem_raw);
    const int rows = TY + Lcp;          // staged input rows = intermediate rows
    const int wcols = TX + Lrp;         // staged input columns
    const int pin = odd_pitch(wcols);
    const int pmid = odd_pitch(TX);
    TC* s_in = s_tap + Lcp + Lrp;
    TC* s_mid = s_in + (size_t)rows * pin;

    const int i0 = blockIdx.y * TY, j0 = blockIdx.x * TX;
    const size_t img = (size_t)blockIdx.z * n1 * n2;
    const TI* xb = x + img;
    for (int t = threadIdx.x; t < Lcp + Lrp; t += blockDim.x) s_tap[t] = taps[t];
    stage_tile<TI, TC>(xb, n1, n2, i0 - cc, j0 - cr, rows, wcols, s_in, pin);
    __syncthreads();
    // row pass: s_mid[r][c] = sum_b gr[b] s_in[r][c + b]
    const TC* gr = s_tap + Lcp;
    TO* yb = y + img;
    if constexpr (PairWindow<TC>::on) {
        // float32: rows r and r + rows / 2 together (rows = TY + Lcp is even)
        const int hr = rows / 2;
        for (int idx = threadIdx.x; idx < hr * (TX / RB); idx += blockDim.x) {
            const int r = idx % hr, sx = idx / hr;
            float2 acc[RB];
#pragma unroll
            for (int k = 0; k < RB; ++k) acc[k] = make_float2(0.0f, 0.0f);
            window8x2(s_in + r * pin + sx * RB, s_in + (r + hr) * pin + sx * RB, 1, gr, Lrp, acc);
#pragma unroll
            for (int k = 0; k < RB; ++k) {
                s_mid[r * pmid + sx * RB + k] = acc[k].x;
                s_mid[(r + hr) * pmid + sx * RB + k] = acc[k].y;
            }
        }
        __syncthreads();
        // column pass: columns c and c + TX / 2 together
        const int hc = TX / 2;
        for (int idx = threadIdx.x; idx < hc * (TY / RB); idx += blockDim.x) {
            const int c = idx % hc, sy = idx / hc;
            float2 acc[RB];
#pragma unroll
            for (int k = 0; k < RB; ++k) acc[k] = make_float2(0.0f, 0.0f);
            const float* base = s_mid + (sy * RB) * pmid + c;
            window8x2(base, base + hc, pmid, s_tap, Lcp, acc);
#pragma unroll
            for (int k = 0; k < RB; ++k) {
                const int gi = i0 + sy * RB + k;
                if (gi >= n1) continue;
                if (j0 + c < n2) stf(yb + (size_t)gi * n2 + j0 + c, acc[k].x);
                if (j0 + c + hc < n2) stf(yb + (size_t)gi * n2 + j0 + c + hc, acc[k].y);
            }
        }
    } else {
        for (int idx = threadIdx.x; idx < rows * (TX / RB); idx += blockDim.x) {
            const int r = idx % rows, sx = idx / rows;
            TC acc[RB];
#pragma unroll
            for (int k = 0; k < RB; ++k) acc[k] = TC(0);
            window8<TC>(s_in + r * pin + sx * RB, 1, gr, Lrp, acc);
#pragma unroll
            for (int k = 0; k < RB; ++k) s_mid[r * pmid + sx * RB + k] = acc[k];
        }
        __syncthreads();
        // column pass: y[i][c] = sum_a gc[a] s_mid[i + a][c]
        for (int idx = threadIdx.x; idx < TX * (TY / RB); idx += blockDim.x) {
            const int c = idx % TX, sy = idx / TX;
            TC acc[RB];
#pragma unroll
            for (int k = 0; k < RB; ++k) acc[k] = TC(0);
            window8<TC>(s_mid + (sy * RB) * pmid + c, pmid, s_tap, Lcp, acc);
            const int gj = j0 + c;
            if (gj < n2) {
#pragma unroll
                for (int k = 0; k < RB; ++k) {
                    const int gi = i0 + sy * RB + k;
                    if (gi < n1) stf(yb + (size_t)gi * n2 + gj, acc[k]);
                }
            }
        }
    }
}

// Sixteen consecutive outputs of two lines a and b (the halves of a float2)
// from a window of 24 values held in registers, eight taps at a time: 16 loads
// (8 of bf16 pairs) and two tap loads per 128 packed FMAs.  L taps (16-byte
// aligned, padded to a multiple of 8, the padding not used).  Reads values up
// to index 8 (L / 8) + 23.
struct Window16 {
    float2 w[24], acc[16];
    const float *sa, *sb;          // float lines
    const unsigned *pa, *pb;       // lines of bf16 pairs
    const float4* g;
    int stride;
    template <bool PAIRS, int AT>  // eight values from index t on into registers AT ..
    __device__ __forceinline__ void load(int t) {
        if constexpr (PAIRS) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const unsigned a = pa[t / 2 + r], b = pb[t / 2 + r];
                w[(AT + 2 * r) % 24] = make_float2(__uint_as_float(a << 16), __uint_as_float(b << 16));
                w[(AT + 2 * r + 1) % 24] = make_float2(__uint_as_float(a & 0xffff0000u), __uint_as_float(b & 0xffff0000u));
            }
        } else {
#pragma unroll
            for (int r = 0; r < 8; ++r) w[(AT + r) % 24] = make_float2(sa[(t + r) * stride], sb[(t + r) * stride]);
        }
    }
    template <bool PAIRS, int O>   // O: register of the window's first value
    __device__ __forceinline__ void taps(int t0, int n) {
        load<PAIRS, O + 16>(t0 + 16);
        const float4 ga = g[t0 / 4], gb = g[t0 / 4 + 1];
        const float tap[8] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
#pragma unroll
        for (int dt = 0; dt < 8; ++dt) {
            if (dt >= n) break;
            const float2 g2 = make_float2(tap[dt], tap[dt]);
#pragma unroll
            for (int r = 0; r < 16; ++r) acc[r] = __ffma2_rn(g2, w[(O + r + dt) % 24], acc[r]);
        }
    }
    template <bool PAIRS>
    __device__ __forceinline__ void run(int L) {
#pragma unroll
        for (int r = 0; r < 16; ++r) acc[r] = make_float2(0.0f, 0.0f);
        load<PAIRS, 0>(0);
        load<PAIRS, 8>(8);
        const int full = L & ~7;
        int t0 = 0;
        for (; t0 + 24 <= full; t0 += 24) {
            taps<PAIRS, 0>(t0, 8);
            taps<PAIRS, 8>(t0 + 8, 8);
            taps<PAIRS, 16>(t0 + 16, 8);
        }
        if (t0 < full) {
            taps<PAIRS, 0>(t0, 8);
            if (t0 + 8 < full) {
                taps<PAIRS, 8>(t0 + 8, 8);
                if (L & 7) taps<PAIRS, 16>(full, L & 7);
            } else if (L & 7) {
                taps<PAIRS, 8>(full, L & 7);
            }
        } else if (L & 7) {
            taps<PAIRS, 0>(full, L & 7);
        }
    }
};

// y = H_col(gc) H_row(gr) x on many bf16 images (the sketch): a CTA walks down
// a strip of TX columns, 64 rows at a time, keeping the row pass of the last
// Lc - 1 rows, so that the row pass is done once per image row (and Lc - 1
// times more at the top of a strip) instead of 1 + Lc / 64 times; the next 64 input rows arrive by cp.async (pairs of columns: n2, cr
// and the start of the strip are even) while these are computed.  The same
// sums in the same order as sepcorr_kernel.  Bound by FP32 FMA issue: 200
// images of 512 x 512 with 49 taps a side (10.3 GFLOP): 241 us, 43 TFLOP/s (tiles with a 56-row halo: 572 us).
constexpr int SY = 64;
template <int TX>
__host__ __device__ inline int stream_pin(int Lr) { return odd_pitch((TX + 8 * (Lr / 8) + 8) / 2); }   // words
__host__ __device__ inline int stream_rows(int Lc) { return SY + 8 * (Lc / 8) + 8; }
template <int TX>
size_t stream_smem(int Lc, int Lr) {
    return 4 * ((size_t)round8(Lc) + round8(Lr) + (size_t)2 * SY * stream_pin<TX>(Lr) + (size_t)stream_rows(Lc) * (TX | 1));
}

template <class TO, int TX>
__global__ void __launch_bounds__(2 * TX, TX == 128 ? 2 : 3)
    sepstream_kernel(const __nv_bfloat16* __restrict__ x, TO* __restrict__ y, int n1, int n2, int batch,
                     const float* __restrict__ taps, int Lc, int Lr, int cc, int cr) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* s_tap = reinterpret_cast<float*>(smem_raw);
    const int Lcp = round8(Lc), Lrp = round8(Lr), pin = stream_pin<TX>(Lr), H = Lc - 1;
    constexpr int pmid = TX | 1, NT = 2 * TX, NW = NT / 32;
    constexpr int MQ = (TX / 2 + 32 + 31) / 32;     // staged pairs per lane and row: (TX + Lr) / 2 <= 32 MQ
    unsigned* s_in = reinterpret_cast<unsigned*>(s_tap + Lcp + Lrp);     // [2][SY][pin] pairs
    float* s_mid = reinterpret_cast<float*>(s_in + 2 * SY * pin);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wq = (TX + Lr) / 2, hn = n2 / 2;      // pairs staged per row, pairs of an image row
    for (int t = threadIdx.x; t < Lcp + Lrp; t += NT) s_tap[t] = taps[t];
    // this CTA's share of the 64-row chunks of all strips, in order: a part of a
    // strip at either end, whole strips between
    const int chunks = (n1 + SY - 1) / SY, strips = (n2 + TX - 1) / TX;
    const int64_t total = (int64_t)batch * strips * chunks;
    const int64_t t_beg = total * blockIdx.x / gridDim.x, t_end = total * (blockIdx.x + 1) / gridDim.x;
    const int above = (H + SY - 1) / SY;            // blocks of input rows above a part
    for (int64_t t = t_beg; t < t_end;) {
        const int64_t strip = t / chunks;
        const int c0 = (int)(t - strip * chunks), nc = (int)min((int64_t)(chunks - c0), t_end - t);
        t += nc;
        const int b_img = (int)(strip / strips), j0 = (int)(strip - (int64_t)b_img * strips) * TX;
        const int ib = c0 * SY, ie = min(n1, (c0 + nc) * SY);
        const unsigned* xb = reinterpret_cast<const unsigned*>(x + (size_t)b_img * n1 * n2);
        TO* yb = y + (size_t)b_img * n1 * n2;
        int gj[MQ];
#pragma unroll
        for (int q = 0; q < MQ; ++q) gj[q] = pmod((j0 - cr) / 2 + lane + 32 * q, hn);
        auto stage = [&](int r0, int buf, int rows) {
            const unsigned d0 = (unsigned)__cvta_generic_to_shared(s_in + buf * SY * pin + lane);
            for (int r = warp; r < rows; r += NW) {
                int gi = r0 + r;
                gi = gi < 0 ? gi + n1 : (gi >= n1 ? gi - n1 : gi);
                if (gi < 0 || gi >= n1) gi = pmod(gi, n1);
                const unsigned* xr = xb + (size_t)gi * hn;
                const unsigned d = d0 + 4 * r * pin;
#pragma unroll
                for (int q = 0; q < MQ; ++q)
                    if (lane + 32 * q < wq)
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 128 * q), "l"(xr + gj[q]));
            }
            asm volatile("cp.async.commit_group;");
        };
        // blocks of input rows in order: those above (H rows), then 64 for every
        // 64 output rows
        const int blocks = above + nc;
        auto first_row = [&](int b) { return ib - cc + (b < above ? b * SY : H + (b - above) * SY); };
        __syncthreads();                            // the previous part is done with the buffers
        stage(first_row(0), 0, above ? min(SY, H) : SY);
        for (int b = 0; b < blocks; ++b) {
            asm volatile("cp.async.wait_group 0;");
            __syncthreads();
            if (b + 1 < blocks) stage(first_row(b + 1), (b + 1) & 1, b + 1 < above ? min(SY, H - (b + 1) * SY) : SY);
            {
                // row pass of rows r and r + 32 of the block
                const int rows = b < above ? min(SY, H - b * SY) : SY, at = b < above ? b * SY : H;
                Window16 w;
                w.pa = s_in + (b & 1) * SY * pin + lane * pin + 8 * warp;
                w.pb = w.pa + 32 * pin;
                w.g = reinterpret_cast<const float4*>(s_tap + Lcp);
                w.run<true>(Lr);
                float* m = s_mid + (at + lane) * pmid + 16 * warp;
                if (lane < rows)
#pragma unroll
                    for (int k = 0; k < 16; ++k) m[k] = w.acc[k].x;
                if (lane + 32 < rows)
#pragma unroll
                    for (int k = 0; k < 16; ++k) m[32 * pmid + k] = w.acc[k].y;
            }
            __syncthreads();
            if (b < above) continue;
            const int i0 = ib + (b - above) * SY;
            // column pass: columns c and c + TX / 2 together
            const int c = threadIdx.x % (TX / 2), sy = threadIdx.x / (TX / 2);
            Window16 w;
            w.sa = s_mid + 16 * sy * pmid + c;
            w.sb = w.sa + TX / 2;
            w.stride = pmid;
            w.g = reinterpret_cast<const float4*>(s_tap);
            w.run<false>(Lc);
            const int left = ie - (i0 + 16 * sy);   // output rows of this thread
            TO* yo = yb + (size_t)(i0 + 16 * sy) * n2 + j0 + c;
            const bool ca = j0 + c < n2, cb = j0 + c + TX / 2 < n2;
            if (left >= 16 && cb) {
#pragma unroll
                for (int k = 0; k < 16; ++k, yo += n2) {
                    stf(yo, w.acc[k].x);
                    stf(yo + TX / 2, w.acc[k].y);
                }
            } else {
#pragma unroll
                for (int k = 0; k < 16; ++k, yo += n2) {
                    if (k < left && ca) stf(yo, w.acc[k].x);
                    if (k < left && cb) stf(yo + TX / 2, w.acc[k].y);
                }
            }
            // the last H rows move to the top, 64 rows at a time
            if (b + 1 < blocks)
                for (int d = 0; d < H; d += SY) {
                    __syncthreads();
                    float* m = s_mid + (d + threadIdx.x / TX) * pmid + threadIdx.x % TX;
                    for (int r = threadIdx.x / TX; r < min(SY, H - d); r += 2, m += 2 * pmid) *m = m[SY * pmid];
                }
        }
    }
}

// General (non-separable) periodic correlation with a kh x kw kernel.
// taps: kh rows of kwp entries (zero padded).
template <class TI, class TO, class TC, int TY, int TX>
__global__ void __launch_bounds__(256) corr2d_kernel(const TI* __restrict__ x, TO* __restrict__ y, int n1,
                                                     int n2, const TC* __restrict__ taps, int kh, int kwp,
                                                     int ch, int cw) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TC* s_tap = reinterpret_cast<TC*>(smem_raw);
    const int rows = TY + kh - 1;
    const int wcols = TX + kwp;
    const int pin = odd_pitch(wcols);
    TC* s_in = s_tap + kh * kwp;
    const int i0 = blockIdx.y * TY, j0 = blockIdx.x * TX;
    const size_t img = (size_t)blockIdx.z * n1 * n2;
    const TI* xb = x + img;
    for (int t = threadIdx.x; t < kh * kwp; t += blockDim.x) s_tap[t] = taps[t];
    stage_tile<TI, TC>(xb, n1, n2, i0 - ch, j0 - cw, rows, wcols, s_in, pin);
    __syncthreads();
    TO* yb = y + img;
    if constexpr (PairWindow<TC>::on) {
        // float32: rows r and r + TY / 2 together
        constexpr int HY = TY / 2;
        for (int idx = threadIdx.x; idx < HY * (TX / RB); idx += blockDim.x) {
            const int r = idx % HY, sx = idx / HY;
            float2 acc[RB];
#pragma unroll
            for (int k = 0; k < RB; ++k) acc[k] = make_float2(0.0f, 0.0f);
            for (int a = 0; a < kh; ++a)
                window8x2(s_in + (r + a) * pin + sx * RB, s_in + (r + HY + a) * pin + sx * RB, 1, s_tap + a * kwp, kwp,
                          acc);
#pragma unroll
            for (int k = 0; k < RB; ++k) {
                const int gj = j0 + sx * RB + k;
                if (gj >= n2) continue;
                if (i0 + r < n1) stf(yb + (size_t)(i0 + r) * n2 + gj, acc[k].x);
                if (i0 + r + HY < n1) stf(yb + (size_t)(i0 + r + HY) * n2 + gj, acc[k].y);
            }
        }
        return;
    }
    for (int idx = threadIdx.x; idx < TY * (TX / RB); idx += blockDim.x) {
        const int r = idx % TY, sx = idx / TY;
        TC acc[RB];
#pragma unroll
        for (int k = 0; k < RB; ++k) acc[k] = TC(0);
        for (int a = 0; a < kh; ++a) window8<TC>(s_in + (r + a) * pin + sx * RB, 1, s_tap + a * kwp, kwp, acc);
        const int gi = i0 + r;
        if (gi < n1) {
#pragma unroll
            for (int k = 0; k < RB; ++k) {
                const int gj = j0 + sx * RB + k;
                if (gj < n2) stf(yb + (size_t)gi * n2 + gj, acc[k]);
            }
        }
    }
}

// ---------------------------------------------------- blur + decimate ----
// One thread per output, 64 to a block so that few outputs spread over more
// SMs; bound by the latency of its chain of taps.  The wrapped row and column
// step along with the taps, whose loads go out eight (four) at a time (a modulo
// and a division per tap, one load after the other: the forward
// 7.7 and the adjoint 7.3 us at 512 x 512, 7 x 7 taps, decimation 4; now 4.6 and
// 5.8.  23 x 23 taps on 128 x 128: 46 to 21 us and 10.4 to 6.0 us).
// y[p,q] = sum_{a,b} h[a,b] x[(d p + a - ch) mod n1, (d q + b - cw) mod n2]
template <class TI, class TO, class TC>
__global__ void __launch_bounds__(64) decim_fwd_kernel(const TI* __restrict__ x, TO* __restrict__ y, int n1, int n2,
                                                       int d, const TC* __restrict__ h, int kh, int kw, int batch) {
    pdl_enter();
    const int m1 = n1 / d, m2 = n2 / d;
    const int64_t total = (int64_t)batch * m1 * m2;
    const int ch = (kh - 1) / 2, cw = (kw - 1) / 2;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int b = (int)(t / ((int64_t)m1 * m2));
        const int rem = (int)(t - (int64_t)b * m1 * m2);
        const int p = rem / m2, q = rem - p * m2;
        const TI* xb = x + (size_t)b * n1 * n2;
        const int j0 = pmod(d * q - cw, n2);
        int gi = pmod(d * p - ch, n1);
        const TC* ha = h;
        TC acc = TC(0);
        for (int a = 0; a < kh; ++a, ha += kw) {
            const TI* row = xb + (size_t)gi * n2;
            int gj = j0;
            for (int bb = 0; bb < kw; bb += 8) {
                TC w[8], v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const bool ok = bb + u < kw;
                    w[u] = ok ? ha[bb + u] : TC(0);
                    v[u] = ok ? (TC)ldf(row + gj) : TC(0);
                    gj = gj + 1 == n2 ? 0 : gj + 1;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) acc = fma(w[u], v[u], acc);
            }
            gi = gi + 1 == n1 ? 0 : gi + 1;
        }
        stf(y + t, acc);
    }
}

// x[i,j] = sum over (a,b) with (i - a + ch) = 0 mod d and (j - b + cw) = 0 mod d of
//          h[a,b] y[((i - a + ch) mod n1)/d, ((j - b + cw) mod n2)/d]
// (each next tap of a pixel takes the sample before)
template <class TI, class TO, class TC>
__global__ void __launch_bounds__(64) decim_adj_kernel(const TI* __restrict__ y, TO* __restrict__ x, int n1, int n2,
                                                       int d, const TC* __restrict__ h, int kh, int kw, int batch) {
    pdl_enter();
    const int m1 = n1 / d, m2 = n2 / d;
    const int64_t total = (int64_t)batch * n1 * n2;
    const int ch = (kh - 1) / 2, cw = (kw - 1) / 2;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int b = (int)(t / ((int64_t)n1 * n2));
        const int rem = (int)(t - (int64_t)b * n1 * n2);
        const int i = rem / n2, j = rem - i * n2;
        const TI* yb = y + (size_t)b * m1 * m2;
        const int a0 = (i + ch) % d, b0 = (j + cw) % d;
        const int j0 = (j + cw - b0) / d % m2;
        int zi = (i + ch - a0) / d % m1;
        TC acc = TC(0);
        for (int a = a0; a < kh; a += d) {
            const TI* row = yb + (size_t)zi * m2;
            int zj = j0;
            for (int bb = b0; bb < kw; bb += 4 * d) {
                TC w[4], v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool ok = bb + u * d < kw;
                    w[u] = ok ? h[a * kw + bb + u * d] : TC(0);
                    v[u] = ok ? (TC)ldf(row + zj) : TC(0);
                    zj = zj ? zj - 1 : m2 - 1;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) acc = fma(w[u], v[u], acc);
            }
            zi = zi ? zi - 1 : m1 - 1;
        }
        stf(x + t, acc);
    }
}

// --------------------------------------------------------------- launch --
template <class TC>
size_t sep_smem(int TY, int TX, int Lcp, int Lrp) {
    const int rows = TY + Lcp;
    return sizeof(TC) * ((size_t)(Lcp + Lrp) + (size_t)rows * odd_pitch(TX + Lrp) + (size_t)rows * odd_pitch(TX));
}
template <class TC>
size_t c2d_smem(int TY, int TX, int kh, int kwp) {
    return sizeof(TC) * ((size_t)kh * kwp + (size_t)(TY + kh - 1) * odd_pitch(TX + kwp));
}

template <class TI, class TO, class TC, int T>
int launch_sep(nys_op* op, const void* x, void* y, int batch, const void* taps, int Lcp, int Lrp, int cc,
               int cr) {
    const size_t sm = sep_smem<TC>(T, T, Lcp, Lrp);
    auto k = sepcorr_kernel<TI, TO, TC, T, T>;
    if (int st = smem_optin(op->ctx, (const void*)k, sm)) return st;
    for (int b0 = 0; b0 < batch; b0 += 65535) {     // images in grid.z
        dim3 grid((op->n2 + T - 1) / T, (op->n1 + T - 1) / T, std::min(65535, batch - b0));
        NYS_CK(op->ctx, launch_pdl(k, grid, 256, sm, op->ctx->stream, (const TI*)x + (size_t)b0 * op->N,
                                   (TO*)y + (size_t)b0 * op->N, op->n1, op->n2, (const TC*)taps, Lcp, Lrp, cc, cr));
        NYS_LAUNCH_CK(op->ctx);
    }
    return NYS_OK;
}

template <class TO, int TX>
int launch_stream(nys_op* op, const __nv_bfloat16* x, TO* y, int batch, const void* taps, int Lc, int Lr, int cc,
                  int cr) {
    auto k = sepstream_kernel<TO, TX>;
    const size_t sm = stream_smem<TX>(Lc, Lr);
    if (int st = smem_optin(op->ctx, (const void*)k, sm)) return st;
    // persistent: the CTAs that stay resident share the chunks evenly
    const int64_t chunks = (int64_t)((op->n1 + SY - 1) / SY) * ((op->n2 + TX - 1) / TX) * batch;
    const int grid = (int)std::min<int64_t>(chunks, (int64_t)op->ctx->sm_count * (TX == 128 ? 2 : 3));
    NYS_CK(op->ctx, launch_pdl(k, grid, 2 * TX, sm, op->ctx->stream, x, y, op->n1, op->n2, batch, (const float*)taps, Lc,
                               Lr, cc, cr));
    NYS_LAUNCH_CK(op->ctx);
    return NYS_OK;
}

template <class TI, class TO, class TC, int T>
int launch_c2d(nys_op* op, const void* x, void* y, int batch, const void* taps) {
    const int kwp = round8(op->kw);
    const size_t sm = c2d_smem<TC>(T, T, op->kh, kwp);
    auto k = corr2d_kernel<TI, TO, TC, T, T>;
    if (int st = smem_optin(op->ctx, (const void*)k, sm)) return st;
    for (int b0 = 0; b0 < batch; b0 += 65535) {     // images in grid.z
        dim3 grid((op->n2 + T - 1) / T, (op->n1 + T - 1) / T, std::min(65535, batch - b0));
        NYS_CK(op->ctx, launch_pdl(k, grid, 256, sm, op->ctx->stream, (const TI*)x + (size_t)b0 * op->N,
                                   (TO*)y + (size_t)b0 * op->N, op->n1, op->n2, (const TC*)taps, op->kh, kwp,
                                   (op->kh - 1) / 2, (op->kw - 1) / 2));
        NYS_LAUNCH_CK(op->ctx);
    }
    return NYS_OK;
}

template <class TC>
constexpr int largest_tile() { return sizeof(TC) == 8 ? 32 : 64; }

// Tile side (largest, a half or a quarter of it), the one whose slowest SM has
// the least work: whole tiles to an SM times the FMAs of a tile with its halo
// (work(T)) and 66 thousand more for staging it and its barriers (float32
// normal operators of 13 to 49 taps on 1 to 400 images of 64 to 512 pixels a
// side: 0.6 us a tile and 9 us per million FMAs fit tiles of 16, 32 and 64
// within 15%).  One 512 x 512 image in float32 takes 32 (64 leaves more than half
// of the SMs idle), a 64 x 64 one in float64 takes 8 (64 CTAs instead of 4:
// 21 to 16 us per normal).
template <class Work>
int pick_tile(const nys_op* op, int batch, int largest, Work&& work) {
    int best = largest;
    double best_cost = 1e300;
    for (int T = largest; T >= largest / 4; T /= 2) {
        const int64_t tiles = (int64_t)((op->n1 + T - 1) / T) * ((op->n2 + T - 1) / T) * batch;
        const double cost = (double)((tiles + op->ctx->sm_count - 1) / op->ctx->sm_count) * (work(T) + 66e3);
        if (cost < best_cost) best = T, best_cost = cost;
    }
    return best;
}

template <class TI, class TO, class TC>
int sep_typed(nys_op* op, const void* x, void* y, int batch, const void* taps, int Lc, int Lr, int cc, int cr) {
    const int Lcp = round8(Lc), Lrp = round8(Lr), SM = op->ctx->sm_count;
    int T = sizeof(TC) == 8 ? 0 : op->blur_tile;      // 0: by size
    // the largest kernel taken: the one that fits the largest tile (or the tuned one)
    if (sep_smem<TC>(T ? T : largest_tile<TC>(), T ? T : largest_tile<TC>(), Lcp, Lrp) > 227 * 1024)
        return fail(op->ctx, NYS_EINVAL, "blur kernel too wide for the shared-memory tile");
    if constexpr (std::is_same<TI, __nv_bfloat16>::value) {
        // Strips with the row pass carried down, TX columns wide with the least
        // padding, when there is a chunk for every other SM; few taps on small
        // images stay with the tiles (13 taps a side at 128 x 128: 45 against
        // 43 us for 400 images; 49 taps at 64 x 64: 22.6 against 26.6 us)
        const int chunks = (op->n1 + SY - 1) / SY;
        const int TX = op->n2 > 64 && (op->n2 + 127) / 128 * 128 - op->n2 < 64 ? 128 : 64;
        const size_t sm = TX == 128 ? stream_smem<128>(Lc, Lr) : stream_smem<64>(Lc, Lr);
        const int64_t strips = (int64_t)((op->n2 + TX - 1) / TX) * batch;
        if (sm <= (TX == 128 ? 113 : 75) * 1024 && Lr <= 64 && op->n2 % 2 == 0 && cr % 2 == 0 &&
            ((uintptr_t)x & 3) == 0 && 2 * strips * chunks >= SM && (Lc + Lr >= 40 || op->n1 >= 190)) {
            const auto* xb = (const __nv_bfloat16*)x;
            return TX == 128 ? launch_stream<TO, 128>(op, xb, (TO*)y, batch, taps, Lc, Lr, cc, cr)
                             : launch_stream<TO, 64>(op, xb, (TO*)y, batch, taps, Lc, Lr, cc, cr);
        }
    }
    auto work = [&](int t) { return (double)(t + Lcp) * t * Lrp + (double)t * t * Lcp; };
    if (!T) T = pick_tile(op, batch, largest_tile<TC>(), work);
    if constexpr (sizeof(TC) == 8) {
        if (T == 8) return launch_sep<TI, TO, TC, 8>(op, x, y, batch, taps, Lcp, Lrp, cc, cr);
    } else {
        if (T == 64) return launch_sep<TI, TO, TC, 64>(op, x, y, batch, taps, Lcp, Lrp, cc, cr);
    }
    if (T == 16) return launch_sep<TI, TO, TC, 16>(op, x, y, batch, taps, Lcp, Lrp, cc, cr);
    return launch_sep<TI, TO, TC, 32>(op, x, y, batch, taps, Lcp, Lrp, cc, cr);
}

template <class TI, class TO, class TC>
int c2d_typed(nys_op* op, const void* x, void* y, int batch, const void* taps) {
    int T = sizeof(TC) == 8 ? 0 : op->blur_tile;      // 0: by size
    const int kwp = round8(op->kw);
    auto work = [&](int t) { return (double)t * t * op->kh * kwp + 4.0 * (t + op->kh) * (t + kwp); };
    if (c2d_smem<TC>(T ? T : largest_tile<TC>(), T ? T : largest_tile<TC>(), op->kh, kwp) > 227 * 1024)
        return fail(op->ctx, NYS_EINVAL, "blur kernel too large for the shared-memory tile");
    if (!T) T = pick_tile(op, batch, largest_tile<TC>(), work);
    if constexpr (sizeof(TC) == 8) {
        if (T == 8) return launch_c2d<TI, TO, TC, 8>(op, x, y, batch, taps);
    } else {
        if (T == 64) return launch_c2d<TI, TO, TC, 64>(op, x, y, batch, taps);
    }
    if (T == 16) return launch_c2d<TI, TO, TC, 16>(op, x, y, batch, taps);
    return launch_c2d<TI, TO, TC, 32>(op, x, y, batch, taps);
}

template <class TI, class TO, class TC>
int blur_typed(nys_op* op, int which, const void* x, void* y, int batch) {
    if (op->separable) {
        if (which == 2)
            return sep_typed<TI, TO, TC>(op, x, y, batch, op->taps_nrm, op->Lc_n, op->Lr_n, op->cc_n, op->cr_n);
        return sep_typed<TI, TO, TC>(op, x, y, batch, which == 0 ? op->taps_fwd : op->taps_adj, op->Lc_f, op->Lr_f,
                                     op->cc_f, op->cr_f);
    }
    if (which != 2) return c2d_typed<TI, TO, TC>(op, x, y, batch, which == 0 ? op->taps_fwd : op->taps_adj);
    // non-separable normal: H^T (H x) through the intermediate buffer, in chunks
    for (int b0 = 0; b0 < batch; b0 += op->chunk) {
        const int nb = std::min(op->chunk, batch - b0);
        const size_t in_off = (size_t)b0 * op->N * sizeof(TI), out_off = (size_t)b0 * op->N * sizeof(TO);
        if (int st = c2d_typed<TI, TC, TC>(op, (const char*)x + in_off, op->inter, nb, op->taps_fwd)) return st;
        if (int st = c2d_typed<TC, TO, TC>(op, op->inter, (char*)y + out_off, nb, op->taps_adj)) return st;
    }
    return NYS_OK;
}

template <class TI, class TO, class TC>
int decim_typed(nys_op* op, int which, const void* x, void* y, int batch) {
    cudaStream_t s = op->ctx->stream;
    const TC* h = (const TC*)op->taps_fwd;
    auto grid = [&](int64_t outs) { return (int)std::min<int64_t>((outs + 63) / 64, (int64_t)op->ctx->sm_count * 32); };
    if (which == 0) {
        NYS_CK(op->ctx, launch_pdl(decim_fwd_kernel<TI, TO, TC>, grid(batch * op->M), 64, 0, s, (const TI*)x, (TO*)y, op->n1,
                                   op->n2, op->decim, h, op->kh, op->kw, batch));
        NYS_LAUNCH_CK(op->ctx);
        return NYS_OK;
    }
    if (which == 1) {
        NYS_CK(op->ctx, launch_pdl(decim_adj_kernel<TI, TO, TC>, grid(batch * op->N), 64, 0, s, (const TI*)x, (TO*)y, op->n1,
                                   op->n2, op->decim, h, op->kh, op->kw, batch));
        NYS_LAUNCH_CK(op->ctx);
        return NYS_OK;
    }
    for (int b0 = 0; b0 < batch; b0 += op->chunk) {
        const int nb = std::min(op->chunk, batch - b0);
        NYS_CK(op->ctx, launch_pdl(decim_fwd_kernel<TI, TC, TC>, grid(nb * op->M), 64, 0, s, (const TI*)x + (size_t)b0 * op->N,
                                   (TC*)op->inter, op->n1, op->n2, op->decim, h, op->kh, op->kw, nb));
        NYS_LAUNCH_CK(op->ctx);
        NYS_CK(op->ctx, launch_pdl(decim_adj_kernel<TC, TO, TC>, grid(nb * op->N), 64, 0, s, (const TC*)op->inter,
                                   (TO*)y + (size_t)b0 * op->N, op->n1, op->n2, op->decim, h, op->kh, op->kw, nb));
        NYS_LAUNCH_CK(op->ctx);
    }
    return NYS_OK;
}

template <template <class, class, class> class F>
struct Dispatch;

// dtype dispatch shared by blur and decimation
template <class Fn>
int dispatch_io(nys_op* op, int in_dt, int out_dt, Fn&& fn) {
    if (op->dtype == NYS_F64) {
        if (in_dt != NYS_F64 || out_dt != NYS_F64) return fail(op->ctx, NYS_EINVAL, "f64 operator needs f64 data");
        return fn((double*)nullptr, (double*)nullptr, (double*)nullptr);
    }
    const bool ib = in_dt == NYS_BF16, ob = out_dt == NYS_BF16;
    if ((in_dt != NYS_F32 && !ib) || (out_dt != NYS_F32 && !ob))
        return fail(op->ctx, NYS_EINVAL, "f32 operator takes f32 or bf16 data");
    if (!ib && !ob) return fn((float*)nullptr, (float*)nullptr, (float*)nullptr);
    if (ib && ob) return fn((__nv_bfloat16*)nullptr, (__nv_bfloat16*)nullptr, (float*)nullptr);
    if (ib) return fn((__nv_bfloat16*)nullptr, (float*)nullptr, (float*)nullptr);
    return fn((float*)nullptr, (__nv_bfloat16*)nullptr, (float*)nullptr);
}

template <class TC>
int upload(nys_op* op, const std::vector<double>& v, void** dst) {
    std::vector<TC> t(v.begin(), v.end());
    NYS_CK(op->ctx, cudaMalloc(dst, t.size() * sizeof(TC) + 16));
    NYS_CK(op->ctx, cudaMemcpy(*dst, t.data(), t.size() * sizeof(TC), cudaMemcpyHostToDevice));
    return NYS_OK;
}

std::vector<double> autocorr(const std::vector<double>& u) {
    const int k = (int)u.size();
    std::vector<double> g(2 * k - 1, 0.0);
    for (int a = 0; a < k; ++a)
        for (int b = 0; b < k; ++b) g[(b - a) + (k - 1)] += u[a] * u[b];
    return g;
}

}  // namespace

int blur_setup(nys_op* op) {
    const int kh = op->kh, kw = op->kw;
    const std::vector<double>& h = op->h;
    // rank-one test: h = u v^T with u = h[:, b*], v = h[a*, :] / h[a*, b*]
    int as = 0, bs = 0;
    double hmax = 0.0;
    for (int a = 0; a < kh; ++a)
        for (int b = 0; b < kw; ++b)
            if (std::fabs(h[a * kw + b]) > hmax) hmax = std::fabs(h[a * kw + b]), as = a, bs = b;
    std::vector<double> u(kh), v(kw);
    for (int a = 0; a < kh; ++a) u[a] = h[a * kw + bs];
    for (int b = 0; b < kw; ++b) v[b] = hmax > 0 ? h[as * kw + b] / h[as * kw + bs] : 0.0;
    double res = 0.0;
    for (int a = 0; a < kh; ++a)
        for (int b = 0; b < kw; ++b) res = std::max(res, std::fabs(h[a * kw + b] - u[a] * v[b]));
    op->separable = hmax > 0 && res <= 1e-13 * hmax;
    const bool f64 = op->dtype == NYS_F64;
    auto up = [&](const std::vector<double>& t, void** dst) {
        return f64 ? upload<double>(op, t, dst) : upload<float>(op, t, dst);
    };
    int st;
    if (op->kind == NYS_OP_BLUR_DECIM) {
        if ((st = up(h, &op->taps_fwd))) return st;
    } else if (op->separable) {
        // forward: [u | v], adjoint: [flip u | flip v]; each padded to a multiple of 8
        op->Lc_f = kh;
        op->Lr_f = kw;
        const int Lcf = round8(kh), Lrf = round8(kw);
        op->cc_f = (kh - 1) / 2;
        op->cr_f = (kw - 1) / 2;
        std::vector<double> f(Lcf + Lrf, 0.0), g(Lcf + Lrf, 0.0);
        for (int a = 0; a < kh; ++a) f[a] = u[a], g[a] = u[kh - 1 - a];
        for (int b = 0; b < kw; ++b) f[Lcf + b] = v[b], g[Lcf + b] = v[kw - 1 - b];
        if ((st = up(f, &op->taps_fwd))) return st;
        if ((st = up(g, &op->taps_adj))) return st;
        std::vector<double> gu = autocorr(u), gv = autocorr(v);
        op->Lc_n = (int)gu.size();
        op->Lr_n = (int)gv.size();
        const int Lcn = round8(op->Lc_n), Lrn = round8(op->Lr_n);
        op->cc_n = kh - 1;
        op->cr_n = kw - 1;
        std::vector<double> n(Lcn + Lrn, 0.0);
        for (size_t a = 0; a < gu.size(); ++a) n[a] = gu[a];
        for (size_t b = 0; b < gv.size(); ++b) n[Lcn + b] = gv[b];
        if ((st = up(n, &op->taps_nrm))) return st;
    } else {
        const int kwp = round8(kw);
        std::vector<double> f((size_t)kh * kwp, 0.0), g((size_t)kh * kwp, 0.0);
        for (int a = 0; a < kh; ++a)
            for (int b = 0; b < kw; ++b) {
                f[a * kwp + b] = h[a * kw + b];
                g[a * kwp + b] = h[(kh - 1 - a) * kw + (kw - 1 - b)];
            }
        if ((st = up(f, &op->taps_fwd))) return st;
        if ((st = up(g, &op->taps_adj))) return st;
    }
    // intermediate for two-pass normals: 16 images of the computing type
    const bool twopass = op->kind == NYS_OP_BLUR_DECIM || !op->separable;
    if (twopass) {
        op->chunk = 16;
        NYS_CK(op->ctx, cudaMalloc(&op->inter, (size_t)op->chunk * op->N * (f64 ? 8 : 4)));
    }
    return NYS_OK;
}

int blur_run(nys_op* op, int which, const void* x, void* y, int batch, int in_dt, int out_dt) {
    return dispatch_io(op, in_dt, out_dt, [&](auto* ti, auto* to, auto* tc) {
        using TI = std::remove_pointer_t<decltype(ti)>;
        using TO = std::remove_pointer_t<decltype(to)>;
        using TC = std::remove_pointer_t<decltype(tc)>;
        return blur_typed<TI, TO, TC>(op, which, x, y, batch);
    });
}

int decim_run(nys_op* op, int which, const void* x, void* y, int batch, int in_dt, int out_dt) {
    return dispatch_io(op, in_dt, out_dt, [&](auto* ti, auto* to, auto* tc) {
        using TI = std::remove_pointer_t<decltype(ti)>;
        using TO = std::remove_pointer_t<decltype(to)>;
        using TC = std::remove_pointer_t<decltype(tc)>;
        return decim_typed<TI, TO, TC>(op, which, x, y, batch);
    });
}

}  // namespace nys
