// Fan-beam ray transform (the second CT geometry of the experiments) and its
// exact transpose, discretised with Joseph's method like the parallel-beam
// one.  A point source on a circle of radius R about the image centre and a
// flat detector at distance D from it: at angle theta, e_s = (cos, sin),
// e_d = (-sin, cos), source S = R e_s, detector centre S - D e_s, bin m at
// offset u_m = (m - (n_bins-1)/2) du along e_d; ray m runs from S to its bin
// along d = -D e_s + u_m e_d.  A ray with |d_y| >= |d_x| samples every row i
// at column position u = a + b i (b = d_x/d_y), weight |d|/|d_y|; any other
// ray samples every column j at row position u = a + b j (b = d_y/d_x),
// weight |d|/|d_x|; linear interpolation between floor(u) and floor(u) + 1,
// zero outside.  Pixel (i, j) sits at (j - c2, i - c1).
//
// The per-ray a, b come from a host table in float64; float32 operators keep
// them as integers with 40 fraction bits and step positions in fixed point (40
// fraction bits in the forward, 27 in the adjoint), so that no weight carries
// the rounding of a float position.
//
// Lanes (ray_lanes.cuh).  Over a full circle, -theta sees the image turned
// upside down with its bins reversed exactly as theta sees the image, and with
// an even number of angles pi - theta and pi + theta do the same with the
// left-right mirrored and the half-turned image: a single image has two or
// four lanes too, whatever its shape.  An orbit whose angles disagree on a
// ray's kind (a ray at exactly 45 degrees) is taken one angle at a time.
//
// Kernels: lane_prep, fan_fwd (rays), lane_bins, fan_adj (pixels), lane_sum.
#include "ray_lanes.cuh"

#include <cmath>
#include <iterator>
#include <memory>
#include <vector>

namespace nys {
namespace {

// a run of bins of one base entry whose rays step along the same kind of line
struct FanSeg {
    int kb, lo, hi;       // bins lo .. hi - 1
    int rs;               // row-step rays
    int sgn;              // sign of dm / d(position along the line)
    int pad;
};

template <class TC> struct FanRay { using type = longlong2; };     // (1 + a, b), 40 fraction bits
template <> struct FanRay<double> { using type = double2; };       // (1 + a, b)

template <class TC>
struct FanTab {
    const typename FanRay<TC>::type* ray;   // [n_angles][n_bins]
    const TC* w;                            // [n_angles][n_bins]
    const unsigned char* rs;                // [n_angles][n_bins] row-step flag
    const float2* ang;                      // [n_angles]: cos, sin
};

__device__ __forceinline__ void ray_at(RayPos<float>& p, const longlong2& r, int l) { p.set40(r.x + l * r.y); }
__device__ __forceinline__ void ray_at(RayPos<double>& p, const double2& r, int l) { p.set(fma(r.y, (double)l, r.x)); }
__device__ __forceinline__ void ray_step(RayPos<float>& p, const longlong2& r) { p.set40(r.y); }
__device__ __forceinline__ void ray_step(RayPos<double>& p, const double2& r) { p.set(r.y); }
__device__ __forceinline__ float ray_a(const longlong2& r) { return (float)r.x * 0x1p-40f; }
__device__ __forceinline__ float ray_a(const double2& r) { return (float)r.x; }
__device__ __forceinline__ float ray_b(const longlong2& r) { return (float)r.y * 0x1p-40f; }
__device__ __forceinline__ float ray_b(const double2& r) { return (float)r.y; }

// Forward: a warp takes 32 CB consecutive bins of one base entry and steps
// along a SEG-th of the lines its rays cross, as radon_fwd_kernel; every ray
// has a slope of its own, and a warp whose rays are of both kinds walks its
// lines once for each.  One 512 x 512 image, 720 angles x 1024 bins: 99 us, the
// L1 data pipe 66% busy (one thread per ray, reading columns of the row-major
// image for column-step rays, took 885 us).  Registers for three CTAs to an SM
// (one image 99 against 104 us with fewer), and a line at a time where a lane
// has two bins (32 images: 2.57 ms, two lines 3.14).
template <class TC, class TO, int IB, int CB, int SEG, bool LANES>
__global__ void __launch_bounds__(256, 3) fan_fwd_kernel(const Lanes<TC, IB>* __restrict__ rows,
                                                         const Lanes<TC, IB>* __restrict__ cols, void* __restrict__ yv,
                                                         int n1, int n2, int n_angles, int n_bins, int batch,
                                                         FanTab<TC> tab, LaneSet set) {
    pdl_enter();
    constexpr int FANG = 8 / SEG;
    __shared__ Lanes<TC, IB> part[SEG > 1 ? SEG - 1 : 1][SEG > 1 ? FANG : 1][SEG > 1 ? CB : 1][32];
    const int nch = (n_bins + 32 * CB - 1) / (32 * CB), ch = blockIdx.x % nch, lane = threadIdx.x & 31;
    const int wa = (threadIdx.x >> 5) % FANG, seg = (threadIdx.x >> 5) / FANG;
    const int kb_me = blockIdx.x / nch * FANG + wa, g = blockIdx.y;
    const int kb = min(kb_me, set.n_base - 1);      // a warp without an angle repeats the last one, unwritten
    const int* ang = set.ang + kb * set.V;
    const size_t r0 = (size_t)ang[0] * n_bins;
    const int m0 = ch * 32 * CB;
    TC acc[CB][IB], wt[CB];
    typename FanRay<TC>::type ray[CB];
    int rs[CB], any[2] = {0, 0};
#pragma unroll
    for (int c = 0; c < CB; ++c) {
        const int m = min(m0 + 32 * c + lane, n_bins - 1);
        ray[c] = tab.ray[r0 + m];
        wt[c] = tab.w[r0 + m];
        rs[c] = tab.rs[r0 + m];
        any[rs[c]] = 1;
#pragma unroll
        for (int q = 0; q < IB; ++q) acc[c][q] = TC(0);
    }
    for (int kind = 0; kind < 2; ++kind) {
        if (!__any_sync(0xffffffffu, kind ? any[1] : any[0])) continue;
        const int nl = kind ? n1 : n2, na = kind ? n2 : n1;
        const size_t pitch = na + PAD;
        // the lines on which one of the warp's rays is inside the image (with
        // two lines of margin): every other sample adds exactly zero
        int l_beg = nl, l_end = 0;
#pragma unroll
        for (int c = 0; c < CB; ++c) {
            if (rs[c] != kind) continue;
            // 0 <= 1 + a + b l < na + 1 with 1 + a anywhere from a0 - 1 to a0 + 1: the
            // rounding of a moves a slow crossing by as much over |b| lines
            const float a0 = floorf(ray_a(ray[c])), b = ray_b(ray[c]);
            int lo = 0, hi = nl;
            if (fabsf(b) * (float)nl > 1.0f) {
                const float e1 = (-1.0f - a0) / b, e2 = ((float)(na + 2) - a0) / b;
                lo = (int)fmaxf(0.0f, floorf(fminf(e1, e2)) - 2.0f);
                hi = (int)fminf((float)nl, ceilf(fmaxf(e1, e2)) + 3.0f);
            } else if (a0 < -5.0f || a0 > (float)(na + 5)) {
                hi = 0;
            }
            if (lo < hi) {
                l_beg = min(l_beg, lo);
                l_end = max(l_end, hi);
            }
        }
        l_beg = __reduce_min_sync(0xffffffffu, l_beg);
        l_end = __reduce_max_sync(0xffffffffu, l_end);
        if (SEG > 1) {
            const int per = (max(0, l_end - l_beg) + SEG - 1) / SEG;
            l_beg += seg * per;
            l_end = min(l_end, l_beg + per);
        }
        RayPos<TC> pos[CB], dt[CB];
#pragma unroll
        for (int c = 0; c < CB; ++c) {
            ray_at(pos[c], ray[c], l_beg);
            ray_step(dt[c], ray[c]);
        }
        const unsigned last = na + 1;   // a position outside [-1, na) reads the two zeros after the line
        const Lanes<TC, IB>* line = (kind ? rows : cols) + ((size_t)g * nl + l_beg) * pitch;
#pragma unroll (CB == 2 ? 1 : 2)
        for (int l = l_beg; l < l_end; ++l, line += pitch) {
#pragma unroll
            for (int c = 0; c < CB; ++c) {
                const unsigned e = rs[c] == kind ? min((unsigned)pos[c].index(), last) : last;
                TC w0, w1;
                pos[c].weights(w0, w1);
                pos[c].step(dt[c]);
                const Lanes<TC, IB> a = line[e], b = line[e + 1];
#pragma unroll
                for (int q = 0; q < IB; ++q) acc[c][q] = fma(w1, b.v[q], fma(w0, a.v[q], acc[c][q]));
            }
        }
    }
    if constexpr (SEG > 1) {
#pragma unroll
        for (int c = 0; c < CB; ++c)
            if (seg) {
                Lanes<TC, IB> w;
#pragma unroll
                for (int q = 0; q < IB; ++q) w.v[q] = acc[c][q];
                part[seg - 1][wa][c][lane] = w;
            }
        __syncthreads();
        if (seg) return;
#pragma unroll
        for (int z = 0; z < SEG - 1; ++z)
#pragma unroll
            for (int c = 0; c < CB; ++c)
#pragma unroll
                for (int q = 0; q < IB; ++q) acc[c][q] += part[z][wa][c][lane].v[q];
    }
#pragma unroll
    for (int c = 0; c < CB; ++c) {
        const int m = m0 + 32 * c + lane;
        if (m >= n_bins || kb_me >= set.n_base) continue;
        if constexpr (LANES) {
            Lanes<TC, IB> w;
#pragma unroll
            for (int q = 0; q < IB; ++q) w.v[q] = ang[q % set.V] >= 0 ? wt[c] * acc[c][q] : TC(0);
            ((Lanes<TC, IB>*)yv)[((size_t)g * set.n_base + kb) * n_bins + m] = w;
        } else {
            TO* y = (TO*)yv;
#pragma unroll
            for (int q = 0; q < IB; ++q) {
                const int b = g * (IB / set.V) + q / set.V, a = ang[q % set.V];
                const int mq = set.sym(q % set.V) & LANE_REV ? n_bins - 1 - m : m;
                if (b < batch && a >= 0) stf(y + ((size_t)b * n_angles + a) * n_bins + mq, wt[c] * acc[c][q]);
            }
        }
    }
}

constexpr int ATS = 32;       // tile side; a thread holds 4 pixels, 8 rows apart
constexpr int AWIN = 192;     // staged bins per segment and piece
constexpr int AJ = 4;         // segments per round
constexpr int AKMAX = 64;     // most candidate bins per pixel of the unrolled path

// Offsets of the rays from a pixel, in fixed point that wraps at 2^(bits -
// frac) pixels (32 in float32, 512 in float64): an offset more than a pixel
// below that keeps a weight of zero (the jobs below see to it)
template <class TC> struct FanOff;
template <> struct FanOff<float> {
    using S = int;
    using U = unsigned;
    struct alignas(8) E { U u, b; };
    // position of ray r at line l0 relative to p0, and its slope (l0 the tile's
    // middle line: the slope's rounding counts at most half a tile's times)
    static __device__ __forceinline__ E make(const longlong2& r, int l0, int p0, int frac) {
        const int sh = 40 - frac;
        const long long h = 1ll << (sh - 1);
        return E{(U)((r.x + l0 * r.y - ((long long)(p0 + 1) << 40) + h) >> sh), (U)((r.y + h) >> sh)};
    }
};
template <> struct FanOff<double> {
    using S = long long;
    using U = unsigned long long;
    struct alignas(16) E { U u, b; };
    static __device__ __forceinline__ E make(const double2& r, int l0, int p0, int frac) {
        const double range = ldexp(1.0, 63 - frac), u = fma(r.y, (double)l0, r.x - (double)(p0 + 1));
        return E{(U)__double2ll_rn(ldexp(u - 2.0 * range * rint(u / (2.0 * range)), frac)),
                 (U)__double2ll_rn(ldexp(r.y, frac))};
    }
};

// a segment as a tile sees it: bins near a point (r, p) (line, position from
// the tile's corner) are around m = mc + g (a0 + ar r + ap p) / (d0 + dr r +
// dp p) from the first staged bin on, to within eps bins
struct FanJob {
    int kb, lo, hi, rs, sgn;
    int mlo, wn, K;           // first staged bin, bins staged, candidates per pixel (0: pixel by pixel)
    float mc, a0, ar, ap, d0, dr, dp, eps;
};

// Adjoint: one CTA per (32 x 32 tile, group of lanes, range of segments).  The
// segments that reach the tile are listed, then taken AJ at a time: their bins
// near the tile are staged in shared memory (offset and slope of the ray in
// tile coordinates, the lanes scaled by the ray's weight), and every pixel
// walks the K bins that can pass within one pixel of it along the line.  K is
// what the pixel with most of them needs; where so many bins reach past the
// wrapping offsets from another pixel (depths several times apart within the
// tile), every pixel finds its own first and last bin.  A
// quarter warp holds 4 x 2 pixels, so that its bins stay close for both kinds
// of ray.  Windows larger than AWIN bins are taken in pieces.
// Bound by instruction issue (about 60%) and the uneven tiles: one 512 x 512
// image, 720 angles x 1024 bins, 0.21 ms, where one thread per pixel testing
// every candidate ray against float tables in L2 took 4.56 ms.
template <class TC, class TO, int IB, bool PLANES>
__global__ void __launch_bounds__(256) fan_adj_kernel(const Lanes<TC, IB>* __restrict__ s, TO* __restrict__ out,
                                                      int n1, int n2, int n_bins, int batch, int ns,
                                                      const FanSeg* __restrict__ segs, int n_seg, float R, float G,
                                                      int frac, FanTab<TC> tab, LaneSet set) {
    pdl_enter();
    using FO = FanOff<TC>;
    using L = Lanes<TC, IB>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    L* win = reinterpret_cast<L*>(smem_raw);                                              // [AJ][AWIN]
    typename FO::E* off = reinterpret_cast<typename FO::E*>(win + AJ * AWIN);       // [AJ][AWIN]
    FanJob* job = reinterpret_cast<FanJob*>(off + AJ * AWIN);                       // [256]
    __shared__ int s_cnt[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tx = (lane & 3) | (lane >> 1 & 4) | (warp & 3) << 3;
    const int ty = (lane >> 2 & 1) | (lane >> 3 & 2) | (warp >> 2) << 2;
    // mirror lanes leave base angles of the first quadrant: the tiles nearest
    // to their sources, the last ones, have most bins per pixel and go first
    const int i0 = (gridDim.y - 1 - blockIdx.y) * ATS, j0 = (gridDim.x - 1 - blockIdx.x) * ATS;
    const int g = blockIdx.z / ns, z = blockIdx.z - g * ns;
    const int per = (n_seg + ns - 1) / ns, q_beg = z * per, q_end = min(n_seg, q_beg + per);
    const L* sg = s + (size_t)g * set.n_base * n_bins;
    // offsets below this many pixels do not wrap onto the hat function
    const float reach = ldexpf(1.0f, 8 * (int)sizeof(typename FO::U) - frac) - 2.0f;
    TC acc[4][IB];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int q = 0; q < IB; ++q) acc[u][q] = TC(0);
    const float ti = (float)(min(ATS, n1 - i0) - 1), tj = (float)(min(ATS, n2 - j0) - 1);
    const TC one = (TC)ldexp(1.0, frac), inv_one = (TC)ldexp(1.0, -frac);
    for (int qb = q_beg; qb < q_end; qb += 256) {
        // ---- the segments of this block of 256 that reach the tile, in order
        FanJob J;
        bool hit = false;
        if (qb + (int)threadIdx.x < q_end) {
            const FanSeg sgm = segs[qb + threadIdx.x];
            const float2 e = tab.ang[set.ang[sgm.kb * set.V]];
            const float px = (float)j0 - 0.5f * (float)(n2 - 1), py = (float)i0 - 0.5f * (float)(n1 - 1);
            J.kb = sgm.kb, J.lo = sgm.lo, J.hi = sgm.hi, J.rs = sgm.rs, J.sgn = sgm.sgn;
            J.a0 = -px * e.y + py * e.x;             // (P - S) . e_d = P . e_d
            J.d0 = R - (px * e.x + py * e.y);
            J.ar = sgm.rs ? e.x : -e.y, J.ap = sgm.rs ? -e.y : e.x;
            J.dr = sgm.rs ? -e.y : -e.x, J.dp = sgm.rs ? -e.x : -e.y;
            const float tr = sgm.rs ? ti : tj, tp = sgm.rs ? tj : ti, sf = (float)sgm.sgn;
            const float cb = 0.5f * (float)(n_bins - 1);
            // lower edge m(p - sgn) and upper edge m(p + sgn) over the tile's corners
            float lo_min = 3e38f, lo_max = -3e38f, hi_max = -3e38f;
            float d_min = 3e38f, d_max = 0.0f, a_max = 0.0f, num = 0.0f, num_min = 3e38f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float r = c & 1 ? tr : 0.0f, p = c & 2 ? tp : 0.0f;
                const float a = J.a0 + J.ar * r + J.ap * p, d = J.d0 + J.dr * r + J.dp * p;
                const float ml = cb + G * (a - sf * J.ap) / (d - sf * J.dp);
                const float mh = cb + G * (a + sf * J.ap) / (d + sf * J.dp);
                lo_min = fminf(lo_min, ml), lo_max = fmaxf(lo_max, ml), hi_max = fmaxf(hi_max, mh);
                d_min = fminf(d_min, d - fabsf(J.dp)), d_max = fmaxf(d_max, d + fabsf(J.dp));
                a_max = fmaxf(a_max, fabsf(a));
                const float nm = fabsf(J.ap * d - a * J.dp);
                num = fmaxf(num, nm), num_min = fminf(num_min, nm);
            }
            // float rounding of m, in bins: eight units of 2^-24 of the terms of a and
            // d (512 x 512, two bins a pixel: 0.001), and a floor well above the usual
            const float terms = fabsf(px) + fabsf(py) + 64.0f;
            J.eps = 0.01f + 0x1p-21f * (G / d_min) * (terms + (a_max / d_min) * (R + terms));
            hit = lo_min < (float)J.hi + 1.0f && hi_max > (float)J.lo - 1.0f;
            // at most span + 1 integers lie between the edges; span from the
            // largest dm/dp on the tile
            const float span = 2.0f * G * num / (d_min * d_min);
            J.K = (int)fminf(span + 4.0f * J.eps, 1.0e6f) + 1;
            J.mlo = (int)floorf(lo_min - J.eps) - 1;
            J.wn = (int)ceilf(fmaxf(lo_max + J.eps + (float)J.K, hi_max)) + 2 - J.mlo;
            J.mc = cb - (float)J.mlo;
            // K bins on from m(p - sgn) a ray is K d^2 / (G num - K d |dp|) pixels away
            // at most (p as a function of m, inverted)
            const float Kd = (float)J.K * d_max;
            if (J.wn > AWIN || J.K > AKMAX || !(Kd * d_max < reach * (G * num_min - Kd * fabsf(J.dp)))) J.K = 0;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, hit);
        __syncthreads();                // the previous list is consumed
        if (lane == 0) s_cnt[warp] = __popc(bal);
        __syncthreads();
        int at = __popc(bal & ((1u << lane) - 1u)), nj = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            if (w < warp) at += s_cnt[w];
            nj += s_cnt[w];
        }
        if (hit) job[at] = J;
        __syncthreads();
        for (int jb = 0; jb < nj; jb += AJ) {
            const int njr = min(AJ, nj - jb);
            int pieces = 1;
            for (int a = 0; a < njr; ++a) pieces = max(pieces, (job[jb + a].wn + AWIN - 1) / AWIN);
            for (int pc = 0; pc < pieces; ++pc) {
                if (jb | pc) __syncthreads();          // the previous windows are consumed
                for (int t = threadIdx.x; t < njr * AWIN; t += 256) {
                    const int a = t / AWIN, w = t - a * AWIN, wg = pc * AWIN + w;
                    const FanJob& J = job[jb + a];
                    if (wg >= J.wn) continue;
                    const int m = J.mlo + wg;
                    L v;
                    typename FO::E e{0, 0};
#pragma unroll
                    for (int q = 0; q < IB; ++q) v.v[q] = TC(0);
                    if (m >= J.lo && m < J.hi) {
                        const size_t ray = (size_t)set.ang[J.kb * set.V] * n_bins + m;
                        v = sg[(size_t)J.kb * n_bins + m];
                        const TC wt = tab.w[ray] * inv_one;
#pragma unroll
                        for (int q = 0; q < IB; ++q) v.v[q] *= wt;
                        e = FO::make(tab.ray[ray], (J.rs ? i0 : j0) + ATS / 2, J.rs ? j0 : i0, frac);
                    }
                    win[t] = v;
                    off[t] = e;
                }
                __syncthreads();
                for (int a = 0; a < njr; ++a) {
                    const FanJob J = job[jb + a];
                    const int wn = min(J.wn - pc * AWIN, AWIN);
                    if (wn <= 0) continue;
                    const L* wa = win + a * AWIN;
                    const typename FO::E* oa = off + a * AWIN;
                    const float sf = (float)J.sgn, mc = J.mc - (float)(pc * AWIN), eps = J.eps;
                    if (J.K) {
                        int idx[4];
                        typename FO::U r[4], p[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int di = ty + 8 * u, rr = J.rs ? di : tx, pp = J.rs ? tx : di;
                            const float fr = (float)rr, fp = (float)pp - sf;
                            const float m = mc + G * __fdividef(J.a0 + J.ar * fr + J.ap * fp, J.d0 + J.dr * fr + J.dp * fp);
                            idx[u] = max(0, min((int)ceilf(m - eps), wn - J.K));   // in range for pixels of the image
                            r[u] = (typename FO::U)(typename FO::S)(rr - ATS / 2);
                            p[u] = (typename FO::U)pp << frac;
                        }
                        for (int c = 0; c < J.K; ++c) {
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const typename FO::E e = oa[idx[u] + c];
                                const L v = wa[idx[u] + c];
                                const TC d = (TC)(typename FO::S)(e.u + r[u] * e.b - p[u]);
                                // (left out, not multiplied by zero: an infinity or a NaN reaches the
                                // pixels of its ray only)
                                const TC w = one - fabs(d);
                                if (w > TC(0)) {
#pragma unroll
                                    for (int q = 0; q < IB; ++q) acc[u][q] = fma(w, v.v[q], acc[u][q]);
                                }
                            }
                        }
                    } else {
                        // bins far denser or sparser than pixels, or a tile next to the source
                        for (int u = 0; u < 4; ++u) {
                            const int di = ty + 8 * u, rr = J.rs ? di : tx, pp = J.rs ? tx : di;
                            if (i0 + di >= n1 || j0 + tx >= n2) continue;
                            const float fr = (float)rr, fp = (float)pp;
                            const float a = J.a0 + J.ar * fr + J.ap * fp, d = J.d0 + J.dr * fr + J.dp * fp;
                            const float ml = mc + G * __fdividef(a - sf * J.ap, d - sf * J.dp);
                            const float mh = mc + G * __fdividef(a + sf * J.ap, d + sf * J.dp);
                            const int c0 = (int)fmaxf(ceilf(ml - eps), 0.0f);
                            const int c1 = (int)fminf(floorf(mh + eps), (float)(wn - 1));
                            for (int c = c0; c <= c1; ++c) {
                                const typename FO::E e = oa[c];
                                const L v = wa[c];
                                const TC dd = (TC)(typename FO::S)(e.u + (typename FO::U)(typename FO::S)(rr - ATS / 2) * e.b -
                                                                  ((typename FO::U)pp << frac));
                                const TC w = one - fabs(dd);
                                if (w > TC(0)) {
#pragma unroll
                                    for (int q = 0; q < IB; ++q) acc[u][q] = fma(w, v.v[q], acc[u][q]);
                                }
                            }
                        }
                    }
                }
            }
        }
    }
    const size_t N = (size_t)n1 * n2;
    const int j = j0 + tx;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int i = i0 + ty + 8 * u;
        if (i >= n1 || j >= n2) continue;
#pragma unroll
        for (int q = 0; q < IB; ++q) {
            if constexpr (PLANES) {
                int si = i, sj = j;
                lane_src(set.sym(q % set.V), si, sj, n1, n2);
                stf(out + (((size_t)g * ns + z) * IB + q) * N + (size_t)si * n2 + sj, acc[u][q]);
            } else {
                const int b = g * IB + q;
                if (b < batch) stf(out + (size_t)b * N + (size_t)i * n2 + j, acc[u][q]);
            }
        }
    }
}

// ------------------------------------------------------------- launching --

// layout of op->rtab: rays, weights, angles, then the lists of the angle sets
// (V = 1, 2, 4) one after the other, then the row-step flags
template <class TC>
FanTab<TC> fan_tab(const nys_op* op) {
    const size_t RA = (size_t)op->n_angles * op->n_bins;
    const char* p = (const char*)op->rtab;
    FanTab<TC> t;
    t.ray = (const typename FanRay<TC>::type*)p;
    t.w = (const TC*)(t.ray + RA);
    t.ang = (const float2*)(p + op->fan.ang_off);
    t.rs = (const unsigned char*)(p + op->fan.rs_off);
    return t;
}

LaneSet fan_set(const nys_op* op, int V) {
    const nys_fan_set& f = op->fan.set[V / 2];
    LaneSet s;
    s.ang = (const int*)((const char*)op->rtab + f.ang_off);
    s.V = V;
    s.n_base = f.n_base;
    // lane v > 0: upside down, mirrored (both with the bins reversed), half a turn
    s.tf = V == 1 ? 0 : (LANE_FI | LANE_REV) << 4 | (LANE_FJ | LANE_REV) << 8 | (LANE_FI | LANE_FJ) << 12;
    return s;
}

// segment ranges of the adjoint: about 20 CTAs to an SM, at least 16 segments
// each (tiles near the sources take several times the bins of those opposite,
// so few long CTAs leave SMs idle: one 512 x 512 image of 720 angles x 1024
// bins, A^T A with 2 ranges 392 us, 7 ranges 342 us, 11 ranges 329 us, 16 341 us)
int adj_ranges(const nys_op* op, int groups, int n_seg) {
    const int64_t ctas = (int64_t)((op->n1 + ATS - 1) / ATS) * ((op->n2 + ATS - 1) / ATS) * groups;
    const int64_t want = (int64_t)op->ctx->sm_count * 20;
    return (int)std::max<int64_t>(1, std::min<int64_t>({want / ctas, n_seg / 16, 16}));
}

template <class TI, class TO, class TC, int IB, bool LANES>
int fwd_part(nys_op* op, const TI* x, void* y, int nb, int V) {
    const LaneSet set = fan_set(op, V);
    if (int st = lane_prep<TI, TC, IB>(op, x, nb, set, true)) return st;
    const int R = IB / V, groups = (nb + R - 1) / R;
    const auto* rows = (const Lanes<TC, IB>*)op->lines;
    const auto* cols = rows + (size_t)groups * op->n1 * (op->n2 + PAD);
    auto go = [&](auto kernel, int CB, int SEG) {
        const int nch = (op->n_bins + 32 * CB - 1) / (32 * CB), fang = 8 / SEG;
        return launch_pdl(kernel, dim3((unsigned)((set.n_base + fang - 1) / fang * nch), groups), 256, 0,
                          op->ctx->stream, rows, cols, y, op->n1, op->n2, op->n_angles, op->n_bins, nb, fan_tab<TC>(op),
                          set);
    };
    const int64_t warps = (int64_t)set.n_base * ((op->n_bins + 63) / 64) * groups;
    if (warps >= (int64_t)op->ctx->sm_count * 32)
        NYS_CK(op->ctx, go(fan_fwd_kernel<TC, TO, IB, 2, 1, LANES>, 2, 1));
    else
        NYS_CK(op->ctx, go(fan_fwd_kernel<TC, TO, IB, 1, 4, LANES>, 1, 4));
    NYS_LAUNCH_CK(op->ctx);
    return NYS_OK;
}

template <class TO, class TC, int IB>
int adj_lanes(nys_op* op, const void* s, TO* x, int nb, int V) {
    const LaneSet set = fan_set(op, V);
    const nys_fan_set& f = op->fan.set[V / 2];
    const int R = IB / V, groups = (nb + R - 1) / R, ns = adj_ranges(op, groups, f.n_seg);
    const dim3 grid((op->n2 + ATS - 1) / ATS, (op->n1 + ATS - 1) / ATS, groups * ns);
    const size_t sm = (size_t)AJ * AWIN * (sizeof(Lanes<TC, IB>) + sizeof(typename FanOff<TC>::E)) +
                      256 * sizeof(FanJob);
    const auto* segs = (const FanSeg*)((const char*)op->rtab + f.seg_off);
    const float Gm = (float)(op->det_dist / op->det_spacing);
    auto go = [&](auto kernel, auto* out) {
        if (int st = smem_optin(op->ctx, (const void*)kernel, sm)) return st;
        NYS_CK(op->ctx, launch_pdl(kernel, grid, 256, sm, op->ctx->stream, (const Lanes<TC, IB>*)s, out, op->n1, op->n2,
                                   op->n_bins, nb, ns, segs, f.n_seg, (float)op->src_dist, Gm, op->fan.frac,
                                   fan_tab<TC>(op), set));
        NYS_LAUNCH_CK(op->ctx);
        return (int)NYS_OK;
    };
    if (V == 1 && ns == 1) return go(fan_adj_kernel<TC, TO, IB, false>, x);
    if (int st = go(fan_adj_kernel<TC, TC, IB, true>, (TC*)op->planes)) return st;
    return lane_sum<TC, TO, IB>(op, x, nb, V, ns);
}

template <class TI, class TO, class TC, int IB>
int part_typed(nys_op* op, int which, const TI* x, TO* y, int nb, int V) {
    if (which == 0) return fwd_part<TI, TO, TC, IB, false>(op, x, y, nb, V);
    if (which == 1) {
        if (int st = lane_bins<TI, TC, IB>(op, x, nb, fan_set(op, V))) return st;
    } else {
        if (int st = fwd_part<TI, TO, TC, IB, true>(op, x, op->inter, nb, V)) return st;
    }
    return adj_lanes<TO, TC, IB>(op, op->inter, y, nb, V);
}

template <class TI, class TO, class TC>
int fan_typed(nys_op* op, int which, const void* x, void* y, int batch) {
    const int64_t in = which == 1 ? op->M : op->N, out = which == 0 ? op->M : op->N;
    for (int b0 = 0; b0 < batch;) {
        const Part p = next_part(op, std::min(op->chunk, batch - b0));
        const TI* xb = (const TI*)x + (size_t)b0 * in;
        TO* yb = (TO*)y + (size_t)b0 * out;
        int st;
        if (p.IB == 4) st = part_typed<TI, TO, TC, 4>(op, which, xb, yb, p.nb, p.V);
        else if (p.IB == 2) st = part_typed<TI, TO, TC, 2>(op, which, xb, yb, p.nb, p.V);
        else st = part_typed<TI, TO, TC, 1>(op, which, xb, yb, p.nb, p.V);
        if (st) return st;
        b0 += p.nb;
    }
    return NYS_OK;
}

}  // namespace

int fanbeam_setup(nys_op* op) {
    const int A = op->n_angles, B = op->n_bins, n1 = op->n1, n2 = op->n2;
    const bool f64 = op->dtype == NYS_F64;
    if (!f64 && std::max(n1, n2) > 2048)
        return fail(op->ctx, NYS_EINVAL, "fan beam: float32 operators take images of at most 2048 lines");
    const double c1 = (n1 - 1) / 2.0, c2 = (n2 - 1) / 2.0, cb = (B - 1) / 2.0;
    const double R = op->src_dist, D = op->det_dist, du = op->det_spacing;
    const size_t RA = (size_t)A * B;
    // rays (two 8-byte words each) and weights as they are uploaded
    const size_t es = f64 ? 8 : 4, w_off = RA * 16;
    std::unique_ptr<char[]> tab(new char[w_off + RA * es]);
    double* abd = (double*)tab.get();
    long long* abq = (long long*)tab.get();
    std::vector<unsigned char> rs(RA), up(RA);     // row-step; sign of the ray's major component
    std::vector<float> ang((size_t)A * 2);
    for (int k = 0; k < A; ++k) {
        const double th = k * (op->span / A);
        const double cs = std::cos(th), sn = std::sin(th);
        const double Sx = R * cs, Sy = R * sn;
        ang[2 * k] = (float)cs;
        ang[2 * k + 1] = (float)sn;
        for (int m = 0; m < B; ++m) {
            const double um = (m - cb) * du;
            const double dx = -D * cs - um * sn, dy = -D * sn + um * cs;
            const double nd = std::sqrt(dx * dx + dy * dy);
            const bool row = std::fabs(dy) >= std::fabs(dx);
            const size_t r = (size_t)k * B + m;
            const double major = row ? dy : dx, minor = row ? dx : dy;
            const double b = minor / major, wt = nd / std::fabs(major);
            const double a = 1.0 + (row ? Sx - (c1 + Sy) * b + c2 : Sy - (c2 + Sx) * b + c1);
            if (f64) {
                abd[2 * r] = a;
                abd[2 * r + 1] = b;
                ((double*)(tab.get() + w_off))[r] = wt;
            } else {
                // a ray that starts further than 2^22 positions outside, with a
                // slope of at most 1, does not reach an image of 2048 lines
                abq[2 * r] = std::llrint(std::min(std::max(a, -4194304.0), 4194304.0) * 0x1p40);
                abq[2 * r + 1] = std::llrint(b * 0x1p40);
                ((float*)(tab.get() + w_off))[r] = (float)wt;
            }
            rs[r] = row;
            up[r] = major > 0.0;
        }
    }
    // the angle sets: orbits of k under the symmetries, split where the angles
    // disagree on the kind of a ray
    std::vector<int> lists[3];
    std::vector<FanSeg> segs[3];
    op->lane_sets = 1;
    for (int vi = 0; vi < 3; ++vi) {
        const int V = 1 << vi;
        if (V > 1 && !(op->span == 2.0 * M_PI && (V == 2 ? A % 2 == 1 : A % 2 == 0))) continue;
        op->lane_sets |= V;
        std::vector<int>& l = lists[vi];
        const int n_orb = V == 1 ? A : A / V + 1;
        for (int k = 0; k < n_orb; ++k) {
            int a[4] = {k, A - k, A / 2 - k, A / 2 + k};
            bool same = true;
            for (int v = 0; v < V; ++v) {
                if (a[v] < 0 || a[v] >= A) a[v] = -1;
                for (int p = 0; p < v; ++p)
                    if (a[p] == a[v]) a[v] = -1;
                if (a[v] < 0 || v == 0) continue;
                const unsigned char *fa = &rs[(size_t)k * B], *fb = &rs[(size_t)a[v] * B];
                same = same && (v == 3 ? std::equal(fa, fa + B, fb)
                                       : std::equal(fa, fa + B, std::reverse_iterator<const unsigned char*>(fb + B)));
            }
            if (same) {
                l.insert(l.end(), a, a + V);
            } else {
                // one angle to an entry: it is its own base, and lane 0
                for (int v = 0; v < V; ++v)
                    if (a[v] >= 0) {
                        l.push_back(a[v]);
                        l.insert(l.end(), V - 1, -1);
                    }
            }
        }
        for (int kb = 0; kb < (int)l.size() / V; ++kb) {
            const size_t r0 = (size_t)l[(size_t)kb * V] * B;
            for (int m = 0; m < B;) {
                int e = m + 1;
                while (e < B && rs[r0 + e] == rs[r0 + m] && up[r0 + e] == up[r0 + m]) ++e;
                // dm/dp has the sign of the ray's y component on a row, of
                // minus its x component on a column
                const int sg = (up[r0 + m] ? 1 : -1) * (rs[r0 + m] ? 1 : -1);
                segs[vi].push_back(FanSeg{kb, m, e, rs[r0 + m], sg, 0});
                m = e;
            }
        }
    }
    // fraction bits of the adjoint's offsets.  A pixel's own bins end within eps
    // (0.01 and some) bins of its neighbours on the line, so a twentieth of the
    // largest spacing of rays along a line has to fit beside the fraction
    const double half_diag = 0.5 * std::sqrt((double)n1 * n1 + (double)n2 * n2);
    const double spacing = std::sqrt(2.0) * du * (R + half_diag + 2.0) / D;
    int ib = f64 ? 9 : 5;
    while (ib < 25 && std::ldexp(1.0, ib) < 8.0 + 0.05 * spacing) ++ib;
    op->fan.frac = (f64 ? 64 : 32) - ib;
    // ---- upload
    size_t total = w_off + RA * es;
    std::vector<std::pair<const void*, std::pair<size_t, size_t>>> puts{{tab.get(), {0, total}}};
    auto put = [&](const void* p, size_t n) {
        const size_t off = (total + 15) & ~size_t(15);
        total = off + n;
        if (n) puts.push_back({p, {off, n}});
        return off;
    };
    op->fan.ang_off = put(ang.data(), ang.size() * sizeof(float));
    for (int vi = 0; vi < 3; ++vi) {
        nys_fan_set& f = op->fan.set[vi];
        f.n_base = (int)(lists[vi].size() >> vi);
        f.n_seg = (int)segs[vi].size();
        f.ang_off = put(lists[vi].data(), lists[vi].size() * sizeof(int));
        f.seg_off = put(segs[vi].data(), segs[vi].size() * sizeof(FanSeg));
    }
    op->fan.rs_off = put(rs.data(), RA);
    NYS_CK(op->ctx, cudaMalloc(&op->rtab, total));
    for (const auto& q : puts)
        NYS_CK(op->ctx, cudaMemcpy((char*)op->rtab + q.second.first, q.first, q.second.second, cudaMemcpyHostToDevice));
    // interleaved sinogram lanes, image lines and the adjoint's planes, for
    // every part that a chunk of images can be cut into
    op->chunk = ray_chunk(op);
    size_t lanes = 0, lines = 0, planes = 0;
    for (int left = 1; left <= op->chunk; ++left) {
        const Part p = next_part(op, left);
        const nys_fan_set& f = op->fan.set[p.V / 2];
        const int Rg = p.IB / p.V, groups = (p.nb + Rg - 1) / Rg, ns = adj_ranges(op, groups, f.n_seg);
        lanes = std::max(lanes, (size_t)groups * f.n_base * p.IB);
        lines = std::max(lines, (size_t)groups * p.IB);
        if (p.V > 1 || ns > 1) planes = std::max(planes, (size_t)groups * ns * p.IB);
    }
    NYS_CK(op->ctx, cudaMalloc(&op->inter, lanes * B * es));
    NYS_CK(op->ctx, cudaMalloc(&op->lines, lines * es * ((size_t)n1 * (n2 + PAD) + (size_t)n2 * (n1 + PAD))));
    if (planes) NYS_CK(op->ctx, cudaMalloc(&op->planes, planes * op->N * es));
    return NYS_OK;
}

int fanbeam_run(nys_op* op, int which, const void* x, void* y, int batch, int in_dt, int out_dt) {
    if (op->dtype == NYS_F64) {
        if (in_dt != NYS_F64 || out_dt != NYS_F64) return fail(op->ctx, NYS_EINVAL, "f64 operator needs f64 data");
        return fan_typed<double, double, double>(op, which, x, y, batch);
    }
    const bool ib = in_dt == NYS_BF16, ob = out_dt == NYS_BF16;
    if (!ib && !ob) return fan_typed<float, float, float>(op, which, x, y, batch);
    if (ib && ob) return fan_typed<__nv_bfloat16, __nv_bfloat16, float>(op, which, x, y, batch);
    if (ib) return fan_typed<__nv_bfloat16, float, float>(op, which, x, y, batch);
    return fan_typed<float, __nv_bfloat16, float>(op, which, x, y, batch);
}

}  // namespace nys
