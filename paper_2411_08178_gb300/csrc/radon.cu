// Parallel-beam ray transform A and its exact transpose A^T (Sec. IV-C, the CT
// forward model), discretised with Joseph's method (P. M. Joseph, "An improved
// algorithm for reprojecting rays through pixel images", IEEE TMI 1982).
//
// Geometry: pixel (i, j) sits at x = j - c2, y = i - c1 (c = (n-1)/2); ray
// (theta_k, t_m) is the line x cos + y sin = t with theta_k = k span / n_angles
// and t_m = m - cb, cb = (n_bins - 1)/2.  A "row-step" angle (|cos| + 1e-9 >=
// |sin|, den = cos) samples the ray once per image row i at column position
//     u(i, m) = c2 + (t_m - (i - c1) sin) / cos
// with linear interpolation between columns floor(u) and floor(u) + 1 and
// weight 1/|den|; a "column-step" angle (den = sin) swaps the roles of rows
// and columns.  Samples that fall outside the image contribute zero.  Seen
// from a pixel, ray m carries the weight
//     max(0, 1/|den| - |m - m*| / den^2),  m* = cb + (j - c2) cos + (i - c1) sin
// (u - position = (m - m*) / den): at most the two bins either side of m*,
// since |den| <= 1.  The forward walks rays, the adjoint gathers per pixel;
// both take their positions from float64 and step them in fixed point, so the
// weights of the two agree to a few roundings of their type (float32 operators:
// 40 fraction bits in the forward, 30 in the adjoint's steps over a 32 x 32
// tile), and the two are transposes of each other to that.
//
// Lanes (ray_lanes.cuh).  Over 180 degrees, angle n_angles - k sees the
// left-right mirrored image exactly as angle k sees the image, and for a
// square image and an even number of angles n_angles/2 -+ k do the same with
// the transposed image and its mirror image: a single image has two or four
// lanes too.
//
// Kernels: lane_prep (images to interleaved lines with zero margins, for
// row-step angles along rows, for column-step ones along columns), radon_fwd
// (rays), lane_bins (a planar sinogram to interleaved lanes), radon_adj
// (pixels), lane_sum (the lanes and angle ranges of one image added up).
#include "ray_lanes.cuh"

#include <cmath>
#include <type_traits>

namespace nys {
namespace {

// per-angle geometry, float64; the ray positions of float32 operators also as
// integers with 40 fraction bits (GB300 issues a float64 operation every 16
// cycles per warp and SM: evaluated in float64, the positions of a few bins per
// warp took as long as a quarter of a warp's lines).  Bins and lines count from
// the middle of the detector and of the image, so that positions near the image
// stay exact whatever the detector's width; the integers may wrap on the way.
struct RGeo {
    double c, inv, t;     // 1 + u(m, l) = c + (m - cb) inv - (l - c_line) t
    long long u0q, invq, tq;         // = u0q + m invq - l tq
    double cs, sn;
    int rs;               // row-step angle
    int b2, l2;           // n_bins - 1, lines - 1
    int m_lo, m_hi;       // rays outside miss the image (further out their integers wrap into it)
};

// the angles of a launch: geo[ang[kb V]] is the geometry of base angle kb
struct RSet : LaneSet {
    const RGeo* geo;
};

__device__ __forceinline__ void ray_at(RayPos<float>& p, const RGeo& g, int m, int l) {
    p.set40(g.u0q + m * g.invq - l * g.tq);
}
__device__ __forceinline__ void ray_at(RayPos<double>& p, const RGeo& g, int m, int l) {
    p.set(fma(m - 0.5 * g.b2, g.inv, fma(-(l - 0.5 * g.l2), g.t, g.c)));
}
__device__ __forceinline__ void ray_step(RayPos<float>& p, const RGeo& g) { p.set40(-g.tq); }
__device__ __forceinline__ void ray_step(RayPos<double>& p, const RGeo& g) { p.set(-g.t); }

// Forward: a warp takes 32 CB consecutive bins of one base angle (CB per lane,
// 32 apart, so that a load's addresses stay together) and steps along a SEG-th
// of the lines its rays cross; the SEG warps of a ray add up in shared memory.
// The 8 / SEG warp groups of a CTA take neighbouring angles and the same bins,
// so that they read the same stripe of the image and L1 serves all but one of
// them (87% of its sectors; one angle per CTA, reading the image from L2 for
// every angle: 35.6 against 25.5 ms for 400 images of 512 x 512, 720 x 736).
// y: planar sinogram of type TO, or the interleaved lanes [g][kb][m] that the
// adjoint reads (LANES).  Bound by the L1 data pipe: 96% busy on that batch,
// where a load's 32 positions, 1 to 1.41 pixels of 16 bytes apart, take about
// 7 wavefronts instead of 4; before the lanes (scalar loads, four images per
// warp) 48.4 ms, and 183 us for one image (now 82 us: 181 base angles leave
// half of the warp slots empty).
// TL: type of the lines, TC or bf16 (a bf16 batch, eight images to a 16-byte
// load: half the L1 traffic per image, 14.0 against 25.5 ms for the batch above).
template <class TL, class TC, class TO, int IB, int CB, int SEG, bool LANES>
__global__ void __launch_bounds__(256) radon_fwd_kernel(const Lanes<TL, IB>* __restrict__ rows,
                                                        const Lanes<TL, IB>* __restrict__ cols, void* __restrict__ yv,
                                                        int n1, int n2, int n_angles, int n_bins, int batch,
                                                        RSet set) {
    pdl_enter();
    constexpr int FANG = 8 / SEG;
    constexpr bool BF = !std::is_same<TL, TC>::value;
    // lines to a loop round: measured, the compiler's order of the loads decides (32
    // images of 4096 x 4096, 90 angles: planar sinograms 21.7 ms with two, 25.2 with
    // four; A^T A 38.3 with two, 34.4 with four)
    constexpr int LU = LANES && !BF ? 4 : 2;
    static_assert(!BF || SEG == 1, "bf16 lines: whole rays");
    __shared__ Lanes<TC, IB> part[SEG > 1 ? SEG - 1 : 1][SEG > 1 ? FANG : 1][SEG > 1 ? CB : 1][32];
    const int nch = (n_bins + 32 * CB - 1) / (32 * CB), ch = blockIdx.x % nch, lane = threadIdx.x & 31;
    const int wa = (threadIdx.x >> 5) % FANG, seg = (threadIdx.x >> 5) / FANG;
    const int kb_me = blockIdx.x / nch * FANG + wa, g = blockIdx.y;
    const int kb = min(kb_me, set.n_base - 1);      // a warp without an angle repeats the last one, unwritten
    const int* ang = set.ang + kb * set.V;
    const RGeo geo = set.geo[ang[0]];
    const int nl = geo.rs ? n1 : n2, na = geo.rs ? n2 : n1;   // lines, positions along a line
    const size_t pitch = na + PAD;
    const Lanes<TL, IB>* src = (geo.rs ? rows : cols) + (size_t)g * nl * pitch;
    const int m0 = ch * 32 * CB;
    // the lines where a sample of the warp's bins can land in [-1, na) form
    // one interval (u is monotone in m), taken with two lines of margin;
    // outside it every sample is out of range and adds exactly zero
    RayPos<TC> pos[CB], dt;
    ray_step(dt, geo);
    ray_at(pos[0], geo, m0, 0);
    const float qa = (float)(pos[0].index() - 1);
    ray_at(pos[0], geo, min(m0 + 32 * CB - 1, n_bins - 1), 0);
    const float qb = (float)(pos[0].index() - 1);
    const float qmin = fminf(qa, qb), qmax = fmaxf(qa, qb) + 1.0f, tl = (float)geo.tq * 0x1p-40f;
    int l_beg = 0, l_end = nl;
    if (fabsf(tl) > 1e-6f) {
        // -1 <= q - l t < na
        const float e1 = (qmin - (float)na) / tl, e2 = (qmax + 1.0f) / tl;
        l_beg = (int)fmaxf(0.0f, floorf(fminf(e1, e2)) - 2.0f);
        l_end = (int)fminf((float)nl, ceilf(fmaxf(e1, e2)) + 3.0f);
    } else if (qmax < -3.0f || qmin > (float)(na + 2)) {
        l_end = 0;
    }
    if (m0 > geo.m_hi || m0 + 32 * CB <= geo.m_lo) l_end = 0;
    if (SEG > 1) {
        const int per = (max(0, l_end - l_beg) + SEG - 1) / SEG;
        l_beg += seg * per;
        l_end = min(l_end, l_beg + per);
    }
    TC acc[CB][IB];
#pragma unroll
    for (int c = 0; c < CB; ++c) {
        ray_at(pos[c], geo, m0 + 32 * c + lane, l_beg);
#pragma unroll
        for (int q = 0; q < IB; ++q) acc[c][q] = TC(0);
    }
    const unsigned last = na + 1;   // a position outside [-1, na) reads the two zeros after the line
    const Lanes<TL, IB>* line = src + (size_t)l_beg * pitch;
#pragma unroll LU
    for (int l = l_beg; l < l_end; ++l, line += pitch) {
#pragma unroll
        for (int c = 0; c < CB; ++c) {
            const unsigned e = min((unsigned)pos[c].index(), last);
            TC w0, w1;
            pos[c].weights(w0, w1);
            pos[c].step(dt);
            if constexpr (BF) {
                // pairs of images in the halves of packed FMAs
                const uint4 ua = *reinterpret_cast<const uint4*>(line + e);
                const uint4 ub = *reinterpret_cast<const uint4*>(line + e + 1);
                const unsigned pa[4] = {ua.x, ua.y, ua.z, ua.w}, pb[4] = {ub.x, ub.y, ub.z, ub.w};
                const float2 w02 = make_float2(w0, w0), w12 = make_float2(w1, w1);
                auto two = [](unsigned u) { return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u)); };
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float2 v = make_float2(acc[c][2 * q], acc[c][2 * q + 1]);
                    v = __ffma2_rn(w12, two(pb[q]), __ffma2_rn(w02, two(pa[q]), v));
                    acc[c][2 * q] = v.x, acc[c][2 * q + 1] = v.y;
                }
            } else {
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
    const TC wt = (TC)fabs(geo.inv);
#pragma unroll
    for (int c = 0; c < CB; ++c) {
        const int m = m0 + 32 * c + lane;
        if (m >= n_bins || kb_me >= set.n_base) continue;
        if constexpr (LANES && BF) {
            // two groups of four lanes, as the adjoint reads them
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                Lanes<TC, 4> w;
#pragma unroll
                for (int q = 0; q < 4; ++q) w.v[q] = wt * acc[c][4 * h + q];
                if (8 * g + 4 * h < batch)
                    ((Lanes<TC, 4>*)yv)[((size_t)(2 * g + h) * set.n_base + kb) * n_bins + m] = w;
            }
        } else if constexpr (LANES) {
            Lanes<TC, IB> w;
#pragma unroll
            for (int q = 0; q < IB; ++q) w.v[q] = ang[q % set.V] >= 0 ? wt * acc[c][q] : TC(0);
            ((Lanes<TC, IB>*)yv)[((size_t)g * set.n_base + kb) * n_bins + m] = w;
        } else {
            TO* y = (TO*)yv;
#pragma unroll
            for (int q = 0; q < IB; ++q) {
                const int b = g * (IB / set.V) + q / set.V, a = ang[q % set.V];
                if (b < batch && a >= 0) stf(y + ((size_t)b * n_angles + a) * n_bins + m, wt * acc[c][q]);
            }
        }
    }
}

// Fixed-point bin position within a tile's window, 0 to 47 (a 32 x 32 tile spans
// at most 31 sqrt(2) + 2 < 46 bins): first pixel and steps from float64, the
// thread's pixel an exact combination of them.  frac() is the fraction f as
// (BIAS + f) / SCALE, in the one operation that the type has for it.
template <class TC>
struct TilePos;
template <>
struct TilePos<float> {
    // 32 fraction bits, steps (at most 1) 30: 2^-31 off, up to 16 times in each
    // direction, below the conversion's 2^-25 (26 bits throughout, in 32-bit words,
    // left weights 1.4e-7 off, rms).  Four positions from one, not each from the
    // last: 400 images of 512 x 512, 720 x 736, 33.9 against 35.0 ms for A^T A
    using type = long long;
    using step = int;
    static constexpr float SCALE = 0x1p-32f;
    static constexpr int BIAS = 0;
    static __device__ __forceinline__ type make(double u) { return __double2ll_rn(u * 4294967296.0); }
    static __device__ __forceinline__ step make_step(double u) { return __double2int_rn(u * 1073741824.0); }
    static __device__ __forceinline__ type at(type p0, int tx, step dj, int ty, step di) {
        return p0 + (((long long)tx * dj + (long long)ty * di) << 2);
    }
    static __device__ __forceinline__ type eight(step d) { return (long long)d << 5; }
    static __device__ __forceinline__ unsigned index(type p) { return (unsigned)(p >> 32); }
    static __device__ __forceinline__ float frac(type p) { return __uint2float_rn((unsigned)p); }
};
template <>
struct TilePos<double> {
    using type = unsigned long long;
    using step = unsigned long long;
    static constexpr double SCALE = 1.0;
    static constexpr int BIAS = 1;
    static constexpr int FRAC = 57;   // below 64: within a signed 64-bit conversion
    static __device__ __forceinline__ step make_step(double u) { return (step)__double2ll_rn(u * 144115188075855872.0); }
    // the fraction is used to 52 bits: half of the last one makes that a rounding
    static __device__ __forceinline__ type make(double u) { return make_step(u) + 16u; }
    static __device__ __forceinline__ type at(type p0, int tx, step dj, int ty, step di) {
        return p0 + (type)(long long)tx * dj + (type)(long long)ty * di;
    }
    static __device__ __forceinline__ type eight(step d) { return d * 8; }
    static __device__ __forceinline__ unsigned index(type p) { return (unsigned)(p >> FRAC); }
    static __device__ __forceinline__ double frac(type p) {
        return __longlong_as_double((long long)(((p >> 5) & 0xfffffffffffffull) | 0x3ff0000000000000ull));
    }
};

constexpr int ATS = 32;     // tile side; a thread holds 4 pixels, 8 rows apart
constexpr int AWIN = 48;    // staged bins per angle: 31 sqrt(2) + 2 + the margin below, rounded up

template <class TC>
struct alignas(16) TileAng {           // one base angle as a tile sees it
    typename TilePos<TC>::type pos0;           // position of the tile's pixel (16, 16)
    typename TilePos<TC>::step dj, di;         // steps along j and i
    TC wb, w0, w1;                     // lower bin's weight w0 - wb F, upper's w1 + wb F where positive, F = frac()
    int mlo;                           // first staged bin
};

// Adjoint: one CTA per (32 x 32 tile, group of lanes, range of base angles).
// AK angles per round: their windows of bins and per-tile constants are staged
// in shared memory (copies of the next round in flight during this one, one
// barrier per round); every pixel then takes its two bins of every angle.
// out: images of type TO (PLANES false: one angle range, no mirror lanes), or
// one plane per (group, angle range, lane), already mirrored back, for
// lane_sum.  RAW: s is the sinogram itself (type TC), its lanes gathered
// while staging, which saves adjoint calls on one to three images the pass
// that interleaves it (257 x 301 pixels, 363 angles, forward and adjoint
// called from Python: 4 launches for 5, 153 to 150 us, host-bound).  Bound
// by shared memory: two 16-byte loads per pixel and angle, 8 wavefronts per
// warp and four lanes, 91% of the L1 data pipe busy on a batch of 400 images
// of 512 x 512, 720 x 736: 18.6 ms (one image: 66 us).  The per-line scatter
// into shared memory before it, 3.7 times the instructions and read-modify-
// writes of a private row, took 117 ms (411 us).
template <class TC, class TO, int IB, bool PLANES, bool RAW>
__global__ void __launch_bounds__(256) radon_adj_kernel(const void* __restrict__ s, TO* __restrict__ out, int n1,
                                                        int n2, int n_angles, int n_bins, int batch, int AK, int per,
                                                        RSet set) {
    pdl_enter();
    using TP = TilePos<TC>;
    using P = typename TP::type;
    using L = Lanes<TC, IB>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    L* win = reinterpret_cast<L*>(smem_raw);                                       // [2][AK][AWIN]
    TileAng<TC>* tab = reinterpret_cast<TileAng<TC>*>(win + 2 * AK * AWIN);        // [3][AK]
    int* ang = reinterpret_cast<int*>(tab + 3 * AK);                               // RAW: [3][AK][IB], a lane's angle or -1
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int i0 = blockIdx.y * ATS, j0 = blockIdx.x * ATS;
    const int g = blockIdx.z % ((batch + IB / set.V - 1) / (IB / set.V)), z = blockIdx.z / ((batch + IB / set.V - 1) / (IB / set.V));
    const int k_beg = z * per, k_end = min(set.n_base, k_beg + per);
    const int rounds = (k_end - k_beg + AK - 1) / AK;
    const L* sg = (const L*)s + (size_t)g * set.n_base * n_bins;
    const int b0 = g * (IB / set.V);
    auto angles_of = [&](int r) {       // the tile's constants of round r
        const int k = k_beg + r * AK + threadIdx.x;
        if (threadIdx.x >= AK || k >= k_end) return;
        const RGeo geo = set.geo[set.ang[k * set.V]];
        // from the detector's middle bin (n_bins - 1) / 2 on
        const double m00 = fma(geo.cs, j0 - 0.5 * (n2 - 1), fma(geo.sn, i0 - 0.5 * (n1 - 1), 0.5 * ((n_bins - 1) & 1)));
        const double lo = floor(m00 + fmin(0.0, (ATS - 1) * geo.cs) + fmin(0.0, (ATS - 1) * geo.sn) - 1e-3);
        const double a = fabs(geo.inv), b = a * a;
        TileAng<TC> t;
        t.pos0 = TP::make(m00 + (ATS / 2) * (geo.cs + geo.sn) - lo);
        t.dj = TP::make_step(geo.cs);
        t.di = TP::make_step(geo.sn);
        // a - b f and a - b (1 - f)
        t.wb = (TC)b * TP::SCALE;
        t.w0 = (TC)(a + TP::BIAS * b);
        t.w1 = (TC)(a - (1 + TP::BIAS) * b);
        t.mlo = (int)lo + (n_bins - 1) / 2;
        tab[(r % 3) * AK + threadIdx.x] = t;
        if (RAW) {
#pragma unroll
            for (int q = 0; q < IB; ++q)
                ang[((r % 3) * AK + threadIdx.x) * IB + q] = b0 + q / set.V < batch ? set.ang[k * set.V + q % set.V] : -1;
        }
    };
    auto stage = [&](int r) {           // the windows of round r
        L* w = win + (r & 1) * AK * AWIN;
        for (int e = threadIdx.x; e < AK * AWIN; e += 256) {
            const int a = e / AWIN, k = k_beg + r * AK + a;
            if (k < k_end) {
                const int m = tab[(r % 3) * AK + a].mlo + (e - a * AWIN);
                const bool ok = (unsigned)m < (unsigned)n_bins;
                if (RAW) {
#pragma unroll
                    for (int q = 0; q < IB; ++q) {
                        const int aq = ang[((r % 3) * AK + a) * IB + q];
                        const int mq = set.sym(q % set.V) & LANE_REV ? n_bins - 1 - m : m;
                        const bool in = ok && aq >= 0;
                        const TC* src = (const TC*)s + (in ? ((size_t)(b0 + q / set.V) * n_angles + aq) * n_bins + mq : 0);
                        cp_async_zfill(&w[e].v[q], src, (int)sizeof(TC), in);
                    }
                    continue;
                }
                const L* src = sg + (size_t)k * n_bins + (ok ? m : 0);
#pragma unroll
                for (int h = 0; h < (int)(sizeof(L) + 15) / 16; ++h)
                    cp_async_zfill((char*)(w + e) + 16 * h, (const char*)src + 16 * h,
                                   sizeof(L) < 16 ? (int)sizeof(L) : 16, ok);
            }
        }
        asm volatile("cp.async.commit_group;");
    };
    TC acc[4][IB];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int q = 0; q < IB; ++q) acc[u][q] = TC(0);
    angles_of(0);
    __syncthreads();
    stage(0);
    angles_of(1);
    for (int r = 0; r < rounds; ++r) {
        asm volatile("cp.async.wait_group 0;");
        __syncthreads();                // round r staged, round r - 1 consumed, constants of round r + 1 there
        if (r + 2 < rounds) angles_of(r + 2);
        if (r + 1 < rounds) stage(r + 1);
        const L* w = win + (r & 1) * AK * AWIN;
        const TileAng<TC>* ta = tab + (r % 3) * AK;
        const int na = min(AK, k_end - k_beg - r * AK);
        // measured, by the compiler's order of the loads: one image 159.5 with four, 161.4
        // us with two; 400 images 33.4 ms with one, 34.9 with two or four
#pragma unroll (PLANES ? 4 : 1)
        for (int a = 0; a < na; ++a, w += AWIN) {
            const TileAng<TC> t = ta[a];
            const P p = TP::at(t.pos0, tx - ATS / 2, t.dj, ty - ATS / 2, t.di);
            const P d8 = TP::eight(t.di);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const P pu = p + u * d8;
                const L* e = w + TP::index(pu);
                const TC F = TP::frac(pu);
                const L s0 = e[0], s1 = e[1];
                // a bin without weight is left out, not multiplied by zero: an infinity or
                // a NaN reaches the pixels of its ray only
                const TC a0 = fma(-t.wb, F, t.w0), a1 = fma(t.wb, F, t.w1);
                if (a0 > TC(0)) {
#pragma unroll
                    for (int q = 0; q < IB; ++q) acc[u][q] = fma(a0, s0.v[q], acc[u][q]);
                }
                if (a1 > TC(0)) {
#pragma unroll
                    for (int q = 0; q < IB; ++q) acc[u][q] = fma(a1, s1.v[q], acc[u][q]);
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
                const size_t plane = ((size_t)g * (gridDim.z / ((batch + IB / set.V - 1) / (IB / set.V))) + z) * IB + q;
                stf(out + plane * N + (size_t)si * n2 + sj, acc[u][q]);
            } else {
                const int b = g * IB + q;
                if (b < batch) stf(out + (size_t)b * N + (size_t)i * n2 + j, acc[u][q]);
            }
        }
    }
}

// ------------------------------------------------------------- launching --

int build_tables(nys_op* op) {
    const int A = op->n_angles, B = op->n_bins, n1 = op->n1, n2 = op->n2;
    const double c1 = (n1 - 1) / 2.0, c2 = (n2 - 1) / 2.0;
    std::vector<RGeo> geo(A);
    for (int k = 0; k < A; ++k) {
        const double th = k * (op->span / A);
        const double cs = std::cos(th), sn = std::sin(th);
        const bool rs = std::fabs(cs) + 1e-9 >= std::fabs(sn);
        const double c = 1.0 + (rs ? c2 : c1);
        const double den = rs ? cs : sn, oth = rs ? sn : cs;
        const double inv = 1.0 / den, t = oth / den;
        const int b2 = B - 1, l2 = (rs ? n1 : n2) - 1;
        // halves of the steps, so that the middles are whole numbers of them
        auto fix = [](double v) { return (unsigned long long)std::llrint(std::ldexp(v, 40)); };
        const unsigned long long ih = fix(0.5 * inv), th2 = fix(0.5 * t);
        const long long far = (int64_t)n1 + n2 + 64;
        geo[k] = RGeo{c, inv, t, (long long)(fix(c) - b2 * ih + l2 * th2), (long long)(2 * ih), (long long)(2 * th2),
                      cs, sn, rs ? 1 : 0, b2, l2, (int)std::max<long long>(0, (b2 - far) / 2),
                      (int)std::min<long long>(b2, (b2 + far) / 2)};
    }
    // the angle sets: every angle by itself, and over exactly 180 degrees the
    // mirror pairs and (square image, even number of angles) the fours
    std::vector<int> ang;
    op->lane_sets = 1;
    for (int k = 0; k < A; ++k) ang.push_back(k);
    auto add = [&](int V, int n_base, auto&& lane) {
        op->lane_sets |= V;
        for (int k = 0; k < n_base; ++k) {
            const size_t first = ang.size();
            for (int v = 0; v < V; ++v) {
                int a = lane(k, v);
                if (a < 0 || a >= A) a = -1;
                for (size_t p = first; p < ang.size(); ++p)
                    if (ang[p] == a) a = -1;
                ang.push_back(a);
            }
        }
    };
    if (op->span == M_PI) {
        add(2, A / 2 + 1, [&](int k, int v) { return v ? A - k : k; });
        if (n1 == n2 && A % 2 == 0)
            add(4, A / 4 + 1, [&](int k, int v) { return v == 0 ? k : v == 1 ? A - k : v == 2 ? A / 2 - k : A / 2 + k; });
    }
    NYS_CK(op->ctx, cudaMalloc(&op->rtab, geo.size() * sizeof(RGeo) + ang.size() * sizeof(int)));
    NYS_CK(op->ctx, cudaMemcpy(op->rtab, geo.data(), geo.size() * sizeof(RGeo), cudaMemcpyHostToDevice));
    NYS_CK(op->ctx, cudaMemcpy((char*)op->rtab + geo.size() * sizeof(RGeo), ang.data(), ang.size() * sizeof(int),
                               cudaMemcpyHostToDevice));
    return NYS_OK;
}

RSet angle_set(const nys_op* op, int V) {
    const int A = op->n_angles;
    const int* ang = (const int*)((const RGeo*)op->rtab + A);
    RSet r;
    r.geo = (const RGeo*)op->rtab;
    r.V = V;
    r.n_base = V == 1 ? A : A / V + 1;
    // lane v > 0: mirrored in j, transposed, both
    r.tf = V == 1 ? 0 : LANE_FJ << 4 | LANE_T << 8 | (LANE_T | LANE_FJ) << 12;
    r.ang = V == 1 ? ang : V == 2 ? ang + A : ang + A + 2 * (A / 2 + 1);
    return r;
}

// angle ranges of the adjoint: as many as keep all CTAs resident at once (4 to
// an SM) when the image has few tiles, at least 16 base angles each (one 512 x
// 512 image, 256 tiles, A^T A: 1 range 216 us, 2 ranges 161, 3 ranges, a second
// wave of a quarter of the SMs, 164 us)
int adj_ranges(const nys_op* op, int groups, int n_base) {
    const int64_t ctas = (int64_t)((op->n1 + ATS - 1) / ATS) * ((op->n2 + ATS - 1) / ATS) * groups;
    const int64_t want = (int64_t)op->ctx->sm_count * 4;
    return (int)std::max<int64_t>(1, std::min<int64_t>({want / ctas, n_base / 16, 16}));
}

template <class TC, int IB>
size_t adj_smem(int AK, bool raw) {
    return sizeof(Lanes<TC, IB>) * 2 * AK * AWIN + (sizeof(TileAng<TC>) + (raw ? IB * sizeof(int) : 0)) * 3 * AK;
}

template <class TI, class TO, class TC, int IB, bool LANES>
int fwd_part(nys_op* op, const TI* x, void* y, int nb, int V) {
    const RSet set = angle_set(op, V);
    if constexpr (std::is_same<TI, __nv_bfloat16>::value && IB == 4) {
        // bf16 images, eight to a group, when that still leaves 32 warps to an SM
        const int g8 = (nb + 7) / 8, nch = (op->n_bins + 63) / 64;
        if (V == 1 && (int64_t)set.n_base * nch * g8 >= (int64_t)op->ctx->sm_count * 32) {
            if (int st = lane_prep<TI, TI, 8>(op, x, nb, set, true)) return st;
            const auto* rows = (const Lanes<TI, 8>*)op->lines;
            NYS_CK(op->ctx, launch_pdl(radon_fwd_kernel<TI, TC, TO, 8, 2, 1, LANES>,
                                       dim3((unsigned)((set.n_base + 7) / 8 * nch), g8), 256, 0, op->ctx->stream, rows,
                                       rows + (size_t)g8 * op->n1 * (op->n2 + PAD), y, op->n1, op->n2, op->n_angles,
                                       op->n_bins, nb, set));
            NYS_LAUNCH_CK(op->ctx);
            return NYS_OK;
        }
    }
    if (int st = lane_prep<TI, TC, IB>(op, x, nb, set, V < 4)) return st;
    const int R = IB / V, groups = (nb + R - 1) / R;
    const auto* rows = (const Lanes<TC, IB>*)op->lines;
    const auto* cols = rows + (size_t)groups * op->n1 * (op->n2 + PAD);
    auto go = [&](auto kernel, int CB, int SEG) {
        const int nch = (op->n_bins + 32 * CB - 1) / (32 * CB), fang = 8 / SEG;
        return launch_pdl(kernel, dim3((unsigned)((set.n_base + fang - 1) / fang * nch), groups), 256, 0,
                          op->ctx->stream, rows, cols, y, op->n1, op->n2, op->n_angles, op->n_bins, nb, set);
    };
    // two bins per lane share the loop and the line when that leaves 32 warps
    // to an SM; otherwise a warp takes one bin per lane and a quarter of the
    // lines, four warps to a ray (one 512 x 512 image, its lines prepared: 94
    // against 141 us without the quarters; two bins per lane for a batch: 25.5
    // against 28.4 ms for three and 35 ms with one)
    const int64_t warps = (int64_t)set.n_base * ((op->n_bins + 63) / 64) * groups;
    if (warps >= (int64_t)op->ctx->sm_count * 32)
        NYS_CK(op->ctx, go(radon_fwd_kernel<TC, TC, TO, IB, 2, 1, LANES>, 2, 1));
    else
        NYS_CK(op->ctx, go(radon_fwd_kernel<TC, TC, TO, IB, 1, 4, LANES>, 1, 4));
    NYS_LAUNCH_CK(op->ctx);
    return NYS_OK;
}

// adjoint of the interleaved lanes s, or of the sinogram s itself (RAW)
template <class TO, class TC, int IB, bool RAW>
int adj_lanes(nys_op* op, const void* s, TO* x, int nb, int V) {
    const RSet set = angle_set(op, V);
    const int R = IB / V, groups = (nb + R - 1) / R, AK = op->radon_adj_ak;
    const int ns = adj_ranges(op, groups, set.n_base), per = (set.n_base + ns - 1) / ns;
    const dim3 grid((op->n2 + ATS - 1) / ATS, (op->n1 + ATS - 1) / ATS, groups * ns);
    const size_t sm = adj_smem<TC, IB>(AK, RAW);
    if (V == 1 && ns == 1) {
        auto kern = radon_adj_kernel<TC, TO, IB, false, RAW>;
        if (int st = smem_optin(op->ctx, (const void*)kern, sm)) return st;
        NYS_CK(op->ctx, launch_pdl(kern, grid, 256, sm, op->ctx->stream, s, x, op->n1, op->n2, op->n_angles, op->n_bins,
                                   nb, AK, per, set));
        NYS_LAUNCH_CK(op->ctx);
        return NYS_OK;
    }
    TC* planes = (TC*)op->planes;
    auto kern = radon_adj_kernel<TC, TC, IB, true, RAW>;
    if (int st = smem_optin(op->ctx, (const void*)kern, sm)) return st;
    NYS_CK(op->ctx, launch_pdl(kern, grid, 256, sm, op->ctx->stream, s, planes, op->n1, op->n2, op->n_angles, op->n_bins,
                               nb, AK, per, set));
    NYS_LAUNCH_CK(op->ctx);
    return lane_sum<TC, TO, IB>(op, x, nb, V, ns);
}

template <class TI, class TO, class TC, int IB>
int part_typed(nys_op* op, int which, const TI* x, TO* y, int nb, int V) {
    if (which == 0) return fwd_part<TI, TO, TC, IB, false>(op, x, y, nb, V);
    if (which == 1) {
        if constexpr (std::is_same<TI, TC>::value)
            if (nb < 4) return adj_lanes<TO, TC, IB, true>(op, x, y, nb, V);
        if (int st = lane_bins<TI, TC, IB>(op, x, nb, angle_set(op, V))) return st;
    } else {
        if (int st = fwd_part<TI, TO, TC, IB, true>(op, x, op->inter, nb, V)) return st;
    }
    return adj_lanes<TO, TC, IB, false>(op, op->inter, y, nb, V);
}

template <class TI, class TO, class TC>
int radon_typed(nys_op* op, int which, const void* x, void* y, int batch) {
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

int radon_setup(nys_op* op) {
    if (int st = build_tables(op)) return st;
    op->chunk = ray_chunk(op);
    const size_t es = op->dtype == NYS_F64 ? 8 : 4;
    // interleaved sinogram lanes, image lines and the adjoint's planes, for
    // every part that a chunk of images can be cut into
    size_t lanes = 0, lines = 0, planes = 0;
    for (int left = 1; left <= op->chunk; ++left) {
        const Part p = next_part(op, left);
        const RSet set = angle_set(op, p.V);
        const int R = p.IB / p.V, groups = (p.nb + R - 1) / R, ns = adj_ranges(op, groups, set.n_base);
        lanes = std::max(lanes, (size_t)groups * set.n_base * p.IB);
        lines = std::max(lines, (size_t)groups * p.IB);
        if (p.V > 1 || ns > 1) planes = std::max(planes, (size_t)groups * ns * p.IB);
    }
    NYS_CK(op->ctx, cudaMalloc(&op->inter, lanes * op->n_bins * es));
    NYS_CK(op->ctx, cudaMalloc(&op->lines, lines * es * ((size_t)op->n1 * (op->n2 + PAD) +
                                                         (size_t)op->n2 * (op->n1 + PAD))));
    if (planes) NYS_CK(op->ctx, cudaMalloc(&op->planes, planes * op->N * es));
    return NYS_OK;
}

int radon_run(nys_op* op, int which, const void* x, void* y, int batch, int in_dt, int out_dt) {
    if (op->dtype == NYS_F64) {
        if (in_dt != NYS_F64 || out_dt != NYS_F64) return fail(op->ctx, NYS_EINVAL, "f64 operator needs f64 data");
        return radon_typed<double, double, double>(op, which, x, y, batch);
    }
    const bool ib = in_dt == NYS_BF16, ob = out_dt == NYS_BF16;
    if (!ib && !ob) return radon_typed<float, float, float>(op, which, x, y, batch);
    if (ib && ob) return radon_typed<__nv_bfloat16, __nv_bfloat16, float>(op, which, x, y, batch);
    if (ib) return radon_typed<__nv_bfloat16, float, float>(op, which, x, y, batch);
    return radon_typed<float, __nv_bfloat16, float>(op, which, x, y, batch);
}

}  // namespace nys
