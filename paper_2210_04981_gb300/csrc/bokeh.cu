// Shaped bokeh for the post-filter (the paper's Discussion: bokeh shapes
// other than the uniform circle, by the shape of the sampling kernel and the
// relative weight of its samples).  Used by hdof_postfilter when
// p->blades >= 3 or p->aberration != 0; the circular path stays as it is.
//
// The thin lens images the aperture point O of a source at CoC c onto the
// screen offset (c / 2A)(-O_right, O_up) (screen y grows downwards): a near
// source's bokeh is the aperture scaled to radius |c|/2 and mirrored
// left-right, a far source's mirrored top-bottom.  With the aperture norm
// D(v) = |v| cos(m - pi/N) / cos(pi/N), m = (atan2(v) - rot) mod 2pi/N (the
// N-gon is {D <= A}; the disk: D = |v|), a source q = p + (dx, dy) weighs at
// receiver p
//   near: s(r_q - D(dx, -dy)) w,   far: s(r_q - D(-dx, dy)) w,
//   w = 1 + aberration (2 min(d / r_q, 1)^2 - 1) (1 while r_q < 1), d = |(dx, dy)|,
// normalised by the weighted lattice area a(r) = sum_o s(r - D(o)) w(|o|, r)
// (mirrors map the lattice onto itself, so one area serves both layers).
//
// k_bokeh_norm: D over the window's offsets (a table, built per call).
// k_bokeh_tables: the lattice points of D < EXACT_R + 1/2 sorted by D, with
//   the running count and sum of d^2; and a(r) on r = k / 256 (a table, for
//   r >= 8): its interpolation's relative error is below 1e-6 there.
// k_bokeh_prep: per pixel r + 1/2, 1/r^2, z and the premultiplied near and far
//   records; per 16x16 tile the largest radius feeding each layer.  a(r)
//   below 8 comes from the sorted points: those of D <= r - 1/2 from the
//   running sums (their d < r), the rim D in (r - 1/2, r + 1/2) point by
//   point (summing the whole lattice per pixel took 98 us at 1279x719, this
//   21 us, all of the kernel).
// k_bokeh_gather: near and far in separate loops, each over the disk of the
//   largest radius that feeds its layer and reaches the tile (D >= d, so
//   taps outside it weigh 0); 2x2 pixels per thread, four thread groups over
//   a tile's source rows, as the round gather (postfilter.cu).  One thread
//   per pixel over one window for both layers took 1310 us on a 1279x719
//   frame of mixed depths with a hexagonal, radially weighted lens; this
//   285 us (930M -> 190M warp instructions).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "batch.cuh"
#include "internal.h"

namespace hdof {
namespace {

constexpr int BT = 16;                  // pixel tile of the prep and the gather
constexpr float AREA_STEP = 1.f / 256.f;
constexpr float EXACT_R = 8.f;          // below: the area from the sorted lattice points
constexpr int AREA_FIRST = (int)(EXACT_R / AREA_STEP);  // first table entry that is read
constexpr int SORT_K = 9;               // offsets [-9, 9]^2 hold every point of D < EXACT_R + 1/2 (D >= d)
constexpr int SORT_N = (2 * SORT_K + 1) * (2 * SORT_K + 1);

struct Shape {
    int K;           // norm table covers offsets [-K, K]^2
    const float* D;  // (2K + 1)^2 aperture norms, row-major in (dy, dx)
    float ab;        // aberration
};

__device__ __forceinline__ float norm_at(const Shape& s, int dx, int dy) {
    return __ldg(&s.D[(dy + s.K) * (2 * s.K + 1) + dx + s.K]);
}
__device__ __forceinline__ float radial_w(const Shape& s, float r, float d) {
    if (r < 1.f) return 1.f;
    const float t = fminf(d / r, 1.f);
    return 1.f + s.ab * (2.f * t * t - 1.f);
}
__device__ __forceinline__ float soft(float x) { return fminf(fmaxf(x + 0.5f, 0.f), 1.f); }

__global__ void __launch_bounds__(256) k_bokeh_norm(int K, int blades, float rot, float* __restrict__ D) {
    const int n = 2 * K + 1;
    for (int e = blockIdx.x * 256 + threadIdx.x; e < n * n; e += gridDim.x * 256) {
        const int dx = e % n - K, dy = e / n - K;
        const float d = sqrtf((float)(dx * dx + dy * dy));
        float v = d;
        if (blades >= 3 && d > 0.f) {
            const float sect = 6.28318530717958648f / blades;
            float m = fmodf(atan2f((float)dy, (float)dx) - rot, sect);
            if (m < 0.f) m += sect;
            v = d * cosf(m - 0.5f * sect) / cosf(0.5f * sect);
        }
        D[e] = v;
    }
}

// The lattice points of [-SORT_K, SORT_K]^2 in order of D: pt[k] = (D, d^2,
// sum of d^2 over the points before k, 0).  A rank sort (ties in index
// order), eight threads per point; the sums are of integers below 2^24,
// exact in any order.
__device__ __forceinline__ void sort_lattice(const Shape& s, int block, float4* __restrict__ pt) {
    __shared__ float sD[SORT_N], sd2[SORT_N];
    constexpr int n = 2 * SORT_K + 1;
    for (int e = threadIdx.x; e < SORT_N; e += 256) {
        const int dx = e % n - SORT_K, dy = e / n - SORT_K;
        // beyond the norm table (r_max < 8): no radius reaches the point
        sD[e] = abs(dx) <= s.K && abs(dy) <= s.K ? norm_at(s, dx, dy) : 1e30f;
        sd2[e] = (float)(dx * dx + dy * dy);
    }
    __syncthreads();
    const int e = block * 32 + (threadIdx.x >> 3);
    const bool on = e < SORT_N;
    const float D = on ? sD[e] : 0.f;
    int rank = 0;
    float sum = 0.f;
    for (int k = threadIdx.x & 7; k < SORT_N; k += 8) {
        const bool before = on && (sD[k] < D || (sD[k] == D && k < e));
        rank += before;
        sum += before ? sd2[k] : 0.f;
    }
    for (int o = 4; o; o >>= 1) {
        rank += __shfl_xor_sync(0xffffffffu, rank, o);
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    if (on && (threadIdx.x & 7) == 0) pt[rank] = make_float4(D, sd2[e], sum, 0.f);
}
constexpr int SORT_BLOCKS = (SORT_N + 31) / 32;

// The first SORT_BLOCKS blocks sort the lattice points; then one block per
// table entry r = k / 256: block sum over the lattice in a fixed order
__global__ void __launch_bounds__(256) k_bokeh_tables(Shape s, int n_r, float4* __restrict__ pt,
                                                      float* __restrict__ area) {
    if (blockIdx.x < SORT_BLOCKS) {
        sort_lattice(s, blockIdx.x, pt);
        return;
    }
    const int k = blockIdx.x - SORT_BLOCKS + AREA_FIRST;
    if (k >= n_r) return;
    const float r = k * AREA_STEP;
    const int kk = (int)ceilf(r + 0.5f), n = 2 * kk + 1;
    float a = 0.f;
    for (int e = threadIdx.x; e < n * n; e += 256) {
        const int dx = e % n - kk, dy = e / n - kk;
        const float w = soft(r - norm_at(s, dx, dy));
        if (w > 0.f) a += w * radial_w(s, r, sqrtf((float)(dx * dx + dy * dy)));
    }
    __shared__ float red[256];
    red[threadIdx.x] = a;
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) area[k] = red[0];
}

// a(r) for r < EXACT_R from the sorted points (pt in shared memory): a point
// of D <= r - 1/2 has s = 1 and d <= D < r, so those add
// n (1 - ab) + 2 ab sum d^2 / r^2 (n for r < 1); the rim point by point
__device__ __forceinline__ float area_sorted(const Shape& s, const float4* pt, float r, float ir2) {
    int lo = 0, hi = SORT_N;  // points of D <= r - 1/2
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (pt[mid].x <= r - 0.5f) lo = mid + 1;
        else hi = mid;
    }
    const float c0 = ir2 > 0.f ? 1.f - s.ab : 1.f, c1 = 2.f * s.ab;
    float a = lo < SORT_N ? fmaf(c1, pt[lo].z * ir2, (float)lo * c0) : 0.f;
    const float rh = r + 0.5f;
    for (int k = lo; k < SORT_N; ++k) {
        const float4 p = pt[k];
        if (p.x >= rh) break;
        a = fmaf(__saturatef(rh - p.x), fmaf(c1, __saturatef(p.y * ir2), c0), a);
    }
    return a;
}

template <class ND, class COL>
struct BokehPrep {
    const ND* nd;
    const COL* col;
    int W, H, ntx;
    Coc coc;
    float rmax;
    Shape s;
    const float* area;  // a(k / 256)
    const float4* pt;   // sorted lattice points
    int n_r;
    float* rh;
    float* zq;
    float* ir2;  // 1 / r^2, 0 where r < 1 (no radial weight)
    float4* nrec;
    float4* frec;
    float4* tmax;  // per tile: largest r feeding the near and the far layer (-1: none); 1: a record is not finite
};

template <class ND, class COL>
__global__ void __launch_bounds__(256) k_bokeh_prep(BokehPrep<ND, COL> a) {
    __shared__ float4 s_pt[SORT_N];
    for (int k = threadIdx.x; k < SORT_N; k += 256) s_pt[k] = __ldg(&a.pt[k]);
    __syncthreads();
    const int i = blockIdx.x * BT + (threadIdx.x & 15), j = blockIdx.y * BT + (threadIdx.x >> 4);
    float rn = -1.f, rf = -1.f;
    bool odd = false;
    if (i < a.W && j < a.H) {
        const size_t q = (size_t)j * a.W + i;
        const float z = ldz(a.nd + q), c = a.coc(z);
        const float r = fminf(fabsf(c) * 0.5f, a.rmax);
        const float ir2 = r < 1.f ? 0.f : 1.f / (r * r);
        float ar;
        if (r < EXACT_R) {
            ar = area_sorted(a.s, s_pt, r, ir2);
        } else {
            const float u = r / AREA_STEP;
            const int k = min((int)u, a.n_r - 2);
            const float f = u - (float)k;
            ar = fmaf(f, __ldg(&a.area[k + 1]) - __ldg(&a.area[k]), __ldg(&a.area[k]));
        }
        const float ia = 1.f / ar, wn = w_near(c), an = wn * ia, af = (1.f - wn) * ia;
        const float4 col = ld4(a.col + q);
        a.rh[q] = r + 0.5f;
        a.zq[q] = z;
        a.ir2[q] = ir2;
        a.nrec[q] = make_float4(col.x * an, col.y * an, col.z * an, an);
        a.frec[q] = make_float4(col.x * af, col.y * af, col.z * af, af);
        odd = !isfinite(col.x) || !isfinite(col.y) || !isfinite(col.z);
        rn = wn > 0.f ? r : -1.f;
        rf = wn < 1.f ? r : -1.f;
    }
    for (int o = 16; o; o >>= 1) {
        rn = fmaxf(rn, __shfl_xor_sync(0xffffffffu, rn, o));
        rf = fmaxf(rf, __shfl_xor_sync(0xffffffffu, rf, o));
    }
    __shared__ float2 red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_float2(rn, rf);
    const int any_odd = __syncthreads_or(odd);
    if (threadIdx.x == 0) {
        float2 m = red[0];
        for (int k = 1; k < 8; ++k) m = make_float2(fmaxf(m.x, red[k].x), fmaxf(m.y, red[k].y));
        a.tmax[blockIdx.y * a.ntx + blockIdx.x] = make_float4(m.x, m.y, any_odd ? 1.f : 0.f, 0.f);
    }
}

template <class COL>
struct BokehGather {
    const float* rh;
    const float* zq;
    const float* ir2;
    const float4* nrec;
    const float4* frec;
    const COL* col;
    const float4* tmax;
    int W, H, ntx, nty, kt;
    float kz_rel;
    Shape s;
    float4* out;
};

constexpr int BG = 4;            // thread groups over a tile's source rows
constexpr int BGT = 64;          // threads of a group: 2x2 pixels each

struct BokehAcc {
    float2 xy, zw;  // (S.x, S.y), (S.z, W)
    float zp, kb;   // far: the depth z_p and 1 / (kz_rel z_p)
};

// One source into the thread's 2x2 pixels.  Row k's left pixel sees it at
// norm D[k] and squared distance d2[k], its right pixel at the previous
// column's, carried in cD and cd2.  The far layer's depth test is
// clamp(1 - (z - z_p) kb): the difference is exact near z_p, where
// (1 + 1 / kz_rel) - z kb would cancel to 2^-24 / kz_rel.  ONLY: a source is
// added only where it weighs (a weight of 0 times an infinite or NaN colour
// would reach every pixel of the window).
template <bool NEAR, bool RAD, bool ONLY>
__device__ __forceinline__ void bk_tap(BokehAcc (&a)[4], float (&cD)[2], float (&cd2)[2], const float (&D)[2],
                                       const float (&d2)[2], float rh, float ir2, float z, float c1, float c0r,
                                       const float4& e) {
    const float c0 = RAD ? (ir2 > 0.f ? c0r : 1.f) : 1.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float Dk = (k & 1) ? cD[k >> 1] : D[k >> 1], dd = (k & 1) ? cd2[k >> 1] : d2[k >> 1];
        float w = __saturatef(rh - Dk);
        if (RAD) w *= fmaf(c1, __saturatef(dd * ir2), c0);
        if (!NEAR) w *= __saturatef(fmaf(a[k].zp - z, a[k].kb, 1.f));
        if (!ONLY || w > 0.f) {
            a[k].xy = fma2(w, e.x, e.y, a[k].xy);
            a[k].zw = fma2(w, e.z, e.w, a[k].zw);
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        cD[k] = D[k];
        cd2[k] = d2[k];
    }
}

// One layer over the disk-shaped window of radius R around the 2x2 block at
// (i, j), rows g, g + BG, ... (see the round gather's pf_layer)
template <bool NEAR, bool RAD, bool ONLY>
__device__ __forceinline__ void bk_layer(BokehAcc (&a)[4], float R, int g, int i, int j, int W, int H, const Shape& s,
                                         const float* __restrict__ rh, const float* __restrict__ ir2,
                                         const float* __restrict__ zq, const float4* __restrict__ rec) {
    const int G = (int)floorf(R + 1e-3f), n = 2 * s.K + 1;
    const int y0 = max(j - G, 0), y1 = min(j + 1 + G, H - 1);
    const float R2 = R * R, c0r = 1.f - s.ab, c1 = 2.f * s.ab;
    const float2* __restrict__ rh2 = reinterpret_cast<const float2*>(rh);
    const float2* __restrict__ ir22 = reinterpret_cast<const float2*>(ir2);
    const float2* __restrict__ zq2 = reinterpret_cast<const float2*>(zq);
    constexpr int SX = NEAR ? 1 : -1;  // near: D(dx, -dy); far: D(-dx, dy)
    for (int y = y0 + g; y <= y1; y += BG) {
        const int dyi = y - j;
        const float dy = (float)dyi, dy0 = dy * dy, dy1 = (dy - 1.f) * (dy - 1.f);
        const float dmin = dyi == 0 || dyi == 1 ? 0.f : fminf(dy0, dy1);
        const int w = (int)(sqrt_approx(fmaxf(R2 - dmin, 0.f)) + 1e-3f);
        const int x0 = max(i - w, 0), x1 = min(i + 1 + w, W - 1);
        // offsets reach one beyond the window (the carried column): K covers it
        const float* __restrict__ D0 = s.D + (s.K - SX * dyi) * n + s.K;
        const float* __restrict__ D1 = s.D + (s.K - SX * (dyi - 1)) * n + s.K;
        int dxi = x0 - i;
        float dx = (float)dxi;
        float cD[2] = {__ldg(&D0[SX * (dxi - 1)]), __ldg(&D1[SX * (dxi - 1)])};
        const float dm = (dx - 1.f) * (dx - 1.f);
        float cd2[2] = {dm + dy0, dm + dy1};
        unsigned q = (unsigned)y * W + x0;
        const unsigned qend = (unsigned)y * W + x1 + 1;
        auto tap = [&](float r, float v, float z, const float4& e) {
            const float D[2] = {__ldg(&D0[SX * dxi]), __ldg(&D1[SX * dxi])}, dx2 = dx * dx;
            const float d2[2] = {dx2 + dy0, dx2 + dy1};
            bk_tap<NEAR, RAD, ONLY>(a, cD, cd2, D, d2, r, v, z, c1, c0r, e);
            ++dxi;
            dx += 1.f;
        };
        if (q & 1) {
            tap(__ldg(&rh[q]), RAD ? __ldg(&ir2[q]) : 0.f, NEAR ? 0.f : __ldg(&zq[q]), ld4(rec + q));
            ++q;
        }
        const unsigned mend = qend >> 1;
        for (unsigned m = q >> 1; m < mend; ++m) {
            const float2 r2 = __ldg(&rh2[m]), v2 = RAD ? __ldg(&ir22[m]) : make_float2(0.f, 0.f);
            const float2 z2 = NEAR ? make_float2(0.f, 0.f) : __ldg(&zq2[m]);
            float4 e0, e1;
            ld_rec_pair(rec + 2 * (size_t)m, e0, e1);
            tap(r2.x, v2.x, z2.x, e0);
            tap(r2.y, v2.y, z2.y, e1);
        }
        if (qend & 1) {
            const unsigned l = qend - 1;
            tap(__ldg(&rh[l]), RAD ? __ldg(&ir2[l]) : 0.f, NEAR ? 0.f : __ldg(&zq[l]), ld4(rec + l));
        }
    }
}

// Bound by issue and load latency together (issue 63% busy; the tap
// arithmetic is 8 instructions per pixel and tap with the radial weight, 10
// in the far layer).  Three resident blocks: 80 registers; four spill.
template <class COL, bool RAD>
__global__ void __launch_bounds__(BG* BGT, 3) k_bokeh_gather(BokehGather<COL> a) {
    const int W = a.W, H = a.H, tx = blockIdx.x, ty = blockIdx.y;
    // each layer's reach: the largest radius + 1/2 among tiles that feed it and can reach this one
    __shared__ int s_reach[2];
    __shared__ float4 s_part[BG][BT * BT];
    if (threadIdx.x < 2) s_reach[threadIdx.x] = -1;
    __syncthreads();
    bool odd = false;  // a tile near enough holds a record that is not finite
    {
        const int n = 2 * a.kt + 1;
        for (int e = threadIdx.x; e < n * n; e += BG * BGT) {
            const int ox = e % n - a.kt, oy = e / n - a.kt, x = tx + ox, y = ty + oy;
            if (x < 0 || y < 0 || x >= a.ntx || y >= a.nty) continue;
            const float4 r = __ldg(&a.tmax[y * a.ntx + x]);
            odd |= r.z > 0.f;
            const float gx = ox == 0 ? 0.f : (float)((abs(ox) - 1) * BT + 1);
            const float gy = oy == 0 ? 0.f : (float)((abs(oy) - 1) * BT + 1);
            const float g2 = gx * gx + gy * gy;
            // positive floats order as their bit patterns
            if (r.x >= 0.f && g2 < (r.x + 0.5f) * (r.x + 0.5f)) atomicMax(&s_reach[0], __float_as_int(r.x + 0.5f));
            if (r.y >= 0.f && g2 < (r.y + 0.5f) * (r.y + 0.5f)) atomicMax(&s_reach[1], __float_as_int(r.y + 0.5f));
        }
    }
    const bool only = __syncthreads_or(odd);
    const int g = threadIdx.x / BGT, t = threadIdx.x % BGT;
    const int li = 2 * (t & 7), lj = 2 * (t >> 3), i = tx * BT + li, j = ty * BT + lj;
    const bool in = i < W && j < H;
    const int p = threadIdx.x, px = tx * BT + (p & 15), py = ty * BT + (p >> 4);  // the pixel this thread finishes
    const bool fin = px < W && py < H;
    const size_t pq = (size_t)py * W + px;
    float4 S[2];  // near, far sums of pixel p
#pragma unroll
    for (int layer = 1; layer >= 0; --layer) {
        S[layer] = make_float4(0.f, 0.f, 0.f, 0.f);
        const int rb = s_reach[layer];
        if (rb < 0) continue;  // nothing within reach feeds this layer (block-uniform)
        if (in) {
            BokehAcc acc[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                acc[k].xy = acc[k].zw = make_float2(0.f, 0.f);
                acc[k].zp = acc[k].kb = 0.f;
                if (layer) {
                    const int x = min(i + (k & 1), W - 1), y = min(j + (k >> 1), H - 1);
                    acc[k].zp = __ldg(&a.zq[(size_t)y * W + x]);
                    acc[k].kb = 1.f / (a.kz_rel * acc[k].zp);
                }
            }
            const float R = __int_as_float(rb);
            if (layer && only) bk_layer<false, RAD, true>(acc, R, g, i, j, W, H, a.s, a.rh, a.ir2, a.zq, a.frec);
            else if (layer) bk_layer<false, RAD, false>(acc, R, g, i, j, W, H, a.s, a.rh, a.ir2, a.zq, a.frec);
            else if (only) bk_layer<true, RAD, true>(acc, R, g, i, j, W, H, a.s, a.rh, a.ir2, a.zq, a.nrec);
            else bk_layer<true, RAD, false>(acc, R, g, i, j, W, H, a.s, a.rh, a.ir2, a.zq, a.nrec);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                s_part[g][(lj + (k >> 1)) * BT + li + (k & 1)] =
                    make_float4(acc[k].xy.x, acc[k].xy.y, acc[k].zw.x, acc[k].zw.y);
        }
        __syncthreads();
        if (fin) {
            float4 v = s_part[0][p];
#pragma unroll
            for (int b = 1; b < BG; ++b) v = add4(v, s_part[b][p]);
            S[layer] = v;
        }
        __syncthreads();
    }
    if (!fin) return;
    const float4 Sn = S[0], Sf = S[1], cp = ld4(a.col + pq);
    const float alpha = fminf(fmaxf(Sn.w, 0.f), 1.f);
    const float in_ = Sn.w > HDOF_PP_MIN_W ? 1.f / Sn.w : 0.f;
    const bool fok = Sf.w > HDOF_PP_MIN_W;
    const float inf_ = fok ? 1.f / Sf.w : 0.f;
    const float3 N = f3(Sn.x * in_, Sn.y * in_, Sn.z * in_);
    const float3 F = fok ? f3(Sf.x * inf_, Sf.y * inf_, Sf.z * inf_) : f3(cp.x, cp.y, cp.z);
    a.out[pq] = make_float4(alpha * N.x + (1.f - alpha) * F.x, alpha * N.y + (1.f - alpha) * F.y,
                            alpha * N.z + (1.f - alpha) * F.z, alpha);
}

}  // namespace

bool bokeh_shaped(const hdof_params* p) { return p->blades >= 3 || p->aberration != 0.f; }

size_t bokeh_scratch_bytes(const hdof_params* p) {
    const int K = (int)std::ceil((p ? p->r_max : 100.f) + 0.5f) + 1;
    const size_t n_r = (size_t)((p ? p->r_max : 100.f) / AREA_STEP) + 2;
    return (((size_t)(2 * K + 1) * (2 * K + 1) * sizeof(float) + 255) & ~size_t(255)) +
           ((n_r * sizeof(float) + 255) & ~size_t(255)) + ((SORT_N * sizeof(float4) + 255) & ~size_t(255));
}

// the shaped post-filter (scratch: the post-filter regions, then bokeh_scratch_bytes)
int launch_bokeh(const hdof_gbuf* in, const Coc& coc, const hdof_params* p, float* pp, void* scratch,
                 cudaStream_t s) {
    const int W = in->width, H = in->height;
    const WsLayout L = ws_layout(W, H, p);
    ViewWs w = {};
    pf_regions(w, static_cast<char*>(scratch), L);
    const int K = (int)std::ceil(p->r_max + 0.5f) + 1;
    const int n_r = (int)(p->r_max / AREA_STEP) + 2;
    float* D = reinterpret_cast<float*>(w.bokeh);
    float* area = reinterpret_cast<float*>(w.bokeh + (((size_t)(2 * K + 1) * (2 * K + 1) * sizeof(float) + 255) &
                                                      ~size_t(255)));
    float4* pt = reinterpret_cast<float4*>(reinterpret_cast<char*>(area) +
                                           (((size_t)n_r * sizeof(float) + 255) & ~size_t(255)));
    Shape sh{K, D, p->aberration};
    ProfScope ps_("pf_bokeh", s);
    k_bokeh_norm<<<(unsigned)std::min((2 * K + 1) * (2 * K + 1) / 256 + 1, 1024), 256, 0, s>>>(K, p->blades,
                                                                                                p->blade_rot, D);
    HDOF_LAUNCHED("post-filter bokeh: norm table");
    k_bokeh_tables<<<SORT_BLOCKS + std::max(n_r - AREA_FIRST, 0), 256, 0, s>>>(sh, n_r, pt, area);
    HDOF_LAUNCHED("post-filter bokeh: area tables");
    const int ntx = (W + BT - 1) / BT, nty = (H + BT - 1) / BT;
    dim3 grid(ntx, nty);
    float4* tmax = w.tmax;
    float* ir2 = reinterpret_cast<float*>(w.pre);  // the round gather's prefix plane
    const bool f32n = in->dtype_nd == HDOF_F32, f32c = in->dtype_col == HDOF_F32;
    const float4* nd4 = static_cast<const float4*>(in->nd);
    const half4s* ndh = static_cast<const half4s*>(in->nd);
    const float4* col4 = static_cast<const float4*>(in->col);
    const bf164s* colb = static_cast<const bf164s*>(in->col);
    auto prep = [&](auto nd, auto col) {
        using ND = std::remove_const_t<std::remove_pointer_t<decltype(nd)>>;
        using COL = std::remove_const_t<std::remove_pointer_t<decltype(col)>>;
        k_bokeh_prep<<<grid, 256, 0, s>>>(BokehPrep<ND, COL>{nd, col, W, H, ntx, coc, p->r_max, sh, area, pt, n_r,
                                                             w.rh, w.zq, ir2, w.nrec, w.frec, tmax});
    };
    if (f32n && f32c) prep(nd4, col4);
    else if (f32n) prep(nd4, colb);
    else if (f32c) prep(ndh, col4);
    else prep(ndh, colb);
    HDOF_LAUNCHED("post-filter bokeh: prep");
    const int kt = (int)std::ceil((p->r_max + 0.5f) / BT) + 1;
    float4* out = reinterpret_cast<float4*>(pp);
    // the radial weight's arithmetic only where there is one
    auto gather = [&](auto col) {
        using COL = std::remove_const_t<std::remove_pointer_t<decltype(col)>>;
        const BokehGather<COL> a{w.rh, w.zq, ir2, w.nrec, w.frec, col, tmax, W, H, ntx, nty, kt, p->kz_rel, sh, out};
        if (p->aberration != 0.f) k_bokeh_gather<COL, true><<<grid, BG * BGT, 0, s>>>(a);
        else k_bokeh_gather<COL, false><<<grid, BG * BGT, 0, s>>>(a);
    };
    if (f32c) gather(col4);
    else gather(colb);
    HDOF_LAUNCHED("post-filter bokeh: gather");
    return HDOF_OK;
}

}  // namespace hdof
