// post-process CoC filter of the sharp image (Design section: the sharp
// rasterised image is blurred by a post-process filter; the Reconstruction
// section gives the gather's rejection rule: a sample counts only if its CoC
// radius reaches the pixel).
//
// Scatter-as-gather with soft disks.  Pixel q scatters its colour over
// s(r_q - d), s(x) = clamp(x + 1/2, 0, 1), r_q = min(|c(z_q)|/2, r_max),
// normalised by the disk's lattice area a(r) = sum_o s(r - |o|) so that each
// pixel scatters unit weight.  a(r) is piecewise linear in r with breaks at
// |o| +- 1/2; a table of its breakpoints is built once per device and
// evaluated by binary search, which is exact up to float rounding.
//
// k_pf_prep: per pixel r + 1/2, z and the premultiplied near and far layer
//   records (c w/a, w/a), row-major; per 16x16
//   tile the largest r feeding each layer and the smallest r feeding the near
//   layer.
// k_pf_rowscan: the row prefix of the near records (row-major).
// k_pf_gather: near and far are gathered in two loops, each bounded per tile
//   by the largest radius among the tiles whose pixels feed that layer and
//   can reach it, and per source row to the columns of that disk; every tap
//   outside has zero weight, so the bounded gathers equal the full ones.
//   Where every near source close to the tile has a large radius, the near
//   taps of weight exactly 1 for all of a thread's pixels (the interior) are
//   summed as one difference of the row prefix and only the ring around them
//   is tapped.  Each thread gathers
//   a 2x2 pixel block so every tap it loads serves four pixels; the per-tap
//   arithmetic is branch-free (saturating adds).  The rows above and below the
//   block are walked in pairs: they share bounds and distances, and their
//   loads are in flight together.  Two thread groups share a tile's window.
//   Bound by the latency of the tap and prefix loads and by issue (57% busy).
//   One common interior per thread (no per-pixel masks, a quarter of the
//   prefix loads), the row pairs and the split took the gather alone from 308
//   to 218 us (1080p room), 3270 to 2116 us (4K room, FP16/BF16 planes), 455
//   to 252 us (1080p, mixed depths) and 43 to 18.5 us (128x128).
#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "batch.cuh"
#include "internal.h"

namespace hdof {
namespace {

using hdof::ld4;  // beside the overloads below
using hdof::ld_rec_pair;
using hdof::st4;

constexpr int TP = HDOF_TILE_PF;
constexpr int PF_GROUP = 64;  // threads that cover a 16x16 tile once (2x2 pixels each; 2x4 slower by 5-30%)
// Thread groups per tile, group g taking the source row pairs g, g + PF_G, ...
// of each pixel's window.  A tile's work runs from nothing to (2 r_max)^2 taps
// a pixel, so with one group the widest windows were the kernel's tail (32 of
// them on one SM outlast the rest of the grid), and a small image had one
// long serial loop a thread.  Gather alone, 1 / 2 / 4 groups: mixed depths at
// 1080p 355 / 252 / 258 us, the 128x128 frame 29 / 18.5 / 14-16 us, the
// 1080p room 224 / 218 / 240 us, 4K 2187 / 2116 / 2148 us.
constexpr int PF_G = 2;
constexpr int GATHER_THREADS = PF_G * PF_GROUP;
constexpr int PF_MINB = 6;    // resident blocks per SM: 80 registers (7, 72 registers: 5-15% slower but for 4K)
constexpr int PF_UNROLL = 2;  // of the tap-pair loop: a pair's four record loads beside the next one's (1: 3% slower)
// A near tile's interior path runs above this share of its reach, and a row
// takes the prefix only for at least PF_MIN_IN columns (two 16-byte loads
// cost about as much as two tap pairs): 0.2 to 0.5, and 2 to 8 columns, are
// within 3% of one another.
constexpr float PF_IN_SHARE = 0.5f;
constexpr int PF_MIN_IN = 4;
// Weight of a window's row above which every pixel sums its own columns
// (pf_gather_body).  An entry of the prefix is rounded in each addition of its
// scan (five in a warp, up to seven warps, one per 256 columns): in a row of
// up to this weight by 2^-22 at most each time, and its colours as finely as
// the row's colour sum allows, so beside a bright source relative to that
// source, on either path.  Errors against 64 bits over 60 drawn images, as
// shares of those with per-pixel sums everywhere: maximum 0.97 and rms 0.98
// (geometric means; one image of the 60 1.17 and 1.10).  With a line at 4 none
// is above 1.01, but a 1080p room's gather takes up to 3% longer; 5 to 7 as at 8.
constexpr float PF_ROW_W = 8.f;
// Shared-memory carve-out (percent of the maximum) for the gather: six
// resident blocks hold 8 KB of partial sums each, and the taps are served
// from L1, so no more than that (20 to 45%: within 2%).
constexpr int GATHER_CARVEOUT = 30;
constexpr int AREA_MAX = 16384;  // breakpoints for radii up to 127.5

// (x_m, a(x_m), slope on [x_m, x_{m+1}], 0)
__device__ float4 g_area[AREA_MAX];
// g_area_at[b]: largest m with x_m <= b / 32.  The breakpoints are at most 4
// to such an interval up to r = 100, so the search within one takes two or
// three dependent reads instead of the fourteen of the whole table, which
// bound k_pf_prep by their latency (1080p 39 to 30 us, 4K FP16/BF16 119 to
// 92 us).
constexpr int AREA_BUCKETS = 4096;
__device__ unsigned short g_area_at[AREA_BUCKETS + 1];

__device__ __forceinline__ float disk_area(float r) {
    const int b = min((int)(r * 32.f), AREA_BUCKETS - 1);
    int lo = __ldg(&g_area_at[b]), hi = __ldg(&g_area_at[b + 1]);  // largest m with x_m <= r
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(&g_area[mid].x) <= r) lo = mid;
        else hi = mid - 1;
    }
    float4 e = __ldg(&g_area[lo]);
    return fmaf(e.z, r - e.x, e.y);
}

// The gather's planes have an even pitch, so that a pair of pixels (2m, 2m + 1)
// of any row is aligned (records to 32 bytes).
__host__ __device__ inline int pf_pitch(int W) { return (W + 1) & ~1; }

// Per source pixel q the gather reads r_q + 1/2, z_q and two premultiplied
// layer records (c_q w/a, w/a) with w = w_near(q) for the near layer and
// 1 - w_near(q) for the far layer; per 16x16 tile, the largest r among its
// pixels that feed each layer (-1: none).  Outside the thin focus zone a
// pixel feeds one layer only, so near and far are gathered in separate loops
// with their own windows (in the workloads here the far field's blur is
// small and the near field's large).
// Layer records in the colour's precision: FP32 colour, float4 records; BF16
// colour (the mixed form), BF16 records (8 bytes: a pair of taps in one
// 128-bit load), accumulated in FP32 like the FP32 ones.
template <class COL>
struct RecOf {
    using T = float4;
    using P = float4;  // an entry of the row prefix
};
template <>
struct RecOf<bf164s> {
    using T = bf164s;
    using P = float4;
};
// The specular plane col.w as an opaque grey colour: FP32 records (s w/a, w/a)
// and as many sums, half the loads and FMAs of a colour's, with the same
// results as the plane filtered as a colour.  That took a pass to write the
// plane and, alone, 245 us at 1279x717 (wide aperture) and 2197 us at 4K in the
// gather; this takes 178 and 1525 us.
template <class COL>
struct Grey {
    COL c;
};
template <class COL>
__device__ __forceinline__ float4 ld4(const Grey<COL>* p) {
    const float s = ld4(&p->c).w;
    return make_float4(s, s, s, s);
}
template <class COL>
struct RecOf<Grey<COL>> {
    using T = float2;
    using P = float2;
};
// a record or prefix entry of two channels stands for the last two of four
__device__ __forceinline__ void st4(float2* p, const float4& v) { *p = make_float2(v.z, v.w); }
__device__ __forceinline__ float4 ld4(const float2* p) {
    const float2 v = __ldg(p);
    return make_float4(0.f, 0.f, v.x, v.y);
}
__device__ __forceinline__ void ld_rec_pair(const float2* p, float2& a, float2& b) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
}

template <class ND, class COL>
struct PrepArgs {
    const ND* nd;
    const COL* col;
    int W, H;
    Coc coc;
    float rmax;
    int ntx;
    float* rh;      // r + 1/2
    float* zq;      // view depth
    typename RecOf<COL>::T* nrec;  // (c w/a, w/a), near layer
    typename RecOf<COL>::T* frec;  // (c (1-w)/a, (1-w)/a), far layer
    float4* tmax;   // per tile: (max r feeding near, max r feeding far, min r feeding near (+inf: none), 0)
    const float* lens;  // optional (focus distance, aperture radius) on the device, replacing coc's lens
    float t;            // tan(fovy / 2), with lens
};

template <class ND, class COL>
__device__ __forceinline__ void pf_prep_body(const PrepArgs<ND, COL>& a, int bx, int by) {
    const int W = a.W, H = a.H;
    int i = bx * TP + (threadIdx.x & 15), j = by * TP + (threadIdx.x >> 4);
    const float INF = __int_as_float(0x7f800000);
    float rn = -1.f, rf = -1.f, rnmin = INF;
    if (i < W && j < H) {
        size_t q = (size_t)j * W + i;
        float z = ldz(a.nd + q);
        float c = lens_coc(a.coc, a.lens, H, a.t)(z);
        float r = fminf(fabsf(c) * 0.5f, a.rmax);
        float ia = 1.f / disk_area(r);
        float wn = w_near(c), an = wn * ia, af = (1.f - wn) * ia;
        float4 col = ld4(a.col + q);
        const size_t o = (size_t)j * pf_pitch(W) + i;
        a.rh[o] = r + 0.5f;
        a.zq[o] = z;
        st4(a.nrec + o, make_float4(col.x * an, col.y * an, col.z * an, an));
        st4(a.frec + o, make_float4(col.x * af, col.y * af, col.z * af, af));
        if (i == W - 1 && (W & 1)) {  // the padding column of an odd width: a source of no weight
            const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
            a.rh[o + 1] = 0.f;
            a.zq[o + 1] = 1.f;
            st4(a.nrec + o + 1, none);
            st4(a.frec + o + 1, none);
        }
        rn = wn > 0.f ? r : -1.f;
        rf = wn < 1.f ? r : -1.f;
        rnmin = wn > 0.f ? r : INF;
    }
    for (int o = 16; o; o >>= 1) {
        rn = fmaxf(rn, __shfl_xor_sync(0xffffffffu, rn, o));
        rf = fmaxf(rf, __shfl_xor_sync(0xffffffffu, rf, o));
        rnmin = fminf(rnmin, __shfl_xor_sync(0xffffffffu, rnmin, o));
    }
    __shared__ float4 red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_float4(rn, rf, rnmin, 0.f);
    __syncthreads();
    if (threadIdx.x == 0) {
        float4 m = red[0];
        for (int k = 1; k < 8; ++k)
            m = make_float4(fmaxf(m.x, red[k].x), fmaxf(m.y, red[k].y), fminf(m.z, red[k].z), 0.f);
        a.tmax[by * a.ntx + bx] = m;
    }
}

template <class ND, class COL>
__global__ void __launch_bounds__(256) k_pf_prep(PrepArgs<ND, COL> a) { pf_prep_body(a, blockIdx.x, blockIdx.y); }

// Row prefix of the near records: pre[y][x] = sum over x' <= x of the near
// record of pixel (x', y), row-major.  The gather sums a pixel's interior
// taps (all of weight exactly 1) as differences of it.  One block per row,
// in rounds of 256 consecutive pixels (a block scan per round plus the
// running total): the summation order is fixed.
template <class REC, class PRE = float4>
struct RowScanArgsT {
    const REC* nrec;  // row-major
    int W, H;
    PRE* pre;
};
using RowScanArgs = RowScanArgsT<float4>;

template <class REC, class PRE>
__device__ __forceinline__ void pf_rowscan_body(const RowScanArgsT<REC, PRE>& a, int y) {
    const int W = pf_pitch(a.W), t = threadIdx.x, lane = t & 31, w = t >> 5;
    const size_t row = (size_t)y * W;
    __shared__ float4 s_warp[8];
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 carry = none, next = t < W ? ld4(a.nrec + row + t) : none;
    for (int x0 = 0; x0 < W; x0 += 256) {
        const int x = x0 + t;
        float4 v = next;
        next = x + 256 < W ? ld4(a.nrec + row + x + 256) : none;  // in flight during this scan (1080p 23.5 to 22.5 us)
        // inclusive warp scan, then the warps' totals
        for (int o = 1; o < 32; o <<= 1) {
            const float4 u = make_float4(__shfl_up_sync(0xffffffffu, v.x, o), __shfl_up_sync(0xffffffffu, v.y, o),
                                         __shfl_up_sync(0xffffffffu, v.z, o), __shfl_up_sync(0xffffffffu, v.w, o));
            if (lane >= o) v = add4(v, u);
        }
        if (lane == 31) s_warp[w] = v;
        __syncthreads();
        float4 before = carry;
        for (int k = 0; k < w; ++k) before = add4(before, s_warp[k]);
        if (x < W) st4(a.pre + row + x, add4(before, v));
        float4 total = carry;
        for (int k = 0; k < 8; ++k) total = add4(total, s_warp[k]);
        carry = total;
        __syncthreads();
    }
}

template <class REC, class PRE>
__global__ void __launch_bounds__(256) k_pf_rowscan(RowScanArgsT<REC, PRE> a) { pf_rowscan_body(a, blockIdx.x); }

// Per target pixel: a layer's sums (S.x, S.y) and (S.z, W) as register
// pairs so one packed FMA updates two of them; the far layer also holds its
// depth test's constants ka, kb.
struct NearAcc {
    float2 xy, zw;
};
struct FarAcc {
    float2 xy, zw;
    float ka, kb;
};
struct GreyNearAcc {  // (S, W)
    float2 zw;
};
struct GreyFarAcc {
    float2 zw;
    float ka, kb;
};
template <class REC>
struct AccOf {
    using Near = NearAcc;
    using Far = FarAcc;
};
template <>
struct AccOf<float2> {
    using Near = GreyNearAcc;
    using Far = GreyFarAcc;
};
template <class A>
__device__ __forceinline__ void acc_clear(A& a) { a.xy = a.zw = make_float2(0.f, 0.f); }
__device__ __forceinline__ void acc_clear(GreyNearAcc& a) { a.zw = make_float2(0.f, 0.f); }
__device__ __forceinline__ void acc_clear(GreyFarAcc& a) { a.zw = make_float2(0.f, 0.f); }
// the sums as (S.x, S.y, S.z, W)
template <class A>
__device__ __forceinline__ float4 acc_sum(const A& a) { return make_float4(a.xy.x, a.xy.y, a.zw.x, a.zw.y); }
__device__ __forceinline__ float4 acc_sum(const GreyNearAcc& a) { return make_float4(a.zw.x, a.zw.x, a.zw.x, a.zw.y); }
__device__ __forceinline__ float4 acc_sum(const GreyFarAcc& a) { return make_float4(a.zw.x, a.zw.x, a.zw.x, a.zw.y); }

// far = (S.x, S.y, S.z, W) of the far layer
template <class COL>
__device__ __forceinline__ float4 pf_finish(const float4& near, const float4& far, const COL* col, size_t pq,
                                            float4* aux) {
    const float3 Sn = f3(near.x, near.y, near.z), Sf = f3(far.x, far.y, far.z);
    const float Wn = near.w, Wf = far.w;
    float alpha = clamp01(Wn);
    float3 N = Wn > HDOF_PP_MIN_W ? (1.f / Wn) * Sn : f3(0, 0, 0);
    float3 F;
    if (Wf > HDOF_PP_MIN_W) F = (1.f / Wf) * Sf;
    else {
        float4 c = ld4(col + pq);
        F = f3(c.x, c.y, c.z);
    }
    if (aux) {  // layer colours and weights, kept for the adjoint
        aux[2 * pq] = make_float4(N.x, N.y, N.z, Wn);
        aux[2 * pq + 1] = make_float4(F.x, F.y, F.z, Wf);
    }
    float3 o = alpha * N + (1.f - alpha) * F;
    return make_float4(o.x, o.y, o.z, alpha);
}

template <class COL>
struct GatherArgs {
    const float* rh;
    const float* zq;
    const typename RecOf<COL>::T* nrec;
    const typename RecOf<COL>::T* frec;
    const COL* col;  // sharp colour (empty far layer)
    const float4* tmax;
    const typename RecOf<COL>::P* pre;  // row prefix of the near records
    int W, H, ntx, nty, kt;
    float kz_rel;
    float4* pp;
    float4* aux;
};

// one source into one target pixel, branch-free: s = clamp(r_q + 1/2 - d, 0, 1)
// (zero outside the disk, and zero layer records, add exact zeros); `in`
// false: the tap lies in the pixel's interior, already summed (weight 0 here)
__device__ __forceinline__ void acc(NearAcc& a, float d, float rh, float, const float4& n, bool in) {
    const float s = in ? __saturatef(rh - d) : 0.f;
    a.xy = fma2(s, n.x, n.y, a.xy);
    a.zw = fma2(s, n.z, n.w, a.zw);
}
__device__ __forceinline__ void acc(FarAcc& a, float d, float rh, float zq, const float4& f, bool) {
    const float t = __saturatef(rh - d) * __saturatef(fmaf(-zq, a.kb, a.ka));
    a.xy = fma2(t, f.x, f.y, a.xy);
    a.zw = fma2(t, f.z, f.w, a.zw);
}
__device__ __forceinline__ void acc(GreyNearAcc& a, float d, float rh, float, const float2& n, bool in) {
    a.zw = fma2(in ? __saturatef(rh - d) : 0.f, n.x, n.y, a.zw);
}
__device__ __forceinline__ void acc(GreyFarAcc& a, float d, float rh, float zq, const float2& f, bool) {
    a.zw = fma2(__saturatef(rh - d) * __saturatef(fmaf(-zq, a.kb, a.ka)), f.x, f.y, a.zw);
}

// Two taps of one column, one in each of the rows ya = j - s and yb = j + 1 + s
// around a thread's 2x2 block of rows j, j + 1.  Row ya lies s above the upper
// pixels and s + 1 above the lower ones, row yb the reverse, so the two rows
// share their distances: dn (s rows away) and df (s + 1).  The left pixels see
// the column at fresh distances, the right ones at the previous column's (the
// same offsets, so the same floats), carried in cn and cf (and the squared
// column offset in pdx2).  MASK: a pixel takes the tap only if its column
// offset exceeds its interior half-width for that row distance (squared: wn,
// wf).
struct TapCarry {
    float cn, cf, pdx2;
};
template <bool MASK, class A, class E>
__device__ __forceinline__ void pf_tap(A (&a)[4], TapCarry& c, float sn2, float sf2, float wn, float wf, float dx,
                                       float ra, float za, const E& ea, float rb, float zb, const E& eb) {
    const float dx2 = dx * dx;
    const float dn = sqrt_approx(dx2 + sn2), df = sqrt_approx(dx2 + sf2);
    acc(a[0], dn, ra, za, ea, !MASK || dx2 > wn);
    acc(a[1], c.cn, ra, za, ea, !MASK || c.pdx2 > wn);
    acc(a[2], df, ra, za, ea, !MASK || dx2 > wf);
    acc(a[3], c.cf, ra, za, ea, !MASK || c.pdx2 > wf);
    acc(a[0], df, rb, zb, eb, !MASK || dx2 > wf);
    acc(a[1], c.cf, rb, zb, eb, !MASK || c.pdx2 > wf);
    acc(a[2], dn, rb, zb, eb, !MASK || dx2 > wn);
    acc(a[3], c.cn, rb, zb, eb, !MASK || c.pdx2 > wn);
    c.cn = dn;
    c.cf = df;
    c.pdx2 = dx2;
}

// a loaded record
template <class REC>
struct EntryOf {
    using T = float4;
};
template <>
struct EntryOf<float2> {
    using T = float2;
};

// The taps of the columns xs .. xe (xs even, xe odd: whole pairs) of the rows
// at plane offsets oa and ob: one 256-bit load of a pair's two records and one
// float2 load of r + 1/2 (and z) per row; the threads of a row, two columns
// apart, read consecutive pairs.  A row outside the image (on_a, on_b false:
// its offset is the other row's) gets radii that reach nothing.
template <bool NEAR, bool MASK, class A, class REC>
__device__ __forceinline__ void pf_segment(A (&a)[4], float sn2, float sf2, float wn, float wf, int xs, int xe, int i,
                                           unsigned oa, unsigned ob, bool on_a, bool on_b,
                                           const float* __restrict__ rh, const float* __restrict__ zq,
                                           const REC* __restrict__ rec) {
    const float2* __restrict__ rh2 = reinterpret_cast<const float2*>(rh);
    const float2* __restrict__ zq2 = reinterpret_cast<const float2*>(zq);
    const float2 none = make_float2(-1e30f, -1e30f), zero = make_float2(0.f, 0.f);
    float dx = (float)(xs - i);
    TapCarry c;
    c.pdx2 = (dx - 1.f) * (dx - 1.f);
    c.cn = sqrt_approx(c.pdx2 + sn2);
    c.cf = sqrt_approx(c.pdx2 + sf2);
    unsigned ma = (oa + xs) >> 1, mb = (ob + xs) >> 1;
#pragma unroll PF_UNROLL
    for (int x = xs; x < xe; x += 2, ++ma, ++mb, dx += 2.f) {
        const float2 ra = on_a ? __ldg(&rh2[ma]) : none, rb = on_b ? __ldg(&rh2[mb]) : none;
        typename EntryOf<REC>::T ea0, ea1, eb0, eb1;
        ld_rec_pair(rec + 2 * (size_t)ma, ea0, ea1);
        ld_rec_pair(rec + 2 * (size_t)mb, eb0, eb1);
        const float2 za = NEAR ? zero : __ldg(&zq2[ma]), zb = NEAR ? zero : __ldg(&zq2[mb]);
        pf_tap<MASK>(a, c, sn2, sf2, wn, wf, dx, ra.x, za.x, ea0, rb.x, zb.x, eb0);
        pf_tap<MASK>(a, c, sn2, sf2, wn, wf, dx + 1.f, ra.y, za.y, ea1, rb.y, zb.y, eb1);
    }
}

template <class A>
__device__ __forceinline__ void add_sum(A& t, const float4& s) {
    t.xy = make_float2(t.xy.x + s.x, t.xy.y + s.y);
    t.zw = make_float2(t.zw.x + s.z, t.zw.y + s.w);
}
template <class A>
__device__ __forceinline__ void add_sum(A& t, const float2& s) {
    t.zw = make_float2(t.zw.x + s.x, t.zw.y + s.y);
}
__device__ __forceinline__ float4 sub_sum(const float4& a, const float4& b) {
    return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
__device__ __forceinline__ float2 sub_sum(const float2& a, const float2& b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float4 both_sums(const float4& a, const float4& b) { return add4(a, b); }
__device__ __forceinline__ float2 both_sums(const float2& a, const float2& b) { return make_float2(a.x + b.x, a.y + b.y); }
// pre[hi] - pre[lo - 1] of one row of the prefix
template <class PRE>
__device__ __forceinline__ PRE prefix_sum(const PRE* __restrict__ row, int lo, int hi) {
    const PRE s = __ldg(&row[hi]);
    return lo > 0 ? sub_sum(s, __ldg(&row[lo - 1])) : s;
}
__device__ __forceinline__ float prefix_weight(const float4* p) { return __ldg(&p->w); }
__device__ __forceinline__ float prefix_weight(const float2* p) { return __ldg(&p->y); }

// One layer's loop over a disk-shaped window of radius R around the 2x2 block
// at (i, j): every source feeding the layer within reach has r + 1/2 <= R, so
// only taps closer than R to one of the four pixels can weigh; per pair of
// source rows (j - s, j + 1 + s), the columns of that disk, in whole pairs of
// pixels (squared distances are exact integers in float).  The two rows share
// their bounds and their distances.
// Near layer with Rin >= 0: every source that feeds the near layer and lies
// within Rin of the block has r - 1/2 >= Rin, so a tap closer than Rin
// weighs exactly 1 and is summed from the row prefix `pre`.  PERPX false: per
// row, the columns closer than Rin to all four pixels are summed once (two
// loads, the same sum for every pixel) and the rest are tapped.  PERPX true:
// each pixel sums its own interior columns (two loads a pixel); the columns
// inside every pixel's interior are skipped, the rest are tapped with each
// pixel's interior masked out.
template <bool NEAR, bool PERPX, class A, class REC, class PRE>
__device__ __forceinline__ void pf_layer(A (&a)[4], float R, float Rin, int g, int i, int j, int W, int H,
                                         const float* __restrict__ rh, const float* __restrict__ zq,
                                         const REC* __restrict__ rec, const PRE* __restrict__ pre) {
    if (R < 0.f) return;  // nothing within reach feeds this layer
    // bounds lean outwards by 1e-3 pixel (float rounding); taps they add weigh 0
    const int G = (int)floorf(R + 1e-3f), Wp = pf_pitch(W);
    const float R2 = R * R, Rin2 = Rin * Rin;
    for (int s = g; s <= G; s += PF_G) {
        const int ya = j - s, yb = j + 1 + s;
        const bool on_a = ya >= 0, on_b = yb < H;
        if (!on_a && !on_b) break;
        const unsigned oa = (unsigned)(on_a ? ya : yb) * Wp, ob = (unsigned)(on_b ? yb : ya) * Wp;
        const float sn2 = (float)(s * s), sf2 = (float)((s + 1) * (s + 1));
        const int w = (int)(sqrt_approx(fmaxf(R2 - sn2, 0.f)) + 1e-3f);
        const int x0 = max(i - w, 0) & ~1, x1 = min(i + 1 + w, W - 1) | 1;
        int ls = x1 + 1, rs = x1;  // [ls, rs]: the columns that are not tapped (none)
        float wn = -1.f, wf = -1.f;
        if (PERPX) {
            // inward: no outward lean here (Rin already has its margin)
            const int in = sn2 <= Rin2 ? (int)floorf(sqrtf(Rin2 - sn2)) : -1;
            const int jf = sf2 <= Rin2 ? (int)floorf(sqrtf(Rin2 - sf2)) : -1;
            wn = in >= 0 ? (float)(in * in) : -1.f;
            wf = jf >= 0 ? (float)(jf * jf) : -1.f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int xa = i + (k & 1), wa = k < 2 ? in : jf, wb = k < 2 ? jf : in;
                if (xa >= W) continue;
                if (on_a && wa >= 0) add_sum(a[k], prefix_sum(pre + oa, max(xa - wa, 0), min(xa + wa, W - 1)));
                if (on_b && wb >= 0) add_sum(a[k], prefix_sum(pre + ob, max(xa - wb, 0), min(xa + wb, W - 1)));
            }
            if (jf >= 2) {
                // columns [i + 1 - jf, i + jf] lie in every pixel's interior
                ls = max(min(x1 + 1, (i + 2 - jf) & ~1), x0);
                rs = min(((i + jf + 1) & ~1) - 1, x1);
            }
        } else if (NEAR && sf2 < Rin2) {
            // columns [i + 1 - wi, i + wi] lie in every pixel's interior
            // (Rin's margin covers the root's rounding); rounded inwards to
            // whole pairs, so that the taps around them are whole pairs too
            const int wi = (int)sqrt_approx(Rin2 - sf2);
            const int la = (max(i + 1 - wi, 0) + 1) & ~1, ra = i + wi >= W - 1 ? Wp - 1 : ((i + wi + 1) & ~1) - 1;
            if (ra - la + 1 >= PF_MIN_IN) {
                PRE sum = on_a ? prefix_sum(pre + oa, la, ra) : PRE{};
                if (on_b) sum = both_sums(sum, prefix_sum(pre + ob, la, ra));
#pragma unroll
                for (int k = 0; k < 4; ++k) add_sum(a[k], sum);
                ls = la;
                rs = ra;
            }
        }
        if (x0 < ls) pf_segment<NEAR, PERPX>(a, sn2, sf2, wn, wf, x0, ls - 1, i, oa, ob, on_a, on_b, rh, zq, rec);
        if (rs < x1) pf_segment<NEAR, PERPX>(a, sn2, sf2, wn, wf, rs + 1, x1, i, oa, ob, on_a, on_b, rh, zq, rec);
    }
}

// the groups' partial sums of pixel p of the tile, in group order
__device__ __forceinline__ float4 pf_group_sum(const float4 (&part)[PF_G][TP * TP], int p) {
    float4 s = part[0][p];
#pragma unroll
    for (int g = 1; g < PF_G; ++g) s = add4(s, part[g][p]);
    return s;
}

// PF_G groups of 64 threads per 16x16 tile; thread t of a group gathers the
// 2x2 pixel block at (2 (t & 7), 2 (t >> 3)) over the group's source rows, so
// each loaded tap serves four pixels; the groups' sums are added in group
// order.
template <class COL>
__device__ __forceinline__ void pf_gather_body(const GatherArgs<COL>& ar, int tx, int ty) {
    const COL* __restrict__ col = ar.col;
    using Acc = AccOf<typename RecOf<COL>::T>;
    const float4* __restrict__ tmax = ar.tmax;
    const int W = ar.W, H = ar.H, ntx = ar.ntx, nty = ar.nty, kt = ar.kt;
    const int nk = (2 * kt + 1) * (2 * kt + 1);
    float4* __restrict__ pp = ar.pp;
    float4* __restrict__ aux = ar.aux;
    __shared__ int s_win[3];
    if (threadIdx.x < 2) s_win[threadIdx.x] = -1;
    if (threadIdx.x == 2) s_win[2] = 0x7f800000;  // +inf
    __syncthreads();
    // per layer: largest r + 1/2 over tiles whose feeding pixels can reach this tile
    for (int k = threadIdx.x; k < nk; k += blockDim.x) {
        int ox = k % (2 * kt + 1) - kt, oy = k / (2 * kt + 1) - kt;
        int x = tx + ox, y = ty + oy;
        if (x < 0 || y < 0 || x >= ntx || y >= nty) continue;
        const float4 r = __ldg(&tmax[y * ntx + x]);
        // pixel gap between the two tiles along each axis
        const float gx = ox == 0 ? 0.f : (float)((abs(ox) - 1) * TP + 1);
        const float gy = oy == 0 ? 0.f : (float)((abs(oy) - 1) * TP + 1);
        const float g2 = gx * gx + gy * gy;
        // positive floats order as their bit patterns
        if (r.x >= 0.f && g2 < (r.x + 0.5f) * (r.x + 0.5f)) atomicMax(&s_win[0], __float_as_int(r.x + 0.5f));
        if (r.y >= 0.f && g2 < (r.y + 0.5f) * (r.y + 0.5f)) atomicMax(&s_win[1], __float_as_int(r.y + 0.5f));
    }
    __syncthreads();
    // the layer's reach R (-1: none); a source weighs only closer than R
    const float Gn = s_win[0] < 0 ? -1.f : __int_as_float(s_win[0]);
    const float Gf = s_win[1] < 0 ? -1.f : __int_as_float(s_win[1]);
    // Near interior radius of the tile: a near source q at distance d weighs
    // exactly 1 if d <= r_q - 1/2, so Rin may grow while every tile T that
    // feeds the near layer and lies closer than Rin to this one has
    // r_min(T) - 1/2 >= Rin: Rin = min over T of max(r_min(T) - 1/2, gap(T)),
    // less a margin, at most Gn.  The interior path (two prefix loads per
    // thread and row) pays only when the interior is a good part of the
    // window: below PF_IN_SHARE Gn the plain loop runs.
    if (Gn >= 0.f) {
        for (int k = threadIdx.x; k < nk; k += blockDim.x) {
            int ox = k % (2 * kt + 1) - kt, oy = k / (2 * kt + 1) - kt;
            int x = tx + ox, y = ty + oy;
            if (x < 0 || y < 0 || x >= ntx || y >= nty) continue;
            const float4 r = __ldg(&tmax[y * ntx + x]);
            if (r.x < 0.f) continue;  // feeds no near layer
            const float gx = ox == 0 ? 0.f : (float)((abs(ox) - 1) * TP + 1);
            const float gy = oy == 0 ? 0.f : (float)((abs(oy) - 1) * TP + 1);
            const float lim = fmaxf(fmaxf(r.z - 0.5f, sqrtf(gx * gx + gy * gy) - 1e-3f), 0.f);
            atomicMin(&s_win[2], __float_as_int(lim));  // non-negative floats order as their bits
        }
        __syncthreads();
    }
    float Rin = Gn >= 0.f ? fminf(__int_as_float(s_win[2]), Gn) - 1e-3f : -1.f;
    if (Rin < PF_IN_SHARE * Gn) Rin = -1.f;
    // A prefix entry's rounding grows with the row's sum, and a sum over the
    // columns that all of a thread's pixels share carries the same rounding
    // into each of them.  Where a row of the window adds up to more than
    // PF_ROW_W (rows that cross the focus zone, whose sources weigh about 1
    // each; a blurred row weighs its length over the disk's area), each pixel
    // keeps its own columns and so its own rounding.
    bool per_px = false;
    if (Rin >= 0.f) {
        const int G = (int)floorf(Gn + 1e-3f), y0 = max(ty * TP - G, 0), y1 = min(ty * TP + TP - 1 + G, H - 1);
        bool big = false;
        for (int y = y0 + threadIdx.x; y <= y1; y += GATHER_THREADS)
            big |= !(prefix_weight(&ar.pre[(size_t)y * pf_pitch(W) + W - 1]) <= PF_ROW_W);
        per_px = __syncthreads_or(big);
    }
    // group g of the block's PF_G takes every PF_G-th source row; t is the
    // thread within its group.  s_part holds the groups' sums of one layer;
    // thread p < 256 adds and finishes pixel p of the tile.
    __shared__ float4 s_part[PF_G][TP * TP];
    const int g = threadIdx.x / PF_GROUP, t = threadIdx.x % PF_GROUP;
    const int li = 2 * (t & 7), lj = 2 * (t >> 3);
    const int i = tx * TP + li, j = ty * TP + lj;
    const bool in = i < W && j < H;
    // far layer first; its sums wait in the pixels' own pp slots (each pixel
    // is one thread's alone) so they hold no registers during the near loop
    if (Gf >= 0.f) {
        typename Acc::Far f[4];  // pixel (i + (k & 1), j + (k >> 1))
        if (in) {
            const float ka = 1.f + 1.f / ar.kz_rel;  // k_z = clamp(ka - z_q kb), kb = 1 / (kz_rel z_p)
            const size_t zo = (size_t)j * pf_pitch(W) + i;
            const float z00 = __ldg(&ar.zq[zo]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int x = i + (k & 1), y = j + (k >> 1);
                const float zp = x < W && y < H ? __ldg(&ar.zq[zo + (size_t)(k >> 1) * pf_pitch(W) + (k & 1)]) : z00;
                f[k].ka = ka;
                f[k].kb = 1.f / (ar.kz_rel * zp);
                acc_clear(f[k]);
            }
            pf_layer<false, false>(f, Gf, -1.f, g, i, j, W, H, ar.rh, ar.zq, ar.frec, ar.pre);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                s_part[g][(lj + (k >> 1)) * TP + li + (k & 1)] = acc_sum(f[k]);
        }
        __syncthreads();
        for (int p = threadIdx.x; p < TP * TP; p += GATHER_THREADS) {
            const int x = tx * TP + (p & 15), y = ty * TP + (p >> 4);
            if (x < W && y < H) pp[(size_t)y * W + x] = pf_group_sum(s_part, p);
        }
        __syncthreads();
    }
    if (in) {
        typename Acc::Near a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) acc_clear(a[k]);
        if (per_px) pf_layer<true, true>(a, Gn, Rin, g, i, j, W, H, ar.rh, ar.zq, ar.nrec, ar.pre);
        else pf_layer<true, false>(a, Gn, Rin, g, i, j, W, H, ar.rh, ar.zq, ar.nrec, ar.pre);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            s_part[g][(lj + (k >> 1)) * TP + li + (k & 1)] = acc_sum(a[k]);
    }
    __syncthreads();
    for (int p = threadIdx.x; p < TP * TP; p += GATHER_THREADS) {
        const int x = tx * TP + (p & 15), y = ty * TP + (p >> 4);
        if (x < W && y < H) {
            const size_t q = (size_t)y * W + x;
            const float4 far = Gf >= 0.f ? pp[q] : make_float4(0.f, 0.f, 0.f, 0.f);
            pp[q] = pf_finish(pf_group_sum(s_part, p), far, col, q, aux);
        }
    }
}

template <class COL>
struct GatherBlocks {
    static constexpr int MIN = PF_MINB;
};
template <class COL>
struct GatherBlocks<Grey<COL>> {
    static constexpr int MIN = 8;  // 64 registers; 6, 7, 8, 10 blocks at 4K: 1663, 1577, 1525, 1742 us
};
template <class COL>
__global__ void __launch_bounds__(GATHER_THREADS, GatherBlocks<COL>::MIN) k_pf_gather(GatherArgs<COL> a) {
    pf_gather_body(a, blockIdx.x, blockIdx.y);
}

using PrepF32 = PrepArgs<float4, float4>;
__global__ void __launch_bounds__(256) k_pf_rowscan_batch(const RowScanArgs* __restrict__ a, BatchGrid g) {
    int v, bx, by;
    g.locate(blockIdx.x, v, bx, by);
    pf_rowscan_body(batch_record(a, v), by);
}
__global__ void __launch_bounds__(256) k_pf_prep_batch(const PrepF32* __restrict__ a, BatchGrid g) {
    int v, bx, by;
    g.locate(blockIdx.x, v, bx, by);
    pf_prep_body(batch_record(a, v), bx, by);
}
__global__ void __launch_bounds__(GATHER_THREADS, PF_MINB)
    k_pf_gather_batch(const GatherArgs<float4>* __restrict__ a, BatchGrid g) {
    int v, bx, by;
    g.locate(blockIdx.x, v, bx, by);
    pf_gather_body(batch_record(a, v), bx, by);
}

// tiles of reach around a tile: radii up to r_max (+1/2 soft edge) span this many
int gather_tiles(float r_max) { return (int)std::ceil((r_max + 0.5f) / TP) + 1; }

std::mutex g_area_mu;
bool g_area_ready[64] = {false};
int g_area_count[64] = {0};

}  // namespace

int ensure_area_table(cudaStream_t s) {
    int dev = 0;
    HDOF_CUDA(cudaGetDevice(&dev), "area table: device");
    if (dev < 0 || dev >= 64) {
        set_error("area table: device index %d unsupported", dev);
        return HDOF_EUNSUPPORTED;
    }
    std::lock_guard<std::mutex> lock(g_area_mu);
    if (g_area_ready[dev]) return HDOF_OK;
    // lattice distances sqrt(k) with multiplicity n(k), |o| < 128.5
    const int R = 129;
    std::vector<int> mult(R * R + 1, 0);
    for (int b = -R; b <= R; ++b)
        for (int a = -R; a <= R; ++a) {
            int k = a * a + b * b;
            if (k <= R * R) mult[k]++;
        }
    std::vector<double> rad, pre_n, pre_nr;  // sorted sqrt(k), prefix sums of n and n*sqrt(k)
    double cn = 0, cnr = 0;
    for (int k = 0; k <= R * R; ++k)
        if (mult[k]) {
            double r = std::sqrt((double)k);
            rad.push_back(r);
            cn += mult[k];
            cnr += mult[k] * r;
            pre_n.push_back(cn);
            pre_nr.push_back(cnr);
        }
    // a(x) = #{|o| <= x - 1/2} + sum_{x-1/2 < |o| < x+1/2} (x + 1/2 - |o|)
    auto area = [&](double x) {
        auto cnt_le = [&](double v, bool strict) -> int {  // number of radii (<= v) or (< v)
            return (int)(strict ? std::lower_bound(rad.begin(), rad.end(), v) - rad.begin()
                                : std::upper_bound(rad.begin(), rad.end(), v) - rad.begin());
        };
        int full = cnt_le(x - 0.5, false);
        int part_end = cnt_le(x + 0.5, true);
        double nf = full ? pre_n[full - 1] : 0.0;
        double np = (part_end ? pre_n[part_end - 1] : 0.0) - nf;
        double nrp = (part_end ? pre_nr[part_end - 1] : 0.0) - (full ? pre_nr[full - 1] : 0.0);
        return nf + (x + 0.5) * np - nrp;
    };
    std::vector<double> bp;
    for (double r : rad) {
        if (r - 0.5 <= 128.0) bp.push_back(r - 0.5);
        if (r + 0.5 <= 128.0) bp.push_back(r + 0.5);
    }
    std::sort(bp.begin(), bp.end());
    bp.erase(std::unique(bp.begin(), bp.end()), bp.end());
    if ((int)bp.size() > AREA_MAX) {
        set_error("area table: %zu breakpoints exceed %d", bp.size(), AREA_MAX);
        return HDOF_EUNSUPPORTED;
    }
    std::vector<float4> tab(bp.size());
    for (size_t m = 0; m < bp.size(); ++m) {
        double a0 = area(bp[m]);
        double slope = 0.0;
        if (m + 1 < bp.size()) slope = (area(bp[m + 1]) - a0) / (bp[m + 1] - bp[m]);
        tab[m] = make_float4((float)bp[m], (float)a0, (float)slope, 0.f);
    }
    int n = (int)tab.size();
    std::vector<unsigned short> at(AREA_BUCKETS + 1);
    for (int b = 0, m = 0; b <= AREA_BUCKETS; ++b) {
        while (m + 1 < n && tab[m + 1].x <= b / 32.f) ++m;
        at[b] = (unsigned short)m;
    }
    HDOF_CUDA(cudaMemcpyToSymbolAsync(g_area_at, at.data(), sizeof(unsigned short) * at.size(), 0,
                                      cudaMemcpyHostToDevice, s),
              "area table: upload");
    HDOF_CUDA(cudaMemcpyToSymbolAsync(g_area, tab.data(), sizeof(float4) * tab.size(), 0, cudaMemcpyHostToDevice, s),
              "area table: upload");
    HDOF_CUDA(cudaStreamSynchronize(s), "area table: upload");
    g_area_ready[dev] = true;
    g_area_count[dev] = n;
    return HDOF_OK;
}

int area_table(const float4** tab, int* n) {
    int dev = 0;
    HDOF_CUDA(cudaGetDevice(&dev), "area table: device");
    void* p = nullptr;
    HDOF_CUDA(cudaGetSymbolAddress(&p, g_area), "area table: symbol");
    *tab = static_cast<const float4*>(p);
    *n = (dev >= 0 && dev < 64) ? g_area_count[dev] : 0;
    return HDOF_OK;
}

}  // namespace hdof

using namespace hdof;

namespace hdof {

template <class ND, class COL>
static int run_postfilter(const hdof_gbuf* in, const Coc& coc, const hdof_params* p, float* pp, float4* aux,
                          void* scratch, cudaStream_t s, const float* lens_dev, float t) {
    using REC = typename RecOf<COL>::T;
    using PRE = typename RecOf<COL>::P;
    int rc;
    if ((rc = ensure_area_table(s))) return rc;
    const int W = in->width, H = in->height;
    ViewWs w = {};
    pf_regions(w, static_cast<char*>(scratch), ws_layout(W, H, p));
    REC* nrec = reinterpret_cast<REC*>(w.nrec);
    REC* frec = reinterpret_cast<REC*>(w.frec);
    PRE* pre = reinterpret_cast<PRE*>(w.pre);
    const COL* col = static_cast<const COL*>(in->col);
    const int ntx = (W + TP - 1) / TP, nty = (H + TP - 1) / TP;
    dim3 grid(ntx, nty);
    {
        ProfScope ps_("pf_prep", s);
        k_pf_prep<<<grid, 256, 0, s>>>(PrepArgs<ND, COL>{static_cast<const ND*>(in->nd), col, W, H, coc, p->r_max, ntx,
                                                         w.rh, w.zq, nrec, frec, w.tmax, lens_dev, t});
        HDOF_LAUNCHED("post-filter prep");
    }
    {
        ProfScope ps_("pf_rowscan", s);
        k_pf_rowscan<<<H, 256, 0, s>>>(RowScanArgsT<REC, PRE>{nrec, W, H, pre});
        HDOF_LAUNCHED("post-filter row prefix");
    }
    // the taps are served from L1: a small shared-memory carve-out
    ProfScope ps_("pf_gather", s);
    cudaFuncSetAttribute(k_pf_gather<COL>, cudaFuncAttributePreferredSharedMemoryCarveout, GATHER_CARVEOUT);
    k_pf_gather<COL><<<grid, GATHER_THREADS, 0, s>>>(GatherArgs<COL>{w.rh, w.zq, nrec, frec, col, w.tmax, pre, W, H, ntx,
                                                                     nty, gather_tiles(p->r_max), p->kz_rel,
                                                                     reinterpret_cast<float4*>(pp), aux});
    HDOF_LAUNCHED("post-filter gather");
    return HDOF_OK;
}

int launch_postfilter(const hdof_gbuf* in, const Coc& coc, const hdof_params* p, float* pp, float4* aux,
                      void* scratch, cudaStream_t s, const float* lens_dev, float t) {
    if (bokeh_shaped(p)) {
        if (aux || lens_dev) {
            set_error("post-filter: shaped bokeh has no adjoint records");
            return HDOF_EUNSUPPORTED;
        }
        return launch_bokeh(in, coc, p, pp, scratch, s);
    }
    const bool f32n = in->dtype_nd == HDOF_F32, f32c = in->dtype_col == HDOF_F32;
    if (f32n && f32c) return run_postfilter<float4, float4>(in, coc, p, pp, aux, scratch, s, lens_dev, t);
    if (f32n) return run_postfilter<float4, bf164s>(in, coc, p, pp, aux, scratch, s, lens_dev, t);
    if (f32c) return run_postfilter<half4s, float4>(in, coc, p, pp, aux, scratch, s, lens_dev, t);
    return run_postfilter<half4s, bf164s>(in, coc, p, pp, aux, scratch, s, lens_dev, t);
}

}  // namespace hdof

extern "C" int hdof_postfilter(const hdof_gbuf* in, const hdof_camera* cam, const hdof_lens* lens,
                               const hdof_params* p, float* pp, void* workspace, size_t workspace_bytes,
                               void* stream) {
    clear_error();
    int rc;
    if ((rc = check_camera(cam, "hdof_postfilter")) || (rc = check_lens(lens, "hdof_postfilter")) ||
        (rc = check_params(p, "hdof_postfilter")) || (rc = check_gbuf(in, "hdof_postfilter", false)))
        return rc;
    HDOF_CHECK_ARG(pp, "hdof_postfilter: pp output is required");
    HDOF_CHECK_ARG(in->width == cam->width && in->height == cam->height, "hdof_postfilter: gbuf/camera size mismatch");
    WsLayout L = ws_layout(in->width, in->height, p);
    HDOF_CHECK_ARG(workspace && workspace_bytes >= L.total, "hdof_postfilter: workspace of %zu bytes < %zu",
                   workspace_bytes, L.total);
    return launch_postfilter(in, make_coc(*lens, in->height, cam->tan_half_fovy), p, pp, nullptr,
                             static_cast<char*>(workspace) + L.pf_off, as_stream(stream));
}

namespace hdof {
namespace {

// The specular luminance (col.w) of every pixel as an opaque grey colour.
template <class COL>
__global__ void __launch_bounds__(256) k_spec_plane(const COL* __restrict__ col, size_t n, float4* __restrict__ out) {
    const size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const float s = ld4(col + q).w;
    out[q] = make_float4(s, s, s, s);
}

}  // namespace
}  // namespace hdof

extern "C" int hdof_postfilter_spec(const hdof_gbuf* in, const hdof_camera* cam, const hdof_lens* lens,
                                    const hdof_params* p, float* pp_spec, void* workspace, size_t workspace_bytes,
                                    void* stream) {
    clear_error();
    int rc;
    if ((rc = check_camera(cam, "hdof_postfilter_spec")) || (rc = check_lens(lens, "hdof_postfilter_spec")) ||
        (rc = check_params(p, "hdof_postfilter_spec")) || (rc = check_gbuf(in, "hdof_postfilter_spec", false)))
        return rc;
    HDOF_CHECK_ARG(pp_spec, "hdof_postfilter_spec: pp_spec output is required");
    HDOF_CHECK_ARG(in->width == cam->width && in->height == cam->height,
                   "hdof_postfilter_spec: gbuf/camera size mismatch");
    WsLayout L = ws_layout(in->width, in->height, p);
    HDOF_CHECK_ARG(workspace && workspace_bytes >= L.total, "hdof_postfilter_spec: workspace of %zu bytes < %zu",
                   workspace_bytes, L.total);
    // the shaped post-filter's grey plane sits below the post-filter's region (the mask and trace
    // scratch, at least 16 bytes per pixel since spp_max >= 1; 16-byte accesses only)
    const size_t n = (size_t)in->width * in->height;
    HDOF_CHECK_ARG(n * sizeof(float4) <= L.pf_off, "hdof_postfilter_spec: no room for the specular plane");
    cudaStream_t s = as_stream(stream);
    const Coc coc = make_coc(*lens, in->height, cam->tan_half_fovy);
    void* scratch = static_cast<char*>(workspace) + L.pf_off;
    if (!bokeh_shaped(p)) {
        const bool f32n = in->dtype_nd == HDOF_F32, f32c = in->dtype_col == HDOF_F32;
        if (f32n && f32c)
            return run_postfilter<float4, Grey<float4>>(in, coc, p, pp_spec, nullptr, scratch, s, nullptr, 0.f);
        if (f32n) return run_postfilter<float4, Grey<bf164s>>(in, coc, p, pp_spec, nullptr, scratch, s, nullptr, 0.f);
        if (f32c) return run_postfilter<half4s, Grey<float4>>(in, coc, p, pp_spec, nullptr, scratch, s, nullptr, 0.f);
        return run_postfilter<half4s, Grey<bf164s>>(in, coc, p, pp_spec, nullptr, scratch, s, nullptr, 0.f);
    }
    HDOF_CHECK_ALIGNED(workspace, 16, "hdof_postfilter_spec");
    float4* plane = static_cast<float4*>(workspace);
    {
        ProfScope ps_("pf_spec_plane", s);
        const unsigned blocks = (unsigned)((n + 255) / 256);
        if (in->dtype_col == HDOF_F32)
            k_spec_plane<<<blocks, 256, 0, s>>>(static_cast<const float4*>(in->col), n, plane);
        else
            k_spec_plane<<<blocks, 256, 0, s>>>(static_cast<const bf164s*>(in->col), n, plane);
    }
    HDOF_LAUNCHED("specular plane");
    hdof_gbuf g = *in;
    g.dtype_col = HDOF_F32;
    g.col = plane;
    return launch_bokeh(&g, coc, p, pp_spec, scratch, s);
}

namespace hdof {

size_t pf_prep_args_size() { return sizeof(PrepF32); }
void pf_prep_fill(const hdof_view& v, const ViewWs& w, unsigned*, void* dst, int* gx, int* gy) {
    const int W = v.cam.width, H = v.cam.height, ntx = (W + TP - 1) / TP;
    *reinterpret_cast<PrepF32*>(dst) =
        PrepF32{static_cast<const float4*>(v.g.nd), static_cast<const float4*>(v.g.col), W, H,
                make_coc(v.lens, H, v.cam.tan_half_fovy), v.params.r_max, ntx, w.rh, w.zq, w.nrec, w.frec, w.tmax};
    *gx = ntx;
    *gy = (H + TP - 1) / TP;
}
void pf_prep_launch_batch(const void* args, BatchGrid g, int blocks, cudaStream_t s) {
    ProfScope ps_("batch_pf_prep", s);
    k_pf_prep_batch<<<blocks, 256, 0, s>>>(static_cast<const PrepF32*>(args), g);
}

size_t pf_rowscan_args_size() { return sizeof(RowScanArgs); }
void pf_rowscan_fill(const hdof_view& v, const ViewWs& w, unsigned*, void* dst, int* gx, int* gy) {
    *reinterpret_cast<RowScanArgs*>(dst) = RowScanArgs{w.nrec, v.cam.width, v.cam.height, w.pre};
    *gx = 1;  // one block per row
    *gy = v.cam.height;
}
void pf_rowscan_launch_batch(const void* args, BatchGrid g, int blocks, cudaStream_t s) {
    ProfScope ps_("batch_pf_rowscan", s);
    k_pf_rowscan_batch<<<blocks, 256, 0, s>>>(static_cast<const RowScanArgs*>(args), g);
}

size_t pf_gather_args_size() { return sizeof(GatherArgs<float4>); }
void pf_gather_fill(const hdof_view& v, const ViewWs& w, unsigned*, void* dst, int* gx, int* gy) {
    const int W = v.cam.width, H = v.cam.height, ntx = (W + TP - 1) / TP, nty = (H + TP - 1) / TP;
    *reinterpret_cast<GatherArgs<float4>*>(dst) =
        GatherArgs<float4>{w.rh, w.zq, w.nrec, w.frec, static_cast<const float4*>(v.g.col), w.tmax, w.pre, W, H, ntx,
                           nty, gather_tiles(v.params.r_max), v.params.kz_rel, reinterpret_cast<float4*>(v.pp),
                           nullptr};
    *gx = ntx;
    *gy = nty;
    cudaFuncSetAttribute(k_pf_gather_batch, cudaFuncAttributePreferredSharedMemoryCarveout, GATHER_CARVEOUT);
}
void pf_gather_launch_batch(const void* args, BatchGrid g, int blocks, cudaStream_t s) {
    ProfScope ps_("batch_pf_gather", s);
    k_pf_gather_batch<<<blocks, GATHER_THREADS, 0, s>>>(static_cast<const GatherArgs<float4>*>(args), g);
}

}  // namespace hdof
