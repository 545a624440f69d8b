// spatio-temporal reconstruction of the ray-traced layers
// (Reconstruction section).
//
// Temporal (k_temporal, one thread per pixel): near and far colours are
// accumulated separately with an exponential moving average, each weighted
// by its share of the hit ratio.  Near terms are reprojected with the
// screen-space motion vector; far terms with the previous-frame projection
// of the average far world position of the pixel's far hits (or of its
// neighbours' when it has none, or of its G-buffer surface).  The composed
// colour uses this frame's hit ratio when the camera moved and the
// accumulated one otherwise; each layer is normalised by its accumulated
// hit-ratio weight.  The reconstructed CoC blends this frame's near and far
// CoC by the accumulated hit ratio.
//
// Spatial (k_spatial, one thread per traced pixel): a circular gather scaled
// by the pixel's CoC that rejects samples whose CoC radius is smaller than
// their distance, blended by the clamped luminance variance so converged
// regions are not over-blurred.
#include "batch.cuh"
#include "internal.h"

namespace hdof {
namespace {

struct TemporalArgs {
    Cam cam, prev;
    int W, H;
    float alpha, alpha_k;  // EMA weight; per-pixel blend factor threshold (0 = fixed weight)
    int moved;
    const float4* rt;  // 3 per pixel
    const uint8_t* spp;
    const float2* mv;
    const float4* hn;  // previous history
    const float4* hf;
    const float2* hm;
    const uint8_t* hl;
    float4* on;  // new history
    float4* of;
    float2* om;
    uint8_t* ol;
    float4* crt;
    float* hacc;
};

__device__ __forceinline__ void acc(float4& o, float w, float4 v) {
    o.x = fmaf(w, v.x, o.x);
    o.y = fmaf(w, v.y, o.y);
    o.z = fmaf(w, v.z, o.z);
    o.w = fmaf(w, v.w, o.w);
}
__device__ __forceinline__ void acc(float2& o, float w, float2 v) {
    o.x = fmaf(w, v.x, o.x);
    o.y = fmaf(w, v.y, o.y);
}
__device__ __forceinline__ void scale(float4& o, float s) {
    o.x *= s;
    o.y *= s;
    o.z *= s;
    o.w *= s;
}
__device__ __forceinline__ void scale(float2& o, float s) {
    o.x *= s;
    o.y *= s;
}
__device__ __forceinline__ void zero(float4& o) { o = make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ void zero(float2& o) { o = make_float2(0.f, 0.f); }

// The four bilinear taps of a history position: their pixels (the pixel
// itself for a tap outside the image) and history lengths (0 there).  All
// four hlen loads are in flight together, and then all of a plane's: with
// each tap's plane load behind its own hlen test the kernel waited on eight
// dependent loads per plane (1080p with half the pixels traced: 107 us; so
// 94).  The sums stay in hist_sample's form, whose bits the mask of the next
// frame depends on.
struct HistTaps {
    unsigned q[4];
    int hl[4];
};
__device__ __forceinline__ HistTaps hist_taps(const TemporalArgs& a, bool valid, float ux, float uy, size_t self) {
    HistTaps h;
    const float x0 = floorf(ux), y0 = floorf(uy);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float x = x0 + (k & 1), y = y0 + (k >> 1);
        const bool in = valid && x >= 0.f && y >= 0.f && x < (float)a.W && y < (float)a.H;
        h.q[k] = in ? (unsigned)y * (unsigned)a.W + (unsigned)x : (unsigned)self;
        h.hl[k] = __ldg(&a.hl[h.q[k]]);
        if (!in) h.hl[k] = 0;
    }
    return h;
}
template <class T>
__device__ __forceinline__ void hist_load(const HistTaps& h, const T* __restrict__ plane, T (&v)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __ldg(&plane[h.q[k]]);
}
// bilinear history sample over taps that hold history (hlen > 0), renormalised;
// invalid below a total tap weight of 1e-3.  hmax: largest hlen among taps
// with non-zero weight.
template <class T>
__device__ __forceinline__ bool hist_sample(const HistTaps& h, const T (&v)[4], float ux, float uy, T& out, int* hmax) {
    const float x0 = floorf(ux), y0 = floorf(uy), fx = ux - x0, fy = uy - y0;
    float ws = 0.f;
    zero(out);
    if (hmax) *hmax = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (h.hl[k] == 0) continue;
        float w = ((k & 1) ? fx : 1.f - fx) * ((k >> 1) ? fy : 1.f - fy);
        ws += w;
        acc(out, w, v[k]);
        if (hmax && w > 0.f && h.hl[k] > *hmax) *hmax = h.hl[k];
    }
    if (!(ws >= HDOF_HIST_MIN_W)) return false;
    scale(out, 1.f / ws);
    return true;
}

template <class ND>
__device__ __forceinline__ void temporal_body(const TemporalArgs& a, const ND* __restrict__ nd, int bx, int by) {
    int i = bx * 32 + (threadIdx.x & 31), j = by * 8 + (threadIdx.x >> 5);
    if (i >= a.W || j >= a.H) return;
    size_t q = (size_t)j * a.W + i;
    if (a.spp[q] == 0) {
        a.ol[q] = 0;
        a.crt[q] = make_float4(0.f, 0.f, 0.f, -1.f);
        return;
    }
    const float4 r0 = __ldg(&a.rt[3 * q]), r1 = __ldg(&a.rt[3 * q + 1]), r2 = __ldg(&a.rt[3 * q + 2]);
    const float h = r0.w, cn = r1.w, cf = r2.w;
    const bool nok = cn >= 0.f, fok = cf >= 0.f;
    float3 Cn = f3(r0.x, r0.y, r0.z), Cf = f3(r1.x, r1.y, r1.z);
    float3 Ccur = nok ? (fok ? h * Cn + (1.f - h) * Cf : Cn) : Cf;
    float Y = luminance(Ccur);
    // near reprojection
    float2 m = __ldg(&a.mv[q]);
    float un = (float)i - m.x, vn = (float)j - m.y;
    const HistTaps tn = hist_taps(a, true, un, vn, q);
    float4 vnear[4];
    float2 vmom[4];
    hist_load(tn, a.hn, vnear);
    hist_load(tn, a.hm, vmom);
    float4 hn;
    float2 hm = make_float2(0.f, 0.f);
    int hl = 0;
    // far world position
    float3 P;
    if (fok) {
        P = f3(r2.x, r2.y, r2.z);
    } else {
        float3 s = f3(0.f, 0.f, 0.f);
        int cnt = 0;
#pragma unroll
        for (int b = -1; b <= 1; ++b) {
            // a row's loads together; rt of an untraced neighbour is not used
            bool on[3];
            float4 p2[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int x = i + c - 1, y = j + b;
                on[c] = (b != 0 || c != 1) && x >= 0 && y >= 0 && x < a.W && y < a.H;
                const size_t qq = on[c] ? (size_t)y * a.W + x : q;
                on[c] = on[c] && __ldg(&a.spp[qq]) != 0;
                p2[c] = __ldg(&a.rt[3 * qq + 2]);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (on[c] && p2[c].w >= 0.f) {
                    s = s + f3(p2[c].x, p2[c].y, p2[c].z);
                    ++cnt;
                }
        }
        if (cnt > 0) {
            P = (1.f / (float)cnt) * s;
        } else {
            float3 d = pinhole_dir(a.cam, i + 0.5f + a.cam.jx, j + 0.5f + a.cam.jy);
            P = a.cam.pos + ldz(nd + q) * d;
        }
    }
    float uf, vf;
    float4 hf;
    const bool seen = project(a.prev, P, uf, vf);
    const HistTaps tf = hist_taps(a, seen, seen ? uf : 0.f, seen ? vf : 0.f, q);
    float4 vfar[4];
    hist_load(tf, a.hf, vfar);
    const bool vn_ok = hist_sample(tn, vnear, un, vn, hn, &hl);
    if (vn_ok) hist_sample(tn, vmom, un, vn, hm, (int*)nullptr);
    const bool vf_ok = seen && hist_sample(tf, vfar, uf, vf, hf, (int*)nullptr);
    // EMA weight: fixed, or per pixel from the temporal gradient (the paper's
    // per-pixel blend factors against ghosting): the larger of this frame's
    // luminance change against the reprojected history beyond alpha_k of its
    // per-frame spread (relative to the larger luminance) and the hit ratio's
    // change beyond alpha_k binomial standard errors; alpha rises towards 1
    float al = a.alpha;
    if (a.alpha_k > 0.f && vn_ok) {
        const float sg = sqrtf(fmaxf(0.f, hm.y - hm.x * hm.x));
        const float den = fmaxf(fmaxf(Y, hm.x), 1e-3f);
        float lam = fminf(fmaxf((fabsf(Y - hm.x) - a.alpha_k * sg) / den, 0.f), 1.f);
        const float hb = hn.w, se = sqrtf(fmaxf(hb * (1.f - hb), 0.f) / (float)a.spp[q]);
        const float lh = fminf(fmaxf(fabsf(h - hb) - a.alpha_k * se, 0.f), 1.f);
        lam = fmaxf(lam, lh);
        al = fmaf(1.f - al, lam, al);
    }
    float4 cur_n = make_float4(h * Cn.x, h * Cn.y, h * Cn.z, h);
    float4 cur_f = make_float4((1.f - h) * Cf.x, (1.f - h) * Cf.y, (1.f - h) * Cf.z, 1.f - h);
    float4 on = vn_ok ? make_float4(fmaf(al, cur_n.x - hn.x, hn.x), fmaf(al, cur_n.y - hn.y, hn.y),
                                    fmaf(al, cur_n.z - hn.z, hn.z), fmaf(al, cur_n.w - hn.w, hn.w))
                      : cur_n;
    float4 of = vf_ok ? make_float4(fmaf(al, cur_f.x - hf.x, hf.x), fmaf(al, cur_f.y - hf.y, hf.y),
                                    fmaf(al, cur_f.z - hf.z, hf.z), fmaf(al, cur_f.w - hf.w, hf.w))
                      : cur_f;
    float2 om = vn_ok ? make_float2(fmaf(al, Y - hm.x, hm.x), fmaf(al, Y * Y - hm.y, hm.y)) : make_float2(Y, Y * Y);
    int nh = vn_ok ? hl + 1 : 1;
    a.on[q] = on;
    a.of[q] = of;
    a.om[q] = om;
    a.ol[q] = (uint8_t)(nh > 255 ? 255 : nh);
    // accumulated hit ratio and composition
    float Bn = on.w, Bf = of.w;
    float Hacc = (Bn + Bf >= HDOF_EMPTY_W) ? Bn / (Bn + Bf) : h;
    bool an = Bn >= HDOF_EMPTY_W, af = Bf >= HDOF_EMPTY_W;
    float hw = a.moved ? h : Hacc;
    float3 CnA = an ? (1.f / Bn) * f3(on.x, on.y, on.z) : f3(0, 0, 0);
    float3 CfA = af ? (1.f / Bf) * f3(of.x, of.y, of.z) : f3(0, 0, 0);
    float3 C = !an ? CfA : (!af ? CnA : hw * CnA + (1.f - hw) * CfA);
    float crt_c = !nok ? cf : (!fok ? cn : Hacc * cn + (1.f - Hacc) * cf);
    a.crt[q] = make_float4(C.x, C.y, C.z, crt_c);
    a.hacc[q] = Hacc;
}

// 3 resident blocks (80 registers): with 2 or 5 the loads in flight of hist_taps gain nothing
template <class ND>
__global__ void __launch_bounds__(256, 3) k_temporal(TemporalArgs a, const ND* __restrict__ nd) {
    temporal_body(a, nd, blockIdx.x, blockIdx.y);
}

struct TemporalBatch {
    TemporalArgs t;
    const float4* nd;
};
// 4 blocks (64 registers; 94 left two): twelve views 43.48 to 43.12 ms, 5 blocks 43.15
__global__ void __launch_bounds__(256, 4) k_temporal_batch(const TemporalBatch* __restrict__ a, BatchGrid g) {
    int v, bx, by;
    g.locate(blockIdx.x, v, bx, by);
    const TemporalBatch& r = batch_record(a, v);
    temporal_body(r.t, r.nd, bx, by);
}

#ifndef HDOF_SP_UNROLL
#define HDOF_SP_UNROLL 4  // unroll of the spatial gather's tap loop
#endif
constexpr int SP_UNROLL = HDOF_SP_UNROLL;

struct SpatialArgs {
    const float4* crt;
    const float2* mom;
    const uint8_t* hlen;
    int W, H;
    float r_s, var_ref;
    float4* crec;
    float4* aux;
};

// a traced pixel's reconstructed colour from its gathered sums: blended with
// its own by beta = clamp(sigma_L / var_ref, 0, 1) (1 while its history is young)
__device__ __forceinline__ void spatial_finish(const SpatialArgs& a, size_t q, const float4& cp, const float3& S,
                                               float Ws) {
    float2 m = __ldg(&a.mom[q]);
    float sig = sqrtf(fmaxf(0.f, m.y - m.x * m.x));
    float beta = __ldg(&a.hlen[q]) < 2 ? 1.f : clamp01(sig / a.var_ref);
    float3 Csp = (1.f / Ws) * S;
    if (a.aux) a.aux[q] = make_float4(Csp.x, Csp.y, Csp.z, Ws);  // kept for the adjoint
    a.crec[q] = make_float4(cp.x + beta * (Csp.x - cp.x), cp.y + beta * (Csp.y - cp.y), cp.z + beta * (Csp.z - cp.z),
                            0.f);
}

// A tile's traced pixels are few or many and their windows 1 to 33 rows, so
// each pixel's rows are shared by SP_G threads: group g takes the source rows
// y with y mod SP_G = g (absolute, so a pixel's sums do not depend on the
// window of the pixel beside it), and the groups are added in order.
constexpr int SP_G = 4;

struct PairSums {
    float4 l, r;  // (S rgb, W) of the left and the right pixel
};

// One thread gathers group g's rows for the horizontally adjacent pixels
// (i, j) and (i + 1, j) (tl, tr: which of them is traced) over the union of
// their windows: each tap is loaded once, and the right pixel's distance to a
// tap is the left pixel's distance to the previous tap (the same float
// operations); the union only adds taps of weight exactly 0.  An untraced
// pixel of the pair gets reach 0.
__device__ __forceinline__ PairSums spatial_pair(const SpatialArgs& a, int i, int j, bool tl, bool tr, int g) {
    const float4* __restrict__ crt = a.crt;
    const int W = a.W, H = a.H;
    const float r_s = a.r_s, Rq = r_s + 0.5f;
    const size_t q = (size_t)j * W + i;
    // a tap weighs only if d < R = min(c/2, r_s) + 1/2: per row, the columns of
    // that disk (the bounds lean outwards by 1e-3 pixel; the taps they add
    // weigh 0).  s(r - d) = clamp(r + 1/2 - d, 0, 1): the half folded into the
    // radii (R here; for the neighbour min(c/2 + 1/2, r_s + 1/2))
    const float Rl = tl ? fminf(__ldg(&crt[q].w) * 0.5f, r_s) + 0.5f : 0.f;
    const float Rr = tr ? fminf(__ldg(&crt[q + 1].w) * 0.5f, r_s) + 0.5f : 0.f;
    const float Rl2 = Rl * Rl, Rr2 = Rr * Rr;
    const int K = (int)floorf(fmaxf(Rl, Rr) + 1e-3f);
    f32x2 lxy = 0ull, lzw = 0ull, rxy = 0ull, rzw = 0ull;  // (S.x, S.y), (S.z, W)
    const int y0 = max(j - K, 0), y1 = min(j + K, H - 1);
    for (int y = y0 + ((g - y0) & (SP_G - 1)); y <= y1; y += SP_G) {
        const float dy = (float)(y - j), dy2 = dy * dy;
        const int wl = (int)(sqrt_approx(fmaxf(Rl2 - dy2, 0.f)) + 1e-3f);
        const int wr = (int)(sqrt_approx(fmaxf(Rr2 - dy2, 0.f)) + 1e-3f);
        const int x0 = max(min(i - wl, i + 1 - wr), 0), x1 = min(max(i + wl, i + 1 + wr), W - 1);
        const float4* row = crt + (size_t)y * W;
        float dx = (float)(x0 - i);
        float dprev = sqrt_approx(fmaf(dx - 1.f, dx - 1.f, dy2));  // the right pixel's distance to x0
#pragma unroll SP_UNROLL
        for (int x = x0; x <= x1; ++x, dx += 1.f) {
            const float4 c = __ldg(&row[x]);
            const float dl = sqrt_approx(fmaf(dx, dx, dy2)), dr = dprev;
            // an untraced neighbour (written as (0, 0, 0, -1)) weighs
            // clamp(-d, 0, 1) = 0 times colour 0: it adds nothing
            const float rq = fminf(fmaf(c.w, 0.5f, 0.5f), Rq);
            const float ql = __saturatef(Rl - dl) * __saturatef(rq - dl);
            const float qr = __saturatef(Rr - dr) * __saturatef(rq - dr);
            const f32x2 cxy = pk2(c.x, c.y), czw = pk2(c.z, 1.f), qql = pk2(ql, ql), qqr = pk2(qr, qr);
            lxy = ffma2(qql, cxy, lxy);
            lzw = ffma2(qql, czw, lzw);
            rxy = ffma2(qqr, cxy, rxy);
            rzw = ffma2(qqr, czw, rzw);
            dprev = dl;
        }
    }
    const float2 l0 = unpk2(lxy), l1 = unpk2(lzw), r0 = unpk2(rxy), r1 = unpk2(rzw);
    PairSums o;
    o.l = make_float4(l0.x, l0.y, l1.x, l1.y);
    o.r = make_float4(r0.x, r0.y, r1.x, r1.y);
    return o;
}

// Block = one 16 x TH tile as 8 x TH horizontal pixel pairs, SP_G threads per
// pair: the n pairs holding a traced pixel are compacted, thread t takes
// group t / n of pair t mod n, so the threads that run fill whole warps and
// all gather.  Bound by the latency of the taps (L1 hits): with one thread
// per pair the widest windows (1089 serial taps) outlasted the rest of the
// grid at 8-17% of the warps active.  75 -> 37 us at 1024x1024 (the fitting
// step's frame), 194 -> 186 us at 1080p with half the pixels traced at random
// CoCs (bound by issue there: lanes of unlike windows).
constexpr int SP_TW = 16;
template <int TH>
constexpr int sp_threads() {
    return SP_G * SP_TW * TH / 2;
}
template <int TH>
__device__ __forceinline__ void spatial_body(const SpatialArgs& a, int bx, int by) {
    constexpr int PW = SP_TW / 2, NP = PW * TH;
    __shared__ unsigned short s_list[NP];
    __shared__ int s_cnt[NP / 32];
    __shared__ float4 s_part[2][sp_threads<TH>()];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    bool tl = false, tr = false;
    unsigned tm = 0;
    if (t < NP) {  // whole warps
        const int i0 = bx * SP_TW + 2 * (t % PW), j0 = by * TH + t / PW;
        const bool row_in = j0 < a.H;
        tl = row_in && i0 < a.W && __ldg(&a.crt[(size_t)j0 * a.W + i0].w) >= 0.f;
        tr = row_in && i0 + 1 < a.W && __ldg(&a.crt[(size_t)j0 * a.W + i0 + 1].w) >= 0.f;
        tm = __ballot_sync(0xffffffffu, tl || tr);
        if (lane == 0) s_cnt[w] = __popc(tm);
    }
    __syncthreads();
    int off = 0, n = 0;
#pragma unroll
    for (int c = 0; c < NP / 32; ++c) {
        off += c < w ? s_cnt[c] : 0;
        n += s_cnt[c];
    }
    if (n == 0) return;  // the whole block
    // the pair's slot and which of its pixels are traced
    if (tl || tr)
        s_list[off + __popc(tm & ((1u << lane) - 1u))] = (unsigned short)(t | (tl ? 0x8000 : 0) | (tr ? 0x4000 : 0));
    __syncthreads();
    if (t < SP_G * n) {
        const int g = t / n, e = s_list[t - g * n], p = e & 0x3fff;
        const PairSums o = spatial_pair(a, bx * SP_TW + 2 * (p % PW), by * TH + p / PW, (e & 0x8000) != 0,
                                        (e & 0x4000) != 0, g);
        s_part[0][t] = o.l;
        s_part[1][t] = o.r;
    }
    __syncthreads();
    for (int k = t; k < 2 * n; k += sp_threads<TH>()) {  // pixel k & 1 of pair k / 2
        const int e = s_list[k >> 1], p = e & 0x3fff;
        if (!(e & ((k & 1) ? 0x4000 : 0x8000))) continue;
        float4 S = s_part[k & 1][k >> 1];
#pragma unroll
        for (int g = 1; g < SP_G; ++g) S = add4(S, s_part[k & 1][g * n + (k >> 1)]);
        const size_t q = (size_t)(by * TH + p / PW) * a.W + bx * SP_TW + 2 * (p % PW) + (k & 1);
        spatial_finish(a, q, __ldg(&a.crt[q]), f3(S.x, S.y, S.z), S.w);
    }
}

constexpr int SP_TILE = 8;  // tile height
// 1280 resident threads (48 registers): 1080p alone 186 to 177 us against 1024, 1536 takes 180; in whole
// frames 4K gains 0.4%, and 128x128, one wave of blocks either way, pays 1.4 us
__global__ void __launch_bounds__(sp_threads<SP_TILE>(), 1280 / sp_threads<SP_TILE>()) k_spatial(SpatialArgs a) {
    spatial_body<SP_TILE>(a, blockIdx.x, blockIdx.y);
}
template <int TH>
__global__ void __launch_bounds__(sp_threads<TH>(), 1024 / sp_threads<TH>()) k_spatial_batch(const SpatialArgs* __restrict__ a, BatchGrid g) {
    int v, bx, by;
    g.locate(blockIdx.x, v, bx, by);
    spatial_body<TH>(batch_record(a, v), bx, by);
}

TemporalArgs temporal_args(const float* rt, const hdof_gbuf* in, const uint8_t* spp, const hdof_camera* cam,
                           const hdof_camera* prev, const hdof_params* p, const hdof_history* hist_in,
                           const hdof_history* hist_out, float* crt, float* hacc) {
    TemporalArgs a;
    a.cam = make_cam(*cam);
    a.prev = make_cam(*prev);
    a.W = cam->width;
    a.H = cam->height;
    a.alpha = p->ema_alpha;
    a.alpha_k = p->alpha_k;
    a.moved = p->camera_moved;
    a.rt = reinterpret_cast<const float4*>(rt);
    a.spp = spp;
    a.mv = reinterpret_cast<const float2*>(in->mv);
    a.hn = reinterpret_cast<const float4*>(hist_in->near_acc);
    a.hf = reinterpret_cast<const float4*>(hist_in->far_acc);
    a.hm = reinterpret_cast<const float2*>(hist_in->mom);
    a.hl = hist_in->hlen;
    a.on = reinterpret_cast<float4*>(hist_out->near_acc);
    a.of = reinterpret_cast<float4*>(hist_out->far_acc);
    a.om = reinterpret_cast<float2*>(hist_out->mom);
    a.ol = hist_out->hlen;
    a.crt = reinterpret_cast<float4*>(crt);
    a.hacc = hacc;
    return a;
}

}  // namespace

int launch_spatial(const float4* crt, const float2* mom, const uint8_t* hlen, int W, int H, float r_s, float var_ref,
                   float4* crec, float4* aux, cudaStream_t s) {
    dim3 g2((W + SP_TW - 1) / SP_TW, (H + SP_TILE - 1) / SP_TILE);
    ProfScope ps_("spatial", s);
    k_spatial<<<g2, sp_threads<SP_TILE>(), 0, s>>>(SpatialArgs{crt, mom, hlen, W, H, r_s, var_ref, crec, aux});
    HDOF_LAUNCHED("spatial reconstruction");
    return HDOF_OK;
}

}  // namespace hdof

using namespace hdof;

static bool hist_ok(const hdof_history* h) { return h && h->near_acc && h->far_acc && h->mom && h->hlen; }

extern "C" int hdof_reconstruct(const float* rt, const hdof_gbuf* in, const uint8_t* spp, const hdof_camera* cam,
                                const hdof_camera* prev, const hdof_lens* lens, const hdof_params* p,
                                const hdof_history* hist_in, const hdof_history* hist_out, float* crt, float* hacc,
                                float* crec, void* stream) {
    clear_error();
    int rc;
    if ((rc = check_camera(cam, "hdof_reconstruct")) || (rc = check_camera(prev, "hdof_reconstruct: prev")) ||
        (rc = check_lens(lens, "hdof_reconstruct")) || (rc = check_params(p, "hdof_reconstruct")) ||
        (rc = check_gbuf(in, "hdof_reconstruct", true)))
        return rc;
    HDOF_CHECK_ARG(rt && spp && crt && hacc && crec, "hdof_reconstruct: NULL buffer");
    HDOF_CHECK_ARG(hist_ok(hist_in) && hist_ok(hist_out), "hdof_reconstruct: history planes are required");
    HDOF_CHECK_ARG(hist_in->near_acc != hist_out->near_acc && hist_in->far_acc != hist_out->far_acc &&
                       hist_in->mom != hist_out->mom && hist_in->hlen != hist_out->hlen,
                   "hdof_reconstruct: hist_in and hist_out must be distinct buffers");
    HDOF_CHECK_ARG(in->width == cam->width && in->height == cam->height && prev->width == cam->width &&
                       prev->height == cam->height,
                   "hdof_reconstruct: size mismatch");
    cudaStream_t s = as_stream(stream);
    const int W = cam->width, H = cam->height;
    TemporalArgs a = temporal_args(rt, in, spp, cam, prev, p, hist_in, hist_out, crt, hacc);
    dim3 g1((W + 31) / 32, (H + 7) / 8);
    {
        ProfScope ps_("temporal", s);
        if (in->dtype_nd == HDOF_F32)
            k_temporal<float4><<<g1, 256, 0, s>>>(a, static_cast<const float4*>(in->nd));
        else
            k_temporal<half4s><<<g1, 256, 0, s>>>(a, static_cast<const half4s*>(in->nd));
        HDOF_LAUNCHED("hdof_reconstruct: temporal");
    }
    return launch_spatial(reinterpret_cast<const float4*>(crt), reinterpret_cast<const float2*>(hist_out->mom),
                          hist_out->hlen, W, H, p->r_s, p->var_ref, reinterpret_cast<float4*>(crec), nullptr, s);
}

namespace hdof {

size_t temporal_args_size() { return sizeof(TemporalBatch); }
void temporal_fill(const hdof_view& v, const ViewWs&, unsigned*, void* dst, int* gx, int* gy) {
    TemporalBatch* b = reinterpret_cast<TemporalBatch*>(dst);
    b->t = temporal_args(v.rt, &v.g, v.spp, &v.cam, &v.prev, &v.params, &v.hist_in, &v.hist_out, v.crt, v.hacc);
    b->nd = static_cast<const float4*>(v.g.nd);
    *gx = (v.cam.width + 31) / 32;
    *gy = (v.cam.height + 7) / 8;
}
void temporal_launch_batch(const void* args, BatchGrid g, int blocks, cudaStream_t s) {
    ProfScope ps_("batch_temporal", s);
    k_temporal_batch<<<blocks, 256, 0, s>>>(static_cast<const TemporalBatch*>(args), g);
}

size_t spatial_args_size() { return sizeof(SpatialArgs); }
void spatial_fill(const hdof_view& v, const ViewWs& w, unsigned*, void* dst, int* gx, int* gy) {
    *reinterpret_cast<SpatialArgs*>(dst) =
        SpatialArgs{reinterpret_cast<const float4*>(v.crt), reinterpret_cast<const float2*>(v.hist_out.mom),
                    v.hist_out.hlen, v.cam.width, v.cam.height, v.params.r_s, v.params.var_ref,
                    reinterpret_cast<float4*>(v.crec), nullptr};
    const int T = w.spatial_tile == 16 ? 16 : SP_TILE;
    *gx = (v.cam.width + SP_TW - 1) / SP_TW;
    *gy = (v.cam.height + T - 1) / T;
}
void spatial_launch_batch(const void* args, BatchGrid g, int blocks, cudaStream_t s) {
    spatial_launch_batch_tile(args, g, blocks, SP_TILE, s);
}
void spatial_launch_batch_tile(const void* args, BatchGrid g, int blocks, int tile, cudaStream_t s) {
    ProfScope ps_("batch_spatial", s);
    if (tile == 16) k_spatial_batch<16><<<blocks, sp_threads<16>(), 0, s>>>(static_cast<const SpatialArgs*>(args), g);
    else k_spatial_batch<SP_TILE><<<blocks, sp_threads<SP_TILE>(), 0, s>>>(static_cast<const SpatialArgs*>(args), g);
}

}  // namespace hdof
