// Differentiable post-path: the frame's reconstruction, post-filter and
// composite as a function of the sharp colour image and of the lens (focus
// distance, aperture), with the ray-traced visibility held fixed, and its
// hand-written adjoint.  The paper has no gradient; this makes the method's
// post-path usable inside an optimisation loop (e.g. fitting the lens to a
// reference image).
//
// Frozen inputs: per-ray hit records (radiance, view depth) from hdof_trace,
// the mask (spp), the depth plane, and the history already sampled at its
// reprojected positions.  Forward: replay of the trace accumulation at the
// new lens (each hit's CoC, split weight and CoC magnitude change, the hits
// do not) -> temporal EMA over the frozen history samples -> spatial gather
// -> post-filter -> composite; the same kernels as the frame path where the
// definitions coincide.  Backward: composite -> spatial (transposed gather)
// -> temporal and replay (per pixel, recomputed) -> post-filter (transposed
// gather over each source pixel's own disk, gather weights recomputed, not
// stored).  The lens gradient is summed in three floats within a warp and in
// double precision beyond, in a fixed order: the result is deterministic.
#include <cmath>

#include "internal.h"
#include "sum3.cuh"

namespace hdof {
namespace {

constexpr float RS2 = 0.35355339059327373f;  // 1 / (2 sqrt2): slope of w_near inside the focus zone

struct LensD {
    float K;           // A H / t
    float izf;         // 1 / zf
    float Ht;          // H / t
    float t;           // tan(fovy / 2)
    const float* dev;  // optional (zf, A) on the device: K and izf are read from it when a kernel starts
};

// K and izf of a lens on the device, by make_lensd's arithmetic
__device__ __forceinline__ LensD lens_at(LensD L, int H) {
    if (L.dev) {
        L.K = __ldg(&L.dev[1]) * (float)H / L.t;
        L.izf = 1.f / __ldg(&L.dev[0]);
    }
    return L;
}

__device__ __forceinline__ float coc_z(float z, const LensD& L) {
    return isinf(z) ? -L.K * L.izf : L.K * (1.f / z - L.izf);
}
// (dc/dzf, dc/dA) of the CoC of a point at depth z (z = inf: the miss CoC)
__device__ __forceinline__ float2 dcoc(float z, const LensD& L) {
    float u = isinf(z) ? -L.izf : 1.f / z - L.izf;
    return make_float2(L.K * L.izf * L.izf, L.Ht * u);
}
__device__ __forceinline__ float wn_slope(float c) { return (c > -HDOF_SQRT2 && c < HDOF_SQRT2) ? RS2 : 0.f; }
__device__ __forceinline__ float dot3f(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ float3 ldf3(const float4& v) { return f3(v.x, v.y, v.z); }

// block sum of a per-thread (float, float), fixed order: in three floats
// (Sum3: the terms cancel, and its bits are more than a double's) within a
// warp, in doubles in a warp with a value that is not finite or that could
// overflow them, and in double across the warps; thread 0 writes the block's
// partial.  Ten shuffle steps of doubles per thread held up the composite
// adjoint (37 us at 1024x1024, 28 so) and the replay's (32 and 25).
__device__ __forceinline__ void block_partial(float2 v, double2* partial) {
    __shared__ double red[2][32];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
    double da = v.x, db = v.y;
    if (__any_sync(0xffffffffu, !(fabsf(v.x) < 1e36f) || !(fabsf(v.y) < 1e36f))) {
        for (int o = 16; o; o >>= 1) {
            da += __shfl_xor_sync(0xffffffffu, da, o);
            db += __shfl_xor_sync(0xffffffffu, db, o);
        }
    } else {
        // the lower half of the warp sums x, the upper half y
        const bool up = l & 16;
        Sum3 s{up ? v.y : v.x, 0.f, 0.f};
        s.add(__shfl_xor_sync(0xffffffffu, up ? v.x : v.y, 16));
        for (int o = 8; o; o >>= 1) s.add(shfl_xor(s, o));
        da = db = s.value();
    }
    if (l == 0) red[0][w] = da;
    if (l == 16) red[1][w] = db;
    __syncthreads();
    if (threadIdx.x == 0) {
        double sa = 0.0, sb = 0.0;
        for (int k = 0; k < nw; ++k) {
            sa += red[0][k];
            sb += red[1][k];
        }
        partial[blockIdx.y * gridDim.x + blockIdx.x] = make_double2(sa, sb);
    }
}

// ------------------------------------------------------------ forward ----

struct ReplaySums {
    float3 SwL, SfL;
    float Sw, Sf, Swc, Sfc;
};

__device__ __forceinline__ ReplaySums replay_sums(const float4* rec, unsigned first, int n, const LensD& L) {
    ReplaySums s;
    s.SwL = s.SfL = f3(0.f, 0.f, 0.f);
    s.Sw = s.Sf = s.Swc = s.Sfc = 0.f;
    for (int k = 0; k < n; ++k) {
        float4 r = __ldg(&rec[first + k]);
        float c = coc_z(r.w, L);
        float w = w_near(c), wf = 1.f - w, ac = fabsf(c);
        s.SwL = s.SwL + w * ldf3(r);
        s.SfL = s.SfL + wf * ldf3(r);
        s.Sw += w;
        s.Sf += wf;
        s.Swc += w * ac;
        s.Sfc += wf * ac;
    }
    return s;
}

__global__ void __launch_bounds__(256) k_replay(const float4* __restrict__ rec, const unsigned* __restrict__ ray_off,
                                                const uint8_t* __restrict__ spp, int W, int H, LensD L,
                                                float4* __restrict__ rt) {
    L = lens_at(L, H);
    int i = blockIdx.x * 32 + (threadIdx.x & 31), j = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (i >= W || j >= H) return;
    size_t q = (size_t)j * W + i;
    int n = spp[q];
    if (!n) return;
    ReplaySums s = replay_sums(rec, ray_off[q], n, L);
    bool nok = s.Sw >= HDOF_EMPTY_W, fok = s.Sf >= HDOF_EMPTY_W;
    float in = nok ? 1.f / s.Sw : 0.f, inf_ = fok ? 1.f / s.Sf : 0.f;
    rt[3 * q] = make_float4(s.SwL.x * in, s.SwL.y * in, s.SwL.z * in, s.Sw / (float)n);
    rt[3 * q + 1] = make_float4(s.SfL.x * inf_, s.SfL.y * inf_, s.SfL.z * inf_, nok ? s.Swc * in : -1.f);
    rt[3 * q + 2] = make_float4(0.f, 0.f, 0.f, fok ? s.Sfc * inf_ : -1.f);
}

// history sampled at the reprojected positions: (near rgb, B) (far rgb, B) (mu1, mu2, flags, hlen)
struct HistS {
    float4 hn, hf;
    float m1, m2;
    bool vn, vf;
    int hl;
};
__device__ __forceinline__ HistS load_hs(const float4* hs, size_t q) {
    HistS h;
    if (!hs) {
        h.hn = h.hf = make_float4(0.f, 0.f, 0.f, 0.f);
        h.m1 = h.m2 = 0.f;
        h.vn = h.vf = false;
        h.hl = 0;
        return h;
    }
    h.hn = __ldg(&hs[3 * q]);
    h.hf = __ldg(&hs[3 * q + 1]);
    float4 t = __ldg(&hs[3 * q + 2]);
    h.m1 = t.x;
    h.m2 = t.y;
    int fl = (int)t.z;
    h.vn = fl & 1;
    h.vf = (fl >> 1) & 1;
    h.hl = (int)t.w;
    return h;
}

// the temporal step with frozen history samples (forward values used by the adjoint)
struct TempF {
    float h, cn, cf;
    bool nok, fok;
    float3 Cn, Cf, Ccur;
    float Y;
    float4 on, of;
    float2 om;
    float Bn, Bf, Hacc, hw;
    bool an, af, hsum;
    float3 CnA, CfA, C;
    float crt_c;
};

__device__ __forceinline__ TempF temporal_fwd(float4 r0, float4 r1, float4 r2, const HistS& hs, float al, int moved) {
    TempF t;
    t.h = r0.w;
    t.cn = r1.w;
    t.cf = r2.w;
    t.nok = t.cn >= 0.f;
    t.fok = t.cf >= 0.f;
    t.Cn = ldf3(r0);
    t.Cf = ldf3(r1);
    t.Ccur = t.nok ? (t.fok ? t.h * t.Cn + (1.f - t.h) * t.Cf : t.Cn) : t.Cf;
    t.Y = luminance(t.Ccur);
    float4 cur_n = make_float4(t.h * t.Cn.x, t.h * t.Cn.y, t.h * t.Cn.z, t.h);
    float4 cur_f = make_float4((1.f - t.h) * t.Cf.x, (1.f - t.h) * t.Cf.y, (1.f - t.h) * t.Cf.z, 1.f - t.h);
    const float4 hn = hs.hn, hf = hs.hf;
    t.on = hs.vn ? make_float4(fmaf(al, cur_n.x - hn.x, hn.x), fmaf(al, cur_n.y - hn.y, hn.y),
                               fmaf(al, cur_n.z - hn.z, hn.z), fmaf(al, cur_n.w - hn.w, hn.w))
                 : cur_n;
    t.of = hs.vf ? make_float4(fmaf(al, cur_f.x - hf.x, hf.x), fmaf(al, cur_f.y - hf.y, hf.y),
                               fmaf(al, cur_f.z - hf.z, hf.z), fmaf(al, cur_f.w - hf.w, hf.w))
                 : cur_f;
    t.om = hs.vn ? make_float2(fmaf(al, t.Y - hs.m1, hs.m1), fmaf(al, t.Y * t.Y - hs.m2, hs.m2))
                 : make_float2(t.Y, t.Y * t.Y);
    t.Bn = t.on.w;
    t.Bf = t.of.w;
    t.hsum = t.Bn + t.Bf >= HDOF_EMPTY_W;
    t.Hacc = t.hsum ? t.Bn / (t.Bn + t.Bf) : t.h;
    t.an = t.Bn >= HDOF_EMPTY_W;
    t.af = t.Bf >= HDOF_EMPTY_W;
    t.hw = moved ? t.h : t.Hacc;
    t.CnA = t.an ? (1.f / t.Bn) * ldf3(t.on) : f3(0, 0, 0);
    t.CfA = t.af ? (1.f / t.Bf) * ldf3(t.of) : f3(0, 0, 0);
    t.C = !t.an ? t.CfA : (!t.af ? t.CnA : t.hw * t.CnA + (1.f - t.hw) * t.CfA);
    t.crt_c = !t.nok ? t.cf : (!t.fok ? t.cn : t.Hacc * t.cn + (1.f - t.Hacc) * t.cf);
    return t;
}

__global__ void __launch_bounds__(256) k_temporal_frozen(const float4* __restrict__ rt, const uint8_t* __restrict__ spp,
                                                         const float4* __restrict__ hs, int W, int H, float al,
                                                         int moved, float4* __restrict__ crt, float* __restrict__ hacc,
                                                         float2* __restrict__ mom, uint8_t* __restrict__ hlen) {
    int i = blockIdx.x * 32 + (threadIdx.x & 31), j = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (i >= W || j >= H) return;
    size_t q = (size_t)j * W + i;
    if (!spp[q]) {
        crt[q] = make_float4(0.f, 0.f, 0.f, -1.f);
        hlen[q] = 0;
        return;
    }
    HistS h = load_hs(hs, q);
    TempF t = temporal_fwd(rt[3 * q], rt[3 * q + 1], rt[3 * q + 2], h, al, moved);
    crt[q] = make_float4(t.C.x, t.C.y, t.C.z, t.crt_c);
    hacc[q] = t.Hacc;
    mom[q] = t.om;
    int nh = h.vn ? h.hl + 1 : 1;
    hlen[q] = (uint8_t)(nh > 255 ? 255 : nh);
}

// ----------------------------------------------------------- backward ----

// composite adjoint: per pixel; grad_col <- f g (the sharp term), gradients of
// pp, crec, crt.w, hacc, and this pixel's share of the lens gradient
__global__ void __launch_bounds__(256) k_composite_bwd(const float4* __restrict__ nd, const float4* __restrict__ col,
                                                       const uint8_t* __restrict__ spp, const float4* __restrict__ pp,
                                                       const float4* __restrict__ crt, const float4* __restrict__ crec,
                                                       const float* __restrict__ hacc, const float4* __restrict__ gout,
                                                       int W, int H, LensD L, float h_tau, float4* __restrict__ gcol,
                                                       float4* __restrict__ gpp, float4* __restrict__ gcrec,
                                                       float4* __restrict__ gcrt, float* __restrict__ ghacc,
                                                       double2* partial) {
    L = lens_at(L, H);
    int i = blockIdx.x * 32 + (threadIdx.x & 31), j = blockIdx.y * 8 + (threadIdx.x >> 5);
    float2 dth = make_float2(0.f, 0.f);
    if (i < W && j < H) {
        size_t q = (size_t)j * W + i;
        float z = __ldg(&nd[q].w);
        float c = coc_z(z, L);
        bool traced = spp[q] > 0;
        float3 C = ldf3(__ldg(&col[q])), P = ldf3(__ldg(&pp[q])), g = ldf3(__ldg(&gout[q]));
        float ce = traced ? __ldg(&crt[q].w) : fabsf(c);
        float fu = HDOF_SQRT2 + 0.5f - ce, f = clamp01(fu);
        float wn = w_near(c);
        float3 nearc = P, farc = P, R = f3(0, 0, 0);
        float b = 0.f, bu = 0.f;
        if (traced) {
            R = ldf3(__ldg(&crec[q]));
            bu = __ldg(&hacc[q]) / h_tau;
            b = clamp01(bu);
            nearc = R;
            farc = R + b * (P - R);
        }
        float3 blur = wn * nearc + (1.f - wn) * farc;
        float3 gb = (1.f - f) * g;
        float gf = dot3f(g, C - blur);
        float gwn = dot3f(gb, nearc - farc);
        float3 gnear = wn * gb, gfar = (1.f - wn) * gb;
        float gc = wn_slope(c) * gwn;
        float gfu = (fu > 0.f && fu < 1.f) ? gf : 0.f;
        gcol[q] = make_float4(f * g.x, f * g.y, f * g.z, 0.f);
        if (traced) {
            float3 gr = gnear + (1.f - b) * gfar;
            float3 gp = b * gfar;
            float gbb = dot3f(gfar, P - R);
            gpp[q] = make_float4(gp.x, gp.y, gp.z, 0.f);
            gcrec[q] = make_float4(gr.x, gr.y, gr.z, 0.f);
            gcrt[q] = make_float4(0.f, 0.f, 0.f, -gfu);
            ghacc[q] = (bu > 0.f && bu < 1.f) ? gbb / h_tau : 0.f;
        } else {
            float3 gp = gnear + gfar;
            gpp[q] = make_float4(gp.x, gp.y, gp.z, 0.f);
            gc += -gfu * (c > 0.f ? 1.f : (c < 0.f ? -1.f : 0.f));
        }
        float2 dc = dcoc(z, L);
        dth = make_float2(gc * dc.x, gc * dc.y);
    }
    block_partial(dth, partial);
}

// spatial adjoint, part 1 (per traced pixel): direct term, the variance blend,
// and the per-gatherer factors a = beta g / W, b = a . C_sp of the gather
__global__ void __launch_bounds__(256) k_spatial_bwd_prep(const float4* __restrict__ crt, const float2* __restrict__ mom,
                                                          const uint8_t* __restrict__ hlen, const float4* __restrict__ aux,
                                                          const float4* __restrict__ gcrec, int W, int H, float var_ref,
                                                          float4* __restrict__ spb, float4* __restrict__ gcrt,
                                                          float2* __restrict__ gmom) {
    int i = blockIdx.x * 32 + (threadIdx.x & 31), j = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (i >= W || j >= H) return;
    size_t q = (size_t)j * W + i;
    float4 cp = crt[q];
    if (cp.w < 0.f) return;
    float2 m = mom[q];
    float v = m.y - m.x * m.x;
    float sig = sqrtf(fmaxf(0.f, v));
    bool young = hlen[q] < 2;
    float bu = sig / var_ref;
    float beta = young ? 1.f : clamp01(bu);
    float4 ax = aux[q];
    float3 Csp = ldf3(ax), Crt = ldf3(cp), g = ldf3(gcrec[q]);
    float gbeta = dot3f(g, Csp - Crt);
    float2 gm = make_float2(0.f, 0.f);
    if (!young && bu > 0.f && bu < 1.f && v > 0.f) {
        float gs = gbeta / var_ref;
        gm = make_float2(gs * (-m.x / sig), gs * (0.5f / sig));
    }
    gmom[q] = gm;
    float3 a = (beta / ax.w) * g;
    spb[q] = make_float4(a.x, a.y, a.z, dot3f(a, Csp));
    float4 gc = gcrt[q];
    float3 gd = (1.f - beta) * g;
    gcrt[q] = make_float4(gc.x + gd.x, gc.y + gd.y, gc.z + gd.z, gc.w);
}

// spatial adjoint, part 2 (per traced pixel x over its own window): x as a
// gathered sample of its neighbours and x as a gatherer.  Block = one 16x8
// tile as pixel pairs; its pairs holding a traced pixel are compacted and
// SBG threads share a pair's rows (y mod SBG), as in the forward gather: one
// thread per pixel took 131 us at 1024x1024 with 20% of the warps active,
// this 60 us (few tiles are traced there: the longest still set the time).
constexpr int SB_TW = 16, SB_TH = 8, SB_NP = SB_TW * SB_TH / 2, SBG = 4, SB_THREADS = SB_NP * SBG;

// one pixel x's share of a tap: gC += sy sx a_y, gcx += sy s'x (x gathered by y + x gathering y)
__device__ __forceinline__ void spatial_bwd_tap(float4& acc, float R, float d, float rq, const float3& Cx,
                                                const float4& bx, const float4& cy, const float4& by) {
    const float ux = R - d, sx = __saturatef(ux), sy = __saturatef(rq - d);
    const float spx = (ux > 0.f && ux < 1.f) ? sy : 0.f, w = sy * sx;
    acc.x = fmaf(w, by.x, acc.x);
    acc.y = fmaf(w, by.y, acc.y);
    acc.z = fmaf(w, by.z, acc.z);
    const float v = (dot3f(ldf3(by), Cx) - by.w) + (dot3f(ldf3(bx), ldf3(cy)) - bx.w);
    acc.w = fmaf(spx, v, acc.w);
}

__global__ void __launch_bounds__(SB_THREADS, 3) k_spatial_bwd(const float4* __restrict__ crt,
                                                               const float4* __restrict__ spb, int W, int H, float r_s,
                                                               float4* __restrict__ gcrt) {
    constexpr int PW = SB_TW / 2;
    __shared__ unsigned short s_list[SB_NP];
    __shared__ int s_cnt[SB_NP / 32];
    __shared__ float4 s_part[2][SB_THREADS];
    const int t = threadIdx.x, lane = t & 31, wi = t >> 5, bx0 = blockIdx.x * SB_TW, by0 = blockIdx.y * SB_TH;
    bool tl = false, tr = false;
    unsigned tm = 0;
    if (t < SB_NP) {  // whole warps
        const int i0 = bx0 + 2 * (t % PW), j0 = by0 + t / PW;
        tl = j0 < H && i0 < W && __ldg(&crt[(size_t)j0 * W + i0].w) >= 0.f;
        tr = j0 < H && i0 + 1 < W && __ldg(&crt[(size_t)j0 * W + i0 + 1].w) >= 0.f;
        tm = __ballot_sync(0xffffffffu, tl || tr);
        if (lane == 0) s_cnt[wi] = __popc(tm);
    }
    __syncthreads();
    int off = 0, n = 0;
#pragma unroll
    for (int k = 0; k < SB_NP / 32; ++k) {
        off += k < wi ? s_cnt[k] : 0;
        n += s_cnt[k];
    }
    if (n == 0) return;  // the whole block
    if (tl || tr)
        s_list[off + __popc(tm & ((1u << lane) - 1u))] = (unsigned short)(t | (tl ? 0x8000 : 0) | (tr ? 0x4000 : 0));
    __syncthreads();
    if (t < SBG * n) {
        const int g = t / n, e = s_list[t - g * n], p = e & 0x3fff;
        const int i = bx0 + 2 * (p % PW), j = by0 + p / PW;
        const size_t q = (size_t)j * W + i;
        const bool hl = e & 0x8000, hr = e & 0x4000;
        const float4 none = make_float4(0.f, 0.f, 0.f, -1.f), zero = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 cl = hl ? __ldg(&crt[q]) : none, cr = hr ? __ldg(&crt[q + 1]) : none;
        const float4 bl = hl ? __ldg(&spb[q]) : zero, br = hr ? __ldg(&spb[q + 1]) : zero;
        // a neighbour takes part only if d < R = min(c/2, r_s) + 1/2 (0 for an
        // untraced pixel of the pair): per row, the columns of that disk
        // (bounds lean outwards by 1e-3 pixel; taps they add weigh 0)
        const float Rl = hl ? fminf(cl.w * 0.5f, r_s) + 0.5f : 0.f, Rr = hr ? fminf(cr.w * 0.5f, r_s) + 0.5f : 0.f;
        const float Rl2 = Rl * Rl, Rr2 = Rr * Rr, Rq = r_s + 0.5f;
        const float3 Cl = ldf3(cl), Cr = ldf3(cr);
        const int K = (int)floorf(fmaxf(Rl, Rr) + 1e-3f);
        float4 al = zero, ar = zero;  // (gC, gcx)
        const int y0 = max(j - K, 0), y1 = min(j + K, H - 1);
        for (int y = y0 + ((g - y0) & (SBG - 1)); y <= y1; y += SBG) {
            const float dy = (float)(y - j), dy2 = dy * dy;
            const int wl = (int)floorf(sqrtf(fmaxf(Rl2 - dy2, 0.f)) + 1e-3f);
            const int wr = (int)floorf(sqrtf(fmaxf(Rr2 - dy2, 0.f)) + 1e-3f);
            const int x0 = max(min(i - wl, i + 1 - wr), 0), x1 = min(max(i + wl, i + 1 + wr), W - 1);
            float dx = (float)(x0 - i);
            float dprev = sqrt_approx(fmaf(dx - 1.f, dx - 1.f, dy2));
            for (int x = x0; x <= x1; ++x, dx += 1.f) {
                const size_t qq = (size_t)y * W + x;
                // branch-free: untraced neighbours (and their unwritten spb)
                // are selected away, out-of-disk pairs weigh exactly zero
                const float4 cy = __ldg(&crt[qq]);
                float4 by = __ldg(&spb[qq]);
                const bool ty = cy.w >= 0.f;
                by = make_float4(ty ? by.x : 0.f, ty ? by.y : 0.f, ty ? by.z : 0.f, ty ? by.w : 0.f);
                const float rq = ty ? fminf(fmaf(cy.w, 0.5f, 0.5f), Rq) : -1.f;
                const float d = sqrt_approx(fmaf(dx, dx, dy2));
                spatial_bwd_tap(al, Rl, d, rq, Cl, bl, cy, by);
                spatial_bwd_tap(ar, Rr, dprev, rq, Cr, br, cy, by);
                dprev = d;
            }
        }
        s_part[0][t] = al;
        s_part[1][t] = ar;
    }
    __syncthreads();
    for (int k = t; k < 2 * n; k += SB_THREADS) {  // pixel k & 1 of pair k / 2
        const int e = s_list[k >> 1], p = e & 0x3fff;
        if (!(e & ((k & 1) ? 0x4000 : 0x8000))) continue;
        float4 S = s_part[k & 1][k >> 1];
#pragma unroll
        for (int g = 1; g < SBG; ++g) S = add4(S, s_part[k & 1][g * n + (k >> 1)]);
        const size_t q = (size_t)(by0 + p / PW) * W + bx0 + 2 * (p % PW) + (k & 1);
        const float rpx = __ldg(&crt[q].w) * 0.5f < r_s ? 0.5f : 0.f;
        const float4 g0 = gcrt[q];
        gcrt[q] = make_float4(g0.x + S.x, g0.y + S.y, g0.z + S.z, g0.w + S.w * rpx);
    }
}

// temporal + replay adjoint (per traced pixel, forward recomputed): the
// gradient of crt, hacc and the moments back to each hit's CoC
__global__ void __launch_bounds__(256) k_temporal_replay_bwd(const float4* __restrict__ rec,
                                                             const unsigned* __restrict__ ray_off,
                                                             const uint8_t* __restrict__ spp,
                                                             const float4* __restrict__ hs, const float4* __restrict__ gcrt,
                                                             const float* __restrict__ ghacc,
                                                             const float2* __restrict__ gmom, int W, int H, LensD L,
                                                             float al, int moved, double2* partial) {
    L = lens_at(L, H);
    int i = blockIdx.x * 32 + (threadIdx.x & 31), j = blockIdx.y * 8 + (threadIdx.x >> 5);
    float2 dth = make_float2(0.f, 0.f);
    size_t q = (size_t)j * W + i;
    int n = (i < W && j < H) ? spp[q] : 0;
    if (n) {
        const unsigned first = ray_off[q];
        ReplaySums s = replay_sums(rec, first, n, L);
        bool nok = s.Sw >= HDOF_EMPTY_W, fok = s.Sf >= HDOF_EMPTY_W;
        float in = nok ? 1.f / s.Sw : 0.f, inf_ = fok ? 1.f / s.Sf : 0.f;
        float4 r0 = make_float4(s.SwL.x * in, s.SwL.y * in, s.SwL.z * in, s.Sw / (float)n);
        float4 r1 = make_float4(s.SfL.x * inf_, s.SfL.y * inf_, s.SfL.z * inf_, nok ? s.Swc * in : -1.f);
        float4 r2 = make_float4(0.f, 0.f, 0.f, fok ? s.Sfc * inf_ : -1.f);
        HistS hsv = load_hs(hs, q);
        TempF t = temporal_fwd(r0, r1, r2, hsv, al, moved);
        // ---- temporal adjoint ----
        float4 g4 = gcrt[q];
        float3 gC = ldf3(g4);
        float gcc = g4.w, gH = ghacc[q];
        float2 gom = gmom[q];
        float3 gCnA = f3(0, 0, 0), gCfA = f3(0, 0, 0);
        float gh = 0.f, ghw = 0.f, gcn = 0.f, gcf = 0.f;
        if (!t.an) gCfA = gC;
        else if (!t.af) gCnA = gC;
        else {
            gCnA = t.hw * gC;
            gCfA = (1.f - t.hw) * gC;
            ghw = dot3f(gC, t.CnA - t.CfA);
        }
        if (moved) gh += ghw;
        else gH += ghw;
        if (!t.nok) gcf += gcc;
        else if (!t.fok) gcn += gcc;
        else {
            gH += gcc * (t.cn - t.cf);
            gcn += t.Hacc * gcc;
            gcf += (1.f - t.Hacc) * gcc;
        }
        float gBn = 0.f, gBf = 0.f;
        if (t.hsum) {
            float S = t.Bn + t.Bf, iS2 = 1.f / (S * S);
            gBn += gH * t.Bf * iS2;
            gBf -= gH * t.Bn * iS2;
        } else {
            gh += gH;
        }
        float3 gon = f3(0, 0, 0), gof = f3(0, 0, 0);
        if (t.an) {
            gon = (1.f / t.Bn) * gCnA;
            gBn -= dot3f(gCnA, ldf3(t.on)) / (t.Bn * t.Bn);
        }
        if (t.af) {
            gof = (1.f / t.Bf) * gCfA;
            gBf -= dot3f(gCfA, ldf3(t.of)) / (t.Bf * t.Bf);
        }
        const float kn = hsv.vn ? al : 1.f, kf = hsv.vf ? al : 1.f;
        float3 gcurn = kn * gon, gcurf = kf * gof;
        float gcurnw = kn * gBn, gcurfw = kf * gBf;
        float gY = kn * (gom.x + 2.f * t.Y * gom.y);
        float3 gCn = t.h * gcurn, gCf = (1.f - t.h) * gcurf;
        gh += dot3f(gcurn, t.Cn) + gcurnw - dot3f(gcurf, t.Cf) - gcurfw;
        float3 gCcur = gY * f3(0.2126f, 0.7152f, 0.0722f);
        if (t.nok && t.fok) {
            gh += dot3f(gCcur, t.Cn - t.Cf);
            gCn = gCn + t.h * gCcur;
            gCf = gCf + (1.f - t.h) * gCcur;
        } else if (t.nok) {
            gCn = gCn + gCcur;
        } else {
            gCf = gCf + gCcur;
        }
        // ---- replay adjoint ----
        float gSw = gh / (float)n, gSf = 0.f, gSwc = 0.f, gSfc = 0.f;
        float3 gSwL = f3(0, 0, 0), gSfL = f3(0, 0, 0);
        if (nok) {
            gSwL = in * gCn;
            gSw -= dot3f(gCn, s.SwL) * in * in;
            gSwc = gcn * in;
            gSw -= gcn * s.Swc * in * in;
        }
        if (fok) {
            gSfL = inf_ * gCf;
            gSf -= dot3f(gCf, s.SfL) * inf_ * inf_;
            gSfc = gcf * inf_;
            gSf -= gcf * s.Sfc * inf_ * inf_;
        }
        for (int k = 0; k < n; ++k) {
            float4 r = __ldg(&rec[first + k]);
            float c = coc_z(r.w, L);
            float w = w_near(c), ac = fabsf(c);
            float gw = gSw - gSf + dot3f(gSwL - gSfL, ldf3(r)) + (gSwc - gSfc) * ac;
            float gac = gSwc * w + gSfc * (1.f - w);
            float gc = gw * wn_slope(c) + gac * (c > 0.f ? 1.f : (c < 0.f ? -1.f : 0.f));
            float2 dc = dcoc(r.w, L);
            dth.x += gc * dc.x;
            dth.y += gc * dc.y;
        }
    }
    block_partial(dth, partial);
}

__device__ __forceinline__ float2 area_and_slope(const float4* tab, int n, float r) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(&tab[mid].x) <= r) lo = mid;
        else hi = mid - 1;
    }
    float4 e = __ldg(&tab[lo]);
    return make_float2(fmaf(e.z, r - e.x, e.y), e.z);
}

// post-filter adjoint, part 1 (per pixel p): factors of dL/d(near weight) =
// A . C_q - E and dL/d(far weight) = Af . C_q - Ef, and the sharp-colour
// fallback of an empty far layer
// Written per pixel q, row-major: (A, E) and (Af, Ef) in two planes, and
// kb_q = 1 / (kz_rel z_q) of the forward's depth test.
__host__ __device__ inline size_t pfb_plane(int W, int H) {  // an even count: both planes' pairs are 32-byte aligned
    return ((size_t)W * H + 1) & ~size_t(1);
}
__global__ void __launch_bounds__(256) k_pf_bwd_prep(const float4* __restrict__ aux, const float4* __restrict__ gpp,
                                                     const float4* __restrict__ nd, float kz_rel, int W, int H,
                                                     float4* __restrict__ pfb, float* __restrict__ kbp,
                                                     float4* __restrict__ gcol) {
    int i = blockIdx.x * 32 + (threadIdx.x & 31), j = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (i >= W || j >= H) return;
    size_t q = (size_t)j * W + i;
    kbp[q] = 1.f / (kz_rel * __ldg(&nd[q].w));
    float4 an = aux[2 * q], af = aux[2 * q + 1];
    float3 g = ldf3(gpp[q]), N = ldf3(an), F = ldf3(af);
    float Wn = an.w, Wf = af.w;
    float alpha = clamp01(Wn);
    float adash = (Wn > 0.f && Wn < 1.f) ? 1.f : 0.f;
    float3 A = Wn > HDOF_PP_MIN_W ? (alpha / Wn) * g : f3(0, 0, 0);
    float E = dot3f(A, N) - adash * dot3f(g, N - F);
    float3 Af = f3(0, 0, 0);
    float Ef = 0.f;
    if (Wf > HDOF_PP_MIN_W) {
        Af = ((1.f - alpha) / Wf) * g;
        Ef = dot3f(Af, F);
    } else {
        float4 gc = gcol[q];  // F is this pixel's sharp colour
        gcol[q] = make_float4(gc.x + (1.f - alpha) * g.x, gc.y + (1.f - alpha) * g.y, gc.z + (1.f - alpha) * g.z, 0.f);
    }
    pfb[q] = make_float4(A.x, A.y, A.z, E);
    pfb[pfb_plane(W, H) + q] = make_float4(Af.x, Af.y, Af.z, Ef);
}

// per source pixel: the radius and the layer weights of the forward map and
// their slopes with respect to the source's CoC
struct PfSrc {
    float R, rp;         // r + 1/2; dr/dc (0 when clipped at r_max)
    float wnia, fia;     // w/a, (1-w)/a
    float dwnia, dfia;   // their derivatives with respect to c
};
__device__ __forceinline__ PfSrc pf_src(float zq, const LensD& L, float rmax, const float4* tab, int ntab) {
    PfSrc o;
    const float c = coc_z(zq, L);
    const bool clip = fabsf(c) * 0.5f >= rmax;
    const float r = clip ? rmax : fabsf(c) * 0.5f;
    o.R = r + 0.5f;
    o.rp = clip ? 0.f : (c > 0.f ? 0.5f : (c < 0.f ? -0.5f : 0.f));
    const float2 as = area_and_slope(tab, ntab, r);
    const float ia = 1.f / as.x, iap = -as.y * ia * ia * o.rp;
    const float wn = w_near(c), wnp = wn_slope(c);
    o.wnia = wn * ia;
    o.fia = (1.f - wn) * ia;
    o.dwnia = wnp * ia + wn * iap;
    o.dfia = -wnp * ia + (1.f - wn) * iap;
    return o;
}

// One layer's sums over the targets of the four sources of a thread, two
// sources (a row's left and right pixel) to a register pair so that one
// packed FMA serves both: per row k, sum s A (gx, gy, gz), sum t s and
// sum t s' with t = A . C_q - E (times the depth test in the far layer),
// s = clamp(R - d, 0, 1) and s' its slope.
struct PfBwdAcc {
    f32x2 gx[2], gy[2], gz[2], S1[2], S2[2];
};
struct PfBwdSrc {
    float R[4], zq[4];
    f32x2 Cx[2], Cy[2], Cz[2];
};

// the four sources of a thread against one target: row k's left source gets a
// fresh distance, its right source the previous target's (the same offsets,
// so the same floats), carried in c
template <bool FAR>
__device__ __forceinline__ void pf_bwd_tap(PfBwdAcc& acc, float (&c)[2], const PfBwdSrc& src, float dx, float dy0,
                                           float dy1, float ka, float kb, const float4& b) {
    const f32x2 Ax = pk2(b.x, b.x), Ay = pk2(b.y, b.y), Az = pk2(b.z, b.z), E = pk2(-b.w, -b.w);
    const float dx2 = dx * dx;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float d = sqrt_approx(dx2 + (k ? dy1 : dy0));
        const float ul = src.R[2 * k] - d, ur = src.R[2 * k + 1] - c[k];
        c[k] = d;
        const float sl = __saturatef(ul), sr = __saturatef(ur);
        float kl = 1.f, kr = 1.f;
        if (FAR) {
            kl = __saturatef(fmaf(-src.zq[2 * k], kb, ka));
            kr = __saturatef(fmaf(-src.zq[2 * k + 1], kb, ka));
        }
        // the clamp's slope: 1 where 0 < u < 1, that is u - u^2 > 0 (the fused
        // form's sign is exact; u of exactly 0 or 1 is met tens of times a frame)
        const f32x2 s = pk2(FAR ? sl * kl : sl, FAR ? sr * kr : sr);
        const f32x2 sp = pk2(fmaf(-ul, ul, ul) > 0.f ? kl : 0.f, fmaf(-ur, ur, ur) > 0.f ? kr : 0.f);
        const f32x2 t = ffma2(Az, src.Cz[k], ffma2(Ay, src.Cy[k], ffma2(Ax, src.Cx[k], E)));
        acc.gx[k] = ffma2(s, Ax, acc.gx[k]);
        acc.gy[k] = ffma2(s, Ay, acc.gy[k]);
        acc.gz[k] = ffma2(s, Az, acc.gz[k]);
        acc.S1[k] = ffma2(t, s, acc.S1[k]);
        acc.S2[k] = ffma2(t, sp, acc.S2[k]);
    }
}

constexpr int PBT = 16, PBG = 4;  // source tile edge, thread groups over the target rows

// One layer's sums of the 2x2 source block at (i, j) over the rows g, g + PBG,
// ... of its window: per target row, the columns closer than the layer's
// reach R to one of the four (bounds lean outwards by 1e-3 pixel; other
// pairs weigh zero, and so do their slopes)
template <bool FAR>
__device__ __forceinline__ void pf_bwd_layer(PfBwdAcc& acc, const PfBwdSrc& src, float R, int g, int i, int j, int W,
                                             int H, float ka, const float4* __restrict__ rec,
                                             const float* __restrict__ kbp) {
#pragma unroll
    for (int k = 0; k < 2; ++k) acc.gx[k] = acc.gy[k] = acc.gz[k] = acc.S1[k] = acc.S2[k] = 0ull;
    const float R2 = R * R;
    const int G = (int)floorf(R + 1e-3f);
    const float2* __restrict__ kb2 = reinterpret_cast<const float2*>(kbp);
    const int y0 = max(j - G, 0), y1 = min(j + 1 + G, H - 1);
    for (int y = y0 + g; y <= y1; y += PBG) {
        const float dy = (float)(y - j);
        const float dy0 = dy * dy, dy1 = (dy - 1.f) * (dy - 1.f);
        const float dmin = dy >= 0.f && dy <= 1.f ? 0.f : fminf(dy0, dy1);
        const int w = (int)(sqrt_approx(fmaxf(R2 - dmin, 0.f)) + 1e-3f);
        const int x0 = max(i - w, 0), x1 = min(i + 1 + w, W - 1);
        float dx = (float)(x0 - i);
        const float dm = (dx - 1.f) * (dx - 1.f);
        float c[2] = {sqrt_approx(dm + dy0), sqrt_approx(dm + dy1)};
        // targets in (even, odd) index pairs; a lone odd first and even last on their own
        unsigned q = (unsigned)y * W + x0;
        const unsigned qend = (unsigned)y * W + x1 + 1;
        if (q & 1) {
            pf_bwd_tap<FAR>(acc, c, src, dx, dy0, dy1, ka, FAR ? __ldg(&kbp[q]) : 0.f, __ldg(&rec[q]));
            ++q;
            dx += 1.f;
        }
        const unsigned mend = qend >> 1;
#pragma unroll 1
        for (unsigned m = q >> 1; m < mend; ++m, dx += 2.f) {
            const float2 kb = FAR ? __ldg(&kb2[m]) : make_float2(0.f, 0.f);
            float4 b0, b1;
            ld_rec_pair(rec + 2 * (size_t)m, b0, b1);
            pf_bwd_tap<FAR>(acc, c, src, dx, dy0, dy1, ka, kb.x, b0);
            pf_bwd_tap<FAR>(acc, c, src, dx + 1.f, dy0, dy1, ka, kb.y, b1);
        }
        if (qend & 1)
            pf_bwd_tap<FAR>(acc, c, src, dx, dy0, dy1, ka, FAR ? __ldg(&kbp[qend - 1]) : 0.f,
                            __ldg(&rec[qend - 1]));
    }
}

// post-filter adjoint, part 2: per source pixel q over the target pixels its
// soft disk reaches, the colour gradient and the gradient of q's CoC.  One
// block per 16x16 tile of sources, PBG groups of 64 threads; thread t of a
// group takes the 2x2 source block at (2 (t & 7), 2 (t >> 3)) over the
// group's target rows, so every target it loads serves four sources.  The
// near and the far layer run one after the other, each only where a source
// of the tile feeds it (a source outside the focus zone feeds one) and as far
// as the largest radius that does; the depth test is the forward's
// clamp(ka - z_q kb_p).  The layer weights w/a and (1-w)/a of a source are
// factored out of its sums.  Thread p finishes source p of the tile.  Bound
// by issue (about 11 instructions per source and target, 58% busy) and the
// latency of the target loads.  Both layers in one loop over every target
// with scalar FMAs took 383 us at 1024x1024 (radii to 10 px, all far); this
// 219 us.
#ifndef HDOF_PFB_MINB
#define HDOF_PFB_MINB 3  // resident blocks per SM the register budget targets (80 registers)
#endif
__global__ void __launch_bounds__(64 * PBG, HDOF_PFB_MINB) k_pf_bwd(const float4* __restrict__ nd, const float4* __restrict__ col,
                                               const float4* __restrict__ pfb, const float* __restrict__ kbp,
                                               const float4* __restrict__ tab, int ntab, int W, int H, LensD L,
                                               float rmax, float kz_rel, float4* __restrict__ gcol,
                                               double2* partial) {
    L = lens_at(L, H);
    __shared__ int s_win[2];                // bit patterns of the layers' reach, -1: not fed
    __shared__ float4 s_src[PBT * PBT];     // (C_q, R)
    __shared__ float s_z[PBT * PBT];
    __shared__ float s_part[PBG][5][PBT * PBT];  // one layer's (gx, gy, gz, S1, S2) per group
    const int p = threadIdx.x;
    if (p < 2) s_win[p] = -1;
    __syncthreads();
    const int pi = blockIdx.x * PBT + (p & 15), pj = blockIdx.y * PBT + (p >> 4);
    const bool ok = pi < W && pj < H;
    const size_t pq = (size_t)pj * W + pi;
    float z = 1.f;
    PfSrc sr{};
    {
        float4 cr = make_float4(0.f, 0.f, 0.f, 0.f);  // R = 0: an absent source weighs nothing
        if (ok) {
            z = __ldg(&nd[pq].w);
            sr = pf_src(z, L, rmax, tab, ntab);
            const float3 C = ldf3(__ldg(&col[pq]));
            cr = make_float4(C.x, C.y, C.z, sr.R);
            // positive floats order as their bits; NaN radii (a lens that is not finite) take the whole cap
            const int rb = __float_as_int(sr.R <= rmax + 0.5f ? sr.R : rmax + 0.5f);
            if (!(sr.wnia == 0.f && sr.dwnia == 0.f)) atomicMax(&s_win[0], rb);
            if (!(sr.fia == 0.f && sr.dfia == 0.f)) atomicMax(&s_win[1], rb);
        }
        s_src[p] = cr;
        s_z[p] = z;
    }
    __syncthreads();
    const int g = threadIdx.x >> 6, t = threadIdx.x & 63;
    const int li = 2 * (t & 7), lj = 2 * (t >> 3), i = blockIdx.x * PBT + li, j = blockIdx.y * PBT + lj;
    const float ka = 1.f + 1.f / kz_rel;
    PfBwdSrc src;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int e = (lj + k) * PBT + li;
        const float4 a = s_src[e], b = s_src[e + 1];
        src.R[2 * k] = a.w;
        src.R[2 * k + 1] = b.w;
        src.zq[2 * k] = s_z[e];
        src.zq[2 * k + 1] = s_z[e + 1];
        src.Cx[k] = pk2(a.x, b.x);
        src.Cy[k] = pk2(a.y, b.y);
        src.Cz[k] = pk2(a.z, b.z);
    }
    float3 gC = f3(0.f, 0.f, 0.f);
    float gc = 0.f;  // gradient of source p's CoC
#pragma unroll
    for (int layer = 0; layer < 2; ++layer) {
        const int rb = s_win[layer];
        if (rb < 0) continue;  // block-uniform
        if (i < W && j < H) {
            PfBwdAcc acc;
            const float reach = __int_as_float(rb);
            if (layer) pf_bwd_layer<true>(acc, src, reach, g, i, j, W, H, ka, pfb + pfb_plane(W, H), kbp);
            else pf_bwd_layer<false>(acc, src, reach, g, i, j, W, H, ka, pfb, kbp);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int e = (lj + k) * PBT + li;
                const float2 v[5] = {unpk2(acc.gx[k]), unpk2(acc.gy[k]), unpk2(acc.gz[k]), unpk2(acc.S1[k]),
                                     unpk2(acc.S2[k])};
#pragma unroll
                for (int m = 0; m < 5; ++m) *reinterpret_cast<float2*>(&s_part[g][m][e]) = v[m];
            }
        }
        __syncthreads();
        if (ok) {
            float v[5];
#pragma unroll
            for (int m = 0; m < 5; ++m) {
                v[m] = s_part[0][m][p];
#pragma unroll
                for (int b = 1; b < PBG; ++b) v[m] += s_part[b][m][p];
            }
            const float wa = layer ? sr.fia : sr.wnia, da = layer ? sr.dfia : sr.dwnia;
            gC = gC + wa * f3(v[0], v[1], v[2]);
            gc += v[3] * da + v[4] * wa * sr.rp;
        }
        __syncthreads();
    }
    float2 dth = make_float2(0.f, 0.f);
    if (ok) {
        const float4 g0 = gcol[pq];
        gcol[pq] = make_float4(g0.x + gC.x, g0.y + gC.y, g0.z + gC.z, 0.f);
        const float2 dc = dcoc(z, L);
        dth = make_float2(gc * dc.x, gc * dc.y);
    }
    block_partial(dth, partial);
}

__global__ void __launch_bounds__(1024) k_reduce(const double2* __restrict__ partial, int n, float* out) {
    __shared__ double red[2][1024];
    double a = 0.0, b = 0.0;
#pragma unroll 4
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        a += partial[k].x;
        b += partial[k].y;
    }
    red[0][threadIdx.x] = a;
    red[1][threadIdx.x] = b;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            red[0][threadIdx.x] += red[0][threadIdx.x + s];
            red[1][threadIdx.x] += red[1][threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = (float)red[0][0];
        out[1] = (float)red[1][0];
    }
}

LensD make_lensd(const hdof_lens& l, int H, float t) {
    LensD L;
    L.K = l.aperture_radius * (float)H / t;
    L.izf = 1.f / l.focus_dist;
    L.Ht = (float)H / t;
    L.t = t;
    L.dev = nullptr;
    return L;
}
LensD make_lensd_dev(const float* lens_dev, int H, float t) {
    LensD L{};
    L.Ht = (float)H / t;
    L.t = t;
    L.dev = lens_dev;
    return L;
}

size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

struct BwdWs {
    float4 *gpp, *gcrec, *gcrt, *spb, *pfb;
    float *ghacc, *kbp;
    float2* gmom;
    double2* partial;
    int n_partial;
    size_t bytes;
};

// regions from the first multiple of PF_ALIGN at or after base (a null base: the size)
BwdWs bwd_layout(int W, int H, char* base) {
    if (base) base = align_up(base, PF_ALIGN);
    BwdWs b{};
    size_t px = (size_t)W * H, o = 0;
    auto take = [&](size_t n) {
        size_t at = o;
        o += up256(n);
        return base ? base + at : nullptr;
    };
    b.gpp = reinterpret_cast<float4*>(take(16 * px));
    b.gcrec = reinterpret_cast<float4*>(take(16 * px));
    b.gcrt = reinterpret_cast<float4*>(take(16 * px));
    b.spb = reinterpret_cast<float4*>(take(16 * px));
    b.pfb = reinterpret_cast<float4*>(take(32 * pfb_plane(W, H)));
    b.kbp = reinterpret_cast<float*>(take(4 * px));
    b.ghacc = reinterpret_cast<float*>(take(4 * px));
    b.gmom = reinterpret_cast<float2*>(take(8 * px));
    int n1 = ((W + 31) / 32) * ((H + 7) / 8), n2 = ((W + 15) / 16) * ((H + 15) / 16);
    b.n_partial = 2 * n1 + n2;
    b.partial = reinterpret_cast<double2*>(take(16 * (size_t)b.n_partial));
    b.bytes = o + PF_ALIGN;
    return b;
}

int check_post(const hdof_gbuf* in, const uint8_t* spp, const float* rec, const uint32_t* ray_off,
               const hdof_camera* cam, const hdof_lens* lens, const hdof_params* p, const hdof_post_state* st,
               const char* who) {
    int rc;
    if ((rc = check_camera(cam, who)) || (lens && (rc = check_lens(lens, who))) || (rc = check_params(p, who)) ||
        (rc = check_gbuf(in, who, false)))
        return rc;
    HDOF_CHECK_ARG(in->dtype_nd == HDOF_F32 && in->dtype_col == HDOF_F32, "%s: the differentiable path is FP32", who);
    HDOF_CHECK_ARG(in->width == cam->width && in->height == cam->height, "%s: gbuf/camera size mismatch", who);
    HDOF_CHECK_ARG(spp && rec && ray_off && st, "%s: spp, rec, ray_off and state are required", who);
    HDOF_CHECK_ARG(st->rt && st->crt && st->hacc && st->mom && st->hlen && st->crec && st->sp_aux && st->pp &&
                       st->pp_aux && st->out,
                   "%s: every state buffer is required", who);
    HDOF_CHECK_ARG(!lens || lens->aperture_radius > 0.f, "%s: the lens gradient needs an aperture > 0", who);
    if (p->alpha_k != 0.f || p->blades != 0 || p->aberration != 0.f || p->spec_pref != 0.f) {
        set_error("%s: the differentiable path takes the fixed EMA weight, the uniform circular lens and no "
                  "specular preference (alpha_k, blades, aberration and spec_pref must be 0)", who);
        return HDOF_EUNSUPPORTED;
    }
    return HDOF_OK;
}

}  // namespace
}  // namespace hdof

using namespace hdof;

extern "C" size_t hdof_post_workspace_bytes(int32_t width, int32_t height, const hdof_params* p) {
    if (width <= 0 || height <= 0) return 0;
    size_t pf = ws_layout(width, height, p).pf;
    size_t bw = bwd_layout(width, height, nullptr).bytes;
    return pf > bw ? pf : bw;
}

namespace hdof {
namespace {

// the forward with the lens as a host record (lens) or on the device (lens_dev)
int post_forward(const hdof_gbuf* in, const uint8_t* spp, const float* rec, const uint32_t* ray_off,
                 const float* hist_samples, const hdof_camera* cam, const hdof_lens* lens, const float* lens_dev,
                 const hdof_params* p, const hdof_post_state* st, void* workspace, size_t workspace_bytes,
                 void* stream, const char* who) {
    clear_error();
    int rc;
    if ((rc = check_post(in, spp, rec, ray_off, cam, lens, p, st, who))) return rc;
    const int W = in->width, H = in->height;
    HDOF_CHECK_ARG(workspace && workspace_bytes >= hdof_post_workspace_bytes(W, H, p), "%s: workspace of %zu bytes < %zu",
                   who, workspace_bytes, hdof_post_workspace_bytes(W, H, p));
    cudaStream_t s = as_stream(stream);
    const float t = cam->tan_half_fovy;
    LensD L = lens ? make_lensd(*lens, H, t) : make_lensd_dev(lens_dev, H, t);
    dim3 g1((W + 31) / 32, (H + 7) / 8);
    k_replay<<<g1, 256, 0, s>>>(reinterpret_cast<const float4*>(rec), ray_off, spp, W, H, L,
                                reinterpret_cast<float4*>(st->rt));
    k_temporal_frozen<<<g1, 256, 0, s>>>(reinterpret_cast<const float4*>(st->rt), spp,
                                         reinterpret_cast<const float4*>(hist_samples), W, H, p->ema_alpha,
                                         p->camera_moved, reinterpret_cast<float4*>(st->crt), st->hacc,
                                         reinterpret_cast<float2*>(st->mom), st->hlen);
    HDOF_LAUNCHED("post-path forward: replay/temporal");
    if ((rc = launch_spatial(reinterpret_cast<const float4*>(st->crt), reinterpret_cast<const float2*>(st->mom),
                             st->hlen, W, H, p->r_s, p->var_ref, reinterpret_cast<float4*>(st->crec),
                             reinterpret_cast<float4*>(st->sp_aux), s)))
        return rc;
    // with lens_dev the kernels replace coc's lens by the device one
    const hdof_lens unit = {1.f, 1.f, 1.f};
    const Coc coc = make_coc(lens ? *lens : unit, H, t);
    if ((rc = launch_postfilter(in, coc, p, st->pp, reinterpret_cast<float4*>(st->pp_aux), workspace, s, lens_dev, t)))
        return rc;
    return launch_composite(in, spp, st->pp, nullptr, st->crt, st->crec, st->hacc, coc, p->h_tau, 0.f, st->out, s,
                            lens_dev, t);
}

// the backward with the lens as a host record (lens) or on the device (lens_dev)
int post_backward(const hdof_gbuf* in, const uint8_t* spp, const float* rec, const uint32_t* ray_off,
                  const float* hist_samples, const hdof_camera* cam, const hdof_lens* lens, const float* lens_dev,
                  const hdof_params* p, const hdof_post_state* st, const float* grad_out, float* grad_col,
                  float* grad_lens, void* workspace, size_t workspace_bytes, void* stream, const char* who) {
    clear_error();
    int rc;
    if ((rc = check_post(in, spp, rec, ray_off, cam, lens, p, st, who))) return rc;
    HDOF_CHECK_ARG(grad_out && grad_col && grad_lens, "%s: grad_out, grad_col, grad_lens required", who);
    const int W = in->width, H = in->height;
    HDOF_CHECK_ARG(workspace && workspace_bytes >= hdof_post_workspace_bytes(W, H, p), "%s: workspace of %zu bytes < %zu",
                   who, workspace_bytes, hdof_post_workspace_bytes(W, H, p));
    cudaStream_t s = as_stream(stream);
    if ((rc = ensure_area_table(s))) return rc;
    const float4* tab = nullptr;
    int ntab = 0;
    if ((rc = area_table(&tab, &ntab))) return rc;
    BwdWs b = bwd_layout(W, H, static_cast<char*>(workspace));
    LensD L = lens ? make_lensd(*lens, H, cam->tan_half_fovy) : make_lensd_dev(lens_dev, H, cam->tan_half_fovy);
    const float4* nd = static_cast<const float4*>(in->nd);
    const float4* col = static_cast<const float4*>(in->col);
    float4* gcol = reinterpret_cast<float4*>(grad_col);
    dim3 g1((W + 31) / 32, (H + 7) / 8), g2((W + 15) / 16, (H + 15) / 16);
    const int n1 = g1.x * g1.y;
    HDOF_CUDA(cudaMemsetAsync(b.gcrt, 0, 16 * (size_t)W * H, s), "post-path backward: clear");
    HDOF_CUDA(cudaMemsetAsync(b.gmom, 0, 8 * (size_t)W * H, s), "post-path backward: clear");
    k_composite_bwd<<<g1, 256, 0, s>>>(nd, col, spp, reinterpret_cast<const float4*>(st->pp),
                                       reinterpret_cast<const float4*>(st->crt), reinterpret_cast<const float4*>(st->crec),
                                       st->hacc, reinterpret_cast<const float4*>(grad_out), W, H, L, p->h_tau, gcol, b.gpp,
                                       b.gcrec, b.gcrt, b.ghacc, b.partial);
    k_spatial_bwd_prep<<<g1, 256, 0, s>>>(reinterpret_cast<const float4*>(st->crt),
                                          reinterpret_cast<const float2*>(st->mom), st->hlen,
                                          reinterpret_cast<const float4*>(st->sp_aux), b.gcrec, W, H, p->var_ref, b.spb,
                                          b.gcrt, b.gmom);
    const dim3 gs((W + SB_TW - 1) / SB_TW, (H + SB_TH - 1) / SB_TH);
    k_spatial_bwd<<<gs, SB_THREADS, 0, s>>>(reinterpret_cast<const float4*>(st->crt), b.spb, W, H, p->r_s, b.gcrt);
    k_temporal_replay_bwd<<<g1, 256, 0, s>>>(reinterpret_cast<const float4*>(rec), ray_off, spp,
                                             reinterpret_cast<const float4*>(hist_samples), b.gcrt, b.ghacc, b.gmom, W,
                                             H, L, p->ema_alpha, p->camera_moved, b.partial + n1);
    k_pf_bwd_prep<<<g1, 256, 0, s>>>(reinterpret_cast<const float4*>(st->pp_aux), b.gpp, nd, p->kz_rel, W, H, b.pfb,
                                     b.kbp, gcol);
    k_pf_bwd<<<g2, 64 * PBG, 0, s>>>(nd, col, b.pfb, b.kbp, tab, ntab, W, H, L, p->r_max, p->kz_rel, gcol,
                               b.partial + 2 * n1);
    k_reduce<<<1, 1024, 0, s>>>(b.partial, b.n_partial, grad_lens);
    HDOF_LAUNCHED("post-path backward");
    return HDOF_OK;
}

}  // namespace
}  // namespace hdof

extern "C" int hdof_post_forward(const hdof_gbuf* in, const uint8_t* spp, const float* rec, const uint32_t* ray_off,
                                 const float* hist_samples, const hdof_camera* cam, const hdof_lens* lens,
                                 const hdof_params* p, const hdof_post_state* st, void* workspace,
                                 size_t workspace_bytes, void* stream) {
    if (!lens) {
        clear_error();
        set_error("hdof_post_forward: lens is required");
        return HDOF_EINVAL;
    }
    return post_forward(in, spp, rec, ray_off, hist_samples, cam, lens, nullptr, p, st, workspace, workspace_bytes,
                        stream, "hdof_post_forward");
}

extern "C" int hdof_post_forward_dlens(const hdof_gbuf* in, const uint8_t* spp, const float* rec,
                                       const uint32_t* ray_off, const float* hist_samples, const hdof_camera* cam,
                                       const float* lens_dev, const hdof_params* p, const hdof_post_state* st,
                                       void* workspace, size_t workspace_bytes, void* stream) {
    if (!lens_dev) {
        clear_error();
        set_error("hdof_post_forward_dlens: lens_dev is required");
        return HDOF_EINVAL;
    }
    return post_forward(in, spp, rec, ray_off, hist_samples, cam, nullptr, lens_dev, p, st, workspace,
                        workspace_bytes, stream, "hdof_post_forward_dlens");
}

extern "C" int hdof_post_backward(const hdof_gbuf* in, const uint8_t* spp, const float* rec, const uint32_t* ray_off,
                                  const float* hist_samples, const hdof_camera* cam, const hdof_lens* lens,
                                  const hdof_params* p, const hdof_post_state* st, const float* grad_out,
                                  float* grad_col, float* grad_lens, void* workspace, size_t workspace_bytes,
                                  void* stream) {
    if (!lens) {
        clear_error();
        set_error("hdof_post_backward: lens is required");
        return HDOF_EINVAL;
    }
    return post_backward(in, spp, rec, ray_off, hist_samples, cam, lens, nullptr, p, st, grad_out, grad_col,
                         grad_lens, workspace, workspace_bytes, stream, "hdof_post_backward");
}

extern "C" int hdof_post_backward_dlens(const hdof_gbuf* in, const uint8_t* spp, const float* rec,
                                        const uint32_t* ray_off, const float* hist_samples, const hdof_camera* cam,
                                        const float* lens_dev, const hdof_params* p, const hdof_post_state* st,
                                        const float* grad_out, float* grad_col, float* grad_lens, void* workspace,
                                        size_t workspace_bytes, void* stream) {
    if (!lens_dev) {
        clear_error();
        set_error("hdof_post_backward_dlens: lens_dev is required");
        return HDOF_EINVAL;
    }
    return post_backward(in, spp, rec, ray_off, hist_samples, cam, nullptr, lens_dev, p, st, grad_out, grad_col,
                         grad_lens, workspace, workspace_bytes, stream, "hdof_post_backward_dlens");
}
