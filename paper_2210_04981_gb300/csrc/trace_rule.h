// A view's default trace: its form and the order of its rays (plain C++, no
// CUDA types).
#pragma once

namespace hdof {

// What a view's trace depends on is how far apart the rays that run together
// are against the scene's triangles.  They spread with the lens's width
// against the view's, kh = A / (zf tan(fovy/2)), or with the CoC scale in
// pixels, K = kh H (pixels of CoC per unit of zf/z - 1), and with the block of
// pixels they come from.  Both choices only set an order or a form: every
// ray's hit is the same.
//
// Order: 32 rays in the tile's order are all samples of 32/spp neighbours and
// spread over the whole lens; listed by lens bin they leave one of its 16
// parts from a block of sqrt(512/spp) pixels a side.  So sorting pays only
// where the lens spreads rays further than that block does, and a line in K
// sqrt(spp) stands beside the one in kh = 0.01 (1080p K = 4.6 unsorted 242,
// sorted 265 us, 7 312/318, 10 359/345, 25 521/381; 4K K = 9.3 390/495).
// In a batch, compaction and trace, unsorted / sorted (the better form of
// each) of 64 views of 256^2, 16 of 640x480, 8 of 720p, 6 of 1080p, 16
// samples; the line is K = 9:
//   K = 4.5  9519/10575, 7598/8655, 8725/9822, 11310/12618 us
//   K = 9    11046/11104, 9236/9071, 10233/10198, 12779/12970
//   K = 13   11738/11471, 10552/9441, 11562/10520, 14090/13283
//   K = 28   13409/12476, 12448/10877, 15148/11855, 18608/14475
// A single view gains earlier, by its scene from K sqrt(spp) = 8 to 80; the
// line is 14: below it a fully sampled image took up to 36% longer sorted
// (258x136, 4 samples, K = 2), above it 0.63 to 1.04 of the unsorted time.
//
// Form: warp packets while their rays stay together, ray level beyond.  Sorted
// packets / rays at 1080p K = 60 458 / 528 us, 100 545 / 568, 140 630 / 600;
// at 480x270 K = 18 283 / 320, 25 316 / 328, 60 422 / 344: kh = 0.1.  In a
// batch, which fills the machine, ray level has no tail to hide and small views
// (whose blocks of pixels are wide) turn earlier: at 256^2 between K = 2 and 9
// (sorted packets 1.12 of rays at 9, 1.20 at 20), at 640x480 at kh = 0.072, at
// 720p 0.091, at 1080p 0.105.
struct TraceRule {
    bool packets;  // warp packets (ray level with refill 4 otherwise)
    bool binned;   // a tile's rays listed by lens bin
};
inline TraceRule trace_rule(float kh, int H, int spp_max, bool batch) {
    const float K = kh * (float)H, rows = (float)H / 400.f;
    TraceRule r;
    r.packets = kh < (batch && rows < 1.f ? 0.1f * rows : 0.1f);
    r.binned = kh >= 0.01f && K * K * (float)spp_max >= (batch ? 1296.f : 200.f);
    return r;
}

}  // namespace hdof
