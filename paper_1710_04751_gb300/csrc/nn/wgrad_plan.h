// wgrad_plan.h -- how the nine-tap weight gradient (conv.cu) splits its voxels.  Host only, no CUDA.
#pragma once

#include <stdint.h>

namespace lbm {
namespace nn {

constexpr int kWgradSMs = 152;

// Slices of the workspace and CTAs that share one (2: a cluster, whose second CTA adds its sums to
// the first's); blocks of 64 voxels per CTA -- the length of its accumulation chain.
struct Wgrad9Plan {
    int slices, ctas, per;
    int64_t work;  // blocks that the busiest SM goes through, prologues and drains included
};

// The tensor core's FP32 accumulation truncates, so the length of its chains shows in the result:
// about 7e-10 of relative error per voxel of a chain.  No chain is longer than the caller's split
// (max_slices) makes it.  Two chains of half the length may take a slice's place up to kPairChain
// voxels, beyond which that would move a result by 2e-5, and then a slice may hold 1.15 times as
// many voxels.  Among these the choice that leaves the least work to the busiest SM.
constexpr int kPairChain = 38400;
inline Wgrad9Plan plan_wgrad9(int total, int cin, int cout, int max_slices) {
    const int tiles = (3 * (cin / 32) + 3) / 4 * ((cout + 31) / 32);
    if (max_slices > total) max_slices = total;
    Wgrad9Plan plan{max_slices, 1, 0, INT64_MAX};
    for (int c = 1; c <= ((int64_t)total * 64 <= (int64_t)kPairChain * max_slices ? 2 : 1); ++c)
        for (int s = max_slices; s >= 1 && s * c >= max_slices && 100 * max_slices <= 115 * s; --s) {
            const int64_t waves = ((int64_t)tiles * s * c + kWgradSMs - 1) / kWgradSMs;
            const int64_t t = waves * ((total + s * c - 1) / (s * c) + 8);  // 8: prologue and drain
            if (t < plan.work) plan.work = t, plan.slices = s, plan.ctas = c;
        }
    const int all = plan.slices * plan.ctas;
    plan.per = (total + all - 1) / all;
    const int filled = plan.per * plan.ctas;
    plan.slices = (total + filled - 1) / filled;  // every slice has work in its first CTA
    return plan;
}

// Whether the nine-tap form takes the weight gradient of a grid from 16^3 with up to 64 output
// channels and M voxels, which the caller splits into `used` slices of `per` blocks.  A nine-tap CTA
// goes through a block in 0.32 us (0.43 where the last 16 output channels are cut in half, whose
// rows TMA fetches in part), a one-tap CTA in about 0.21, but there are nine times as many of those
// for a third of the operand reads, so the work of the busiest SM decides: with few splits the nine-tap
// CTAs leave most SMs idle.  Calls with the host wait, us, one-tap / nine-tap: 64^3 batch 2, 32 -> 32
// channels in 43 splits 115 / 79, 16: 122 / 126, 8: 204 / 364, 1: 1535 / 2605; 96 -> 32 in 14
// 251 / 144, 8: 378 / 367, 4: 521 / 688; 128 -> 40 in 11 664 / 362; 32 -> 24 in 43 133 / 93, 8:
// 274 / 484; 32^3 batch 4, 256 -> 64 in 5 178 / 121, 2: 273 / 396; 128^3, 32 -> 32 in 43 345 / 285,
// 16: 521 / 688.  Below 2^23 voxels x input channels its long ramp shows in any split: 32^3, 64 -> 64
// 79 / 82, 16^3 batch 4, 64 -> 48 64 / 75.
inline bool nine_taps_pay(int64_t M, int cin, int cout, int Kp, int used, int per) {
    if (M * cin < (int64_t(1) << 23)) return false;
    const int64_t ctas = (int64_t)((Kp + 127) / 128) * used;
    const int64_t one = (ctas + kWgradSMs - 1) / kWgradSMs * per;
    return plan_wgrad9((int)(M / 64), cin, cout, used).work * (cout % 16 == 8 ? 7 : 6) < one * 4;
}

}  // namespace nn
}  // namespace lbm
