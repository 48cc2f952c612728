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
    Wgrad9Plan plan{max_slices, 1, 0};
    int64_t best = INT64_MAX;
    for (int c = 1; c <= ((int64_t)total * 64 <= (int64_t)kPairChain * max_slices ? 2 : 1); ++c)
        for (int s = max_slices; s >= 1 && s * c >= max_slices && 100 * max_slices <= 115 * s; --s) {
            const int64_t waves = ((int64_t)tiles * s * c + kWgradSMs - 1) / kWgradSMs;
            const int64_t t = waves * ((total + s * c - 1) / (s * c) + 8);  // 8: prologue and drain
            if (t < best) best = t, plan.slices = s, plan.ctas = c;
        }
    const int all = plan.slices * plan.ctas;
    plan.per = (total + all - 1) / all;
    const int filled = plan.per * plan.ctas;
    plan.slices = (total + filled - 1) / filled;  // every slice has work in its first CTA
    return plan;
}

}  // namespace nn
}  // namespace lbm
