// range_table.h -- the costs that decide where a bf16 GEMM's K is cut.
//
// An fp32 accumulator in tensor memory rounds at every MMA, so what a bf16 sum
// rounds to depends on the K ranges it is formed in: N(0, 1) operands with K =
// 4096 are off the nearest bf16 in 0.24 % of the results as one chain and in
// 0.13 % as two chains of 2048 added in fp32.  The ranges are therefore a
// property of the GEMM's sizes: the K split of the plan that is fastest by the
// costs below, which stay as they are when plan_table.h is fitted again.  A
// kernel then sums those ranges in order, in fp32, as split-K partials or in
// registers (kTmaOutSlabs); tests/test_bf16_ranges.py holds both to each other.
// A split tail cuts K for the tiles of the last round alone: a plan with one by
// these costs runs as it is, tile and family included, and no other plan gets
// one.  (60 seeded shapes whose tail the later fit had changed: 2 % slower than
// by that fit, 1.18 at worst and 0.88 at best, and 5 % faster than before it.)
// The costs are those of kernels whose MMA loops were issued by one lane.  A
// later fit alone moved the cuts (128 x 12288 x 4096 to one range); with the
// ranges kept, that GEMM runs unsplit in 20.5 us where the split takes 27.6 and
// one chain 20.2, and 128 x 4096 x 11008 in its six splits in 24.4 us where
// four take 23.0.
#pragma once

#include "plan_table.h"

namespace gb300 {
namespace range_table {

// plan_table.h's entries for bf16: [0][0 single CTA, 1 CTA pair][BN 64, 96, 128, 192, 224, 256]
constexpr plan_table::StepCost kCost[1][2][6] = {
    {
        {{0.26885f, 0.0812f}, {0.27958f, 0.0000f}, {0.27863f, 0.1047f}, {0.29486f, 0.5838f}, {0.28341f, 2.6772f}, {0.35269f, 1.0832f}},
        {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.27831f, 0.7914f}, {0.28422f, 1.2185f}, {0.27975f, 3.0965f}, {0.29593f, 1.6487f}},
    },
};
constexpr float kSplitFixedUs[1] = {2.6661f};
constexpr float kSplitUsPerMB[1] = {0.34096f};

}  // namespace range_table
}  // namespace gb300
