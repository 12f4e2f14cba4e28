// plan_table.h -- GENERATED by paper_2512_13282_gb300/tile_model.py from
// plan_measurements.json (tile_sweep.py on one GB300); do not edit by hand.
//
// Per compiled tensor-core kernel variant: the fitted time of one K step of
// BK = 64 (eff of Eq. 1 measured) and the fixed time of one unit (start and
// epilogue), in microseconds; and per operand type the split-K terms
// (reduction launch, and time per MB of fp32/int32 partials).  The planner
// minimises the busiest CTA's K steps * kstep + its units * unit + split
// terms (Eq. 9 with wave quantisation; a split tail adds one round of a
// tail unit's steps to the full rounds) + kMemWeight * the DRAM time of
// Eq. 6-8, 10 (the share of B's re-reads the kernels do not hide).
#pragma once

namespace gb300 {
namespace plan_table {

struct StepCost {
  float kstep_us;  // one K step of 64 for one unit
  float unit_us;   // per unit: start, accumulator drain, stores
};

// [0 bf16, 1 int8][0 single CTA, 1 CTA pair][BN 64, 96, 128, 192, 224, 256]; {0, 0}: not compiled
constexpr StepCost kCost[2][2][6] = {
    {
        {{0.14600f, 0.1401f}, {0.16741f, 0.3322f}, {0.21090f, 0.3281f}, {0.28599f, 0.6118f}, {0.25697f, 3.7654f}, {0.34977f, 1.1271f}},
        {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.16995f, 1.3202f}, {0.23027f, 1.8002f}, {0.23069f, 4.5338f}, {0.29964f, 1.9946f}},
    },
    {
        {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.18873f, 1.2100f}, {0.30843f, 0.8441f}, {0.28810f, 1.9227f}, {0.35987f, 1.4159f}},
        {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.16863f, 2.4881f}, {0.21109f, 3.0536f}, {0.23396f, 4.0198f}, {0.27329f, 3.6180f}},
    },
};

// split-K: [0 bf16, 1 int8]
constexpr float kSplitFixedUs[2] = {3.0379f, 1.5380f};
constexpr float kSplitUsPerMB[2] = {0.25321f, 0.20626f};

// Eq. 10: DRAM bandwidth (GB/s) and the L2 capacity the reuse factors use.
constexpr double kHbmGBs = 6693.8;
constexpr double kL2Bytes = 129000000.0;
constexpr double kMemWeight = 0.100;

}  // namespace plan_table
}  // namespace gb300
