// When a Sinkhorn iteration of the scaling form has nothing left to move, for tiles of up to 639 pruned tokens (plain C++:
// the rule is also compiled for the host by its test).
#pragma once
#include <stdlib.h>

#ifndef __CUDACC__
#define __host__
#define __device__
#endif

namespace rtp {

// A dual's value after this iteration, the last and the one before that, as the bit patterns of positive floats (neighbours
// differ by one).  Settled: within one unit in the last place of the last value, or cycling: within four units of it and back
// within one unit of the one before (the rounding of sums of a few hundred terms can go round such a cycle for good).  Two
// iterations then move it by a unit, no more than the first clause lets each of them do; steps of a few units that all lead
// one way are no cycle.
__host__ __device__ inline bool dual_settled(int now, int last, int before)
{
    const int d = abs(now - last), back = abs(now - before);
    const int cycle = d - 3 > back ? d - 3 : back;             // (no branches: the test is on the way to the next iteration)
    return (d < cycle ? d : cycle) <= 1;
}

// The recursion leaves U -> U/c, V -> cV free, and rounding moves c by a unit or two per iteration long after the plan U K V
// has settled.  lo and hi: the smallest and largest relative move (V - V_last) / V_last of an iteration over all columns, the
// dustbin's among them.  Settled: they lie within two units of 2^-23 of each other, that is every column within one unit of a
// common factor: what single duals that each move by one unit at most, up or down, can spread over.  A column that still
// drifts against the others keeps the loop going.  Measured against 64 bits on the device, 64 to 1156 tokens, eps 1, 0.3 and
// 0.1: the weights' rms error is that of the rule for single duals within 2 % either way (bf16 storage 0.2 to 2.2e-6, fp32
// 1.9 to 3.3e-7), and the loop is shorter by 1 iteration of 7 at eps = 1, 2 of 15 at 0.3, 3 of 32 at 0.1, the longest of a
// batch of 64 or 128 images at eps = 1 by 6 of 15 and 7 of 18: 1 x 400 48.3 -> 45.6 us, 32 x 256 65.4 -> 61.7, 64 x 400 105.5
// -> 103.9, 128 of 456-1156 433 -> 424, 64 of them at eps = 0.1 590 -> 576.
constexpr float kPlanSpread = 2.38418579e-7f;      // 2 * 2^-23
// (Where a column is not a number, lo and hi are none either: the rule for single duals decides.)
__host__ __device__ inline bool plan_settled(float lo, float hi) { return hi - lo <= kPlanSpread; }

}  // namespace rtp
