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
// dustbin's among them.  Settled: they lie within 2^-22 of each other, so that every column is within 2^-23 of its value (one to
// two units in the last place, by its mantissa) of a common factor: what single duals that each move by 2^-23 at most, up or down,
// can spread over.  One column alone may move by two or three units; one that drifts by more against the others keeps the loop
// going.  Measured against 64 bits on the device: the weights' rms error is that of the rule for single
// duals and of all 100 iterations within 1 % (bf16 storage 1.0e-6 at eps = 1, 1.6e-6 at 0.3, 2.2e-6 at 0.1, 3.6 to 4.2e-6 at 0.05; fp32
// 1.6 to 1.9e-6 at 0.05 to 0.07; 64 to 1156 tokens), and images leave after 6.4 iterations instead of 7.5 on average at eps = 1 (the
// longest of 64 after 8 instead of 12), 12.4 instead of 14.9 at 0.3, 25 instead of 28 at 0.1, 34 to 82 instead of 37 to 83 at 0.05.
constexpr float kPlanSpread = 2.38418579e-7f;      // 2 * 2^-23
// (Where a column is not a number, lo and hi are none either: the rule for single duals decides.)
__host__ __device__ inline bool plan_settled(float lo, float hi) { return hi - lo <= kPlanSpread; }

}  // namespace rtp
