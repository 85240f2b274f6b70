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

}  // namespace rtp
