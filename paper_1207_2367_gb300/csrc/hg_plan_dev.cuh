// hg_plan_dev.cuh -- the evaluation planner on one CTA.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "hg_internal.cuh"

namespace hg {
namespace {

// The evaluation plan for block size m, by every thread of one CTA (at least
// kPlanCandidates threads would score one candidate each; fewer loop): the
// lowest cost wins, ties to the lowest candidate index (make_plan's choice on
// the host).  A tuned candidate of m's bucket that is admissible wins outright.
// Thread 0 writes *out (global or shared memory).
__device__ void plan_on_block(int64_t m, const PlanParams &q, Plan *out)
{
    __shared__ int64_t s_cost[32];
    __shared__ int s_cand[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    Plan p;
    const int tc = q.tuned[tune_bucket(m)];
    if (tc >= 0 && plan_candidate(m, q, tc, p) >= 0) {   // measured choice
        if (threadIdx.x == 0) *out = p;
        return;
    }
    int64_t best = -1;
    int bc = 0x7fffffff;
    for (int c = threadIdx.x; c < plan_total(q); c += blockDim.x) {
        const int64_t cost = plan_candidate(m, q, c, p);
        if (cost >= 0 && (best < 0 || cost < best)) {
            best = cost;
            bc = c;
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        const int64_t ob = __shfl_xor_sync(0xffffffffu, best, off);
        const int oc = __shfl_xor_sync(0xffffffffu, bc, off);
        if (ob >= 0 && (best < 0 || ob < best || (ob == best && oc < bc))) {
            best = ob;
            bc = oc;
        }
    }
    if (lane == 0) {
        s_cost[w] = best;
        s_cand[w] = bc;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < nw; ++k) {
            const int64_t ob = s_cost[k];
            const int oc = s_cand[k];
            if (ob >= 0 && (best < 0 || ob < best || (ob == best && oc < bc))) {
                best = ob;
                bc = oc;
            }
        }
        if (best >= 0)
            plan_candidate(m, q, bc, p);
        else
            p = plan_unsplit(m, q);
        *out = p;
    }
}

}  // namespace
}  // namespace hg
