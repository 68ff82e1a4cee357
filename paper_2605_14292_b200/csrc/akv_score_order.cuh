// Where event_pool_kernel (akv_event_pool.cuh) keeps the rows of an event while it scores them. Plain C++, so that it also compiles for
// the host by itself.
#pragma once

#ifdef __CUDACC__
#define AKV_ORDER_HD __host__ __device__ __forceinline__
#else
#define AKV_ORDER_HD inline
#endif

namespace akv {

// An event's blocks of 16 rows are two chains of score_steps(n) blocks (the second may be shorter by one): step i scores block i and block
// score_steps(n) + i side by side, each with the rotation of the block before it in its chain turned by one step of positions. All forms of the
// kernel do, so that a rotation, and with it a score, is the same to the bit in each.
AKV_ORDER_HD int score_steps(int n) { return (((n + 15) >> 4) + 1) >> 1; }

// 193 to 256 rows where shared memory has room for 192, half of it for each chain. What the last two steps score comes late, into the slots of
// what the first two have scored. The slot of a row of step `step` as a distance from the row's own number:
constexpr int kLateSteps = 2, kChainSlots = 96;
AKV_ORDER_HD int late_slot_shift(int step, int steps, int chain) {
    return chain * (kChainSlots - 16 * steps) - (step < steps - kLateSteps ? 0 : 16 * (steps - kLateSteps));
}

}  // namespace akv
