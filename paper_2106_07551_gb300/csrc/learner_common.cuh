// What the learner's gradient kernels share: the sample order of a batch and the
// CTAs' shares of its tiles.
#pragma once

#include "internal.h"

namespace malib {

constexpr int kH = 64, kA = 5;                           // hidden width, actions
constexpr int kTile = 128, kThreads = 256;               // samples of a tile, threads of a CTA

// Sample s of the policy's sample order: (slot, episode, step, env) -> the
// trajectory index of its (episode, step, env, agent).
__device__ __forceinline__ int64_t sample_index(const LearnArgs& a, const int32_t* slots, int64_t s, int epp) {
    int r, t;
    int64_t e, slot;
    if ((s | a.n_episodes) <= 0x7fffffff) {              // 32-bit divisions where they do
        const uint32_t q = (uint32_t)s / (uint32_t)epp, q2 = q / (uint32_t)a.T;
        r = (int)((uint32_t)s - q * (uint32_t)epp);
        t = (int)(q - q2 * (uint32_t)a.T);
        slot = q2 / (uint32_t)a.n_episodes;
        e = q2 - (uint32_t)slot * (uint32_t)a.n_episodes;
    } else {
        r = (int)(s % epp);
        const int64_t q = s / epp;                        // (slot, e, t)
        t = (int)(q % a.T);
        const int64_t q2 = q / a.T;
        e = q2 % a.n_episodes;
        slot = q2 / a.n_episodes;
    }
    const int ck = slots[slot];
    const int c = ck / a.n_agents, ka = ck - c * a.n_agents;
    const int64_t env = (int64_t)c * epp + r;
    return ((e * a.T + t) * a.n_envs + env) * a.n_agents + ka;
}

// A CTA's contiguous share [lo, hi) of the batch's tiles (all policies' tiles
// in policy order).
__device__ __forceinline__ int64_t share_lo(const LearnArgs& a, int64_t c) {
    return a.tile_off[a.nb] * c / a.grid;
}

// Observation widths up to this one take the tensor-core kernel (learner_x3.cu): the
// next one's two X tiles and W1 images would not fit its shared memory. 18 wide it
// takes 1.08 ms where the general kernel takes 2.92; nearly all ReLU branches are the same.
constexpr int kLearnX3MaxIn = 20;
cudaError_t launch_learn_grad_x3(const LearnArgs& a, cudaStream_t s);

}  // namespace malib
