// Batched rollout of the cooperative particle-spread scenario (App. B.1: N
// agents cover N landmarks; shared reward minus the summed distance from each
// landmark to its closest agent, minus one per collision) under policy
// combinations (Sec. 3.1: X ~ P(s, a, s' | a ~ Comb_t)), fp32 MLP policies on
// the tensor cores (mlp_x3.cuh: fp32 operands as three bf16 parts).
//
// Work unit = 128 rows of one combination for T steps: as many whole episodes
// of its envs_per_pair (<= 128) environments as fit (two of 60, sixteen of 8).
// A group of four warps plays a unit, one environment per thread with its
// state in registers: per step and agent the thread writes its observation row
// (the trajectory's row, and split for the MMAs), turns its row of layer 1
// into layer 2's operand, forms its logits and draws its action; the group's
// first thread issues the MMAs. Up to three groups of a CTA share the
// combination's policies in shared memory and overlap each other's MMAs and
// waits. Within a group the next agent's observations are written while layer
// 2 runs, and its layer 1 runs while this agent's logits and draw are formed.
// An item is a combination's chunk of units; CTAs take items in turn, and the
// policies are converted from the population's fp32 images when the
// combination changes. Where a call has fewer units than the chip takes, the
// groups of a CTA share a unit instead: each plays its own agents' tiles and
// steps a copy of the environments, and they exchange actions once a step. The
// plan (units per chunk, groups, shared or not) takes the smallest sum of
// rounds, weighted by their measured costs.
//
// What bounds it: the chain of a tile through its group (about 5,000 cycles:
// conversion 900, layer 2 1,000, logits 800, observation and stores 1,100, draw
// 300), overlapped by three groups a CTA; tensor pipe 35 % busy, issue 48 %.
// 256-row passes of packed fp32 FMAs before (61 % of the FMA pipe, one episode
// pair per CTA): spread 4,096 environments x 10 episodes 1,343 us, now 355;
// tag 9 x 125 environments x 3 episodes 990 us, now 275.
// The same kernel, templated on the scenario, runs the simple adversary, the
// simple speaker listener, the simple push, the simple tag and the simple
// reference (App. B.1) with their own environment code, and spread with contact
// forces between agents.
#include "adversary_env.cuh"
#include "push_env.cuh"
#include "ref_env.cuh"
#include "sl_env.cuh"
#include "tag_env.cuh"
#include "device_common.cuh"
#include "internal.h"
#include "mlp_x3.cuh"
#include "spread_env.cuh"

namespace malib {

namespace {

// kScen: kSpread - cooperative spread (N agents, N landmarks); kAdversary - the
// simple adversary (N = 3, two landmarks, obs 14); kSpeakerListener - the simple
// speaker listener (N = 2, three landmarks, obs 11; the speaker may take
// actions 0..2 only); kPush - the simple push (N = 2, one landmark, obs 8);
// kTag - the simple tag (N = 4, two obstacles, obs 16); kSpreadContact -
// spread whose agents also push each other apart; kReference - the simple
// reference (N = 2, three landmarks, obs 14, 15 actions: move and message).
constexpr int kSpread = 0, kAdversary = 1, kSpeakerListener = 2, kPush = 3, kTag = 4, kSpreadContact = 5,
              kReference = 6;
__host__ __device__ constexpr int actions_of(int scen) { return scen == kReference ? kRefActions : 5; }

template <int kScen, int N>
struct ScenarioEnv {
    using type = SpreadEnv<N>;
};
template <int N>
struct ScenarioEnv<kAdversary, N> {
    using type = AdvEnv;
};
template <int N>
struct ScenarioEnv<kSpeakerListener, N> {
    using type = SlEnv;
};
template <int N>
struct ScenarioEnv<kPush, N> {
    using type = PushEnv;
};
template <int N>
struct ScenarioEnv<kTag, N> {
    using type = TagEnv;
};
template <int N>
struct ScenarioEnv<kReference, N> {
    using type = RefEnv;
};

constexpr int kGroupThreads = 128;
constexpr int kMaxGroups = 3;

// How a call's units are dealt (rollout_plan).
struct RolloutPlan {
    int epu;                      // episodes per unit
    int64_t upp;                  // units per combination
    int64_t per;                  // units per chunk
    int64_t chunks;               // chunks per combination
    int64_t items;                // n_pairs * chunks
    int share;                    // the groups of a CTA share each unit's agents
};

template <int N, int IN, int kScen>
struct RolloutSmem {
    using M = MlpX3<IN, actions_of(kScen)>;
    static constexpr uint32_t kOnes = N * M::kPolicy;
    static constexpr uint32_t kX = kOnes + M::kOnesBytes;
    // Per warp, a buffer through which its rows of observations (or logits) leave
    // in the trajectory's order: kRows rows at a time, an odd number of 16-byte
    // units apart (the simple tag's four policies leave room for 16 rows only).
    static constexpr int kRows = N == 4 ? 16 : 32;
    static constexpr int kQ = M::XS / 4, kRowUnits = kQ | 1;
    static constexpr uint32_t kStage = (uint32_t)kRows * kRowUnits * 16;
    static_assert(kStage >= 32u * actions_of(kScen) * 4 || kRows == 16, "holds a warp's logits");
    static_assert(kStage >= (uint32_t)kRows * actions_of(kScen) * 4, "holds the rows' logits");
    __host__ __device__ static constexpr uint32_t stage_at(int groups) { return kX + (uint32_t)groups * M::kXBytes; }
    __host__ __device__ static constexpr uint32_t bytes(int groups) { return stage_at(groups) + 4u * groups * kStage; }
    static_assert(bytes(kMaxGroups) + 2048 <= 232448, "fits the 227 KB of shared memory of a CTA");
    static_assert(kMaxGroups * M::kCols <= 512, "fits tensor memory");
};

template <int N, int kScen, int XS, class Env>
__device__ __forceinline__ void scenario_obs(const Env& s, int i, float* o) {
    if constexpr (kScen == kAdversary) adv_obs<XS>(s, i, o);
    else if constexpr (kScen == kSpeakerListener) sl_obs<XS>(s, i, o);
    else if constexpr (kScen == kPush) push_obs<XS>(s, i, o);
    else if constexpr (kScen == kTag) tag_obs<XS>(s, i, o);
    else if constexpr (kScen == kReference) ref_obs<XS>(s, i, o);
    else spread_obs<N, XS>(s, i, o);
}

// The actions an agent may take.
template <int kScen>
__device__ __forceinline__ unsigned legal_of(int i) {
    return (kScen == kSpeakerListener && i == 0) ? kSlSpeakerLegal : (1u << actions_of(kScen)) - 1u;
}

// One thread, one step: the agents whose bits from 16 on are set in act_pk (their
// operands' parts were not finite somewhere) take their actions from a forward in fp32
// FMAs of their observations, which are in the trajectory; ix: the step's agent 0.
template <int N, int IN, int kScen, bool kLogits>
__device__ __noinline__ uint32_t redo_agents(const RolloutArgs& a, int pair, int64_t ix, uint64_t g, uint32_t t,
                                             uint32_t act_pk) {
    constexpr int A = actions_of(kScen), XS = MlpX3<IN, A>::XS;
    for (int i = 0; i < N; ++i) {
        if (((act_pk >> (16 + i)) & 1u) == 0u) continue;
        float z[A];
        forward_fma<IN, MlpX3<IN, A>::H, A>(a.arena + a.pol_offset[a.pairs[pair * N + i]], a.obs + (ix + i) * XS, z);
        const float uu = u24(draw(g, t, (uint32_t)i, a.seed).x);
        act_pk = (act_pk & ~(0xfu << (4 * i))) | (uint32_t)sample_masked<A>(z, legal_of<kScen>(i), uu) << (4 * i);
        if (kLogits)
            for (int k = 0; k < A; ++k) a.logits[(ix + i) * A + k] = z[k];
    }
    return act_pk;
}

// kLogits: the call records the logits (the recording code is compiled out of
// the other instance). blockDim.x = 128 groups.
template <int N, int IN, int kScen = kSpread, bool kLogits = false>
__global__ void __launch_bounds__(kGroupThreads * kMaxGroups, 1)
    spread_rollout_x3_kernel(const __grid_constant__ RolloutArgs a, const __grid_constant__ RolloutPlan plan) {
    static_assert(kScen != kAdversary || (N == 3 && IN == kAdvObs), "the simple adversary has 3 agents, obs 14");
    static_assert(kScen != kSpeakerListener || (N == 2 && IN == kSlObs),
                  "the simple speaker listener has 2 agents, obs 11");
    static_assert(kScen != kPush || (N == 2 && IN == kPushObs), "the simple push has 2 agents, obs 8");
    static_assert(kScen != kTag || (N == 4 && IN == kTagObs), "the simple tag has 4 agents, obs 16");
    static_assert(kScen != kReference || (N == 2 && IN == kRefObs), "the simple reference has 2 agents, obs 14");
    static_assert(N <= 4 && actions_of(kScen) <= 16, "four bits per agent's action in a 16-bit word");
    constexpr int A = actions_of(kScen);
    using SM = RolloutSmem<N, IN, kScen>;
    using M = typename SM::M;
    constexpr int XS = M::XS;           // == obs_pad
    extern __shared__ __align__(1024) uint8_t smem[];
    // [group][layer]: its MMAs are complete. One barrier per layer: a thread still
    // waiting for layer 2 must not meet the completion of the next layer 1, issued
    // as soon as the issuing warp has seen layer 2 done (with one barrier that
    // would be its own phase again). Each is completed again only after a
    // barrier of the group that follows every thread's wait.
    __shared__ __align__(8) uint64_t bars[kMaxGroups][2];
    __shared__ uint32_t tmem_base;
    __shared__ uint32_t dead;           // a bounded wait expired: nobody waits any more
    __shared__ uint16_t acts[2][kMaxGroups][kGroupThreads];   // shared units: each group's actions of a step

    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int grp = warp >> 2, r = tid & 127;            // group, row of its tiles
    const int groups = blockDim.x >> 7;
    const bool issuer = (warp & 3) == 0;                 // this warp issues the group's MMAs
    if (tid == 0) {
        for (int g = 0; g < 2 * kMaxGroups; ++g) mbar_init(&bars[0][0] + g, 1);
        dead = 0u;
    }
    if (grp == 0) M::put_ones(smem + SM::kOnes, r);      // fenced with the first policies
    if (warp == 0) {
        tc::tmem_alloc(&tmem_base, 512);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tb = tmem_base + (uint32_t)grp * M::kCols;
    const uint32_t lane_q = (uint32_t)(32 * (warp & 3)) << 16;
    uint8_t* X = smem + SM::kX + (uint32_t)grp * M::kXBytes;
    float4* buf = reinterpret_cast<float4*>(smem + SM::stage_at(groups) + (uint32_t)warp * SM::kStage);
    uint64_t* bar = bars[grp];
    uint32_t phase[2] = {0, 0};
    uint32_t turn = 0;                                   // buffer of acts, alternating over units and items
    auto is_dead = [&] { return *(volatile uint32_t*)&dead != 0u; };
    auto group_sync = [&] { asm volatile("bar.sync %0, 128;" ::"r"(grp + 1) : "memory"); };
    // layer `layer` (0, 1) of the group's current tile has completed
    auto mma_wait = [&](int layer) {
        if (!is_dead() && !mbar_wait_bounded(bar + layer, phase[layer], kWaitLimitNs)) {
            *(volatile uint32_t*)&dead = 1u;
            atomicOr(a.err, ERRBIT_TIMEOUT);
            mbar_wait_bounded(bar + layer, phase[layer], kWaitLimitNs);     // its MMAs in flight; none are issued after
        }
        phase[layer] ^= 1u;
        tc::fence_after_sync();
    };

    const int epp = (int)(a.n_envs / a.n_pairs);
    const int T = a.episode_len;
    int staged = -1;
    for (int64_t item = blockIdx.x; item < plan.items; item += gridDim.x) {
        const int pair = (int)(item / plan.chunks);
        const int64_t u_lo = (item - (int64_t)pair * plan.chunks) * plan.per;
        const int64_t u_hi = u_lo + plan.per < plan.upp ? u_lo + plan.per : plan.upp;
        if (pair != staged) {
            bool ok = true;
            for (int i = 0; i < N; ++i) {
                const int p = a.pairs[pair * N + i];
                ok = ok && p >= 0 && p < a.n_pol;
            }
            if (!ok) {
                if (tid == 0) atomicOr(a.err, ERRBIT_BAD_PAIR);
                continue;
            }
            __syncthreads();   // every group is done with the previous policies
            for (int i = 0; i < N; ++i)
                M::stage(smem + i * M::kPolicy, a.arena + a.pol_offset[a.pairs[pair * N + i]], tid, blockDim.x);
            fence_proxy_async_smem();
            __syncthreads();
            staged = pair;
        }
        // agents i0, i0 + di, ... are this group's
        const int i0 = plan.share ? grp : 0, di = plan.share ? groups : 1;
        for (int64_t u = plan.share ? u_lo : u_lo + grp; u < u_hi; u += plan.share ? 1 : groups) {
            const int slot = r / epp, v = r - slot * epp;
            const int64_t ep = u * plan.epu + slot;
            const bool mine = slot < plan.epu && ep < a.n_episodes;
            const bool busy = __any_sync(0xffffffffu, mine);     // warps without rows only keep step
            const int64_t env = (int64_t)pair * epp + v;
            const uint64_t g = (uint64_t)ep * (uint64_t)a.n_envs + (uint64_t)env;
            typename ScenarioEnv<kScen, N>::type s;
            if (mine) {
                if constexpr (kScen == kAdversary) adv_reset(s, g, a.seed);
                else if constexpr (kScen == kSpeakerListener) sl_reset(s, g, a.seed);
                else if constexpr (kScen == kPush) push_reset(s, g, a.seed);
                else if constexpr (kScen == kTag) tag_reset(s, g, a.seed);
                else if constexpr (kScen == kReference) ref_reset(s, g, a.seed);
                else spread_reset<N>(s, g, a.seed);
            } else {
                M::zero_row(X, r);      // stays zero for the unit
            }
            int64_t ix = (ep * T * a.n_envs + env) * N;          // this step's (env, agent 0)
            // Agent i's observation into the tile. It leaves for the trajectory
            // only after the barrier that follows: the proxy fence waits for the
            // thread's earlier stores, and with the global ones before it that
            // took 2,000 cycles.
            float o[XS];
            auto observe = [&](int i) {
                if (mine) {
#pragma unroll
                    for (int j = 0; j < N; ++j)
                        if (j == i) scenario_obs<N, kScen, XS>(s, j, o);
                    M::put_row(X, r, o);
                }
                fence_proxy_async_smem();
            };
            // The warp's rows through its buffer, so that consecutive lanes store
            // consecutive 16-byte units (4-byte ones for logits) of an
            // environment's row: stored by each thread for itself, a warp's store
            // touched 32 lines, and a step's stores took 2,500 cycles.
            auto store_obs = [&](int i) {
                if (!busy) return;
                const unsigned rows = __ballot_sync(0xffffffffu, mine);
                const int64_t at = (ix + i) * SM::kQ;
#pragma unroll
                for (int h = 0; h < 32; h += SM::kRows) {
                    __syncwarp();                            // the buffer is read
                    if (lane >= h && lane < h + SM::kRows)
#pragma unroll
                        for (int q = 0; q < SM::kQ; ++q)
                            buf[(lane - h) * SM::kRowUnits + q] =
                                make_float4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < SM::kRows * SM::kQ / 32; ++k) {
                        const int c = lane + 32 * k, row = c / SM::kQ, q = c - row * SM::kQ;
                        const int64_t to = __shfl_sync(0xffffffffu, at, row + h);
                        if ((rows >> (row + h)) & 1u)
                            reinterpret_cast<float4*>(a.obs)[to + q] = buf[row * SM::kRowUnits + q];
                    }
                }
            };
            auto store_logits = [&](int i, const float (&lg)[A]) {
                const unsigned rows = __ballot_sync(0xffffffffu, mine);
                const int64_t at = (ix + i) * A;
                float* fb = reinterpret_cast<float*>(buf);
#pragma unroll
                for (int h = 0; h < 32; h += SM::kRows) {
                    __syncwarp();
                    if (lane >= h && lane < h + SM::kRows)
#pragma unroll
                        for (int k = 0; k < A; ++k) fb[(lane - h) * A + k] = lg[k];
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < (SM::kRows * A + 31) / 32; ++k) {
                        const int c = lane + 32 * k, row = c / A, q = c - row * A;
                        const int64_t to = __shfl_sync(0xffffffffu, at, (row + h) & 31);
                        if (row < SM::kRows && ((rows >> (row + h)) & 1u)) a.logits[to + q] = fb[c];
                    }
                }
            };
            // the group's tile is written (and layer 2 of the tile before is done): layer 1
            auto layer1 = [&](int i) {
                if (issuer && !is_dead() && tc::elect_one())
                    M::issue1(tb, smem_u32(X), smem_u32(smem + SM::kOnes), smem_u32(smem + i * M::kPolicy), bar);
                __syncwarp();
            };
            observe(i0);
            tc::fence_before_sync();
            group_sync();
            tc::fence_after_sync();
            layer1(i0);
            store_obs(i0);
            for (int t = 0; t < T; ++t) {
                uint32_t act_pk = 0;
#pragma unroll 1
                for (int i = i0; i < N; i += di) {
                    const uint8_t* pol = smem + i * M::kPolicy;
                    mma_wait(0);                             // layer 1
                    if (busy) M::hidden(tb, lane_q);
                    tc::fence_before_sync();
                    group_sync();
                    tc::fence_after_sync();
                    if (issuer && !is_dead() && tc::elect_one()) M::issue2(tb, smem_u32(smem + SM::kOnes), smem_u32(pol), bar + 1);
                    __syncwarp();
                    const float uu = u24(draw(g, (uint32_t)t, (uint32_t)i, a.seed).x);
                    if (i + di < N) {
                        observe(i + di);                     // layer 1 no longer reads the tile
                        group_sync();
                        store_obs(i + di);
                    }
                    mma_wait(1);                             // layer 2
                    if (i + di < N) layer1(i + di);
                    if (busy) {
                        float lg[A];
                        M::logits(tb, lane_q, pol, lg);
                        if (mine) {
                            act_pk |= (uint32_t)sample_masked<A>(lg, legal_of<kScen>(i), uu) << (4 * i);
                            if (parts_failed(lg[0])) act_pk |= 0x10000u << i;
                        }
                        if (kLogits) store_logits(i, lg);
                    }
                }
                // agents whose parts failed (a call in their own loop cost it 1 to 5 %)
                if (__any_sync(0xffffffffu, act_pk >> 16 != 0u)) {
                    __syncwarp();                            // after the other lanes' stores of this row
                    if (act_pk >> 16 != 0u) act_pk = redo_agents<N, IN, kScen, kLogits>(a, pair, ix, g, (uint32_t)t, act_pk);
                }
                if (plan.share) {
                    // the other groups' actions (a buffer is written again only
                    // after the next exchange's barrier, be it in the next unit)
                    acts[turn][grp][r] = (uint16_t)act_pk;
                    asm volatile("bar.sync %0, %1;" ::"r"(kMaxGroups + 1), "r"((int)blockDim.x) : "memory");
                    for (int q = 0; q < groups; ++q)
                        if (q != grp) act_pk |= acts[turn][q][r];
                    turn ^= 1u;
                }
                int act[N];
                float rw[N];
#pragma unroll
                for (int i = 0; i < N; ++i) act[i] = (int)((act_pk >> (4 * i)) & 0xfu);
                if (mine) {
                    if constexpr (kScen == kAdversary) adv_step(s, act, rw);
                    else if constexpr (kScen == kSpeakerListener) sl_step(s, act, rw);
                    else if constexpr (kScen == kPush) push_step(s, act, rw);
                    else if constexpr (kScen == kTag) tag_step(s, act, rw);
                    else if constexpr (kScen == kReference) ref_step(s, act, rw, a.local_ratio < 0.f ? 0.5f : a.local_ratio);
                    else spread_step<N, kScen == kSpreadContact>(s, act, rw, a.local_ratio);
                }
                if (t + 1 < T) {
                    observe(i0);
                    tc::fence_before_sync();
                    group_sync();
                    tc::fence_after_sync();
                    layer1(i0);
                }
                if (mine) {
#pragma unroll
                    for (int i = 0; i < N; ++i) {
                        if (plan.share && i % groups != grp) continue;
                        a.action[ix + i] = (uint8_t)act[i];
                        a.reward[ix + i] = rw[i];
                    }
                    if (i0 == 0) a.done[(ep * T + t) * a.n_envs + env] = (t == T - 1) ? 1 : 0;
                }
                ix += a.n_envs * N;
                if (t + 1 < T) store_obs(i0);
            }
            // the next unit's first barrier orders its MMAs after this unit's
            // last reads of D2
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem_base, 512);
}

// Costs in units of one unit played by one group alone (152 CTAs, 128
// environments; spread 242 us): a round of g groups took 1.14 to 1.26 (g = 2)
// and 1.37 to 1.56 (3), a unit shared by its agents' groups 0.70 to 0.82 over
// the seven scenarios; converting a combination's policies about 5 us.
constexpr double kRoundCost[kMaxGroups + 1] = {0.0, 1.0, 1.2, 1.46};
constexpr double kShareCost = 0.76;
constexpr double kStageCost = 0.03;

RolloutPlan rollout_plan(int32_t n_pairs, int n_agents, int64_t epp, int64_t n_episodes, int n_sm, int* groups,
                         int64_t* grid) {
    RolloutPlan p{};
    p.epu = (int)(kGroupThreads / epp);
    p.upp = (n_episodes + p.epu - 1) / p.epu;
    const int gs = n_agents == 3 ? 3 : 2;              // groups of a shared unit: equal numbers of agents
    double best = 1e300;
    // chunks of `per` units: all sizes up to 96, then doubling
    for (int64_t per = 1; per <= p.upp; per = per < 96 ? per + 1 : (per * 2 < p.upp || per == p.upp ? per * 2 : p.upp)) {
        const int64_t chunks = (p.upp + per - 1) / per;
        const int64_t turns = ((int64_t)n_pairs * chunks + n_sm - 1) / n_sm;
        for (int g = 0; g <= kMaxGroups && g <= per; ++g) {   // 0: shared units
            const double rounds = g == 0 ? (double)per * kShareCost : (double)((per + g - 1) / g) * kRoundCost[g];
            const double cost = (double)turns * (kStageCost + rounds);
            if (cost < best) {
                best = cost;
                p.per = per;
                p.chunks = chunks;
                p.share = g == 0;
                *groups = g == 0 ? gs : g;
            }
        }
    }
    p.items = (int64_t)n_pairs * p.chunks;
    *grid = p.items < n_sm ? p.items : n_sm;
    return p;
}

template <int N, int IN, int kScen = kSpread>
cudaError_t launch_rollout(const RolloutArgs& a, int n_sm, cudaStream_t s) {
    using SM = RolloutSmem<N, IN, kScen>;
    int groups = 1;
    int64_t grid = 1;
    const RolloutPlan plan = rollout_plan(a.n_pairs, N, a.n_envs / a.n_pairs, a.n_episodes, n_sm, &groups, &grid);
    auto kern = a.logits ? spread_rollout_x3_kernel<N, IN, kScen, true> : spread_rollout_x3_kernel<N, IN, kScen, false>;
    // the limit is the process's: the most that any call takes, so that a call of another
    // thread never lowers it between this one's two steps
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM::bytes(kMaxGroups));
    if (err != cudaSuccess) return err;
    kern<<<(unsigned)grid, kGroupThreads * groups, SM::bytes(groups), s>>>(a, plan);
    return cudaGetLastError();
}

}  // namespace

bool scenario_f32_supported(int hidden) { return hidden == 64; }

bool spread_f32_supported(int n_agents, int obs_dim, int hidden) {
    return n_agents == 3 && obs_dim == 18 && hidden == 64;
}

cudaError_t launch_spread_rollout_f32(const RolloutArgs& a, int hidden, int n_sm, cudaStream_t s) {
    if (a.n_pairs == 0 || a.n_episodes == 0) return cudaSuccess;
    if (a.env_kind == MALIB_ENV_ADVERSARY) {
        if (hidden == 64) return launch_rollout<3, kAdvObs, kAdversary>(a, n_sm, s);
        return cudaErrorInvalidValue;
    }
    if (a.env_kind == MALIB_ENV_SPEAKER_LISTENER) {
        if (hidden == 64) return launch_rollout<2, kSlObs, kSpeakerListener>(a, n_sm, s);
        return cudaErrorInvalidValue;
    }
    if (a.env_kind == MALIB_ENV_PUSH) {
        if (hidden == 64) return launch_rollout<2, kPushObs, kPush>(a, n_sm, s);
        return cudaErrorInvalidValue;
    }
    if (a.env_kind == MALIB_ENV_REFERENCE) {
        if (hidden == 64) return launch_rollout<2, kRefObs, kReference>(a, n_sm, s);
        return cudaErrorInvalidValue;
    }
    if (a.env_kind == MALIB_ENV_TAG) {
        if (hidden == 64) return launch_rollout<4, kTagObs, kTag>(a, n_sm, s);
        return cudaErrorInvalidValue;
    }
    if (a.n_agents == 3 && a.obs_dim == 18 && hidden == 64)
        return a.contact ? launch_rollout<3, 18, kSpreadContact>(a, n_sm, s)
                         : launch_rollout<3, 18>(a, n_sm, s);
    return cudaErrorInvalidValue;
}

}  // namespace malib
