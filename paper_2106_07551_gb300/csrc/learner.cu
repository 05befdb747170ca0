// Learner-side update on the device: one independent learner's policy-gradient
// step on the samples a rollout wrote (Sec. 3.3 "Independent Learning": one
// learner per policy, trained on its own agents' experience; App. C.2: the
// training workflow's optimize() with Adam and an entropy coefficient).
//
// For policy p with samples S_p (each (episode, step, environment, agent) whose
// combination gives that agent policy p; M = |S_p|):
//   L = -(1/M) sum_i [ (G_i - b) log pi(a_i | o_i) + beta H(pi(. | o_i)) ],
// G the discounted return-to-go within the episode, b the mean of G over S_p,
// H the entropy of the softmax over the 5 actions. The gradient by the chain
// rule: dL/dz_j = (1/M) [ (G - b)(pi_j - [j = a]) + beta pi_j (log pi_j + H) ],
// back through W3, the ReLUs (pre-activation > 0) and W2, W1.
// The PPO variant (clip > 0; Schulman et al. 2017's clipped surrogate, the
// same advantage A = G - b) replaces (G - b) log pi(a | o) by
// min(rho A, clip(rho, 1 - eps, 1 + eps) A), rho = pi(a | o) / mu(a | o) with mu
// the behavior policy whose logits the rollout recorded; the unclipped term
// carries the gradient A rho (pi_j - [j = a]) where it is the minimum (ties
// to it), the clipped one none.
//
// Kernels, in stream order:
//  1. learn_slots_kernel: the (combination, agent) slots acting with p, in
//     ascending order (one block).
//  2. learn_returns_kernel: G of every sample by the backward recursion
//     G_t = r_t + gamma G_{t+1}, one thread per (slot, episode, env), and
//     per-block fp64 sums of G.
//  3. learn_baseline_kernel: M and b = sum G / M in a fixed order (one block).
//  4. learn_grad_x3_kernel (learner_x3.cu; observations up to 20 wide) or
//     learn_grad_kernel (up to 32): persistent CTAs over tiles of 128 samples:
//     forward (fp32, hidden 64), logits, softmax, dL/dz, the backward pass, and
//     the weight gradients, summed over the CTA's tiles; each CTA writes its
//     partial gradient. learn_grad_kernel in fp32 FMAs (learner_fma.cuh):
//     each thread keeps a 4 x 4 block of dW2 and a few entries of the rest in
//     registers; the tile's activations are stored feature-major in shared
//     memory so that every product reads 16-byte vectors.
//  5. learn_reduce_kernel: the partials summed over CTAs in a fixed order into
//     the gradient (the malib_policy_desc layout) and the loss statistics.
// Deterministic: no atomics, every sum in a fixed order.
// Adam (Kingma and Ba): learn_adam_kernel, elementwise with bias correction.
#include <cmath>

#include "device_common.cuh"
#include "learner_fma.cuh"

namespace malib {

namespace {

// One block per policy b of the batch: the slots acting with it, ascending.
__global__ void __launch_bounds__(1024) learn_slots_kernel(LearnArgs a) {
    __shared__ int warp_n[32];
    __shared__ int base;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = blockIdx.x;
    const int total = a.n_pairs * a.n_agents;
    const int policy = a.pols[b];
    int32_t* slots = a.slots + (int64_t)b * total;
    if (tid == 0) base = 0;
    __syncthreads();
    for (int c0 = 0; c0 < total; c0 += blockDim.x) {
        const int i = c0 + tid;
        const int pid = i < total ? a.pairs[i] : -1;
        if (b == 0 && i < total && (pid < 0 || pid >= a.n_pol)) atomicOr(a.err, ERRBIT_BAD_PAIR);
        const bool mine = i < total && pid == policy;
        const unsigned m = __ballot_sync(0xffffffffu, mine);
        if (lane == 0) warp_n[warp] = __popc(m);
        __syncthreads();
        int before = base;
        for (int w = 0; w < warp; ++w) before += warp_n[w];
        if (mine) slots[before + __popc(m & ((1u << lane) - 1u))] = i;   // c * n_agents + k
        __syncthreads();
        if (tid == 0) {
            int n = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) n += warp_n[w];
            base += n;
        }
        __syncthreads();
    }
    if (tid == 0) a.n_slots[b] = base;
}

// The batch's sample and tile offsets (prefix sums over the policies; one thread).
__global__ void learn_plan_kernel(LearnArgs a) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int64_t per_slot = a.n_episodes * a.T * (a.n_envs / a.n_pairs);
    int64_t s = 0, t = 0;
    for (int b = 0; b < a.nb; ++b) {
        a.samp_off[b] = s;
        a.tile_off[b] = t;
        const int64_t M = (int64_t)a.n_slots[b] * per_slot;
        s += M;
        t += (M + 127) / 128;
    }
    a.samp_off[a.nb] = s;
    a.tile_off[a.nb] = t;
}

// Grid (blocks, nb): G of every sample of policy b by the backward recursion
// G_t = r_t + gamma G_{t+1}, one thread per (slot, episode, env), and per-block
// fp64 sums of G.
__global__ void __launch_bounds__(256) learn_returns_kernel(LearnArgs a) {
    __shared__ double red[256];
    const int b = blockIdx.y;
    const int epp = (int)(a.n_envs / a.n_pairs);
    const int64_t n_seq = (int64_t)a.n_slots[b] * a.n_episodes * epp;
    const int32_t* slots = a.slots + (int64_t)b * a.n_pairs * a.n_agents;
    float* G = a.G + a.samp_off[b];
    if ((int64_t)blockIdx.x * blockDim.x >= n_seq) {
        // no sequence of policy b reaches this block: its partial is 0, as the
        // reduction below would give, without the barriers
        if (threadIdx.x == 0) a.gsum[(int64_t)b * gridDim.x + blockIdx.x] = 0.0;
        return;
    }
    double sum = 0.0;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n_seq;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t slot = q / (a.n_episodes * epp);
        const int64_t rem = q - slot * a.n_episodes * epp;
        const int64_t e = rem / epp;
        const int r = (int)(rem - e * epp);
        const int ck = slots[slot];
        const int c = ck / a.n_agents, k = ck - c * a.n_agents;
        const int64_t env = (int64_t)c * epp + r;
        // backward over the episode, 8 steps at a time: the 8 rewards are loaded
        // together (the stores to G would otherwise hold each load behind the
        // previous step's store), then the same recurrence in the same order
        float g = 0.f;
        for (int t_hi = a.T; t_hi > 0; t_hi -= 8) {
            float rv[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int t = t_hi - 1 - u;
                rv[u] = t >= 0 ? a.reward[((e * a.T + t) * a.n_envs + env) * a.n_agents + k] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int t = t_hi - 1 - u;
                if (t >= 0) {
                    g = __fadd_rn(rv[u], __fmul_rn(a.gamma, g));
                    G[((slot * a.n_episodes + e) * a.T + t) * epp + r] = g;
                    sum += (double)g;
                }
            }
        }
    }
    red[threadIdx.x] = sum;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) a.gsum[(int64_t)b * gridDim.x + blockIdx.x] = red[0];
}

// One warp per policy b: lane l sums blocks l, l + 32, ... in order, then a
// fixed xor tree; M and the baseline b = sum G / M.
__global__ void learn_baseline_kernel(LearnArgs a, int n_blocks) {
    const int lane = threadIdx.x & 31;
    const int b = blockIdx.x;
    double s = 0.0;
    for (int k = lane; k < n_blocks; k += 32) s += a.gsum[(int64_t)b * n_blocks + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x != 0) return;
    const double M = (double)(a.samp_off[b + 1] - a.samp_off[b]);
    a.stats[4 * b] = M;
    a.stats[4 * b + 1] = M > 0 ? s / M : 0.0;
}

__global__ void __launch_bounds__(kThreads, 1) learn_grad_kernel(LearnArgs a) {
    extern __shared__ __align__(16) float sm[];
    learn_tiles_fma(a, sm, share_lo(a, blockIdx.x), share_lo(a, blockIdx.x + 1));
}

// Grid (blocks, nb): policy b's gradient as the sum of the partials of the CTAs
// whose tile share meets b's tiles; its loss and mean entropy. A block takes 64
// entries; four groups of threads sum a quarter of the CTAs each (eight loads in
// flight), combined in a fixed order. One thread per entry with the CTAs' shares
// recomputed by a division per step and its partial sums in local memory took 58
// us for 3 policies; this 17.
constexpr int kRedEntries = 64, kRedGroups = 4;

__global__ void __launch_bounds__(kRedEntries * kRedGroups) learn_reduce_kernel(LearnArgs a, int P) {
    __shared__ double part[kRedGroups][kRedEntries];
    __shared__ int range[2];
    const int b = blockIdx.y;
    const int64_t t_lo = a.tile_off[b], t_hi = a.tile_off[b + 1], n_t = a.tile_off[a.nb];
    if (threadIdx.x == 0) {
        int c_lo = 0, c_hi = 0;              // CTAs [c_lo, c_hi) hold partials of b
        if (t_hi > t_lo) {
            // c_lo: the first CTA whose share ends past t_lo; c_hi: the first CTA
            // after it whose share starts at or past t_hi (or the grid's end). Both
            // start from the shares' proportional position and step to the exact one.
            c_lo = (int)min((int64_t)a.grid - 1, t_lo * a.grid / n_t);
            while (c_lo > 0 && share_lo(a, c_lo) > t_lo) --c_lo;
            while (share_lo(a, c_lo + 1) <= t_lo) ++c_lo;
            c_hi = (int)max((int64_t)c_lo + 1, min((int64_t)a.grid, (t_hi * a.grid + n_t - 1) / n_t));
            while (c_hi > c_lo + 1 && share_lo(a, c_hi - 1) >= t_hi) --c_hi;
            while (c_hi < a.grid && share_lo(a, c_hi) < t_hi) ++c_hi;
        }
        range[0] = c_lo;
        range[1] = c_hi;
    }
    __syncthreads();
    const int e = threadIdx.x & (kRedEntries - 1), grp = threadIdx.x / kRedEntries;
    const int j = blockIdx.x * kRedEntries + e;
    const int n = range[1] - range[0], per = (n + kRedGroups - 1) / kRedGroups;
    const int c0 = range[0] + grp * per, c1 = min(range[1], c0 + per);
    // with fewer tiles than CTAs some shares are empty, and those CTAs wrote no partial
    const bool all = n_t >= a.grid;
    const float* src = a.gpart + (int64_t)b * a.grid * (P + 2) + j;
    double s = 0.0;
    if (j < P + 2)
        for (int c = c0; c < c1; c += 8) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                v[u] = c + u < c1 && (all || share_lo(a, c + u + 1) > share_lo(a, c + u))
                           ? __ldcg(src + (int64_t)(c + u) * (P + 2)) : 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) s += (double)v[u];
        }
    part[grp][e] = s;
    __syncthreads();
    if (grp != 0 || j >= P + 2) return;
#pragma unroll
    for (int q = 1; q < kRedGroups; ++q) s += part[q][e];
    double* st = a.stats + 4 * b;
    if (j < P) a.grad[(int64_t)b * P + j] = (float)s;
    else if (j == P) st[2] = st[0] > 0 ? s / st[0] : 0.0;   // loss: (1/M) sum of -(A log pi + beta H)
    else st[3] = st[0] > 0 ? s / st[0] : 0.0;              // mean entropy
}

__global__ void learn_adam_kernel(float* p, const float* g, float* m, float* v, int64_t n, float lr, float b1,
                                  float b2, float eps, float c1, float c2) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

}  // namespace

int64_t learn_param_count(int in) { return (int64_t)kH * in + kH + kH * kH + kH + kA * kH + kA; }

bool learn_supported(int in, int h1, int h2, int n_actions) {
    return in >= 1 && in <= kLearnMaxIn && h1 == kH && h2 == kH && n_actions == kA;
}

// Upper bounds of the work space (bytes, each region on a 256-byte boundary):
// the distinct policies of a batch own disjoint slots, so their samples together
// are at most every (episode, step, env, agent).
int64_t learn_work_bytes(int32_t nb, int32_t n_pairs, int32_t n_agents, int64_t n_envs, int64_t n_episodes,
                         int32_t T, int in, int grid, int ret_blocks) {
    auto up = [](int64_t b) { return (b + 255) / 256 * 256; };
    const int64_t slots = (int64_t)n_pairs * n_agents;
    const int64_t samples = slots * n_episodes * T * (n_envs / n_pairs);
    return up((int64_t)nb * 4) + up((int64_t)nb * 8) + up((int64_t)nb * slots * 4) + up((int64_t)nb * 4) +
           2 * up((int64_t)(nb + 1) * 8) + up(samples * 4) + up((int64_t)nb * ret_blocks * 8) +
           up((int64_t)nb * 4 * 8) + up((int64_t)nb * grid * (learn_param_count(in) + 2) * 4);
}

void learn_work_layout(uint8_t* base, int32_t nb, int32_t n_pairs, int32_t n_agents, int64_t n_envs,
                       int64_t n_episodes, int32_t T, int in, int grid, int ret_blocks, LearnArgs* a) {
    int64_t off = 0;
    auto take = [&](int64_t bytes) {
        uint8_t* p = base + off;
        off += (bytes + 255) / 256 * 256;
        return p;
    };
    const int64_t slots = (int64_t)n_pairs * n_agents;
    const int64_t samples = slots * n_episodes * T * (n_envs / n_pairs);
    a->pols = reinterpret_cast<int32_t*>(take((int64_t)nb * 4));
    a->pol_offs = reinterpret_cast<int64_t*>(take((int64_t)nb * 8));
    a->slots = reinterpret_cast<int32_t*>(take((int64_t)nb * slots * 4));
    a->n_slots = reinterpret_cast<int32_t*>(take((int64_t)nb * 4));
    a->samp_off = reinterpret_cast<int64_t*>(take((int64_t)(nb + 1) * 8));
    a->tile_off = reinterpret_cast<int64_t*>(take((int64_t)(nb + 1) * 8));
    a->G = reinterpret_cast<float*>(take(samples * 4));
    a->gsum = reinterpret_cast<double*>(take((int64_t)nb * ret_blocks * 8));
    a->stats = reinterpret_cast<double*>(take((int64_t)nb * 4 * 8));
    a->gpart = reinterpret_cast<float*>(take((int64_t)nb * grid * (learn_param_count(in) + 2) * 4));
    a->nb = nb;
    a->grid = grid;
}

static cudaError_t launch_learn_grad_f32(const LearnArgs& a, cudaStream_t s) {
    const cudaError_t err = cudaFuncSetAttribute(learn_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)kSBytes);
    if (err != cudaSuccess) return err;
    learn_grad_kernel<<<a.grid, kThreads, kSBytes, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_learn_pg(const LearnArgs& a, int ret_blocks, cudaStream_t s, cudaEvent_t g0, cudaEvent_t g1) {
    if (a.nb <= 0) return cudaSuccess;
    learn_slots_kernel<<<a.nb, 1024, 0, s>>>(a);
    learn_plan_kernel<<<1, 32, 0, s>>>(a);
    learn_returns_kernel<<<dim3(ret_blocks, a.nb), 256, 0, s>>>(a);
    learn_baseline_kernel<<<a.nb, 32, 0, s>>>(a, ret_blocks);
    if (g0) cudaEventRecord(g0, s);
    cudaError_t err = a.in <= kLearnX3MaxIn ? launch_learn_grad_x3(a, s) : launch_learn_grad_f32(a, s);
    if (err != cudaSuccess) return err;
    if (g1) cudaEventRecord(g1, s);
    const int P = (int)learn_param_count(a.in);
    learn_reduce_kernel<<<dim3((P + 2 + kRedEntries - 1) / kRedEntries, a.nb), kRedEntries * kRedGroups, 0, s>>>(a, P);
    return cudaGetLastError();
}

cudaError_t launch_learn_adam(float* p, const float* g, float* m, float* v, int64_t n, float lr, float b1,
                              float b2, float eps, float c1, float c2, int n_sm, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 4 * (int64_t)n_sm) blocks = 4 * (int64_t)n_sm;
    learn_adam_kernel<<<(unsigned)blocks, 256, 0, s>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

}  // namespace malib
