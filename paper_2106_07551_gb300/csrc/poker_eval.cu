// Payoff-table evaluation of Kuhn poker (Sec. 3.2 Evaluator, Sec. 4.2: each
// entry of the empirical payoff table is the Monte-Carlo mean over simulated
// hands of one policy combination): one thread per hand, tabular policies in
// registers. (Leduc: leduc_x3.cu for fp32 policies, leduc_tc.cu for bf16.)
#include "device_common.cuh"
#include "internal.h"
#include "eval_common.cuh"

namespace malib {

namespace {

// ---------------------------------------------------------------- Kuhn
// Cards J=0 < Q=1 < K=2, ante 1, one bet of 1. Infoset index card*2 + h with
// h = 1 when the seat faces a bet. Decision t uses counter (g, t, seat).
struct KuhnHand { int n; int act[3]; float p[3]; int payoff; };

// Entry idx of a 6-entry register table without dynamic indexing.
__device__ __forceinline__ float tab6(const float (&t)[6], int idx) {
    float v = t[0];
#pragma unroll
    for (int i = 1; i < 6; ++i) v = idx == i ? t[i] : v;
    return v;
}

// Seat 0 acts at decisions 0 and 2, seat 1 at decision 1, whatever the
// actions, so the three decision draws (g, t, seat) are known before the hand
// is played: they are drawn up front and the hand is resolved with selects, so
// the threads of a warp never run the generator on divergent paths. The third
// draw is used only after pass-bet.
__device__ __forceinline__ KuhnHand kuhn_play(const float (&t0)[6], const float (&t1)[6], uint64_t g,
                                              uint64_t seed) {
    const U4 d = draw(g, 0, kChance, seed);
    const int c0 = (int)pick(d.x, 3);
    const int j = (int)pick(d.y, 2);
    const int c1 = j + (j >= c0 ? 1 : 0);
    const int sd = c0 > c1 ? 1 : -1;
    const float u0 = u24(draw(g, 0, 0, seed).x);
    const float u1 = u24(draw(g, 1, 1, seed).x);
    const float u2 = u24(draw(g, 2, 0, seed).x);
    KuhnHand h;
    h.p[0] = tab6(t0, c0 * 2);                                  // seat 0 opens: P(bet)
    h.act[0] = u0 < h.p[0] ? 1 : 0;
    h.p[1] = tab6(t1, c1 * 2 + h.act[0]);                       // seat 1: P(bet) or P(call)
    h.act[1] = u1 < h.p[1] ? 1 : 0;
    h.p[2] = tab6(t0, c0 * 2 + 1);                              // seat 0 facing a bet: P(call)
    h.act[2] = u2 < h.p[2] ? 1 : 0;
    const bool third = h.act[0] == 0 && h.act[1] == 1;          // pass, bet
    h.n = third ? 3 : 2;
    h.payoff = h.act[0] ? (h.act[1] ? 2 * sd : 1)
                        : (h.act[1] ? (h.act[2] ? 2 * sd : -1) : sd);
    return h;
}

// A thread's share of a pair's hands: e0, e0 + stride, ...; adds the payoffs, their
// squares and the decisions to s1, s2, nd and records the first n_dump hands.
template <class Sum>
__device__ __forceinline__ void kuhn_hands(const EvalArgs& a, int pair, int p0, int p1, int64_t e0, int64_t stride,
                                           Sum& s1, Sum& s2, Sum& nd) {
    float t0[6], t1[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        t0[i] = a.arena[a.pol_offset[p0] + i];
        t1[i] = a.arena[a.pol_offset[p1] + i];
    }
    for (int64_t e = e0; e < a.n_episodes; e += stride) {
        const uint64_t g = (uint64_t)pair * (uint64_t)a.n_episodes + (uint64_t)e;
        const KuhnHand h = kuhn_play(t0, t1, g, a.seed);
        s1 += h.payoff;
        s2 += (Sum)(h.payoff * h.payoff);
        nd += h.n;
        if (e < a.n_dump) {
            const int64_t base = ((int64_t)pair * a.n_dump + e) * 3;
            for (int t = 0; t < 3; ++t) {
                const bool on = t < h.n;
                if (a.d_action) a.d_action[base + t] = on ? (uint8_t)h.act[t] : (uint8_t)255;
                if (a.d_reward) a.d_reward[base + t] = (t == h.n - 1) ? (float)h.payoff : 0.f;
                if (a.d_done) a.d_done[base + t] = (t >= h.n - 1) ? 1 : 0;
                if (a.d_logits) {
                    a.d_logits[(base + t) * 2] = on ? 1.f - h.p[t] : 0.f;
                    a.d_logits[(base + t) * 2 + 1] = on ? h.p[t] : 0.f;
                }
            }
        }
    }
}

// (four blocks on an SM: with 72 registers a thread three were, 992 pairs x 3,073 hands 47 -> 51 us)
__global__ void __launch_bounds__(256, 4) kuhn_eval_kernel(EvalArgs a) {
    const int pair = blockIdx.y;
    const int p0 = a.pairs[2 * pair], p1 = a.pairs[2 * pair + 1];
    const bool ok = pair_ok(a, p0, p1);
    if (!ok && threadIdx.x == 0 && blockIdx.x == 0) atomicOr(a.err, ERRBIT_BAD_PAIR);
    long long s1 = 0, s2 = 0, nd = 0;
    if (ok)
        kuhn_hands(a, pair, p0, p1, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x,
                   s1, s2, nd);
    block_add_sums(s1, s2, nd, a.acc + 2 * pair, a.n_dec);
    // the pair's last block to finish writes its table row (its sums are final:
    // every block fenced its additions before counting itself)
    if (a.fin_out && threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(a.work + pair, 1ull) == (unsigned long long)gridDim.x - 1ull) {
            __threadfence();
            const long long f1 = (long long)__ldcg(a.acc + 2 * pair);
            const long long f2 = (long long)__ldcg(a.acc + 2 * pair + 1);
            finalize_pair(f1, f2, a.n_episodes, a.fin_out + 4 * (int64_t)pair);
        }
    }
}

// The same with a cluster per pair: the CTAs' sums (32-bit: at most 3,072 hands a
// CTA) meet in the first one's shared memory, which writes the pair's row and
// its decision count. No accumulators in global memory to clear, add to and count
// blocks with: a table of 16 pairs x 10,000 hands is bound by latencies (the
// policies' loads, two hands a thread, the fp64 division and square root of the
// row), and took 14.0 us a call with them and takes 10.2 so.
constexpr int kKuhnMaxThreads = 768, kKuhnMaxCluster = 8;

__global__ void __launch_bounds__(kKuhnMaxThreads, 2) kuhn_cluster_kernel(EvalArgs a) {
    __shared__ int warp_sums[3][32], cta_sums[kKuhnMaxCluster][4];
    uint32_t rank, size;
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");        // this CTA runs
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(size));
    const int pair = (int)(blockIdx.x / size), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p0 = a.pairs[2 * pair], p1 = a.pairs[2 * pair + 1];
    const bool ok = pair_ok(a, p0, p1);
    int s[3] = {0, 0, 0};
    if (ok)
        kuhn_hands(a, pair, p0, p1, (int64_t)(rank * blockDim.x + threadIdx.x), (int64_t)(size * blockDim.x), s[0], s[1], s[2]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int v = __reduce_add_sync(0xffffffffu, s[i]);
        if (lane == 0) warp_sums[i][warp] = v;
    }
    asm volatile("barrier.cluster.wait;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int i = 0; i < 3; ++i)
            s[i] = __reduce_add_sync(0xffffffffu, lane < (int)(blockDim.x >> 5) ? warp_sums[i][lane] : 0);
        if (lane == 0) {
            uint32_t first;
            asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(first) : "r"(smem_u32(&cta_sums[rank][0])));
            asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(first), "r"(s[0]), "r"(s[1]), "r"(s[2]),
                         "r"(0)
                         : "memory");
        }
    }
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
    if (rank != 0 || warp != 0) return;
#pragma unroll
    for (int i = 0; i < 3; ++i) s[i] = __reduce_add_sync(0xffffffffu, lane < (int)size ? cta_sums[lane & (kKuhnMaxCluster - 1)][i] : 0);
    if (lane != 0) return;
    if (!ok) atomicOr(a.err, ERRBIT_BAD_PAIR);
    a.work[pair] = (unsigned long long)s[2];
    finalize_pair(s[0], s[1], a.n_episodes, a.fin_out + 4 * (int64_t)pair);
}

// CTAs per pair of kuhn_cluster_kernel; 0: kuhn_eval_kernel takes the call. A pair's
// cluster of at most 8 CTAs plays up to 3,072 hands a CTA; longer calls are bound by
// the generator and go over all the SMs. Both sides, in us a call (clusters, blocks):
// 1 x 2,000 hands 6.2, 9.2; 1 x 24,000 10.3, 10.3; 16 x 24,000 14.9, 16.5;
// 64 x 24,000 26.7, 28.8; 256 x 6,000 (2 CTAs a pair) 26.7, 28.8; 1,000 x 3,000 41, 44.
int kuhn_cluster(int32_t n_pairs, int64_t n_episodes, int n_sm) {
    int c = kKuhnMaxCluster;
    while (c > 1 && ((int64_t)n_pairs * c > 4 * (int64_t)n_sm || (int64_t)c * 64 > n_episodes)) c /= 2;
    return n_episodes <= (int64_t)c * kKuhnMaxThreads * 4 ? c : 0;
}

// Exact expected seat-0 payoff: the 6 deals, each 1/6, times the betting tree.
__global__ void kuhn_exact_kernel(EvalArgs a, double* out) {
    const int pair = blockIdx.x * blockDim.x + threadIdx.x;
    if (pair >= a.n_pairs) return;
    const int p0 = a.pairs[2 * pair], p1 = a.pairs[2 * pair + 1];
    double v = 0.0;
    if (!pair_ok(a, p0, p1)) {
        atomicOr(a.err, ERRBIT_BAD_PAIR);
        v = __longlong_as_double(0x7ff8000000000000ll);
    } else {
        const float* t0 = a.arena + a.pol_offset[p0];
        const float* t1 = a.arena + a.pol_offset[p1];
        for (int c0 = 0; c0 < 3; ++c0)
            for (int c1 = 0; c1 < 3; ++c1) {
                if (c0 == c1) continue;
                const double sd = c0 > c1 ? 1.0 : -1.0;
                const double pb = t0[c0 * 2], pc = t1[c1 * 2 + 1];
                const double qb = t1[c1 * 2], qc = t0[c0 * 2 + 1];
                const double bet = pc * 2.0 * sd + (1.0 - pc);
                const double chk = (1.0 - qb) * sd + qb * (qc * 2.0 * sd - (1.0 - qc));
                v += (pb * bet + (1.0 - pb) * chk) / 6.0;
            }
    }
    out[4 * pair + 0] = v;
    out[4 * pair + 1] = 0.0;
    out[4 * pair + 2] = 0.0;
    out[4 * pair + 3] = 0.0;
}

}  // namespace

bool kuhn_counts_itself(int32_t n_pairs, int64_t n_episodes, int n_sm) {
    return kuhn_cluster(n_pairs, n_episodes, n_sm) != 0;
}

cudaError_t launch_kuhn_eval(const EvalArgs& a, int n_sm, cudaStream_t s) {
    if (a.n_pairs == 0) return cudaSuccess;
    if (const int c = a.fin_out ? kuhn_cluster(a.n_pairs, a.n_episodes, n_sm) : 0) {
        const int64_t per = (a.n_episodes + c - 1) / c;                      // hands of a CTA
        // Few CTAs: as many threads as there are, one hand each (latency). More than two an
        // SM: blocks of 256, so that one's last steps (a row's fp64 division and root)
        // overlap others' hands; 40,000 pairs x 768 hands 705 -> 344 us, x 2,000 1,076 -> 817
        // (kuhn_eval_kernel 490, 911)
        const int64_t most = (int64_t)a.n_pairs * c >= 2 * (int64_t)n_sm ? 256 : kKuhnMaxThreads;
        const int64_t turns = (per + most - 1) / most;
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)c;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(a.n_pairs * c));
        cfg.blockDim = dim3((unsigned)(((per + turns - 1) / turns + 31) / 32 * 32));
        cfg.stream = s;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kuhn_cluster_kernel, a);
    }
    int64_t blocks_per_pair = (a.n_episodes + 255) / 256;
    const int64_t cap = max(1, (n_sm * 8) / max(1, a.n_pairs));
    if (blocks_per_pair > cap) blocks_per_pair = cap;
    if (blocks_per_pair > 65535) blocks_per_pair = 65535;
    dim3 grid((unsigned)blocks_per_pair, (unsigned)a.n_pairs);
    kuhn_eval_kernel<<<grid, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_kuhn_exact(const EvalArgs& a, double* out, cudaStream_t s) {
    if (a.n_pairs == 0) return cudaSuccess;
    kuhn_exact_kernel<<<(a.n_pairs + 127) / 128, 128, 0, s>>>(a, out);
    return cudaGetLastError();
}

}  // namespace malib
