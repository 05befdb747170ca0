// Payoff-table evaluation of Leduc hold'em with fp32 MLP policies on the tensor
// cores (Sec. 3.2 payoff table, Sec. 4.2 Monte-Carlo simulations per policy
// combination). fp32 operands are the exact sum of three bf16 parts, and a
// product is taken as its six largest part products, the smallest first, in
// fp32 accumulators (mlp_x3.cuh).
//
// Work units are (pair, segment of at most kMaxHands hands), claimed by the CTAs
// from a counter. A CTA plays a unit's hands all at once, in phases: in a phase
// every live hand whose acting seat is s makes one decision through seat s's
// policy; phases alternate between the seats. Policies are converted from the
// population's fp32 images: 128 wide only the acting seat's fits in shared memory,
// between the phases, 64 wide both seats' stay until a unit has others. Hands
// live in shared memory: a 27-bit state word each, and a list of hand numbers per
// acting seat. A phase takes its seat's list whole; hands that act next as the
// other seat join the other list, hands that act again as s a third one, which
// becomes the seat's list when the phase ends (a list is never written while it
// is read). So the call needs no device scratch but the sums and the claim
// counter.
//
// Two groups of eight warps take a phase's 128-row tiles in turn. Row r of a
// tile belongs to two threads (tensor-memory lane r; warps w and w + 4), one per
// half of the hidden units; the first of them holds the hand: it writes the
// observation, and from the logits draws the action, steps the hand and queues
// it. Per tile and group:
//   X (shared memory) x W1 -> D1; relu, split -> HID (tensor memory);
//   per 64 output units: HID x W2, + b2 -> D2; relu(D2) x W3 summed in the
//   threads; the next tile's observations are written while the last of these
//   products runs, and its layer 1 runs while this tile's actions are drawn.
// Tensor memory per group: HID 3 H / 2 columns, D2 64 (H = 128: 256, two groups
// fill the SM's 512). D1 is the last H of these columns; the parts of the first
// half of the hidden units go to HID's upper half (over their own D1 columns,
// read before), the others' to the lower half, so the two threads of a row need
// no barrier in between.
//
// Leduc observations are small exact numbers but for the two contributions / 13,
// so a row of X is 16 features (feature 15, constant 1, is a bias), the middle
// and low parts of those two, and ones for the biases: two K = 16 steps, five
// MMAs for layer 1.
//
// What bounds it (17-128-128-3): layer 2's 98 MMAs of N = 64 take 1,620 cycles per
// 64 output units, near the pipe's rate; on 64 x 65,536 hands the tensor pipe is
// 62 % busy (two groups overlap), and a phase costs about 4,000 cycles of policy
// conversion and 7,800 of its first tile's chain, which is all there is in small
// calls. 64 pairs x 65,536 hands: 12.24 ms with packed fp32 FMAs on 248 hands in
// flight per CTA (0.64 of the FMA pipe), now 2.64 ms; 18 pairs x 338 hands: 237
// us, now 74. 64 wide, many pairs of few hands are units' fixed costs: 4,900 pairs x
// 20 hands 757 us before, 740 with both policies resident (832 converting in every
// phase). The logits are off by 1.44e-7 of their norm against 64 bits (FMAs:
// 1.73e-7; H = 64: 1.02e-7, before 1.18e-7).
#include "device_common.cuh"
#include "eval_common.cuh"
#include "internal.h"
#include "leduc_env.cuh"
#include "mlp_x3.cuh"
#include "segments.h"

namespace malib {

namespace {

constexpr int kGroups = 2;
constexpr int kGroupThreads = 256;
constexpr int kThreads = kGroups * kGroupThreads;
constexpr int kMaxHands = 8192;            // hands of a unit
constexpr int kMaxDec = 8;
constexpr int kF9 = 9, kF10 = 10;          // the contributions' features

template <int H>
struct LeducX3 {
    static_assert(H == 64 || H == 128, "hidden widths built");
    using L = F32Layout<17, H, 3>;
    static constexpr int kOut = H / 64;                        // 64-unit products of layer 2
    static constexpr uint32_t kD2 = 3 * H / 2, kCols = kD2 + 64, kD1 = kCols - H;
    static_assert(kGroups * kCols <= 512, "tensor memory");
    // block b = 32 hidden units: its D1 columns, and its parts (16 columns each)
    __host__ __device__ static constexpr uint32_t d1_col(int b) { return kD1 + 32u * b; }
    __host__ __device__ static constexpr uint32_t hid_col(int b, int part) {
        return (b < H / 64 ? 3u * H / 4 + 48u * b : 48u * (b - H / 64)) + 16u * part;
    }
    // shared memory (bytes): the policies (64 wide, both seats'; 128 wide, the acting seat's)
    static constexpr int kPols = H == 64 ? 2 : 1;
    static constexpr uint32_t kLboX = 128 / 8 * 128, kLboW = H / 8 * 128;
    static constexpr uint32_t kStep = 2 * kLboW;               // one K = 16 step of a weight image
    static constexpr uint32_t kPart2 = (uint32_t)H * H * 2;
    static constexpr uint32_t kW2 = 0;                         // parts h, m, l
    static constexpr uint32_t kW1 = kW2 + 3 * kPart2;          // steps [wh 2][wm 2][wl 1]
    static constexpr uint32_t kB2 = kW1 + 5 * kStep;           // bias step [H][16]
    static constexpr uint32_t kW3 = kB2 + kStep;               // fp32 [3][H], b3
    static constexpr uint32_t kPolicy = (kW3 + (3 * H + 4) * 4 + 127) / 128 * 128;
    static constexpr uint32_t kOnes = kPols * kPolicy;         // [128][16] rows 1 1 1 0 ..
    static constexpr uint32_t kXBytes = 128 * 32 * 2;
    static constexpr uint32_t kX = kOnes + 128 * 16 * 2;
    static constexpr uint32_t kP = kX + kGroups * kXBytes;     // partial logits [group][128] float4
    static constexpr uint32_t kState = kP + kGroups * 128 * 16;
    static constexpr uint32_t kList = kState + kMaxHands * 4;  // uint16 [3][kMaxHands]
    static constexpr uint32_t kBytes = kList + 3 * kMaxHands * 2;
    static_assert(kBytes + 1280 <= 232448, "fits the 227 KB of shared memory of a CTA");

    // Converts a policy (fp32 image in global memory) into shared memory at sm; all
    // threads, the caller fences for the async proxy and synchronises.
    __device__ static void stage(uint8_t* sm, const float* __restrict__ src, int tid) {
        // W2: a thread converts 8 k of one row at a time (coalesced loads, 16-byte stores)
#pragma unroll 4
        for (int e = tid; e < H * (H / 8); e += kThreads) {
            const int j = e & (H - 1), c = e / H;
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __ldg(src + L::kW2T + (8 * c + i) * H + j);
            uint32_t w[3][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) split3(v[2 * i], v[2 * i + 1], w[0][i], w[1][i], w[2][i]);
#pragma unroll
            for (int q = 0; q < 3; ++q)
                *reinterpret_cast<uint4*>(sm + kW2 + q * kPart2 + tc::cm_offset(j, 8 * c, H, 2)) =
                    make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
        }
        // W1: images wh (chunks 0-3 of 8 elements), wm (4-7), wl (8, 9). A thread
        // converts 8 features of one row for all three, or the row's elements
        // 16 .. 31: the contributions against X's middle and low parts, and in wh
        // b1 and the constant feature against the ones.
        for (int e = tid; e < 3 * H; e += kThreads) {
            const int j = e & (H - 1), c = e / H;
            auto put = [&](int chunk, uint32_t x, uint32_t y, uint32_t z, uint32_t u) {
                *reinterpret_cast<uint4*>(sm + kW1 + tc::cm_offset(j, 8 * chunk, H, 2)) = make_uint4(x, y, z, u);
            };
            uint32_t w[3][4];
            if (c < 2) {
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = __ldg(src + L::kW1T + (8 * c + i == 15 ? 16 : 8 * c + i) * H + j);
#pragma unroll
                for (int i = 0; i < 4; ++i) split3(v[2 * i], v[2 * i + 1], w[0][i], w[1][i], w[2][i]);
                put(c, w[0][0], w[0][1], w[0][2], w[0][3]);
                put(4 + c, w[1][0], w[1][1], w[1][2], w[1][3]);
                put(8 + c, w[2][0], w[2][1], w[2][2], w[2][3]);
            } else {
                const float f9 = __ldg(src + L::kW1T + kF9 * H + j), f10 = __ldg(src + L::kW1T + kF10 * H + j);
                const float b = __ldg(src + L::kB1 + j), k = __ldg(src + L::kW1T + kLeducConstFeature * H + j);
                split3(f9, f10, w[0][0], w[1][0], w[2][0]);
                split3(b, k, w[0][1], w[1][1], w[2][1]);           // b1 in the low halves
                // 16 f9 17 f10 18 f9 19 f10, 20-22 b1's parts, 23-25 the constant's
                put(2, w[0][0], w[0][0], (w[0][1] & 0xffffu) | (w[1][1] << 16), (w[2][1] & 0xffffu) | (w[0][1] & 0xffff0000u));
                put(3, (w[1][1] >> 16) | (w[2][1] & 0xffff0000u), 0u, 0u, 0u);
                put(6, w[1][0], 0u, 0u, 0u);
                put(7, 0u, 0u, 0u, 0u);
            }
        }
        for (int j = tid; j < H; j += kThreads) {
            uint32_t w[3];
            split3(__ldg(src + L::kB2 + j), 0.f, w[0], w[1], w[2]);
            *reinterpret_cast<uint4*>(sm + kB2 + tc::cm_offset(j, 0, H, 2)) = make_uint4(w[0] | (w[1] << 16), w[2], 0u, 0u);
            *reinterpret_cast<uint4*>(sm + kB2 + tc::cm_offset(j, 8, H, 2)) = make_uint4(0u, 0u, 0u, 0u);
        }
        float* f = reinterpret_cast<float*>(sm + kW3);
        for (int i = tid; i < 3 * H + 3; i += kThreads) f[i] = __ldg(src + L::kW3 + i);   // W3, then b3
    }
    static_assert(L::kB3 == L::kW3 + 3 * H, "b3 follows W3");

    // Row r of X from the observation.
    __device__ static void put_row(uint8_t* X, int r, const float (&o)[17]) {
        uint32_t w[8], m, l, h910;
#pragma unroll
        for (int q = 0; q < 7; ++q) w[q] = tc::pack_bf16(o[2 * q], o[2 * q + 1]);
        w[7] = tc::pack_bf16(o[14], o[16]);
        split3(o[kF9], o[kF10], h910, m, l);
        *reinterpret_cast<uint4*>(X + tc::cm_offset(r, 0, 128, 2)) = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4*>(X + tc::cm_offset(r, 8, 128, 2)) = make_uint4(w[4], w[5], w[6], w[7]);
        *reinterpret_cast<uint4*>(X + tc::cm_offset(r, 16, 128, 2)) = make_uint4(m, l, 0x3f803f80u, 0x3f803f80u);
        *reinterpret_cast<uint4*>(X + tc::cm_offset(r, 24, 128, 2)) = make_uint4(0x3f803f80u, 0u, 0u, 0u);
    }
    __device__ static void zero_row(uint8_t* X, int r) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            *reinterpret_cast<uint4*>(X + tc::cm_offset(r, 8 * c, 128, 2)) = make_uint4(0u, 0u, 0u, 0u);
    }

    __device__ static void mma_ts(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t idesc, bool acc) {
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d),
            "r"(a_tmem), "l"(b), "r"(idesc), "r"((uint32_t)acc)
            : "memory");
    }

    // One elected thread: layer 1 into D1 (steps h wl, m wm, h wm, then m wh, l wh
    // and the biases, then h wh).
    __device__ static void issue1(uint32_t tb, uint32_t sm, uint32_t x, uint64_t* bar) {
        const uint32_t idesc = tc::instr_desc(128, H, 1);
        const uint64_t x0 = tc::smem_desc(x, kLboX, 128), x1 = x0 + ((2u * kLboX) >> 4);
        const uint64_t w = tc::smem_desc(sm + kW1, kLboW, 128);
        tc::mma_bf16(tb + kD1, x0, w + (uint64_t)4 * (kStep >> 4), idesc, false);
        tc::mma_bf16(tb + kD1, x1, w + (uint64_t)3 * (kStep >> 4), idesc, true);
        tc::mma_bf16(tb + kD1, x0, w + (uint64_t)2 * (kStep >> 4), idesc, true);
        tc::mma_bf16(tb + kD1, x1, w + (uint64_t)1 * (kStep >> 4), idesc, true);
        tc::mma_bf16(tb + kD1, x0, w, idesc, true);
        tc::mma_commit(bar);
    }

    // One elected thread: layer 2's output units 64 n .. into D2 (sm: the policy's).
    __device__ static void issue2(uint32_t tb, uint32_t sm, uint32_t ones, int n, uint64_t* bar) {
        const uint32_t idesc = tc::instr_desc(128, 64, 1);
        const uint64_t w = tc::smem_desc(sm + kW2 + 1024u * n, kLboW, 128);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const int px = q == 0 ? 2 : (q == 1 || q == 3) ? 1 : 0, pw = q == 2 ? 2 : (q == 1 || q == 4) ? 1 : 0;
            if (q == 5)
                tc::mma_bf16(tb + kD2, tc::smem_desc(ones, kLboX, 128),
                             tc::smem_desc(sm + kB2 + 1024u * n, kLboW, 128), idesc, true);
#pragma unroll
            for (int k = 0; k < H / 16; ++k)
                mma_ts(tb + kD2, tb + hid_col(k >> 1, px) + 8u * (k & 1),
                       w + (uint64_t)(pw * (kPart2 >> 4) + k * (kStep >> 4)), idesc, q + k != 0);
        }
        tc::mma_commit(bar);
    }

    // A warp: the hidden units of half `hh` of its rows, split into HID.
    __device__ static void hidden(uint32_t tb, uint32_t lane_q, int hh) {
#pragma unroll
        for (int c = 0; c < H / 64; ++c) {
            const int b = hh * (H / 64) + c;
            uint32_t v[32], w[3][16];
            tc::tmem_ld32x1(tb + lane_q + d1_col(b), v);
#pragma unroll
            for (int i = 0; i < 16; ++i)
                split3(relu_nan(__uint_as_float(v[2 * i])), relu_nan(__uint_as_float(v[2 * i + 1])), w[0][i], w[1][i],
                       w[2][i]);
#pragma unroll
            for (int q = 0; q < 3; ++q) tc::tmem_st16(tb + lane_q + hid_col(b, q), w[q]);
        }
        tc::tmem_wait_st();
    }

    // A warp: the 32 units 64 n + 32 hh .. of its rows added to the partial logits.
    __device__ static void logits(uint32_t tb, uint32_t lane_q, const uint8_t* sm, int n, int hh,
                                  unsigned long long (&acc)[3][2]) {
        const float* f = reinterpret_cast<const float*>(sm + kW3) + 64 * n + 32 * hh;
        uint32_t d[32];
        tc::tmem_ld32x1(tb + lane_q + kD2 + 32u * hh, d);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const unsigned long long z0 = f2_relu_nan(f2_pack(d[4 * i], d[4 * i + 1]));
            const unsigned long long z1 = f2_relu_nan(f2_pack(d[4 * i + 2], d[4 * i + 3]));
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(f + q * H + 4 * i);
                f2_fma(acc[q][0], z0, w.x);
                f2_fma(acc[q][1], z1, w.y);
            }
        }
    }
};

// A hand in one word: cards, round, raises, actions this round, actor,
// decisions so far, contributions.
__device__ __forceinline__ uint32_t pack_hand(const LeducHand& h, int t) {
    return (uint32_t)h.c0 | ((uint32_t)h.c1 << 3) | ((uint32_t)h.pub << 6) | ((uint32_t)h.round << 9) |
           ((uint32_t)h.raises << 10) | ((uint32_t)h.nact << 12) | ((uint32_t)h.actor << 14) | ((uint32_t)t << 15) |
           ((uint32_t)h.con0 << 19) | ((uint32_t)h.con1 << 23);
}
__device__ __forceinline__ void unpack_hand(uint32_t w, LeducHand& h, int& t) {
    h.c0 = (int)(w & 7u);
    h.c1 = (int)((w >> 3) & 7u);
    h.pub = (int)((w >> 6) & 7u);
    h.round = (int)((w >> 9) & 1u);
    h.raises = (int)((w >> 10) & 3u);
    h.nact = (int)((w >> 12) & 3u);
    h.actor = (int)((w >> 14) & 1u);
    t = (int)((w >> 15) & 15u);
    h.con0 = (int)((w >> 19) & 15u);
    h.con1 = (int)((w >> 23) & 15u);
    h.done = 0;
    h.payoff = 0;
}

// The logits of the hand w in fp32 FMAs (its operands' parts were not finite
// somewhere), a function of its own to keep its registers out of the tiles' loop.
template <int H>
__device__ __noinline__ float3 redo_logits(const float* __restrict__ img, uint32_t w) {
    LeducHand h;
    int t;
    unpack_hand(w, h, t);
    float o[17], z[3];
    leduc_obs(h, o);
    forward_fma<17, H, 3>(img, o, z);
    return make_float3(z[0], z[1], z[2]);
}

// Units of a call: n_seg segments of `per` hands per pair.
struct LeducUnits {
    int64_t n_seg, per, n_units;
};

// kDump: the call records its first n_dump hands of every pair (the recording
// code is compiled out of the other instance).
template <int H, bool kDump>
__global__ void __launch_bounds__(kThreads, 1) leduc_eval_x3_kernel(EvalArgs a, LeducUnits units) {
    using E = LeducX3<H>;
    using u64 = unsigned long long;
    extern __shared__ __align__(1024) uint8_t smem[];
    // [group][layer 1, layer 2's products]: complete. Each barrier is completed
    // again only after a barrier of the group that follows every thread's wait.
    __shared__ __align__(8) uint64_t bars[kGroups][1 + E::kOut];
    __shared__ uint32_t tmem_base;
    __shared__ uint32_t dead;              // a bounded wait expired: nobody waits any more
    __shared__ long long unit_s;
    __shared__ int len[3];                 // entries of the lists

    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int grp = warp >> 3, hh = (warp >> 2) & 1, r = (warp & 3) * 32 + lane;   // group, half, row
    const bool issuer = (warp & 7) == 0;
    if (tid == 0) {
        for (int i = 0; i < kGroups * (1 + E::kOut); ++i) mbar_init(&bars[0][0] + i, 1);
        dead = 0u;
    }
    if (tid < 128) {
        *reinterpret_cast<uint4*>(smem + E::kOnes + tc::cm_offset(tid, 0, 128, 2)) = make_uint4(0x3f803f80u, 0x3f80u, 0u, 0u);
        *reinterpret_cast<uint4*>(smem + E::kOnes + tc::cm_offset(tid, 8, 128, 2)) = make_uint4(0u, 0u, 0u, 0u);
    }
    if (warp == 0) {
        tc::tmem_alloc(&tmem_base, 512);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tb = tmem_base + (uint32_t)grp * E::kCols;
    const uint32_t lane_q = (uint32_t)(32 * (warp & 3)) << 16;
    uint8_t* X = smem + E::kX + (uint32_t)grp * E::kXBytes;
    float4* P = reinterpret_cast<float4*>(smem + E::kP) + 128 * grp;
    uint32_t* state = reinterpret_cast<uint32_t*>(smem + E::kState);
    uint16_t* lists = reinterpret_cast<uint16_t*>(smem + E::kList);
    uint64_t* bar = bars[grp];
    uint32_t phase_bit = 0;                // the group's tiles so far, mod 2
    auto is_dead = [&] { return *(volatile uint32_t*)&dead != 0u; };
    auto group_sync = [&] { asm volatile("bar.sync %0, 256;" ::"r"(grp + 1) : "memory"); };
    auto mma_wait = [&](int b) {
        if (!is_dead() && !mbar_wait_bounded(bar + b, phase_bit, kWaitLimitNs)) {
            *(volatile uint32_t*)&dead = 1u;
            atomicOr(a.err, ERRBIT_TIMEOUT);
            mbar_wait_bounded(bar + b, phase_bit, kWaitLimitNs);   // its MMAs in flight; none are issued after
        }
        tc::fence_after_sync();
    };
    long long nd = 0;                      // this thread's decisions
    int staged[2] = {-1, -1};              // the policies in shared memory

    while (true) {
        __syncthreads();                                     // unit_s and len are read by all
        if (tid == 0) {
            const long long u = (long long)atomicAdd(a.work, 1ull);
            unit_s = u < units.n_units ? u : -1;
            len[0] = len[1] = len[2] = 0;
        }
        __syncthreads();
        const long long unit = unit_s;
        if (unit < 0 || is_dead()) break;
        const int pair = (int)(unit / units.n_seg);
        const int64_t e_lo = (unit - (int64_t)pair * units.n_seg) * units.per;
        const int64_t e_hi = e_lo + units.per < a.n_episodes ? e_lo + units.per : a.n_episodes;
        const int n_hands = e_hi > e_lo ? (int)(e_hi - e_lo) : 0;
        const int pid[2] = {a.pairs[2 * pair], a.pairs[2 * pair + 1]};
        if (!pair_ok(a, pid[0], pid[1])) {
            if (tid == 0) atomicOr(a.err, ERRBIT_BAD_PAIR);
            continue;
        }
        if (n_hands == 0) continue;
        const uint64_t g0 = (uint64_t)pair * (uint64_t)a.n_episodes + (uint64_t)e_lo;
        int s1 = 0, s2 = 0;                                  // of at most 8,192 hands
        int mine[2] = {0, 1}, spare = 2;                     // the seats' lists, and the third
        bool first = true;                                   // the phase that deals the hands
        for (int s = 0;; s ^= 1) {
            // (every thread has passed the barrier that ended the last phase)
            const int n0 = first ? n_hands : len[mine[0]], n1 = len[mine[1]];
            const int n = s == 0 ? n0 : n1;
            if (n == 0) {
                if (n0 == 0 && n1 == 0) break;
                continue;
            }
            const int pol = pid[s], at = E::kPols == 2 ? s : 0;
            uint8_t* const ps = smem + (uint32_t)at * E::kPolicy;
            const uint32_t pu = smem_u32(ps);
            if (pol != (at ? staged[1] : staged[0])) {
                E::stage(ps, a.arena + a.pol_offset[pol], tid);
                (at ? staged[1] : staged[0]) = pol;
            }
            fence_proxy_async_smem();
            __syncthreads();                                 // also: everyone has read len
            const uint16_t* q_in = lists + mine[s] * kMaxHands;
            // hand (number in the unit) and state of the row's tile i; -1: no hand
            auto fetch = [&](int i, int& id, uint32_t& w) {
                const int idx = i * 128 + r;
                id = -1;
                w = 0u;
                if (idx >= n) return;
                if (first) {
                    id = idx;
                    LeducHand h;
                    leduc_deal(h, g0 + (uint64_t)idx, a.seed);
                    w = pack_hand(h, 0);
                } else {
                    id = (int)q_in[idx];
                    w = state[id];
                }
            };
            auto observe = [&](int id, uint32_t w) {
                if (id >= 0) {
                    LeducHand h;
                    int t;
                    unpack_hand(w, h, t);
                    float o[17];
                    leduc_obs(h, o);
                    E::put_row(X, r, o);
                } else {
                    E::zero_row(X, r);
                }
                fence_proxy_async_smem();
            };
            const int tiles = (n + 127) / 128;
            int id = -1, id_next = -1;
            uint32_t w = 0u, w_next = 0u;
            if (grp < tiles) {
                if (hh == 0) {
                    fetch(grp, id, w);
                    observe(id, w);
                }
                tc::fence_before_sync();
                group_sync();
                tc::fence_after_sync();
                if (issuer && !is_dead() && tc::elect_one()) E::issue1(tb, pu, smem_u32(X), bar);
                __syncwarp();
            }
            for (int i = grp; i < tiles; i += kGroups) {
                mma_wait(0);
                E::hidden(tb, lane_q, hh);
                u64 acc[3][2] = {};
                float u = 0.f;
#pragma unroll
                for (int p = 0; p < E::kOut; ++p) {
                    tc::fence_before_sync();
                    group_sync();                            // HID is written; D2 is read
                    tc::fence_after_sync();
                    if (issuer && !is_dead() && tc::elect_one()) E::issue2(tb, pu, smem_u32(smem + E::kOnes), p, bar + 1 + p);
                    __syncwarp();
                    if (hh == 0) {
                        if (p == 0 && id >= 0) u = u24(draw(g0 + (uint64_t)id, (w >> 15) & 15u, (uint32_t)s, a.seed).x);
                        if (p == E::kOut - 1 && i + kGroups < tiles) {
                            fetch(i + kGroups, id_next, w_next);   // layer 1 no longer reads the tile
                            observe(id_next, w_next);
                        }
                    }
                    mma_wait(1 + p);
                    E::logits(tb, lane_q, ps, p, hh, acc);
                }
                float lg[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const float2 v = f2_split(f2_add(acc[q][0], acc[q][1]));
                    lg[q] = __fadd_rn(v.x, v.y);
                }
                if (hh == 1) P[r] = make_float4(lg[0], lg[1], lg[2], 0.f);
                tc::fence_before_sync();
                group_sync();                                // partials and the next tile are written; D2 is read
                tc::fence_after_sync();
                phase_bit ^= 1u;
                if (i + kGroups < tiles) {
                    if (issuer && !is_dead() && tc::elect_one()) E::issue1(tb, pu, smem_u32(X), bar);
                    __syncwarp();
                }
                if (hh == 0) {
                    const float* b3 = reinterpret_cast<const float*>(ps + E::kW3) + 3 * H;
                    int next = -1;
                    if (id >= 0) {
                        const float4 o = P[r];
                        lg[0] = __fadd_rn(__fadd_rn(lg[0], o.x), b3[0]);
                        lg[1] = __fadd_rn(__fadd_rn(lg[1], o.y), b3[1]);
                        lg[2] = __fadd_rn(__fadd_rn(lg[2], o.z), b3[2]);
                        LeducHand h;
                        int t;
                        unpack_hand(w, h, t);
                        if (parts_failed(lg[0])) {
                            const float3 z = redo_logits<H>(a.arena + a.pol_offset[pol], w);
                            lg[0] = z.x; lg[1] = z.y; lg[2] = z.z;
                        }
                        const int act = sample_masked<3>(lg, leduc_legal(h), u);
                        const int64_t e = e_lo + id;
                        const bool rec = kDump && e < a.n_dump;
                        const int64_t rb = ((int64_t)pair * a.n_dump + e) * kMaxDec;
                        if (rec) {
                            if (a.d_obs) {
                                float ob[17];
                                leduc_obs(h, ob);
                                float* od = a.d_obs + (rb + t) * 20;
#pragma unroll
                                for (int q = 0; q < 17; ++q) od[q] = ob[q];
                                od[17] = 0.f; od[18] = 0.f; od[19] = 0.f;
                            }
                            if (a.d_logits) {
                                float* l = a.d_logits + (rb + t) * 3;
                                l[0] = lg[0]; l[1] = lg[1]; l[2] = lg[2];
                            }
                            if (a.d_action) a.d_action[rb + t] = (uint8_t)act;
                        }
                        leduc_apply(h, act);
                        if (rec) {
                            if (a.d_reward) a.d_reward[rb + t] = h.done ? (float)h.payoff : 0.f;
                            if (a.d_done) a.d_done[rb + t] = h.done ? 1 : 0;
                        }
                        ++t;
                        ++nd;
                        if (h.done) {
                            s1 += h.payoff;
                            s2 += h.payoff * h.payoff;
                            if (rec) {
                                for (int k = t; k < kMaxDec; ++k) {
                                    if (a.d_obs)
                                        for (int q = 0; q < 20; ++q) a.d_obs[(rb + k) * 20 + q] = 0.f;
                                    if (a.d_logits)
                                        for (int q = 0; q < 3; ++q) a.d_logits[(rb + k) * 3 + q] = 0.f;
                                    if (a.d_action) a.d_action[rb + k] = 255;
                                    if (a.d_reward) a.d_reward[rb + k] = 0.f;
                                    if (a.d_done) a.d_done[rb + k] = 1;
                                }
                            }
                        } else {
                            state[id] = pack_hand(h, t);
                            next = h.actor;
                        }
                    }
                    // the hand joins the list of its next acting seat (one
                    // shared-memory atomic per warp and list)
#pragma unroll
                    for (int again = 0; again < 2; ++again) {
                        const bool go = next >= 0 && (next == s) == (again == 1);
                        const unsigned m = __ballot_sync(0xffffffffu, go);
                        if (m == 0u) continue;
                        const int to = again ? spare : mine[s ^ 1];
                        const int leader = __ffs(m) - 1;
                        int base = 0;
                        if (lane == leader) base = atomicAdd(&len[to], __popc(m));
                        base = __shfl_sync(0xffffffffu, base, leader);
                        if (go) lists[to * kMaxHands + base + __popc(m & ((1u << lane) - 1u))] = (uint16_t)id;
                    }
                    id = id_next;
                    w = w_next;
                }
            }
            __syncthreads();                                 // the phase is over
            if (is_dead()) break;
            if (tid == 0) len[mine[s]] = 0;                  // (next written after a barrier)
            const int done_list = mine[s];
            mine[s] = spare;
            spare = done_list;
            first = false;
        }
        if (hh == 0) {                                       // (integers: exact in any order)
            s1 = __reduce_add_sync(0xffffffffu, s1);
            s2 = __reduce_add_sync(0xffffffffu, s2);
            if (lane == 0 && s2 != 0) {
                atomicAdd(a.acc + 2 * pair, (u64)(long long)s1);
                atomicAdd(a.acc + 2 * pair + 1, (u64)(long long)s2);
            }
        }
    }
    nd = warp_sum_ll(nd);
    if (lane == 0 && nd != 0) atomicAdd(a.n_dec, (u64)nd);
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem_base, 512);
}

// Segments per pair: the smallest estimated time. A unit's phase costs a policy
// conversion and the first tile's chain (4 us), and each pair of tiles a chain (6).
LeducUnits plan_units(int32_t n_pairs, int64_t n, int n_sm) {
    const int64_t lo = (n + kMaxHands - 1) / kMaxHands;
    int64_t hi = 2 * (int64_t)n_sm / n_pairs + 2;            // up to two waves of units
    if (hi < 4 * lo) hi = 4 * lo;
    if (hi > (n + 63) / 64) hi = (n + 63) / 64 > lo ? (n + 63) / 64 : lo;
    if (hi > lo + 4096) hi = lo + 4096;
    const int64_t seg = cheapest_segments(n_pairs, n, n_sm, lo, hi, 4.0, 6.0, 256.0);
    return LeducUnits{seg, (n + seg - 1) / seg, (int64_t)n_pairs * seg};
}

template <int H>
cudaError_t launch_h(const EvalArgs& a, int n_sm, cudaStream_t s) {
    auto kern = a.n_dump > 0 ? leduc_eval_x3_kernel<H, true> : leduc_eval_x3_kernel<H, false>;
    const cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LeducX3<H>::kBytes);
    if (err != cudaSuccess) return err;
    const LeducUnits u = plan_units(a.n_pairs, a.n_episodes, n_sm);
    const int64_t grid = u.n_units < n_sm ? u.n_units : n_sm;
    kern<<<(unsigned)grid, kThreads, LeducX3<H>::kBytes, s>>>(a, u);
    return cudaGetLastError();
}

}  // namespace

bool leduc_f32_supported(int hidden) { return hidden == 128 || hidden == 64; }

cudaError_t launch_leduc_eval_f32(const EvalArgs& a, int hidden, int n_sm, cudaStream_t s) {
    if (a.n_pairs == 0) return cudaSuccess;
    if (!a.work) return cudaErrorInvalidValue;               // the kernel claims units from a.work[0]
    if (hidden == 128) return launch_h<128>(a, n_sm, s);
    if (hidden == 64) return launch_h<64>(a, n_sm, s);
    return cudaErrorInvalidValue;
}

}  // namespace malib
