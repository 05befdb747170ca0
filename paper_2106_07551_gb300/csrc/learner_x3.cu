// The learner's gradient kernel on the tensor cores (learner.cu has the loss and
// the other kernels of the step): fp32 MLPs in-64-64-5 with in <= 20, every fp32
// operand as the exact sum of three bf16 parts, products in fp32 accumulators,
// the smallest first (mlp_x3.cuh). Per tile of 128 samples:
//   h1 = relu(X W1 + b1), h2 = relu(h1 W2 + b2)           (forward)
//   z, softmax, dL/dz                                       (fp32, in the threads)
//   d2 = (dz W3) [h2 > 0]                                   (fp32, in the threads)
//   d1 = (d2 W2) [h1 > 0]
//   dW2 += d2^T h1, dW1 | db1 += d1^T X, dW3 += h2^T dz      (sums over the samples)
//
// Eight warps; row r of a tile belongs to two threads (tensor-memory lane r;
// warps w and w + 4), one per half of the 64 hidden units. The rows' operands are
// stored as [sample][unit] tiles in the core-matrix layout: with the samples as
// rows they are K-major operands, and for the sums over samples the same bytes
// are MN-major operands (chunks of 8 units SBO apart, groups of 8 samples LBO
// apart), so nothing is transposed: X (forward A, gradient B), W2 (forward B, and
// MN-major for d2 W2), h1 (B), and [d2 d1], whose 128 units make one A operand
// (M = 128) of both layers' gradients. X carries three ones per row, against b1's
// parts in W1's image and as the columns that give db1 and db2. MN-major operands
// run at the K-major rate (N = 128: 65 cycles, 256: 129).
// dW3 is summed in fp32 FMAs while d2 W2 runs. Each tile's other gradients leave
// tensor memory for running fp32 sums in registers (thread = unit), so that no
// accumulator runs over more than 128 samples.
// X is double-buffered: the next tile's X and layer 1 go in behind this tile's
// sums. Its sample's index comes from counters that a tile advances by 128 (three
// divisions and a dependent load per sample took 900 cycles a tile).
//
// Of a tile's ~13,500 cycles the tensor core is busy 4,700: the phases of a tile
// depend on one another, and operands of a second tile (h1 and [d2 d1] in three
// parts: 144 KB) do not fit beside the first's. 16 warps with four threads a row
// were slower (the conversions are bound by issue, not by latency). Measured with
// 16 policies, 3.07 M samples of 18 features: 2.92 -> 1.08 ms (learn_grad_kernel ->
// this one); 3 policies, 105,000 samples of 8: 115 -> 56 us.
// Error against 64 bits, 105,000 samples: 2.0e-7 .. 2.8e-7 of the gradient's norm
// (learn_grad_kernel 2.2e-7 .. 3.3e-7).
#include "device_common.cuh"
#include "f32x2.cuh"
#include "learner_fma.cuh"
#include "mlp_x3.cuh"

namespace malib {

namespace {

template <int PP>                          // input width rounded up (zeros past the width)
struct LearnX3 {
    static constexpr int kOnes = 3 * PP;                       // X row: [h m l] of PP, three ones, zeros
    static constexpr int kK1 = (kOnes + 3 + 15) / 16 * 16;
    // K = 16 steps of X that W1's images [wh wh wh b1], [wm wm], [wl] reach
    static constexpr int kS1 = kK1 / 16, kS2 = (2 * PP + 15) / 16, kS3 = (PP + 15) / 16;
    static constexpr int kOnesStep = kOnes / 16, kOnesAt = kOnes % 16;
    static_assert(kOnesAt <= 13 && kK1 <= 64 && PP % 4 == 0, "layout");
    static constexpr uint32_t kLboX = 128 / 8 * 128, kLboW = kH / 8 * 128, kStepW = 2 * kLboW;
    static constexpr uint32_t kPart2 = kH * kH * 2;
    // shared memory (bytes)
    static constexpr uint32_t kW1 = 0;
    static constexpr uint32_t kW2 = kW1 + (kS1 + kS2 + kS3) * kStepW;
    static constexpr uint32_t kB2 = kW2 + 3 * kPart2;          // bias step [64][16]
    static constexpr uint32_t kW3 = kB2 + kStepW;              // fp32 W3 [5][64], b3
    // [sample][X, even tiles | three parts of h1 | X, odd tiles]: even tiles store h1
    // as [h m l] and odd ones as [l m h], so that X and the first parts are always
    // one B operand of the sums
    static constexpr uint32_t kXBytes = 128u * kK1 * 2, kPartH1 = 128u * kH * 2;
    static constexpr uint32_t kX0 = kW3 + 1408;
    static constexpr uint32_t kH1 = kX0 + kXBytes;
    static constexpr uint32_t kX1 = kH1 + 3 * kPartH1;
    static constexpr uint32_t kDU = kX1 + kXBytes;             // 3 parts x [128][d2 64 | d1 64]
    static constexpr uint32_t kPartDU = 128u * 128 * 2;
    static constexpr uint32_t kBytes = kDU + 3 * kPartDU;
    static_assert(kBytes + 1024 <= 232448, "fits the 227 KB of shared memory of a CTA");
    // Until d1 is known its three 16 KB blocks hold, in fp32: h2, 48 rows of 68 a
    // block; past them the partial logits [5][128] of half 0 and half 1 (blocks 0
    // and 1) and dz [128][8] (block 2)
    static constexpr uint32_t kRow = 272, kRows = 48;
    __host__ __device__ static constexpr uint32_t h2_at(int row) {
        return kDU + (uint32_t)row / kRows * kPartDU + kPartDU / 2 + (uint32_t)row % kRows * kRow;
    }
    __host__ __device__ static constexpr uint32_t p_at(int half) {
        return kDU + (uint32_t)half * kPartDU + kPartDU / 2 + kRows * kRow;
    }
    static constexpr uint32_t kDZ = kDU + 2 * kPartDU + kPartDU / 2 + (128 - 2 * kRows) * kRow;
    static_assert(kRows * kRow + kA * 128 * 4 <= kPartDU / 2 && kDZ + 4096 <= kBytes, "fits d1's blocks");
    // tensor memory columns: HID (parts of 64 units), D (64), the sums (in the
    // order of their B operands)
    static constexpr uint32_t kHid = 0, kD = 96, kGX0 = 160, kG2 = kGX0 + kK1, kGX1 = kG2 + 192;
    static_assert(kGX1 + kK1 <= 512 && 192 + kK1 <= 256, "tensor memory, N of an MMA");
    static constexpr int kMnA = 1 << 15, kMnB = 1 << 16;       // instruction descriptor: MN-major operands

    __host__ __device__ static constexpr uint32_t hid_col(int b, int part) { return kHid + (b == 0 ? 48u : 0u) + 16u * part; }
    __host__ __device__ static constexpr int part_x(int q) { return q == 0 ? 2 : (q == 1 || q == 3) ? 1 : 0; }
    __host__ __device__ static constexpr int part_w(int q) { return q == 2 ? 2 : (q == 1 || q == 4) ? 1 : 0; }

    __device__ static void mma_ts(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t idesc, bool acc) {
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d),
            "r"(a_tmem), "l"(b), "r"(idesc), "r"((uint32_t)acc)
            : "memory");
    }
    // MN-major operand at `addr`: chunks of 8 units `sbo` apart, groups of 8 K rows 128 B apart
    __device__ static uint64_t mn_desc(uint32_t addr, uint32_t sbo) { return tc::smem_desc(addr, 128, sbo); }

    // Converts policy pol (F32Layout: W1T [in][64], b1, W2T [64][64], b2, W3, b3)
    // into shared memory; all threads, the caller fences and synchronises.
    __device__ static void stage(uint8_t* sm, const float* __restrict__ pol, int in, int tid) {
        const float *W1T = pol, *b1 = W1T + in * kH, *W2T = b1 + kH, *b2 = W2T + kH * kH, *W3 = b2 + kH;
        for (int e = tid; e < kH * 2 * (kS1 + kS2 + kS3); e += kThreads) {
            const int j = e & (kH - 1), c = e / kH;
            const int img = c < 2 * kS1 ? 0 : c < 2 * (kS1 + kS2) ? 1 : 2;
            const int k0 = 8 * (c - (img == 0 ? 0 : img == 1 ? 2 * kS1 : 2 * (kS1 + kS2)));
            float v[8];
            int part[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int k = k0 + i, f = k % PP;
                const bool feat = k < (3 - img) * PP && f < in, bias = img == 0 && k >= kOnes && k < kOnes + 3;
                part[i] = feat ? img : bias ? k - kOnes : 3;
                v[i] = __ldg(feat ? W1T + f * kH + j : b1 + j);
            }
            uint32_t out[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t w[3];
                split3(v[2 * i], v[2 * i + 1], w[0], w[1], w[2]);
                const int p0 = part[2 * i], p1 = part[2 * i + 1];
                out[i] = ((p0 == 0 ? w[0] : p0 == 1 ? w[1] : p0 == 2 ? w[2] : 0u) & 0xffffu) |
                         ((p1 == 0 ? w[0] : p1 == 1 ? w[1] : p1 == 2 ? w[2] : 0u) & 0xffff0000u);
            }
            *reinterpret_cast<uint4*>(sm + kW1 + tc::cm_offset(j, 8 * c, kH, 2)) = make_uint4(out[0], out[1], out[2], out[3]);
        }
        for (int e = tid; e < kH * kH / 8; e += kThreads) {
            const int j = e & (kH - 1), c = e / kH;
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __ldg(W2T + (8 * c + i) * kH + j);
            uint32_t w[3][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) split3(v[2 * i], v[2 * i + 1], w[0][i], w[1][i], w[2][i]);
#pragma unroll
            for (int q = 0; q < 3; ++q)
                *reinterpret_cast<uint4*>(sm + kW2 + q * kPart2 + tc::cm_offset(j, 8 * c, kH, 2)) =
                    make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
        }
        for (int j = tid; j < kH; j += kThreads) {
            uint32_t w[3];
            split3(__ldg(b2 + j), 0.f, w[0], w[1], w[2]);
            for (int k = 0; k < 16; ++k)
                *reinterpret_cast<uint16_t*>(sm + kB2 + tc::cm_offset(j, k, kH, 2)) =
                    (uint16_t)(k == kOnesAt ? w[0] : k == kOnesAt + 1 ? w[1] : k == kOnesAt + 2 ? w[2] : 0u);
        }
        float* f = reinterpret_cast<float*>(sm + kW3);
        for (int i = tid; i < kA * kH + kA; i += kThreads) f[i] = __ldg(W3 + i);   // W3, then b3
    }

    // Row r of X: [h m l] of o, three ones, zeros.
    __device__ static void put_row(uint8_t* X, int r, const float (&o)[PP]) {
        uint32_t w[3][PP / 2];
#pragma unroll
        for (int p = 0; p < PP / 2; ++p) split3(o[2 * p], o[2 * p + 1], w[0][p], w[1][p], w[2][p]);
#pragma unroll
        for (int c = 0; c < kK1 / 8; ++c) {
            uint32_t v[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int i = 4 * c + h, q = i / (PP / 2), p = i % (PP / 2);      // word i: part q, pair p
                v[h] = q < 3 ? w[q < 3 ? q : 0][p] : i == kOnes / 2 ? 0x3f803f80u : i == kOnes / 2 + 1 ? 0x3f80u : 0u;
            }
            *reinterpret_cast<uint4*>(X + tc::cm_offset(r, 8 * c, 128, 2)) = make_uint4(v[0], v[1], v[2], v[3]);
        }
    }

    // 32 values of row r (units u0 ..), split: to HID (block b) and to the [sample][unit]
    // tile at t0, whose parts are `stride` bytes apart.
    __device__ static void spread(const float (&v)[32], uint32_t tmem, int b, bool to_hid, uint8_t* t0, int stride,
                                  int r, int u0) {
        uint32_t w[3][16];
#pragma unroll
        for (int i = 0; i < 16; ++i) split3(v[2 * i], v[2 * i + 1], w[0][i], w[1][i], w[2][i]);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            if (to_hid) tc::tmem_st16(tmem + hid_col(b, q), w[q]);
            uint8_t* t = t0 + q * stride;
#pragma unroll
            for (int c = 0; c < 4; ++c)
                *reinterpret_cast<uint4*>(t + tc::cm_offset(r, u0 + 8 * c, 128, 2)) =
                    make_uint4(w[q][4 * c], w[q][4 * c + 1], w[q][4 * c + 2], w[q][4 * c + 3]);
        }
    }

    // ---- MMA batches, one elected thread each
    __device__ static void issue_l1(uint32_t tb, uint32_t sm, int odd, uint64_t* bar) {
        const uint32_t id = tc::instr_desc(128, kH, 1);
        const uint64_t x = tc::smem_desc(sm + (odd ? kX1 : kX0), kLboX, 128), w = tc::smem_desc(sm + kW1, kLboW, 128);
        auto step = [&](int k, int i, bool acc) {
            tc::mma_bf16(tb + kD, x + (uint64_t)k * ((2u * kLboX) >> 4), w + (uint64_t)i * (kStepW >> 4), id, acc);
        };
#pragma unroll
        for (int k = 0; k < kS3; ++k) step(k, kS1 + kS2 + k, k != 0);
#pragma unroll
        for (int k = kS2 - 1; k >= 0; --k) step(k, kS1 + k, true);
#pragma unroll
        for (int k = kS1 - 1; k >= 0; --k) step(k, k, true);
        tc::mma_commit(bar);
    }
    __device__ static void issue_l2(uint32_t tb, uint32_t sm, int odd, uint64_t* bar) {
        const uint32_t id = tc::instr_desc(128, kH, 1);
        const uint64_t w = tc::smem_desc(sm + kW2, kLboW, 128);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            if (q == 5)
                tc::mma_bf16(tb + kD, tc::smem_desc(sm + (odd ? kX1 : kX0) + kOnesStep * 2 * kLboX, kLboX, 128),
                             tc::smem_desc(sm + kB2, kLboW, 128), id, true);
#pragma unroll
            for (int k = 0; k < kH / 16; ++k)
                mma_ts(tb + kD, tb + hid_col(k >> 1, part_x(q)) + 8u * (k & 1),
                       w + (uint64_t)(part_w(q) * (kPart2 >> 4) + k * (kStepW >> 4)), id, q + k != 0);
        }
        tc::mma_commit(bar);
    }
    // d2 W2: the same image of W2, MN-major (units k of layer 1 as N, units j as K)
    __device__ static void issue_d1(uint32_t tb, uint32_t sm, uint64_t* bar) {
        const uint32_t id = tc::instr_desc(128, kH, 1) | kMnB;
        const uint64_t w = mn_desc(sm + kW2, kLboW);
#pragma unroll
        for (int q = 0; q < 6; ++q)
#pragma unroll
            for (int k = 0; k < kH / 16; ++k)
                mma_ts(tb + kD, tb + hid_col(k >> 1, part_x(q)) + 8u * (k & 1),
                       w + (uint64_t)(part_w(q) * (kPart2 >> 4) + k * (256u >> 4)), id, q + k != 0);
        tc::mma_commit(bar);
    }
    // [d2 d1]^T [X h1]: the part l of d meets X and h1's part h (its first step all
    // of them: it sets the columns), m also h1's m, h all three
    template <bool kOdd>
    __device__ static void issue_grads(uint32_t tb, uint32_t sm, uint64_t* bar) {
        const uint64_t du = mn_desc(sm + kDU, 2048), x0 = mn_desc(sm + kX0, 2048);
#pragma unroll
        for (int pa = 2; pa >= 0; --pa)
#pragma unroll
            for (int k = 0; k < kTile / 16; ++k) {
                const bool first = pa == 2 && k == 0;
                const int parts = first ? 3 : 3 - pa, skip = kOdd ? kK1 + 64 * (3 - parts) : 0;   // columns
                tc::mma_bf16(tb + kGX0 + skip, du + (uint64_t)(pa * (kPartDU >> 4) + k * 16),
                             x0 + (uint64_t)((skip / 8 * 2048 >> 4) + k * 16),
                             tc::instr_desc(128, kK1 + 64 * parts, 1) | kMnA | kMnB, !first);
            }
        tc::mma_commit(bar);
    }
};

// Which of the row's pre-activations marked in `near` (units u0 + bit; the row is
// lane's, of the 32 from r0) are positive in the fp32 FMA chain that
// learn_grad_kernel takes (bias first, inputs ascending). The whole warp works on
// each lane's marks in turn; X holds the rows' observations as their parts.
template <int PP>
__device__ __noinline__ uint32_t chain_signs(const float* __restrict__ pol, int in, const uint8_t* X, int r0, int u0,
                                             int layer, uint32_t near) {
    const int lane = threadIdx.x & 31;
    const float *W1T = pol, *b1 = W1T + in * kH, *W2T = b1 + kH, *b2 = W2T + kH * kH;
    uint32_t out = 0u;
    for (uint32_t who = __ballot_sync(0xffffffffu, near != 0u); who != 0u; who &= who - 1) {
        const int src = __ffs(who) - 1;
        auto x = [&](int f) {
            float v = 0.f;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                v += __uint_as_float((uint32_t)*reinterpret_cast<const uint16_t*>(X + tc::cm_offset(r0 + src, q * PP + f, 128, 2)) << 16);
            return v;
        };
        auto layer1 = [&](int u) {
            float z = __ldg(b1 + u);
            for (int f = 0; f < in; ++f) z = fmaf(x(f), __ldg(W1T + f * kH + u), z);
            return z;
        };
        float h0 = 0.f, h1 = 0.f;                        // layer 2's inputs lane, lane + 32
        if (layer == 2) {
            h0 = fmaxf(layer1(lane), 0.f);
            h1 = fmaxf(layer1(lane + 32), 0.f);
        }
        uint32_t got = 0u;
        for (uint32_t m = __shfl_sync(0xffffffffu, near, src); m != 0u; m &= m - 1) {
            const int i = __ffs(m) - 1, j = u0 + i;
            float z;
            if (layer == 2) {
                const float w0 = __ldg(W2T + lane * kH + j), w1 = __ldg(W2T + (lane + 32) * kH + j);
                z = __ldg(b2 + j);
                for (int k = 0; k < 32; ++k) z = fmaf(__shfl_sync(0xffffffffu, h0, k), __shfl_sync(0xffffffffu, w0, k), z);
                for (int k = 0; k < 32; ++k) z = fmaf(__shfl_sync(0xffffffffu, h1, k), __shfl_sync(0xffffffffu, w1, k), z);
            } else {
                z = layer1(j);
            }
            got |= z > 0.f ? 1u << i : 0u;
        }
        if (lane == src) out = got;
    }
    return out;
}

// Tiles once more in fp32 FMAs, from the CTA's first policy whose partial is not
// finite to its last one: an infinity, a NaN or a value beyond bf16's range
// (3.3962e38) among the weights, the activations, the observations or the gradients
// has no parts (mlp_x3.cuh), and what comes out then shows it (the ReLUs keep a NaN,
// which reaches the row's logits and with them db3) but need not be what IEEE
// arithmetic gives. Called at the kernel's end, where nothing is live: from flush
// it cost the tiles 1 to 2 %.
__device__ __noinline__ void redo_tiles(LearnArgs a, float* sm, int64_t lo, int64_t hi) { learn_tiles_fma(a, sm, lo, hi); }

template <int PP>
__global__ void __launch_bounds__(kThreads, 1) learn_grad_x3_kernel(LearnArgs a) {
    using E = LearnX3<PP>;
    using u64 = unsigned long long;
    extern __shared__ __align__(1024) uint8_t sm[];
    // layer 1, layer 2, d1, the sums: complete (once a tile each, and again only
    // after a CTA barrier that follows every thread's wait)
    __shared__ __align__(8) uint64_t bars[4];
    __shared__ uint32_t tmem_base, dead;
    __shared__ int step[4];                              // 128 samples as (env, step, episode, slot)
    __shared__ int64_t redo[2];                          // tiles for redo_tiles (none: empty)
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int qt = warp & 3, hh = warp >> 2, r = 32 * qt + lane;      // lane quarter, half, row
    const int in = a.in;
    const int epp = (int)(a.n_envs / a.n_pairs);
    const int P = kH * in + kH + kH * kH + kH + kA * kH + kA;
    const int64_t lo = share_lo(a, blockIdx.x), hi = share_lo(a, blockIdx.x + 1);
    if (lo >= hi) return;                                // an empty share writes no partial
    if (tid == 0) {
        for (int i = 0; i < 4; ++i) mbar_init(&bars[i], 1);
        dead = 0u;
        redo[0] = redo[1] = 0;
        int q = kTile / epp;
        step[0] = kTile - q * epp;
        step[1] = q % a.T;
        q /= a.T;
        step[2] = (int)(q % a.n_episodes);
        step[3] = (int)(q / a.n_episodes);
    }
    if (warp == 0) {
        tc::tmem_alloc(&tmem_base, 512);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tb = tmem_base, lane_q = (uint32_t)(32 * qt) << 16, tq = tb + lane_q;
    const uint32_t smu = smem_u32(sm);
    const float* W3s = reinterpret_cast<const float*>(sm + E::kW3);
    float* const Ps = reinterpret_cast<float*>(sm + E::p_at(hh));
    const float* const Po = reinterpret_cast<const float*>(sm + E::p_at(hh ^ 1));
    uint32_t parity = 0;
    auto is_dead = [&] { return *(volatile uint32_t*)&dead != 0u; };
    auto mma_wait = [&](int i) {
        if (!is_dead() && !mbar_wait_bounded(&bars[i], parity, kWaitLimitNs)) {
            *(volatile uint32_t*)&dead = 1u;
            atomicOr(a.err, ERRBIT_TIMEOUT);
            mbar_wait_bounded(&bars[i], parity, kWaitLimitNs);   // its MMAs in flight; none are issued after
        }
        __syncwarp();
        tc::fence_after_sync();
    };
    // every thread's shared and tensor memory accesses so far, before what follows
    auto hand_over = [&] {
        fence_proxy_async_smem();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
    };
    auto issues = [&] { return warp == 0 && !is_dead() && tc::elect_one(); };

    // running sums. Rows 0 .. 63 (d2 units): dW2 of the thread's 32 columns and db2;
    // rows 64 .. (d1 units): the thread's X columns. dW3 of units 2 lane, 2 lane + 1
    // over the tiles' samples 16 warp .. + 15, db3 of the thread's row
    float gacc[32] = {}, gb2 = 0.f, gb3[kA] = {}, lsum = 0.f, hsum = 0.f;
    u64 gw3[kA] = {};
    int b = -1;
    int64_t M = 0, t0 = 0;
    float invM = 0.f, base = 0.f;
    const int32_t* slots = nullptr;
    const float* Gb = nullptr;
    constexpr int kChunks = E::kK1 / 16;                 // 16-column chunks of X's block; this thread's: hh, hh + 2
    auto flush = [&] {
        float* out = a.gpart + ((int64_t)b * a.grid + blockIdx.x) * (P + 2);
        bool finite = true;
        auto put = [&](int e, float v) {
            out[e] = v;
            finite = finite && fabsf(v) <= 3.402823466e38f;
        };
        const int oW2 = kH * in + kH, oW3 = oW2 + kH * kH + kH;
        float* S = reinterpret_cast<float*>(sm + E::kH1);            // [64][kK1] of d1^T X
        float* R = reinterpret_cast<float*>(sm + E::kDU);            // [7][128]
        float* R3 = R + 7 * 128;                                      // [8][5][64]
        if (qt < 2) {
#pragma unroll
            for (int i = 0; i < 32; ++i) put(oW2 + r * kH + 32 * hh + i, gacc[i]);
            if (hh == 0) put(oW2 + kH * kH + r, gb2);
        } else {
#pragma unroll
            for (int c = 0; c < (kChunks + 1) / 2; ++c)
                if (2 * c + hh < kChunks)
#pragma unroll
                    for (int i = 0; i < 16; ++i) S[(r - 64) * E::kK1 + 16 * (2 * c + hh) + i] = gacc[16 * c + i];
        }
        if (hh == 0) {
#pragma unroll
            for (int c = 0; c < kA; ++c) R[c * 128 + r] = gb3[c];
            R[5 * 128 + r] = lsum;
            R[6 * 128 + r] = hsum;
        }
#pragma unroll
        for (int c = 0; c < kA; ++c) *reinterpret_cast<u64*>(R3 + (warp * kA + c) * kH + 2 * lane) = gw3[c];
        __syncthreads();
        for (int e = tid; e < kH * in; e += kThreads) {
            const int j = e / in, f = e - j * in;
            const float* s = S + j * E::kK1;
            put(e, (s[2 * PP + f] + s[PP + f]) + s[f]);
        }
        if (tid < kH) put(kH * in + tid, S[tid * E::kK1 + E::kOnes]);
        for (int e = tid; e < kA * kH; e += kThreads) {
            float v[8];
#pragma unroll
            for (int g = 0; g < 8; ++g) v[g] = R3[g * kA * kH + e];
            put(oW3 + e, ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7])));
        }
        if (warp < 7) {
            float s = (R[warp * 128 + lane] + R[warp * 128 + 32 + lane]) + (R[warp * 128 + 64 + lane] + R[warp * 128 + 96 + lane]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) put(warp < 5 ? oW3 + kA * kH + warp : P + warp - 5, s);
        }
        if (__syncthreads_or(!finite) && tid == 0) {
            redo[0] = redo[1] > redo[0] ? redo[0] : max(lo, a.tile_off[b]);
            redo[1] = min(hi, a.tile_off[b + 1]);
        }
    };
    // this row's sample of a tile of policy b (both threads the action, return and
    // behavior logits; the first the observation): the loads only
    float4 o[PP / 4];
    float ret = 0.f, bl[kA];
    int act = 0;
    bool valid = false;
    const bool vec = ((uintptr_t)a.obs & 15u) == 0;
    // The row's sample of the next tile in the policy's order (slot, episode, step,
    // env): counters that a tile advances by 128 (its digits in step[]) without a
    // division, the slot's (combination, agent), and the trajectory index (-1: none)
    int sr = 0, st = 0, sslot = 0, sc = 0, ska = 0;
    int64_t se = 0, ix = -1;
    auto locate = [&](int64_t tile, bool restart) {
        const int64_t s = (tile - t0) * kTile + r;
        int was = sslot;
        if (restart) {
            int64_t q = s / epp;
            sr = (int)(s - q * epp);
            st = (int)(q % a.T);
            q /= a.T;
            sslot = (int)(q / a.n_episodes);
            se = q - sslot * a.n_episodes;
            was = -1;
        } else {
            sr += step[0];
            int c = sr >= epp ? 1 : 0;
            sr -= c ? epp : 0;
            st += step[1] + c;
            c = st >= a.T ? 1 : 0;
            st -= c ? a.T : 0;
            se += step[2] + c;
            c = se >= a.n_episodes ? 1 : 0;
            se -= c ? a.n_episodes : 0;
            sslot += step[3] + c;
        }
        ix = -1;
        if (s >= M) return;
        if (sslot != was) {
            const int ck = slots[sslot];
            sc = ck / a.n_agents;
            ska = ck - sc * a.n_agents;
        }
        ix = ((se * a.T + st) * a.n_envs + (int64_t)sc * epp + sr) * a.n_agents + ska;
    };
    auto gather = [&](int64_t tile) {
        valid = ix >= 0;
        if (!valid) return;
        if (hh == 0) {
            const float* row = a.obs + ix * a.xs;
#pragma unroll
            for (int f = 0; f < PP / 4; ++f) {
                const float* p = row + (4 * f < in ? 4 * f : 0);
                o[f] = vec ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
            }
        }
        act = a.action[ix];
        ret = Gb[(tile - t0) * kTile + r];
        if (a.clip > 0.f)
#pragma unroll
            for (int c = 0; c < kA; ++c) bl[c] = a.blogits[ix * kA + c];
    };
    // the observation to X (zeros past its width, and without a sample)
    auto put = [&](int odd) {
        if (hh != 0) return;
        float v[PP];
#pragma unroll
        for (int f = 0; f < PP; ++f) {
            const float4 q = o[f / 4];
            const float x = f % 4 == 0 ? q.x : f % 4 == 1 ? q.y : f % 4 == 2 ? q.z : q.w;
            v[f] = valid && f < in ? x : 0.f;
        }
        E::put_row(sm + (odd ? E::kX1 : E::kX0), r, v);
    };

    // A ReLU whose input is within rounding of zero may go either way, and each such
    // sample moves the gradient (a mean of terms of both signs) by ~1e-4 of its norm:
    // inputs below 2^-20 of the largest of eight of the row's (13 times the usual
    // difference of two fp32 sums) take the sign of the fp32 chain, so that nearly
    // always both kernels take the same branch. Not always: the sums' difference goes
    // with their terms, and a unit whose terms cancel far below them can differ by more.
    // About one tile in 50 has an input this close to zero.
    auto settle = [&](float (&z)[32], int layer, int odd) {
        float mn = fabsf(z[0]), mx = mn;
#pragma unroll
        for (int i = 1; i < 32; ++i) mn = fminf(mn, fabsf(z[i]));
#pragma unroll
        for (int i = 4; i < 32; i += 4) mx = fmaxf(mx, fabsf(z[i]));
        mx *= 0x1p-20f;
        if (!__any_sync(0xffffffffu, valid && mn < mx)) return;
        uint32_t near = 0u;
#pragma unroll
        for (int i = 0; i < 32; ++i) near |= valid && fabsf(z[i]) < mx ? 1u << i : 0u;
        const uint32_t pos = chain_signs<PP>(a.arena + a.pol_offs[b], in, sm + (odd ? E::kX1 : E::kX0), 32 * qt, 32 * hh, layer, near);
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if ((near >> i) & 1u) z[i] = (pos >> i) & 1u ? fmaxf(fabsf(z[i]), 1.17549435e-38f) : -fabsf(z[i]);
    };

    bool fetched = false;                                // the tile's X is stored and its layer 1 issued
    int odd = 0;
    for (int64_t tile = lo; tile < hi; ++tile) {
        if (b < 0 || tile >= a.tile_off[b + 1]) {
            // the next policy of the batch with tiles: flush the previous one's
            // partials, stage this one, restart the sums
            if (b >= 0) flush();
            if (b < 0) b = 0;
            while (tile >= a.tile_off[b + 1]) ++b;
            E::stage(sm, a.arena + a.pol_offs[b], in, tid);
            M = a.samp_off[b + 1] - a.samp_off[b];
            invM = M > 0 ? (float)(1.0 / (double)M) : 0.f;
            base = (float)a.stats[4 * b + 1];
            slots = a.slots + (int64_t)b * a.n_pairs * a.n_agents;
            Gb = a.G + a.samp_off[b];
            t0 = a.tile_off[b];
#pragma unroll
            for (int i = 0; i < 32; ++i) gacc[i] = 0.f;
#pragma unroll
            for (int c = 0; c < kA; ++c) {
                gb3[c] = 0.f;
                gw3[c] = 0ull;
            }
            gb2 = 0.f;
            lsum = hsum = 0.f;
            fetched = false;
        }
        if (!fetched) {
            locate(tile, true);
            gather(tile);
            put(odd);
            hand_over();
            if (issues()) E::issue_l1(tb, smu, odd, &bars[0]);
            __syncwarp();
        }
        // PPO: log mu(a | o), the behavior policy's log-softmax at the action taken
        float lmu = 0.f;
        if (valid && a.clip > 0.f) {
            float m = bl[0];
#pragma unroll
            for (int c = 1; c < kA; ++c) m = fmaxf(m, bl[c]);
            float S = 0.f;
#pragma unroll
            for (int c = 0; c < kA; ++c) S += expf(bl[c] - m);
            float la = bl[0];
#pragma unroll
            for (int c = 1; c < kA; ++c)
                if (c == act) la = bl[c];
            lmu = la - m - logf(S);
        }
        // h1: this thread's 32 units
        uint32_t m1 = 0u;
        mma_wait(0);
        {
            uint32_t d[32];
            float v[32];
            tc::tmem_ld32x1(tq + E::kD + 32u * hh, d);
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(d[i]);
            settle(v, 1, odd);
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                m1 |= v[i] > 0.f ? 1u << i : 0u;
                v[i] = relu_nan(v[i]);
            }
            E::spread(v, tq, hh, true, sm + E::kH1 + (odd ? 2 * E::kPartH1 : 0u),
                      odd ? -(int)E::kPartH1 : (int)E::kPartH1, r, 32 * hh);
            tc::tmem_wait_st();
        }
        hand_over();
        if (issues()) E::issue_l2(tb, smu, odd, &bars[1]);
        __syncwarp();
        fetched = tile + 1 < hi && tile + 1 < a.tile_off[b + 1];
        if (fetched) locate(tile + 1, false);
        mma_wait(1);
        float h2[32];
        {
            uint32_t d[32];
            tc::tmem_ld32x1(tq + E::kD + 32u * hh, d);
#pragma unroll
            for (int i = 0; i < 32; ++i) h2[i] = __uint_as_float(d[i]);
            settle(h2, 2, odd);
#pragma unroll
            for (int i = 0; i < 32; ++i) h2[i] = relu_nan(h2[i]);
            float4* p = reinterpret_cast<float4*>(sm + E::h2_at(r)) + 8 * hh;
#pragma unroll
            for (int i = 0; i < 8; ++i) p[i] = make_float4(h2[4 * i], h2[4 * i + 1], h2[4 * i + 2], h2[4 * i + 3]);
        }
        // logits: the two halves' sums through shared memory
        float z[kA];
        {
            u64 acc[kA][2] = {};
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
                const u64 x0 = f2_pack(__float_as_uint(h2[i]), __float_as_uint(h2[i + 1]));
                const u64 x1 = f2_pack(__float_as_uint(h2[i + 2]), __float_as_uint(h2[i + 3]));
#pragma unroll
                for (int c = 0; c < kA; ++c) {
                    const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(W3s + c * kH + 32 * hh + i);
                    f2_fma(acc[c][0], x0, w.x);
                    f2_fma(acc[c][1], x1, w.y);
                }
            }
#pragma unroll
            for (int c = 0; c < kA; ++c) {
                const float2 v = f2_split(f2_add(acc[c][0], acc[c][1]));
                z[c] = v.x + v.y;
                Ps[c * 128 + r] = z[c];
            }
        }
        __syncthreads();
        float dz[kA] = {0.f, 0.f, 0.f, 0.f, 0.f};
        if (valid) {
            const float adv = ret - base;
#pragma unroll
            for (int c = 0; c < kA; ++c) z[c] = (z[c] + Po[c * 128 + r]) + W3s[kA * kH + c];
            float m = z[0];
#pragma unroll
            for (int c = 1; c < kA; ++c) m = fmaxf(m, z[c]);
            float S = 0.f;
#pragma unroll
            for (int c = 0; c < kA; ++c) S += expf(z[c] - m);
            const float lS = logf(S);
            float logp[kA], pi[kA], Hn = 0.f;
#pragma unroll
            for (int c = 0; c < kA; ++c) {
                logp[c] = z[c] - m - lS;
                pi[c] = expf(logp[c]);
                Hn -= pi[c] * logp[c];
            }
            float lp_a = logp[0];
#pragma unroll
            for (int c = 1; c < kA; ++c)
                if (c == act) lp_a = logp[c];
            float gain = adv * lp_a, w = adv;
            if (a.clip > 0.f) {
                // PPO: min(rho A, clip(rho) A); the unclipped term carries the
                // gradient A rho (pi - [c = a]) when it is the minimum (ties to it)
                const float rho = expf(lp_a - lmu);
                const float unc = rho * adv;
                const float clp = fminf(fmaxf(rho, 1.f - a.clip), 1.f + a.clip) * adv;
                w = unc <= clp ? unc : 0.f;
                gain = fminf(unc, clp);
            }
#pragma unroll
            for (int c = 0; c < kA; ++c)
                dz[c] = (w * (pi[c] - (c == act ? 1.f : 0.f)) + a.beta * pi[c] * (logp[c] + Hn)) * invM;
            lsum -= gain + a.beta * Hn;
            hsum += Hn;
        }
        // d2, as operand of d2 W2 and of the sums
        {
            float v[32];
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
                u64 x0 = 0ull, x1 = 0ull;
#pragma unroll
                for (int c = 0; c < kA; ++c) {
                    const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(W3s + c * kH + 32 * hh + i);
                    const u64 d = f2_dup(dz[c]);
                    f2_fma(x0, d, w.x);
                    f2_fma(x1, d, w.y);
                }
                const float2 p = f2_split(x0), q = f2_split(x1);
                v[i] = h2[i] > 0.f ? p.x : 0.f;
                v[i + 1] = h2[i + 1] > 0.f ? p.y : 0.f;
                v[i + 2] = h2[i + 2] > 0.f ? q.x : 0.f;
                v[i + 3] = h2[i + 3] > 0.f ? q.y : 0.f;
            }
            E::spread(v, tq, hh, true, sm + E::kDU, (int)E::kPartDU, r, 32 * hh);
        }
        if (hh == 0) {
            float4* p = reinterpret_cast<float4*>(sm + E::kDZ) + 2 * r;
            p[0] = make_float4(dz[0], dz[1], dz[2], dz[3]);
            p[1] = make_float4(dz[4], 0.f, 0.f, 0.f);
#pragma unroll
            for (int c = 0; c < kA; ++c) gb3[c] += dz[c];
        }
        tc::tmem_wait_st();
        hand_over();
        if (issues()) E::issue_d1(tb, smu, &bars[2]);
        __syncwarp();
        if (fetched) gather(tile + 1);
        // dW3 meanwhile
        {
            u64 t[kA] = {};
            const uint8_t* hp = sm + E::h2_at(16 * warp) + 8 * lane;
            const float* dp = reinterpret_cast<const float*>(sm + E::kDZ) + 8 * 16 * warp;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const u64 h = *reinterpret_cast<const u64*>(hp + i * E::kRow);
                const float4 d = *reinterpret_cast<const float4*>(dp + 8 * i);
                f2_fma(t[0], h, f2_dup(d.x));
                f2_fma(t[1], h, f2_dup(d.y));
                f2_fma(t[2], h, f2_dup(d.z));
                f2_fma(t[3], h, f2_dup(d.w));
                f2_fma(t[4], h, f2_dup(dp[8 * i + 4]));
            }
#pragma unroll
            for (int c = 0; c < kA; ++c) gw3[c] = f2_add(gw3[c], t[c]);
        }
        __syncthreads();                                 // h2 and dz are read
        mma_wait(2);
        {
            uint32_t d[32];
            float d1[32];
            tc::tmem_ld32x1(tq + E::kD + 32u * hh, d);
#pragma unroll
            for (int i = 0; i < 32; ++i) d1[i] = (m1 >> i) & 1u ? __uint_as_float(d[i]) : 0.f;
            E::spread(d1, tq, hh, false, sm + E::kDU, (int)E::kPartDU, r, 64 + 32 * hh);
        }
        hand_over();
        if (issues()) {
            if (odd) E::template issue_grads<true>(tb, smu, &bars[3]);
            else E::template issue_grads<false>(tb, smu, &bars[3]);
        }
        __syncwarp();
        // the next tile's layer 1 behind them
        if (fetched) {
            put(odd ^ 1);
            hand_over();
            if (issues()) E::issue_l1(tb, smu, odd ^ 1, &bars[0]);
            __syncwarp();
        }
        mma_wait(3);
        parity ^= 1u;
        // the tile's sums to the running ones, the small parts' columns first
        const uint32_t gx = tq + (odd ? E::kGX1 : E::kGX0);
        if (qt < 2) {
            uint32_t l[32], m[32];
            tc::tmem_ld32x1(tq + E::kG2 + (odd ? 0u : 128u) + 32u * hh, l);
            tc::tmem_ld32x1(tq + E::kG2 + 64u + 32u * hh, m);
#pragma unroll
            for (int i = 0; i < 32; ++i) l[i] = __float_as_uint(__uint_as_float(l[i]) + __uint_as_float(m[i]));
            tc::tmem_ld32x1(tq + E::kG2 + (odd ? 128u : 0u) + 32u * hh, m);
#pragma unroll
            for (int i = 0; i < 32; ++i) gacc[i] += __uint_as_float(l[i]) + __uint_as_float(m[i]);
            if (hh == 0) {
                float c16[16];
                tc::tmem_ld16(gx + 16u * E::kOnesStep, c16);
                gb2 += c16[E::kOnesAt];
            }
        } else {
#pragma unroll
            for (int c = 0; c < (kChunks + 1) / 2; ++c)
                if (2 * c + hh < kChunks) {
                    float c16[16];
                    tc::tmem_ld16(gx + 16u * (2 * c + hh), c16);
#pragma unroll
                    for (int i = 0; i < 16; ++i) gacc[16 * c + i] += c16[i];
                }
        }
        odd ^= 1;
    }
    tc::fence_before_sync();
    flush();
    if (warp == 0) tc::tmem_dealloc(tmem_base, 512);
    __syncthreads();
    if (redo[1] > redo[0]) redo_tiles(a, reinterpret_cast<float*>(sm), redo[0], redo[1]);
}

template <int PP>
cudaError_t launch_pp(const LearnArgs& a, cudaStream_t s) {
    constexpr size_t bytes = LearnX3<PP>::kBytes > kSBytes ? LearnX3<PP>::kBytes : kSBytes;    // redo_tiles needs kSBytes
    const cudaError_t e = cudaFuncSetAttribute(learn_grad_x3_kernel<PP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)bytes);
    if (e != cudaSuccess) return e;
    learn_grad_x3_kernel<PP><<<a.grid, kThreads, bytes, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_learn_grad_x3(const LearnArgs& a, cudaStream_t s) {
    if (a.in <= 8) return launch_pp<8>(a, s);
    if (a.in <= 12) return launch_pp<12>(a, s);
    if (a.in <= 16) return launch_pp<16>(a, s);
    if (a.in <= 20) return launch_pp<20>(a, s);
    return cudaErrorInvalidValue;
}

}  // namespace malib
