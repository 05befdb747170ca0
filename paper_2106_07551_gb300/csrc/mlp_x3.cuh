// fp32 policy forward in-64-64-A on the 5th-generation tensor cores: every fp32
// operand is the exact sum of three bf16 parts (x = h + m + l: h = bf16(x), m =
// bf16(x - h), l = x - h - m, 8 + 8 + 8 significant bits) and a product x w is
// taken as the six part products down to 2^-16,
//   l wh + m wm + h wl + m wh + h wm + h wh,
// accumulated in fp32 in tensor memory, the smallest first. The products left
// out are below 2^-24 of x w. In this order the accumulator is small until the
// last K / 16 steps, so only those round at the sum's size: measured against 64
// bits, a K = 64 sum of ReLU activations is off by 6.6e-8 of its norm (fp32 FMA
// chain 1.02e-7; the largest products first 7.1e-7).
//
// A group of four warps owns a tile of 128 rows, one row per thread (warp w of
// the group the tensor-memory lanes 32 w ..), so a row's observation, hidden
// activations and logits never leave its thread but through tensor memory:
//   X (shared memory, bf16 parts)  x  W1, + b1 -> D1   (fp32, 64 columns of H)
//   ReLU(D1), split                            -> H    (96 columns of bf16 pairs)
//   H (tensor memory)              x  W2, + b2 -> D2   (fp32, 64 columns)
//   ReLU(D2) times W3 + b3 in fp32 FMAs in the row's thread.
// A bias is one more K = 16 step, [1 1 1 0 ..] x [bh bm bl 0 ..], taken after the
// small products: exact but for the accumulator's rounding, and the row's
// threads need neither load nor add it.
// Tensor memory per group: 160 columns, so three groups fit the SM's 512. D1
// lies in H's own columns, so the next tile's layer 1 needs only layer 2 done
// and runs while this tile's logits are formed from D2. H holds the parts h, m,
// l of neurons 0 .. 31 in its columns 0 .. 47 and those of 32 .. 63 in 48 .. 95,
// 16 columns a part; D1 is columns 32 .. 95, so converting the first half
// overwrites only what has been read, and the second half its own columns.
//
// Layer 1: with the input width rounded up to even (P), a row of X is [h m l],
// 3 P elements padded with zeros to whole K = 16 steps, and W1 comes as three
// images, [wl 0 0], [wm wm 0] and [wh wh wh], each multiplied with the steps of
// X that it reaches (2 + 3 + 4 steps for 18 inputs, where parts padded one by
// one would take 12); the steps of the last image run from l to h.
//
// An infinity, and a finite value that rounds to a bf16 infinity (from 3.3962e38),
// has no such parts: they are infinite and NaN, and so are the products. The ReLUs
// keep a NaN, which makes every unit of the next layer and every logit NaN, so the
// first logit tells, and the caller takes that row again in fp32 FMAs
// (forward_fma), which give such weights and activations their IEEE meaning. At
// the other end, values below 2^-110 lose their low parts to bf16's smallest
// magnitude, 2^-133: that shows in a sum only next to weights beyond 2^100.
#pragma once

#include <cstdint>

#include "device_common.cuh"
#include "f32x2.cuh"
#include "tc_common.cuh"

namespace malib {

// The three bf16 parts of two floats, packed (v0 in the low halves).
__device__ __forceinline__ void split3(float v0, float v1, uint32_t& h, uint32_t& m, uint32_t& l) {
    h = tc::pack_bf16(v0, v1);
    const float r0 = __fsub_rn(v0, __uint_as_float(h << 16));
    const float r1 = __fsub_rn(v1, __uint_as_float(h & 0xffff0000u));
    m = tc::pack_bf16(r0, r1);
    l = tc::pack_bf16(__fsub_rn(r0, __uint_as_float(m << 16)), __fsub_rn(r1, __uint_as_float(m & 0xffff0000u)));
}

// True for a row whose parts were not finite somewhere (any of its logits tells).
__device__ __forceinline__ bool parts_failed(float logit) { return !(fabsf(logit) <= 3.402823466e38f); }

// The forward of one row x by one thread in fp32 FMAs (bias first, inputs
// ascending), from the population's image; slow, for rows whose parts failed.
template <int IN, int H, int A>
__device__ __noinline__ void forward_fma(const float* __restrict__ img, const float* x, float* lg) {
    using L = F32Layout<IN, H, A>;
    float h1[H], s[A];
#pragma unroll 1
    for (int j = 0; j < H; ++j) {
        float z = __ldg(img + L::kB1 + j);
        for (int k = 0; k < IN; ++k) z = fmaf(x[k], __ldg(img + L::kW1T + k * H + j), z);
        h1[j] = fmaxf(z, 0.f);
    }
    for (int a = 0; a < A; ++a) s[a] = 0.f;
#pragma unroll 1
    for (int j = 0; j < H; ++j) {
        float z = __ldg(img + L::kB2 + j);
#pragma unroll 8
        for (int k = 0; k < H; ++k) z = fmaf(h1[k], __ldg(img + L::kW2T + k * H + j), z);
        z = fmaxf(z, 0.f);
#pragma unroll
        for (int a = 0; a < A; ++a) s[a] = fmaf(z, __ldg(img + L::kW3 + a * H + j), s[a]);
    }
#pragma unroll
    for (int a = 0; a < A; ++a) lg[a] = s[a] + __ldg(img + L::kB3 + a);
}

template <int IN, int A>
struct MlpX3 {
    static constexpr int H = 64;
    using L = F32Layout<IN, H, A>;
    static constexpr int XS = (IN + 3) / 4 * 4;                 // observation row of the trajectory (floats)
    static constexpr int P = (IN + 1) / 2 * 2;
    // K = 16 steps of X that the images [wh wh wh], [wm wm 0], [wl 0 0] reach
    static constexpr int kS1 = (3 * P + 15) / 16, kS2 = (2 * P + 15) / 16, kS3 = (P + 15) / 16;
    static constexpr int kK1 = 16 * kS1;                        // stored elements of a row
    static constexpr uint32_t kStep1 = (uint32_t)64 * 16 * 2;   // bytes of one W1 step
    static constexpr uint32_t kLboX = 128 / 8 * 128, kLboW = H / 8 * 128;   // K-chunk strides (bytes)
    // shared memory of one policy
    static constexpr uint32_t kW1 = 0;
    static constexpr uint32_t kW2 = kW1 + (kS1 + kS2 + kS3) * kStep1;       // parts h, m, l
    static constexpr uint32_t kPart2 = (uint32_t)H * H * 2;
    static constexpr uint32_t kB1 = kW2 + 3 * kPart2;                       // bias steps [64][16]
    static constexpr uint32_t kB2 = kB1 + (uint32_t)H * 16 * 2;
    static constexpr uint32_t kF32 = kB2 + (uint32_t)H * 16 * 2;            // fp32 W3 [A][64], b3
    static constexpr int kFW3 = 0, kFB3 = A * H;
    static constexpr uint32_t kPolicy = (kF32 + (uint32_t)(kFB3 + (A + 3) / 4 * 4) * 4 + 127u) / 128u * 128u;
    static constexpr uint32_t kXBytes = 128u * kK1 * 2;                     // one tile's observations
    static constexpr uint32_t kOnesBytes = 128u * 16 * 2;                   // rows [1 1 1 0 ..] (bias steps)
    // tensor memory columns of one group
    static constexpr uint32_t kD2 = 0, kHid = 64, kD1 = kHid + 32, kCols = 160;
    // column of H holding part `part` of the 16 inputs 16 k .. of layer 2
    __host__ __device__ static constexpr uint32_t h_col(int part, int k) {
        return kHid + 48u * (uint32_t)(k >> 1) + 16u * (uint32_t)part + 8u * (uint32_t)(k & 1);
    }
    static_assert(A <= 16 && IN <= 32, "shapes built");

    // The six products of layer 2 in order: parts (0 h, 1 m, 2 l) of the operands.
    __host__ __device__ static constexpr int part_x(int q) { return q == 0 ? 2 : (q == 1 || q == 3) ? 1 : 0; }
    __host__ __device__ static constexpr int part_w(int q) { return q == 2 ? 2 : (q == 1 || q == 4) ? 1 : 0; }

    // Converts a policy (fp32 F32Layout image in global memory) into the
    // tensor-core image at pol (all nt threads of the CTA; the caller fences
    // for the async proxy and synchronises).
    __device__ static void stage(uint8_t* pol, const float* __restrict__ src, int tid, int nt) {
        // W1: a thread writes the pair (k, k + 1) of one row of one image
        constexpr int kPairs = 8 * (kS1 + kS2 + kS3);
        for (int e = tid; e < H * kPairs; e += nt) {
            const int j = e & (H - 1), p = e >> 6;               // pair p of the concatenated images
            const int img = p < 8 * kS1 ? 0 : p < 8 * (kS1 + kS2) ? 1 : 2;
            const int k = 2 * (p - (img == 0 ? 0 : img == 1 ? 8 * kS1 : 8 * (kS1 + kS2)));
            uint32_t w[3] = {0u, 0u, 0u};
            if (k < (3 - img) * P) {
                const int f = k % P;
                split3(src[L::kW1T + f * H + j], f + 1 < IN ? src[L::kW1T + (f + 1) * H + j] : 0.f, w[0], w[1], w[2]);
            }
            *reinterpret_cast<uint32_t*>(pol + kW1 + tc::cm_offset(j, 2 * p, H, 2)) =
                img == 0 ? w[0] : img == 1 ? w[1] : w[2];
        }
#pragma unroll 4
        for (int e = tid; e < H * (H / 2); e += nt) {
            const int j = e & (H - 1), p = e >> 6;
            uint32_t w[3];
            split3(src[L::kW2T + 2 * p * H + j], src[L::kW2T + (2 * p + 1) * H + j], w[0], w[1], w[2]);
#pragma unroll
            for (int q = 0; q < 3; ++q)
                *reinterpret_cast<uint32_t*>(pol + kW2 + q * kPart2 + tc::cm_offset(j, 2 * p, H, 2)) = w[q];
        }
        float* f = reinterpret_cast<float*>(pol + kF32);
        for (int e = tid; e < 2 * H; e += nt) {
            const int j = e & (H - 1);
            uint32_t w[3];
            split3(src[(e < H ? L::kB1 : L::kB2) + j], 0.f, w[0], w[1], w[2]);
            uint8_t* row = pol + (e < H ? kB1 : kB2);
            *reinterpret_cast<uint4*>(row + tc::cm_offset(j, 0, H, 2)) = make_uint4(w[0] | (w[1] << 16), w[2], 0u, 0u);
            *reinterpret_cast<uint4*>(row + tc::cm_offset(j, 8, H, 2)) = make_uint4(0u, 0u, 0u, 0u);
        }
        for (int e = tid; e < A * H; e += nt) f[kFW3 + e] = src[L::kW3 + e];
        for (int e = tid; e < A; e += nt) f[kFB3 + e] = src[L::kB3 + e];
    }

    // Row r of the ones tile.
    __device__ static void put_ones(uint8_t* ones, int r) {
        *reinterpret_cast<uint4*>(ones + tc::cm_offset(r, 0, 128, 2)) = make_uint4(0x3f803f80u, 0x3f80u, 0u, 0u);
        *reinterpret_cast<uint4*>(ones + tc::cm_offset(r, 8, 128, 2)) = make_uint4(0u, 0u, 0u, 0u);
    }

    // Writes row r of the tile X from its observation o[XS] (zeros past IN).
    __device__ static void put_row(uint8_t* X, int r, const float* o) {
        uint32_t w[3][P / 2];
#pragma unroll
        for (int p = 0; p < P / 2; ++p) split3(o[2 * p], o[2 * p + 1], w[0][p], w[1][p], w[2][p]);
#pragma unroll
        for (int c = 0; c < kK1 / 8; ++c) {
            uint32_t v[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int i = 4 * c + h, q = i / (P / 2), p = i % (P / 2);   // word i: part q, pair p
                v[h] = q < 3 ? w[q < 3 ? q : 0][p] : 0u;
            }
            *reinterpret_cast<uint4*>(X + tc::cm_offset(r, 8 * c, 128, 2)) = make_uint4(v[0], v[1], v[2], v[3]);
        }
    }
    __device__ static void zero_row(uint8_t* X, int r) {
#pragma unroll
        for (int c = 0; c < kK1 / 8; ++c)
            *reinterpret_cast<uint4*>(X + tc::cm_offset(r, 8 * c, 128, 2)) = make_uint4(0u, 0u, 0u, 0u);
    }

    // One thread: layer 1 of the tile X into D1, then an arrival on bar. The
    // bias comes before the last step, which holds the first h wh products.
    __device__ static void issue1(uint32_t tbase, uint32_t x, uint32_t ones, uint32_t pol, uint64_t* bar) {
        const uint32_t idesc = tc::instr_desc(128, H, 1);
        const uint64_t dx = tc::smem_desc(x, kLboX, 128), dw = tc::smem_desc(pol + kW1, kLboW, 128);
        auto step = [&](int k, int w, bool acc) {
            tc::mma_bf16(tbase + kD1, dx + (uint64_t)k * ((2u * kLboX) >> 4), dw + (uint64_t)w * (kStep1 >> 4), idesc, acc);
        };
#pragma unroll
        for (int k = 0; k < kS3; ++k) step(k, kS1 + kS2 + k, k != 0);
#pragma unroll
        for (int k = kS2 - 1; k >= 0; --k) step(k, kS1 + k, true);
#pragma unroll
        for (int k = kS1 - 1; k >= 0; --k) {
            if (k == 0)
                tc::mma_bf16(tbase + kD1, tc::smem_desc(ones, kLboX, 128), tc::smem_desc(pol + kB1, kLboW, 128), idesc,
                             true);
            step(k, k, true);
        }
        tc::mma_commit(bar);
    }

    // One thread: layer 2 (A operand from tensor memory) into D2, then an
    // arrival on bar.
    __device__ static void issue2(uint32_t tbase, uint32_t ones, uint32_t pol, uint64_t* bar) {
        const uint32_t idesc = tc::instr_desc(128, H, 1);
        const uint64_t dw = tc::smem_desc(pol + kW2, kLboW, 128);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            if (q == 5)
                tc::mma_bf16(tbase + kD2, tc::smem_desc(ones, kLboX, 128), tc::smem_desc(pol + kB2, kLboW, 128), idesc,
                             true);
#pragma unroll
            for (int k = 0; k < H / 16; ++k)
                mma_ts(tbase + kD2, tbase + h_col(part_x(q), k),
                       dw + (uint64_t)(part_w(q) * (kPart2 >> 4) + k * ((2u * kLboW) >> 4)), idesc, q + k != 0);
        }
        tc::mma_commit(bar);
    }

    __device__ static void mma_ts(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t idesc, bool acc) {
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d),
            "r"(a_tmem), "l"(b), "r"(idesc), "r"((uint32_t)acc)
            : "memory");
    }

    // All lanes of a warp (lane_q: its tensor-memory lanes << 16): the hidden
    // activations relu(D1) of its rows, split into H.
    __device__ static void hidden(uint32_t tbase, uint32_t lane_q) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            uint32_t v[32], w[3][16];
            tc::tmem_ld32x1(tbase + lane_q + kD1 + 32u * c, v);
#pragma unroll
            for (int i = 0; i < 16; ++i)
                split3(relu_nan(__uint_as_float(v[2 * i])), relu_nan(__uint_as_float(v[2 * i + 1])), w[0][i], w[1][i],
                       w[2][i]);
#pragma unroll
            for (int q = 0; q < 3; ++q) tc::tmem_st16(tbase + lane_q + h_col(q, 2 * c), w[q]);
        }
        tc::tmem_wait_st();
    }

    // All lanes of a warp: its rows' logits W3 relu(D2) + b3, in packed pairs
    // of hidden units.
    __device__ static void logits(uint32_t tbase, uint32_t lane_q, const uint8_t* pol, float (&lg)[A]) {
        using u64 = unsigned long long;
        constexpr int kSums = A <= 8 ? 4 : 2;      // chains per action (fewer where registers run out)
        const float* f = reinterpret_cast<const float*>(pol + kF32);
        u64 acc[A][kSums];
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
            for (int q = 0; q < kSums; ++q) acc[a][q] = 0ull;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            uint32_t d[32];
            tc::tmem_ld32x1(tbase + lane_q + kD2 + 32u * c, d);
            u64 z[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) z[i] = f2_relu_nan(f2_pack(d[2 * i], d[2 * i + 1]));
#pragma unroll
            for (int i = 0; i < 8; ++i) {
#pragma unroll
                for (int a = 0; a < A; ++a) {
                    const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(f + kFW3 + a * H + 32 * c + 4 * i);
                    f2_fma(acc[a][(2 * i) % kSums], z[2 * i], w.x);
                    f2_fma(acc[a][(2 * i + 1) % kSums], z[2 * i + 1], w.y);
                }
            }
        }
#pragma unroll
        for (int a = 0; a < A; ++a) {
#pragma unroll
            for (int q = kSums / 2; q > 0; q >>= 1)
#pragma unroll
                for (int i = 0; i < q; ++i) acc[a][i] = f2_add(acc[a][i], acc[a][i + q]);
            const float2 q = f2_split(acc[a][0]);
            lg[a] = __fadd_rn(__fadd_rn(q.x, q.y), f[kFB3 + a]);
        }
    }
};

}  // namespace malib
