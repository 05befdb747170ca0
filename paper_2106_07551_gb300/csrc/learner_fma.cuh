// The learner's gradient of a range of tiles in fp32 FMAs on the CUDA cores:
// learn_grad_kernel's whole work, and what learn_grad_x3_kernel takes again where
// its operands have no finite bf16 parts.
#pragma once

#include "device_common.cuh"
#include "f32x2.cuh"
#include "learner_common.cuh"

namespace malib {

// The per-tile activations are stored feature-major ([feature][sample], rows of
// kTS floats, 16-byte aligned), so that a thread's 8 samples or 4 consecutive
// samples are one or two 16-byte loads; kTS = 132 spreads rows 16 apart over
// the banks.
constexpr int kTS = kTile + 4;
constexpr int kXR = kLearnMaxIn;     // observation feature rows

// Shared-memory layout of learn_tiles_fma (floats).
constexpr int kSW1T = 0;                          // [in][64]: W1T[k][j] = W1[j][k]
constexpr int kSB1 = kSW1T + kLearnMaxIn * kH;
constexpr int kSW2T = kSB1 + kH;                  // [64][64]: W2T[k][j] = W2[j][k]
constexpr int kSW2 = kSW2T + kH * kH;             // [64][64]: W2[j][k]
constexpr int kSB2 = kSW2 + kH * kH;
constexpr int kSW3 = kSB2 + kH;                   // [5][64]
constexpr int kSB3 = kSW3 + kA * kH;              // [8]
constexpr int kSX = kSB3 + 8;                     // XT [in][kTS] observations
constexpr int kSH1 = kSX + kXR * kTS;             // H1T [64][kTS] post-ReLU layer 1
constexpr int kSH2 = kSH1 + kH * kTS;             // H2T [64][kTS] post-ReLU layer 2
constexpr int kSD2 = kSH2 + kH * kTS;             // D2T [64][kTS] dL/d(pre-activation 2)
constexpr int kSD1 = kSD2 + kH * kTS;             // D1T [64][kTS] dL/d(pre-activation 1)
constexpr int kSDZ = kSD1 + kH * kTS;             // DZT [8][kTS] dL/dz
constexpr int kSFloats = kSDZ + 8 * kTS;
constexpr size_t kSBytes = (size_t)kSFloats * 4;
static_assert(kSBytes <= 232448, "fits the 227 KB of shared memory of a CTA");
static_assert(kSX % 4 == 0 && kTS % 4 == 0, "16-byte aligned rows");

// H_out[j][s] = relu(b[j] + sum_k W[k][j] H_in[k][s]) for this thread's 8
// samples (8 sg ..) and 4 outputs (ng + 16 q): per k two 16-byte loads of H_in
// (four sample pairs) and four weights, each duplicated into a pair, for 16
// packed FMAs (each lane an fmaf in the same order as a scalar loop).
__device__ __forceinline__ void dense_relu(const float* __restrict__ Win, const float* __restrict__ b,
                                           const float* __restrict__ Hin, int K, float* __restrict__ Hout,
                                           int sg, int ng) {
    using u64 = unsigned long long;
    u64 acc[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const u64 b2 = f2_dup(b[ng + 16 * q]);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[q][i] = b2;
    }
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const ulonglong2 x0 = *reinterpret_cast<const ulonglong2*>(Hin + k * kTS + 8 * sg);
        const ulonglong2 x1 = *reinterpret_cast<const ulonglong2*>(Hin + k * kTS + 8 * sg + 4);
        const u64 x[4] = {x0.x, x0.y, x1.x, x1.y};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const u64 w = f2_dup(Win[k * kH + ng + 16 * q]);
#pragma unroll
            for (int i = 0; i < 4; ++i) f2_fma(acc[q][i], x[i], w);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        ulonglong2* o = reinterpret_cast<ulonglong2*>(Hout + (ng + 16 * q) * kTS + 8 * sg);
        o[0] = make_ulonglong2(f2_relu(acc[q][0]), f2_relu(acc[q][1]));
        o[1] = make_ulonglong2(f2_relu(acc[q][2]), f2_relu(acc[q][3]));
    }
}

// The 8 values of a sample-pair row (four pairs) where the activations h are
// positive, else 0 (the ReLU's derivative), stored at o.
__device__ __forceinline__ void store_masked(float* __restrict__ o, const unsigned long long (&v)[4],
                                             const float* __restrict__ h) {
    const float4 h0 = *reinterpret_cast<const float4*>(h);
    const float4 h1 = *reinterpret_cast<const float4*>(h + 4);
    const float2 v0 = f2_split(v[0]), v1 = f2_split(v[1]), v2 = f2_split(v[2]), v3 = f2_split(v[3]);
    *reinterpret_cast<float4*>(o) = make_float4(h0.x > 0.f ? v0.x : 0.f, h0.y > 0.f ? v0.y : 0.f,
                                                h0.z > 0.f ? v1.x : 0.f, h0.w > 0.f ? v1.y : 0.f);
    *reinterpret_cast<float4*>(o + 4) = make_float4(h1.x > 0.f ? v2.x : 0.f, h1.y > 0.f ? v2.y : 0.f,
                                                    h1.z > 0.f ? v3.x : 0.f, h1.w > 0.f ? v3.y : 0.f);
}

// Tiles [lo, hi) of the batch, all threads of the CTA: the partial gradient of
// every policy with tiles among them, in the dynamic shared memory sm (kSBytes).
__device__ __forceinline__ void learn_tiles_fma(const LearnArgs& a, float* sm, int64_t lo, int64_t hi) {
    const int tid = threadIdx.x;
    const int in = a.in;
    const int epp = (int)(a.n_envs / a.n_pairs);
    const int P = kH * in + kH + kH * kH + kH + kA * kH + kA;

    float* XT = sm + kSX;
    float* H1T = sm + kSH1;
    float* H2T = sm + kSH2;
    float* D2T = sm + kSD2;
    float* D1T = sm + kSD1;
    float* DZT = sm + kSDZ;
    const int sg = tid >> 4, ng = tid & 15;           // layers: samples 8 sg .., outputs ng + 16 q
    // this thread's gradient entries, accumulated over the CTA's tiles
    float gW2[4][4] = {};                              // dW2[ng' + 16 p][kb + 16 q], ng' = sg
    const int w1j = tid & 63, w1k = tid >> 6;          // dW1[w1j][w1k + 4 q]
    float gW1[kLearnMaxIn / 4] = {};
    float gW3[2] = {};                                 // dW3 entries tid, tid + 256 of [5][64]
    float gB = 0.f;                                    // b1 (tid < 64), b2 (64..127), b3 (128..132)
    float lsum = 0.f, hsum = 0.f;                      // loss and entropy of this thread's samples
    int b = -1;                                        // the batch's policy of the current tiles
    int64_t M = 0, t0 = 0;
    float invM = 0.f, base = 0.f;
    const int32_t* slots = nullptr;
    const float* Gb = nullptr;
    // this CTA's partial gradient of policy b, in the malib_policy_desc layout:
    // W1 [64][in], b1, W2 [64][64], b2, W3 [5][64], b3, then loss and entropy sums
    auto flush = [&]() {
        float* out = a.gpart + ((int64_t)b * a.grid + blockIdx.x) * (P + 2);
#pragma unroll
        for (int q = 0; q < kLearnMaxIn / 4; ++q) {
            const int k = w1k + 4 * q;
            if (k < in) out[w1j * in + k] = gW1[q];
        }
        const int oW2 = kH * in + kH;
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) out[oW2 + (sg + 16 * p) * kH + ng + 16 * q] = gW2[p][q];
        const int oW3 = oW2 + kH * kH + kH;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int e = tid + kThreads * q;
            if (e < kA * kH) out[oW3 + e] = gW3[q];
        }
        if (tid < kH) out[kH * in + tid] = gB;                          // b1
        else if (tid < 2 * kH) out[oW2 + kH * kH + tid - kH] = gB;      // b2
        else if (tid < 2 * kH + kA) out[oW3 + kA * kH + tid - 2 * kH] = gB;   // b3
        // loss and entropy sums (fixed-order tree in shared memory; the tiles'
        // buffers are free between tiles)
        float* red = sm + kSX;
        red[tid] = lsum;
        red[kThreads + tid] = hsum;
        __syncthreads();
        for (int w = kThreads / 2; w > 0; w >>= 1) {
            if (tid < w) {
                red[tid] += red[tid + w];
                red[kThreads + tid] += red[kThreads + tid + w];
            }
            __syncthreads();
        }
        if (tid == 0) {
            out[P] = red[0];
            out[P + 1] = red[kThreads];
        }
        __syncthreads();
    };
    for (int64_t tile = lo; tile < hi; ++tile) {
        if (b < 0 || tile >= a.tile_off[b + 1]) {
            // the next policy of the batch with tiles: flush the previous one's
            // partials, stage this one (F32Layout: W1T [in][64], b1, W2T [64][64],
            // b2, W3 [5][64], b3), restart the sums
            if (b >= 0) flush();
            if (b < 0) b = 0;
            while (tile >= a.tile_off[b + 1]) ++b;
            const float* pol = a.arena + a.pol_offs[b];
            for (int i = tid; i < in * kH; i += kThreads) sm[kSW1T + i] = pol[i];
            for (int i = tid; i < kH; i += kThreads) sm[kSB1 + i] = pol[in * kH + i];
            for (int i = tid; i < kH * kH; i += kThreads) {
                const float w = pol[in * kH + kH + i];               // W2T[k][j], i = k * 64 + j
                sm[kSW2T + i] = w;
                sm[kSW2 + (i & (kH - 1)) * kH + (i >> 6)] = w;        // W2[j][k]
            }
            for (int i = tid; i < kH; i += kThreads) sm[kSB2 + i] = pol[in * kH + kH + kH * kH + i];
            for (int i = tid; i < kA * kH; i += kThreads) sm[kSW3 + i] = pol[in * kH + 2 * kH + kH * kH + i];
            if (tid < kA) sm[kSB3 + tid] = pol[in * kH + 2 * kH + kH * kH + kA * kH + tid];
            M = a.samp_off[b + 1] - a.samp_off[b];
            invM = M > 0 ? (float)(1.0 / (double)M) : 0.f;
            base = (float)a.stats[4 * b + 1];
            slots = a.slots + (int64_t)b * a.n_pairs * a.n_agents;
            Gb = a.G + a.samp_off[b];
            t0 = a.tile_off[b];
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) gW2[p][q] = 0.f;
#pragma unroll
            for (int q = 0; q < kLearnMaxIn / 4; ++q) gW1[q] = 0.f;
            gW3[0] = gW3[1] = 0.f;
            gB = 0.f;
            lsum = hsum = 0.f;
            __syncthreads();
        }
        const int64_t s0 = (tile - t0) * kTile;
        // the tile's observations (feature-major; zero columns past M), and for
        // the logits phase each sample's action and return
        int act = 0;
        float ret = 0.f, lmu = 0.f;
        {
            const int r = tid & (kTile - 1), half = tid >> 7;
            const int64_t s = s0 + r;
            if (s < M) {
                const int64_t ix = sample_index(a, slots, s, epp);
                const float* orow = a.obs + ix * a.xs;
                for (int k = half; k < in; k += 2) XT[k * kTS + r] = orow[k];
                if (half == 0) {
                    act = a.action[ix];
                    ret = Gb[s];
                    if (a.clip > 0.f) {
                        // log mu(a | o): the behavior policy's log-softmax at the action taken
                        const float* bl = a.blogits + ix * kA;
                        float l[kA];
#pragma unroll
                        for (int j = 0; j < kA; ++j) l[j] = bl[j];
                        float m = l[0];
#pragma unroll
                        for (int j = 1; j < kA; ++j) m = fmaxf(m, l[j]);
                        float S = 0.f;
#pragma unroll
                        for (int j = 0; j < kA; ++j) S += expf(l[j] - m);
                        float la = l[0];
#pragma unroll
                        for (int j = 1; j < kA; ++j)
                            if (j == act) la = l[j];
                        lmu = la - m - logf(S);
                    }
                }
            } else {
                for (int k = half; k < in; k += 2) XT[k * kTS + r] = 0.f;
            }
        }
        __syncthreads();
        dense_relu(sm + kSW1T, sm + kSB1, XT, in, H1T, sg, ng);
        __syncthreads();
        dense_relu(sm + kSW2T, sm + kSB2, H1T, kH, H2T, sg, ng);
        __syncthreads();
        // logits, softmax and dL/dz, one sample per thread (threads 0 .. 127)
        if (tid < kTile) {
            const int64_t s = s0 + tid;
            float dz[kA] = {0.f, 0.f, 0.f, 0.f, 0.f};
            if (s < M) {
                const float adv = ret - base;
                float z[kA];
#pragma unroll
                for (int j = 0; j < kA; ++j) z[j] = sm[kSB3 + j];
#pragma unroll 8
                for (int h = 0; h < kH; ++h) {
                    const float x = H2T[h * kTS + tid];
#pragma unroll
                    for (int j = 0; j < kA; ++j) z[j] = fmaf(sm[kSW3 + j * kH + h], x, z[j]);
                }
                float m = z[0];
#pragma unroll
                for (int j = 1; j < kA; ++j) m = fmaxf(m, z[j]);
                float S = 0.f;
#pragma unroll
                for (int j = 0; j < kA; ++j) S += expf(z[j] - m);
                const float lS = logf(S);
                float logp[kA], pi[kA], H = 0.f;
#pragma unroll
                for (int j = 0; j < kA; ++j) {
                    logp[j] = z[j] - m - lS;
                    pi[j] = expf(logp[j]);
                    H -= pi[j] * logp[j];
                }
                float lp_a = logp[0];
#pragma unroll
                for (int j = 1; j < kA; ++j)
                    if (j == act) lp_a = logp[j];
                if (a.clip > 0.f) {
                    // PPO: min(rho A, clip(rho) A); the unclipped term carries the
                    // gradient A rho (pi - [j = a]) when it is the minimum (ties to it)
                    const float rho = expf(lp_a - lmu);
                    const float unc = rho * adv;
                    const float clp = fminf(fmaxf(rho, 1.f - a.clip), 1.f + a.clip) * adv;
                    const float w = unc <= clp ? unc : 0.f;
#pragma unroll
                    for (int j = 0; j < kA; ++j)
                        dz[j] = (w * (pi[j] - (j == act ? 1.f : 0.f)) + a.beta * pi[j] * (logp[j] + H)) * invM;
                    lsum -= fminf(unc, clp) + a.beta * H;
                } else {
#pragma unroll
                    for (int j = 0; j < kA; ++j)
                        dz[j] = (adv * (pi[j] - (j == act ? 1.f : 0.f)) + a.beta * pi[j] * (logp[j] + H)) * invM;
                    lsum -= adv * lp_a + a.beta * H;
                }
                hsum += H;
            }
#pragma unroll
            for (int j = 0; j < kA; ++j) DZT[j * kTS + tid] = dz[j];
        }
        __syncthreads();
        // D2 = (dz W3) * [h2 > 0]: samples 8 sg .. (four pairs), units ng + 16 q
        {
            using u64 = unsigned long long;
            u64 dzv[kA][4];
#pragma unroll
            for (int c = 0; c < kA; ++c) {
                const ulonglong2 d0 = *reinterpret_cast<const ulonglong2*>(DZT + c * kTS + 8 * sg);
                const ulonglong2 d1 = *reinterpret_cast<const ulonglong2*>(DZT + c * kTS + 8 * sg + 4);
                dzv[c][0] = d0.x; dzv[c][1] = d0.y; dzv[c][2] = d1.x; dzv[c][3] = d1.y;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int j = ng + 16 * q;
                u64 v[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
                for (int c = 0; c < kA; ++c) {
                    const u64 w = f2_dup(sm[kSW3 + c * kH + j]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) f2_fma(v[i], dzv[c][i], w);
                }
                store_masked(D2T + j * kTS + 8 * sg, v, H2T + j * kTS + 8 * sg);
            }
        }
        __syncthreads();
        // D1 = (D2 W2) * [h1 > 0]: samples 8 sg .. (four pairs), units ng + 16 q
        {
            using u64 = unsigned long long;
            u64 acc[4][4] = {};
#pragma unroll 4
            for (int j = 0; j < kH; ++j) {
                const ulonglong2 d0 = *reinterpret_cast<const ulonglong2*>(D2T + j * kTS + 8 * sg);
                const ulonglong2 d1 = *reinterpret_cast<const ulonglong2*>(D2T + j * kTS + 8 * sg + 4);
                const u64 d[4] = {d0.x, d0.y, d1.x, d1.y};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const u64 w = f2_dup(sm[kSW2 + j * kH + ng + 16 * q]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) f2_fma(acc[q][i], d[i], w);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = ng + 16 * q;
                store_masked(D1T + k * kTS + 8 * sg, acc[q], H1T + k * kTS + 8 * sg);
            }
        }
        __syncthreads();
        // the tile's weight gradients, 4 samples per 16-byte load; packed pairs
        // of consecutive samples (the even and odd samples' sums, added at the
        // tile's end)
        {
            using u64 = unsigned long long;
            u64 t2[4][4] = {};
#pragma unroll 2
            for (int s = 0; s < kTile; s += 4) {
                ulonglong2 d[4], h[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    d[p] = *reinterpret_cast<const ulonglong2*>(D2T + (sg + 16 * p) * kTS + s);
                    h[p] = *reinterpret_cast<const ulonglong2*>(H1T + (ng + 16 * p) * kTS + s);
                }
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        f2_fma(t2[p][q], d[p].x, h[q].x);
                        f2_fma(t2[p][q], d[p].y, h[q].y);
                    }
            }
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float2 v = f2_split(t2[p][q]);
                    gW2[p][q] += v.x + v.y;
                }
        }
        {
            using u64 = unsigned long long;
            u64 t1[kLearnMaxIn / 4] = {};
            for (int s = 0; s < kTile; s += 4) {
                const ulonglong2 d = *reinterpret_cast<const ulonglong2*>(D1T + w1j * kTS + s);
#pragma unroll
                for (int q = 0; q < kLearnMaxIn / 4; ++q) {
                    const int k = w1k + 4 * q;
                    if (k < in) {
                        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(XT + k * kTS + s);
                        f2_fma(t1[q], d.x, x.x);
                        f2_fma(t1[q], d.y, x.y);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < kLearnMaxIn / 4; ++q) {
                const float2 v = f2_split(t1[q]);
                gW1[q] += v.x + v.y;
            }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int e = tid + kThreads * q;
            if (e < kA * kH) {
                const int c = e / kH, j = e - c * kH;
                unsigned long long t3 = 0ull;
                for (int s = 0; s < kTile; s += 4) {
                    const ulonglong2 d = *reinterpret_cast<const ulonglong2*>(DZT + c * kTS + s);
                    const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(H2T + j * kTS + s);
                    f2_fma(t3, d.x, x.x);
                    f2_fma(t3, d.y, x.y);
                }
                const float2 v = f2_split(t3);
                gW3[q] += v.x + v.y;
            }
        }
        if (tid < 2 * kH + kA) {
            const float* row = tid < kH ? D1T + tid * kTS : tid < 2 * kH ? D2T + (tid - kH) * kTS
                                                                         : DZT + (tid - 2 * kH) * kTS;
            float g = gB;
            for (int s = 0; s < kTile; s += 4) {
                const float4 d = *reinterpret_cast<const float4*>(row + s);
                g += d.x;
                g += d.y;
                g += d.z;
                g += d.w;
            }
            gB = g;
        }
        __syncthreads();                        // the tile's buffers are rewritten next
    }

    if (b >= 0) flush();
}

}  // namespace malib
