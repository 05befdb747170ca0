// Collisions as forces between disks (App. B.1: agents that collide, obstacles
// that block the way), for the particle scenarios on the device. The paper
// gives no force law; the model is the soft contact of the particle
// environments it runs: for disks at a and b whose radii sum to dmin, with
// delta = a - b and d = |delta|, the overlap is smoothed by a softplus of
// margin k = 0.001,
//   pen = k log(1 + exp((dmin - d) / k)),
// and a feels F_c pen delta / d (F_c = 100), b its negative. Every step is one
// correctly rounded fp32 operation in a fixed order, so the forces are the same
// bits wherever these steps are evaluated.
#pragma once

#include "device_common.cuh"

namespace malib {

constexpr float kContactMargin = 0.001f;
constexpr float kContactForce = 100.0f;

// log(1 + y) for y in [0, 1]: 2 atanh(z) with z = y / (2 + y) <= 1/3, the odd
// series of atanh up to z^17 (the rest is below 2^-32 of the sum) in Horner
// form in z^2 with fused multiply-adds.
__device__ __forceinline__ float det_log1pf(float y) {
    if (!(y > 0.0f)) return 0.0f;
    const float z = __fdiv_rn(y, __fadd_rn(2.0f, y));
    const float w = __fmul_rn(z, z);
    float p = 0x1.e1e1e2p-5f;          // 1/17
    p = fmaf(p, w, 0x1.111112p-4f);    // 1/15
    p = fmaf(p, w, 0x1.3b13b2p-4f);    // 1/13
    p = fmaf(p, w, 0x1.745d18p-4f);    // 1/11
    p = fmaf(p, w, 0x1.c71c72p-4f);    // 1/9
    p = fmaf(p, w, 0x1.24924ap-3f);    // 1/7
    p = fmaf(p, w, 0x1.99999ap-3f);    // 1/5
    p = fmaf(p, w, 0x1.555556p-2f);    // 1/3
    p = fmaf(p, w, 1.0f);
    return __fmul_rn(__fmul_rn(2.0f, z), p);
}

// The force on disk a from disk b, in the order dx, dy, q = dx dx + dy dy,
// d = sqrt(q), x = (dmin - d) / k, softplus(x) = max(x, 0) + log1p(exp(-|x|)),
// pen = k softplus, c = (F_c pen) / d, (c dx, c dy). False (no force) when
// d = 0 or pen = 0 (the latter once d - dmin >= 87 k: det_expf gives 0).
__device__ __forceinline__ bool contact_force(float ax, float ay, float bx, float by, float dmin,
                                              float& fx, float& fy) {
    const float dx = __fsub_rn(ax, bx), dy = __fsub_rn(ay, by);
    const float d = __fsqrt_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)));
    if (d == 0.0f) return false;
    const float x = __fdiv_rn(__fsub_rn(dmin, d), kContactMargin);
    const float sp = __fadd_rn(x > 0.0f ? x : 0.0f, det_log1pf(det_expf(-fabsf(x))));
    const float pen = __fmul_rn(kContactMargin, sp);
    if (pen == 0.0f) return false;
    const float c = __fdiv_rn(__fmul_rn(kContactForce, pen), d);
    fx = __fmul_rn(c, dx);
    fy = __fmul_rn(c, dy);
    return true;
}

// Adds to F the contact forces among N movable disks (pairs a < b ascending: a
// +f, b -f), then those of M immovable disks on each movable one (a ascending,
// then o ascending). A force is added only where one acts, so without contact
// F keeps its bits.
template <int N, int M>
__device__ __forceinline__ void add_contacts(const float (&px)[N], const float (&py)[N], const float (&rad)[N],
                                             const float* ox, const float* oy, const float* orad,
                                             float (&Fx)[N], float (&Fy)[N]) {
#pragma unroll
    for (int a = 0; a < N; ++a)
#pragma unroll
        for (int b = a + 1; b < N; ++b) {
            float fx, fy;
            if (contact_force(px[a], py[a], px[b], py[b], __fadd_rn(rad[a], rad[b]), fx, fy)) {
                Fx[a] = __fadd_rn(Fx[a], fx);
                Fy[a] = __fadd_rn(Fy[a], fy);
                Fx[b] = __fsub_rn(Fx[b], fx);
                Fy[b] = __fsub_rn(Fy[b], fy);
            }
        }
#pragma unroll
    for (int a = 0; a < N; ++a)
#pragma unroll
        for (int o = 0; o < M; ++o) {
            float fx, fy;
            if (contact_force(px[a], py[a], ox[o], oy[o], __fadd_rn(rad[a], orad[o]), fx, fy)) {
                Fx[a] = __fadd_rn(Fx[a], fx);
                Fy[a] = __fadd_rn(Fy[a], fy);
            }
        }
}

// True unless the disks are surely too far apart for a force: pen = 0 once d -
// dmin >= 87 k = 0.087, and q (the squared distance as contact_force rounds it)
// is above (dmin + 0.0885)^2, a margin of 1.5e-3 that no rounding reaches.
__device__ __forceinline__ bool contact_near(float ax, float ay, float bx, float by, float dmin) {
    const float dx = __fsub_rn(ax, bx), dy = __fsub_rn(ay, by);
    const float q = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
    const float far = dmin + 0.0885f;
    return !(q > far * far);
}

// add_contacts, the same bits, for many pairs of which an environment touches
// few (the simple tag: 14). One force takes about 150 dependent instructions
// (square root, divisions, softplus), and some lane of a warp needs nearly
// every pair; here each lane walks its own near pairs, in add_contacts' order,
// so a warp runs as many forces as its busiest lane has (3 to 5). The tag
// step's transition went from 10,000 to 4,300 cycles.
template <int N, int M>
__device__ __forceinline__ void add_contacts_sparse(const float (&px)[N], const float (&py)[N], const float (&rad)[N],
                                                    const float* ox, const float* oy, const float* orad,
                                                    float (&Fx)[N], float (&Fy)[N]) {
    static_assert(N <= 4 && N + M <= 8 && N * (N - 1) / 2 + N * M <= 16, "pair codes of 5 bits in three words");
    uint32_t mask = 0;
    // pair e: its disks a (2 bits) and b (3 bits, obstacles from N on), 6 pairs a word
    uint32_t code[3] = {0u, 0u, 0u};
    int e = 0;
#pragma unroll
    for (int a = 0; a < N; ++a)
#pragma unroll
        for (int b = a + 1; b < N; ++b) {
            if (contact_near(px[a], py[a], px[b], py[b], __fadd_rn(rad[a], rad[b]))) mask |= 1u << e;
            code[e / 6] |= (uint32_t)(a | (b << 2)) << (5 * (e % 6));
            ++e;
        }
#pragma unroll
    for (int a = 0; a < N; ++a)
#pragma unroll
        for (int o = 0; o < M; ++o) {
            if (contact_near(px[a], py[a], ox[o], oy[o], __fadd_rn(rad[a], orad[o]))) mask |= 1u << e;
            code[e / 6] |= (uint32_t)(a | ((N + o) << 2)) << (5 * (e % 6));
            ++e;
        }
#pragma unroll 1
    while (mask != 0u) {
        const int p = __ffs(mask) - 1;
        mask &= mask - 1u;
        const uint32_t c = (p < 6 ? code[0] >> (5 * p) : p < 12 ? code[1] >> (5 * (p - 6)) : code[2] >> (5 * (p - 12)));
        const int a = (int)(c & 3u), b = (int)((c >> 2) & 7u);
        float ax = px[0], ay = py[0], ar = rad[0], bx = px[0], by = py[0], br = rad[0];
#pragma unroll
        for (int k = 1; k < N; ++k) {
            if (a == k) { ax = px[k]; ay = py[k]; ar = rad[k]; }
            if (b == k) { bx = px[k]; by = py[k]; br = rad[k]; }
        }
#pragma unroll
        for (int o = 0; o < M; ++o)
            if (b == N + o) { bx = ox[o]; by = oy[o]; br = orad[o]; }
        float fx, fy;
        if (!contact_force(ax, ay, bx, by, __fadd_rn(ar, br), fx, fy)) continue;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            if (a == k) { Fx[k] = __fadd_rn(Fx[k], fx); Fy[k] = __fadd_rn(Fy[k], fy); }
            if (b == k) { Fx[k] = __fsub_rn(Fx[k], fx); Fy[k] = __fsub_rn(Fy[k], fy); }
        }
    }
}

// Unit force of the five discrete actions (0 noop, 1 +x, 2 -x, 3 +y, 4 -y).
__device__ __forceinline__ void unit_force(int act, float& fx, float& fy) {
    fx = act == 1 ? 1.f : (act == 2 ? -1.f : 0.f);
    fy = act == 3 ? 1.f : (act == 4 ? -1.f : 0.f);
}

}  // namespace malib
