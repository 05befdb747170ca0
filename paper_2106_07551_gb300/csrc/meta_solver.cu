// Meta-game solvers on the payoff table (Sec. 4.2: the PSRO loop on Leduc uses
// fictitious play as its meta-solver and names an exact LP solver; App. C.2:
// payoffs aggregated under the equilibrium). A[i][j] is seat 0's payoff when
// row policy i meets column policy j; the games are zero-sum.
//
// One CTA solves one game of fictitious play, the sides on different warps and
// each play's argmax / argmin by integer warp reductions; an LP is dealt over the
// CTAs of a cluster by columns. What a game needs stays on chip where it fits: the
// payoff matrix (or the LP tableau) in shared memory, cumulative payoffs in
// registers.
#include <cstdint>
#include <type_traits>

#include "internal.h"
#include "malib.h"
#include "quotient.cuh"

namespace malib {

namespace {

constexpr int kFpWarps = 8;                     // warps per side
constexpr int kFpPer = 4;                       // rows (columns) per thread: m, n <= 1024
constexpr int kFpMaxDim = 32 * kFpWarps * kFpPer;
// Bytes of payoff / tableau kept on chip; also the kernels' dynamic shared memory limit,
// which is the process's, so that calls of several threads never lower one another's.
constexpr int kSmemLimit = 200 * 1024;

// Order-preserving integer key of a finite double (larger double, larger
// key), and its inverse. The comparisons of a play run on these keys: fp64
// arithmetic is a narrow pipe on this part, integer compares and shuffles are
// not. The cumulative payoffs start at +0.0 and every sum with +0.0 is +0.0,
// so -0.0 never occurs and key equality is value equality.
__device__ __forceinline__ long long okey(double v) {
    const long long b = __double_as_longlong(v);
    return b >= 0 ? b : b ^ 0x7fffffffffffffffll;
}
__device__ __forceinline__ double okey_inv(long long k) {
    return __longlong_as_double(k >= 0 ? k : k ^ 0x7fffffffffffffffll);
}

struct Cand {
    long long k;      // key to maximise; kNone for "no candidate"
    int i;            // index; ties go to the lower one
};
constexpr long long kNone = (long long)0x8000000000000000ull;   // below every finite key

// Branch-free: b replaces a when its key is larger, or equal with a lower index.
__device__ __forceinline__ Cand pick(Cand a, Cand b) {
    const bool take = (b.k > a.k) | ((b.k == a.k) & (b.i < a.i));
    return Cand{take ? b.k : a.k, take ? b.i : a.i};
}

// The best candidate of a warp (every lane gets it): the largest key by its high
// then its low word, then the lowest index, each one warp-wide integer
// reduction. Five rounds of 64-bit shuffles and selects took about twice as long.
__device__ __forceinline__ Cand warp_best(Cand a) {
    const int hi = (int)(a.k >> 32);
    const unsigned lo = (unsigned)a.k;
    const int mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    const unsigned i = __reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? (unsigned)a.i : 0xffffffffu);
    return Cand{((long long)mh << 32) | (long long)ml, (int)i};
}

// Simultaneous fictitious play: both play policy 0 first; then each plays the
// first best response to the other's plays so far. u_row[i] = sum over plays of
// A[i][j_s] and u_col[j] = sum of A[i_s][j] are fp64 sums in play order, held in
// registers. The column player's argmin is the argmax of the negated key.
//
// A play is a chain: load, fp64 addition (64 cycles), argmax in the warp (three
// integer reductions of 24), one CTA barrier, argmax over the side's warps;
// nothing of the next play can start before. So the two sides are on different
// warps (two additions would take turns on a scheduler), and after the barrier
// every thread reads both sides' at most eight candidates from shared memory (a
// buffer selected by the play's parity, so one barrier per play) and takes the
// best by a fixed tree; the play counts are compares in registers, off the
// chain. 64 x 64, one game: 165 ns a play; with both sides on every warp, the
// argmax by 64-bit shuffles and the candidates reduced again in every warp 575.
// Warps 0 .. wr - 1 hold the rows (row lane + 32 w + 32 wr k), the rest the
// columns. K: rows (columns) per thread; W: candidates per side read (1, 2, 4, 8).
// kTable: the payoffs on chip, or read where they lie with strides that fit 32 bits (a
// 64-bit product is on the chain of a play: 1 % at 256 x 256), or with any.
enum FpTable { kFpOnChip, kFpNear, kFpFar };
template <FpTable kTable, int K, int W>
__global__ void __launch_bounds__(64 * W) fictitious_play_kernel(
    const double* __restrict__ P, int32_t n_games, int32_t m, int32_t n, int32_t stride,
    int64_t T, int32_t wr, double* __restrict__ x_out, double* __restrict__ y_out,
    double* __restrict__ bounds_out) {
    constexpr bool kOnChip = kTable == kFpOnChip;
    // This side's best while the payoffs arrive (256 x 256: 797 -> 769 ns a play), where
    // they come from L2; from shared memory at once with the other's (64 x 64: 348 -> 328
    // us for 2,000 plays), and with four rows a thread too (513 x 513: 1,183 -> 1,120 ns).
    constexpr bool kOwnLate = !kOnChip && K <= 2;
    extern __shared__ double sA[];              // [m][ld] when on chip
    __shared__ Cand red[2][2][W];               // [play's parity][side][warp]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nt = blockDim.x;
    const int ld = n | 1;                       // odd row stride: column reads hit distinct banks
    const int side = warp >= wr ? 1 : 0, ws = side ? (nt >> 5) - wr : wr, w = warp - side * wr;
    const int dim = side ? n : m;
    // strides of this side's entries and of the other side's policies
    const int64_t sq = kOnChip ? (side ? 1 : ld) : (int64_t)stride * (side ? 1 : n);
    const int64_t so = kOnChip ? (side ? ld : 1) : (int64_t)stride * (side ? n : 1);

    for (int g = blockIdx.x; g < n_games; g += gridDim.x) {
        const double* Pg = P + (int64_t)g * m * n * stride;
        __syncthreads();                        // the previous game's readers are done
        if (kOnChip) {
            for (int k = tid; k < m * n; k += nt) {
                const int i = k / n, j = k - i * n;
                sA[i * ld + j] = Pg[(int64_t)k * stride];
            }
        }
        if (tid < 4 * W) (&red[0][0][0])[tid] = Cand{kNone, 0x7fffffff};   // warps that do not exist
        __syncthreads();
        double u[K];
        long long cnt[K];
        const double* at[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int q = lane + 32 * (w + ws * k);
            u[k] = 0.0;
            cnt[k] = 0;
            at[k] = (kOnChip ? sA : Pg) + (q < dim ? q * sq : 0);
        }
        int other = 0, own = 0;
        // the best of the other side's candidates (of == 1) or of this side's (of == 0)
        auto best_of = [&](int par, int of) {
            Cand c[W];
#pragma unroll
            for (int q = 0; q < W; ++q) c[q] = red[par][side ^ of][q];
#pragma unroll
            for (int h = W / 2; h > 0; h >>= 1)
#pragma unroll
                for (int q = 0; q < h; ++q) c[q] = pick(c[q], c[q + h]);
            return c[0];
        };
        Cand best_other{kNone, 0};
        for (int64_t t = 0; t < T; ++t) {
            const int par = (int)(t & 1);
            Cand b{kNone, 0x7fffffff};
            double a[K];
#pragma unroll
            for (int k = 0; k < K; ++k)
                a[k] = kOnChip             ? at[k][other * (int)so]
                       : kTable == kFpNear ? __ldg(at[k] + (int64_t)other * (int)so)
                                           : __ldg(at[k] + other * so);
            if (kOwnLate && t > 0) own = best_of(par ^ 1, 0).i;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int q = lane + 32 * (w + ws * k);
                cnt[k] += q == own ? 1 : 0;
                u[k] += a[k];
                const long long key = side ? -okey(u[k]) : okey(u[k]);
                if (q < dim) b = pick(b, Cand{key, q});
            }
            b = warp_best(b);
            if (lane == 0) red[par][side][w] = b;
            __syncthreads();
            best_other = best_of(par, 1);
            other = best_other.i;
            if (!kOwnLate) own = best_of(par, 0).i;
        }
        const Cand best_own = best_of((int)((T - 1) & 1), 0);
        const double Td = (double)T;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int q = lane + 32 * (w + ws * k);
            if (q < dim) (side ? y_out : x_out)[(int64_t)g * dim + q] = (double)cnt[k] / Td;
        }
        if (tid == 0) {                                            // a row thread
            bounds_out[2 * g] = okey_inv(-best_other.k) / Td;      // min_j (x^T A)_j
            bounds_out[2 * g + 1] = okey_inv(best_own.k) / Td;     // max_i (A y)_i
        }
    }
}

// Payoffs under a pair of mixtures: A y (per row), x^T A (per column), x^T A y.
// One block of W warps per game. Rows: kRowLanes lanes each over the columns (32 /
// kRowLanes rows of a warp at once). Columns: a lane each, the rows dealt over the
// warps of its column group. kRowLanes = 0 is for narrow tables, `lanes` (the columns,
// rounded up to a power of two) at most 16: up to 4 lanes a row, and in the second
// pass 32 / lanes rows of a warp at once. Partial sums are combined in a fixed order.
template <int W, int kRowLanes>
__global__ void __launch_bounds__(32 * W) aggregate_kernel(
    const double* __restrict__ P, int32_t n_games, int32_t m, int32_t n, int32_t stride, int32_t lanes,
    const double* __restrict__ x, const double* __restrict__ y, double* __restrict__ ay_out,
    double* __restrict__ xa_out, double* __restrict__ val_out) {
    __shared__ double red[W];
    __shared__ double col[W][32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int L = kRowLanes ? kRowLanes : min(lanes, 4);         // lanes of a row, first pass
    const int C = kRowLanes ? 32 : lanes;                        // columns of a warp, second pass
    for (int g = blockIdx.x; g < n_games; g += gridDim.x) {
        const double* Pg = P + (int64_t)g * m * n * stride;
        const double* xg = x + (int64_t)g * m;
        const double* yg = y + (int64_t)g * n;
        double part = 0.0;                       // of x^T A y: this lane group's rows, in row order
        for (int i0 = warp * (32 / L); i0 < m; i0 += W * (32 / L)) {
            const int i = i0 + lane / L;
            double s = 0.0;
            if (i < m)
#pragma unroll 4
                for (int j = lane & (L - 1); j < n; j += L) s = fma(Pg[((int64_t)i * n + j) * stride], yg[j], s);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (o < L) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (i < m) {
                if ((lane & (L - 1)) == 0) ay_out[(int64_t)g * m + i] = s;
                part = fma(xg[i], s, part);
            }
        }
        for (int o = L; o < 32; o <<= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if (lane == 0) red[warp] = part;
        // columns, W groups of them at a time over all warps
        const int groups = (n + 31) / 32;
        for (int c0 = 0; c0 < groups; c0 += W) {
            const int here = min(W, groups - c0);                // column groups of this round
            const int per = W / here;                            // warps per group
            const int grp = warp / per, sub = warp - grp * per;
            const int j = (c0 + grp) * 32 + (lane & (C - 1));
            double s = 0.0;
            if (grp < here && j < n)
#pragma unroll 4
                for (int i = sub * (32 / C) + lane / C; i < m; i += per * (32 / C))
                    s = fma(xg[i], Pg[((int64_t)i * n + j) * stride], s);
            for (int o = C; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            col[warp][lane] = s;
            __syncthreads();
            if (grp < here && sub == 0 && lane < C && j < n) {
                for (int q = 1; q < per; ++q) s += col[warp + q][lane];
                xa_out[(int64_t)g * n + j] = s;
            }
            __syncthreads();
        }
        if (tid == 0) {
            double v = 0.0;
            for (int w = 0; w < W; ++w) v += red[w];
            val_out[g] = v;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Exact equilibrium by the simplex method. With B = A - min(A) + 1 > 0, the
// column player's problem max sum(q) s.t. B q <= 1, q >= 0 has optimum
// 1 / v_B; y = q v_B, and the row player's x = p v_B from the duals p (the
// objective row under the slack columns). v_A = v_B + min(A) - 1.
// The tableau is kept condensed: rows 0..m-1 hold the nonbasic columns of [B | I]
// and the right side (1), row m the reduced costs (-1 at the start, 0 on the
// right). A pivot on (p, q) scales row p by 1 / a_pq, subtracts a_rq times it
// from every other row r, and puts the leaving variable's column, (1 / a_pq at p,
// -a_rq / a_pq elsewhere), in the entering one's place.
// Entering column: the most negative reduced cost (Dantzig); after 2 (m + n)
// consecutive degenerate pivots the rule switches for good to Bland's (lowest
// index with a negative reduced cost), which cannot cycle. Leaving row: the
// minimum ratio, ties to the lowest basic variable index. A pivot limit (at
// most that many pivots; optimality is still recognised after the last one)
// guards regardless. Comparisons run on the integer keys above; the tableau
// arithmetic is fp64.
//
// A pivot is (m + 1)(n + 1) independent fp64 FMAs between two reductions, and
// fp64 is this part's slowest pipe (2 lanes a clock and SM: 5,000 cycles at 100 x
// 100), so a game's columns are dealt over the CTAs of a cluster. Each CTA has
// its columns and a copy of the right side and the basis; per pivot it offers
// its best entering column (key and label to every CTA, the column in a buffer
// the others read), one cluster barrier decides, and the ratio test and the
// update run in every CTA without further exchange. The column buffer is
// selected by the pivot's parity, so it is written again only after the next
// barrier. One 100 x 100 game (its pivots depend on its entries): 298 us on 8 CTAs
// where the full tableau (identity columns included, a division per element to find
// its row) on one CTA takes 1,237.
// ---------------------------------------------------------------------------
constexpr int kLpThreads = 256, kLpWarps = kLpThreads / 32;
constexpr int kLpMaxDim = 512, kLpMaxCluster = 8;

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
// Without .aligned: a warp's lanes may arrive one by one (its loops before the
// barrier have lane-dependent trip counts).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
    cluster_arrive();
    cluster_wait();
}

struct LpShape {
    int32_t m, n, stride;
    int32_t cluster;             // CTAs per game
    int32_t cols;                // columns of a CTA: ceil(n / cluster)
    int32_t hs;                  // column stride (doubles, odd, >= m + 1)
    int32_t on_chip;
    int32_t rows, rows_log2;     // threads over rows in an update: a power of two, at most 128
    int64_t cta_doubles;         // (cols + 1) * hs
};

template <bool kCluster>
__global__ void __launch_bounds__(kLpThreads) lp_nash_kernel(
    const double* __restrict__ P, int32_t n_games, LpShape sh, double* __restrict__ x_out,
    double* __restrict__ y_out, double* __restrict__ val_out, double* __restrict__ gscratch,
    int32_t pivot_limit, int* __restrict__ err) {
    struct Offer {
        long long key;
        int label, col;          // variable, and its column in the offering CTA
    };
    extern __shared__ double smem_tab[];
    __shared__ double offered[2][kLpMaxDim + 1];             // [parity] this CTA's best entering column
    __shared__ __align__(16) Offer offers[2][kLpMaxCluster]; // [parity][CTA]
    __shared__ double colq[kLpMaxDim + 1], invs[kLpMaxDim], prow[kLpMaxDim + 1];
    __shared__ int basis[kLpMaxDim], label[kLpMaxDim];       // label: variable of each own column
    __shared__ Cand red[2][kLpWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if constexpr (kCluster) cluster_arrive();                // this CTA runs: its peers may store into it
    bool peers_run = false;
    const int m = sh.m, n = sh.n, hs = sh.hs;
    const int rank = kCluster ? (int)cluster_rank() : 0, size = kCluster ? sh.cluster : 1;
    const int c_lo = rank * sh.cols, w = max(0, min(sh.cols, n - c_lo));   // own columns
    double* Tb = sh.on_chip ? smem_tab : gscratch + (int64_t)blockIdx.x * sh.cta_doubles;   // [w + 1][hs]
    const Cand none{kNone, 0x7fffffff};
    const double eps = 1e-12;
    const long long k_neg_eps = okey(-eps);
    int rp = 0;                                              // parity of red
    // the best candidate over the CTA (all threads get it; one barrier)
    auto cta_best = [&](Cand c) {
        c = warp_best(c);
        rp ^= 1;
        if (lane == 0) red[rp][warp] = c;
        __syncthreads();
        Cand b = red[rp][0];
#pragma unroll
        for (int q = 1; q < kLpWarps; ++q) b = pick(b, red[rp][q]);
        return b;
    };

    for (int g = blockIdx.x / size; g < n_games; g += gridDim.x / size) {
        const double* Pg = P + (int64_t)g * m * n * sh.stride;
        __syncthreads();                                     // the previous game's tableau is read
        Cand lo = none;                                      // min(A): the largest negated key
        for (int k = tid; k < m * n; k += kLpThreads) lo = pick(lo, Cand{-okey(Pg[(int64_t)k * sh.stride]), k});
        lo = cta_best(lo);
        const double shift = 1.0 - okey_inv(-lo.k);
        for (int r = warp; r <= m; r += kLpWarps)
            for (int c = lane; c <= w; c += 32)
                Tb[(int64_t)c * hs + r] = r < m ? (c < w ? Pg[((int64_t)r * n + c_lo + c) * sh.stride] + shift : 1.0)
                                               : (c < w ? -1.0 : 0.0);
        for (int r = tid; r < m; r += kLpThreads) basis[r] = n + r;
        for (int c = tid; c < w; c += kLpThreads) label[c] = c_lo + c;
        __syncthreads();
        if constexpr (kCluster) {
            // before the first remote access (a CTA that has not started has no shared memory yet)
            if (!peers_run) cluster_wait();
            peers_run = true;
        }

        const int max_pivots = pivot_limit > 0 ? pivot_limit : 50 * (m + n) + 1000;
        bool done = false, bland = false;
        int degenerate = 0;
        for (int piv = 0;; ++piv) {
            const int par = piv & 1;
            // entering column: this CTA's best (ties by label: a column's label
            // is its candidate index), then the cluster's
            Cand ce = none;
            int col = 0;
            for (int c = tid; c < w; c += kLpThreads) {
                const long long k = okey(Tb[(int64_t)c * hs + m]);
                const Cand x{bland ? 0ll : -k, label[c]};
                if (k < k_neg_eps && ((x.k > ce.k) | ((x.k == ce.k) & (x.i < ce.i)))) { ce = x; col = c; }
            }
            const Cand mine = cta_best(ce);
            // the one thread whose column it is notes where it lies here
            if (mine.k != kNone && ce.k == mine.k && ce.i == mine.i) offers[par][rank].col = col;
            __syncthreads();
            const int oc = offers[par][rank].col;
            int q_rank = 0;
            if constexpr (kCluster) {
                if (mine.k != kNone)
                    for (int r = tid; r <= m; r += kLpThreads) offered[par][r] = Tb[(int64_t)oc * hs + r];
                if (tid < size)
                    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                                     peer_addr(&offers[par][rank], (uint32_t)tid)),
                                 "r"((uint32_t)(unsigned long long)mine.k), "r"((uint32_t)((unsigned long long)mine.k >> 32)),
                                 "r"((uint32_t)mine.i), "r"((uint32_t)oc)
                                 : "memory");
                cluster_sync();
                ce = none;
                for (int q = 0; q < size; ++q) {
                    const Cand o{offers[par][q].key, offers[par][q].label};
                    if ((o.k > ce.k) | ((o.k == ce.k) & (o.i < ce.i))) { ce = o; q_rank = q; }
                }
            } else {
                ce = mine;
            }
            if (ce.k == kNone) { done = true; break; }
            if (piv == max_pivots) break;                    // another pivot is needed: limit reached
            const int q = ce.i;
            const int q_col = q_rank == rank ? oc : -1;      // its column here, when this CTA owns it
            // leaving row: minimum ratio (ratios are >= 0), ties to the lowest
            // basic index; the candidate index packs (basic index, row)
            Cand cl = none;
            for (int r = tid; r <= m; r += kLpThreads) {
                double a;
                if constexpr (kCluster)
                    asm volatile("ld.shared::cluster.f64 %0, [%1];"
                                 : "=d"(a)
                                 : "r"(peer_addr(&offered[par][r], (uint32_t)q_rank))
                                 : "memory");
                else
                    a = Tb[(int64_t)oc * hs + r];
                colq[r] = a;
                if (r < m && a > eps) {
                    const double inv = 1.0 / a;
                    invs[r] = inv;
                    cl = pick(cl, Cand{-okey(quotient(Tb[(int64_t)w * hs + r], a, inv)), basis[r] * 1024 + r});
                }
            }
            cl = cta_best(cl);
            if (cl.k == kNone) break;                        // unbounded: cannot happen with B > 0
            const int p = cl.i & 1023;
            degenerate = (okey_inv(-cl.k) == 0.0) ? degenerate + 1 : 0;
            if (degenerate > 2 * (m + n)) bland = true;
            // pivot on (p, q): the scaled row p first
            const double inv = invs[p];
            for (int c = tid; c <= w; c += kLpThreads) prow[c] = c == q_col ? inv : Tb[(int64_t)c * hs + p] * inv;
            const int leaving = basis[p];
            __syncthreads();
            if (tid == 0) {
                basis[p] = q;
                if (q_col >= 0) label[q_col] = leaving;
            }
            for (int r = tid & (sh.rows - 1); r <= m; r += sh.rows) {   // sh.rows threads over rows, the rest over columns
                const double f = colq[r];
                for (int c = tid >> sh.rows_log2; c <= w; c += kLpThreads >> sh.rows_log2) {
                    double* t = Tb + (int64_t)c * hs + r;
                    if (r == p) *t = prow[c];
                    else if (c == q_col) *t = f != 0.0 ? -f * prow[c] : 0.0;
                    else if (f != 0.0) *t = fma(-f, prow[c], *t);
                }
            }
            __syncthreads();
        }
        if (!done && tid == 0 && rank == 0) atomicOr(err, ERRBIT_NOT_CONVERGED);
        // read out: z = sum q = the right side of row m; v_B = 1 / z; basic
        // variables from the right side, the others are 0; x from the reduced
        // costs of the slacks (0 for basic ones)
        const double vB = 1.0 / Tb[(int64_t)w * hs + m];
        if (rank == 0)
            for (int r = tid; r < m; r += kLpThreads) {
                const int v = basis[r];
                if (v < n) y_out[(int64_t)g * n + v] = Tb[(int64_t)w * hs + r] * vB;
                else x_out[(int64_t)g * m + v - n] = 0.0;
            }
        for (int c = tid; c < w; c += kLpThreads) {
            const int v = label[c];
            if (v < n) y_out[(int64_t)g * n + v] = 0.0;
            else x_out[(int64_t)g * m + v - n] = Tb[(int64_t)c * hs + m] * vB;
        }
        if (tid == 0 && rank == 0) val_out[g] = vB - shift;
        if constexpr (kCluster) cluster_sync();              // nobody reads this game's offers any more
    }
}

}  // namespace

int fp_grid(int32_t n_games, int n_sm) { return n_games < 4 * n_sm ? n_games : 4 * n_sm; }

cudaError_t launch_fictitious_play(const double* P, int32_t G, int32_t m, int32_t n, int32_t stride,
                                   int64_t T, double* x, double* y, double* bounds, int n_sm,
                                   cudaStream_t s) {
    const int ld = n | 1;
    const int64_t bytes = (int64_t)m * ld * 8;
    const bool on_chip = bytes <= kSmemLimit;
    const size_t dyn = on_chip ? (size_t)bytes : 0;
    // a warp per 32 rows and per 32 columns, at most kFpWarps a side
    const int per = ((m > n ? m : n) + 32 * kFpWarps - 1) / (32 * kFpWarps);
    auto warps = [&](int d) { return (d + 32 * per - 1) / (32 * per); };
    const int wr = warps(m), wc = warps(n);
    const int most = wr > wc ? wr : wc;
    auto pick_kernel = [&](auto where) {
        constexpr FpTable T = decltype(where)::value;
        return per > 2     ? fictitious_play_kernel<T, kFpPer, 8>
               : per > 1   ? fictitious_play_kernel<T, 2, 8>     // (fp64 additions of absent rows cost as much as others)
               : most <= 1 ? fictitious_play_kernel<T, 1, 1>
               : most <= 2 ? fictitious_play_kernel<T, 1, 2>
               : most <= 4 ? fictitious_play_kernel<T, 1, 4>
                           : fictitious_play_kernel<T, 1, 8>;
    };
    auto kern = on_chip ? pick_kernel(std::integral_constant<FpTable, kFpOnChip>{})
                : (int64_t)stride * n <= INT32_MAX ? pick_kernel(std::integral_constant<FpTable, kFpNear>{})
                                                   : fictitious_play_kernel<kFpFar, kFpPer, 8>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e != cudaSuccess) return e;
    kern<<<fp_grid(G, n_sm), 32 * (wr + wc), dyn, s>>>(P, G, m, n, stride, T, wr, x, y, bounds);
    return cudaGetLastError();
}

cudaError_t launch_aggregate(const double* P, int32_t G, int32_t m, int32_t n, int32_t stride,
                             const double* x, const double* y, double* ay, double* xa, double* val,
                             int n_sm, cudaStream_t s) {
    int32_t lanes = 1;
    while (lanes < n && lanes < 32) lanes *= 2;
    // Small tables come many at a time: fewer warps a game, more games at once (16
    // warps and a warp per row throughout: 10,000 games 2 x 2 91 us, 60 x 10 409, 45 x 45
    // 421; a thread per row and column in 8 warps: 44, 129, 375; so: 19, 72, 198). Wide
    // rows want all lanes; others share a warp, whose fp64 pipe (2 lanes a clock and SM)
    // would otherwise spend five additions a row on combining lanes (one game 100 x 100
    // 12.6 us, 32 lanes a row 20.5; 2,000 x 2,000 4,160 us with 8 lanes, 2,910 with 32).
    const int64_t size = (int64_t)m * n;
    void (*kern)(const double*, int32_t, int32_t, int32_t, int32_t, int32_t, const double*, const double*, double*,
                 double*, double*);
    const int W = n > 256 || size > 4096 ? 16 : size > 1024 ? 8 : size > 256 ? 4 : 2;
    if (lanes <= 16)
        kern = W == 2 ? aggregate_kernel<2, 0> : W == 4 ? aggregate_kernel<4, 0> : W == 8 ? aggregate_kernel<8, 0>
                                                                                 : aggregate_kernel<16, 0>;
    else
        kern = n > 256  ? aggregate_kernel<16, 32>
               : W == 2 ? aggregate_kernel<2, 8>
               : W == 4 ? aggregate_kernel<4, 8>
               : W == 8 ? aggregate_kernel<8, 8>
                        : aggregate_kernel<16, 8>;
    const int64_t most = (int64_t)n_sm * (W == 2 ? 32 : 64 / W);               // resident blocks
    kern<<<(unsigned)(G < most ? G : most), 32 * W, 0, s>>>(P, G, m, n, stride, lanes, x, y, ay, xa, val);
    return cudaGetLastError();
}

// The CTAs of a game: a cluster of 8, 4 or 2 while the games leave SMs free (an
// eight-CTA cluster needs eight SMs of one GPC: 15 clusters at once were seen on
// this part) and the update is long enough: below 40 x 40 the cluster's barrier
// and remote loads (about 1,000 cycles a pivot) cost more than they save.
static LpShape lp_shape(int32_t n_games, int32_t m, int32_t n, int32_t stride, int n_sm) {
    LpShape s{};
    s.m = m;
    s.n = n;
    s.stride = stride;
    s.cluster = 1;
    if ((int64_t)m * n >= 1600)
        while (s.cluster < kLpMaxCluster && (int64_t)n_games * s.cluster * 2 <= n_sm - n_sm / 5) s.cluster *= 2;
    while (s.cluster > 1 && n < 2 * s.cluster) s.cluster /= 2;
    s.cols = (n + s.cluster - 1) / s.cluster;
    s.hs = (m + 1) | 1;
    s.rows = 1;
    while (s.rows < 128 && s.rows < m + 1) {
        s.rows *= 2;
        ++s.rows_log2;
    }
    s.cta_doubles = (int64_t)(s.cols + 1) * s.hs;
    s.on_chip = s.cta_doubles * 8 <= kSmemLimit ? 1 : 0;
    return s;
}

static int lp_grid(int32_t n_games, int n_sm) { return n_games < n_sm ? n_games : n_sm; }

int64_t lp_scratch_bytes(int32_t n_games, int32_t m, int32_t n, int n_sm) {
    const LpShape s = lp_shape(n_games, m, n, 1, n_sm);
    return s.on_chip ? 0 : (int64_t)lp_grid(n_games, n_sm) * s.cluster * s.cta_doubles * 8;
}

cudaError_t launch_lp_nash(const double* P, int32_t G, int32_t m, int32_t n, int32_t stride,
                           double* x, double* y, double* val, double* scratch, int32_t pivot_limit,
                           int* err, int n_sm, cudaStream_t s) {
    const LpShape sh = lp_shape(G, m, n, stride, n_sm);
    const size_t dyn = sh.on_chip ? (size_t)sh.cta_doubles * 8 : 0;
    auto kern = sh.cluster > 1 ? lp_nash_kernel<true> : lp_nash_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(lp_grid(G, n_sm) * sh.cluster));
    cfg.blockDim = dim3(kLpThreads);
    cfg.dynamicSmemBytes = dyn;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)sh.cluster;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kern, P, G, sh, x, y, val, scratch, pivot_limit, err);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace malib

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
using namespace malib;

namespace {

// Device memory of the context's own device.
bool dev_ptr(int device, const void* p) { return p && ptr_where(p, device) == kPtrHere; }

int check_table(malib_ctx* ctx, int device, const double* payoff, int32_t G, int32_t m, int32_t n,
                int32_t stride, int32_t max_dim) {
    if (G < 0) return ctx_fail(ctx, MALIB_EINVAL, "n_games < 0");
    if (m < 1 || n < 1 || m > max_dim || n > max_dim)
        return ctx_fail(ctx, m < 1 || n < 1 ? MALIB_EINVAL : MALIB_EUNSUPPORTED,
                        "payoff table dimensions outside 1..limit (see malib.h)");
    if (stride < 1) return ctx_fail(ctx, MALIB_EINVAL, "stride < 1");
    if ((int64_t)G * m * n * stride > ((int64_t)1 << 40))
        return ctx_fail(ctx, MALIB_EINVAL, "payoff table too large");
    if (G > 0 && !dev_ptr(device, payoff)) return ctx_fail(ctx, MALIB_EINVAL, "payoff must be device memory of the context's device");
    return MALIB_OK;
}

int launched(malib_ctx* ctx, cudaError_t e, int n_launch) {
    if (e != cudaSuccess) return ctx_fail(ctx, MALIB_ECUDA, cudaGetErrorString(e));
    ctx_count_launches(ctx, n_launch);
    return MALIB_OK;
}

}  // namespace

extern "C" int malib_meta_fictitious_play(malib_ctx* ctx, const double* payoff, int32_t n_games,
                                          int32_t m, int32_t n, int32_t stride, int64_t iters,
                                          double* x_out, double* y_out, double* bounds_out) {
    CtxView v;
    if (!ctx_view(ctx, &v)) return MALIB_EINVAL;
    int r = check_table(ctx, v.device, payoff, n_games, m, n, stride, kFpMaxDim);
    if (r != MALIB_OK) return r;
    if (iters < 1) return ctx_fail(ctx, MALIB_EINVAL, "iters must be >= 1");
    if (n_games == 0) return MALIB_OK;
    if (!dev_ptr(v.device, x_out) || !dev_ptr(v.device, y_out) || !dev_ptr(v.device, bounds_out))
        return ctx_fail(ctx, MALIB_EINVAL, "x_out, y_out and bounds_out must be device memory of the context's device");
    DevSel d(v.device);
    if (!d.ok) return ctx_fail(ctx, MALIB_ECUDA, "cannot select the context's device");
    return launched(ctx, launch_fictitious_play(payoff, n_games, m, n, stride, iters, x_out, y_out,
                                                bounds_out, v.n_sm, v.stream), 1);
}

extern "C" int malib_meta_aggregate(malib_ctx* ctx, const double* payoff, int32_t n_games,
                                    int32_t m, int32_t n, int32_t stride, const double* x,
                                    const double* y, double* row_payoff_out,
                                    double* col_payoff_out, double* value_out) {
    CtxView v;
    if (!ctx_view(ctx, &v)) return MALIB_EINVAL;
    int r = check_table(ctx, v.device, payoff, n_games, m, n, stride, 1 << 20);
    if (r != MALIB_OK) return r;
    if (n_games == 0) return MALIB_OK;
    if (!dev_ptr(v.device, x) || !dev_ptr(v.device, y) || !dev_ptr(v.device, row_payoff_out) ||
        !dev_ptr(v.device, col_payoff_out) || !dev_ptr(v.device, value_out))
        return ctx_fail(ctx, MALIB_EINVAL, "mixtures and outputs must be device memory of the context's device");
    DevSel d(v.device);
    if (!d.ok) return ctx_fail(ctx, MALIB_ECUDA, "cannot select the context's device");
    return launched(ctx, launch_aggregate(payoff, n_games, m, n, stride, x, y, row_payoff_out,
                                          col_payoff_out, value_out, v.n_sm, v.stream), 1);
}

extern "C" int malib_meta_lp_nash_ex(malib_ctx* ctx, const double* payoff, int32_t n_games,
                                     int32_t m, int32_t n, int32_t stride, int32_t max_pivots,
                                     double* x_out, double* y_out, double* value_out) {
    CtxView v;
    if (!ctx_view(ctx, &v)) return MALIB_EINVAL;
    int r = check_table(ctx, v.device, payoff, n_games, m, n, stride, 512);
    if (r != MALIB_OK) return r;
    if (max_pivots < 0) return ctx_fail(ctx, MALIB_EINVAL, "max_pivots < 0");
    if (n_games == 0) return MALIB_OK;
    if (!dev_ptr(v.device, x_out) || !dev_ptr(v.device, y_out) || !dev_ptr(v.device, value_out))
        return ctx_fail(ctx, MALIB_EINVAL, "x_out, y_out and value_out must be device memory of the context's device");
    DevSel d(v.device);
    if (!d.ok) return ctx_fail(ctx, MALIB_ECUDA, "cannot select the context's device");
    double* scratch = nullptr;
    const int64_t bytes = lp_scratch_bytes(n_games, m, n, v.n_sm);
    if (bytes > 0) {
        void* p = nullptr;
        r = ctx_scratch(ctx, bytes, &p);
        if (r != MALIB_OK) return r;
        scratch = static_cast<double*>(p);
    }
    return launched(ctx, launch_lp_nash(payoff, n_games, m, n, stride, x_out, y_out, value_out,
                                        scratch, max_pivots, v.err, v.n_sm, v.stream), 1);
}

extern "C" int malib_meta_lp_nash(malib_ctx* ctx, const double* payoff, int32_t n_games, int32_t m,
                                  int32_t n, int32_t stride, double* x_out, double* y_out,
                                  double* value_out) {
    return malib_meta_lp_nash_ex(ctx, payoff, n_games, m, n, stride, 0, x_out, y_out, value_out);
}
