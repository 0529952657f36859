// Stage 2 of the emulator: the chain-rule sampler (arXiv:2511.14923, Sec. "The
// sampling algorithm", Sec. Methods and App. "Approximating marginals efficiently
// with a chain rule"), for a batch of S samples drawn in lockstep.
//
// The rule. For bits x_1..x_M (bit n = mode n-1), Eq. probs_corr_cumulants_3
// truncated at order K expands p(x_n..x_1) over the spin cumulants kappa(R+{n}),
// |R| < K, times marginals p(x_{[n-1]-R}) that are approximated by tables:
//   P[a] = p(x_a..x_1),  Pp[a][b] = p+(x_a..x_b),  P1[a][e] = p1(x_a..~x_e..x_1),
//   P2[a][e][d] = p2(x_a..~x_e..~x_d..x_1)  (K = 5 only),
// filled by truncated forms of the same rule: K = 3 single elision (Eq. methprob,
// Eq. b, Eq. a), K = 5 double elision (Eq. probade, Eq. probpartialade,
// Eq. probelidedade, Eq. probdoubleelidedade; orders 3, 3, 2 for p+, p1, p2 unless
// the caller lowers them), K = 4 the same without the |R| = 4 term (orders
// 2, 2, 1 by default). Boundary cases: P[0] = 1, an empty p+ range is 1,
// P1[a][a] = P[a-1], P2[a][a][d] = P1[a-1][d].
//
// Scaling. Each table entry over a variable set A is stored times prod_{v in A}
// s_v, with s_v = exp(H_v) and H_v the click entropy of mode v - 1 (from
// kappa({v})), so that a typical sample's values stay near 1 instead of
// decaying like e^{-sum H}. Writing hs_v = s_v / 2 and kappa'(S) = kappa(S)
// prod_{v in S} hs_v, every rule keeps its form with the factors 2^{-(|R|+1)}
// absorbed: the term of R becomes chi kappa'(R + {n}) times the scaled
// marginal, and the leading 1/2 (1 + gamma_n) becomes hs_n + chi_n kappa'_n.
// Then p(x_n = 0) and p(x_n = 1) are proportional to hs_n P~[n-1] +- B~, with B~
// the scaled odd part, and the probability of a bitstring is
// P~[M] exp(-sum_v H_v).
//
// Factorisation of the expensive terms. The terms of the bias B that reach back
// to a table row j - 1 through P2[j-1] (or P1[j-1] for K = 3) are sums over
// pairs (or single indices) below j of kappa(.., j, i, m) W_j, with
// W_j(e, d) = chi_e chi_d P2~[j-1][e][d] (K = 3: W_j(d) = chi_d P1~[j-1][d]).
// W_j only involves bits below j, so right after bit j - 1 is drawn one matrix
// product per step,
//   Z_j[row][s] = sum_r kappa[base(row) + r] W_j[r][s],
// evaluates those sums for every later (i, m) at once; in colex order the
// kappa entries of one row are contiguous, so each row is a segment of the
// table. The rows at step j are (K = 5) the order-3 set {., ., j} (used at this
// step), the order-4 sets {., ., j, n}, the order-5 sets {., ., j, i, m} and the
// pairs below j of the order-3 sets {., ., n} (X_j(n), the part of the p1 update
// whose largest index is the elided one);
// (K = 3) the order-2 set {., j} and the order-3 sets {., j, n}. At step n the
// bias then only combines stored Z values with p+ factors:
//   K = 5: B~ = kappa'_n P~[n-1] + sum_i kappa'(i,n) chi_i P1~[n-1][i] + G3
//             + sum_{i<n} chi_i Pp~[n-1][i+1] (Z3_i(n) + sum_{j<i} chi_j Pp~[i-1][j+1] Z5_j(i,n))
//   K = 3: B~ = kappa'_n P~[n-1] + G2 + sum_{i<n} chi_i Pp~[n-1][i+1] Z_i(n)
// (chi_n taken as +1: every term but hs_n P~[n-1] is odd in x_n; kappa' in every
// product row).
//
// Drawing. x_n = 0 when u_n < q0 = max(p0, 0) / (max(p0, 0) + max(p1, 0))
// (1/2 if both are <= 0); P[n] keeps the chosen branch unclipped.
//
// Layout. The samples form groups of SG; every per-sample table of a group is
// [entry][SG] (sample fastest, see SG), so a warp always touches consecutive
// samples of one entry: 32 VW of them, VW per lane.
#include <cstdint>
#include <cstdio>
#include <cstdlib>

#include "gbs.h"
#include "gbs_common.cuh"
#include "gbs_sampler.cuh"

namespace gbs {
namespace smp {


__host__ __device__ __forceinline__ uint64_t cb(int n, int k) { return binom(n, k); }

// Entry indices (variables 1-based).
__host__ __device__ __forceinline__ uint64_t i_pp(int a, int b) { return cb(a, 2) + (uint64_t)(b - 1); }       // 1<=b<=a
__host__ __device__ __forceinline__ uint64_t i_p1(int a, int e) { return cb(a - 1, 2) + (uint64_t)(e - 1); }   // 1<=e<a
__host__ __device__ __forceinline__ uint64_t i_p2(int a, int e, int d) {                                          // d<e<a
    return cb(a - 1, 3) + cb(e - 1, 2) + (uint64_t)(d - 1);
}
__host__ __device__ __forceinline__ uint64_t i_z(int t, int n) { return cb(n - 1, 2) + (uint64_t)(t - 1); }     // t<n
__host__ __device__ __forceinline__ uint64_t i_z5(int t, int i, int m) {                                         // t<i<m
    return cb(m - 1, 3) + cb(i - 1, 2) + (uint64_t)(t - 1);
}

// Samples per group. The per-sample tables of one group of SG consecutive samples
// form one block ([entry][SG], sample fastest; Args::tab, gs elements per block),
// so an entry's row is 512 bytes in FP32 and consecutive entries are neighbours
// in memory. (With one row of all S samples per entry, neighbouring entries lay
// 4 S bytes apart: at S = 8192 every warp's load opened another DRAM page.)
constexpr int SG = 128;

// First entry of each table inside a group's block.
struct Tabs {
    size_t chi, P, Pp, P1, P2, Z, Z5, G, Y, X, CA, CB, CC, T, R2, entries;
};

template <class R>
struct Args {
    const R *kap;          // spin cumulants, orders 1..K, gbs.h layout
    uint64_t off[6];       // order offsets of the cumulant table
    int M, K, S, opp, op1, op2;
    R *tab;                // the groups' tables
    size_t gs;             // elements per group block (Tabs::entries x SG)
    Tabs o;
    R *W;
    const R *kb;           // kappa(i, n) regrouped for p2_block_kernel, or null (p2_kernel then walks every row itself)
    float *At;             // tensor-core product: the step's rows, split and tiled (operands_kernel)
    const R *lead;         // per-variable pairs (kappa'({v}), hs[v]) at lead[2v], lead[2v+1]
    const double *H;       // per-variable log scale ln s_v (the click entropy of mode v - 1)
    unsigned *status;      // status word (ST_* bits), first bytes of the workspace
    int use_tc;            // FP32: step product on the tensor cores
    int wait_limit;        // polls of an mbarrier before a wait gives up (ST_TIMEOUT)
    int no_loads;          // test hook: the step product issues no copies (its first wait runs out)
    uint32_t *bw;          // spins as bits: word w of sample s at bw[w * S + s], bit v & 31 = x_v
    const double *u;       // [n_samples][M] uniforms (chunk base)
    const uint8_t *force;  // [n_samples][M] or null
    uint8_t *bits;         // [n_samples][M]
    double *q0;            // [n_samples][M] or null
    int n_valid;           // samples of this chunk that are real
};

// The tables of one group, each shifted to the calling thread's (first) sample.
template <class R>
struct Grp {
    R *chi, *P, *Pp, *P1, *P2, *Z, *Z5, *G, *Y, *X, *CA, *CB, *CC, *T, *R2;
    __device__ __forceinline__ Grp(const Args<R> &a, int s) {
        R *b = a.tab + (size_t)(s / SG) * a.gs + (s % SG);
        chi = b + a.o.chi * SG;
        P = b + a.o.P * SG;
        Pp = b + a.o.Pp * SG;
        P1 = b + a.o.P1 * SG;
        P2 = b + a.o.P2 * SG;
        Z = b + a.o.Z * SG;
        Z5 = b + a.o.Z5 * SG;
        G = b + a.o.G * SG;
        Y = b + a.o.Y * SG;
        X = b + a.o.X * SG;
        CA = b + a.o.CA * SG;
        CB = b + a.o.CB * SG;
        CC = b + a.o.CC * SG;
        T = b + a.o.T * SG;
        R2 = b + a.o.R2 * SG;
    }
};

// Spins of one sample read from its packed bits; the current 32-bit word is
// cached, so a loop over ascending variables loads one word per 32 of them.
template <class R>
struct Spins {
    const uint32_t *bw;
    int S, s, w;
    uint32_t cur;
    __device__ Spins(const Args<R> &a, int s_) : bw(a.bw), S(a.S), s(s_), w(-1), cur(0) {}
    __device__ __forceinline__ R operator()(int v) {
        if ((v >> 5) != w) {
            w = v >> 5;
            cur = bw[(size_t)w * S + s];
        }
        return (cur >> (v & 31)) & 1u ? R(-1) : R(1);
    }
};

// (kappa'({n}), hs_n) in one vector load: the leading coefficient of every rule
// at step n is hs_n + chi_n kappa'({n}).
template <class R>
struct Pair2;
template <>
struct Pair2<float> {
    using T = float2;
};
template <>
struct Pair2<double> {
    using T = double2;
};
template <class R>
__device__ __forceinline__ typename Pair2<R>::T lead(const Args<R> &a, int n) {
    return reinterpret_cast<const typename Pair2<R>::T *>(a.lead)[n];
}

// kappa of the sorted variable set (v_1 < .. < v_d), 1-based.
template <class R>
__device__ __forceinline__ R k1(const Args<R> &a, int n) { return a.kap[a.off[1] + (n - 1)]; }

// Pair rank -> (hi, lo), hi > lo >= 0 (colex: rank = C(hi, 2) + lo). The root
// estimate is taken in FP32 (GB300's FP64 pipe is narrow and every lane of the
// table kernels decodes its pair) and corrected exactly by the loops.
__device__ __forceinline__ void pair_of(uint64_t r, int &hi, int &lo) {
    int c = (int)(0.5f * (1.f + sqrtf(1.f + 8.f * (float)r)));
    if (c < 1) c = 1;
    while (cb(c, 2) > r) --c;
    while (cb(c + 1, 2) <= r) ++c;
    hi = c;
    lo = (int)(r - cb(c, 2));
}

// ---------------------------------------------------------------- step t: Z rows

// Row q of the product at step t: kbase = offset of its segment in the cumulant
// table, dst = the entry of the group's block its result goes to.
__device__ __forceinline__ void zrow(int K, int M, int t, uint64_t q, const uint64_t *off, const Tabs &o,
                                     uint64_t &kbase, uint64_t &dst) {
    if (K == 3) {
        if (q == 0) {
            kbase = off[2] + cb(t - 1, 2);
            dst = o.G;
        } else {
            const int n = t + (int)q;
            kbase = off[3] + cb(n - 1, 3) + cb(t - 1, 2);
            dst = o.Z + i_z(t, n);
        }
        return;
    }
    if (q == 0) {
        kbase = off[3] + cb(t - 1, 3);
        dst = o.G;
    } else if (q <= (uint64_t)(M - t)) {
        const int n = t + (int)q;
        kbase = off[4] + cb(n - 1, 4) + cb(t - 1, 3);
        dst = o.Z + i_z(t, n);
    } else if (q <= 2 * (uint64_t)(M - t)) {
        // the pairs below t of the order-3 set {., ., n}: X_t(n) for the p1 update
        const int n = t + (int)(q - (uint64_t)(M - t));
        kbase = off[3] + cb(n - 1, 3);
        dst = o.X + i_z(t, n);
    } else {  // K = 5 only
        int hi, lo;
        pair_of(q - 1 - 2 * (uint64_t)(M - t), hi, lo);
        const int i = t + 1 + lo, m = t + 1 + hi;
        kbase = off[5] + cb(m - 1, 5) + cb(i - 1, 4) + cb(t - 1, 3);
        dst = o.Z5 + i_z5(t, i, m);
    }
}

// Blocks with the samples on the slow grid axis: y, and z beyond the 65535 blocks y
// may have (FP64 batches of 2^21, 32 samples a block). The number of blocks, a
// multiple of 4 (S is one of 128), halves evenly.
static dim3 sample_grid(unsigned x, unsigned blocks) {
    unsigned z = 1;
    for (; blocks > 65535; blocks /= 2) z *= 2;
    return dim3(x, blocks, z);
}
__device__ __forceinline__ int sample_block() { return (int)(blockIdx.z * gridDim.y + blockIdx.y); }

// W_t[r][s], the inner operand of the step-t product: K = 5, pair r = (e, d) of
// bits below t, chi_e chi_d P2~[t-1][e][d]; K = 3, d = r + 1, chi_d P1~[t-1][d].
// Grid: (samples / ETB, entries); the entry index is uniform in a block.
constexpr int ETB = 64;  // threads per block of the per-(entry, sample) kernels

template <class R, int K>
__global__ void __launch_bounds__(ETB) w_kernel(Args<R> a, int t, int D) {
    await_previous();
    if constexpr (K == 3) release_next();
    const int s = blockIdx.x * ETB + threadIdx.x;
    const size_t S = (size_t)a.S;
    // this block's share of r = 0 .. D-1, walked in order
    const int per = (D + (int)gridDim.y - 1) / (int)gridDim.y;
    const int r0 = blockIdx.y * per, r1 = r0 + per < D ? r0 + per : D;
    if (r0 >= r1) return;
    Spins<R> sp(a, s);
    const Grp<R> tb(a, s);
    R *W = a.W + s;
    if (K == 3) {
        // W_t(d) = chi_d P1~[t-1][d], d = r + 1; d = t - 1 -> P~[t-2]
        const R *q = tb.P1 + (t >= 3 ? i_p1(t - 1, 1) : 0) * SG;
        for (int r = r0; r < r1; ++r) {
            const int d = r + 1;
            const R v = d == t - 1 ? tb.P[(size_t)(t - 2) * SG] : q[(size_t)r * SG];
            W[(size_t)r * S] = v * sp(d);
        }
        return;
    }
    // K = 5: pair r = (e, d); for e < t - 1 the p2 row t - 1 holds the same pairs in
    // the same order (offset C(t-2, 3)); e = t - 1 comes from P1~[t-2][d] (P~[t-3]
    // when d = t - 2)
    int hi, lo;
    pair_of((uint64_t)r0, hi, lo);
    int e = hi + 1, d = lo + 1;
    Spins<R> sd(a, s);
    const uint64_t rowlen = cb(t - 2, 2);
    const R *q2 = tb.P2 + (t >= 4 ? cb(t - 2, 3) : 0) * SG;
    for (int r = r0; r < r1; ++r) {
        R v;
        if ((uint64_t)r < rowlen) v = q2[(size_t)r * SG];
        else v = d == t - 2 ? tb.P[(size_t)(t - 3) * SG] : tb.P1[i_p1(t - 2, d) * SG];
        W[(size_t)r * S] = v * sp(e) * sd(d);
        if (++d == e) {
            ++e;
            d = 1;
        }
    }
}

// Z[row][s] = sum_{r < D} kappa[kbase(row) + r] W_t[r][s] for rows [0, rows) and
// all samples: one chain of FMAs per result, in ascending r, whatever the tile.
// 256 threads, a tile of 16 T x 16 T results per CTA, T x T per thread (two 4-wide
// halves each way when T = 8), BK inner entries per stage with the next stage
// prefetched into registers. Late steps have few rows and long chains, so the
// tile is chosen by the CTAs it leaves (launch_zgemm).
template <class R, int K, int T>
__global__ void __launch_bounds__(256) zgemm_kernel(Args<R> a, int t, uint64_t rows, int D) {
    await_previous();
    if constexpr (K == 3) release_next();
    constexpr int BT = 16 * T, BK = T == 1 ? 16 : 8;
    constexpr int E = BT * BK / 256;  // elements of each operand per thread per stage
    __shared__ __align__(16) R As[2][BK][BT];
    __shared__ __align__(16) R Bs[2][BK][BT];
    __shared__ uint64_t kb[BT];
    __shared__ uint64_t dst[BT];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const uint64_t m0 = (uint64_t)blockIdx.x * BT;
    const int s0 = sample_block() * BT;
    for (int m = tid; m < BT; m += 256) {
        const uint64_t q = m0 + m;
        if (q < rows) zrow(K, a.M, t, q, a.off, a.o, kb[m], dst[m]);
        else kb[m] = ~0ull;
    }
    __syncthreads();
    // stage loaders: A element e = tid + 256 q -> (row e / BK, inner e % BK);
    // B: E consecutive samples of inner row tid / (BT / E)
    const int bk = tid / (BT / E), bs = (tid % (BT / E)) * E;
    R ra[E], rb[E];
    auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < E; ++q) {
            const int e = tid + 256 * q, m = e / BK, k = e % BK;
            ra[q] = (kb[m] != ~0ull && k0 + k < D) ? a.kap[kb[m] + k0 + k] : R(0);
        }
        const R *w = a.W + (size_t)(k0 + bk) * a.S + s0 + bs;
#pragma unroll
        for (int q = 0; q < E; ++q) rb[q] = (k0 + bk < D) ? w[q] : R(0);
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int q = 0; q < E; ++q) {
            const int e = tid + 256 * q;
            As[buf][e % BK][e / BK] = ra[q];
        }
#pragma unroll
        for (int q = 0; q < E; ++q) Bs[buf][bk][bs + q] = rb[q];
    };
    auto at = [](int th, int i) { return T == 8 ? (i < 4 ? 0 : BT / 2) + th * 4 + (i & 3) : th * T + i; };
    R acc[T][T];
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
        for (int j = 0; j < T; ++j) acc[i][j] = R(0);
    load(0);
    store(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < D; k0 += BK) {
        const bool more = k0 + BK < D;
        if (more) load(k0 + BK);
#pragma unroll
        for (int k = 0; k < BK; ++k) {
            R av[T], bv[T];
#pragma unroll
            for (int i = 0; i < T; ++i) av[i] = As[buf][k][at(ty, i)];
#pragma unroll
            for (int j = 0; j < T; ++j) bv[j] = Bs[buf][k][at(tx, j)];
#pragma unroll
            for (int i = 0; i < T; ++i)
#pragma unroll
                for (int j = 0; j < T; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
        }
        if (more) {
            store(buf ^ 1);
            __syncthreads();
            buf ^= 1;
        }
    }
    R *const out0 = a.tab + (size_t)(s0 / SG) * a.gs + s0 % SG;  // the tile lies in one group
#pragma unroll
    for (int i = 0; i < T; ++i) {
        const int m = at(ty, i);
        if (kb[m] == ~0ull) continue;
#pragma unroll
        for (int j = 0; j < T; ++j) out0[dst[m] * SG + at(tx, j)] = acc[i][j];
    }
}

// FP32: the largest of the 128, 64 and 32-wide tiles that leaves two CTAs for
// every multiprocessor. FP64: the FP64 pipe (2 FMAs per clock) binds with any
// tile, so only the split counts: 32 wide from eight CTAs per multiprocessor on
// (the last wave then costs little), else 16 wide. At M = 100, K = 5, 256 samples
// the 64-wide FP64 tiles used before left 56-80 CTAs for 152 multiprocessors at
// the heaviest steps: 179 ms a call, 31 ms being the pipe's.
template <class R, int K>
static cudaError_t launch_zgemm(const Args<R> &a, int t, uint64_t rows, int D, int sms, cudaStream_t st) {
    auto ctas = [&](int bt) { return (rows + bt - 1) / bt * (uint64_t)(a.S / bt); };
    auto grid = [&](int bt) { return sample_grid((unsigned)((rows + bt - 1) / bt), (unsigned)(a.S / bt)); };
    cudaError_t e;
    if constexpr (sizeof(R) == 4) {
        if (ctas(128) >= 2 * (uint64_t)sms) e = launch_next(K == 3, zgemm_kernel<R, K, 8>, grid(128), 256, 0, st, a, t, rows, D);
        else if (ctas(64) >= 2 * (uint64_t)sms) e = launch_next(K == 3, zgemm_kernel<R, K, 4>, grid(64), 256, 0, st, a, t, rows, D);
        else e = launch_next(K == 3, zgemm_kernel<R, K, 2>, grid(32), 256, 0, st, a, t, rows, D);
    } else {
        if (ctas(32) >= 8 * (uint64_t)sms) e = launch_next(K == 3, zgemm_kernel<R, K, 2>, grid(32), 256, 0, st, a, t, rows, D);
        else e = launch_next(K == 3, zgemm_kernel<R, K, 1>, grid(16), 256, 0, st, a, t, rows, D);
    }
    return e;
}

// ---------------------------------------------------------------- step product on the tensor cores
// FP32 calls with a batch that is a multiple of 256 run the step product on the
// 5th-generation tensor cores: tcgen05.mma kind::tf32 with the 3-term split
// x = hi + lo (hi, lo TF32), Z = Ahi Bhi + Ahi Blo + Alo Bhi accumulated in FP32
// in tensor memory (the dropped Alo Blo term is ~2^-22 relative). A CTA of 128
// threads owns 128 rows x 256 samples. W arrives from operands_kernel already split
// and laid out as the MMA's K-major core matrices (8 rows x 16 bytes, no
// swizzle), one contiguous block per TC_KC-wide K chunk and sample tile, and
// is brought in by one TMA bulk copy per chunk; the rows (cumulant segments)
// arrive the same way from operands_kernel. One elected thread issues the MMAs. A
// ring of TC_NS stages, each with a "full" mbarrier (the bulk copies' bytes) and
// an "empty" one (the MMAs' commit), keeps TC_NS - 1 chunks loading while the
// MMAs of one run; the ring takes 96 KB of shared memory, so two CTAs share a
// multiprocessor (and its 512 tensor-memory columns) and one's epilogue
// overlaps the other's MMAs. Every wait is bounded; one that runs out sets ST_TIMEOUT in the status
// word.
constexpr int TC_M = 128, TC_N = 256, TC_KC = 8;
constexpr int TC_ACH = TC_M * TC_KC;            // floats of one A copy (hi or lo) of one chunk
constexpr int TC_BCH = TC_N * TC_KC;            // floats of one B copy of one chunk
constexpr int TC_AB = TC_M * TC_KC * 4;         // bytes of one A copy per stage (4 KB)
constexpr int TC_NS = 4, TC_NS_DEEP = 8;         // stages of the ring, of TN samples (see launch_ztc)
constexpr int TC_NARROW = 64;
constexpr int tc_stage(int tn) { return 2 * TC_AB + 2 * tn * TC_KC * 4; }  // A hi, A lo, B hi, B lo
constexpr int tc_smem(int ns, int tn) { return ns * tc_stage(tn) + 256; }  // then 2 x 8 mbarriers, TMEM slot, flag
// instruction descriptor: D f32, A and B tf32, both K-major, N = n, M = 128
constexpr uint32_t tc_idesc(int n) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// byte offset of element (row r, inner k) of an operand copy of one chunk
__device__ __forceinline__ uint32_t tc_off(int r, int k) {
    const int core = (r >> 3) * (TC_KC / 4) + (k >> 2);  // core matrix: 8-row group, then 4-wide K slice
    return (uint32_t)((core * 8 + (r & 7)) * 16 + (k & 3) * 4);
}

// shared-memory matrix descriptor: K-major, no swizzle; leading byte offset 128
// (next core matrix along K), stride byte offset 32 TC_KC (next group of 8 rows)
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)((32 * TC_KC) >> 4) << 32) |
           ((uint64_t)1 << 46);
}

__device__ __forceinline__ float to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

__device__ __forceinline__ void mbar_init(uint64_t *b, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

// Bounded wait for phase `parity` of the mbarrier: at most `limit` polls
// (try_wait may itself suspend the thread briefly); false if it did not complete.
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t parity, int limit) {
    for (int it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(smem_u32(b)), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// TMA bulk copies global -> shared that complete their bytes on an mbarrier;
// the expected byte count is announced once per phase.
__device__ __forceinline__ void mbar_expect(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_bulk(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

template <int TN>
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}" ::"r"(d),
        "l"(a), "l"(b), "r"(tc_idesc(TN)), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void tc_commit(uint64_t *b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(b))
                 : "memory");
}

// 32 consecutive accumulator columns of this thread's lane
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// W_t split into TF32 hi / lo in the tensor-core tile layout: element (r, s),
// r < KC ceil(D / KC) (zero beyond D; KC = TC_KC inner entries per chunk), at
// float offset ((c nsb + sb) 2 + part) 256 KC + tc_off(s % 256, r % KC) / 4,
// c = r / KC, sb = s / 256, nsb = S / 256. A thread forms four consecutive r (one 16-byte
// row of a core matrix) of one sample, so 8 consecutive samples write one
// 128-byte line. Block (bx, by) of (samples / PREP, ny): quads by, by + ny, ...
constexpr int PREP = 128;  // threads of the operand kernels
template <int K>
__device__ __forceinline__ void w_operand(const Args<float> &a, int t, int D, int bx, int by, int ny) {
    const int s = bx * PREP + threadIdx.x;
    const int Dp = (D + TC_KC - 1) / TC_KC * TC_KC;
    const int nsb = a.S / TC_N, sb = s / TC_N, sl = s % TC_N;
    Spins<float> sp(a, s), sd(a, s);
    // K = 4, 5: pair r = (e, d) with e < t - 1 is entry C(t-2, 3) + r of the p2
    // table (row t - 1 lists its pairs in colex order); e = t - 1 reads P1~[t-2][d]
    const Grp<float> tb(a, s);
    const uint64_t rowlen = K == 3 ? 0 : cb(t - 2, 2);
    const float *q2 = tb.P2 + (K != 3 && t >= 4 ? cb(t - 2, 3) : 0) * SG;
    for (int qd = by; qd < Dp / 4; qd += ny) {
        const int r0 = 4 * qd;
        float v[4];
        int e = 0, d = 0;
        if (K != 3 && r0 < D) {
            int hi, lo;
            pair_of((uint64_t)r0, hi, lo);
            e = hi + 1;
            d = lo + 1;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = r0 + j;
            v[j] = 0.f;
            if (r < D) {
                if (K == 3) {
                    v[j] = (r + 1 == t - 1 ? tb.P[(size_t)(t - 2) * SG] : tb.P1[i_p1(t - 1, r + 1) * SG]) * sp(r + 1);
                } else {
                    const float p = (uint64_t)r < rowlen ? q2[(size_t)r * SG]
                                    : d == t - 2         ? tb.P[(size_t)(t - 3) * SG]
                                                         : tb.P1[i_p1(t - 2, d) * SG];
                    v[j] = p * sp(e) * sd(d);
                    if (++d == e) {  // next pair in colex order
                        ++e;
                        d = 1;
                    }
                }
            }
        }
        float4 h, l;
        h.x = to_tf32(v[0]); l.x = to_tf32(v[0] - h.x);
        h.y = to_tf32(v[1]); l.y = to_tf32(v[1] - h.y);
        h.z = to_tf32(v[2]); l.z = to_tf32(v[2] - h.z);
        h.w = to_tf32(v[3]); l.w = to_tf32(v[3] - h.w);
        const size_t blk = ((size_t)(r0 / TC_KC) * nsb + sb) * 2 * TC_BCH;
        const uint32_t o = tc_off(sl, r0 % TC_KC) / 4;
        *reinterpret_cast<float4 *>(a.W + blk + o) = h;
        *reinterpret_cast<float4 *>(a.W + blk + TC_BCH + o) = l;
    }
}

// The rows of the step product (cumulant segments) split into TF32 hi / lo and
// laid out like W: row tile rt (128 rows), chunk c (TC_KC inner entries) at
// float offset (rt nk + c) 2 128 TC_KC, hi then lo, each in the core-matrix layout.
// Rows beyond `rows` and entries beyond D are zero. Thread i = row i of tile rt.
template <int K>
__device__ __forceinline__ void a_operand(const Args<float> &a, int t, uint64_t rows, int D, int rt, int c, int nk) {
    static_assert(PREP == TC_M, "one thread per row of a tile");
    const int tid = threadIdx.x;
    const uint64_t q = (uint64_t)rt * TC_M + tid;
    uint64_t kb = 0, dst = 0;
    if (q < rows) zrow(K, a.M, t, q, a.off, a.o, kb, dst);
    float *blk = a.At + ((size_t)rt * nk + c) * 2 * TC_ACH;
    const float *kp = a.kap + kb;
#pragma unroll 2
    for (int j = 0; j < TC_KC; j += 4) {
        const int k = c * TC_KC + j;
        float v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = (q < rows && k + i < D) ? kp[k + i] : 0.f;
        float4 h, l;
        h.x = to_tf32(v[0]); l.x = to_tf32(v[0] - h.x);
        h.y = to_tf32(v[1]); l.y = to_tf32(v[1] - h.y);
        h.z = to_tf32(v[2]); l.z = to_tf32(v[2] - h.z);
        h.w = to_tf32(v[3]); l.w = to_tf32(v[3] - h.w);
        const uint32_t o = tc_off(tid, j) / 4;
        *reinterpret_cast<float4 *>(blk + o) = h;
        *reinterpret_cast<float4 *>(blk + TC_ACH + o) = l;
    }
}

// Both operands of step t's product in one launch: nw blocks of W (S / PREP per
// row of blocks), then row tiles x chunks of the rows.
template <int K>
__global__ void __launch_bounds__(PREP) operands_kernel(Args<float> a, int t, uint64_t rows, int D, unsigned nw,
                                                        unsigned nrt, unsigned nk) {
    await_previous();
    if constexpr (K == 3) release_next();
    const unsigned nx = (unsigned)(a.S / PREP);
    if (blockIdx.x < nw) {
        w_operand<K>(a, t, D, (int)(blockIdx.x % nx), (int)(blockIdx.x / nx), (int)(nw / nx));
    } else {
        const unsigned q = blockIdx.x - nw;
        a_operand<K>(a, t, rows, D, (int)(q % nrt), (int)(q / nrt), (int)nk);
    }
}

// Z rows of one 128-row tile x 256 samples. Thread 0 streams both operands by
// TMA bulk copies (A: 128 rows, W: 256 samples, hi and lo, per TC_KC-wide
// chunk) into a ring of TC_NS stages and issues the MMAs; chunk c-1+TC_NS is
// loaded into the stage of chunk c-1 once the MMAs of chunk c-1 have completed,
// while those of chunk c run. All threads then read
// the accumulator (thread i = row i) and write the rows out.
template <int K, int NS, int TN>
__global__ void __launch_bounds__(128, NS == TC_NS ? 2 : 1) ztc_kernel(Args<float> a, int t, uint64_t rows, int D) {
    await_previous();
    if constexpr (K == 3) release_next();
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int STAGE = tc_stage(TN), BB = TN * TC_KC * 4;
    static_assert(NS <= 8 && NS * STAGE >= 4 * 32 * 36 * 4, "barrier area, epilogue tiles");
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + NS * STAGE);
    uint64_t *empty = full + 8;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + NS * STAGE + 128);
    int *flag = reinterpret_cast<int *>(smem + NS * STAGE + 192);
    const int tid = threadIdx.x, warp = tid >> 5;
    const uint64_t m0 = (uint64_t)blockIdx.x * TC_M;
    const int rt = blockIdx.x, s0 = (int)blockIdx.y * TN, sb = s0 / TC_N, nsb = a.S / TC_N;
    const int nk = (D + TC_KC - 1) / TC_KC;
    if (tid == 0) {
        for (int i = 0; i < NS; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        *flag = 1;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(TN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    if (tid == 0) {
        const uint32_t sbase = smem_u32(smem);
        const float *Ab = a.At + (size_t)rt * nk * 2 * TC_ACH;
        // TN samples of W's 256-sample tile: a contiguous part of its hi and of its lo copy
        const float *Wb = a.W + (size_t)sb * 2 * TC_BCH + s0 % TC_N * TC_KC;
        auto load = [&](int c) {
            const int st = c % NS;
            unsigned char *sp = smem + st * STAGE;
            mbar_expect(&full[st], 2 * TC_AB + 2 * BB);
            tma_bulk(sp, Ab + (size_t)c * 2 * TC_ACH, 2 * TC_AB, &full[st]);
            const float *wc = Wb + (size_t)c * nsb * 2 * TC_BCH;
            if constexpr (TN == TC_N) {
                tma_bulk(sp + 2 * TC_AB, wc, 2 * BB, &full[st]);
            } else {
                tma_bulk(sp + 2 * TC_AB, wc, BB, &full[st]);
                tma_bulk(sp + 2 * TC_AB + BB, wc + TC_BCH, BB, &full[st]);
            }
        };
        // chunk c uses stage c % NS and completes phase (c / NS) & 1 of its
        // barriers; nl chunks loaded, nf of them waited for (full), nc committed,
        // ne of those waited for (empty)
        int nl = 0, nf = 0, nc = 0, ne = 0;
        const int lim = a.wait_limit;
        auto wait_full = [&](int c) { return mbar_wait(&full[c % NS], (uint32_t)(c / NS) & 1u, lim); };
        auto wait_empty = [&](int c) { return mbar_wait(&empty[c % NS], (uint32_t)(c / NS) & 1u, lim); };
        bool ok = true;
        if (!a.no_loads)
            for (int c = 0; c < NS && c < nk; ++c) {
                load(c);
                ++nl;
            }
        for (int c = 0; c < nk && ok; ++c) {
            const int st = c % NS;
            ok = wait_full(c);
            if (!ok) break;
            ++nf;
            tc_fence_after();
            const uint32_t sbs = sbase + st * STAGE;
#pragma unroll
            for (int j = 0; j < TC_KC / 8; ++j) {
                const uint32_t o = j * 256;  // two core matrices per 8-wide slice of K
                const uint64_t ahi = tc_desc(sbs + o), alo = tc_desc(sbs + TC_AB + o);
                const uint64_t bhi = tc_desc(sbs + 2 * TC_AB + o), blo = tc_desc(sbs + 2 * TC_AB + BB + o);
                tc_mma<TN>(tmem, ahi, bhi, (c > 0 || j > 0) ? 1u : 0u);
                tc_mma<TN>(tmem, ahi, blo, 1u);
                tc_mma<TN>(tmem, alo, bhi, 1u);
            }
            tc_commit(&empty[st]);
            ++nc;
            // refill the stage of chunk c-1 with chunk c-1+NS once its MMAs are
            // done (those of chunk c are queued behind them meanwhile)
            if (c >= 1 && c - 1 + NS < nk) {
                ok = wait_empty(c - 1);
                if (ok) {
                    ++ne;
                    load(c - 1 + NS);
                    ++nl;
                }
            }
        }
        // the loop waited for chunks 0 .. nk-1-NS; wait for the rest
        while (ok && ne < nc) {
            ok = wait_empty(ne);
            if (ok) ++ne;
        }
        if (!ok) {
            *flag = 0;
            if (a.status) atomicOr(a.status, ST_TIMEOUT);
            // drain what this thread issued before leaving: copies not yet waited
            // for, then committed MMAs, each wait bounded again; what is still
            // outstanding after that is abandoned (the kernel has already failed)
            for (int c = nf; c < nl; ++c) wait_full(c);
            for (int c = ne; c < nc; ++c) wait_empty(c);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (*flag) {
        uint64_t kb = 0, dst = 0;
        float *out = nullptr;
        if (m0 + tid < rows) {
            zrow(K, a.M, t, m0 + tid, a.off, a.o, kb, dst);
            out = a.tab + dst * SG;
        }
        // The warp's 32 rows leave through shared memory (the ring is idle now):
        // a lane holds 32 columns of its own row after tcgen05.ld; the warp
        // writes them to a 32 x 36-float tile and reads them back as 8 lanes per
        // row, so every store instruction writes four whole 128-byte row pieces.
        const int lane = tid & 31, rsub = lane >> 3, c4 = (lane & 7) * 4;
        float *tile = reinterpret_cast<float *>(smem) + warp * 32 * 36;
        float *optr[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int src = 4 * i + rsub;  // row of the tile this lane stores in round i
            const unsigned long long p = __shfl_sync(0xffffffffu, (unsigned long long)out, src);
            optr[i] = reinterpret_cast<float *>(p);
        }
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
        for (int cc = 0; cc < TN / 32; ++cc) {
            const int sc = s0 + cc * 32;
            const size_t col = (size_t)(sc / SG) * a.gs + sc % SG + c4;  // group block and sample within it
            uint32_t v[32];
            tc_ld32(lane_base + (uint32_t)(cc * 32), v);
            float4 *row = reinterpret_cast<float4 *>(tile + lane * 36);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                row[q] = make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]),
                                     __uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3]));
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 w = *reinterpret_cast<const float4 *>(tile + (4 * i + rsub) * 36 + c4);
                if (optr[i]) *reinterpret_cast<float4 *>(optr[i] + col) = w;
            }
            __syncwarp();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TN) : "memory");
}

// Two CTAs with four stages share a multiprocessor, one's epilogue overlapping the
// other's MMAs. A launch that leaves few CTAs is bound by each one's chain of
// chunks: at one CTA or less per multiprocessor eight stages keep seven chunks'
// copies in flight; at half of that 64-sample tiles split the MMAs of a chunk over
// four times the CTAs (the same accumulations, so the same bits). K = 3, M = 1152,
// 256 samples (9 wide tiles of up to 144 chunks a step): 33 us a step with wide
// tiles, 26 with narrow ones.
template <int K>
static cudaError_t launch_ztc(const Args<float> &a, int t, uint64_t rows, int D, int sms, cudaStream_t st) {
    const unsigned nrt = (unsigned)((rows + TC_M - 1) / TC_M);
    const uint64_t wide = (uint64_t)nrt * (unsigned)(a.S / TC_N);
    auto go = [&](auto fn, int ns, int tn) {
        const int smem = tc_smem(ns, tn);
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        return launch_next(K == 3, fn, dim3(nrt, (unsigned)(a.S / tn)), 128, (size_t)smem, st, a, t, rows, D);
    };
    if (2 * wide <= (uint64_t)sms) return go(ztc_kernel<K, TC_NS_DEEP, TC_NARROW>, TC_NS_DEEP, TC_NARROW);
    if (wide <= (uint64_t)sms) return go(ztc_kernel<K, TC_NS_DEEP, TC_N>, TC_NS_DEEP, TC_N);
    return go(ztc_kernel<K, TC_NS, TC_N>, TC_NS, TC_N);
}

// ---------------------------------------------------------------- table rows of one step
// The kernels below take one table entry (or a few) and 32 VW consecutive samples
// per warp, VW per lane, the sample groups on the slow grid axis, so that all
// entries of a group are in flight together and its rows are shared in L2. Every
// sum over earlier variables is one chain of FMAs per sample in ascending order,
// whatever VW: the results don't depend on the schedule. The loads of a chain
// don't depend on it, so walk() issues U of them ahead of the FMAs that use them.

// VW consecutive samples of one lane, loaded and stored as one vector.
template <class R, int VW>
struct Lanes {
    R v[VW];
};
template <class R, int VW>
__device__ __forceinline__ Lanes<R, VW> ldl(const R *p) {
    Lanes<R, VW> r;
    if constexpr (VW == 1) {
        r.v[0] = *p;
    } else if constexpr (VW == 2) {
        const auto q = *reinterpret_cast<const typename Pair2<R>::T *>(p);
        r.v[0] = q.x;
        r.v[1] = q.y;
    } else {
        static_assert(VW == 4 && sizeof(R) == 4, "four lanes: float only");
        const float4 q = *reinterpret_cast<const float4 *>(p);
        r.v[0] = q.x;
        r.v[1] = q.y;
        r.v[2] = q.z;
        r.v[3] = q.w;
    }
    return r;
}
template <class R, int VW>
__device__ __forceinline__ void stl(R *p, const R (&x)[VW]) {
    if constexpr (VW == 1) {
        *p = x[0];
    } else if constexpr (VW == 2) {
        typename Pair2<R>::T q;
        q.x = x[0];
        q.y = x[1];
        *reinterpret_cast<typename Pair2<R>::T *>(p) = q;
    } else {
        *reinterpret_cast<float4 *>(p) = make_float4(x[0], x[1], x[2], x[3]);
    }
}
template <class R, int VW>
__device__ __forceinline__ Lanes<R, VW> ones() {
    Lanes<R, VW> r;
#pragma unroll
    for (int k = 0; k < VW; ++k) r.v[k] = R(1);
    return r;
}

// for i = i0 .. i1-1: use(i, load(i)), the loads of U terms issued before the
// first of them is used (load may keep running offsets: it is called in order).
template <int U, class Load, class Use>
__device__ __forceinline__ void walk(int i0, int i1, Load load, Use use) {
    using T = decltype(load(0));
    int i = i0;
    for (; i + U <= i1; i += U) {
        T b[U];
#pragma unroll
        for (int u = 0; u < U; ++u) b[u] = load(i + u);
#pragma unroll
        for (int u = 0; u < U; ++u) use(i + u, b[u]);
    }
    if (i < i1) {
        T b[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u < i1) b[u] = load(i + u);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u < i1) use(i + u, b[u]);
    }
}

// C(i, 2) in 32 bits, i <= 4096.
__device__ __forceinline__ unsigned c2u(int i) { return (unsigned)i * (unsigned)(i - 1) / 2u; }

// Sample-independent part of the address of P2~[x][e][d] (with its boundary
// cases P2~[x][x][d] = P1~[x-1][d], P1~[y][y] = P~[y-1]).
template <class R>
__device__ __forceinline__ const R *p2_row(const Grp<R> &t, int x, int e, int d) {
    if (e != x) return t.P2 + i_p2(x, e, d) * SG;
    return d == x - 1 ? t.P + (size_t)(x - 2) * SG : t.P1 + i_p1(x - 1, d) * SG;
}
// P1~[x][e] with P1~[x][x] = P~[x-1].
template <class R>
__device__ __forceinline__ const R *p1_row(const Grp<R> &t, int x, int e) {
    return e == x ? t.P + (size_t)(x - 1) * SG : t.P1 + i_p1(x, e) * SG;
}
// Pp~[x][b] (1 when the range is empty, b > x).
template <class R, int VW>
__device__ __forceinline__ Lanes<R, VW> ppl(const Grp<R> &t, int x, int b) {
    if (b > x) return ones<R, VW>();
    return ldl<R, VW>(t.Pp + i_pp(x, b) * SG);
}

template <class R, int VW>
struct Two {
    Lanes<R, VW> c, v;
};

// K = 5: Y[i][s] = Z3_i(n) + sum_{3 <= j < i} chi_j Pp~[i-1][j+1] Z5_j(i, n), 3 <= i < n.
template <class R, int VW, int U, int WPB>
__global__ void __launch_bounds__(32 * WPB) yv_kernel(Args<R> a, int n) {
    const int i = 3 + (int)blockIdx.x * WPB + (int)(threadIdx.x >> 5);
    if (i >= n) return;
    const Grp<R> t(a, sample_block() * (32 * VW) + (int)(threadIdx.x & 31) * VW);
    Lanes<R, VW> y = ldl<R, VW>(t.Z + i_z(i, n) * SG);
    const R *z5 = t.Z5 + i_z5(0, i, n) * SG, *q = t.Pp + (size_t)c2u(i - 1) * SG;  // Z5_j(i, n) and Pp~[i-1][j+1] at j
    struct Three {
        Lanes<R, VW> c, w, z;
    };
    walk<U>(
        3, i,
        [&](int j) {
            return Three{ldl<R, VW>(t.chi + j * SG), j == i - 1 ? ones<R, VW>() : ldl<R, VW>(q + (size_t)j * SG),
                         ldl<R, VW>(z5 + (size_t)j * SG)};
        },
        [&](int, const Three &b) {
#pragma unroll
            for (int k = 0; k < VW; ++k) y.v[k] = fma(b.c.v[k] * b.w.v[k], b.z.v[k], y.v[k]);
        });
    stl<R, VW>(t.Y + (size_t)i * SG, y.v);
}

// ---------------------------------------------------------------- step n: bias and draw
// The bias of 32 samples per block. Its sums over i are one chain of FMAs per
// sample, which one warp runs out of shared memory while all BIAS_W warps bring
// in the next tile of its operands (a thread per sample that loads its own terms
// waits for memory at every few of up to M steps of the chain: 340 us of a step
// at M = 1152, K = 3, 256 samples). The same tiles leave the step's coefficient
// rows behind, one per (i < n, sample):
//   CA = chi_i Pp~[n-1][i+1],  CB = kappa(i,n) chi_i,  CC = kappa(i,n) chi_i Pp~[n-1][i+1].
constexpr int BIAS_W = 16;

template <class R, int K>
__global__ void __launch_bounds__(32 * BIAS_W) bias_kernel(Args<R> a, int n) {
    await_previous();
    if constexpr (K == 3) release_next();
    constexpr int TI = 256 / sizeof(R);  // i per tile
    constexpr int PER = TI / BIAS_W;     // per thread
    __shared__ R cs[2][TI][32], vs[2][TI][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, s = (int)blockIdx.x * 32 + lane;
    const Grp<R> t(a, s);
    const R *k2n = a.kap + a.off[2] + c2u(n - 1) - 1;       // kappa(i, n) at i
    const R *ppn = t.Pp + (size_t)c2u(n - 1) * SG;          // Pp~[n-1][i+1] at i < n-1
    const R *yz = K == 5 ? t.Y : t.Z + ((size_t)c2u(n - 1) - 1) * SG;  // Y_i, or Z_i(n), at i
    R B = R(0), Pm = R(0);
    if (w == 0) {
        Pm = t.P[(size_t)(n - 1) * SG];
        B = k1(a, n) * Pm;
        if (K == 3 && n >= 2) B += t.G[0];
    }
    // pass 0 (K = 4, 5): kappa(i, n) chi_i P1~[n-1][i]; pass 1: chi_i Pp~[n-1][i+1] Y_i
    // (K = 4: Z_i, from i = 3; K = 3: Z_i, from i = 2) and the coefficient rows
#pragma unroll
    for (int pass = K == 3 ? 1 : 0; pass < 2; ++pass) {
        const int first = pass == 0 ? 1 : K == 3 ? 2 : 3;
        // loads of a tile (all of them before any of their uses or stores), then its
        // operands into shared memory
        R rx[PER], rk[PER], rp[PER], rv[PER];
        auto load = [&](int i0) {
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int i = i0 + w + BIAS_W * q;
                const bool in = i < n;
                rx[q] = in ? t.chi[(size_t)i * SG] : R(0);
                rk[q] = in ? k2n[i] : R(0);
                if (pass == 0) {
                    rv[q] = in ? *p1_row(t, n - 1, i) : R(0);
                } else {
                    rp[q] = i < n - 1 ? ppn[(size_t)i * SG] : R(1);
                    rv[q] = in && i >= first ? yz[(size_t)i * SG] : R(0);
                }
            }
        };
        auto put = [&](int buf, int i0) {
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int i = i0 + w + BIAS_W * q;
                const R cbv = rk[q] * rx[q], ca = pass == 0 ? R(0) : rx[q] * rp[q];
                if (pass == 1 && i < n) {
                    if (K != 3) t.CA[(size_t)i * SG] = ca;
                    t.CB[(size_t)i * SG] = cbv;
                    t.CC[(size_t)i * SG] = cbv * rp[q];
                }
                cs[buf][w + BIAS_W * q][lane] = pass == 0 ? cbv : ca;
                vs[buf][w + BIAS_W * q][lane] = rv[q];
            }
        };
        load(1);
        int buf = 0;
        for (int i0 = 1; i0 < n; i0 += TI, buf ^= 1) {
            put(buf, i0);
            __syncthreads();
            if (i0 + TI < n) load(i0 + TI);
            if (w == 0) {
                const int hi = min(TI, n - i0);
#pragma unroll 8
                for (int q = max(0, first - i0); q < hi; ++q) B = fma(cs[buf][q][lane], vs[buf][q][lane], B);
            }
        }
        if (K != 3 && pass == 0) {
            if (w == 0 && n >= 3) B += t.G[0];
            __syncthreads();  // the tiles are free again
        }
    }
    if (w != 0) return;
    const R hn = lead(a, n).y;
    const R p0 = fma(hn, Pm, B), p1v = fma(hn, Pm, -B);
    const R c0 = p0 > R(0) ? p0 : R(0), c1 = p1v > R(0) ? p1v : R(0);
    const R q = (c0 + c1 > R(0)) ? c0 / (c0 + c1) : R(0.5);
    int x = 0;
    if (s < a.n_valid) {
        const size_t o = (size_t)s * a.M + (n - 1);
        if (a.force) x = a.force[o] ? 1 : 0;
        else x = (a.u[o] < (double)q) ? 0 : 1;
        a.bits[o] = (uint8_t)x;
        if (a.q0) a.q0[o] = (double)q;
    }
    t.chi[(size_t)n * SG] = x ? R(-1) : R(1);
    if (x) a.bw[(size_t)(n >> 5) * a.S + s] |= 1u << (n & 31);
    t.P[(size_t)n * SG] = x ? p1v : p0;
}

// ---------------------------------------------------------------- step n: table rows

// Order-3 part of the p+ update, factored: the term
//   sum_{i > j >= l} kappa(j,i,n) chi_i chi_j chi_n Pp~[n-1][i+1] Pp~[i-1][j+1] Pp~[j-1][l]
// equals chi_n sum_{j >= l} Pp~[j-1][l] v(j) with
//   v(j) = chi_j sum_{i > j} kappa(j,i,n) chi_i Pp~[n-1][i+1] Pp~[i-1][j+1],
// which does not depend on l. v goes to Y (free after the bias).
template <class R, int VW, int U, int WPB>
__global__ void __launch_bounds__(32 * WPB) pvv_kernel(Args<R> a, int n) {
    const int j = 1 + (int)blockIdx.x * WPB + (int)(threadIdx.x >> 5);
    if (j >= n) return;
    const Grp<R> t(a, sample_block() * (32 * VW) + (int)(threadIdx.x & 31) * VW);
    const R *k3n = a.kap + a.off[3] + cb(n - 1, 3) + (j - 1);  // kappa(j, i, n) at C(i-1, 2)
    Lanes<R, VW> v;
#pragma unroll
    for (int k = 0; k < VW; ++k) v.v[k] = R(0);
    struct Term {
        Lanes<R, VW> c, q;
        R k3;
    };
    walk<U>(
        j + 1, n,
        [&](int i) {
            const unsigned o = c2u(i - 1);  // Pp~[i-1][j+1] is entry C(i-1, 2) + j
            return Term{ldl<R, VW>(t.CA + (size_t)i * SG),
                        i == j + 1 ? ones<R, VW>() : ldl<R, VW>(t.Pp + (size_t)(o + j) * SG), k3n[o]};
        },
        [&](int, const Term &b) {
#pragma unroll
            for (int k = 0; k < VW; ++k) v.v[k] = fma(b.k3 * b.c.v[k], b.q.v[k], v.v[k]);
        });
    const auto cj = ldl<R, VW>(t.chi + (size_t)j * SG);
#pragma unroll
    for (int k = 0; k < VW; ++k) v.v[k] = v.v[k] * cj.v[k];
    stl<R, VW>(t.Y + (size_t)j * SG, v.v);
}

// Terms i < e of P2~[n][e][d]: use(i, {coef row i, P2~[e-1][max(i,d)][min(i,d)]})
// for i = 1 .. e-1, i != d, ascending; coef is an [i][SG] table.
template <class R, int VW, int U, class Use>
__device__ __forceinline__ void p2_row_terms(const Grp<R> &t, int e, int d, const R *coef, Use use) {
    // i < d: P2~[e-1][d][i]; for d = e - 1 that row is P1~[e-2][i], ending with P~[e-3]
    const R *q = d < e - 1 ? t.P2 + i_p2(e - 1, d, 0) * SG : t.P1 + (e >= 3 ? i_p1(e - 2, 0) : 0) * SG;
    const R *pb = t.P + (size_t)(e - 3) * SG;
    walk<U>(
        1, d,
        [&](int i) {
            return Two<R, VW>{ldl<R, VW>(coef + (size_t)i * SG),
                              ldl<R, VW>(d == e - 1 && i == e - 2 ? pb : q + (size_t)i * SG)};
        },
        use);
    // d < i < e - 1: P2~[e-1][i][d]
    const R *qc = t.P2 + (i_p2(e - 1, 1, 0) + d) * SG;
    walk<U>(
        d + 1, e - 1,
        [&](int i) {
            return Two<R, VW>{ldl<R, VW>(coef + (size_t)i * SG), ldl<R, VW>(qc + (size_t)c2u(i - 1) * SG)};
        },
        use);
    if (d < e - 1) use(e - 1, Two<R, VW>{ldl<R, VW>(coef + (size_t)(e - 1) * SG), ldl<R, VW>(p1_row(t, e - 2, d))});
}

// The sums over i < e of the p2 update at steps n0 .. n0 + P2_NB - 1, for every
// pair (e, d) with e < n0: sum_i kappa(i,n) chi_i P2~[e-1][max(i,d)][min(i,d)] only
// needs bits and rows below n0, so one pass over the table serves P2_NB steps:
// a value loaded once feeds P2_NB chains of FMAs (kappa(i,n) uniform, chi_i times
// the value formed once; the products are the ones p2_kernel would form, in the
// same order). Left in R2 for p2_kernel. What p2_kernel still walks each step is
// the column i > e, whose weights Pp~[n-1][i+1] are known at step n only, and the
// rows e >= n0.
constexpr int P2_NB = 8;

template <class R, int VW>
__global__ void __launch_bounds__(32, 16) p2_block_kernel(Args<R> a, int n0, unsigned npairs) {
    const Grp<R> t(a, (int)blockIdx.y * (32 * VW) + (int)threadIdx.x * VW);
    const unsigned r = blockIdx.x;
    int hi, lo;
    pair_of(r, hi, lo);
    const R *kb = a.kb + (size_t)((n0 - 1) / P2_NB) * (a.M + 1) * P2_NB;
    R x[P2_NB][VW];
#pragma unroll
    for (int m = 0; m < P2_NB; ++m)
#pragma unroll
        for (int k = 0; k < VW; ++k) x[m][k] = R(0);
    p2_row_terms<R, VW, 4>(t, hi + 1, lo + 1, t.chi, [&](int i, const Two<R, VW> &b) {
        R v[VW], kn[P2_NB];
#pragma unroll
        for (int k = 0; k < VW; ++k) v[k] = b.c.v[k] * b.v.v[k];
        constexpr int KV = 16 / sizeof(R);
#pragma unroll
        for (int m = 0; m < P2_NB; m += KV) {
            const auto q = ldl<R, KV>(kb + (size_t)i * P2_NB + m);
#pragma unroll
            for (int u = 0; u < KV; ++u) kn[m + u] = q.v[u];
        }
#pragma unroll
        for (int m = 0; m < P2_NB; ++m)
#pragma unroll
            for (int k = 0; k < VW; ++k) x[m][k] = fma(kn[m], v[k], x[m][k]);
    });
#pragma unroll
    for (int m = 0; m < P2_NB; ++m)
        if (n0 + m <= a.M) stl<R, VW>(t.R2 + ((size_t)m * npairs + r) * SG, x[m]);
}

// kb[b][i][m] = kappa(i, n), n = 1 + P2_NB b + m (0 where i >= n or n > M).
template <class R>
__global__ void kb_kernel(const R *__restrict__ kap2, int M, int n, R *__restrict__ kb) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const int m = q % P2_NB, i = q / P2_NB % (M + 1), v = 1 + q / (P2_NB * (M + 1)) * P2_NB + m;
    kb[q] = i >= 1 && i < v && v <= M ? kap2[c2u(v - 1) + (unsigned)(i - 1)] : R(0);
}

// P2~[n][e][d], n-1 >= e > d >= 1 (Eq. probdoubleelidedade).
// Order 2: i > e reaches P2~[i-1][e][d] (factor Pp~[n-1][i+1]); i < e reaches
// P2~[e-1][max(i,d)][min(i,d)] (common factor Pp~[n-1][e+1]).
// The same values P2~[i-1][e][d], i > e, are every term of the p1 order-3 sums
// whose largest index is i (Eq. probelidedade with (a, b, c) = (i, e, d)): they
// enter P1~[n][e] with weight CA[i] kappa(d,i,n) chi_d and P1~[n][d] with weight
// CA[i] kappa(e,i,n) chi_e. Both sums are formed here, without chi_d / chi_e, and
// left in T for rows_kernel, so each value is read once per step.
// Schedule: one warp (one block) per pair (e, d) and 32 VW consecutive samples.
// The kernel is bound by load latency: the bounds cap it at 64 registers, so that
// 32 one-warp blocks (the per-SM block limit) stay resident.
template <class R, int VW>
__global__ void __launch_bounds__(32, 32) p2_kernel(Args<R> a, int n, unsigned npairs) {
    const Grp<R> t(a, (int)blockIdx.y * (32 * VW) + (int)threadIdx.x * VW);
    const unsigned r = blockIdx.x;
    int hi, lo;
    pair_of(r, hi, lo);
    const int e = hi + 1, d = lo + 1;
    R acc[VW], tE[VW], tD[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) acc[k] = tE[k] = tD[k] = R(0);
    if (a.op2 >= 2) {
        const int m = (n - 1) % P2_NB;
        Lanes<R, VW> x;
        if (a.kb && e < n - m) {  // formed by p2_block_kernel at step n - m
            x = ldl<R, VW>(t.R2 + ((size_t)m * npairs + r) * SG);
        } else {
#pragma unroll
            for (int k = 0; k < VW; ++k) x.v[k] = R(0);
            p2_row_terms<R, VW, 4>(t, e, d, t.CB, [&](int, const Two<R, VW> &b) {
#pragma unroll
                for (int k = 0; k < VW; ++k) x.v[k] = fma(b.c.v[k], b.v.v[k], x.v[k]);
            });
        }
        const auto w = ppl<R, VW>(t, n - 1, e + 1);
#pragma unroll
        for (int k = 0; k < VW; ++k) acc[k] = w.v[k] * x.v[k];
    }
    if ((a.op2 >= 2 || a.op1 >= 3) && e + 1 < n) {
        const R *k3n = a.kap + a.off[3] + cb(n - 1, 3) - 1;  // k3n[C(i-1,2) + j] = kappa(j, i, n)
        R a2[VW];
        // i = e + 1: P1~[e-1][d], or P~[e-2] when d = e - 1
        {
            const auto v = ldl<R, VW>(p1_row(t, e - 1, d));
            const R *kp = k3n + c2u(e);
            const R kd = kp[d], ke = kp[e];
            const auto ca = ldl<R, VW>(t.CA + (size_t)(e + 1) * SG), cc = ldl<R, VW>(t.CC + (size_t)(e + 1) * SG);
#pragma unroll
            for (int k = 0; k < VW; ++k) {
                a2[k] = cc.v[k] * v.v[k];
                tE[k] = ca.v[k] * kd * v.v[k];
                tD[k] = ca.v[k] * ke * v.v[k];
            }
        }
        struct Col {
            Lanes<R, VW> v, ca, cc;
            R kd, ke;
        };
        const R *q = t.P2 + i_p2(e + 1, e, d) * SG;
        walk<2>(
            e + 2, n,
            [&](int i) {
                const R *kp = k3n + c2u(i - 1);
                const Col b{ldl<R, VW>(q), ldl<R, VW>(t.CA + (size_t)i * SG), ldl<R, VW>(t.CC + (size_t)i * SG), kp[d], kp[e]};
                q += (size_t)c2u(i - 2) * SG;
                return b;
            },
            [&](int, const Col &b) {
#pragma unroll
                for (int k = 0; k < VW; ++k) {
                    a2[k] = fma(b.cc.v[k], b.v.v[k], a2[k]);
                    tE[k] = fma(b.ca.v[k] * b.kd, b.v.v[k], tE[k]);
                    tD[k] = fma(b.ca.v[k] * b.ke, b.v.v[k], tD[k]);
                }
            });
        if (a.op2 >= 2) {
#pragma unroll
            for (int k = 0; k < VW; ++k) acc[k] += a2[k];
        }
    }
    if (a.op1 >= 3) {
        stl<R, VW>(t.T + (size_t)(2 * r) * SG, tE);
        stl<R, VW>(t.T + (size_t)(2 * r + 1) * SG, tD);
    }
    const auto cn = ldl<R, VW>(t.chi + (size_t)n * SG);
    const auto ld = lead(a, n);
    const auto pv = ldl<R, VW>(p2_row(t, n - 1, e, d));
    R out[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) out[k] = fma(cn.v[k], acc[k], fma(ld.x, cn.v[k], ld.y) * pv.v[k]);
    stl<R, VW>(t.P2 + i_p2(n, e, d) * SG, out);
}

// Pp~[n][l] (Eq. a / Eq. probpartialade).
template <class R, int VW, int U>
__device__ __forceinline__ void pp_row(const Args<R> &a, const Grp<R> &t, int n, int l) {
    const auto cn = ldl<R, VW>(t.chi + (size_t)n * SG);
    const auto ld = lead(a, n);
    R acc[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) acc[k] = R(0);
    auto use = [&](int, const Two<R, VW> &b) {
#pragma unroll
        for (int k = 0; k < VW; ++k) acc[k] = fma(b.c.v[k], b.v.v[k], acc[k]);
    };
    // coef rows (CC, then the order-3 factors Y) against Pp~[i-1][l] (1 at i = l)
    auto sum = [&](const R *coef, int hi) {
        if (l < hi) use(l, Two<R, VW>{ldl<R, VW>(coef + (size_t)l * SG), ones<R, VW>()});
        const R *p = t.Pp + ((size_t)l - 1) * SG;
        walk<U>(
            l + 1, hi,
            [&](int i) {
                return Two<R, VW>{ldl<R, VW>(coef + (size_t)i * SG), ldl<R, VW>(p + (size_t)c2u(i - 1) * SG)};
            },
            use);
    };
    if (a.opp >= 2) sum(t.CC, n);
    if (a.opp >= 3) sum(t.Y, n - 1);
    const auto w = ppl<R, VW>(t, n - 1, l);
    R out[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) out[k] = fma(cn.v[k], acc[k], fma(ld.x, cn.v[k], ld.y) * w.v[k]);
    stl<R, VW>(t.Pp + i_pp(n, l) * SG, out);
}

// K = 3: P1~[n][e] (Eq. b), i < e with weight kappa(i,n) chi_i Pp~[n-1][e+1] and
// i > e with CC_i.
template <class R, int VW, int U>
__device__ __forceinline__ void p1_row_k3(const Args<R> &a, const Grp<R> &t, int n, int e) {
    const auto cn = ldl<R, VW>(t.chi + (size_t)n * SG), w = ppl<R, VW>(t, n - 1, e + 1);
    const auto ld = lead(a, n);
    R acc[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) acc[k] = R(0);
    auto below = [&](int, const Two<R, VW> &b) {
#pragma unroll
        for (int k = 0; k < VW; ++k) acc[k] = fma(b.c.v[k] * w.v[k], b.v.v[k], acc[k]);
    };
    auto above = [&](int, const Two<R, VW> &b) {
#pragma unroll
        for (int k = 0; k < VW; ++k) acc[k] = fma(b.c.v[k], b.v.v[k], acc[k]);
    };
    auto cb_ = [&](int i) { return ldl<R, VW>(t.CB + (size_t)i * SG); };
    auto cc_ = [&](int i) { return ldl<R, VW>(t.CC + (size_t)i * SG); };
    const R *p = t.P1 + ((size_t)c2u(e - 2) - 1) * SG;  // P1~[e-1][i], i < e - 1
    if (e >= 3) walk<U>(1, e - 1, [&](int i) { return Two<R, VW>{cb_(i), ldl<R, VW>(p + (size_t)i * SG)}; }, below);
    if (e >= 2) below(e - 1, Two<R, VW>{cb_(e - 1), ldl<R, VW>(t.P + (size_t)(e - 2) * SG)});
    if (e + 1 < n) above(e + 1, Two<R, VW>{cc_(e + 1), ldl<R, VW>(t.P + (size_t)(e - 1) * SG)});
    p = t.P1 + ((size_t)e - 1) * SG;  // P1~[i-1][e] at C(i-2, 2)
    walk<U>(
        e + 2, n, [&](int i) { return Two<R, VW>{cc_(i), ldl<R, VW>(p + (size_t)c2u(i - 2) * SG)}; }, above);
    const auto pv = ldl<R, VW>(p1_row(t, n - 1, e));
    R out[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) out[k] = fma(cn.v[k], acc[k], fma(ld.x, cn.v[k], ld.y) * pv.v[k]);
    stl<R, VW>(t.P1 + i_p1(n, e) * SG, out);
}

// K = 4, 5: P1~[n][e] (Eq. probelidedade). Order 3: with (a, b, c) the decreasing
// order of (i, j, e), the terms with a = e come from the product rows (X_e(n),
// times Pp~[n-1][e+1]); the others (a = i > e) from the per-pair sums p2_kernel
// leaves in T: pairs (e, d), d < e, carry chi_d-weighted parts for e; pairs (j, e),
// j > e, for e.
template <class R, int VW, int U>
__device__ __forceinline__ void p1_row_k45(const Args<R> &a, const Grp<R> &t, int n, int e) {
    const auto cn = ldl<R, VW>(t.chi + (size_t)n * SG);
    const auto ld = lead(a, n);
    R acc[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) acc[k] = R(0);
    auto use = [&](int, const Two<R, VW> &b) {
#pragma unroll
        for (int k = 0; k < VW; ++k) acc[k] = fma(b.c.v[k], b.v.v[k], acc[k]);
    };
    if (a.op1 >= 2) {
        walk<U>(
            1, e,
            [&](int i) { return Two<R, VW>{ldl<R, VW>(t.CB + (size_t)i * SG), ldl<R, VW>(p2_row(t, n - 1, e, i))}; }, use);
        const R *q = t.P2 + (i_p2(n - 1, 1, 0) + e) * SG;  // P2~[n-1][i][e] at C(i-1, 2)
        walk<U>(
            e + 1, n - 1,
            [&](int i) {
                return Two<R, VW>{ldl<R, VW>(t.CB + (size_t)i * SG), ldl<R, VW>(q + (size_t)c2u(i - 1) * SG)};
            },
            use);
        if (e < n - 1)
            use(n - 1, Two<R, VW>{ldl<R, VW>(t.CB + (size_t)(n - 1) * SG), ldl<R, VW>(p1_row(t, n - 2, e))});
    }
    if (a.op1 >= 3) {
        if (e >= 3) use(e, Two<R, VW>{ppl<R, VW>(t, n - 1, e + 1), ldl<R, VW>(t.X + i_z(e, n) * SG)});
        const R *T = t.T + 2 * ((size_t)c2u(e - 1) - 1) * SG;  // pair (e, d) at 2 d
        walk<U>(
            1, e,
            [&](int d) { return Two<R, VW>{ldl<R, VW>(t.chi + (size_t)d * SG), ldl<R, VW>(T + (size_t)(2 * d) * SG)}; },
            use);
        T = t.T + (2 * (size_t)(e - 1) + 1) * SG;  // pair (j, e) at 2 C(j-1, 2)
        walk<U>(
            e + 1, n,
            [&](int j) {
                return Two<R, VW>{ldl<R, VW>(t.chi + (size_t)j * SG), ldl<R, VW>(T + (size_t)(2 * c2u(j - 1)) * SG)};
            },
            use);
    }
    const auto pv = ldl<R, VW>(p1_row(t, n - 1, e));
    R out[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) out[k] = fma(cn.v[k], acc[k], fma(ld.x, cn.v[k], ld.y) * pv.v[k]);
    stl<R, VW>(t.P1 + i_p1(n, e) * SG, out);
}

// The p1 rows e = 1..n-1 and the p+ rows l = 1..n of one step in one launch (they
// read rows below n only): the p1 warps first, the p+ warps by falling length.
template <class R, int K, int VW, int U, int WPB>
__global__ void __launch_bounds__(32 * WPB, 32 / WPB) rows_kernel(Args<R> a, int n) {
    await_previous();
    if (K == 3 && n < a.M) release_next();
    const Grp<R> t(a, sample_block() * (32 * VW) + (int)(threadIdx.x & 31) * VW);
    const int item = (int)blockIdx.x * WPB + (int)(threadIdx.x >> 5);
    if (item < n - 1) {
        if constexpr (K == 3) p1_row_k3<R, VW, U>(a, t, n, 1 + item);
        else p1_row_k45<R, VW, U>(a, t, n, 1 + item);
    } else if (item < 2 * n - 1) {
        pp_row<R, VW, U>(a, t, n, item - n + 2);
    }
}

template <class R>
__global__ void init_kernel(Args<R> a) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < a.S) {
        const Grp<R> t(a, s);
        t.P[0] = R(1);
        for (int w = 0; w <= a.M / 32; ++w) a.bw[(size_t)w * a.S + s] = 0u;
    }
}

// ln of the estimated probability: ln P~[M] - sum_v ln s_v (NaN if P~[M] <= 0).
template <class R>
__global__ void logp_kernel(Args<R> a, double *logp) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= a.n_valid) return;
    double h = 0.0;
    for (int v = 1; v <= a.M; ++v) h += a.H[v];
    const double P = (double)Grp<R>(a, s).P[(size_t)a.M * SG];
    logp[s] = P > 0.0 ? log(P) - h : __longlong_as_double(0x7ff8000000000000ULL);
}

// Per-variable scales from the order-1 cumulants: kappa({v}) = c_v = <(-1)^{x_v}>,
// so mode v - 1 is silent with probability (1 + c_v) / 2; s_v = exp(H_v) with H_v
// that binary entropy in nats (s_v in [1, 2]).
template <class R>
__global__ void scale_kernel(const double *__restrict__ kap, int M, R *hs, R *lead, double *H) {
    const int v = 1 + blockIdx.x * blockDim.x + threadIdx.x;
    if (v > M) return;
    double p0 = 0.5 * (1.0 + kap[v - 1]);
    p0 = p0 < 0.0 ? 0.0 : (p0 > 1.0 ? 1.0 : p0);
    const double p1 = 1.0 - p0;
    const double h = (p0 > 0.0 ? -p0 * log(p0) : 0.0) + (p1 > 0.0 ? -p1 * log(p1) : 0.0);
    const double half = 0.5 * exp(h);
    H[v] = h;
    hs[v] = (R)half;
    lead[2 * v] = (R)(kap[v - 1] * half);
    lead[2 * v + 1] = (R)half;
}

// x rounded to R; FP32 results in the normal range by integer rounding (the
// conversion instruction runs on GB300's narrow FP64 pipe).
template <class R>
__device__ __forceinline__ R round_to(double x) {
    if constexpr (sizeof(R) == 8) {
        return x;
    } else {
        const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
        const int e = (int)((hi >> 20) & 0x7ffu) - 896;
        if (e < 1 || e > 253) return (float)x;
        unsigned r = (hi & 0x80000000u) | ((unsigned)e << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
        const unsigned rest = lo << 3;  // to nearest, ties to even; a carry moves into the exponent
        r += rest > 0x80000000u || (rest == 0x80000000u && (r & 1u));
        return __uint_as_float(r);
    }
}

// kappa'(S) = kappa(S) prod_{v in S} s_v / 2 for every entry of order d, in the
// arithmetic precision R, the product formed from the largest mode down. A warp
// takes `run` consecutive entries, 32 at a time (coalesced); each lane keeps the
// modes c_2 < .. < c_{d-1} of its entry, whose C(c_2, 2) pairs (c_0, c_1) are
// consecutive ranks, and their scales' product, and moves on to the next such set
// when its rank leaves them. Bound by the FP64 pipe (3 multiplications per entry)
// and HBM (12 bytes per entry): M = 144, K = 5 took 9.3 ms with one thread walking
// 64 entries, whose loads did not coalesce.
template <class R, int D>
__global__ void __launch_bounds__(256) kscale_kernel(const double *__restrict__ kap, int M, uint64_t off, uint64_t n,
                                                     const R *__restrict__ hs, R *__restrict__ out, int run) {
    extern __shared__ double hd[];  // hd[c] = scale of mode c
    for (int c = threadIdx.x; c < M; c += blockDim.x) hd[c] = (double)hs[c + 1];
    __syncthreads();
    const uint64_t r0 = ((uint64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * run;
    if (r0 >= n) return;
    const uint64_t r1 = r0 + run < n ? r0 + run : n;
    uint64_t r = r0 + (threadIdx.x & 31);
    if (r >= r1) return;
    int c[D + 1];
    colex_unrank(r, D, c);
    c[D] = M + 1;  // beyond the last mode
    unsigned t = 0, len = 0;  // rank within the pairs of c[2..], and their number
    double fu = 1.0;          // product of the scales of c[2..D-1]
    auto upper = [&]() {
        fu = 1.0;
#pragma unroll
        for (int i = D - 1; i >= 2; --i) fu *= hd[c[i]];
        len = D >= 3 ? (unsigned)binom2(c[2]) : ~0u;
    };
    if constexpr (D >= 2) {
        t = (unsigned)binom2(c[1]) + (unsigned)c[0];
        upper();
    }
    for (; r < r1; r += 32) {
        const double x = kap[off + r];
        if constexpr (D == 1) {
            out[off + r] = round_to<R>(x * (1.0 * hd[(int)r]));
        } else {
            while (t >= len) {  // next set of upper modes (colex successor)
                t -= len;
                int i = 2;
#pragma unroll
                for (int k = 2; k < D - 1; ++k)
                    if (i == k && c[k] + 1 == c[k + 1]) i = k + 1;
#pragma unroll
                for (int k = 2; k < D; ++k) c[k] = k < i ? k : k == i ? c[k] + 1 : c[k];
                upper();
            }
            int c1, c0;
            pair_decode(t, c1, c0);
            out[off + r] = round_to<R>(x * ((fu * hd[c1]) * hd[c0]));
            t += 32;
        }
    }
}

template <class R>
static void launch_kscale(const double *kap, int M, int K, const R *hs, R *out, cudaStream_t st) {
    uint64_t off = 0;
    for (int d = 1; d <= K; ++d) {
        const uint64_t n = cb(M, d);
        // 8 warps a block; short runs until they fill the GPU's warps several times
        const int run = n >= 1u << 25 ? 4096 : 512;
        const unsigned grid = (unsigned)((n + 8 * run - 1) / (8 * run));
        const size_t smem = sizeof(double) * (size_t)M;  // at most 32 KB
        if (d == 1) kscale_kernel<R, 1><<<grid, 256, smem, st>>>(kap, M, off, n, hs, out, run);
        if (d == 2) kscale_kernel<R, 2><<<grid, 256, smem, st>>>(kap, M, off, n, hs, out, run);
        if (d == 3) kscale_kernel<R, 3><<<grid, 256, smem, st>>>(kap, M, off, n, hs, out, run);
        if (d == 4) kscale_kernel<R, 4><<<grid, 256, smem, st>>>(kap, M, off, n, hs, out, run);
        if (d == 5) kscale_kernel<R, 5><<<grid, 256, smem, st>>>(kap, M, off, n, hs, out, run);
        off += n;
    }
}

// ---------------------------------------------------------------- host side

static size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

static Tabs sampler_tabs(int M, int K) {
    Tabs o{};
    size_t n = 0;
    auto take = [&](size_t &field, size_t entries) {
        field = n;
        n += entries;
    };
    take(o.chi, (size_t)M + 1);
    take(o.P, (size_t)M + 1);
    take(o.G, 1);
    take(o.CA, K >= 4 ? (size_t)M + 1 : 0);
    take(o.CB, (size_t)M + 1);
    take(o.CC, (size_t)M + 1);
    take(o.Y, K >= 4 ? (size_t)M + 1 : 0);
    take(o.Pp, cb(M, 2) + (size_t)M);
    take(o.P1, cb(M, 2));
    take(o.Z, cb(M, 2));
    take(o.X, K >= 4 ? cb(M, 2) : 0);
    take(o.T, K >= 4 ? 2 * cb(M - 1, 2) : 0);
    take(o.R2, K == 5 ? P2_NB * cb(M - 1, 2) : 0);  // K = 4 runs order 1 (no such sums) unless told otherwise
    take(o.P2, K >= 4 ? cb(M, 3) : 0);
    take(o.Z5, K == 5 ? cb(M, 3) : 0);
    o.entries = n;
    return o;
}

SamplerLayout sampler_layout(int M, int K, int S, int precision) {
    SamplerLayout L{};
    const size_t es = precision == 0 ? sizeof(double) : sizeof(float);
    const size_t Ss = (size_t)S;
    size_t off = 256;  // status word first (read by gbs_stream_status)
    L.tab = off;       // S is a multiple of SG: whole groups
    off = a256(off + sampler_tabs(M, K).entries * Ss * es);
    // W: plain [r][S], or for the tensor-core product hi / lo copies of TC_KC-wide chunks
    L.W = off;
    off = a256(off + 2 * ((K >= 4 ? cb(M - 1, 2) : (size_t)M) + 32) * Ss * es);
    // tensor-core product rows: max over the steps of (row tiles x chunks) x 2 TC_ACH floats
    size_t at = 0;
    if (precision != 0)
        for (int t = 1; t <= M; ++t) {
            const uint64_t D = K == 3 ? (uint64_t)(t - 1) : cb(t - 1, 2);
            const uint64_t rows = K == 3   ? 1 + (uint64_t)(M - t)
                                  : K == 4 ? 1 + 2 * (uint64_t)(M - t)
                                           : 1 + 2 * (uint64_t)(M - t) + cb(M - t, 2);
            const size_t n = (size_t)((rows + TC_M - 1) / TC_M) * ((D + TC_KC - 1) / TC_KC) * 2 * TC_ACH;
            if (n > at) at = n;
        }
    L.At = off;
    off = a256(off + at * sizeof(float));
    L.bw = off;
    off = a256(off + (size_t)(M / 32 + 1) * Ss * sizeof(uint32_t));
    L.kap = off;  // the rescaled cumulants kappa', in the arithmetic precision
    uint64_t nk = 0;
    for (int d = 1; d <= K; ++d) nk += cb(M, d);
    off = a256(off + nk * es);
    L.hs = off;
    off = a256(off + ((size_t)M + 1) * es);
    L.H = off;
    off = a256(off + ((size_t)M + 1) * sizeof(double));
    L.lead = off;
    off = a256(off + 2 * ((size_t)M + 1) * es);
    L.kb = off;
    off = a256(off + (K == 5 ? (size_t)((M - 1) / P2_NB + 1) * (M + 1) * P2_NB : 0) * es);
    L.total = off;
    return L;
}

// Grid of a per-(entry, sample) kernel: samples along x, entries along y, about
// 10^4 blocks in all (each block loops over its share of the entries).
static dim3 egrid(int S, uint64_t entries) {
    const uint64_t bx = (uint64_t)(S / ETB);
    uint64_t cap = 10000 / bx;
    if (cap < 16) cap = 16;
    uint64_t by = entries < cap ? entries : cap;
    if (by < 1) by = 1;
    return dim3((unsigned)bx, (unsigned)by);
}

// Steps of K = 3 are chains of four kernels of 6 to 110 us; chained (launch_next) their
// gaps go: M = 1152, 256 samples 191.8 -> 184.9 ms a call. At K = 5 (1.6 ms a step, M =
// 144, 8192 samples) chaining every kernel was 0.6 % slower, 222.9 -> 224.2 ms: blocks
// in place early keep the kernel before's split of shared memory and first-level cache,
// which the table walk reads through. K = 4 and 5 stay with ordinary launches.
//
// The kernels of step t after its products: VW samples per lane, U loads of a
// chain ahead, WPB warps per block. Two samples per lane in FP32 and one in FP64,
// eight loads ahead, two warps: the fastest or within 2 % of it at every size tried
// (K = 3, M = 1152, 256 samples: 195 ms; four samples and four loads 213; one
// sample and 16 loads 200).
template <class R, int K>
static cudaError_t step_rows(const Args<R> &a, int t, cudaStream_t st) {
    constexpr int VW = sizeof(R) == 4 ? 2 : 1, U = 8, WPB = 2, NT = 32 * WPB;
    const unsigned gy = (unsigned)(a.S / (32 * VW));
    auto grid = [&](int warps) { return sample_grid((unsigned)((warps + WPB - 1) / WPB), gy); };
    cudaError_t e = cudaSuccess;
    auto next = [&](auto fn, dim3 g, int nt, auto... args) {
        if (e == cudaSuccess) e = launch_next(K == 3, fn, g, nt, 0, st, a, args...);
    };
    if (K == 5 && t > 3) next(yv_kernel<R, VW, U, WPB>, grid(t - 3), NT, t);
    next(bias_kernel<R, K>, (unsigned)(a.S / 32), 32 * BIAS_W, t);
    if (K >= 4 && a.opp >= 3 && t > 1) next(pvv_kernel<R, VW, U, WPB>, grid(t - 1), NT, t);
    if (K >= 4 && t > 2) {  // before the p1 rows: fills T
        constexpr int VP = sizeof(R) == 4 ? 4 : 2;
        const unsigned gs = (unsigned)(a.S / (32 * VP)), npairs = (unsigned)cb(a.M - 1, 2);
        const dim3 pairs((unsigned)cb(t - 1, 2), gs);  // e < t
        if (a.kb && (t - 1) % P2_NB == 0 && t > 3) next(p2_block_kernel<R, VP>, pairs, 32, t, npairs);
        next(p2_kernel<R, VP>, pairs, 32, t, npairs);
    }
    next(rows_kernel<R, K, VW, U, WPB>, grid(2 * t - 1), NT, t);
    return e;
}

template <class R, int K>
static cudaError_t run_chunk(Args<R> a, double *prob, int sms, cudaStream_t st) {
    const int S = a.S, M = a.M;
    const int TB = 256;
    cudaError_t e = cudaSuccess;
    init_kernel<R><<<(S + TB - 1) / TB, TB, 0, st>>>(a);
    for (int t = 1; t <= M; ++t) {
        // products for this step and later ones (inputs: rows < t of the tables)
        const int D = K == 3 ? t - 1 : (int)cb(t - 1, 2);  // K = 4, 5: pairs below t
        if (D > 0) {
            bool tc = false;
            if constexpr (sizeof(R) == 4) tc = a.use_tc != 0;
            if (!tc) e = launch_next(K == 3, w_kernel<R, K>, egrid(S, (uint64_t)D), ETB, 0, st, a, t, D);
            if (e != cudaSuccess) return e;
            const uint64_t rows = K == 3   ? 1 + (uint64_t)(M - t)
                                  : K == 4 ? 1 + 2 * (uint64_t)(M - t)
                                           : 1 + 2 * (uint64_t)(M - t) + cb(M - t, 2);
            if constexpr (sizeof(R) == 4) {
                if (tc) {
                    const unsigned nrt = (unsigned)((rows + TC_M - 1) / TC_M), nk = (unsigned)((D + TC_KC - 1) / TC_KC);
                    // W: about 5000 blocks, each taking its share of the quads
                    const unsigned nx = (unsigned)(S / PREP), quads = (unsigned)((D + TC_KC - 1) / TC_KC * TC_KC / 4);
                    const unsigned cap = 5000 / nx < 16 ? 16 : 5000 / nx, nw = nx * (quads < cap ? quads : cap);
                    e = launch_next(K == 3, operands_kernel<K>, nw + nrt * nk, PREP, 0, st, a, t, rows, D, nw, nrt, nk);
                    if (e == cudaSuccess) e = launch_ztc<K>(a, t, rows, D, sms, st);
                } else {
                    e = launch_zgemm<R, K>(a, t, rows, D, sms, st);
                }
            } else {
                e = launch_zgemm<R, K>(a, t, rows, D, sms, st);
            }
            if (e != cudaSuccess) return e;
        }
        e = step_rows<R, K>(a, t, st);
        if (e != cudaSuccess) return e;
    }
    if (prob) logp_kernel<R><<<(S + TB - 1) / TB, TB, 0, st>>>(a, prob);
    return cudaGetLastError();
}

template <class R>
static cudaError_t run_all(const SamplerCall &c, cudaStream_t st) {
    const SamplerLayout L = sampler_layout(c.M, c.K, c.S, c.precision);
    char *w = static_cast<char *>(c.ws);
    int dev = 0, sms = 0;
    {
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
    }
    Args<R> a{};
    a.M = c.M;
    a.K = c.K;
    a.S = c.S;
    a.opp = c.K == 3 ? 2 : c.orders[0];
    a.op1 = c.K == 3 ? 2 : c.orders[1];
    a.op2 = c.orders[2];  // the caller resolves the defaults per K
    a.off[0] = 0;
    for (int d = 1; d <= 5; ++d) a.off[d] = order_offset(c.M, d);
    a.tab = reinterpret_cast<R *>(w + L.tab);
    a.o = sampler_tabs(c.M, c.K);
    a.gs = a.o.entries * SG;
    a.W = reinterpret_cast<R *>(w + L.W);
    a.At = reinterpret_cast<float *>(w + L.At);
    a.bw = reinterpret_cast<uint32_t *>(w + L.bw);
    a.status = reinterpret_cast<unsigned *>(w);
    {
        cudaError_t e = cudaMemsetAsync(w, 0, 256, st);
        if (e != cudaSuccess) return e;
    }
    a.use_tc = 0;
    a.wait_limit = 1 << 22;
    a.no_loads = 0;
    if (fault_injected("sampler_no_loads")) {
        a.no_loads = 1;
        a.wait_limit = 1 << 10;
    }
    if (sizeof(R) == 4) {
        const char *env = getenv("GBS_SAMPLER_SIMT");
        a.use_tc = (env && *env && *env != '0') || c.S % TC_N != 0 ? 0 : 1;
    }
    {
        R *hs = reinterpret_cast<R *>(w + L.hs);
        double *H = reinterpret_cast<double *>(w + L.H);
        R *ldp = reinterpret_cast<R *>(w + L.lead);
        R *kf = reinterpret_cast<R *>(w + L.kap);
        scale_kernel<R><<<(c.M + 255) / 256, 256, 0, st>>>(c.kappa, c.M, hs, ldp, H);
        launch_kscale<R>(c.kappa, c.M, c.K, hs, kf, st);
        if (c.K == 5 && a.op2 >= 2) {
            R *kb = reinterpret_cast<R *>(w + L.kb);
            const int n = ((c.M - 1) / P2_NB + 1) * (c.M + 1) * P2_NB;
            kb_kernel<R><<<(n + 255) / 256, 256, 0, st>>>(kf + a.off[2], c.M, n, kb);
            a.kb = kb;
        }
        a.kap = kf;
        a.lead = ldp;
        a.H = H;
    }
    for (int s0 = 0; s0 < c.n_samples; s0 += c.S) {
        a.n_valid = c.n_samples - s0 < c.S ? c.n_samples - s0 : c.S;
        const size_t o = (size_t)s0 * c.M;
        a.u = c.u ? c.u + o : nullptr;
        a.force = c.force ? c.force + o : nullptr;
        a.bits = c.bits + o;
        a.q0 = c.q0 ? c.q0 + o : nullptr;
        double *pr = c.prob ? c.prob + s0 : nullptr;
        cudaError_t e = c.K == 3 ? run_chunk<R, 3>(a, pr, sms, st) : c.K == 4 ? run_chunk<R, 4>(a, pr, sms, st) : run_chunk<R, 5>(a, pr, sms, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_sampler(const SamplerCall &c, cudaStream_t st) {
    return c.precision == 0 ? run_all<double>(c, st) : run_all<float>(c, st);
}

}  // namespace smp
}  // namespace gbs

// ---------------------------------------------------------------- C ABI

namespace gbs {
int record_error(int code, const char *msg);
}

namespace {

bool dev_ptr(const void *p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

bool valid_shape(int M, int K, int batch, int precision) {
    return K >= 3 && K <= 5 && M >= K && M <= (K == 3 ? GBS_MAX_MODES_K3 : GBS_MAX_MODES) && batch >= 128 &&
           batch <= GBS_MAX_SAMPLE_BATCH && batch % 128 == 0 &&
           (precision == GBS_SAMPLE_FP64 || precision == GBS_SAMPLE_FP32);
}

}  // namespace

extern "C" {

size_t gbs_sampler_workspace_bytes(int M, int K, int batch, int precision) {
    if (!valid_shape(M, K, batch, precision)) return 0;
    return gbs::smp::sampler_layout(M, K, batch, precision).total;
}

int gbs_sample(const double *kappa, int M, int K, const int *orders, int n_samples, const double *u,
               const uint8_t *force, uint8_t *bits_out, double *logp_out, double *q0_out, int batch, int precision,
               void *workspace, size_t ws_bytes, void *cuda_stream) {
    using gbs::record_error;
    if (!valid_shape(M, K, batch, precision))
        return record_error(GBS_ERR_INVALID_ARG,
                            "need K in {3, 4, 5}, K <= M <= 1024 (4096 for K = 3), batch a multiple of 128 in "
                            "[128, GBS_MAX_SAMPLE_BATCH] and precision GBS_SAMPLE_FP64 or GBS_SAMPLE_FP32");
    if (n_samples < 0) return record_error(GBS_ERR_INVALID_ARG, "n_samples must be >= 0");
    int ord[3] = {3, 3, 2};  // K = 5; K = 4: one order lower, as the paper's rule gives
    if (K == 4) ord[0] = ord[1] = 2, ord[2] = 1;
    if (orders) {
        for (int i = 0; i < 3; ++i) ord[i] = orders[i];
        if (ord[0] < 1 || ord[0] > 3 || ord[1] < 1 || ord[1] > 3 || ord[2] < 1 || ord[2] > 2)
            return record_error(GBS_ERR_INVALID_ARG, "orders must be {1..3, 1..3, 1..2}");
    }
    if (!kappa || !bits_out || !workspace || (!u && !force))
        return record_error(GBS_ERR_INVALID_ARG, "kappa, bits_out, workspace and one of u / force must be non-NULL");
    if (((uintptr_t)kappa & 7) || (u && ((uintptr_t)u & 7)) || (logp_out && ((uintptr_t)logp_out & 7)) ||
        (q0_out && ((uintptr_t)q0_out & 7)) || ((uintptr_t)workspace & 255))
        return record_error(GBS_ERR_INVALID_ARG, "double arrays must be 8-byte aligned, the workspace 256-byte aligned");
    if (!dev_ptr(kappa) || !dev_ptr(bits_out) || !dev_ptr(workspace) || (u && !dev_ptr(u)) ||
        (force && !dev_ptr(force)) || (logp_out && !dev_ptr(logp_out)) || (q0_out && !dev_ptr(q0_out)))
        return record_error(GBS_ERR_INVALID_ARG, "all arrays must be CUDA device (or managed) memory");
    const gbs::smp::SamplerLayout L = gbs::smp::sampler_layout(M, K, batch, precision);
    if (ws_bytes < L.total) return record_error(GBS_ERR_WORKSPACE, "workspace smaller than gbs_sampler_workspace_bytes()");
    if (n_samples == 0) return record_error(GBS_OK, "");
    gbs::smp::SamplerCall c{};
    c.kappa = kappa;
    c.M = M;
    c.K = K;
    c.S = batch;
    c.precision = precision;
    c.n_samples = n_samples;
    for (int i = 0; i < 3; ++i) c.orders[i] = ord[i];
    c.u = u;
    c.force = force;
    c.bits = bits_out;
    c.prob = logp_out;
    c.q0 = q0_out;
    c.ws = workspace;
    cudaError_t e = gbs::smp::launch_sampler(c, static_cast<cudaStream_t>(cuda_stream));
    if (e != cudaSuccess) return record_error(GBS_ERR_CUDA, cudaGetErrorString(e));
    return record_error(GBS_OK, "");
}

}  // extern "C"
