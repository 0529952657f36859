// Device code shared by the single-instance forward kernels (gbs_fwd.cu) and the
// batched kernel (gbs_batch.cu): the combine step, the per-order entry
// functions and one work item of the prefix-tree elimination. See gbs_fwd.cu
// for the formulas.
#pragma once
#include <cooperative_groups.h>

#include <type_traits>

#include "gbs.h"
#include "gbs_common.cuh"
#include "gbs_fwd.cuh"
#include "gbs_refined.cuh"

namespace gbs {

constexpr int FLAT_THREADS = 256;
constexpr int TREE_THREADS = 512;
constexpr int XCAP = 1152;  // per-batch x-entries in shared memory (>= GBS_MAX_MODES)
constexpr int CCAP = kMaxChildren;  // per-batch children

// x * 2^K by its exponent on the integer pipe (GB300 issues 2 FP64 instructions per
// clock and multiprocessor): exact where x and the result are normal numbers; zero,
// infinity, NaN and what lies within 2^|K| of the range's ends come back as they are.
template <int K>
__device__ __forceinline__ double mul_pow2(double x) {
    const unsigned h = (unsigned)__double2hiint(x), e = (h >> 20) & 0x7ffu;
    constexpr unsigned lo = K < 0 ? 1 - K : 1, hi = K < 0 ? 0x7ff : 0x7ff - K;
    const unsigned g = e - lo < hi - lo ? h + (unsigned)(K * (1 << 20)) : h;
    return __hiloint2double((int)g, __double2loint(x));
}

// ---------------------------------------------------------------- shared combine step

// Per-child constants of the gathers. P = {c_3, .., c_D} ascending, NP = D-2
// elements, subsets of P by bitmask over P's positions.
//   baseJ[Q]: table index of {x} + Q is baseJ[Q] + x   (x < min P)
//   baseT[Q]: table index of {j, c2} + Q is baseT[Q] + t, t = C(c2,2) + j
//   idxQ[Q] : table index of Q (Q nonempty)
template <int NP>
__device__ __forceinline__ void child_bases(const int *P, int M, uint64_t *baseJ, uint64_t *baseT, uint64_t *idxQ) {
    uint64_t off[GBS_MAX_ORDER + 2];
    off[0] = 0;
    off[1] = 0;
    for (int m = 2; m <= NP + 2; ++m) off[m] = off[m - 1] + binom(M, m - 1);
#pragma unroll
    for (int q = 0; q < (1 << NP); ++q) {
        int m = __popc(q);
        uint64_t sJ = off[m + 1], sT = off[m + 2], sQ = off[m];
        int i = 0;
#pragma unroll
        for (int e = 0; e < NP; ++e)
            if (q >> e & 1) {
                ++i;
                sJ += binom(P[e], i + 1);
                sT += binom(P[e], i + 2);
                sQ += binom(P[e], i);
            }
        baseJ[q] = sJ;
        baseT[q] = sT;
        idxQ[q] = sQ;
    }
}

template <int NP, int MODE>
__host__ __device__ constexpr double lead_sign();
template <int NP, int MODE>
__device__ __forceinline__ double combine_tail(double acc, int j, int c2, uint32_t t, const uint64_t *baseJ,
                                               const uint64_t *baseT, const double *p0R,
                                               const double *__restrict__ p0tab, const double *__restrict__ outtab);

// Mode-specific value of the leaf S = {j, c2} + P (|P| = NP) given P0(S).
// p0R[R] = P0(R) for nonempty R subset of P.
template <int NP, int MODE>
__device__ __forceinline__ double combine(double P0S, int j, int c2, uint32_t t, const uint64_t *baseJ,
                                          const uint64_t *baseT, const double *p0R, const double *__restrict__ p0tab,
                                          const double *__restrict__ outtab) {
    constexpr int PALL = (1 << NP) - 1;
    if (MODE == MODE_P0) return P0S;
    if (MODE == MODE_MU) {
        double acc = outtab[baseJ[PALL] + c2];  // mu(S')
#pragma unroll
        for (int q = 0; q <= PALL; ++q) {
            const double sg = (__popc(q) & 1) ? -1.0 : 1.0;
            acc = fma(-sg, p0tab[baseJ[q] + j], acc);
            const double t2 = (q == PALL) ? P0S : p0tab[baseT[q] + t];
            acc = fma(sg, t2, acc);
        }
        return acc;
    }
    if (MODE == MODE_SPINC) {
        // c(S) = -c(S') - 2 (-1)^d sum_{R' subset S'} (-2)^{|R'|} P0({j} + R'), d = |S|
        // (the sum of Eq. correlator_sum_cov split by whether R contains j)
        constexpr double lead = ((NP + 2) & 1) ? 2.0 : -2.0;  // -2 (-1)^d
        double acc = -outtab[baseJ[PALL] + c2];                // -c(S')
#pragma unroll
        for (int q = 0; q <= PALL; ++q) {
            const double w = lead * ((__popc(q) & 1) ? -1.0 : 1.0) * (double)(1 << __popc(q));  // (-2)^{|q|}
            acc = fma(w, p0tab[baseJ[q] + j], acc);
            const double t2 = (q == PALL) ? P0S : p0tab[baseT[q] + t];
            acc = fma(-2.0 * w, t2, acc);                      // R' = Q + {c2}
        }
        return acc;
    }
    // MODE_KAPPA: kt(S) = (-1)^d [bracket];  MODE_SPINK: kappa(S) = (-2)^d kt(S) = 2^d [bracket],
    // with the lower-order table holding kappa = (-2)^{|Q|} kt (exact power-of-two scalings).
    // The bracket is accumulated already multiplied by lead_sign (the sign of the
    // order for MODE_KAPPA), which every FMA absorbs as an operand negation.
    constexpr double sd = lead_sign<NP, MODE>();
    return combine_tail<NP, MODE>(fma(-sd * p0tab[j], p0tab[baseJ[PALL] + c2], sd * P0S), j, c2, t, baseJ, baseT,
                                  p0R, p0tab, outtab);
}

// The recursion's weights for the table value of R + {j}, n = |R| (R within P, or
// R = Q + {c2} with n = |Q| + 1): (-1)^n of the order's sign for the click cumulant,
// -2^{-(n+1)} for the spin cumulant (an exponent, no FP64 instruction).
template <int MODE, int N>
__device__ __forceinline__ double weighted(double x, double sd) {
    if constexpr (MODE == MODE_SPINK) return -mul_pow2<-(N + 1)>(x);
    else return (N & 1) ? -sd * x : sd * x;
}
__host__ __device__ constexpr int bits_of(int q) { return q ? (q & 1) + bits_of(q >> 1) : 0; }
// f(integral constant q) for q = Q0 .. Q1 - 1
template <int Q0, int Q1, class F>
__device__ __forceinline__ void for_subsets(F f) {
    if constexpr (Q0 < Q1) {
        f(std::integral_constant<int, Q0>{});
        for_subsets<Q0 + 1, Q1>(f);
    }
}

// Sign carried by the accumulator of the cumulant recursion: (-1)^d for the
// click cumulant (d = NP + 2), + for the spin cumulant.
template <int NP, int MODE>
__host__ __device__ constexpr double lead_sign() {
    return (MODE == MODE_KAPPA && ((NP + 2) & 1)) ? -1.0 : 1.0;
}

// The cumulant recursion (MODE_KAPPA, MODE_SPINK) after its leading term
// acc = lead_sign (P0(S) - P0({j}) P0(S')): the 2^{d-1} - 2 products with
// lower-order cumulants (signs folded into each FMA), then, for the spin
// cumulant, the power of two.
template <int NP, int MODE>
__device__ __forceinline__ double combine_tail(double acc, int j, int c2, uint32_t t, const uint64_t *baseJ,
                                               const uint64_t *baseT, const double *p0R,
                                               const double *__restrict__ p0tab, const double *__restrict__ outtab) {
    constexpr int PALL = (1 << NP) - 1;
    constexpr double sd = lead_sign<NP, MODE>();
    for_subsets<1, PALL + 1>([&](auto q) {
        acc = fma(weighted<MODE, bits_of(q())>(outtab[baseJ[q()] + j], sd), p0tab[baseJ[PALL ^ q()] + c2], acc);
    });
    for_subsets<0, PALL>([&](auto q) {
        acc = fma(weighted<MODE, bits_of(q()) + 1>(outtab[baseT[q()] + t], sd), p0R[PALL ^ q()], acc);
    });
    if constexpr (MODE == MODE_SPINK) return mul_pow2<NP + 2>(acc);
    return acc;
}

// The cumulant recursion of the refined path (MODE_KAPPA, MODE_SPINK) in terms of
// the no-click cumulants ky (kt = (-1)^d ky, kappa = 2^d ky):
//   ky(S) = P0(S) - P0({j}) P0(S') - sum_{empty != R proper subset S'} ky(R + {j}) P0(S' - R).
// The lead term P0(S') (r0 (1 + eta) - P0({j})) and the products whose factors are
// particular to j and to c2 (R within P) run on pairs from the tables' float-pair
// copies: every order-5 entry then takes 8 FP64 instructions instead of 15, and
// GB300's FP64 pipe (1/63 of the FP32 rate) no longer binds alone. The products
// with c2 in R keep FP64: one factor is the same for a whole child. The pairs'
// error, about 2^-46 of a product, is below the determinants' own.
// In two parts, so that the table values are not live across the determinant step:
// the products, then the lead term.
struct PairSum {
    Acc g;       // -sum over R within P
    double acc;  // sum over R with c2, with the order's sign
};
// k[q] = ky({j} + Q), p[q] = P0({c2} + Q) as pairs, u[q] = the mode's table at
// {j, c2} + Q, for the subsets Q of P (bitmasks q).
template <int NP, int MODE>
__device__ __forceinline__ PairSum combine_products(const float2 (&k)[1 << NP], const float2 (&p)[1 << NP],
                                                    const double (&u)[1 << NP], const double *p0R) {
    constexpr int PALL = (1 << NP) - 1;
    constexpr double sd = lead_sign<NP, MODE>();
    PairSum r;
    r.acc = weighted<MODE, 1>(u[0], sd) * p0R[PALL];
    for_subsets<1, PALL>([&](auto q) { r.acc = fma(weighted<MODE, bits_of(q()) + 1>(u[q()], sd), p0R[PALL ^ q()], r.acc); });
    const DF f = df_mulu(DF{-k[1].x, -k[1].y}, DF{p[PALL ^ 1].x, p[PALL ^ 1].y});
    r.g = Acc{f.h, f.l};
#pragma unroll
    for (int q = 2; q <= PALL; ++q) acc_sub(r.g, DF{k[q].x, k[q].y}, DF{p[PALL ^ q].x, p[PALL ^ q].y});
    return r;
}
// ps = P0(S'), pj = P0({j}) as pairs.
template <int NP, int MODE>
__device__ __forceinline__ double combine_lead(PairSum r, float r0, float eta, float2 pj, float2 ps) {
    // w = r0 + r0 eta - P0({j}): two-sum of the leading parts, the rest gathered
    const float s = __fsub_rn(r0, pj.x);
    const float bb = __fsub_rn(s, r0);
    const float e1 = __fsub_rn(__fsub_rn(r0, __fsub_rn(s, bb)), __fadd_rn(pj.x, bb));
    const float pr = r0 * eta;
    const float lo = __fadd_rn(__fsub_rn(e1, pj.y), __fadd_rn(pr, __fmaf_rn(r0, eta, -pr)));
    acc_sub(r.g, DF{-ps.x, -ps.y}, df_norm(s, lo));
    // into FP64, with the order's sign
    const unsigned flip = lead_sign<NP, MODE>() < 0 ? 0x80000000u : 0u;
    const double v = r.acc + f2d_bits(__uint_as_float(__float_as_uint(r.g.s) ^ flip)) +
                     f2d_bits(__uint_as_float(__float_as_uint(r.g.t) ^ flip));
    if constexpr (MODE == MODE_SPINK) return mul_pow2<NP + 2>(v);
    return v;
}

template <int MODE>
__device__ __forceinline__ void store_entry(const FwdArgs &a, int d, uint64_t idx, double P0, double v, bool write_p0);

// ---------------------------------------------------------------- small kernels

// Block (x, y) of A = (V+I)/2 from V.
__device__ __forceinline__ Blk vblk(const double *__restrict__ V, int M, int x, int y) {
    const size_t n2 = 2 * (size_t)M;
    double a00 = V[x * n2 + y], a01 = V[x * n2 + y + M];
    double a10 = V[(x + M) * n2 + y], a11 = V[(x + M) * n2 + y + M];
    if (x == y) {
        a00 += 1.0;
        a11 += 1.0;
    }
    return Blk{0.5 * a00, 0.5 * a01, 0.5 * a10, 0.5 * a11};
}

// Writes block idx = x*M + y of A = (V+I)/2 as 4 doubles, and (if Af is not
// null) as 4 hi floats then 4 lo floats for the refined path.
__device__ __forceinline__ void pack_entry(const double *__restrict__ V, int M, double *__restrict__ A,
                                           float *__restrict__ Af, int idx) {
    const int x = idx / M, y = idx - x * M;
    const Blk b = vblk(V, M, x, y);
    store_blk(A + 4 * (size_t)idx, b);
    if (Af) {
        float4 h, l;
        split_df(b.a00, h.x, l.x);
        split_df(b.a01, h.y, l.y);
        split_df(b.a10, h.z, l.z);
        split_df(b.a11, h.w, l.w);
        float4 *f = reinterpret_cast<float4 *>(Af) + 2 * (size_t)idx;
        f[0] = h;
        f[1] = l;
    }
}


// P0 of one mode from its block of A; NaN (ok = false) unless positive definite.
template <bool DISP>
__device__ __forceinline__ double p0_single(const Blk &b, const double *mean, int M, int j, bool &ok) {
    const Sym s = blk_sym(b);
    const double det = det_sym(s);
    const double rs = rsqrt(det);
    double P0 = rs;
    if (DISP) P0 *= exp(-quad_inv(s, rs * rs, half_mean(mean, M, j)));
    ok = det > 0.0 && s.s00 > 0.0;
    return ok ? P0 : __longlong_as_double(0x7ff8000000000000ULL);
}
// mu({j}) = kt({j}) = 1 - P0({j});  c({j}) = kappa({j}) = 2 P0({j}) - 1
template <int MODE>
__device__ __forceinline__ double single_value(double P0) {
    return (MODE == MODE_MU || MODE == MODE_KAPPA) ? 1.0 - P0 : (MODE == MODE_SPINC || MODE == MODE_SPINK) ? fma(2.0, P0, -1.0) : P0;
}

// Orders 1 and 2 read V itself (order 2 forms its modes' own P0), so that they can
// share a launch with the packing.
template <int MODE, bool DISP = false>
__device__ __forceinline__ void order1_entry(const FwdArgs &a, int j, bool write_p0) {
    bool ok;
    const double P0 = p0_single<DISP>(vblk(a.V, a.M, j, j), a.mean, a.M, j, ok);
    if (!ok) flag_status(a.status, ST_NOT_POSDEF);
    store_entry<MODE>(a, 1, (uint64_t)j, P0, single_value<MODE>(P0), write_p0);
}


template <int MODE, bool DISP = false>
__device__ __forceinline__ void order2_entry(const FwdArgs &a, uint32_t t, bool write_p0) {
    const int M = a.M;
    int c2, j;
    pair_decode(t, c2, j);
    bool ok, ok2, okj;
    double detp;
    const Blk b2 = vblk(a.V, M, c2, c2), bj = vblk(a.V, M, j, j);
    const double p2 = p0_single<DISP>(b2, a.mean, M, c2, ok2), pj = p0_single<DISP>(bj, a.mean, M, j, okj);
    const LInv m2 = chol2_inv(blk_sym(b2), ok, detp);
    const Blk w = lmul(m2, vblk(a.V, M, c2, j));
    const Sym sch = sym_sub_gram(blk_sym(bj), w);
    const double det2 = det_sym(sch);
    const double rs = rsqrt(det2);
    double P0 = p2 * rs;
    if (DISP) {
        const Vec2 r = sub_wtg(half_mean(a.mean, M, j), w, lvec(m2, half_mean(a.mean, M, c2)));
        P0 *= exp(-quad_inv(sch, rs * rs, r));
    }
    if (!(det2 > 0.0) || !ok) {
        flag_status(a.status, ST_NOT_POSDEF);
        P0 = __longlong_as_double(0x7ff8000000000000ULL);
    }
    const uint64_t idx = (uint64_t)M + t;
    double v = P0;
    if (MODE == MODE_MU) v = single_value<MODE>(p2) - pj + P0;
    if (MODE == MODE_KAPPA) v = fma(-pj, p2, P0);
    // c({j,c2}) = -c({c2}) - 2 (P0({j}) - 2 P0(S));  kappa(S) = 4 (P0(S) - P0({j}) P0({c2}))
    if (MODE == MODE_SPINC) v = fma(4.0, P0, fma(-2.0, pj, -single_value<MODE>(p2)));
    if (MODE == MODE_SPINK) v = 4.0 * fma(-pj, p2, P0);
    store_entry<MODE>(a, 2, idx, P0, v, write_p0);
}


template <int MODE, bool DISP = false>
__device__ __forceinline__ void order3_entry(const FwdArgs &a, uint64_t r, bool write_p0) {
    const int M = a.M;
    int s[3];
    colex_unrank(r, 3, s);
    const int j = s[0], c2 = s[1], c3 = s[2];
    const uint32_t t = (uint32_t)binom2(c2) + j;
    bool ok3, ok2;
    double dd;
    const LInv m3 = chol2_inv(blk_sym(ablk(a.A, M, c3, c3)), ok3, dd);
    const Blk z2 = lmul(m3, ablk(a.A, M, c3, c2));
    const Blk zj = lmul(m3, ablk(a.A, M, c3, j));
    const LInv m2 = chol2_inv(sym_sub_gram(blk_sym(ablk(a.A, M, c2, c2)), z2), ok2, dd);
    const Sym dj = sym_sub_gram(blk_sym(ablk(a.A, M, j, j)), zj);
    const Blk X = blk_sub_cross(ablk(a.A, M, c2, j), z2, zj);
    const Blk w = lmul(m2, X);
    const Sym sch = sym_sub_gram(dj, w);
    const double det2 = det_sym(sch);
    uint64_t baseJ[2], baseT[2], idxQ[2];
    const int P[1] = {c3};
    child_bases<1>(P, M, baseJ, baseT, idxQ);
    const double rs = rsqrt(det2);
    double P0 = a.p0[baseJ[1] + c2] * rs;
    if (DISP) {
        const Vec2 g3 = lvec(m3, half_mean(a.mean, M, c3));
        const Vec2 r2 = sub_wtg(half_mean(a.mean, M, c2), z2, g3);
        const Vec2 rj = sub_wtg(half_mean(a.mean, M, j), zj, g3);
        P0 *= exp(-quad_inv(sch, rs * rs, sub_wtg(rj, w, lvec(m2, r2))));
    }
    if (!(det2 > 0.0) || !ok3 || !ok2) {
        flag_status(a.status, ST_NOT_POSDEF);
        P0 = __longlong_as_double(0x7ff8000000000000ULL);
    }
    const double p0R[2] = {0.0, a.p0[idxQ[1]]};
    const double v = combine<1, MODE>(P0, j, c2, t, baseJ, baseT, p0R, a.p0, a.out);
    store_entry<MODE>(a, 3, baseT[1] + t, P0, v, write_p0);
}


// ---------------------------------------------------------------- tree kernel

// CC: children per batch it has room for. YC > 0: the slot-free form of the
// refined path, which keeps the item's elimination rows Y(x) (x < c4 <= YC) in
// yq for the whole item and forms every Schur-complement block it needs from
// them instead of reading a slot.
template <int D, int XC = XCAP, bool DISP = false, int CC = CCAP, int YC = 0>
struct TreeShared {
    static constexpr int NP = D - 2;       // |P|
    static constexpr int NQ = 1 << NP;     // subsets of P
    // item decode: K + 1 <= M - 2 prefix entries, M <= XC + 1 for the shapes whose
    // x-entry area is smaller than GBS_MAX_MODES
    uint32_t c4pref[XC < GBS_MAX_MODES ? XC + 3 : GBS_MAX_MODES + 2];
    uint32_t item;
    // uniform pivots of the item's U (and, displaced, their whitened half-means)
    double upiv[DISP ? 10 : 8];
    // children of the current batch
    int c3[CC];
    int xoff[CC + 1];
    // (refined cumulants: subsets without c3, whose bases all children share, first)
    alignas(16) uint64_t baseJ[CC][NQ];
    alignas(16) uint64_t baseT[CC][NQ];
    alignas(16) double p0R[CC][NQ];
    double m3[CC][3];
    float p3f[CC][6];  // refined path: the c3 pivot's factors i0, l, i1 as pairs (Piv)
    double g3[DISP ? CC : 1][2];  // displaced: whitened half-mean of each child's c3 pivot
    // Per x-entry data, structure of arrays. FP64 path (10 double rows):
    // z(x) = m3 * S_U[c3, x] (rows 0-3), d(x) = S_U[x,x] - z^T z (rows 4-6),
    // inverse c2-pivot factor m2(x) (rows 7-9). Refined-FP32 path (6 float4
    // rows, consecutive entries in consecutive 16-byte words): z hi (0), z lo (1),
    // (d hi 00 01 11, d lo 00) (2), (d lo 01 11, 0, 0) (3), the c2 pivot's factors
    // (i0 h l, l h l) (4), (i1 h l, 0, 0) (5). A leaf loads rows 0-3 of j and
    // 0, 1, 4, 5 of c2.
    // Displaced states add 4 double rows: the reduced half-mean r(x) after
    // eliminating U and c3 (rows 10-11) and its whitened form g2(x) = m2(x) r(x)
    // as a c2 pivot (rows 12-13).
    // Before the batches of an item start, the same storage holds Y(x) of the
    // elimination of U (8 doubles per mode x < c4, or 4 float4 rows of pairs).
    static constexpr int XROWS = DISP ? 14 : 10;
    static constexpr int XBYTES = (6 * 16 > XROWS * 8 ? 6 * 16 : XROWS * 8) * XC;
    alignas(16) unsigned char xraw[XBYTES];
    // slot-free form: Y(x) as 16 floats (hi, lo of y5 00 01 10 11, then of y4) in
    // four float4 rows, row r holding floats 4r..4r+3 of every x
    alignas(16) float4 yq[YC > 0 ? 4 : 1][YC > 0 ? YC : 1];
    __device__ double (*xe())[XC] { return reinterpret_cast<double(*)[XC]>(xraw); }
    __device__ float4 (*xq())[XC] { return reinterpret_cast<float4(*)[XC]>(xraw); }
};

// Schur-complement slots: 2x2 blocks at pair index, then the diagonal blocks, 32
// bytes each. FP64 path: 4 doubles (diagonal: 00 01 11). Refined path: 4 hi floats
// then 4 lo floats (diagonal: h00 h01 h11 l00 | l01 l11).
__device__ __forceinline__ Sym slot_diag(const double *sdiag, int x) {
    return Sym{sdiag[4 * x], sdiag[4 * x + 1], sdiag[4 * x + 2]};
}
__device__ __forceinline__ ABlk slot_pair_df(const double *slot, size_t q) {
    const float4 *f = reinterpret_cast<const float4 *>(slot) + 2 * q;
    const float4 h = f[0], l = f[1];
    return ABlk{Acc{h.x, l.x}, Acc{h.y, l.y}, Acc{h.z, l.z}, Acc{h.w, l.w}};
}
__device__ __forceinline__ ASym slot_diag_df(const double *sdiag, int x) {
    const float4 *f = reinterpret_cast<const float4 *>(sdiag) + 2 * (size_t)x;
    const float4 a = f[0];
    const float2 b = *reinterpret_cast<const float2 *>(f + 1);
    return ASym{Acc{a.x, a.w}, Acc{a.y, b.x}, Acc{a.z, b.y}};
}

// Schur-complement block S_U[x][y] (x >= y) of the refined path formed from A's
// blocks and the rows Y(x), Y(y) of the eliminated modes U (rows 0, 1 of c5 for
// D = 5, then 2, 3 of c4), normalised:
// b_uv -= sum_k y(x)_ku y(y)_kv. Shared by the slot build and the slot-free form,
// so both give the same bits.
template <int D, class Rows>
__device__ __forceinline__ DFBlk su_block(const float *__restrict__ Af, int M, const Rows yq, int x, int y) {
    const float4 *f = reinterpret_cast<const float4 *>(Af) + 2 * ((size_t)x * M + y);
    const float4 h = f[0], l = f[1];
    ABlk b{Acc{h.x, l.x}, Acc{h.y, l.y}, Acc{h.z, l.z}, Acc{h.w, l.w}};
#pragma unroll
    for (int k = (D == 5 ? 0 : 2); k < 4; ++k) {
        const float4 u = yq[k][x], v = yq[k][y];
        acc_sub_row(b, DF{u.x, u.y}, DF{u.z, u.w}, DF{v.x, v.y}, DF{v.z, v.w});
    }
    return DFBlk{acc_norm(b.a00), acc_norm(b.a01), acc_norm(b.a10), acc_norm(b.a11)};
}
__device__ __forceinline__ ABlk acc_of(const DFBlk &b) {
    return ABlk{Acc{b.a00.h, b.a00.l}, Acc{b.a01.h, b.a01.l}, Acc{b.a10.h, b.a10.l}, Acc{b.a11.h, b.a11.l}};
}
__device__ __forceinline__ ASym acc_sym(const DFBlk &b) {
    return ASym{Acc{b.a00.h, b.a00.l}, Acc{b.a01.h, b.a01.l}, Acc{b.a11.h, b.a11.l}};
}

// Number of stride classes the children c3 in [2, c4) of one U are split into.
__host__ __device__ __forceinline__ int n_classes(int c4, uint64_t target) {
    const uint64_t leaves = binom(c4, 3);
    uint64_t n = (leaves + target - 1) / target;
    if (n < 1) n = 1;
    if (n > (uint64_t)(c4 - 2)) n = (uint64_t)(c4 - 2);
    return (int)n;
}

// Items of the order-D prefix tree whose top element (c5 for D = 5, c4 for
// D = 4) lies in [lo, hi): the largest c4 that has any, and the items of one c4.
template <int D>
__host__ __device__ __forceinline__ int c4_max(int M, int hi) {
    const int top = hi < M ? hi : M;
    return D == 5 ? top - 2 : top - 1;
}
template <int D>
__host__ __device__ __forceinline__ int c4_max(int M) {
    return c4_max<D>(M, M);
}

// First top element c5 of the items of one c4 (D = 5).
__host__ __device__ __forceinline__ int c5_first(int c4, int lo) { return c4 + 1 > lo ? c4 + 1 : lo; }

template <int D>
__host__ __device__ __forceinline__ uint32_t items_for_c4(int M, int c4, uint64_t target, int lo, int hi) {
    int nU;
    if (D == 5) {
        const int first = c5_first(c4, lo), last = hi < M ? hi : M;
        nU = last > first ? last - first : 0;
    } else {
        nU = (c4 >= lo && c4 < hi) ? 1 : 0;
    }
    return (uint32_t)nU * (uint32_t)n_classes(c4, target);
}
template <int D>
__host__ __device__ __forceinline__ uint32_t items_for_c4(int M, int c4, uint64_t target) {
    return items_for_c4<D>(M, c4, target, 0, M);
}

// Stores entry idx (table layout) of order d: into the caller's slice of order
// kmax during a range call, else into the P0 table (write_p0) and the mode's table.
template <int MODE>
__device__ __forceinline__ void store_entry(const FwdArgs &a, int d, uint64_t idx, double P0, double v, bool write_p0) {
    if (a.top && d == a.kmax) {
        a.top[idx - a.top_base] = (MODE == MODE_P0) ? P0 : v;
        return;
    }
    if (write_p0) a.p0[idx] = P0;
    if (MODE != MODE_P0) a.out[idx] = v;
    if constexpr (MODE == MODE_KAPPA || MODE == MODE_SPINK) {
        if (a.p0p && d < a.kmax) {
            // ky = (-1)^d kt = 2^{-d} kappa
            a.p0p[idx] = pair_of_double(P0);
            a.kyp[idx] = pair_of_double(MODE == MODE_SPINK ? v * (1.0 / (double)(1 << d)) : (d & 1) ? -v : v);
        }
    }
}

// One work item of the prefix-tree kernel: U = {c4, c5} (D = 5) or {c4} (D = 4),
// children c3 = c4-1-s, c4-1-s-nc, ... >= 2 (stride class s of nc). Called by all
// threads of the block; sh is the block's shared memory, slot its scratch slot.
//
// Displaced states (DISP, FP64 only) carry the reduced half-means along: the
// slot holds r_U(x) after the Schur blocks, the x-entries r(x) and g2(x), and
// each leaf multiplies its P0 by exp(-r^T Sch^{-1} r).
//
// CL: the CTAs of a thread-block cluster share one slot and one U. CTA `part` of
// `nparts` writes every nparts-th chunk of NT Schur blocks, and a cluster-wide
// barrier (release / acquire, so the other CTAs' global writes are visible)
// replaces the block barrier after the build; the caller passes s = part,
// nc = nparts, so each CTA then takes one stride class of the children.
//
// YC > 0 (refined path only): no slot. Y(x) stays in shared memory for the
// whole item and each Schur-complement block is formed where it is used
// (su_block): the c3 pivots, z(x) and d(x) of the batch setup, and one block per
// leaf pair and batch. That trades FP32 work (about 60 more FP32 instructions
// per order-5 leaf with a 384-entry x area) for the slot's DRAM writes and
// re-reads.
template <int D, int MODE, int PREC, int NT = TREE_THREADS, int XC = XCAP, bool DISP = false, bool CL = false,
          int CC = CCAP, int YC = 0>
__device__ __forceinline__ void tree_item(const FwdArgs &a, TreeShared<D, XC, DISP, CC, YC> &sh, double *const slot,
                                          const int c4, const int c5, const int s, const int nc, const bool write_p0,
                                          const int ccap_in = CCAP, const int part = 0, const int nparts = 1) {
    static_assert(!DISP || PREC == 0, "displaced states run in FP64");
    static_assert(!(DISP && CL), "displaced states run without clusters");
    constexpr bool NOSLOT = YC > 0;
    static_assert(!NOSLOT || (PREC == 1 && !CL), "the slot-free form is the refined path's, without clusters");
    constexpr bool PAIRS = PREC == 1 && (MODE == MODE_KAPPA || MODE == MODE_SPINK);  // combine_products
    const int ccap = ccap_in < CC ? ccap_in : CC;
    using SH = TreeShared<D, XC, DISP, CC, YC>;
    constexpr int NP = SH::NP;
    constexpr int NQ = SH::NQ;
    constexpr int PALL = NQ - 1;
    double(*const xe)[XC] = sh.xe();
    float4(*const xq)[XC] = sh.xq();
    const int tid = threadIdx.x;
    const int M = a.M;
    double *const sdiag = slot + 4 * binom2(M);
    double *const rU = sdiag + 4 * (size_t)M;  // displaced: reduced half-means, 2 per mode
    const double *__restrict__ A = a.A;

    if constexpr (NOSLOT) {
        if (c4 > YC) {  // Y rows beyond the shared area (the launcher bounds M): reject, block-uniformly
            if (tid == 0) flag_status(a.status, ST_BAD_INDEX);
            return;
        }
    }
    // ---- Schur complement of A after eliminating U, modes < c4 -> slot
    // uniform pivots: m5 = chol(A[c5,c5])^{-1}, y5(c4), m4 = chol(Pi4)^{-1}
    if (tid == 0) {
        bool ok = true, ok2 = true;
        double dd;
        LInv m5{0, 0, 0};
        Blk y5c4{0, 0, 0, 0};
        Sym pi4 = blk_sym(ablk(A, M, c4, c4));
        if (D == 5) {
            m5 = chol2_inv(blk_sym(ablk(A, M, c5, c5)), ok, dd);
            y5c4 = lmul(m5, ablk(A, M, c5, c4));
            pi4 = sym_sub_gram(pi4, y5c4);
        }
        const LInv m4 = chol2_inv(pi4, ok2, dd);
        if (!ok || !ok2) flag_status(a.status, ST_NOT_POSDEF);
        sh.upiv[0] = m5.m00; sh.upiv[1] = m5.m10; sh.upiv[2] = m5.m11;
        sh.upiv[3] = m4.m00; sh.upiv[4] = m4.m10; sh.upiv[5] = m4.m11;
        if constexpr (DISP) {
            Vec2 g5{0, 0}, r4 = half_mean(a.mean, M, c4);
            if (D == 5) {
                g5 = lvec(m5, half_mean(a.mean, M, c5));
                r4 = sub_wtg(r4, y5c4, g5);
            }
            const Vec2 g4 = lvec(m4, r4);
            sh.upiv[6] = g5.v0; sh.upiv[7] = g5.v1; sh.upiv[8] = g4.v0; sh.upiv[9] = g4.v1;
        }
    }
    __syncthreads();
    {
        // Y(x) = [y5(x); y4(x)] into the x-entry area (it is free until the batches start):
        // 8 doubles per x (FP64 path) or 4 float4 rows of pairs (refined path); x < c4 <= 1023
        double *Y = &xe[0][0];
        const LInv m5{sh.upiv[0], sh.upiv[1], sh.upiv[2]};
        const LInv m4{sh.upiv[3], sh.upiv[4], sh.upiv[5]};
        Blk y5c4{0, 0, 0, 0};
        if (D == 5) y5c4 = lmul(m5, ablk(A, M, c5, c4));
        for (int x = tid; x < c4; x += NT) {
            Blk y5{0, 0, 0, 0};
            Blk r4 = ablk(A, M, c4, x);
            if (D == 5) {
                y5 = lmul(m5, ablk(A, M, c5, x));
                r4 = blk_sub_cross(r4, y5c4, y5);
            }
            const Blk y4 = lmul(m4, r4);
            if constexpr (DISP) {
                Vec2 r = half_mean(a.mean, M, x);
                if (D == 5) r = sub_wtg(r, y5, Vec2{sh.upiv[6], sh.upiv[7]});
                r = sub_wtg(r, y4, Vec2{sh.upiv[8], sh.upiv[9]});
                rU[2 * x] = r.v0;
                rU[2 * x + 1] = r.v1;
            }
            const double v[8] = {y5.a00, y5.a01, y5.a10, y5.a11, y4.a00, y4.a01, y4.a10, y4.a11};
            if constexpr (PREC == 0) {
#pragma unroll
                for (int k = 0; k < 8; ++k) Y[8 * x + k] = v[k];
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float4 r;
                    split_df(v[2 * k], r.x, r.y);
                    split_df(v[2 * k + 1], r.z, r.w);
                    if constexpr (NOSLOT) sh.yq[k][x] = r;
                    else xq[k][x] = r;
                }
            }
        }
        __syncthreads();
        // the slot build (the slot-free form has nothing more to do: Y is in place)
        if constexpr (!NOSLOT) {
        const uint32_t npairs = (uint32_t)binom2(c4);
        for (uint32_t qi = (uint32_t)(part * NT + tid); qi < npairs + (uint32_t)c4; qi += (uint32_t)(nparts * NT)) {
            int x, y;
            if (qi < npairs) pair_decode(qi, x, y);
            else x = y = (int)(qi - npairs);
            if (PREC == 0) {
                const double *px = Y + 8 * x, *py = Y + 8 * y;
                Blk b = ablk(A, M, x, y);
                const Blk y5x{px[0], px[1], px[2], px[3]}, y5y{py[0], py[1], py[2], py[3]};
                const Blk y4x{px[4], px[5], px[6], px[7]}, y4y{py[4], py[5], py[6], py[7]};
                if (D == 5) b = blk_sub_cross(b, y5x, y5y);
                b = blk_sub_cross(b, y4x, y4y);
                if (qi < npairs) store_blk(slot + 4 * (size_t)qi, b);
                else store_blk(sdiag + 4 * (size_t)x, Blk{b.a00, 0.5 * (b.a01 + b.a10), b.a11, 0.0});
            } else {
                const DFBlk g = su_block<D>(a.Af, M, xq, x, y);
                const DF b[4] = {g.a00, g.a01, g.a10, g.a11};
                if (qi < npairs) {
                    float4 *f = reinterpret_cast<float4 *>(slot) + 2 * (size_t)qi;
                    f[0] = make_float4(b[0].h, b[1].h, b[2].h, b[3].h);
                    f[1] = make_float4(b[0].l, b[1].l, b[2].l, b[3].l);
                } else {
                    float4 *f = reinterpret_cast<float4 *>(sdiag) + 2 * (size_t)x;
                    f[0] = make_float4(b[0].h, b[1].h, b[3].h, b[0].l);
                    f[1] = make_float4(b[1].l, b[3].l, 0.f, 0.f);
                }
            }
        }
        if constexpr (CL) cooperative_groups::this_cluster().sync();
        else __syncthreads();
        }
    }

    // ---- children c3 = c4-1-s, c4-1-s-nc, ... >= 2, processed in batches
    const int cfirst = c4 - 1 - s;
    const int nchild = (cfirst >= 2) ? (cfirst - 2) / nc + 1 : 0;
    int k0 = 0;
    while (k0 < nchild) {
        // batch [k0, k0+nb): identical arithmetic in every thread
        int nb = 0, xs = 0;
        while (k0 + nb < nchild && nb < ccap) {
            const int c3 = cfirst - (k0 + nb) * nc;
            if (xs + c3 > XC) break;
            xs += c3;
            ++nb;
        }
        if (nb == 0) {  // a child wider than the x-entry area: reject instead of spinning
            if (tid == 0) flag_status(a.status, ST_BAD_INDEX);
            break;
        }
        // pre-setup: one thread per child
        if (tid < nb) {
            const int b = tid;
            const int c3 = cfirst - (k0 + b) * nc;
            int xo = 0;
            for (int q = 0; q < b; ++q) {
                const int cq = cfirst - (k0 + q) * nc;
                xo += cq;
            }
            sh.c3[b] = c3;
            sh.xoff[b] = xo;
            if (b == nb - 1) sh.xoff[nb] = xo + c3;
            int P[3] = {c3, c4, c5};
            uint64_t bj[NQ], bt[NQ], idxQ[NQ];
            child_bases<NP>(P, M, bj, bt, idxQ);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int at = PAIRS ? (q & 1) * (NQ / 2) + (q >> 1) : q;
                sh.baseJ[b][at] = bj[q];
                sh.baseT[b][at] = bt[q];
            }
            sh.p0R[b][0] = 0.0;
#pragma unroll
            for (int q = 1; q < NQ; ++q) sh.p0R[b][q] = a.p0[idxQ[q]];
            bool ok;
            if constexpr (PREC == 0) {
                double dd;
                const LInv m3 = chol2_inv(slot_diag(sdiag, c3), ok, dd);
                sh.m3[b][0] = m3.m00; sh.m3[b][1] = m3.m10; sh.m3[b][2] = m3.m11;
                if constexpr (DISP) {
                    const Vec2 g3 = lvec(m3, Vec2{rU[2 * c3], rU[2 * c3 + 1]});
                    sh.g3[b][0] = g3.v0;
                    sh.g3[b][1] = g3.v1;
                }
            } else {
                ASym p;
                if constexpr (NOSLOT) p = acc_sym(su_block<D>(a.Af, M, sh.yq, c3, c3));
                else p = slot_diag_df(sdiag, c3);
                const Piv p3 = pivot_of(p, ok);
                sh.p3f[b][0] = p3.i0.h; sh.p3f[b][1] = p3.i0.l; sh.p3f[b][2] = p3.l.h;
                sh.p3f[b][3] = p3.l.l; sh.p3f[b][4] = p3.i1.h; sh.p3f[b][5] = p3.i1.l;
            }
            if (!ok) flag_status(a.status, ST_NOT_POSDEF);
        }
        __syncthreads();
        // setup: eliminate c3 for every x < c3 of every child in the batch
        for (int e = tid; e < xs; e += NT) {
            int lo2 = 0, hi2 = nb;
            while (hi2 - lo2 > 1) {
                const int mid = (lo2 + hi2) >> 1;
                if (sh.xoff[mid] <= e) lo2 = mid;
                else hi2 = mid;
            }
            const int b = lo2;
            const int c3 = sh.c3[b];
            const int x = e - sh.xoff[b];
            if (PREC == 0) {
                const LInv m3{sh.m3[b][0], sh.m3[b][1], sh.m3[b][2]};
                const Blk z = lmul(m3, load_blk(slot + 4 * (binom2(c3) + x)));
                const Sym dx = sym_sub_gram(slot_diag(sdiag, x), z);
                xe[0][e] = z.a00; xe[1][e] = z.a01; xe[2][e] = z.a10; xe[3][e] = z.a11;
                xe[4][e] = dx.s00; xe[5][e] = dx.s01; xe[6][e] = dx.s11;
                Vec2 r3{0, 0};
                if constexpr (DISP) {
                    r3 = sub_wtg(Vec2{rU[2 * x], rU[2 * x + 1]}, z, Vec2{sh.g3[b][0], sh.g3[b][1]});
                    xe[10][e] = r3.v0; xe[11][e] = r3.v1;
                }
                if (x >= 1) {
                    bool ok;
                    double dd;
                    const LInv m2 = chol2_inv(dx, ok, dd);
                    if (!ok) flag_status(a.status, ST_NOT_POSDEF);
                    xe[7][e] = m2.m00; xe[8][e] = m2.m10; xe[9][e] = m2.m11;
                    if constexpr (DISP) {
                        const Vec2 g2 = lvec(m2, r3);
                        xe[12][e] = g2.v0; xe[13][e] = g2.v1;
                    }
                }
            } else {
                // the pivot rows z(x) of c3, d(x) = S_U[x, x] - z^T z, and x as a c2 pivot
                ABlk S;
                ASym dx;
                if constexpr (NOSLOT) {
                    S = acc_of(su_block<D>(a.Af, M, sh.yq, c3, x));
                    dx = acc_sym(su_block<D>(a.Af, M, sh.yq, x, x));
                } else {
                    S = slot_pair_df(slot, binom2(c3) + x);
                    dx = slot_diag_df(sdiag, x);
                }
                const float *pf = sh.p3f[b];
                DFBlk z = pivot_rows(S, Piv{DF{pf[0], pf[1]}, DF{pf[2], pf[3]}, DF{pf[4], pf[5]}});
                z = DFBlk{df_norm(z.a00.h, z.a00.l), df_norm(z.a01.h, z.a01.l), df_norm(z.a10.h, z.a10.l),
                          df_norm(z.a11.h, z.a11.l)};
                dx = acc_sub_gram(dx, z);
                xq[0][e] = make_float4(z.a00.h, z.a01.h, z.a10.h, z.a11.h);
                xq[1][e] = make_float4(z.a00.l, z.a01.l, z.a10.l, z.a11.l);
                xq[2][e] = make_float4(dx.s00.s, dx.s01.s, dx.s11.s, dx.s00.t);
                xq[3][e] = make_float4(dx.s01.t, dx.s11.t, 0.f, 0.f);
                if (x >= 1) {
                    bool ok;
                    const Piv p = pivot_of(dx, ok);
                    if (!ok) flag_status(a.status, ST_NOT_POSDEF);
                    xq[4][e] = make_float4(p.i0.h, p.i0.l, p.l.h, p.l.l);
                    xq[5][e] = make_float4(p.i1.h, p.i1.l, 0.f, 0.f);
                }
            }
        }
        __syncthreads();
        // leaves (c2, j), j < c2 < c3: pairs t = C(c2, 2) + j on the outer loop and
        // the batch's children (c3 decreasing with b) inside, so each 2x2 block of
        // the slot is read once per batch instead of once per child
        const uint32_t L0 = (uint32_t)binom2(sh.c3[0]);
        for (uint32_t t = tid; t < L0; t += NT) {
            int c2, j;
            pair_decode(t, c2, j);
            Blk S64{0, 0, 0, 0};
            ABlk Sg{};
            if constexpr (PREC == 0) S64 = load_blk(slot + 4 * (size_t)t);
            else if constexpr (NOSLOT) Sg = acc_of(su_block<D>(a.Af, M, sh.yq, c2, j));
            else Sg = slot_pair_df(slot, t);
            // refined cumulants: table values of the subsets without c3, the same for every
            // child of the batch (half of a leaf's gathers)
            [[maybe_unused]] float2 pj, kq[NQ], pq[NQ];
            [[maybe_unused]] double uq[NQ];
            if constexpr (PAIRS) {
                pj = a.p0p[j];
                kq[0] = float2{};
#pragma unroll
                for (int h = 0; h < NQ / 2; ++h) {
                    const uint64_t bj = sh.baseJ[0][h];
                    if (h) kq[2 * h] = a.kyp[bj + j];
                    pq[2 * h] = a.p0p[bj + c2];
                }
            }
            for (int b = 0; b < nb && c2 < sh.c3[b]; ++b) {
                const int xo = sh.xoff[b];
                const int e2 = xo + c2, ej = xo + j;
                const uint64_t *bJ = sh.baseJ[b];
                const uint64_t *bT = sh.baseT[b];
                double P0;
                bool ok;
                if constexpr (PREC == 0) {
                    const double P0Sp = a.p0[bJ[PALL] + c2];
                    const Blk z2{xe[0][e2], xe[1][e2], xe[2][e2], xe[3][e2]};
                    const Blk zj{xe[0][ej], xe[1][ej], xe[2][ej], xe[3][ej]};
                    const LInv m2{xe[7][e2], xe[8][e2], xe[9][e2]};
                    const Sym dj{xe[4][ej], xe[5][ej], xe[6][ej]};
                    const Blk X = blk_sub_cross(S64, z2, zj);
                    const Blk w = lmul(m2, X);
                    const Sym sch = sym_sub_gram(dj, w);
                    const double det2 = det_sym(sch);
                    const double rs = rsqrt(det2);
                    P0 = P0Sp * rs;
                    if constexpr (DISP) {
                        const Vec2 r = sub_wtg(Vec2{xe[10][ej], xe[11][ej]}, w, Vec2{xe[12][e2], xe[13][e2]});
                        P0 *= exp(-quad_inv(sch, rs * rs, r));
                    }
                    ok = det2 > 0.0;
                } else {
                    [[maybe_unused]] PairSum sums;
                    [[maybe_unused]] uint64_t topT = 0, topJ = 0;
                    if constexpr (PAIRS) {
                        // the subsets with c3: odd bitmasks, at NQ / 2 .. NQ - 1
                        const ulonglong2 *bo = reinterpret_cast<const ulonglong2 *>(bJ + NQ / 2);
                        const ulonglong2 *to = reinterpret_cast<const ulonglong2 *>(bT + NQ / 2);
                        const double2 *r2 = reinterpret_cast<const double2 *>(sh.p0R[b]);
                        double p0R[NQ];
#pragma unroll
                        for (int h = 0; h < NQ / 4; ++h) {
                            const ulonglong2 x = bo[h], y = to[h];
                            const uint64_t jo[2] = {x.x, x.y}, tt[2] = {y.x, y.y};
#pragma unroll
                            for (int g = 0; g < 2; ++g) {
                                const int q = 2 * (2 * h + g) + 1;
                                kq[q] = a.kyp[jo[g] + j];
                                pq[q] = a.p0p[jo[g] + c2];
                                uq[q] = q < PALL ? a.out[tt[g] + t] : 0.0;
                            }
                            topJ = x.y;
                            topT = y.y;
                        }
#pragma unroll
                        for (int h = 0; h < NQ / 2; ++h) {
                            const double2 x = r2[h];
                            p0R[2 * h] = x.x;
                            p0R[2 * h + 1] = x.y;
                        }
                        {
                            const ulonglong2 *be = reinterpret_cast<const ulonglong2 *>(bT);
#pragma unroll
                            for (int h = 0; h < NQ / 4; ++h) {
                                const ulonglong2 x = be[h];
                                uq[4 * h] = a.out[x.x + t];
                                uq[4 * h + 2] = a.out[x.y + t];
                            }
                        }
                        sums = combine_products<NP, MODE>(kq, pq, uq, p0R);
                    }
                    const float4 zh2 = xq[0][e2], zl2 = xq[1][e2], zhj = xq[0][ej], zlj = xq[1][ej];
                    const float4 d0 = xq[2][ej], p4 = xq[4][e2];
                    const float2 d1 = *reinterpret_cast<const float2 *>(&xq[3][ej]);
                    const float2 p5 = *reinterpret_cast<const float2 *>(&xq[5][e2]);
                    const DFBlk z2{DF{zh2.x, zl2.x}, DF{zh2.y, zl2.y}, DF{zh2.z, zl2.z}, DF{zh2.w, zl2.w}};
                    const DFBlk zj{DF{zhj.x, zlj.x}, DF{zhj.y, zlj.y}, DF{zhj.z, zlj.z}, DF{zhj.w, zlj.w}};
                    const ASym dj{Acc{d0.x, d0.w}, Acc{d0.y, d1.x}, Acc{d0.z, d1.y}};
                    const Piv pv{DF{p4.x, p4.y}, DF{p4.z, p4.w}, DF{p5.x, p5.y}};
                    float r0, eta;
                    refined_leaf_factor(Sg, z2, zj, dj, pv, r0, eta, ok);
                    if constexpr (PAIRS) {
                        P0 = write_p0 ? refined_leaf_p0(a.p0[topJ + c2], r0, eta) : 0.0;
                        double v = combine_lead<NP, MODE>(sums, r0, eta, pj, pq[PALL]);
                        if (!ok) {
                            flag_status(a.status, ST_NOT_POSDEF);
                            P0 = v = __longlong_as_double(0x7ff8000000000000ULL);
                        }
                        store_entry<MODE>(a, NP + 2, topT + t, P0, v, write_p0);
                        continue;
                    }
                    P0 = refined_leaf_p0(a.p0[bJ[PALL] + c2], r0, eta);
                }
                if (!ok) {
                    flag_status(a.status, ST_NOT_POSDEF);
                    P0 = __longlong_as_double(0x7ff8000000000000ULL);
                }
                const double v = combine<NP, MODE>(P0, j, c2, t, bJ, bT, sh.p0R[b], a.p0, a.out);
                store_entry<MODE>(a, NP + 2, bT[PALL] + t, P0, v, write_p0);
            }
        }
        __syncthreads();
        k0 += nb;
    }
}

}  // namespace gbs
