// Orders 3 and 4 by chunks of pairs: a CTA takes one prefix P = {c3} or {c3, c4}
// and L consecutive pairs t = C(c2, 2) + j, j < c2 < c3, of the subsets
// {j, c2} + P. It eliminates P once for every mode x <= max c2 into shared memory
// (the pivot rows z(x), the reduced diagonal block d(x), and the pivot factor of
// the chunk's own rows c2), and each leaf is then one 2x2 block of A, its updates
// by the pivot rows, a triangular solve and a Schur step. Same operations on the
// same operands in the same order as the prefix-tree kernels (tree_item), so the
// same bits; what it does not have is their global scratch slot, item queue and
// batches of children, whose block-wide barriers bound small and medium tables.
#pragma once
#include "gbs_tree.cuh"

namespace gbs {

constexpr int CHUNK_THREADS = 128;
// Dynamic shared memory a chunk may take: 227 KB less the kernel's static part.
constexpr size_t kChunkSmem = 226 * 1024;

// Shared memory: doubles per mode x <= max c2 and per row c2 of the chunk.
template <int NP, int PREC, bool DISP>
struct ChunkShape {
    // FP64: z of each prefix mode, d (, r); refined (float4 rows): pivot rows of U =
    // P - {c3} and of c3, d
    static constexpr int PX = PREC == 0 ? 4 * NP + 3 + (DISP ? 2 : 0) : 2 * (2 * (NP - 1) + 4);
    static constexpr int PR = PREC == 0 ? 3 + (DISP ? 2 : 0) : 4;
};

// The prefix's own elimination, largest mode first: inverse pivot factors, the
// earlier pivots' rows at the later modes, whitened half-means.
template <int NP>
struct ChunkPrefix {
    LInv m[NP];
    Blk z[NP][NP];  // z[i][k], i < k: pivot row of the i-th mode eliminated at the k-th
    Vec2 g[NP];
    int bad;
};

// The two pivot rows of a block as pairs, one float4 (0h 0l 1h 1l) each.
__device__ __forceinline__ void split_rows(const Blk &y, float4 &r0, float4 &r1) {
    split_df(y.a00, r0.x, r0.y);
    split_df(y.a01, r0.z, r0.w);
    split_df(y.a10, r1.x, r1.y);
    split_df(y.a11, r1.z, r1.w);
}

template <int NP, int MODE, int PREC, bool DISP>
__global__ void __launch_bounds__(CHUNK_THREADS, DISP ? 4 : 6)
    chunk_kernel(FwdArgs a, bool write_p0, int top_hi, uint32_t L) {
    static_assert(NP >= 1 && NP <= 2 && !(DISP && PREC == 1) && !(NP == 1 && PREC == 1), "forms in use");
    constexpr int NQ = 1 << NP, PALL = NQ - 1;
    extern __shared__ __align__(16) double shc[];
    __shared__ ChunkPrefix<NP> pre;
    await_previous();
    if (NP + 2 < a.kmax) release_next();
    const int M = a.M;
    // prefixes with the largest top element first
    int P[3] = {0, 0, 0};
    if constexpr (NP == 1) {
        P[0] = top_hi - (int)blockIdx.x;
    } else {
        int c4, c3;
        pair_decode((uint32_t)binom2(top_hi + 1) - 1 - blockIdx.x, c4, c3);
        P[0] = c3;
        P[1] = c4;
    }
    const int c3 = P[0];
    const uint32_t np = (uint32_t)binom2(c3), t0 = blockIdx.y * L;
    if (t0 >= np) return;
    const uint32_t t1 = t0 + L < np ? t0 + L : np;
    int ca, cl, unused;
    pair_decode(t0, ca, unused);
    pair_decode(t1 - 1, cl, unused);
    const int nx = cl + 1, nr = cl - ca + 1;
    const double nan = __longlong_as_double(0x7ff8000000000000ULL);
    const double *__restrict__ A = a.A;
    auto mode = [&](int k) { return P[NP - 1 - k]; };  // k-th mode eliminated
    // the FP64 pivots of the refined path end with U; its c3 pivot comes from pairs
    constexpr int NE = PREC == 0 ? NP : NP - 1;
    if (threadIdx.x < 32) {
        ChunkPrefix<NP> q;
        q.bad = 0;
#pragma unroll
        for (int k = 0; k < NE; ++k) {
            Sym s = blk_sym(ablk(A, M, mode(k), mode(k)));
#pragma unroll
            for (int i = 0; i < k; ++i) s = sym_sub_gram(s, q.z[i][k]);
            bool ok;
            double dd;
            q.m[k] = chol2_inv(s, ok, dd);
            if (!ok) q.bad = 1;
            if constexpr (DISP) {
                Vec2 r = half_mean(a.mean, M, mode(k));
#pragma unroll
                for (int i = 0; i < k; ++i) r = sub_wtg(r, q.z[i][k], q.g[i]);
                q.g[k] = lvec(q.m[k], r);
            }
#pragma unroll
            for (int n = k + 1; n < NE; ++n) {
                Blk b = ablk(A, M, mode(k), mode(n));
#pragma unroll
                for (int i = 0; i < k; ++i) b = blk_sub_cross(b, q.z[i][k], q.z[i][n]);
                q.z[k][n] = lmul(q.m[k], b);
            }
        }
        if (threadIdx.x == 0) pre = q;
    }
    __syncthreads();
    double *const xs = shc;                                          // FP64: [PX][nx]
    double *const rs = shc + ChunkShape<NP, PREC, DISP>::PX * nx;    // FP64: [PR][nr]
    float4 *const xq = reinterpret_cast<float4 *>(shc);              // refined: [PX / 2][nx]
    float4 *const rq = xq + ChunkShape<NP, PREC, DISP>::PX / 2 * nx;  // refined: [2][nr]
    const bool bad = pre.bad != 0;
    if (bad && threadIdx.x == 0) flag_status(a.status, ST_NOT_POSDEF);
    // U's pivot rows (refined: as pairs), then c3's, d(x), the c2 pivots
    for (int x = threadIdx.x; x < nx; x += CHUNK_THREADS) {
        Blk y[NP];
        Vec2 r{0, 0};
        if constexpr (DISP) r = half_mean(a.mean, M, x);
#pragma unroll
        for (int k = 0; k < NE; ++k) {
            Blk b = ablk(A, M, mode(k), x);
#pragma unroll
            for (int i = 0; i < k; ++i) b = blk_sub_cross(b, pre.z[i][k], y[i]);
            y[k] = lmul(pre.m[k], b);
            if constexpr (DISP) r = sub_wtg(r, y[k], pre.g[k]);
        }
        if constexpr (PREC == 0) {
            Sym d = blk_sym(ablk(A, M, x, x));
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                d = sym_sub_gram(d, y[k]);
                xs[(4 * k) * nx + x] = y[k].a00;
                xs[(4 * k + 1) * nx + x] = y[k].a01;
                xs[(4 * k + 2) * nx + x] = y[k].a10;
                xs[(4 * k + 3) * nx + x] = y[k].a11;
            }
            xs[(4 * NP) * nx + x] = d.s00;
            xs[(4 * NP + 1) * nx + x] = d.s01;
            xs[(4 * NP + 2) * nx + x] = d.s11;
            if constexpr (DISP) {
                xs[(4 * NP + 3) * nx + x] = r.v0;
                xs[(4 * NP + 4) * nx + x] = r.v1;
            }
            if (x >= ca) {
                bool ok;
                double dd;
                LInv m2 = chol2_inv(d, ok, dd);
                if (!ok) m2 = LInv{nan, nan, nan};  // its leaves' determinants are then NaN and reported
                const int q = x - ca;
                rs[q] = m2.m00;
                rs[nr + q] = m2.m10;
                rs[2 * nr + q] = m2.m11;
                if constexpr (DISP) {
                    const Vec2 g2 = lvec(m2, r);
                    rs[3 * nr + q] = g2.v0;
                    rs[4 * nr + q] = g2.v1;
                }
            }
        } else {
#pragma unroll
            for (int k = 0; k < NE; ++k) {
                split_rows(y[k], xq[(2 * k) * nx + x], xq[(2 * k + 1) * nx + x]);
            }
        }
    }
    __syncthreads();
    // refined: Schur-complement block S_U[x][y] from A's block and U's rows, those
    // of x given by ux
    auto su = [&](int x, int y, auto ux) {
        const float4 *f = reinterpret_cast<const float4 *>(a.Af) + 2 * ((size_t)x * M + y);
        const float4 h = f[0], l = f[1];
        ABlk b{Acc{h.x, l.x}, Acc{h.y, l.y}, Acc{h.z, l.z}, Acc{h.w, l.w}};
#pragma unroll
        for (int k = 0; k < 2 * NE; ++k) {
            const float4 u = ux(k), v = x == y ? u : xq[k * nx + y];
            acc_sub_row(b, DF{u.x, u.y}, DF{u.z, u.w}, DF{v.x, v.y}, DF{v.z, v.w});
        }
        return DFBlk{acc_norm(b.a00), acc_norm(b.a01), acc_norm(b.a10), acc_norm(b.a11)};
    };
    if constexpr (PREC == 1) {
        static_assert(NE == 1, "U is one mode");
        // c3's rows of U (c3 lies above the chunk's modes) and its pivot, in every thread
        float4 u3[2];
        split_rows(lmul(pre.m[0], ablk(A, M, mode(0), c3)), u3[0], u3[1]);
        auto at3 = [&](int k) { return u3[k]; };
        bool ok3;
        const Piv p3 = pivot_of(acc_sym(su(c3, c3, at3)), ok3);
        if (!ok3 && threadIdx.x == 0) flag_status(a.status, ST_NOT_POSDEF);
        for (int x = threadIdx.x; x < nx; x += CHUNK_THREADS) {
            DFBlk z = pivot_rows(acc_of(su(c3, x, at3)), p3);
            z = DFBlk{df_norm(z.a00.h, z.a00.l), df_norm(z.a01.h, z.a01.l), df_norm(z.a10.h, z.a10.l),
                      df_norm(z.a11.h, z.a11.l)};
            const ASym d = acc_sub_gram(acc_sym(su(x, x, [&](int k) { return xq[k * nx + x]; })), z);
            float4 *const e = xq + (2 * NE) * nx + x;
            e[0] = make_float4(z.a00.h, z.a01.h, z.a10.h, z.a11.h);
            e[nx] = make_float4(z.a00.l, z.a01.l, z.a10.l, z.a11.l);
            e[2 * nx] = make_float4(d.s00.s, d.s01.s, d.s11.s, d.s00.t);
            e[3 * nx] = make_float4(d.s01.t, d.s11.t, 0.f, 0.f);
            if (x >= ca) {
                bool ok;
                const Piv p = pivot_of(d, ok);
                if (!ok) flag_status(a.status, ST_NOT_POSDEF);
                const int q = x - ca;
                rq[q] = make_float4(p.i0.h, p.i0.l, p.l.h, p.l.l);
                rq[nr + q] = make_float4(p.i1.h, p.i1.l, 0.f, 0.f);
            }
        }
        __syncthreads();
    }
    uint64_t baseJ[NQ], baseT[NQ], idxQ[NQ];
    child_bases<NP>(P, M, baseJ, baseT, idxQ);
    double p0R[NQ];
    p0R[0] = 0.0;
#pragma unroll
    for (int q = 1; q < NQ; ++q) p0R[q] = a.p0[idxQ[q]];
    for (uint32_t t = t0 + threadIdx.x; t < t1; t += CHUNK_THREADS) {
        int c2, j;
        pair_decode(t, c2, j);
        const int q = c2 - ca;
        double P0, v;
        bool ok;
        if constexpr (PREC == 0) {
            Blk X = ablk(A, M, c2, j);
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const double *z = xs + 4 * k * nx;
                X = blk_sub_cross(X, Blk{z[c2], z[nx + c2], z[2 * nx + c2], z[3 * nx + c2]},
                                  Blk{z[j], z[nx + j], z[2 * nx + j], z[3 * nx + j]});
            }
            const double *d = xs + 4 * NP * nx;
            const Blk w = lmul(LInv{rs[q], rs[nr + q], rs[2 * nr + q]}, X);
            const Sym sch = sym_sub_gram(Sym{d[j], d[nx + j], d[2 * nx + j]}, w);
            const double det2 = det_sym(sch);
            const double rd = rsqrt(det2);
            P0 = a.p0[baseJ[PALL] + c2] * rd;
            if constexpr (DISP)
                P0 *= exp(-quad_inv(sch, rd * rd, sub_wtg(Vec2{d[3 * nx + j], d[4 * nx + j]}, w,
                                                          Vec2{rs[3 * nr + q], rs[4 * nr + q]})));
            ok = det2 > 0.0 && !bad;
            if (!ok) P0 = nan;
            v = combine<NP, MODE>(P0, j, c2, t, baseJ, baseT, p0R, a.p0, a.out);
        } else {
            const float4 *const z = xq + 2 * NE * nx;
            const float4 zh2 = z[c2], zl2 = z[nx + c2], zhj = z[j], zlj = z[nx + j];
            const float4 d0 = z[2 * nx + j], d1 = z[3 * nx + j], p4 = rq[q], p5 = rq[nr + q];
            float r0, eta;
            refined_leaf_factor(acc_of(su(c2, j, [&](int k) { return xq[k * nx + c2]; })),
                                DFBlk{DF{zh2.x, zl2.x}, DF{zh2.y, zl2.y}, DF{zh2.z, zl2.z}, DF{zh2.w, zl2.w}},
                                DFBlk{DF{zhj.x, zlj.x}, DF{zhj.y, zlj.y}, DF{zhj.z, zlj.z}, DF{zhj.w, zlj.w}},
                                ASym{Acc{d0.x, d0.w}, Acc{d0.y, d1.x}, Acc{d0.z, d1.y}},
                                Piv{DF{p4.x, p4.y}, DF{p4.z, p4.w}, DF{p5.x, p5.y}}, r0, eta, ok);
            ok = ok && !bad;
            constexpr bool pairs = MODE == MODE_KAPPA || MODE == MODE_SPINK;
            P0 = !ok ? nan : write_p0 || !pairs ? refined_leaf_p0(a.p0[baseJ[PALL] + c2], r0, eta) : 0.0;
            if constexpr (pairs) {
                float2 kq[NQ], pq[NQ];
                double uq[NQ];
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    kq[q] = q ? a.kyp[baseJ[q] + j] : float2{};
                    pq[q] = a.p0p[baseJ[q] + c2];
                    uq[q] = q < PALL ? a.out[baseT[q] + t] : 0.0;
                }
                v = combine_lead<NP, MODE>(combine_products<NP, MODE>(kq, pq, uq, p0R), r0, eta, a.p0p[j], pq[PALL]);
                if (!ok) v = nan;
            } else {
                v = combine<NP, MODE>(P0, j, c2, t, baseJ, baseT, p0R, a.p0, a.out);
            }
        }
        if (!ok) flag_status(a.status, ST_NOT_POSDEF);
        store_entry<MODE>(a, NP + 2, baseT[PALL] + t, P0, v, write_p0);
    }
}

// Shared-memory bytes of chunks of L pairs below the top mode c3 = top: PX doubles
// per mode up to the chunk's largest c2, PR per row of it. A chunk that starts at
// c2 = 1 touches about sqrt(2 L) rows; one that ends in the upper half has few.
constexpr size_t chunk_smem(int top, uint32_t L, int px, int pr) {
    size_t rows = 2;
    while (rows * (rows - 1) / 2 < L && rows < (size_t)top) ++rows;
    rows += 2;
    const size_t half = (size_t)top / 2, few = half > rows ? L / (half - rows) + 3 : rows;
    const size_t hi = px * (size_t)top + pr * (few < rows ? few : rows), lo = px * (half + 1) + pr * rows;
    return sizeof(double) * (hi > lo ? hi : lo);
}

// Queues the chunked kernel over the prefixes with top element in [c_lo, c_hi).
template <int NP, int MODE, int PREC, bool DISP>
static cudaError_t launch_chunk(const FwdArgs &a, bool write_p0, int c_lo, int c_hi, uint32_t L, size_t smem,
                                cudaStream_t st) {
    auto fn = chunk_kernel<NP, MODE, PREC, DISP>;
    // the static part takes a little of the 48 KB that need no opt-in. The limit belongs
    // to the kernel, not to this call: every call sets the same one, so that no host
    // thread lowers it between another's two calls
    if (smem > 40 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kChunkSmem);
        if (e != cudaSuccess) return e;
    }
    const int hi = c_hi - 1, lo = c_lo > NP + 1 ? c_lo : NP + 1;  // largest and smallest top element
    const int c3 = hi - (NP - 1);
    const uint64_t prefixes = NP == 1 ? (uint64_t)(hi - lo + 1) : binom2(hi + 1) - binom2(lo);
    return launch_next(!a.ev, fn, dim3((unsigned)prefixes, (unsigned)((binom2(c3) + L - 1) / L)), CHUNK_THREADS, smem, st, a,
                       write_p0, hi, L);
}

}  // namespace gbs
