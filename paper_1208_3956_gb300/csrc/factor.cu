// Algorithm 1 (preparation) on the GPU: factor every strip operator S^(j) A^(j)
// as a block-tridiagonal matrix along y, partitioned into P chunks separated by
// single separator rows (one level of nested dissection along y):
//
//   chunk p covers rows r0[p] .. r1[p]-1, separator p is row r1[p] (p < P-1).
//
// Every block-tridiagonal system (each chunk, and the separator system) is
// factored "twisted": eliminated from both ends toward a middle twist row, so
// that a solve runs its two halves concurrently and needs about m+1 dependent
// steps instead of 2m-1.  For a chunk with twist row t = r0 + (m-1)/2:
//   rows r0..t-1:   S_k = D_k - C_k S_{k-1}^{-1} C_k          (top down)
//   rows r1-1..t+1: S_k = D_k - C_{k+1} S_{k+1}^{-1} C_{k+1}  (bottom up)
//   row t:          S_t = D_t - C_t S_{t-1}^{-1} C_t - C_{t+1} S_{t+1}^{-1} C_{t+1}
// and Sinv_k = S_k^{-1} is stored for every row.  The chunk solve is
//   z_k = Sinv_k (b_k - C_k z_{k-1})        k < t
//   z_k = Sinv_k (b_k - C_{k+1} z_{k+1})    k > t
//   y_t = Sinv_t (b_t - C_t z_{t-1} - C_{t+1} z_{t+1})
//   y_k = z_k - Sinv_k C_{k+1} y_{k+1}      k < t (outward)
//   y_k = z_k - Sinv_k C_k y_{k-1}          k > t (outward).
// Spikes (k_factor_chunk): GB = A_p^{-1} E_last C_{r1} (response to the
// separator below) and GT = A_p^{-1} E_first C_{r0} (separator above), so that
// the chunk solution is x_p = y_p - GT x_sep(p-1) - GB x_sep(p).
//
// Separator system (k_factor_sep_*), q = 0..Q-1, Q = P-1, solved in groups (a second level of
// nested dissection):
//   T_q = D_s - C_s GB_q(last) - C_{s+1} GT_{q+1}(first),   s = r1[q]
//   L_q = -C_s GT_q(last),  U_q = -C_{s+1} GB_{q+1}(first)
// twisted at tq = (Q-1)/2.  Stored per separator: Rinv_q, an "outer" coupling
// E_q (toward the ends) and an "inner" coupling F_q (toward the twist):
//   q < tq: R_q = T_q - L_q F_{q-1},  E_q = Rinv_q L_q,  F_q = Rinv_q U_q
//   q > tq: R_q = T_q - U_q F_{q+1},  E_q = Rinv_q U_q,  F_q = Rinv_q L_q
//   q = tq: R_q = T_q - L_q F_{q-1} - U_q F_{q+1},  E_q = Rinv_q L_q,  F_q = Rinv_q U_q
// and the separator solve is z_q = a_q - E_q z_{outer neighbour},
// x_tq = a_tq - E_tq z_{tq-1} - F_tq z_{tq+1}, x_q = z_q - F_q x_{inner neighbour},
// with a_q = Rinv_q bhat_q.
#include "common.cuh"
#include "strip_ops.cuh"
#include "internal.h"

namespace helm {

// Blocks between shared memory (column-major W x W) and the factor pools (row-major, a warp to a
// row so that global accesses are contiguous): the sweep layout (leading dimension ld, zero
// pad) and the spikes' (row length spld(W), so that the correction step reads rows).
template <typename C>
__device__ void load_block(C* dst, const C* src, int W, int ld) {
    for (int r = threadIdx.x >> 5; r < W; r += blockDim.x >> 5)
        for (int a = threadIdx.x & 31; a < W; a += 32) dst[a * W + r] = src[(int64_t)r * ld + a];
}
template <typename C>
__device__ void store_block(C* dst, const C* src, int W, int ld) {
    for (int r = threadIdx.x >> 5; r < W; r += blockDim.x >> 5)
        for (int a = threadIdx.x & 31; a < ld; a += 32) dst[(int64_t)r * ld + a] = a < W ? src[a * W + r] : CT<C>::zero();
}
template <typename C>
__device__ void load_rows(C* dst, const C* src, int W) {
    load_block(dst, src, W, spld(W));
}
template <typename C>
__device__ void store_rows(C* dst, const C* src, int W) {
    const int ld = spld(W);
    for (int r = threadIdx.x >> 5; r < W; r += blockDim.x >> 5)
        for (int a = threadIdx.x & 31; a < W; a += 32) dst[(int64_t)r * ld + a] = src[a * W + r];
}
template <typename C>
__device__ void fill_zero(C* dst, int count) {
    for (int e = threadIdx.x; e < count; e += blockDim.x) dst[e] = CT<C>::zero();
}
template <typename C>
__device__ void load_coupling(C* dv, const Geom& g, const double2* sx, int W, int k) {
    for (int c = threadIdx.x; c < W; c += blockDim.x) dv[c] = CT<C>::from(strip_coupling(g, sx[c], k));
}
// s_x of the strip's columns into shared memory (one complex division per column and CTA)
__device__ inline void load_sx(double2* sx, const Geom& g, const StripDev& st) {
    for (int c = threadIdx.x; c < st.W; c += blockDim.x) sx[c] = strip_sx(g, st, c);
    __syncthreads();
}
// M -= diag(d) X diag(d)
template <typename C, int NI>
__device__ void sub_congruence(C* M, const C* X, const C* d, int W) {
    const int ti = threadIdx.x & 15, tj = threadIdx.x >> 4;
#pragma unroll
    for (int j = 0; j < NI; ++j)
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int r = ti + 16 * i, c = tj + 16 * j;
            if (r < W && c < W) M[c * W + r] = csub(M[c * W + r], cmul(cmul(d[r], X[c * W + r]), d[c]));
        }
}

// Spike solve A_p Y = E_rs Rhs for the chunk [r0, r1) with twist t (rs = r0 or
// r1-1, Rhs = diag(C_{r0}) or diag(C_{r1}) given as the vector dr).  Y goes to
// OUT (global, row-major).  Z values of the elimination are parked in OUT.
// smem: M (Sinv), X (current), Y (scratch), dv (coupling vector).
template <typename C, int NI>
__device__ void spike_solve(const Geom& g, const StripDev& st, const C* SinvS, C* OUT, int r0, int r1, int t,
                            int rs, const C* dr, C*& M, C*& X, C*& Y, C* dv, const double2* sx) {
    using R = typename CT<C>::R;
    const int W = st.W;
    const int64_t bs = st.bs;
    auto swap = [&]() { C* h = X; X = Y; Y = h; };   // the result of a product is the next one's input
    // X <- Sinv_rs diag(dr): the eliminated block at row rs
    load_block(M, SinvS + (int64_t)rs * bs, W, st.ld);
    __syncthreads();
    for (int c = threadIdx.x >> 4; c < W; c += 16)
        for (int r = threadIdx.x & 15; r < W; r += 16) X[c * W + r] = cmul(M[c * W + r], dr[c]);
    __syncthreads();
    if (rs != t) {
        store_rows(OUT + (int64_t)rs * bs, X, W);
        const int dir = rs < t ? 1 : -1;   // elimination runs toward the twist
        for (int k = rs + dir; k != t; k += dir) {
            load_block(M, SinvS + (int64_t)k * bs, W, st.ld);
            load_coupling(dv, g, sx, W, dir > 0 ? k : k + 1);   // coupling to the previous row
            __syncthreads();
            block_gemm_dscale<C, NI>(Y, M, dv, X, W, false, (R)-1);   // z_k = -Sinv_k C z_prev
            store_rows(OUT + (int64_t)k * bs, Y, W);
            swap();
        }
        // twist row: y_t = Sinv_t (-C z_{t-dir})
        load_block(M, SinvS + (int64_t)t * bs, W, st.ld);
        load_coupling(dv, g, sx, W, dir > 0 ? t : t + 1);
        __syncthreads();
        block_gemm_dscale<C, NI>(Y, M, dv, X, W, false, (R)-1);
        swap();
    }
    store_rows(OUT + (int64_t)t * bs, X, W);   // X = y_t
    __syncthreads();
    // outward back substitution on both sides; Y_k = z_k - Sinv_k C y_inner
    for (int side = 0; side < 2; ++side) {
        const int dir = side == 0 ? -1 : 1;      // -1: rows t-1..r0, +1: rows t+1..r1-1
        if (side == 1) load_rows(X, OUT + (int64_t)t * bs, W);   // y_t
        for (int k = t + dir; k >= r0 && k < r1; k += dir) {
            load_block(M, SinvS + (int64_t)k * bs, W, st.ld);
            load_coupling(dv, g, sx, W, dir < 0 ? k + 1 : k);   // coupling to the inner row
            const bool has_z = (rs < t) ? (dir < 0 && k >= rs) : (rs > t && dir > 0 && k <= rs);
            if (has_z) load_rows(Y, OUT + (int64_t)k * bs, W);
            __syncthreads();
            block_gemm_dscale<C, NI>(Y, M, dv, X, W, has_z, (R)-1);
            store_rows(OUT + (int64_t)k * bs, Y, W);
            swap();
        }
        __syncthreads();
    }
}

// MINB: CTAs to fit on an SM (0: as the registers come, two); see launch_factor_ni.
template <typename C, int NI, int MINB>
__global__ void __launch_bounds__(kBlockThreads, MINB) k_factor_chunk(Geom g, C* __restrict__ Sinv,
                                                                      C* __restrict__ GT, C* __restrict__ GB,
                                                                      int* __restrict__ status) {
    const StripDev st = g.strips[blockIdx.y];
    const int p = blockIdx.x;
    const int W = st.W;
    const int r0 = g.r0[p], r1 = g.r1[p];
    const int t = r0 + (r1 - r0 - 1) / 2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ InvScratch<C> sc;
    __shared__ double2 sx[64];
    __shared__ C dv[64], dr[64];
    C* M = reinterpret_cast<C*>(smem_raw);
    C* X = M + W * W;
    C* Y = X + W * W;
    C* SinvS = Sinv + st.fac;
    const int64_t bs = st.bs;
    load_sx(sx, g, st);

    // M -> its inverse, stored as row k's block; X the same inverse (the next row's neighbour)
    auto finish_row = [&](int k) -> bool {
        if (!block_inverse<C, NI>(M, W, sc)) {
            if (threadIdx.x == 0) atomicExch(status, 1);
            return false;
        }
        store_block(SinvS + (int64_t)k * bs, M, W, st.ld);
        C* h = X; X = M; M = h;
        return true;
    };
    // ---- top-down rows r0 .. t-1
    for (int k = r0; k < t; ++k) {
        build_diag_block(g, st, k, M, sx);
        if (k > r0) {
            load_coupling(dv, g, sx, W, k);
            __syncthreads();
            sub_congruence<C, NI>(M, X, dv, W);
            __syncthreads();
        }
        if (!finish_row(k)) return;
    }
    // ---- bottom-up rows r1-1 .. t+1
    for (int k = r1 - 1; k > t; --k) {
        build_diag_block(g, st, k, M, sx);
        if (k < r1 - 1) {
            load_coupling(dv, g, sx, W, k + 1);
            __syncthreads();
            sub_congruence<C, NI>(M, X, dv, W);
            __syncthreads();
        }
        if (!finish_row(k)) return;
    }
    // ---- twist row
    build_diag_block(g, st, t, M, sx);
    if (t > r0) {
        load_block(X, SinvS + (int64_t)(t - 1) * bs, W, st.ld);
        load_coupling(dv, g, sx, W, t);
        __syncthreads();
        sub_congruence<C, NI>(M, X, dv, W);
        __syncthreads();
    }
    if (t < r1 - 1) {
        load_block(X, SinvS + (int64_t)(t + 1) * bs, W, st.ld);
        load_coupling(dv, g, sx, W, t + 1);
        __syncthreads();
        sub_congruence<C, NI>(M, X, dv, W);
        __syncthreads();
    }
    if (!finish_row(t)) return;
    __syncthreads();

    // ---- spikes
    if (p < g.P - 1) {   // bottom spike, driven by separator row r1
        load_coupling(dr, g, sx, W, r1);
        __syncthreads();
        spike_solve<C, NI>(g, st, SinvS, GB + st.fac, r0, r1, t, r1 - 1, dr, M, X, Y, dv, sx);
        __syncthreads();
    }
    if (p > 0) {         // top spike, driven by separator row r0-1
        load_coupling(dr, g, sx, W, r0);
        __syncthreads();
        spike_solve<C, NI>(g, st, SinvS, GT + st.fac, r0, r1, t, r0, dr, M, X, Y, dv, sx);
    }
}

template <typename C>
struct SepPools {
    C* Rinv;   // per separator slot, sweep layout
    C* E;
    C* F;
    C* GT2;    // group spikes, W rows of spld(W)
    C* GB2;
    C* P2L;    // level-2 right-hand-side products Rinv2 L, Rinv2 U (sweep layout)
    C* P2U;
    C* Q2L;    // level-2 contributions of a group separator's right-hand side (sweep layout)
    C* Q2U;
};

// a * b with its roundings spelled out (the second product of each component rounded, the first
// fused), and t - a * b rounded after it: the separator blocks cancel, and how the compiler
// would contract the plain expression depends on the code around it.
__device__ __forceinline__ float2 cmul_fixed(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -__fmul_rn(a.y, b.y)), fmaf(a.x, b.y, __fmul_rn(a.y, b.x)));
}
__device__ __forceinline__ double2 cmul_fixed(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -__dmul_rn(a.y, b.y)), fma(a.x, b.y, __dmul_rn(a.y, b.x)));
}
__device__ __forceinline__ float2 csub_fixed(float2 t, float2 v) {
    return make_float2(__fadd_rn(t.x, -v.x), __fadd_rn(t.y, -v.y));
}
__device__ __forceinline__ double2 csub_fixed(double2 t, double2 v) {
    return make_double2(__dadd_rn(t.x, -v.x), __dadd_rn(t.y, -v.y));
}

// What the separator kernels share: one strip's pools and tables, the shared-memory blocks and
// the level-1 separator blocks.
template <typename C, int NI>
struct SepStrip {
    using R = typename CT<C>::R;
    const Geom& g;
    const StripDev& st;
    const C *GTs, *GBs;
    SepPools<C> P;
    const double2* sx;
    C *M, *X, *Y, *Z;      // Z: level-2 scratch (null in a single group)
    InvScratch<C>& sc;
    int* status;
    int W;
    int64_t bs;
    __device__ SepStrip(const Geom& g_, const StripDev& st_, const C* GT, const C* GB, const SepPools<C>& pl, C* smem,
                        bool z, double2* sx_, InvScratch<C>& sc_, int* status_)
        : g(g_), st(st_), GTs(GT + st_.fac), GBs(GB + st_.fac), P(pl), sx(sx_), sc(sc_), status(status_), W(st_.W),
          bs(st_.bs) {
        M = smem;
        X = M + W * W;
        Y = X + W * W;
        Z = z ? Y + W * W : nullptr;
        P.Rinv += st.red; P.E += st.red; P.F += st.red; P.GT2 += st.red; P.GB2 += st.red; P.P2L += st.red;
        P.P2U += st.red;
        if (P.Q2L) { P.Q2L += st.red; P.Q2U += st.red; }
        load_sx(sx_, g, st);
    }
    __device__ void gemm(C* Out, const C* A, const C* B, bool acc, R sgn) {
        block_gemm_dscale<C, NI>(Out, A, (const C*)nullptr, B, W, acc, sgn);
    }
    // D <- -diag(C_k) times a spike block (row-major)
    __device__ void coupled_spike(C* D, const C* spike, int k) {
        C* ck = sc.col[0];   // scratch outside the inverse
        __syncthreads();
        load_coupling(ck, g, sx, W, k);
        load_rows(D, spike, W);
        __syncthreads();
        for_entries([&](int r, int e) { D[e] = cneg(cmul_fixed(ck[r], D[e])); });
        __syncthreads();
    }
    // f(row, index) for this thread's entries of a column-major block
    template <typename F>
    __device__ void for_entries(F f) {
        const int ti = threadIdx.x & 15, tj = threadIdx.x >> 4;
#pragma unroll
        for (int j = 0; j < NI; ++j)
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                const int r = ti + 16 * i, c = tj + 16 * j;
                if (r < W && c < W) f(r, c * W + r);
            }
    }
    // level-1 blocks of separator q (row s = r1[q])
    __device__ void build_T1(int q) {   // M <- T_q = D_s - C_s GB_q(last) - C_{s+1} GT_{q+1}(first)
        const int s = g.r1[q];
        C *c0 = sc.col[0], *c1 = sc.col[1];
        __syncthreads();
        load_coupling(c0, g, sx, W, s);
        load_coupling(c1, g, sx, W, s + 1);
        load_rows(X, GBs + (int64_t)(s - 1) * bs, W);
        load_rows(Y, GTs + (int64_t)g.r0[q + 1] * bs, W);
        build_diag_block(g, st, s, M, sx);
        for_entries([&](int r, int e) { M[e] = csub_fixed(csub_fixed(M[e], cmul_fixed(c0[r], X[e])), cmul_fixed(c1[r], Y[e])); });
        __syncthreads();
    }
    __device__ void build_L1(int q, C* D) {   // L_q = -C_s GT_q(last)
        const int s = g.r1[q];
        coupled_spike(D, GTs + (int64_t)(s - 1) * bs, s);
    }
    __device__ void build_U1(int q, C* D) {   // U_q = -C_{s+1} GB_{q+1}(first)
        coupled_spike(D, GBs + (int64_t)g.r0[q + 1] * bs, g.r1[q] + 1);
    }
    __device__ void load(C* dst, const C* pool, int q) { load_block(dst, pool + (int64_t)q * bs, W, st.ld); }
    __device__ void store(C* pool, int q, const C* src) { store_block(pool + (int64_t)q * bs, src, W, st.ld); }

    // Twisted LU of a block-tridiagonal system with dense couplings, elements i = 0..n-1 stored at
    // separator slots sl(i): bT(i) builds the diagonal block into M, bL(i, D) / bU(i, D) build
    // the couplings to i-1 / i+1 into D (they may use Y and Z as scratch but not M).  Stores
    // Rinv, the outer coupling E and the inner coupling F of every element (file header).
    template <typename SL, typename BT_, typename BL, typename BU>
    __device__ bool twisted_lu(int n, SL sl, BT_ bT, BL bL, BU bU) {
        auto sub_nb = [&](int inb) {   // M -= X F_nb
            load(Y, P.F, sl(inb));
            __syncthreads();
            gemm(M, X, Y, true, (R)-1);
        };
        auto inv_store = [&](int i) -> bool {
            if (!block_inverse<C, NI>(M, W, sc)) {
                if (threadIdx.x == 0) atomicExch(status, 2);
                return false;
            }
            store(P.Rinv, sl(i), M);
            __syncthreads();
            return true;
        };
        auto prod_store = [&](C* pool, int i) {   // pool_i = M X (M = Rinv)
            gemm(Y, M, X, false, (R)1);
            store(pool, sl(i), Y);
            __syncthreads();
        };
        auto zero_store = [&](C* pool, int i) {
            fill_zero(pool + (int64_t)sl(i) * bs, W * st.ld);
            __syncthreads();
        };
        const int tq = (n - 1) / 2;
        for (int u = 0; u < n; ++u) {   // top down 0 .. tq-1, bottom up n-1 .. tq+1, the twist
            const int i = u < tq ? u : u < n - 1 ? n - 1 - (u - tq) : tq;
            const bool tw = u == n - 1, top = u < tq;
            // neighbours already eliminated: above (top half, twist) and below (bottom half, twist)
            const bool hl = (top || tw) && i >= 1, hu = (!top || tw) && i <= n - 2;
            bT(i);
            if (hl) { bL(i, X); sub_nb(i - 1); }
            if (hu) { bU(i, X); sub_nb(i + 1); }
            if (!inv_store(i)) return false;
            // E: the outer coupling; F: the inner one (the twist: E above, F below)
            if (top || tw) {
                if (i >= 1) { bL(i, X); prod_store(P.E, i); } else zero_store(P.E, i);
                if (i <= n - 2) { bU(i, X); prod_store(P.F, i); } else zero_store(P.F, i);
            } else {
                if (i <= n - 2) { bU(i, X); prod_store(P.E, i); } else zero_store(P.E, i);
                bL(i, X);
                prod_store(P.F, i);
            }
        }
        return true;
    }
};
#define HELM_SEP_STRIP(zbuf)                                                                               \
    extern __shared__ __align__(16) unsigned char smem_raw[];                                              \
    __shared__ InvScratch<C> sc;                                                                           \
    __shared__ double2 sx[64];                                                                             \
    using R = typename CT<C>::R;                                                                           \
    const StripDev st = g.strips[blockIdx.y];                                                              \
    SepStrip<C, NI> S(g, st, GT, GB, pl, reinterpret_cast<C*>(smem_raw), zbuf, sx, sc, status);            \
    const SepPools<C>& P = S.P;                                                                            \
    const int W = S.W;                                                                                     \
    const int64_t bs = S.bs;                                                                               \
    C *M = S.M, *X = S.X, *Y = S.Y, *Z = S.Z;

// The separator system in three launches, each as wide as its dependencies allow.  One CTA per
// strip ran all of it; with that, an uncoalesced read per spike entry, an FP64 division per
// coupling and one product entry per thread, it took 33.5 ms of a 65 ms factorisation on the
// 1023 x 1023 grid (64 strips) and 21 of 30 ms on 511 x 511 (32 strips); now 4.8 of 27.5 and
// 2.2 of 9.0 ms, bound by the chain of block inversions of the longest group and of level 2.
// k_factor_sep_group (group x strip): twisted LU of the group's separators, then the group
// spikes, the response of the group to the level-2 separator above (right-hand side L_{q0} at
// its first element) and below (U_{q1-1} at its last).
template <typename C, int NI, int MINB>
__global__ void __launch_bounds__(kBlockThreads, MINB) k_factor_sep_group(Geom g, const C* __restrict__ GT,
                                                                          const C* __restrict__ GB, SepPools<C> pl,
                                                                          int* __restrict__ status) {
    HELM_SEP_STRIP(g.G > 1)
    const int G = g.G, gi = blockIdx.x;
    const int q0 = g.gq0[gi], q1 = g.gq1[gi], n = q1 - q0, tq = (n - 1) / 2;
    if (!S.twisted_lu(n, [&](int i) { return q0 + i; }, [&](int i) { S.build_T1(q0 + i); },
                      [&](int i, C* D) { S.build_L1(q0 + i, D); }, [&](int i, C* D) { S.build_U1(q0 + i, D); }))
        return;
    for (int side = 0; side < 2; ++side) {
        const bool top = side == 0;
        if (top && gi == 0) continue;
        if (!top && gi == G - 1) continue;
        C* OUT = top ? P.GT2 : P.GB2;
        auto out = [&](int i) { return OUT + (int64_t)(q0 + i) * bs; };
        const int rs = top ? 0 : n - 1;
        // X <- Rinv_rs B, B = L_{q0} (top) or U_{q1-1} (bottom)
        if (top) S.build_L1(q0, Z); else S.build_U1(q1 - 1, Z);
        S.load(M, P.Rinv, q0 + rs);
        __syncthreads();
        S.gemm(X, M, Z, false, (R)1);
        auto swap = [&]() { C* h = X; X = Y; Y = h; };
        if (rs != tq) {
            store_rows(out(rs), X, W);
            const int dir = rs < tq ? 1 : -1;
            for (int i = rs + dir; i != tq; i += dir) {   // z_i = -E_i z_prev
                S.load(M, P.E, q0 + i);
                __syncthreads();
                S.gemm(Y, M, X, false, (R)-1);
                store_rows(out(i), Y, W);
                swap();
            }
            // twist: x_t = -E_t z_{t-1} (from above) or -F_t z_{t+1} (from below)
            S.load(M, dir > 0 ? P.E : P.F, q0 + tq);
            __syncthreads();
            S.gemm(Y, M, X, false, (R)-1);
            swap();
        }
        store_rows(out(tq), X, W);
        __syncthreads();
        for (int sd = 0; sd < 2; ++sd) {   // outward: x_i = z_i - F_i x_inner
            const int dir = sd == 0 ? -1 : 1;
            if (sd == 1) load_rows(X, out(tq), W);
            for (int i = tq + dir; i >= 0 && i < n; i += dir) {
                S.load(M, P.F, q0 + i);
                const bool has_z = top ? (dir < 0 && i >= rs) : (dir > 0 && i <= rs);
                if (has_z) load_rows(Y, out(i), W);
                __syncthreads();
                S.gemm(Y, M, X, has_z, (R)-1);
                store_rows(out(i), Y, W);
                swap();
            }
            __syncthreads();
        }
    }
}

// k_factor_sep_l2 (strip): the level-2 system over r = 0..G-2 (separator sigma_r = gq1[r]) and its
// right-hand-side products P2L_r = Rinv2_r L_s, P2U_r = Rinv2_r U_s.
template <typename C, int NI>
__global__ void __launch_bounds__(kBlockThreads) k_factor_sep_l2(Geom g, const C* __restrict__ GT,
                                                                 const C* __restrict__ GB, SepPools<C> pl,
                                                                 int* __restrict__ status) {
    HELM_SEP_STRIP(true)
    const int G = g.G;
    auto sig = [&](int r) { return g.gq1[r]; };
    auto spike = [&](C* dst, const C* pool, int q) { load_rows(dst, pool + (int64_t)q * bs, W); };
    auto bT2 = [&](int r) {   // T_s - L_s GB2_r(last) - U_s GT2_{r+1}(first)
        const int q = sig(r);
        S.build_T1(q);
        S.build_L1(q, Z);
        spike(Y, P.GB2, q - 1);
        __syncthreads();
        S.gemm(M, Z, Y, true, (R)-1);
        S.build_U1(q, Z);
        spike(Y, P.GT2, g.gq0[r + 1]);
        __syncthreads();
        S.gemm(M, Z, Y, true, (R)-1);
    };
    auto bL2 = [&](int r, C* D) {   // -L_s GT2_r(last)
        const int q = sig(r);
        S.build_L1(q, Z);
        spike(Y, P.GT2, q - 1);
        __syncthreads();
        S.gemm(D, Z, Y, false, (R)-1);
    };
    auto bU2 = [&](int r, C* D) {   // -U_s GB2_{r+1}(first)
        const int q = sig(r);
        S.build_U1(q, Z);
        spike(Y, P.GB2, g.gq0[r + 1]);
        __syncthreads();
        S.gemm(D, Z, Y, false, (R)-1);
    };
    if (!S.twisted_lu(G - 1, sig, bT2, bL2, bU2)) return;
    for (int r = 0; r < G - 1; ++r) {
        const int q = sig(r);
        S.load(M, P.Rinv, q);
        S.build_L1(q, X);
        S.gemm(Y, M, X, false, (R)1);
        S.store(P.P2L, q, Y);
        S.build_U1(q, X);
        S.gemm(Y, M, X, false, (R)1);
        S.store(P.P2U, q, Y);
        __syncthreads();
    }
}

// k_factor_sep_q (2 x group, strip): level-2 contributions of the group separators.  A group's part
// of a level-2 right-hand side is -P2L y(last) (to the level-2 separator below it) or
// -P2U y(first) (above), and the group solution's end values are linear in the group's
// right-hand sides a_i = Rinv_i bhat_i: y(last) = sum_i K_i a_i, y(first) = sum_i K'_i a_i.  The
// K blocks follow from the twisted solve's recurrences run backwards (the derivative of its
// last or first output with respect to every intermediate):
//   y(last):  G_{n-1} = I, G_{j-1} = -G_j F_j (j > tq); K_tq = G_tq;
//             K_{tq-1} = -G_tq E_tq, K_{j-1} = -K_j E_j (j < tq);
//             K_{tq+1} = G_{tq+1} - G_tq F_tq, K_j = G_j - K_{j-1} E_{j-1} (j > tq + 1)
//   y(first): G'_0 = I, G'_{j+1} = -G'_j F_j (j < tq); K'_tq = G'_tq;
//             K'_{tq+1} = -G'_tq F_tq, K'_{j+1} = -K'_j E_j (j > tq);
//             K'_{tq-1} = G'_{tq-1} - G'_tq E_tq, K'_{j-1} = G'_{j-1} - K'_j E_j (j < tq - 1)
// Stored per separator: Q2L_i = -P2L K_i, Q2U_i = -P2U K'_i, so that every chunk adds its
// share of the level-2 right-hand sides from its own separator parts.
template <typename C, int NI>
__global__ void __launch_bounds__(kBlockThreads) k_factor_sep_q(Geom g, const C* __restrict__ GT,
                                                                const C* __restrict__ GB, SepPools<C> pl,
                                                                int* __restrict__ status) {
    const int gi = blockIdx.x >> 1;
    const bool last = (blockIdx.x & 1) == 0;   // y(last): level-2 separator below; y(first): above
    if (last ? gi == g.G - 1 : gi == 0) return;
    HELM_SEP_STRIP(true)
    const int q0 = g.gq0[gi], q1 = g.gq1[gi], n = q1 - q0, tq = (n - 1) / 2;
    const C one = CT<C>::from(make_double2(1.0, 0.0));
    auto ident = [&](C* D) {
        fill_zero(D, W * W);
        __syncthreads();
        for (int e = threadIdx.x; e < W; e += blockDim.x) D[e * W + e] = one;
        __syncthreads();
    };
    C* OUT = last ? P.Q2L : P.Q2U;
    auto slot = [&](int i) { return OUT + (int64_t)(q0 + i) * bs; };
    auto put = [&](int i, const C* src) {
        store_rows(slot(i), src, W);
        __syncthreads();
    };
    auto get = [&](C* dst, int i) { load_rows(dst, slot(i), W); };
    auto blk = [&](C* dst, const C* pool, int i) { S.load(dst, pool, q0 + i); };
    if (last) {
        ident(X);
        put(n - 1, X);
        for (int j = n - 1; j > tq; --j) {   // G_{j-1} = -G_j F_j
            blk(M, P.F, j);
            __syncthreads();
            S.gemm(Y, X, M, false, (R)-1);
            block_copy(X, Y, W * W);
            put(j - 1, X);
        }
        block_copy(Z, X, W * W);             // G_tq = K_tq
        for (int j = tq; j >= 1; --j) {      // K_{j-1} = -K_j E_j (K_tq = G_tq)
            blk(M, P.E, j);
            __syncthreads();
            S.gemm(Y, Z, M, false, (R)-1);
            block_copy(Z, Y, W * W);
            put(j - 1, Z);
        }
        if (n - 1 > tq) {                    // K_{tq+1} = G_{tq+1} - G_tq F_tq
            get(Z, tq);
            blk(M, P.F, tq);
            get(Y, tq + 1);
            __syncthreads();
            S.gemm(Y, Z, M, true, (R)-1);
            put(tq + 1, Y);
            block_copy(Z, Y, W * W);
            for (int j = tq + 2; j < n; ++j) {   // K_j = G_j - K_{j-1} E_{j-1}
                blk(M, P.E, j - 1);
                get(Y, j);
                __syncthreads();
                S.gemm(Y, Z, M, true, (R)-1);
                put(j, Y);
                block_copy(Z, Y, W * W);
            }
        }
    } else {
        ident(X);
        put(0, X);
        for (int j = 0; j < tq; ++j) {       // G'_{j+1} = -G'_j F_j
            blk(M, P.F, j);
            __syncthreads();
            S.gemm(Y, X, M, false, (R)-1);
            block_copy(X, Y, W * W);
            put(j + 1, X);
        }
        if (n - 1 > tq) {                    // K'_{tq+1} = -G'_tq F_tq, K'_{j+1} = -K'_j E_j
            blk(M, P.F, tq);
            __syncthreads();
            S.gemm(Z, X, M, false, (R)-1);
            put(tq + 1, Z);
            for (int j = tq + 1; j + 1 < n; ++j) {
                blk(M, P.E, j);
                __syncthreads();
                S.gemm(Y, Z, M, false, (R)-1);
                block_copy(Z, Y, W * W);
                put(j + 1, Z);
            }
        }
        if (tq >= 1) {                       // K'_{tq-1} = G'_{tq-1} - G'_tq E_tq
            block_copy(Z, X, W * W);
            blk(M, P.E, tq);
            get(Y, tq - 1);
            __syncthreads();
            S.gemm(Y, Z, M, true, (R)-1);
            put(tq - 1, Y);
            block_copy(Z, Y, W * W);
            for (int j = tq - 1; j >= 1; --j) {   // K'_{j-1} = G'_{j-1} - K'_j E_j
                blk(M, P.E, j);
                get(Y, j - 1);
                __syncthreads();
                S.gemm(Y, Z, M, true, (R)-1);
                put(j - 1, Y);
                block_copy(Z, Y, W * W);
            }
        }
    }
    // Q = -P2 K with P2L of the level-2 separator below, P2U of the one above
    S.load(M, last ? P.P2L : P.P2U, last ? q1 : q0 - 1);
    for (int i = 0; i < n; ++i) {
        get(X, i);
        __syncthreads();
        S.gemm(Y, M, X, false, (R)-1);
        store_block(slot(i), Y, W, st.ld);
        __syncthreads();
    }
}
#undef HELM_SEP_STRIP

// Transfer composites (with separator groups): for every chunk row k of chunk p and
// transfer column c (forward to0, to1, backward to0, to1; StripDev::xc) the row vectors
//   XF[k][col][0] = GT_p(k)[c,:] GT2_{p-1},   XF[k][col][1] = GT_p(k)[c,:] GB2_{p-1},
//   XF[k][col][2] = GB_p(k)[c,:] GT2_p,       XF[k][col][3] = GB_p(k)[c,:] GB2_p
// (zero where the level-2 spike does not exist).  With them the transfer of row k
// follows from the chain solution, the group solutions of the chunk's two separators
// and the level-2 values around their groups, before those separators are final:
//   x_k[c] = y_k[c] - GT[c,:] y2_{p-1} - GB[c,:] y2_p + XF[0] x2a + XF[1] x2b + XF[2] x2a' + XF[3] x2b'.
// One CTA per (chunk, strip); two level-2 blocks staged at a time.
template <typename C>
__global__ void k_factor_xfer(Geom g, const C* __restrict__ GT, const C* __restrict__ GB,
                              const C* __restrict__ GT2, const C* __restrict__ GB2, C* __restrict__ XF) {
    const StripDev st = g.strips[blockIdx.y];
    const int p = blockIdx.x;
    const int W = st.W, SL = spld(W);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* blk = reinterpret_cast<C*>(smem_raw);   // [2][W][SL]
    const int4 m0 = g.cmeta[2 * p];
    const int r0 = m0.x, r1 = m0.y, gA = m0.z, gB = m0.w;
    const int G = g.G;
    for (int half = 0; half < 2; ++half) {   // 0: separator above (p-1), 1: separator below (p)
        const int gi = half == 0 ? gA : gB;
        const bool has[2] = {gi > 0, gi >= 0 && gi < G - 1};   // GT2, GB2 of that separator exist
        const int q = half == 0 ? p - 1 : p;
        __syncthreads();
        for (int e = threadIdx.x; e < 2 * W * SL; e += blockDim.x) {
            const int k = e / (W * SL), o = e % (W * SL);
            blk[e] = has[k] ? (k == 0 ? GT2 : GB2)[st.red + (int64_t)q * st.bs + o] : CT<C>::zero();
        }
        __syncthreads();
        for (int k = r0; k < r1; ++k)
            for (int col = 0; col < 4; ++col) {
                const int c = st.xc[col];
                const C* v = (half == 0 ? GT : GB) + st.fac + (int64_t)k * st.bs + (int64_t)c * SL;
                for (int o = threadIdx.x; o < 2 * SL; o += blockDim.x) {
                    const int k2 = o / SL, a = o % SL;
                    C acc = CT<C>::zero();
                    if (has[k2] && a < W) {
                        const C* M = blk + k2 * W * SL + a;
                        for (int cc = 0; cc < W; ++cc) acc = cfma(v[cc], M[cc * SL], acc);
                    }
                    XF[st.xf + (((int64_t)k * 4 + col) * 4 + half * 2 + k2) * SL + a] = acc;
                }
            }
    }
}

size_t factor_smem_bytes(int Wmax, size_t esize, int nbuf) {
    const size_t fixed = 8 * 64 * esize + 64 * sizeof(int) + 64 * sizeof(double2);   // InvScratch, dv, dr; sx
    return (size_t)nbuf * Wmax * Wmax * esize + fixed;
}

template <typename C, int NI>
static cudaError_t launch_factor_ni(const Geom& g, int Wmax, void* const* pool, int* status, cudaStream_t s,
                                    KernelTimer* tm) {
    auto attr = [](const void* fn, size_t bytes) {
        return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    const size_t blk = (size_t)Wmax * Wmax * sizeof(C);
    const C *GT = (const C*)pool[1], *GB = (const C*)pool[2];
    // A chunk's chain of inversions and products leaves most issue slots empty (barriers, shared
    // memory), so a third CTA per SM helps once the grid has more than two for each: complex64
    // 3 x 3 tiles fit in its 80 registers without spills.  Factor of 1023 x 1023 30.5 -> 27.5 ms,
    // 511 x 511 9.6 -> 9.0; four CTAs (64 registers, spills) 27.9 and 9.35.  Smaller grids keep
    // the registers (127 x 127: 2.75 ms against 2.79), and so does complex128, bound by the FP64
    // pipe.
    constexpr int kMinB = sizeof(C) == 8 && NI == 3 ? 3 : 0;
    int dev = 0, nsm = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if ((err = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return err;
    const auto chunk_fn = g.P * g.J > 2 * nsm ? k_factor_chunk<C, NI, kMinB> : k_factor_chunk<C, NI, 0>;
    if ((err = attr((const void*)chunk_fn, 3 * blk)) != cudaSuccess) return err;
    {
        TimedLaunch t(tm, "factor_chunk", s);
        chunk_fn<<<dim3(g.P, g.J), kBlockThreads, 3 * blk, s>>>(g, (C*)pool[0], (C*)pool[1], (C*)pool[2], status);
    }
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    if (g.P > 1) {
        SepPools<C> pl{(C*)pool[3], (C*)pool[4], (C*)pool[5], (C*)pool[6], (C*)pool[7], (C*)pool[8], (C*)pool[9],
                       g.G > 1 ? (C*)pool[11] : nullptr, g.G > 1 ? (C*)pool[12] : nullptr};
        const size_t smem = (g.G > 1 ? 4 : 3) * blk;
        const auto group_fn = g.G * g.J > 2 * nsm ? k_factor_sep_group<C, NI, kMinB> : k_factor_sep_group<C, NI, 0>;
        for (const void* fn : {(const void*)group_fn, (const void*)k_factor_sep_l2<C, NI>,
                               (const void*)k_factor_sep_q<C, NI>})
            if ((err = attr(fn, smem)) != cudaSuccess) return err;
        TimedLaunch t(tm, "factor_sep", s);
        group_fn<<<dim3(g.G, g.J), kBlockThreads, smem, s>>>(g, GT, GB, pl, status);
        if (g.G > 1) {
            k_factor_sep_l2<C, NI><<<dim3(1, g.J), kBlockThreads, smem, s>>>(g, GT, GB, pl, status);
            k_factor_sep_q<C, NI><<<dim3(2 * g.G, g.J), kBlockThreads, smem, s>>>(g, GT, GB, pl, status);
        }
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
    if (g.G > 1) {
        const size_t xs = (size_t)2 * Wmax * spld(Wmax) * sizeof(C);
        err = attr((const void*)k_factor_xfer<C>, xs);
        if (err != cudaSuccess) return err;
        TimedLaunch t(tm, "factor_xfer", s);
        k_factor_xfer<C><<<dim3(g.P, g.J), 256, xs, s>>>(g, GT, GB, (const C*)pool[6], (const C*)pool[7],
                                                          (C*)pool[10]);
    }
    return cudaGetLastError();
}

template <typename C>
cudaError_t launch_factor(const Geom& g, int Wmax, void* const* pool, int* status, cudaStream_t s, KernelTimer* tm) {
    if (factor_smem_bytes(Wmax, sizeof(C), g.G > 1 ? 4 : 3) > kFactorSmemMax) return cudaErrorInvalidConfiguration;
    return Wmax <= 48 ? launch_factor_ni<C, 3>(g, Wmax, pool, status, s, tm)
                      : launch_factor_ni<C, 4>(g, Wmax, pool, status, s, tm);
}

template cudaError_t launch_factor<float2>(const Geom&, int, void* const*, int*, cudaStream_t, KernelTimer*);
template cudaError_t launch_factor<double2>(const Geom&, int, void* const*, int*, cudaStream_t, KernelTimer*);

}  // namespace helm
