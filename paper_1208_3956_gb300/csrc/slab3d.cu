// Three-dimensional strips (Section 2.2, Algorithm 1 and the sweeps of Section
// 2.1 on a 3-D grid).  A strip is a slab of W x-columns by all N_z planes; at
// grid row y = k its unknowns form one block of n = W N_z points, ordered
// e = z W + c (strip-local column c fastest).  S^(j) A^(j) is block tridiagonal
// along y with these dense-after-elimination blocks and diagonal couplings:
//   D_k(e,e)     = [s_y s_z (a_x(c+1/2) + a_x(c-1/2))
//                   + s_x s_z (a_y(k+1/2) + a_y(k-1/2))
//                   + s_x s_y (a_z(z+1/2) + a_z(z-1/2))] / h^2 - s_x s_y s_z k^2
//   D_k(e,e+1)   = -s_y s_z a_x(c+1/2) / h^2            (c+1 < W, same plane)
//   D_k(e,e+W)   = -s_x s_y a_z(z+1/2) / h^2
//   C_k(e)       = -s_x(c) s_z(z) a_y(k-1/2) / h^2      (couples rows k-1, k)
// with s = 1/alpha at integer points and a = alpha at half points.
//
// Factorisation (Algorithm 1) from both ends toward a middle row t = (N_y-1)/2, so that the
// elimination and the solves are two independent chains: X_k = S_k^{-1},
//   k < t:  S_k = D_k - C_k X_{k-1} C_k              (top down)
//   k > t:  S_k = D_k - C_{k+1} X_{k+1} C_{k+1}      (bottom up)
//   S_t = D_t - C_t X_{t-1} C_t - C_{t+1} X_{t+1} C_{t+1}
// each S_k inverted by Gauss-Jordan elimination with partial (row) pivoting: complex64 on the
// tensor cores, the rows of both chains of several strips side by side (slab_tc.cu), complex128
// on the whole GPU (one cooperative launch per block).  Solve of a strip (block elimination
// toward t and substitution outward):
//   y_k = X_k (r_k - C_k y_{k-1}),      k < t;    y_k = X_k (r_k - C_{k+1} y_{k+1}),  k > t
//   x_t = X_t (r_t - C_t y_{t-1} - C_{t+1} y_{t+1})
//   x_k = y_k - X_k C_{k+1} x_{k+1},    k < t;    x_k = y_k - X_k C_k x_{k-1},        k > t
// all 2 N_y - 1 block steps in one cooperative launch (k_slab_sweep), each a matrix product
// with the right-hand sides' vectors that streams X_k from HBM through shared memory.
#include <algorithm>

#include <type_traits>

#include "common.cuh"
#include "slab_ops.cuh"
#include "internal.h"

namespace helm {
namespace {

constexpr uint32_t kBarPolls = 1u << 20;   // polls of a grid barrier before it gives up (about a second)
constexpr int kGjThreads = 256;
constexpr int kGjRowsPerThread = 8;        // n <= kGjThreads * kGjRowsPerThread
constexpr int kGjMaxCols = 64;             // columns owned by one CTA
constexpr size_t kGjCacheMax = 200 * 1024; // the owned columns in shared memory, at most

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

template <typename C> __device__ __forceinline__ C ldcg(const C* p);
template <> __device__ __forceinline__ float2 ldcg(const float2* p) { return __ldcg(p); }
template <> __device__ __forceinline__ double2 ldcg(const double2* p) { return __ldcg(p); }

// One thread waits (bounded) until the counter reaches target; a wait that gives up
// records 7 in the status word and returns false.
__device__ bool wait_count(const unsigned* ctr, unsigned target, int* status) {
    unsigned v = ld_acquire_gpu(ctr);
    for (uint32_t it = 0; v < target && it < kBarPolls; ++it) {
        __nanosleep(20);
        v = ld_acquire_gpu(ctr);
    }
    if (v >= target) return true;
    atomicExch(status, 7);
    return false;
}
__device__ __forceinline__ void add_release(unsigned* ctr) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
}

// M (column-major, ldm) = - C_k Xp C_k - C_{k+1} Xn C_{k+1}, Xp = X_{k-1} and Xn = X_{k+1} in the
// tile layout (null: no such term); k_slab_dadd then adds D_k.
template <typename C>
__global__ void __launch_bounds__(256) k_slab_build(Geom g, StripDev st, int k, const C* __restrict__ Xp,
                                                    const C* __restrict__ Xn, C* __restrict__ M, int ldm) {
    slab_build_entries<C>(g, st, k, Xp, Xn, M, ldm);
}

template <typename C>
__global__ void __launch_bounds__(64) k_slab_dadd(Geom g, StripDev st, int k, C* __restrict__ M, int ldm) {
    slab_dadd_entries<C>(g, st, k, M, ldm);
}

// In-place Gauss-Jordan inverse with partial pivoting of the n x n matrix M
// (column-major, ldm), columns dealt round-robin to the CTAs of a cooperative
// launch.  Step i: rows i and p (the largest |M(r,i)|, r >= i) are exchanged,
// the pivot row is scaled by 1/M(p,i) with M(i,i) <- 1/pivot, and every other
// row r loses m_r times it with M(r,i) <- -m_r/pivot (m_r = M(r,i) after the
// exchange).  The owner of column i publishes p and the exchanged column m (one
// buffer per step, never reused, so a CTA may trail the others by any number of
// steps) and raises the published-step counter bar[0] (release, zero at launch); a
// CTA starts step i once that counter says so (acquire).  Only the owner of the next
// column, which it updates first, is on the critical path.  The
// result is (P M)^{-1} for the product P of the exchanges; pinv[c] = the
// position of original row c after all exchanges, so M^{-1}(:, c) = result(:, pinv[c]).
// cached != 0: a CTA keeps its columns in shared memory for the whole elimination.
template <typename C>
__global__ void __launch_bounds__(kGjThreads) k_gj_invert(C* __restrict__ M, int n, int ldm, int* __restrict__ perm,
                                                         int* __restrict__ pinv, C* __restrict__ mult,
                                                         int* __restrict__ pivrow, unsigned* __restrict__ bar,
                                                         int* __restrict__ status, int cached) {
    using R = typename CT<C>::R;
    extern __shared__ __align__(16) unsigned char gj_smem[];
    __shared__ C s_ai[kGjMaxCols], s_ap[kGjMaxCols];
    __shared__ R s_best[kGjThreads / 32];
    __shared__ int s_bidx[kGjThreads / 32];
    __shared__ int s_p, s_ok;
    __shared__ int s_rows[kGjThreads * kGjRowsPerThread];
    const int nb = gridDim.x, b = blockIdx.x, tid = threadIdx.x;
    const int ncol = b < n ? (n - 1 - b) / nb + 1 : 0;   // owned columns b, b+nb, ...
    C* cache = reinterpret_cast<C*>(gj_smem);            // [ncol][n] when cached
    auto colp = [&](int lc) -> C* {
        return cached ? cache + (int64_t)lc * n : M + (int64_t)(b + lc * nb) * ldm;
    };
    if (cached) {
        for (int lc = 0; lc < ncol; ++lc)
            for (int r = tid; r < n; r += kGjThreads) cache[(int64_t)lc * n + r] = M[(int64_t)(b + lc * nb) * ldm + r];
        __syncthreads();
    }

    // pivot search and publication for column i (owned by this CTA, up to date)
    auto publish = [&](int i) {
        const C* col = colp(i / nb);   // i = b + (i / nb) nb
        R best = (R)-1;
        int bi = n;
        for (int r = i + tid; r < n; r += kGjThreads) {
            const R v = cabs2(col[r]);
            if (v > best) { best = v; bi = r; }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const R ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        if ((tid & 31) == 0) { s_best[tid >> 5] = best; s_bidx[tid >> 5] = bi; }
        __syncthreads();
        if (tid == 0) {
            R bb = s_best[0];
            int bx = s_bidx[0];
            for (int w = 1; w < kGjThreads / 32; ++w)
                if (s_best[w] > bb || (s_best[w] == bb && s_bidx[w] < bx)) { bb = s_best[w]; bx = s_bidx[w]; }
            if (!(bb > (R)0) || !(bb < (R)INFINITY) || bx >= n) {
                atomicExch(status, 6);   // zero or non-finite pivot: the result is invalid
                bx = i;
            }
            s_p = bx;
            pivrow[i] = bx;
        }
        __syncthreads();
        const int p = s_p;
        C* mu = mult + (int64_t)i * ldm;
        for (int r = tid; r < n; r += kGjThreads) mu[r] = col[r == i ? p : (r == p ? i : r)];
        __syncthreads();
        if (tid == 0) add_release(bar);   // step i published
    };

    if (b == 0 && ncol > 0) publish(0);   // column 0 belongs to CTA 0
    for (int i = 0; i < n; ++i) {
        if (tid == 0) s_ok = wait_count(bar, (unsigned)(i + 1), status);
        __syncthreads();
        if (!s_ok) return;
        const int p = __ldcg(pivrow + i);
        const C* mu = mult + (int64_t)i * ldm;
        const C ip = cinv(ldcg(mu + i));
        if (b == 0 && tid == 0) perm[i] = p;
        C m_r[kGjRowsPerThread];
#pragma unroll
        for (int u = 0; u < kGjRowsPerThread; ++u) {
            const int r = tid + u * kGjThreads;
            m_r[u] = r < n ? ldcg(mu + r) : CT<C>::zero();
        }
        for (int lc = tid; lc < ncol; lc += kGjThreads) {
            const C* col = colp(lc);
            s_ai[lc] = col[i];
            s_ap[lc] = col[p];
        }
        __syncthreads();
        auto update = [&](int lc) {
            const int c = b + lc * nb;
            C* col = colp(lc);
            const C t = c == i ? ip : cmul(s_ap[lc], ip);
            const C ai = s_ai[lc];
#pragma unroll
            for (int u = 0; u < kGjRowsPerThread; ++u) {
                const int r = tid + u * kGjThreads;
                if (r >= n) continue;
                const C base = c == i ? CT<C>::zero() : (r == p ? ai : col[r]);
                col[r] = r == i ? t : csub(base, cmul(m_r[u], t));
            }
        };
        const int cn = i + 1;
        const int lcn = (cn < n && cn % nb == b) ? cn / nb : -1;
        if (lcn >= 0) {
            update(lcn);
            __syncthreads();
            publish(cn);
        }
        for (int lc = 0; lc < ncol; ++lc)
            if (lc != lcn) update(lc);
        __syncthreads();   // s_ai / s_ap are rewritten at the next step
    }
    if (cached) {
        __syncthreads();
        for (int lc = 0; lc < ncol; ++lc)
            for (int r = tid; r < n; r += kGjThreads) M[(int64_t)(b + lc * nb) * ldm + r] = cache[(int64_t)lc * n + r];
    }
    // the exchanges, replayed: s_rows[r] = original row at position r
    if (b == 0) {
        __syncthreads();
        for (int r = tid; r < n; r += kGjThreads) s_rows[r] = r;
        __syncthreads();
        if (tid == 0)
            for (int i = 0; i < n; ++i) {
                const int p = perm[i], t = s_rows[i];
                s_rows[i] = s_rows[p];
                s_rows[p] = t;
            }
        __syncthreads();
        for (int r = tid; r < n; r += kGjThreads) pinv[s_rows[r]] = r;
    }
}

// X (tile layout) = M^{-1} from the Gauss-Jordan result: X(a, c) = Mgj(a, pinv[c]) =
// M[pinv[c] * ldm + a]; rows n .. of the last tile are zero.
template <typename C>
__global__ void __launch_bounds__(256) k_slab_store(const C* __restrict__ M, int n, int ldm,
                                                    const int* __restrict__ pinv, C* __restrict__ X) {
    const int a = blockIdx.x * 64 + (threadIdx.x & 63), c = blockIdx.y * 4 + (threadIdx.x >> 6);
    if (c < n) X[slab_at(n, a, c)] = a < n ? M[(int64_t)pinv[c] * ldm + a] : CT<C>::zero();
}

// ------------------------------------------------------------------ sweeps
// Right-hand side of a strip solve in the symmetric form (as the 2-D sweep):
//   r(b,k,e) = s_x s_y s_z ([mlo <= gc <= mhi] src(b,z,k,gc)
//                           + [gc == t0 or t0+1] tcoef (xp(to1) - xp(to0)))
// xp: the previous strip solve's solution (strip pst, its transfer columns).
template <typename C>
__global__ void k_slab_rhs(Geom g, StripDev st, SweepStep sp, StripDev pst, const C* __restrict__ ct,
                           int64_t ct_sz, const C* __restrict__ prevY, int pld, C* __restrict__ Rb, int ld, int B) {
    const int W = st.W, Nz = g.Nz, Ny = g.Ny, n = W * Nz;
    const int cofs = st.lo - st.lpml;
    const int64_t tot = (int64_t)B * Ny * ld;
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < tot; o += (int64_t)gridDim.x * blockDim.x) {
        const int e = (int)(o % ld);
        const int k = (int)((o / ld) % Ny);
        const int b = (int)(o / ((int64_t)ld * Ny));
        if (e >= n) { Rb[o] = CT<C>::zero(); continue; }
        const int c = e % W, z = e / W, gc = cofs + c;
        const C s = cmul(cmul(ct[st.ctab + c], ct[g.ct_sy + k]), ct[ct_sz + z]);
        double2 f = make_double2(0.0, 0.0);
        if (gc >= sp.mlo && gc <= sp.mhi) f = sp.src[(((int64_t)b * Nz + z) * Ny + k) * g.Nx + gc];
        C v = cmul(CT<C>::from(f), s);
        if (prevY && (gc == sp.t0 || gc == sp.t0 + 1)) {
            const C* py = prevY + ((int64_t)b * Ny + k) * pld + (int64_t)z * pst.W;
            const C tv = csub(py[pst.xc[2 * sp.pdir + 1]], py[pst.xc[2 * sp.pdir]]);
            v = cadd(v, cmul(cscale(tv, (typename CT<C>::R)sp.tcoef), s));
        }
        Rb[o] = v;
    }
}

// A whole strip solve (2 N_y - 1 block steps) in one cooperative launch, one CTA per SM.
//
// Every block is cut into mr x nq tiles of 128 rows by kc columns; CTA (m, q) streams its tile
// of every block and multiplies it with its kc entries of the step's input vector z (for NB
// right-hand sides).  A step of a chain is
//   product: partial sums of the CTA's 128 rows into P[chain][q], counter part[m] raised;
//   sum:     the CTA's own `epc` entries of its row tile: y = sum over q of P (plus y_k on the
//            way out), stored to Y, and the next step's z = r - C y on them, counter vec[m]
//            raised.
// A CTA's sums wait for the nq CTAs of its row tile only, and its copy of z for the row tiles that
// hold its kc columns (two or three at 1800 unknowns, up to nine at 4000).  Z and P are double buffered by the step's parity: a CTA
// enters product s+2 after the products s+1 of its row tile, each of which followed its
// CTA's sums of step s; and it writes z of step s+2 after all of its row tile's products
// s+1, which together waited for every CTA's z of step s+1 and so for every product s.
// The two chains are independent up to the middle row, and the warps are specialised, so that
// one chain's sums, counters and vector loads run while the other chain's tile is multiplied:
//   8 product warps  walk both chains in turn (top, bottom, top, ...);
//   2 x 3 sum warps  one group per chain: sums, z, and the copy of z into shared memory (by
//                    plain loads: a bulk copy would queue behind the ring's tiles);
//   1 producer warp  streams the tiles, step after step, through a ring of column slots
//                    (cp.async.bulk + mbarriers) ahead of the products and never waits for z.
// Splitting the columns too (instead of giving a CTA whole rows) keeps a CTA's share of z at
// kc entries: with whole rows the vectors of 8 right-hand sides were more L2 traffic than the
// blocks themselves (63^3 grid, blocks of 1659: 19 us per block and 8 right-hand sides).
// A warp's lane holds 4 of the 128 rows (two adjacent ones in each 64-row half), so a product
// needs no reduction over lanes; the warps split the slot's columns (and, for 16 right-hand
// sides, the right-hand sides in two), their sums meet in shared memory once per step.
// What bounds it: with one right-hand side the chain's latency under the stream's load (tile
// 7.4k cycles, the rest of a step about 12k, half of it hidden by the other chain); with 16
// instruction issue (54 %, the FMA pipe 40 %, shared memory 30 % on a 39^3 grid) and the barriers
// that end a step; in complex128 the FP64 pipe (83 % with two on 33 x 37 x 29).  One application of P on the 63^3 grid
// (8 strips, blocks of 1659-1817, 15 strip solves; top-down elimination with whole rows per
// CTA and tiles of 4 right-hand sides before): 16.4 -> 11.3 ms with one right-hand side (3.2
// -> 4.7 TB/s of blocks), 127 -> 28.3 ms with 16.  Complex128 on 33 x 37 x 29 (blocks of 779 and
// 820): 21.3 -> 6.5, 60.1 -> 9.7 and 59.9 -> 19.2 ms with 1, 2 and 4.
// Every wait is bounded: on time-out the kernel records 7 in the status word, waits (bounded)
// for its copies in flight and returns.
template <typename C>
struct SlabSweepArgs {
    const C* X;          // block 0 of the strip in the tile layout (slab_ops.cuh); block k at X + k * bs
    int64_t bs;
    int n, Ny;
    int nq, kc, epc, slots;
    const C* rhs;        // [B][Ny][ld] right-hand sides
    C* Y;                // [B][Ny][ld] solution
    int ld, B;           // row stride of rhs / Y; right-hand sides of this launch (<= NB)
    const C* sxz;        // s_x(c) s_z(z) per block entry
    const C* cyt;        // -alpha_y(y_{k-1/2}) / h^2, k = 0 .. Ny
    C* Z;                // [chain][step parity][nz][NB] input vectors, nz = n rounded up to even
    C* P;                // [chain][step parity][nq][n][NB] partial sums
    unsigned* bar;       // counters [part, vec][chain][kMaxRowTiles], kCtrStride apart, zero at launch
    int* status;
};
constexpr int kCtrStride = 32;      // counters on separate 128-byte lines
constexpr int kMaxRowTiles = 32;    // blocks of up to 4096 unknowns
constexpr size_t kCtrBytes = (size_t)4 * kMaxRowTiles * kCtrStride * sizeof(unsigned);   // 16 KB
__device__ __forceinline__ unsigned* slab_ctr(unsigned* bar, int vec, int ch, int m) {
    return bar + ((vec * 2 + ch) * kMaxRowTiles + m) * kCtrStride;
}
constexpr int kProdWarps = 8, kSumThreads = 96;
constexpr int kSweepThreads = 32 * kProdWarps + 2 * kSumThreads + 32;
constexpr int kSlotBytes = 16 * 1024;   // a ring slot: 16 (complex64) or 8 columns of 128 rows
constexpr int kMaxSlots = 16;
constexpr size_t kSlabSmemMax = 227 * 1024;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mb_init(uint64_t* m, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(m)), "r"(count) : "memory");
}
__device__ __forceinline__ void mb_expect_tx(uint64_t* m, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(m)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mb_arrive(uint64_t* m) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(m)) : "memory");
}
// bounded; gives up early once the CTA has recorded a failed wait
__device__ __forceinline__ bool mb_wait(uint64_t* m, uint32_t parity, const volatile int* abort_flag = nullptr) {
    for (uint32_t it = 0; it < kBarPolls; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(smem_addr(m)), "r"(parity)
            : "memory");
        if (ok) return true;
        if (abort_flag && *abort_flag) return false;
    }
    return false;
}
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* m) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(m))
        : "memory");
}
__device__ __forceinline__ void group_sync(int id, int nthr) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthr) : "memory");
}

// Barrier of the group that returns, to all its threads alike, whether any of them passed v != 0.
__device__ __forceinline__ bool group_or(int id, int nthr, int v) {
    uint32_t r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %1, 0;\n bar.red.or.pred q, %2, %3, p;\n selp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"(v), "r"(id), "r"(nthr)
        : "memory");
    return r != 0;
}

// The grid row of step i of a chain: the top chain (0) walks rows 0 .. t-1, t, t-1 .. 0, the
// bottom chain (1) rows N_y-1 .. t+1, t+1 .. N_y-1, with t = (N_y-1)/2.
__device__ __forceinline__ int slab_row(int chain, int i, int Ny) {
    const int t = (Ny - 1) / 2, nu = Ny - 1 - t;
    if (chain == 0) return i <= t ? i : 2 * t - i;
    return i < nu ? Ny - 1 - i : t + 1 + (i - nu);
}
// Step p of the walk over both chains: their forward steps in turn, the middle row, the
// outward steps in turn; the bottom chain's extra row (N_y even) comes last of its half.
__device__ __forceinline__ int slab_chain(int p, int Ny) {
    const int t = (Ny - 1) / 2, nu = Ny - 1 - t, nf = t + nu;
    if (p == nf) return 0;
    const int q = p < nf ? p : p - nf - 1;
    return q >= 2 * t ? 1 : q & 1;
}

// two adjacent entries of shared memory (16-byte aligned in complex64)
__device__ __forceinline__ void ld_pair(const float2* p, float2& a, float2& b) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void ld_pair(const double2* p, double2& a, double2& b) { a = p[0]; b = p[1]; }

__device__ __forceinline__ void ldcg_pair(const float2* p, float2& a, float2& b) {
    const float4 v = __ldcg(reinterpret_cast<const float4*>(p));
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void ldcg_pair(const double2* p, double2& a, double2& b) { a = __ldcg(p); b = __ldcg(p + 1); }

// Right-hand sides of a tile and how the product warps share them: kRG groups of warps take
// NB / kRG each, the others split the columns.
template <int NB> struct SlabTile {
    static constexpr int kRG = NB > 8 ? 2 : 1, kN = NB / kRG, kKG = kProdWarps / kRG;
    // the column groups' sums, [group][4 rows][NB][33] (the last dimension padded so that the
    // lanes of a warp read and write different banks)
    static constexpr int kRed = kKG * 4 * NB * 33;
    static constexpr int kMaxEpc = NB > 8 ? 18 : 36;                         // own entries of a CTA, at most
    static constexpr int kVals = (kMaxEpc * NB + kSumThreads - 1) / kSumThreads;   // values of a sum thread
};

template <typename C, int NB>
__host__ __device__ inline size_t slab_sweep_fixed(int kc) {
    return (size_t)2 * kc * NB * sizeof(C) + (size_t)SlabTile<NB>::kRed * sizeof(C) +
           (2 * kMaxSlots + 4) * 8 + 16;
}

template <typename C, int NB>
__global__ void __launch_bounds__(kSweepThreads, 1) k_slab_sweep(SlabSweepArgs<C> A) {
    using T = SlabTile<NB>;
    constexpr int SC = kSlotBytes / (128 * (int)sizeof(C));   // columns of a slot
    extern __shared__ __align__(128) unsigned char sweep_smem[];
    C* ring = reinterpret_cast<C*>(sweep_smem);                                   // [slots][2][SC][64]
    C* zs = reinterpret_cast<C*>(sweep_smem + (size_t)A.slots * kSlotBytes);      // [2][kc][NB]
    C* red = zs + (size_t)2 * A.kc * NB;                                          // [column group][4 rows][NB][33]
    uint64_t* full = reinterpret_cast<uint64_t*>(red + T::kRed);
    uint64_t* empty = full + kMaxSlots;
    uint64_t* zfull = empty + kMaxSlots;   // [2] z of the chain's step is in zs
    uint64_t* xdone = zfull + 2;           // [0] middle row summed, [1] bottom chain's forward half summed
    volatile int* abort_flag = reinterpret_cast<volatile int*>(xdone + 2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int Ny = A.Ny, n = A.n, nz = (n + 1) & ~1;
    const int m = (int)blockIdx.x / A.nq, q = (int)blockIdx.x % A.nq;
    const int row0 = m * 128;
    const int c0 = q * A.kc, ncol = imin(A.kc, n - c0);
    const bool half2 = row0 + 64 < n;   // the tile's second 64-row half exists
    const int nslot = (ncol + SC - 1) / SC;
    const int t = (Ny - 1) / 2, nu = Ny - 1 - t;
    if (tid == 0) {
        for (int i = 0; i < A.slots; ++i) { mb_init(&full[i], 1); mb_init(&empty[i], kProdWarps); }
        for (int i = 0; i < 2; ++i) { mb_init(&zfull[i], kSumThreads); mb_init(&xdone[i], 1); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    auto give_up = [&]() { atomicExch(A.status, 7); *abort_flag = 1; };

    if (warp == kSweepThreads / 32 - 1) {   // ---- producer
        if (lane == 0) {
            uint32_t g = 0;
            bool ok = true;
            int step[2] = {0, 0};
            for (int p = 0; p < 2 * Ny - 1 && ok; ++p) {
                const int ch = slab_chain(p, Ny);
                const int k = slab_row(ch, ch ? step[1]++ : step[0]++, Ny);
                const C* lo = A.X + (int64_t)k * A.bs + ((int64_t)(2 * m) * n + c0) * 64;
                const C* hi = lo + (int64_t)n * 64;
                for (int i = 0; i < nslot; ++i, ++g) {
                    const int slot = (int)(g % (uint32_t)A.slots);
                    const uint32_t use = g / (uint32_t)A.slots;
                    if (use > 0 && !mb_wait(&empty[slot], (use - 1) & 1, abort_flag)) { ok = false; break; }
                    const uint32_t bytes = (uint32_t)(imin(SC, ncol - i * SC) * 64 * (int)sizeof(C));
                    C* dst = ring + (int64_t)slot * (kSlotBytes / (int)sizeof(C));
                    mb_expect_tx(&full[slot], half2 ? 2 * bytes : bytes);
                    bulk_copy(dst, lo + (int64_t)i * SC * 64, bytes, &full[slot]);
                    if (half2) bulk_copy(dst + SC * 64, hi + (int64_t)i * SC * 64, bytes, &full[slot]);
                }
            }
            if (!ok && !*abort_flag) give_up();
            // copies still in flight land before the CTA exits
            const uint32_t lo = g > (uint32_t)A.slots ? g - (uint32_t)A.slots : 0;
            for (uint32_t i = lo; i < g; ++i) mb_wait(&full[i % (uint32_t)A.slots], (i / (uint32_t)A.slots) & 1);
        }
        return;
    }

    if (warp >= kProdWarps) {   // ---- sum warps of chain ch
        const int ch = (tid - 32 * kProdWarps) / kSumThreads, at = (tid - 32 * kProdWarps) % kSumThreads;
        const int nstep = ch == 0 ? 2 * t + 1 : 2 * nu;
        const int e0 = row0 + q * A.epc, ne = imax(0, imin(A.epc, imin(n, row0 + 128) - e0));
        unsigned* c_part = slab_ctr(A.bar, 0, ch, m);
        unsigned* c_vec = slab_ctr(A.bar, 1, ch, m);
        const int mz0 = c0 / 128, mz1 = (c0 + ncol - 1) / 128;   // row tiles that hold this CTA's columns
        // waits (one thread) until a counter reaches `target`
        auto poll = [&](const unsigned* ctr, unsigned target) -> bool {
            unsigned v = ld_acquire_gpu(ctr);
            for (uint32_t it = 0; v < target && it < kBarPolls && !*abort_flag; ++it) v = ld_acquire_gpu(ctr);
            return v >= target;
        };
        int ve[T::kVals], vb[T::kVals];   // this thread's values: entry (clamped), right-hand side
        bool on[T::kVals], st[T::kVals];  // value exists / is a right-hand side of this launch
        C sx[T::kVals], y[T::kVals];
#pragma unroll
        for (int i = 0; i < T::kVals; ++i) {
            const int v = at + i * kSumThreads;
            on[i] = v < ne * NB;
            ve[i] = imin(e0 + v / NB, n - 1);
            vb[i] = v % NB;
            st[i] = on[i] && vb[i] < A.B;
            sx[i] = A.sxz[ve[i]];
            y[i] = CT<C>::zero();
        }
        auto yp = [&](int i, int k) -> C* { return A.Y + ((int64_t)imin(vb[i], A.B - 1) * Ny + k) * A.ld + ve[i]; };
        auto forward = [&](int s) { return ch == 0 ? s <= t : s < nu; };
        // of step s: the right-hand side, or y_k on the way out (the bottom chain turns on the row
        // it has just summed, whose value is still in y)
        C base[T::kVals], next[T::kVals], cy0 = CT<C>::zero(), cy1 = CT<C>::zero();
        auto load_step = [&](int s) {   // and the couplings to the step before and, at the middle row, to y_{t+1}
            const int k = slab_row(ch, s, Ny);
            const bool fwd = forward(s);
            cy0 = A.cyt[ch == 0 ? (s <= t ? k : k + 1) : (s < nu ? k + 1 : k)];
            cy1 = A.cyt[k + 1];
            if (ch == 1 && s == nu) return;
#pragma unroll
            for (int i = 0; i < T::kVals; ++i)
                next[i] = !st[i] ? CT<C>::zero()
                          : fwd  ? ldcg(A.rhs + ((int64_t)vb[i] * Ny + k) * A.ld + ve[i])
                                 : ldcg(yp(i, k));
        };
        if (nstep > 0) load_step(0);
        for (int s = 0; s < nstep; ++s) {
            const int k = slab_row(ch, s, Ny);
            const bool mid = ch == 0 && s == t, fwd = forward(s);
#pragma unroll
            for (int i = 0; i < T::kVals; ++i) base[i] = ch == 1 && s == nu ? y[i] : next[i];
            // the other chain's values of the same entries: y_{t+1} at the middle row, x_t for the
            // bottom chain's way out
            bool ok = true;
            const bool cross = (mid && nu > 0) || (ch == 1 && s == nu);
            if (cross) ok = mb_wait(&xdone[mid ? 1 : 0], 0, abort_flag);
            C* zg = A.Z + (int64_t)(ch * 2 + (s & 1)) * nz * NB;
#pragma unroll
            for (int i = 0; i < T::kVals; ++i) {
                if (!on[i]) continue;
                C z = fwd ? base[i] : CT<C>::zero();
                if (st[i]) {
                    C prev = y[i];
                    if (ch == 1 && s == nu) prev = ldcg(yp(i, t));
                    if (s > 0) z = csub(z, cmul(cmul(cy0, sx[i]), prev));
                    if (mid && nu > 0) z = csub(z, cmul(cmul(cy1, sx[i]), ldcg(yp(i, t + 1))));
                }
                zg[(int64_t)ve[i] * NB + vb[i]] = z;
            }
            if (!ok) give_up();
            group_sync(2 + ch, kSumThreads);
            const unsigned target = (unsigned)(s + 1) * (unsigned)A.nq;
            if (at == 0) {
                asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(c_vec) : "memory");
                bool zok = !*abort_flag;
                for (int mm = mz0; mm <= mz1 && zok; ++mm) zok = poll(slab_ctr(A.bar, 1, ch, mm), target);
                if (!zok && !*abort_flag) give_up();
            }
            if (group_or(2 + ch, kSumThreads, *abort_flag)) return;
            // z of this CTA's columns into shared memory, two entries a load; every product of the
            // previous step has read zs (its partial sums are in)
            {
                const C* src = zg + (int64_t)c0 * NB;
                C* dst = zs + (size_t)ch * A.kc * NB;
                const int tot = (ncol * NB + 1) / 2;
                constexpr int kBatch = sizeof(C) == sizeof(float2) ? 8 : 4;
                for (int o0 = at; o0 < tot; o0 += kBatch * kSumThreads) {
                    C v[kBatch][2];
#pragma unroll
                    for (int j = 0; j < kBatch; ++j)
                        ldcg_pair(src + 2 * imin(o0 + j * kSumThreads, tot - 1), v[j][0], v[j][1]);
#pragma unroll
                    for (int j = 0; j < kBatch; ++j) {
                        const int o = o0 + j * kSumThreads;
                        if (o < tot) { dst[2 * o] = v[j][0]; dst[2 * o + 1] = v[j][1]; }
                    }
                }
                mb_arrive(&zfull[ch]);
            }
            if (s + 1 < nstep) load_step(s + 1);   // in flight during the wait
            if (at == 0 && !poll(c_part, target) && !*abort_flag) give_up();
            if (group_or(2 + ch, kSumThreads, *abort_flag)) return;
            // y = [y_k +] the sum of the partial sums
            const C* pp = A.P + (int64_t)(ch * 2 + (s & 1)) * A.nq * n * NB;
#pragma unroll
            for (int i = 0; i < T::kVals; ++i) y[i] = fwd ? CT<C>::zero() : base[i];
            constexpr int kBatch = 6;   // partial sums in flight per value
            for (int j0 = 0; j0 < A.nq; j0 += kBatch) {
                C v[T::kVals][kBatch];
#pragma unroll
                for (int i = 0; i < T::kVals; ++i)
#pragma unroll
                    for (int j = 0; j < kBatch; ++j)
                        v[i][j] = ldcg(pp + ((int64_t)imin(j0 + j, A.nq - 1) * n + ve[i]) * NB + vb[i]);
#pragma unroll
                for (int i = 0; i < T::kVals; ++i)
#pragma unroll
                    for (int j = 0; j < kBatch; ++j)
                        if (j0 + j < A.nq) y[i] = cadd(y[i], v[i][j]);
            }
#pragma unroll
            for (int i = 0; i < T::kVals; ++i)
                if (st[i]) *yp(i, k) = y[i];
            if (mid || (ch == 1 && s == nu - 1)) {
                group_sync(2 + ch, kSumThreads);
                if (at == 0) mb_arrive(&xdone[mid ? 0 : 1]);
            }
        }
        return;
    }

    // ---- product warps
    const int rg = warp % T::kRG, kg = warp / T::kRG;   // right-hand sides, columns
    const int rl = 2 * lane;                            // rows rl, rl+1 of each half
    uint32_t g = 0;
    int step[2] = {0, 0};
    for (int p = 0; p < 2 * Ny - 1; ++p) {
        const int ch = slab_chain(p, Ny);
        const int s = ch ? step[1]++ : step[0]++;
        bool ok = __all_sync(0xffffffffu, mb_wait(&zfull[ch], (uint32_t)(s & 1), abort_flag));
        const C* zc = zs + (size_t)ch * A.kc * NB + rg * T::kN;
        C acc[4][T::kN];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int b = 0; b < T::kN; ++b) acc[r][b] = CT<C>::zero();
        for (int i = 0; i < nslot && ok; ++i, ++g) {
            const int slot = (int)(g % (uint32_t)A.slots);
            ok = mb_wait(&full[slot], (g / (uint32_t)A.slots) & 1, abort_flag);
            if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
            const C* xs = ring + (int64_t)slot * (kSlotBytes / (int)sizeof(C)) + rl;
            const int nc = imin(SC, ncol - i * SC);
#pragma unroll 2
            for (int c = kg; c < nc; c += T::kKG) {
                C x[4], z[T::kN];
                ld_pair(xs + c * 64, x[0], x[1]);
                ld_pair(xs + (SC + c) * 64, x[2], x[3]);
                const C* zp = zc + (size_t)(i * SC + c) * NB;
                if constexpr (T::kN == 1) {
                    z[0] = zp[0];
                } else {
#pragma unroll
                    for (int b = 0; b < T::kN; b += 2) ld_pair(zp + b, z[b], z[b + 1]);
                }
#pragma unroll
                for (int b = 0; b < T::kN; ++b)
#pragma unroll
                    for (int r = 0; r < 4; ++r) acc[r][b] = cfma(x[r], z[b], acc[r][b]);
            }
            __syncwarp();
            if (lane == 0) mb_arrive(&empty[slot]);
        }
        if (!ok && lane == 0 && !*abort_flag) give_up();
        C* pp = A.P + (int64_t)((ch * 2 + (s & 1)) * A.nq + q) * n * NB;
        C* rr = red + (size_t)kg * 4 * NB * 33 + (size_t)rg * T::kN * 33 + lane;
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int b = 0; b < T::kN; ++b) rr[(r * NB + b) * 33] = acc[r][b];
        group_sync(1, 32 * kProdWarps);
        for (int o = tid; o < 128 * NB; o += 32 * kProdWarps) {   // adjacent threads: adjacent right-hand sides
            const int b = o % NB, rw = o / NB;                    // row of the tile
            const int h2 = rw >> 6, l = (rw & 63) >> 1, r = 2 * h2 + (rw & 1);
            C v = CT<C>::zero();
#pragma unroll
            for (int h = 0; h < T::kKG; ++h) v = cadd(v, red[((size_t)(h * 4 + r) * NB + b) * 33 + l]);
            if (row0 + rw < n) pp[(int64_t)(row0 + rw) * NB + b] = v;
        }
        if (group_or(1, 32 * kProdWarps, *abort_flag)) return;
        if (tid == 0)
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(slab_ctr(A.bar, 0, ch, m)) : "memory");
    }
}

// dst(b,z,k,gc) = [base] + x(b,k,e) on padded columns olo..ohi of the strip
template <typename C>
__global__ void k_slab_out(Geom g, StripDev st, int dir, const C* __restrict__ Y, int ld, double2* __restrict__ dst,
                           const double2* __restrict__ base, int B) {
    const int cofs = st.lo - st.lpml;
    const int olo = st.olo[dir], ohi = min(st.ohi[dir], cofs + st.W - 1), nc = ohi - olo + 1;
    const int64_t tot = (int64_t)B * g.Nz * g.Ny * nc;
    for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < tot; o += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(o % nc);
        int64_t t = o / nc;
        const int k = (int)(t % g.Ny);
        t /= g.Ny;
        const int z = (int)(t % g.Nz);
        const int b = (int)(t / g.Nz);
        const int gc = olo + i, c = gc - cofs;
        const double2 x = to_d2(Y[((int64_t)b * g.Ny + k) * ld + (int64_t)z * st.W + c]);
        const int64_t idx = (((int64_t)b * g.Nz + z) * g.Ny + k) * g.Nx + gc;
        dst[idx] = base ? cadd(base[idx], x) : x;
    }
}

int grid_for(int64_t work, int threads) {
    const int64_t blocks = (work + threads - 1) / threads;
    return (int)(blocks < 1 ? 1 : (blocks > 152 * 16 ? 152 * 16 : blocks));
}

}  // namespace

// ------------------------------------------------------------------ host
cudaError_t launch_slab_factor(const Geom& g, const StripDev& st, void* pool, const SlabScratch& sc, int* status,
                               cudaStream_t s, KernelTimer* tm) {
    using C = double2;
    const int n = st.W * g.Nz;
    if (n > kGjThreads * kGjRowsPerThread) return cudaErrorInvalidValue;
    int dev = 0, nsm = 0, occ = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int nb = imin(nsm, n);
    if ((n + nb - 1) / nb > kGjMaxCols) return cudaErrorInvalidConfiguration;
    // the owned columns stay in shared memory when they fit
    const size_t cache = (size_t)((n + nb - 1) / nb) * n * sizeof(C);
    int cached = cache <= kGjCacheMax ? 1 : 0;
    size_t dsmem = cached ? cache : 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_gj_invert<C>, kGjThreads, dsmem);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    C* X = reinterpret_cast<C*>(pool) + st.fac;
    C* M = reinterpret_cast<C*>(sc.M);
    C* mult = reinterpret_cast<C*>(sc.mult);
    const dim3 tiles((n + 63) / 64, (n + 3) / 4), tiles_st((n + 63) / 64, (n + 3) / 4);
    const int tmid = (g.Ny - 1) / 2;
    for (int i = 0; i < g.Ny; ++i) {   // rows 0 .. t-1, N_y-1 .. t+1, t
        const int k = i < tmid ? i : i < g.Ny - 1 ? g.Ny - 1 - (i - tmid) : tmid;
        const C* Xp = k > 0 && k <= tmid ? X + (int64_t)(k - 1) * st.bs : nullptr;
        const C* Xn = k + 1 < g.Ny && k >= tmid ? X + (int64_t)(k + 1) * st.bs : nullptr;
        {
            TimedLaunch t(tm, "slab_build", s);
            k_slab_build<C><<<tiles, 256, 0, s>>>(g, st, k, Xp, Xn, M, sc.ldm);
            k_slab_dadd<C><<<(5 * n + 63) / 64, 64, 0, s>>>(g, st, k, M, sc.ldm);
        }
        e = cudaMemsetAsync(sc.bar, 0, 2 * sizeof(unsigned), s);
        if (e != cudaSuccess) return e;
        {
            TimedLaunch t(tm, "slab_gj_invert", s);
            int nn = n, ldm = sc.ldm;
            void* args[] = {&M, &nn, &ldm, (void*)&sc.perm, (void*)&sc.pinv, &mult, (void*)&sc.pivrow,
                            (void*)&sc.bar, &status, &cached};
            e = cudaLaunchCooperativeKernel((const void*)k_gj_invert<C>, dim3(nb), dim3(kGjThreads), args, dsmem, s);
            if (e != cudaSuccess) return e;
        }
        {
            TimedLaunch t(tm, "slab_store", s);
            k_slab_store<C><<<tiles_st, 256, 0, s>>>(M, n, sc.ldm, sc.pinv, X + (int64_t)k * st.bs);
        }
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// The tile grid of a strip solve: mr row tiles of 128, nq column chunks of kc, at most one tile
// per SM and at least 32 columns in a chunk (below that the partial sums of the chunks cost
// more than the tiles).
struct SlabGrid {
    int nq, kc, ncta, epc;
};
static SlabGrid slab_grid(int n, int nsm) {
    SlabGrid r;
    const int mr = (n + 127) / 128;
    r.nq = imax(1, imin(nsm / mr, (n + 31) / 32));
    r.kc = ((n + r.nq - 1) / r.nq + 1) & ~1;   // even: every chunk of z starts 16-byte aligned
    r.nq = (n + r.kc - 1) / r.kc;
    r.ncta = mr * r.nq;
    r.epc = (imin(n, 128) + r.nq - 1) / r.nq;
    return r;
}
// The strip-solve kernel for tiles of NB right-hand sides, if the vectors and a ring of at least
// four slots fit in shared memory.
struct SlabKernel {
    const void* fn = nullptr;
    int nb = 0, slots = 0;
    size_t smem = 0;
};
template <typename C, int NB>
static bool slab_kernel(const SlabGrid& gr, SlabKernel& k) {
    const size_t fixed = slab_sweep_fixed<C, NB>(gr.kc);
    if (gr.epc > SlabTile<NB>::kMaxEpc || fixed + 4 * kSlotBytes > kSlabSmemMax) return false;
    k.fn = (const void*)k_slab_sweep<C, NB>;
    k.nb = NB;
    k.slots = (int)std::min<size_t>(kMaxSlots, (kSlabSmemMax - fixed) / kSlotBytes);
    k.smem = fixed + (size_t)k.slots * kSlotBytes;
    return true;
}
// For `left` remaining right-hand sides: the widest useful tile that fits (a tile streams every
// block once whatever its width).  Complex128 takes two at most: the FP64 pipe is 83 % busy
// then and DRAM 9 %, so a wider tile would stream less and take as long.
template <typename C>
static SlabKernel pick_slab_kernel(const SlabGrid& gr, int left) {
    SlabKernel k;
    if constexpr (std::is_same<C, float2>::value) {
        if (left > 8 && slab_kernel<C, 16>(gr, k)) return k;
        if (left > 4 && slab_kernel<C, 8>(gr, k)) return k;
        if (left > 1 && slab_kernel<C, 4>(gr, k)) return k;
    } else {
        if (left > 1 && slab_kernel<C, 2>(gr, k)) return k;
    }
    slab_kernel<C, 1>(gr, k);
    return k;
}
constexpr int kSlabMaxNb = 16;
static cudaError_t sm_count(int& nsm) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    return e;
}
// Z and P of the strip solve, for strips of up to nmax unknowns.
size_t slab_sweep_scratch(int nmax, size_t esize) {
    int nsm = 0;
    if (sm_count(nsm) != cudaSuccess) return 0;
    size_t p = 0;
    for (int n = 1; n <= nmax; ++n) p = std::max(p, (size_t)4 * slab_grid(n, nsm).nq * n * kSlabMaxNb * esize);
    return (size_t)4 * (nmax + 1) * kSlabMaxNb * esize + p;
}

template <typename C>
cudaError_t launch_slab_solve(const Geom& g, const StripDev& st, const StripDev* pst, const SweepStep& sp,
                              const SlabWork& wk, const void* pool, cudaStream_t s, KernelTimer* tm) {
    const int n = st.W * g.Nz, Ny = g.Ny, ld = wk.ld, B = wk.B;
    const C* ct = reinterpret_cast<const C*>(g.ct);
    C* Rb = reinterpret_cast<C*>(wk.rbuf);
    C* Y = reinterpret_cast<C*>(wk.ybuf);
    const C* X = reinterpret_cast<const C*>(pool) + st.fac;
    const C* sxz = reinterpret_cast<const C*>(wk.sxz);
    {
        TimedLaunch t(tm, "slab_rhs", s);
        const StripDev pd = pst ? *pst : st;
        k_slab_rhs<C><<<grid_for((int64_t)B * Ny * ld, 256), 256, 0, s>>>(
            g, st, sp, pd, ct, wk.ct_sz, pst ? reinterpret_cast<const C*>(wk.pybuf) : nullptr, ld, Rb, ld, B);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int nsm = 0;
    e = sm_count(nsm);
    if (e != cudaSuccess) return e;
    if (n > 128 * kMaxRowTiles) return cudaErrorInvalidValue;
    const SlabGrid gr = slab_grid(n, nsm);
    for (int b0 = 0; b0 < B;) {
        const SlabKernel kr = pick_slab_kernel<C>(gr, B - b0);
        if (!kr.fn) return cudaErrorInvalidValue;
        const int nb = imin(kr.nb, B - b0);
        SlabSweepArgs<C> A{};
        A.X = X;
        A.bs = st.bs;
        A.n = n;
        A.Ny = Ny;
        A.nq = gr.nq;
        A.kc = gr.kc;
        A.epc = gr.epc;
        A.slots = kr.slots;
        A.rhs = Rb + (int64_t)b0 * Ny * ld;
        A.Y = Y + (int64_t)b0 * Ny * ld;
        A.ld = ld;
        A.B = nb;
        A.sxz = sxz;
        A.cyt = ct + g.ct_cy;
        A.Z = reinterpret_cast<C*>(wk.scratch);
        A.P = A.Z + (size_t)4 * ((n + 1) & ~1) * kr.nb;
        A.bar = wk.bar;
        A.status = wk.status;
        e = cudaMemsetAsync(wk.bar, 0, kCtrBytes, s);
        if (e != cudaSuccess) return e;
        TimedLaunch t(tm, "slab_sweep", s);
        void* args[] = {&A};
        e = cudaLaunchCooperativeKernel(kr.fn, dim3(gr.ncta), dim3(kSweepThreads), args, kr.smem, s);
        if (e != cudaSuccess) return e;
        b0 += nb;
    }
    return cudaGetLastError();
}

template <typename C>
cudaError_t launch_slab_out(const Geom& g, const StripDev& st, int dir, const void* ybuf, int ld, double2* dst,
                            const double2* base, int B, cudaStream_t s, KernelTimer* tm) {
    TimedLaunch t(tm, "slab_out", s);
    const int64_t work = (int64_t)B * g.Nz * g.Ny *
                         (std::min(st.ohi[dir], st.lo - st.lpml + st.W - 1) - st.olo[dir] + 1);
    k_slab_out<C><<<grid_for(work, 256), 256, 0, s>>>(g, st, dir, reinterpret_cast<const C*>(ybuf), ld, dst, base,
                                                     B);
    return cudaGetLastError();
}

cudaError_t preload_slab_kernels(size_t esize) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaSuccess;
    auto limit = [&](const void* fn, size_t bytes) {   // (this also loads the kernel)
        if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    if (esize == sizeof(float2)) {
        for (const void* fn : {(const void*)k_slab_sweep<float2, 1>, (const void*)k_slab_sweep<float2, 4>,
                               (const void*)k_slab_sweep<float2, 8>, (const void*)k_slab_sweep<float2, 16>})
            limit(fn, kSlabSmemMax);
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_slab_rhs<float2>);
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_slab_out<float2>);
    } else {
        limit((const void*)k_slab_sweep<double2, 1>, kSlabSmemMax);
        limit((const void*)k_slab_sweep<double2, 2>, kSlabSmemMax);
        limit((const void*)k_gj_invert<double2>, kGjCacheMax);
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_slab_rhs<double2>);
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_slab_out<double2>);
    }
    return e;
}

#define HELM_SLAB_INST(C)                                                                                       \
    template cudaError_t launch_slab_solve<C>(const Geom&, const StripDev&, const StripDev*, const SweepStep&, \
                                              const SlabWork&, const void*, cudaStream_t, KernelTimer*);       \
    template cudaError_t launch_slab_out<C>(const Geom&, const StripDev&, int, const void*, int, double2*,     \
                                            const double2*, int, cudaStream_t, KernelTimer*);
HELM_SLAB_INST(float2)
HELM_SLAB_INST(double2)
#undef HELM_SLAB_INST

}  // namespace helm
