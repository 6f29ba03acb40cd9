// Block-row coefficients of the symmetrised strip operator S^(j) A^(j) and the
// block-level dense kernels (Gauss-Jordan inverse, products) shared by the
// factorisation kernels.
//
// Ordering: the strip's unknowns are grouped by grid row y = k (block k holds
// the W columns of the strip).  S^(j) A^(j) is then block tridiagonal:
//   diagonal block D_k  = tridiagonal W x W (x-part of Section 2.2 plus the
//                         y-diagonal and -S k^2),
//   coupling   C_k      = diagonal, couples rows k-1 and k,
//                         C_k(c) = -s_x(c) alpha_y(y_{k-1/2}) / h^2.
// Symmetrised entries (row (c,k) of A times s_x(c) s_y(k), s = 1/alpha):
//   D_k(c,c)   = s_y(k)[a_x(c+1/2) + a_x(c-1/2)]/h^2 + s_x(c)[a_y(k+1/2) + a_y(k-1/2)]/h^2
//                - s_x(c) s_y(k) k^2(c,k)
//   D_k(c,c+1) = D_k(c+1,c) = -s_y(k) a_x(c+1/2)/h^2
// With Robin transmission the strips carry no added layers and the diagonal of an
// internal boundary column gains s_x s_y (a/b)/h^2 (Geom::rab).
#pragma once

#include "common.cuh"

namespace helm {

__device__ __forceinline__ double2 strip_ax_int(const Geom& g, const StripDev& st, int c) {
    return g.stab[st.tab + c];
}
__device__ __forceinline__ double2 strip_ax_half(const Geom& g, const StripDev& st, int m) {
    return g.stab[st.tab + st.W + m];   // alpha at strip half point m - 1/2
}
__device__ __forceinline__ int strip_k2_col(const StripDev& st, int c) {
    return imin(imax(st.lo - st.lpml + c, st.lo), st.hi);
}
__device__ __forceinline__ double2 strip_sx(const Geom& g, const StripDev& st, int c) {
    return cinv(strip_ax_int(g, st, c));
}
__device__ __forceinline__ double2 glob_sy(const Geom& g, int k) { return cinv(g.gy_int[k]); }

// C_k(c): coupling between rows k-1 and k (k >= 1), symmetric form; sx = s_x(c).
__device__ __forceinline__ double2 strip_coupling(const Geom& g, double2 sx, int k) {
    return cscale(cmul(sx, g.gy_half[k]), -g.inv_h2);
}

// diagonal and super-diagonal entries of D_k; sx = s_x(c), sy = s_y(k)
__device__ __forceinline__ double2 strip_diag(const Geom& g, const StripDev& st, int k, int c, double2 sx, double2 sy) {
    double2 xs = cadd(strip_ax_half(g, st, c + 1), strip_ax_half(g, st, c));
    double2 ys = cadd(g.gy_half[k + 1], g.gy_half[k]);
    double2 d = cscale(cadd(cmul(sy, xs), cmul(sx, ys)), g.inv_h2);
    double k2 = g.k2[(int64_t)k * g.Nx + strip_k2_col(st, c)];
    d = csub(d, cscale(cmul(sx, sy), k2));
    if (g.rab) {
        // Robin rows (Section 4.4): the ghost value beyond an internal boundary column,
        // eliminated through a u_in + b u_ghost = data, adds (a/b)/h^2 to the diagonal
        if (c == 0 && st.j > 0) d = cadd(d, cscale(cmul(cmul(sx, sy), g.rab[(int64_t)st.j * g.Ny + k]), g.inv_h2));
        if (c == st.W - 1 && st.j < g.J - 1)
            d = cadd(d, cscale(cmul(cmul(sx, sy), g.rab[(int64_t)(st.j + 1) * g.Ny + k]), g.inv_h2));
    }
    return d;
}
__device__ __forceinline__ double2 strip_offdiag(const Geom& g, const StripDev& st, int c, double2 sy) {
    // entry (c, c+1) = (c+1, c)
    return cscale(cmul(sy, strip_ax_half(g, st, c + 1)), -g.inv_h2);
}

// ---- W x W block kernels of a 256-thread CTA, blocks column-major in shared memory.  Thread
// (ti, tj) of 16 x 16 owns entries (ti + 16 i, tj + 16 j), i, j < NI (W <= 16 NI): a product
// reads 2 NI entries per NI^2 multiply-adds (one entry to a thread read 2 per multiply-add and
// was bound by shared memory: 48 x 48 complex64 products 3.4 times the FMA time).
constexpr int kBlockThreads = 256;

// M <- D_k; sx: s_x of the strip's columns (shared memory)
template <typename C>
__device__ void build_diag_block(const Geom& g, const StripDev& st, int k, C* M, const double2* sx) {
    const int W = st.W;
    for (int e = threadIdx.x; e < W * W; e += blockDim.x) M[e] = CT<C>::zero();
    __syncthreads();
    if ((int)threadIdx.x < W) {
        const int c = threadIdx.x;
        const double2 sy = glob_sy(g, k);
        M[c * W + c] = CT<C>::from(strip_diag(g, st, k, c, sx[c], sy));
        if (c + 1 < W) {
            C o = CT<C>::from(strip_offdiag(g, st, c, sy));
            M[(c + 1) * W + c] = o;
            M[c * W + c + 1] = o;
        }
    }
    __syncthreads();
}

// Scratch of block_inverse: two pivot columns, two pairs of rows, the column order.
template <typename C>
struct InvScratch {
    C col[2][64], rowk[2][64], rowp[2][64];
    int dst[64];
};

// In-place Gauss-Jordan inverse with partial (row) pivoting of the W x W matrix A, the entries in
// registers for the whole elimination: the owners of column k publish it, every warp finds the
// pivot row p for itself (largest |entry|^2 at or below row k, the first of equals), the owners
// of rows k and p publish those, and every thread updates its entries (two barriers a step).
// The column order of the inverse is restored as the entries go back.  Returns false
// (uniformly) on a zero or non-finite pivot.
template <typename C, int NI>
__device__ bool block_inverse(C* A, int n, InvScratch<C>& sc) {
    using R = typename CT<C>::R;
    const int tid = threadIdx.x, ti = tid & 15, tj = tid >> 4, lane = tid & 31;
    C a[NI][NI];
#pragma unroll
    for (int j = 0; j < NI; ++j)
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int r = ti + 16 * i, c = tj + 16 * j;
            a[i][j] = (r < n && c < n) ? A[c * n + r] : CT<C>::zero();
        }
    if (tid < 64) sc.dst[tid] = tid;
    bool ok = true;
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
        C* col = sc.col[k & 1];
        C* rk = sc.rowk[k & 1];
        C* rp = sc.rowp[k & 1];
        // entries of a thread at a run-time row or column group, by selects (an indexed register
        // array would go to local memory)
        auto pick_col = [&](int i, int q) -> C {
            C v = a[i][0];
#pragma unroll
            for (int j = 1; j < NI; ++j)
                if (q == j) v = a[i][j];
            return v;
        };
        auto pick_row = [&](int q, int j) -> C {
            C v = a[0][j];
#pragma unroll
            for (int i = 1; i < NI; ++i)
                if (q == i) v = a[i][j];
            return v;
        };
        if (tj == (k & 15)) {
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                const C v = pick_col(i, k >> 4);
                if (ti + 16 * i < n) col[ti + 16 * i] = v;
            }
        }
        __syncthreads();
        R best = (R)-1;
        int p = k;
        for (int i = k + lane; i < n; i += 32) {
            const R v = cabs2(col[i]);
            if (v > best) { best = v; p = i; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const R ov = __shfl_xor_sync(0xffffffffu, best, o);
            const int oi = __shfl_xor_sync(0xffffffffu, p, o);
            if (ov > best || (ov == best && oi < p)) { best = ov; p = oi; }
        }
        if (!(best > (R)0) || !isfinite(best)) { ok = false; break; }   // uniform: every warp sees the same column
        if (tid == 0) {   // dst[c]: the place of column c once the row exchanges are undone on the columns
            const int x = sc.dst[k];
            sc.dst[k] = sc.dst[p];
            sc.dst[p] = x;
        }
        const C inv = cinv(col[p]);
        if (ti == (k & 15)) {
#pragma unroll
            for (int j = 0; j < NI; ++j) {
                const C v = pick_row(k >> 4, j);
                if (tj + 16 * j < n) rk[tj + 16 * j] = v;
            }
        }
        if (ti == (p & 15)) {
#pragma unroll
            for (int j = 0; j < NI; ++j) {
                const C v = pick_row(p >> 4, j);
                if (tj + 16 * j < n) rp[tj + 16 * j] = v;
            }
        }
        __syncthreads();
        C m[NI], t[NI], bk[NI];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int r = imin(ti + 16 * i, n - 1);
            m[i] = r == p ? col[k] : col[r];   // the multipliers after the exchange of rows k and p
        }
#pragma unroll
        for (int j = 0; j < NI; ++j) {
            const int c = imin(tj + 16 * j, n - 1);
            t[j] = c == k ? inv : cmul(rp[c], inv);
            bk[j] = rk[c];
        }
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int r = ti + 16 * i;
#pragma unroll
            for (int j = 0; j < NI; ++j) {
                const int c = tj + 16 * j;
                C base = r == p ? bk[j] : a[i][j];
                if (c == k) base = CT<C>::zero();
                a[i][j] = r == k ? t[j] : csub(base, cmul(m[i], t[j]));
            }
        }
    }
    __syncthreads();
    if (!ok) return false;
#pragma unroll
    for (int j = 0; j < NI; ++j) {
        const int c = tj + 16 * j;
        if (c >= n) continue;
        const int d = sc.dst[c];
#pragma unroll
        for (int i = 0; i < NI; ++i)
            if (ti + 16 * i < n) A[d * n + ti + 16 * i] = a[i][j];
    }
    __syncthreads();
    return true;
}

// Out(r,c) = [Out(r,c) +] sgn * sum_a A(r,a) d(a) B(a,c)   (W x W; d: optional diagonal scaling between
// the factors; Out may alias neither A nor B).
template <typename C, int NI>
__device__ void block_gemm_dscale(C* Out, const C* A, const C* d, const C* B, int n, bool accumulate,
                                  typename CT<C>::R sgn) {
    const int ti = threadIdx.x & 15, tj = threadIdx.x >> 4;
    C acc[NI][NI];
    const C* Ar[NI];
    const C* Bc[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        Ar[i] = A + imin(ti + 16 * i, n - 1);
        Bc[i] = B + imin(tj + 16 * i, n - 1) * n;
#pragma unroll
        for (int j = 0; j < NI; ++j) acc[i][j] = CT<C>::zero();
    }
#pragma unroll 2
    for (int a = 0; a < n; ++a) {
        C x[NI], y[NI];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            x[i] = Ar[i][a * n];
            y[i] = Bc[i][a];
        }
        if (d) {
            const C da = d[a];
#pragma unroll
            for (int j = 0; j < NI; ++j) y[j] = cmul(da, y[j]);
        }
#pragma unroll
        for (int i = 0; i < NI; ++i)
#pragma unroll
            for (int j = 0; j < NI; ++j) acc[i][j] = cfma(x[i], y[j], acc[i][j]);
    }
#pragma unroll
    for (int j = 0; j < NI; ++j)
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int r = ti + 16 * i, c = tj + 16 * j;
            if (r >= n || c >= n) continue;
            const C v = cscale(acc[i][j], sgn);
            Out[c * n + r] = accumulate ? cadd(Out[c * n + r], v) : v;
        }
    __syncthreads();
}

template <typename C>
__device__ void block_copy(C* dst, const C* src, int count) {
    for (int e = threadIdx.x; e < count; e += blockDim.x) dst[e] = src[e];
    __syncthreads();
}

}  // namespace helm
