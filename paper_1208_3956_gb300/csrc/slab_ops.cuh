// Entries of the 3-D strip blocks (see slab3d.cu for the ordering and the formulas) and the
// assembly of a block before its inversion, shared by the SIMT (slab3d.cu) and tensor-core
// (slab_tc.cu) factorisations.
#pragma once

#include "strip_ops.cuh"

namespace helm {

__device__ __forceinline__ double2 slab_sz(const Geom& g, int z) { return cinv(g.gz_int[z]); }

__device__ inline double2 slab_diag(const Geom& g, const StripDev& st, int k, int c, int z) {
    const double2 sx = strip_sx(g, st, c), sy = glob_sy(g, k), sz = slab_sz(g, z);
    const double2 xs = cadd(strip_ax_half(g, st, c + 1), strip_ax_half(g, st, c));
    const double2 ys = cadd(g.gy_half[k + 1], g.gy_half[k]);
    const double2 zs = cadd(g.gz_half[z + 1], g.gz_half[z]);
    double2 d = cadd(cadd(cmul(cmul(sy, sz), xs), cmul(cmul(sx, sz), ys)), cmul(cmul(sx, sy), zs));
    d = cscale(d, g.inv_h2);
    const double k2 = g.k2[((int64_t)z * g.Ny + k) * g.Nx + strip_k2_col(st, c)];
    return csub(d, cscale(cmul(cmul(sx, sy), sz), k2));
}
// entry (e, e+1), e = z W + c, c + 1 < W
__device__ inline double2 slab_xoff(const Geom& g, const StripDev& st, int k, int c, int z) {
    return cscale(cmul(cmul(glob_sy(g, k), slab_sz(g, z)), strip_ax_half(g, st, c + 1)), -g.inv_h2);
}
// entry (e, e+W), z + 1 < N_z
__device__ inline double2 slab_zoff(const Geom& g, const StripDev& st, int k, int c, int z) {
    return cscale(cmul(cmul(strip_sx(g, st, c), glob_sy(g, k)), g.gz_half[z + 1]), -g.inv_h2);
}
// D_k(r, a) for any pair (zero off the stencil)
__device__ inline double2 slab_dentry(const Geom& g, const StripDev& st, int k, int r, int a) {
    const int W = st.W;
    const int lo = imin(r, a), d = r > a ? r - a : a - r;
    if (d != 0 && d != 1 && d != W) return make_double2(0.0, 0.0);
    const int c = lo % W, z = lo / W;
    if (d == 0) return slab_diag(g, st, k, c, z);
    if (d == 1 && c + 1 < W) return slab_xoff(g, st, k, c, z);
    if (d == W) return slab_zoff(g, st, k, c, z);
    return make_double2(0.0, 0.0);
}

// Layout of a stored block X (n x n): 64-row tiles, each column after column with its 64 rows
// contiguous, so that any column range of a tile is one contiguous piece (a bulk copy) and
// the lanes of a warp read adjacent rows.  slab_block_elems(n) elements per block.
__host__ __device__ __forceinline__ int64_t slab_block_elems(int n) { return (int64_t)((n + 63) / 64) * 64 * n; }
__device__ __forceinline__ int64_t slab_at(int n, int r, int c) { return ((int64_t)(r >> 6) * n + c) * 64 + (r & 63); }

// M (column-major, ldm) = - C_k Xp C_k - C_{k+1} Xn C_{k+1}, Xp / Xn in the tile layout or null.
// CTA (x, y): rows 64 x .., columns 4 y .., 256 threads.
template <typename C>
__device__ __forceinline__ void slab_build_entries(const Geom& g, const StripDev& st, int k, const C* __restrict__ Xp,
                                                   const C* __restrict__ Xn, C* __restrict__ M, int ldm) {
    const int n = st.W * g.Nz;
    const int r = blockIdx.x * 64 + (threadIdx.x & 63), a = blockIdx.y * 4 + (threadIdx.x >> 6);
    if (r >= n || a >= n) return;
    // C_k(e) = s_x(c) s_z(z) (-alpha_y(y_{k-1/2}) / h^2) from the working-precision table
    const C* ct = reinterpret_cast<const C*>(g.ct);
    const C sr = cmul(ct[st.ctab + r % st.W], ct[g.ct_sz + r / st.W]);
    const C sa = cmul(ct[st.ctab + a % st.W], ct[g.ct_sz + a / st.W]);
    C acc = CT<C>::zero();
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const C* X = side == 0 ? Xp : Xn;
        if (!X) continue;   // uniform
        const C cy = ct[g.ct_cy + k + side];
        acc = csub(acc, cmul(cmul(cmul(sr, cy), X[slab_at(n, r, a)]), cmul(sa, cy)));
    }
    M[(int64_t)a * ldm + r] = acc;
}

// M(r, a) += D_k(r, a) on the stencil entries of row r: a = r, r +- 1 (same z), r +- W; one
// entry per thread (the entries are evaluated in FP64, so they are spread over the GPU).
template <typename C>
__device__ __forceinline__ void slab_dadd_entries(const Geom& g, const StripDev& st, int k, C* __restrict__ M,
                                                  int ldm) {
    const int n = st.W * g.Nz, W = st.W;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < 5 * n; e += gridDim.x * blockDim.x) {
        const int r = e / 5, i = e % 5, c = r % W;
        const int a = i == 0 ? r : i == 1 ? (c > 0 ? r - 1 : -1) : i == 2 ? (c + 1 < W ? r + 1 : -1) : i == 3 ? r - W : r + W;
        if (a < 0 || a >= n) continue;
        C* p = M + (int64_t)a * ldm + r;
        *p = cadd(*p, CT<C>::from(slab_dentry(g, st, k, r, a)));
    }
}

}  // namespace helm
