// Device part of the hierarchy setup: Galerkin coarse operator, reordering of
// each level into its smoothing order, dense inverse of the coarsest matrix
// and the scaled float32 level copies.

#include <algorithm>
#include <numeric>

#include "device.h"

namespace amg {

namespace {

inline int blocks_for(int64_t threads, int block = kBlock) {
    return (int)((threads + block - 1) / block);
}

// ---------------------------------------------------------------------------
// Galerkin product G = P^T A P (Eq. prolongation and the coarse operator that
// follows it).  One warp builds coarse row I: it stages the (J = agg(j), A_ij)
// pairs of the rows i of aggregate I -- members in ascending order, entries
// in row order -- in shared memory, marks the first occurrence of each J,
// and for each distinct J sums its entries left to right in that staged
// order, which is the fine CSR order.  The result is therefore independent
// of the launch configuration and bit-identical to a sequential sum.
// Pass 1 (FILL = false) counts the distinct J of every row; pass 2 writes
// the sorted columns and the sums at the row offsets.
// ---------------------------------------------------------------------------
template <bool FILL>
__global__ void k_galerkin(int nc, const int32_t* __restrict__ mptr, const int32_t* __restrict__ mem,
                           const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                           const double* __restrict__ va, const int32_t* __restrict__ agg, int cap,
                           int32_t* __restrict__ cnt, const int32_t* __restrict__ grp,
                           int32_t* __restrict__ gci, double* __restrict__ gva) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int wpb = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double* sV = reinterpret_cast<double*>(smem) + (size_t)warp * cap;
    int32_t* sJ = reinterpret_cast<int32_t*>(reinterpret_cast<double*>(smem) + (size_t)wpb * cap) +
                  (size_t)warp * cap;
    uint8_t* sF = reinterpret_cast<uint8_t*>(reinterpret_cast<int32_t*>(
                      reinterpret_cast<double*>(smem) + (size_t)wpb * cap) + (size_t)wpb * cap) +
                  (size_t)warp * cap;
    const int I = blockIdx.x * wpb + warp;
    if (I >= nc) return;
    int m = 0;
    for (int t = mptr[I]; t < mptr[I + 1]; ++t) {
        const int i = mem[t];
        const int k0 = rp[i], len = rp[i + 1] - k0;
        for (int q = lane; q < len; q += 32) {
            sJ[m + q] = agg[ci[k0 + q]];
            if (FILL) sV[m + q] = va[k0 + q];
        }
        m += len;
    }
    __syncwarp();
    for (int e = lane; e < m; e += 32) {
        const int J = sJ[e];
        bool first = J >= 0;
        for (int f = 0; f < e && first; ++f)
            if (sJ[f] == J) first = false;
        sF[e] = first ? 1 : 0;
    }
    __syncwarp();
    if (!FILL) {
        int c = 0;
        for (int e = lane; e < m; e += 32) c += sF[e];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
        if (lane == 0) cnt[I] = c;
        return;
    }
    const int base = grp[I];
    for (int e = lane; e < m; e += 32) {
        if (!sF[e]) continue;
        const int J = sJ[e];
        int rank = 0;
        for (int f = 0; f < m; ++f) rank += (sF[f] && sJ[f] < J) ? 1 : 0;
        double s = sV[e];
        for (int f = e + 1; f < m; ++f)
            if (sJ[f] == J) s = s + sV[f];
        gci[base + rank] = J;
        gva[base + rank] = s;
    }
}

// Copy row inv[r] of A into row r of the smoothing-order level: off-diagonal
// entries (in their stored order, columns renumbered by perm) and diagonal.
// With rlow set, the entries towards earlier colours (positions below r: equal
// colours are not coupled) come first, in their stored order, and their number
// goes to rlow.
__global__ void k_reorder_rows(int n, const int32_t* __restrict__ inv, const int32_t* __restrict__ perm,
                               const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                               const double* __restrict__ va, const int32_t* __restrict__ nrp,
                               int32_t* __restrict__ nci, double* __restrict__ nva,
                               double* __restrict__ diag, double* __restrict__ dinv,
                               uint16_t* __restrict__ rlow) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int i = inv[r];
    int low = 0;
    if (rlow) {
        for (int k = rp[i]; k < rp[i + 1]; ++k) low += perm[ci[k]] < r ? 1 : 0;
        rlow[r] = (uint16_t)low;
    }
    int out = nrp[r], up = nrp[r] + low;
    double d = 0.0;
    for (int k = rp[i]; k < rp[i + 1]; ++k) {
        const int j = ci[k];
        if (j == i) {
            d = va[k];
        } else {
            const int pj = perm[j];
            int& at = (rlow && pj > r) ? up : out;
            nci[at] = pj;
            nva[at] = va[k];
            ++at;
        }
    }
    diag[r] = d;
    dinv[r] = 1.0 / d;
}

// Scatter the off-diagonal CSR rows into the SELL-32 arrays; padding entries
// point at the row itself with value 0.  Split rows (rlow set) put their first
// rlow entries into the slots 0, 1, ... and the others into width - 1,
// width - 2, ...
__global__ void k_csr_to_sell(int n, const int32_t* __restrict__ nrp, const int32_t* __restrict__ nci,
                              const double* __restrict__ nva, const uint16_t* __restrict__ rlow,
                              int width, int32_t* __restrict__ scol, double* __restrict__ sval) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int64_t base = (int64_t)(r >> 5) * 32 * width + (r & 31);
    const int k0 = nrp[r], len = nrp[r + 1] - k0;
    const int low = rlow ? (int)rlow[r] : len;
    for (int k = 0; k < width; ++k) {
        const int64_t e = base + 32 * (int64_t)k;
        const int q = k < low ? k : low + (width - 1 - k);   // entry of the row in slot k
        if (q < len) {
            scol[e] = nci[k0 + q];
            sval[e] = nva[k0 + q];
        } else {
            scol[e] = r;
            sval[e] = 0.0;
        }
    }
}

// Copy the sliced arrays (common width W) into the layout with per-slice
// widths: slice s starts at soff[s] and keeps K_s = (soff[s+1] - soff[s]) / 32
// entries a row, slot k of lane i at soff[s] + 32 k + i (padding entries as
// in the common layout: the row itself with value 0); the upper parts of split
// rows (rlow set) move to the end of their slice.  One thread per row.
template <typename T>
__global__ void k_sell_own_width(int n, int width, const uint16_t* __restrict__ rlow,
                                 const int64_t* __restrict__ soff,
                                 const int32_t* __restrict__ scol, const T* __restrict__ sval,
                                 int32_t* __restrict__ ccol, T* __restrict__ cval) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int64_t src = (int64_t)(r >> 5) * 32 * width + (r & 31);
    const int64_t dst = soff[r >> 5] + (r & 31);
    const int ks = (int)((soff[(r >> 5) + 1] - soff[r >> 5]) >> 5);
    const int low = rlow ? (int)rlow[r] : ks;
    for (int k = 0; k < ks; ++k) {
        const int64_t from = src + 32 * (int64_t)(k < low ? k : k + width - ks);
        if (ccol) ccol[dst + 32 * (int64_t)k] = scol[from];
        cval[dst + 32 * (int64_t)k] = sval[from];
    }
}

// ---------------------------------------------------------------------------
// coarsest level: dense Cholesky factor (lower triangle, row-major, in place)
// and the inverse through two triangular solves per unit vector
// ---------------------------------------------------------------------------
__global__ void k_dense_from_csr(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                 const double* __restrict__ va, double* __restrict__ M) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int k = rp[i]; k < rp[i + 1]; ++k) M[(size_t)i * n + ci[k]] = va[k];
}

// ---------------------------------------------------------------------------
// Dense inverse of the coarsest matrix M (n x n, row-major), float64:
// blocked Cholesky M = L L^T in 32-column panels, then Y = L^-1 by blocked
// forward substitution and M^-1 = Y^T Y.  Work is n^3/6 fused multiply-adds
// per phase, almost all of it in 64 x 64 (or 32 x 32) output tiles staged in
// shared memory.  Only the lower triangle of the working matrix W is read.
// ---------------------------------------------------------------------------
constexpr int kPanel = 32;

// Factor the diagonal block W[k0.., k0..] (m <= 32 rows) in shared memory,
// one thread per entry (32 x 32 threads); write L_kk back (upper part zero)
// and D = L_kk^-1 to Dk (32 x 32, row-major).  A pivot <= 0 sets *err and
// continues with 1.
//
// A warp-wide float64 operation takes 64 cycles of a sub-partition whatever
// its active lanes, and a division about twenty of them.  Dividing a column by
// its pivot with one thread in each of the 32 warps took 5 us a column; here
// one thread forms the pivot's square root and reciprocal, and a column is one
// warp's multiplication.  The inverse of 275 rows: 1.96 -> 1.59 ms (0.96 with the
// smaller output tiles, see invert_dense).
__global__ void __launch_bounds__(kPanel * kPanel) k_potrf_block(int n, int k0, double* __restrict__ W,
                                                                 double* __restrict__ Dk,
                                                                 int* __restrict__ err) {
    __shared__ double T[kPanel][kPanel + 1];
    __shared__ double Y[kPanel][kPanel + 1];
    __shared__ double rinv[kPanel];
    const int r = threadIdx.x / kPanel, c = threadIdx.x % kPanel;
    const int m = min(kPanel, n - k0);
    T[r][c] = (r < m && c <= r) ? W[(size_t)(k0 + r) * n + k0 + c] : 0.0;
    Y[r][c] = (r == c && r < m) ? 1.0 : 0.0;
    __syncthreads();
    // right-looking Cholesky: column j (by the first warp, lane = row), then
    // the rank-1 update of the rest
    for (int j = 0; j < m; ++j) {
        if (r == 0) {
            double inv = 0.0;
            if (c == 0) {
                double d = T[j][j];
                if (!(d > 0.0)) {
                    *err = 1;
                    d = 1.0;
                }
                const double root = sqrt(d);
                T[j][j] = root;
                inv = 1.0 / root;
                rinv[j] = inv;
            }
            inv = __shfl_sync(0xffffffffu, inv, 0);
            if (c > j && c < m) T[c][j] *= inv;
        }
        __syncthreads();
        if (r > j && r < m && c > j && c <= r) T[r][c] -= T[r][j] * T[c][j];
        __syncthreads();
    }
    // D = L_kk^-1 by forward elimination on the identity, row j at a time
    for (int j = 0; j < m; ++j) {
        if (r == j && c <= j) Y[j][c] *= rinv[j];
        __syncthreads();
        if (r > j && r < m && c <= j) Y[r][c] -= T[r][j] * Y[j][c];
        __syncthreads();
    }
    if (r < m && c < m) W[(size_t)(k0 + r) * n + k0 + c] = T[r][c];
    Dk[r * kPanel + c] = Y[r][c];
}

// Panel below the diagonal block: W[i, k0:k0+m] <- W[i, k0:k0+m] D^T for
// i >= k0 + m (solves x L_kk^T = a), one warp per row, lane = column.
__global__ void __launch_bounds__(kBlock) k_panel(int n, int k0, int m, double* __restrict__ W,
                                                  const double* __restrict__ Dk) {
    __shared__ double D[kPanel][kPanel + 1];
    const int lane = threadIdx.x & 31;
    for (int t = threadIdx.x; t < kPanel * kPanel; t += blockDim.x)
        D[t / kPanel][t % kPanel] = Dk[t];
    __syncthreads();
    const int i = k0 + m + (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    if (i >= n) return;
    double* row = W + (size_t)i * n + k0;
    const double a = lane < m ? row[lane] : 0.0;
    double out = 0.0;
    for (int t = 0; t < m; ++t) {
        const double at = __shfl_sync(0xffffffffu, a, t);
        if (t <= lane) out = fma(at, D[lane][t], out);
    }
    if (lane < m) row[lane] = out;
}

// Tile index of the lower-triangle tile pair number b: (I, J), I >= J.
__device__ __forceinline__ void tri_pair(int b, int& I, int& J) {
    I = (int)((sqrt(8.0 * (double)b + 1.0) - 1.0) * 0.5);
    while ((I + 1) * (I + 2) / 2 <= b) ++I;
    while (I * (I + 1) / 2 > b) --I;
    J = b - I * (I + 1) / 2;
}

// Trailing update W[i][j] -= sum_t P[i][t] P[j][t] over the lower tiles of
// rows/columns >= r0 (P = the panel W[:, k0:k0+m]); TS x TS tiles, 256
// threads, TS/16 x TS/16 outputs per thread.
template <int TS>
__global__ void __launch_bounds__(256) k_syrk(int n, int r0, int k0, int m, double* __restrict__ W) {
    constexpr int TU = TS / 16;
    __shared__ double Pa[TS][kPanel + 1];
    __shared__ double Pb[TS][kPanel + 1];
    int I, J;
    tri_pair((int)blockIdx.x, I, J);
    const int i0 = r0 + TS * I, j0 = r0 + TS * J;
    for (int t = threadIdx.x; t < TS * kPanel; t += blockDim.x) {
        const int r = t / kPanel, q = t % kPanel;
        Pa[r][q] = (i0 + r < n && q < m) ? W[(size_t)(i0 + r) * n + k0 + q] : 0.0;
        Pb[r][q] = (j0 + r < n && q < m) ? W[(size_t)(j0 + r) * n + k0 + q] : 0.0;
    }
    __syncthreads();
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    double acc[TU][TU] = {};
    for (int q = 0; q < m; ++q) {
        double av[TU], bv[TU];
#pragma unroll
        for (int u = 0; u < TU; ++u) {
            av[u] = Pa[ty * TU + u][q];
            bv[u] = Pb[tx * TU + u][q];
        }
#pragma unroll
        for (int u = 0; u < TU; ++u)
#pragma unroll
            for (int v = 0; v < TU; ++v) acc[u][v] = fma(av[u], bv[v], acc[u][v]);
    }
#pragma unroll
    for (int u = 0; u < TU; ++u)
#pragma unroll
        for (int v = 0; v < TU; ++v) {
            const int i = i0 + ty * TU + u, j = j0 + tx * TU + v;
            if (i < n && j < n && j <= i) W[(size_t)i * n + j] -= acc[u][v];
        }
}

// Y = L^-1, right-looking by 32-row block rows.  Row block j of Y holds
// the running sums S_jc = sum_{c <= t < i} L_jt Y_tc until its turn; then
// Y_jc = -D_j S_jc for c < j and Y_jj = D_j.
//
// Finalise block row i0 (m rows): column tile c = blockIdx.x (c0 <= i0).
// 32 x 32 threads, one output each.
__global__ void __launch_bounds__(kPanel * kPanel) k_trinv_final(int n, int i0, int m,
                                                                 double* __restrict__ Y,
                                                                 const double* __restrict__ Di) {
    __shared__ double D[kPanel][kPanel + 1];
    __shared__ double S[kPanel][kPanel + 1];
    const int r = threadIdx.x / kPanel, c = threadIdx.x % kPanel;
    const int c0 = kPanel * (int)blockIdx.x;
    D[r][c] = Di[r * kPanel + c];
    if (c0 == i0) {
        if (r < m && c0 + c < n) Y[(size_t)(i0 + r) * n + c0 + c] = D[r][c];
        return;
    }
    S[r][c] = (r < m) ? Y[(size_t)(i0 + r) * n + c0 + c] : 0.0;
    __syncthreads();
    if (r >= m) return;
    double out = 0.0;
    for (int q = 0; q <= r; ++q) out = fma(D[r][q], S[q][c], out);
    Y[(size_t)(i0 + r) * n + c0 + c] = -out;
}

// Update after block row i0 is final: S_jc += L_j,i Y_i,c for the block rows
// j > i0 and column tiles c <= i0, TS x TS output tiles of (rows >= i0 + m,
// columns < i0 + m), K = m; 256 threads, TS/16 x TS/16 outputs each.
template <int TS>
__global__ void __launch_bounds__(256) k_trinv_update(int n, int i0, int m, const double* __restrict__ L,
                                                      double* __restrict__ Y) {
    constexpr int TU = TS / 16;
    __shared__ double Pa[TS][kPanel + 1];   // L[j rows, i0 .. i0+m)
    __shared__ double Pb[kPanel][TS + 1];   // Y[i0 .. i0+m, c columns]
    const int r0 = i0 + m, ncol = i0 + m;
    const int tiles_c = (ncol + TS - 1) / TS;
    const int J = (int)blockIdx.x / tiles_c, C = (int)blockIdx.x % tiles_c;
    const int j0 = r0 + TS * J, c0 = TS * C;
    for (int t = threadIdx.x; t < TS * kPanel; t += blockDim.x) {
        const int rr = t / kPanel, q = t % kPanel;
        Pa[rr][q] = (j0 + rr < n && q < m) ? L[(size_t)(j0 + rr) * n + i0 + q] : 0.0;
        const int qq = t / TS, cc = t % TS;
        Pb[qq][cc] = (qq < m && c0 + cc < ncol) ? Y[(size_t)(i0 + qq) * n + c0 + cc] : 0.0;
    }
    __syncthreads();
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    double acc[TU][TU] = {};
    for (int q = 0; q < m; ++q) {
        double av[TU], bv[TU];
#pragma unroll
        for (int u = 0; u < TU; ++u) {
            av[u] = Pa[ty * TU + u][q];
            bv[u] = Pb[q][tx * TU + u];
        }
#pragma unroll
        for (int u = 0; u < TU; ++u)
#pragma unroll
            for (int v = 0; v < TU; ++v) acc[u][v] = fma(av[u], bv[v], acc[u][v]);
    }
#pragma unroll
    for (int u = 0; u < TU; ++u)
#pragma unroll
        for (int v = 0; v < TU; ++v) {
            const int j = j0 + ty * TU + u, cc = c0 + tx * TU + v;
            if (j < n && cc < ncol) Y[(size_t)j * n + cc] += acc[u][v];
        }
}

// X = Y^T Y for the lower tiles (I >= J) of TS x TS, mirrored to the upper
// part: X[i][j] = sum_{k >= TS I} Y[k][i] Y[k][j] (Y is lower triangular).
template <int TS>
__global__ void __launch_bounds__(256) k_yty(int n, const double* __restrict__ Y, double* __restrict__ X) {
    constexpr int TU = TS / 16;
    __shared__ double Ya[kPanel][TS + 1];
    __shared__ double Yb[kPanel][TS + 1];
    int I, J;
    tri_pair((int)blockIdx.x, I, J);
    const int i0 = TS * I, j0 = TS * J;
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    double acc[TU][TU] = {};
    for (int k0 = i0; k0 < n; k0 += kPanel) {
        for (int t = threadIdx.x; t < kPanel * TS; t += blockDim.x) {
            const int kk = t / TS, c = t % TS;
            const bool ok = k0 + kk < n;
            Ya[kk][c] = (ok && i0 + c < n) ? Y[(size_t)(k0 + kk) * n + i0 + c] : 0.0;
            Yb[kk][c] = (ok && j0 + c < n) ? Y[(size_t)(k0 + kk) * n + j0 + c] : 0.0;
        }
        __syncthreads();
        for (int q = 0; q < kPanel; ++q) {
            double av[TU], bv[TU];
#pragma unroll
            for (int u = 0; u < TU; ++u) {
                av[u] = Ya[q][ty * TU + u];
                bv[u] = Yb[q][tx * TU + u];
            }
#pragma unroll
            for (int u = 0; u < TU; ++u)
#pragma unroll
                for (int v = 0; v < TU; ++v) acc[u][v] = fma(av[u], bv[v], acc[u][v]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < TU; ++u)
#pragma unroll
        for (int v = 0; v < TU; ++v) {
            const int i = i0 + ty * TU + u, j = j0 + tx * TU + v;
            if (i < n && j < n && j <= i) {
                X[(size_t)i * n + j] = acc[u][v];
                X[(size_t)j * n + i] = acc[u][v];
            }
        }
}

// Minv_s = S Minv S with S = diag(sqrt(A_ii)): the inverse of S^-1 A S^-1
__global__ void k_scale_inverse(int n, const double* __restrict__ diag, const double* __restrict__ X,
                                double* __restrict__ Xs) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)n * n) return;
    const int i = (int)(t / n), j = (int)(t % n);
    Xs[t] = sqrt(diag[i]) * X[t] * sqrt(diag[j]);
}

// float32 level: A^ = S^-1 A S^-1 (off-diagonal, diagonal and its inverse),
// and the transfer weights t_i = s_i / s_coarse(agg(i)).
__global__ void k_level_fp32(int n, int width, const int32_t* __restrict__ scol,
                             const double* __restrict__ sval, const double* __restrict__ diag,
                             const int32_t* __restrict__ agg, const double* __restrict__ cdiag,
                             float* __restrict__ sval32, float* __restrict__ diag32,
                             float* __restrict__ dinv32, float* __restrict__ t32) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double si = sqrt(diag[i]);
    const int64_t base = (int64_t)(i >> 5) * 32 * width + (i & 31);
    for (int k = 0; k < width; ++k) {
        const int64_t e = base + 32 * (int64_t)k;
        sval32[e] = (float)(sval[e] / (si * sqrt(diag[scol[e]])));
    }
    const double dh = diag[i] / (si * si);
    diag32[i] = (float)dh;
    dinv32[i] = (float)(1.0 / dh);
    if (t32) {
        const int a = agg[i];
        t32[i] = a >= 0 ? (float)(si / sqrt(cdiag[a])) : 0.0f;
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// host-side drivers
// ---------------------------------------------------------------------------

void galerkin_device(const DevCsr& A, const HostCsr& Ah, const AggResult& R, DevArena& arena,
                     DevCsr& Gd, HostCsr& Gh, cudaStream_t s) {
    const int32_t n = Ah.n, nc = R.nc;
    // members of each aggregate in ascending order (counting sort)
    std::vector<int32_t> mptr(nc + 1, 0), mem;
    for (int32_t i = 0; i < n; ++i)
        if (R.agg[i] >= 0) ++mptr[R.agg[i] + 1];
    for (int32_t I = 0; I < nc; ++I) mptr[I + 1] += mptr[I];
    mem.resize(mptr[nc]);
    {
        std::vector<int32_t> fill(mptr.begin(), mptr.end() - 1);
        for (int32_t i = 0; i < n; ++i)
            if (R.agg[i] >= 0) mem[fill[R.agg[i]]++] = i;
    }
    // staging capacity: largest number of fine entries feeding one coarse row
    int64_t cap = 1;
    for (int32_t I = 0; I < nc; ++I) {
        int64_t m = 0;
        for (int32_t t = mptr[I]; t < mptr[I + 1]; ++t) m += Ah.rp[mem[t] + 1] - Ah.rp[mem[t]];
        cap = std::max(cap, m);
    }
    cap = (cap + 15) / 16 * 16;
    const size_t per_warp = (size_t)cap * (sizeof(double) + sizeof(int32_t) + 1);
    const size_t smem_limit = 200 * 1024;
    if (per_warp > smem_limit)
        throw Error{AMG_EINVAL, "Galerkin product: a coarse row gathers " + std::to_string(cap) +
                                    " fine entries, more than the shared-memory staging holds"};
    int wpb = (int)std::max<size_t>(1, std::min<size_t>(8, smem_limit / per_warp));
    const size_t smem = per_warp * wpb;
    if (smem > 40 * 1024) {   // the 48 KB default also holds static shared memory
        raise_dyn_smem(k_galerkin<false>, smem);
        raise_dyn_smem(k_galerkin<true>, smem);
    }
    DevArena tmp(s);
    int32_t* d_agg = tmp.alloc<int32_t>(n);
    int32_t* d_mptr = tmp.alloc<int32_t>(nc + 1);
    int32_t* d_mem = tmp.alloc<int32_t>(mem.size());
    int32_t* d_cnt = tmp.alloc<int32_t>(nc);
    AMG_CUDA_TRY(cudaMemcpyAsync(d_agg, R.agg.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice, s));
    AMG_CUDA_TRY(cudaMemcpyAsync(d_mptr, mptr.data(), sizeof(int32_t) * (nc + 1), cudaMemcpyHostToDevice, s));
    AMG_CUDA_TRY(cudaMemcpyAsync(d_mem, mem.data(), sizeof(int32_t) * mem.size(), cudaMemcpyHostToDevice, s));
    const int grid = (nc + wpb - 1) / wpb;
    k_galerkin<false><<<grid, 32 * wpb, smem, s>>>(nc, d_mptr, d_mem, A.rp, A.ci, A.va, d_agg, (int)cap,
                                                   d_cnt, nullptr, nullptr, nullptr);
    AMG_CUDA_TRY(cudaGetLastError());
    std::vector<int32_t> cnt(nc);
    AMG_CUDA_TRY(cudaMemcpyAsync(cnt.data(), d_cnt, sizeof(int32_t) * nc, cudaMemcpyDeviceToHost, s));
    AMG_CUDA_TRY(cudaStreamSynchronize(s));
    Gh.n = nc;
    Gh.rp.assign(nc + 1, 0);
    for (int32_t I = 0; I < nc; ++I) {
        if ((int64_t)Gh.rp[I] + cnt[I] >= INT32_MAX)
            throw Error{AMG_EINVAL, "coarse matrix exceeds int32 entries"};
        Gh.rp[I + 1] = Gh.rp[I] + cnt[I];
    }
    const int64_t gnnz = Gh.rp[nc];
    Gd.n = nc;
    Gd.nnz = gnnz;
    Gd.rp = arena.alloc<int32_t>(nc + 1);
    Gd.ci = arena.alloc<int32_t>(gnnz);
    Gd.va = arena.alloc<double>(gnnz);
    AMG_CUDA_TRY(cudaMemcpyAsync(Gd.rp, Gh.rp.data(), sizeof(int32_t) * (nc + 1), cudaMemcpyHostToDevice, s));
    k_galerkin<true><<<grid, 32 * wpb, smem, s>>>(nc, d_mptr, d_mem, A.rp, A.ci, A.va, d_agg, (int)cap,
                                                  nullptr, Gd.rp, Gd.ci, Gd.va);
    AMG_CUDA_TRY(cudaGetLastError());
    Gh.ci.resize(gnnz);
    Gh.va.resize(gnnz);
    AMG_CUDA_TRY(cudaMemcpyAsync(Gh.ci.data(), Gd.ci, sizeof(int32_t) * gnnz, cudaMemcpyDeviceToHost, s));
    AMG_CUDA_TRY(cudaMemcpyAsync(Gh.va.data(), Gd.va, sizeof(double) * gnnz, cudaMemcpyDeviceToHost, s));
    AMG_CUDA_TRY(cudaStreamSynchronize(s));
}

void build_level_device(const DevCsr& A, const HostCsr& Ah, const std::vector<int32_t>& perm,
                        bool split, DevArena& arena, DevLevel& L, std::vector<uint16_t>& low,
                        cudaStream_t s) {
    const int32_t n = Ah.n;
    std::vector<int32_t> inv(n), nrp(n + 1, 0);
    std::vector<uint16_t> rlen(n);
    for (int32_t i = 0; i < n; ++i) inv[perm[i]] = i;
    for (int32_t r = 0; r < n; ++r) {
        const int32_t i = inv[r];
        const int32_t len = Ah.rp[i + 1] - Ah.rp[i] - 1;
        if (len > 65535) throw Error{AMG_EINVAL, "a matrix row has more than 65535 off-diagonal entries"};
        rlen[r] = (uint16_t)len;
        nrp[r + 1] = nrp[r] + len;
    }
    const int32_t nslices = (n + 31) / 32;
    int width = 0;
    for (int32_t r = 0; r < n; ++r) width = std::max<int>(width, rlen[r]);
    L.n = n;
    L.nnz_off = nrp[n];
    L.width = width;
    L.sw = 32 * (int64_t)width;
    L.padded = (int64_t)nslices * L.sw;
    // staged blocks cover 8 consecutive slices (256 rows) starting at any
    // slice (colours start anywhere): their tile bounds are maxima over every
    // window of 8 slices
    constexpr int kSlicesPerStage = 8;
    auto window_max = [&](const std::vector<int64_t>& per_slice) {
        int64_t run = 0, best = 0;
        for (int32_t sl = 0; sl < nslices; ++sl) {
            run += per_slice[sl];
            if (sl >= kSlicesPerStage) run -= per_slice[sl - kSlicesPerStage];
            best = std::max(best, run);
        }
        return best;
    };
    // per-slice widths: each slice padded only to its own longest row
    std::vector<int64_t> kmax(nslices, 0), soff(nslices + 1, 0);
    for (int32_t r = 0; r < n; ++r) kmax[r >> 5] = std::max<int64_t>(kmax[r >> 5], rlen[r]);
    for (int32_t sl = 0; sl < nslices; ++sl) soff[sl + 1] = soff[sl] + 32 * kmax[sl];
    // kept where the common width pads more than a tenth over that (the
    // coarse levels; the fine level's rows are nearly all W long)
    const bool compact = width > 0 && 10 * L.padded > 11 * soff[nslices];
    L.stage_cap = compact ? 32 * window_max(kmax) : 256 * (int64_t)width;
    L.rlen = arena.alloc<uint16_t>(n);
    L.split = split;
    L.rlow = split ? arena.alloc<uint16_t>(n) : nullptr;
    L.scol = arena.alloc<int32_t>(L.padded);
    L.sval = arena.alloc<double>(L.padded);
    L.diag = arena.alloc<double>(n);
    L.dinv = arena.alloc<double>(n);
    DevArena tmp(s);
    int32_t* d_inv = tmp.alloc<int32_t>(n);
    int32_t* d_perm = tmp.alloc<int32_t>(n);
    const bool keep_nrp = split && n < kTailMaxRows;
    int32_t* d_nrp = (keep_nrp ? arena : tmp).alloc<int32_t>(n + 1);
    int32_t* d_nci = tmp.alloc<int32_t>(L.nnz_off);
    double* d_nva = tmp.alloc<double>(L.nnz_off);
    AMG_CUDA_TRY(cudaMemcpyAsync(d_inv, inv.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice, s));
    AMG_CUDA_TRY(cudaMemcpyAsync(d_perm, perm.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice, s));
    AMG_CUDA_TRY(cudaMemcpyAsync(d_nrp, nrp.data(), sizeof(int32_t) * (n + 1), cudaMemcpyHostToDevice, s));
    AMG_CUDA_TRY(cudaMemcpyAsync(L.rlen, rlen.data(), sizeof(uint16_t) * n, cudaMemcpyHostToDevice, s));
    k_reorder_rows<<<blocks_for(n), kBlock, 0, s>>>(n, d_inv, d_perm, A.rp, A.ci, A.va, d_nrp, d_nci,
                                                    d_nva, L.diag, L.dinv, L.rlow);
    k_csr_to_sell<<<blocks_for(n), kBlock, 0, s>>>(n, d_nrp, d_nci, d_nva, L.rlow, width, L.scol, L.sval);
    AMG_CUDA_TRY(cudaGetLastError());
    if (compact) {
        const int64_t ce = soff[nslices];
        L.stage_entries = ce;
        L.soff = arena.alloc<int64_t>(nslices + 1);
        L.ccol = arena.alloc<int32_t>(ce);
        L.cval = arena.alloc<double>(ce);
        AMG_CUDA_TRY(cudaMemcpyAsync(L.soff, soff.data(), sizeof(int64_t) * (nslices + 1),
                                     cudaMemcpyHostToDevice, s));
        // rows past n in the last slice: padding entries of no row
        AMG_CUDA_TRY(cudaMemsetAsync(L.ccol, 0, sizeof(int32_t) * ce, s));
        AMG_CUDA_TRY(cudaMemsetAsync(L.cval, 0, sizeof(double) * ce, s));
        k_sell_own_width<double><<<blocks_for(n), kBlock, 0, s>>>(n, width, L.rlow, L.soff, L.scol,
                                                                  L.sval, L.ccol, L.cval);
        AMG_CUDA_TRY(cudaGetLastError());
    }
    // lanes per row: the staged one-row-per-thread kernels on sparse rows
    // (bandwidth bound), several lanes on the denser coarse rows (gather
    // latency bound).  On a split level a pass reads about half a row, and the
    // fewer rows it has, the more its time is one row's chain of loads, sums and
    // instruction fetches, which more lanes shorten; the longer the rows, the
    // further up that holds.  V-cycle from the level in float64, us, by lanes in
    // blocks of 128 (256 with the same lanes: at most 2 % faster, up to 14 % slower):
    //   rows       entries a row     8      4      2      1
    //   8,268          11.4         60     66     74    111
    //   16,187          6.0         57     57     60     74
    //   34,032         15.5        108    118    129    199
    //   49,278         15.6        154    163    171    237
    //   51,932         11.7        144    141    148    189
    //   76,393         14.9        186    180    192    257
    //   105,089         8.6        193    165    164    198
    //   128,547        11.8        222    186    185    220
    //   259,103         7.6        281    249    234    229
    //   269,587        11.9        313    291    269    295
    //   314,662         6.4        307    251    245    227
    //   391,841        11.9        410    355    346    352
    //   612,615        10.9        546    447    422    414
    //   1,661,243      10.9       1168    874    806    754
    //   36,115         29.9        179    229    257    483
    //   70,655         30.3        270    319    348    574
    //   137,869        30.6        374    409    451    727
    //   237,932        30.8        548    538    571    896
    //   463,995        31.0        757    745    723    973
    const double avg = n > 0 ? (double)L.nnz_off / n : 0.0;
    if (split) {
        if (avg > 16.0) L.lpr = n <= 200000 ? 8 : n <= 350000 ? 4 : 2;
        else L.lpr = n <= 50000 ? 8 : n <= 100000 ? 4 : n <= (avg > 8.0 ? 450000 : 250000) ? 2 : 1;
        L.block = 128;
    } else {
        L.lpr = (avg <= 7.0 && staged_fits(L)) ? 0 : avg <= 16.0 ? 4 : 8;
    }
    L.lpr_wide = L.lpr;
    if (keep_nrp) {
        L.nrp = d_nrp;
        L.nrp_host = nrp;
    }
    // entries of each colour's lower parts (the colours' first rows are known
    // to the caller only: it sums low over them)
    if (split) {
        low.resize(n);
        AMG_CUDA_TRY(cudaMemcpyAsync(low.data(), L.rlow, sizeof(uint16_t) * n, cudaMemcpyDeviceToHost, s));
    }
    AMG_CUDA_TRY(cudaStreamSynchronize(s));
}

// Minv = W^-1 for the dense matrix whose lower triangle is W (overwritten)
template <int TS>
static bool invert_dense_tiles(int n, double* W, double* Minv, cudaStream_t s) {
    const int np = (n + kPanel - 1) / kPanel;
    DevArena tmp(s);
    double* Y = tmp.alloc<double>((size_t)n * n);
    double* D = tmp.alloc<double>((size_t)np * kPanel * kPanel);
    int* err = tmp.alloc<int>(1);
    AMG_CUDA_TRY(cudaMemsetAsync(Y, 0, sizeof(double) * (size_t)n * n, s));
    AMG_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), s));
    // Cholesky, right-looking by 32-column panels
    for (int p = 0; p < np; ++p) {
        const int k0 = p * kPanel, m = std::min(kPanel, n - k0), r0 = k0 + m;
        k_potrf_block<<<1, kPanel * kPanel, 0, s>>>(n, k0, W, D + (size_t)p * kPanel * kPanel, err);
        if (r0 < n) {
            k_panel<<<blocks_for((int64_t)(n - r0) * 32), kBlock, 0, s>>>(n, k0, m, W,
                                                                           D + (size_t)p * kPanel * kPanel);
            const int t = (n - r0 + TS - 1) / TS;
            k_syrk<TS><<<t * (t + 1) / 2, 256, 0, s>>>(n, r0, k0, m, W);
        }
    }
    // Y = L^-1 (Y starts at zero: the running sums), then M^-1 = Y^T Y
    for (int p = 0; p < np; ++p) {
        const int i0 = p * kPanel, m = std::min(kPanel, n - i0), r0 = i0 + m;
        k_trinv_final<<<p + 1, kPanel * kPanel, 0, s>>>(n, i0, m, Y, D + (size_t)p * kPanel * kPanel);
        if (r0 < n) {
            const int tiles = ((n - r0 + TS - 1) / TS) * ((r0 + TS - 1) / TS);
            k_trinv_update<TS><<<tiles, 256, 0, s>>>(n, i0, m, W, Y);
        }
    }
    const int t = (n + TS - 1) / TS;
    k_yty<TS><<<t * (t + 1) / 2, 256, 0, s>>>(n, Y, Minv);
    AMG_CUDA_TRY(cudaGetLastError());
    int herr = 0;
    AMG_CUDA_TRY(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    AMG_CUDA_TRY(cudaStreamSynchronize(s));
    return herr == 0;
}

// Output tiles of 64 x 64, or of 32 x 32 where those would leave most SMs idle: a
// tile's float64 work runs at one SM's two multiply-adds a clock, 300 us for the
// last product of a 64 x 64 tile at 275 rows (whose inverse took 1.59 ms, and takes
// 0.96).
static bool invert_dense(int n, double* W, double* Minv, cudaStream_t s) {
    return n < 1024 ? invert_dense_tiles<32>(n, W, Minv, s) : invert_dense_tiles<64>(n, W, Minv, s);
}

bool dense_inverse_device(const DevCsr& A, double* Minv, cudaStream_t s) {
    const int n = A.n;
    DevArena tmp(s);
    double* W = tmp.alloc<double>((size_t)n * n);
    AMG_CUDA_TRY(cudaMemsetAsync(W, 0, sizeof(double) * (size_t)n * n, s));
    k_dense_from_csr<<<blocks_for(n), kBlock, 0, s>>>(n, A.rp, A.ci, A.va, W);
    return invert_dense(n, W, Minv, s);
}

// ---------------------------------------------------------------------------
// the dissected coarsest solve (see DissDesc)
// ---------------------------------------------------------------------------
namespace {

// W rows: segment g of a separator row is sum_l a_il B_k[l][.] over the row's
// entries l in part k.  One block per segment.
__global__ void k_diss_w(const int32_t* __restrict__ gseg, const int32_t* __restrict__ grow,
                         const int32_t* __restrict__ spp, const int32_t* __restrict__ spc,
                         const double* __restrict__ spv, const int64_t* __restrict__ boff,
                         const double* __restrict__ B, double* __restrict__ W) {
    const int g = (int)blockIdx.x;
    const int p0 = gseg[3 * g], len = gseg[3 * g + 1], at = gseg[3 * g + 2], i = grow[g];
    const double* Bk = B + boff[g];
    for (int j = threadIdx.x; j < len; j += blockDim.x) {
        double s = 0.0;
        for (int k = spp[i]; k < spp[i + 1]; ++k) {
            const int l = spc[k] - p0;
            if (l >= 0 && l < len) s = fma(spv[k], Bk[(size_t)l * len + j], s);
        }
        W[(size_t)at + j] = s;
    }
}

// Schur complement, lower triangle: S_ij = A_ij - sum_l W_il a_jl over the
// interior entries l of row j
__global__ void k_diss_schur(int ns, const int32_t* __restrict__ segp, const int32_t* __restrict__ seg,
                             const double* __restrict__ W, const int32_t* __restrict__ spp,
                             const int32_t* __restrict__ spc, const double* __restrict__ spv,
                             double* __restrict__ S) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int i = (int)(t / ns), j = (int)(t % ns);
    if (i >= ns || j > i) return;
    double s = 0.0;
    for (int k = spp[j]; k < spp[j + 1]; ++k) {
        const int l = spc[k];
        for (int g = segp[i]; g < segp[i + 1]; ++g) {
            const int q = l - seg[3 * g];
            if (q >= 0 && q < seg[3 * g + 1]) s = fma(W[(size_t)seg[3 * g + 2] + q], spv[k], s);
        }
    }
    S[(size_t)i * ns + j] -= s;
}

__global__ void k_diss_fill(int m, const int32_t* __restrict__ at_r, const int32_t* __restrict__ at_c,
                            const double* __restrict__ v, int ns, double* __restrict__ S) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < m) S[(size_t)at_r[k] * ns + at_c[k]] = v[k];
}

// scaled copies: entry (r, c) times sqrt(d_r)^pr sqrt(d_c)^pc
__global__ void k_diss_scale_dense(int64_t count, int r0, int len, const double* __restrict__ diag,
                                   const double* __restrict__ in, double* __restrict__ out) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= count) return;
    out[t] = sqrt(diag[r0 + t / len]) * in[t] * sqrt(diag[r0 + t % len]);
}
__global__ void k_diss_scale_w(int nI, const int32_t* __restrict__ gseg, const int32_t* __restrict__ grow,
                               const double* __restrict__ diag, const double* __restrict__ in,
                               double* __restrict__ out) {
    const int g = (int)blockIdx.x;
    const int p0 = gseg[3 * g], len = gseg[3 * g + 1];
    const size_t at = (size_t)gseg[3 * g + 2];
    const double si = sqrt(diag[nI + grow[g]]);
    for (int j = threadIdx.x; j < len; j += blockDim.x) out[at + j] = in[at + j] * sqrt(diag[p0 + j]) / si;
}
__global__ void k_diss_scale_wt(int64_t count, int p0, int m, int nI, const int32_t* __restrict__ adj,
                                const double* __restrict__ diag, const double* __restrict__ in,
                                double* __restrict__ out) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= count) return;
    out[t] = in[t] * sqrt(diag[p0 + t / m]) / sqrt(diag[nI + adj[t % m]]);
}

// W^T of one part: row l over the part's separator rows (j-th: its segment starts at place[j])
__global__ void k_diss_wt(int len, int m, const int32_t* __restrict__ place, const double* __restrict__ W,
                          double* __restrict__ WT) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)len * m) return;
    const int l = (int)(t / m), j = (int)(t % m);
    WT[t] = W[(size_t)place[j] + l];
}

template <typename T>
T* to_device(DevArena& arena, const std::vector<T>& v, cudaStream_t s) {
    T* d = arena.alloc<T>(v.size());
    if (!v.empty())
        AMG_CUDA_TRY(cudaMemcpyAsync(d, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice, s));
    return d;
}

}  // namespace

bool dissect_device(const HostCsr& A, const Dissection& P, DevArena& arena, Dissected& out,
                    cudaStream_t s) {
    const int np = P.parts();
    const int32_t n = A.n, nI = P.ptr[np], ns = n - nI;
    DevArena tmp(s);
    std::vector<int32_t> pos(n), part(n, -1);
    for (int32_t k = 0; k < n; ++k) pos[P.order[k]] = k;
    for (int k = 0; k < np; ++k)
        for (int32_t q = P.ptr[k]; q < P.ptr[k + 1]; ++q) part[P.order[q]] = k;
    // dense inverses of the parts
    std::vector<int64_t> b0(np + 1, 0);
    for (int k = 0; k < np; ++k) {
        const int64_t m = P.ptr[k + 1] - P.ptr[k];
        b0[k + 1] = b0[k] + m * m;
    }
    double* B = arena.alloc<double>((size_t)b0[np]);
    int32_t longest = 1;
    for (int k = 0; k < np; ++k) {
        const int32_t p0 = P.ptr[k], m = P.ptr[k + 1] - p0;
        longest = std::max(longest, m);
        HostCsr sub;
        sub.n = m;
        sub.rp.assign(m + 1, 0);
        for (int32_t q = 0; q < m; ++q) {
            const int32_t i = P.order[p0 + q];
            for (int32_t e = A.rp[i]; e < A.rp[i + 1]; ++e)
                if (part[A.ci[e]] == k) {
                    sub.ci.push_back(pos[A.ci[e]] - p0);
                    sub.va.push_back(A.va[e]);
                }
            sub.rp[q + 1] = (int32_t)sub.ci.size();
        }
        DevArena sm(s);
        DevCsr D;
        D.n = m;
        D.nnz = sub.nnz();
        D.rp = to_device(sm, sub.rp, s);
        D.ci = to_device(sm, sub.ci, s);
        D.va = to_device(sm, sub.va, s);
        if (!dense_inverse_device(D, B + b0[k], s)) return false;   // (waits for the stream)
    }
    // separator rows: interior entries, segments of W, A_SS
    std::vector<int32_t> spp(1, 0), spc, segp(1, 0), seg, grow, ssr, ssc;
    std::vector<int64_t> gb;
    std::vector<double> spv, ssv;
    std::vector<std::vector<int32_t>> adj(np), place(np);   // a part's separator rows, their W segments
    int64_t nW = 0;
    std::vector<char> has(np);
    for (int32_t q = 0; q < ns; ++q) {
        const int32_t i = P.order[nI + q];
        std::fill(has.begin(), has.end(), 0);
        for (int32_t e = A.rp[i]; e < A.rp[i + 1]; ++e) {
            const int32_t j = A.ci[e];
            if (part[j] >= 0) {
                spc.push_back(pos[j]);
                spv.push_back(A.va[e]);
                has[part[j]] = 1;
            } else if (pos[j] - nI <= q) {
                ssr.push_back(q);
                ssc.push_back(pos[j] - nI);
                ssv.push_back(A.va[e]);
            }
        }
        spp.push_back((int32_t)spc.size());
        for (int k = 0; k < np; ++k)
            if (has[k]) {
                const int32_t m = P.ptr[k + 1] - P.ptr[k];
                seg.insert(seg.end(), {P.ptr[k], m, (int32_t)nW});
                grow.push_back(q);
                gb.push_back(b0[k]);
                adj[k].push_back(q);
                place[k].push_back((int32_t)nW);
                nW += m;
            }
        segp.push_back((int32_t)grow.size());
    }
    // blocks of kDissRows rows
    std::vector<int32_t> blk, adj_all, adj_ptr(1, 0);
    std::vector<int64_t> wt0(np, 0);
    int32_t most_adj = 0;
    {
        int64_t at = 0;
        for (int k = 0; k < np; ++k) {
            const int32_t p0 = P.ptr[k], m = P.ptr[k + 1] - p0, na = (int32_t)adj[k].size();
            wt0[k] = at;
            for (int32_t r = 0; r < m; r += kDissRows)
                blk.insert(blk.end(), {p0, m, (int32_t)b0[k], r, (int32_t)adj_all.size(), na, (int32_t)at, 0});
            adj_all.insert(adj_all.end(), adj[k].begin(), adj[k].end());
            adj_ptr.push_back((int32_t)adj_all.size());
            most_adj = std::max(most_adj, na);
            at += (int64_t)m * na;
        }
    }
    const int ng = (int)grow.size();
    int32_t* d_seg = to_device(arena, seg, s);
    int32_t* d_segp = to_device(arena, segp, s);
    int32_t* d_grow = to_device(arena, grow, s);
    int32_t* d_spp = to_device(tmp, spp, s);
    int32_t* d_spc = to_device(tmp, spc, s);
    double* d_spv = to_device(tmp, spv, s);
    int64_t* d_gb = to_device(tmp, gb, s);
    double* W = arena.alloc<double>((size_t)nW);
    double* WT = arena.alloc<double>((size_t)nW);
    double* S = arena.alloc<double>((size_t)ns * ns);
    if (ng > 0) {
        k_diss_w<<<ng, 128, 0, s>>>(d_seg, d_grow, d_spp, d_spc, d_spv, d_gb, B, W);
        for (int k = 0; k < np; ++k) {
            const int len = P.ptr[k + 1] - P.ptr[k], m = (int)adj[k].size();
            if (m > 0)
                k_diss_wt<<<blocks_for((int64_t)len * m), kBlock, 0, s>>>(len, m, to_device(tmp, place[k], s),
                                                                          W, WT + wt0[k]);
        }
        AMG_CUDA_TRY(cudaGetLastError());
    }
    bool ok = true;
    if (ns > 0) {
        double* M = tmp.alloc<double>((size_t)ns * ns);
        AMG_CUDA_TRY(cudaMemsetAsync(M, 0, sizeof(double) * (size_t)ns * ns, s));
        k_diss_fill<<<blocks_for((int64_t)ssr.size()), kBlock, 0, s>>>(
            (int)ssr.size(), to_device(tmp, ssr, s), to_device(tmp, ssc, s), to_device(tmp, ssv, s), ns, M);
        k_diss_schur<<<blocks_for((int64_t)ns * ns), kBlock, 0, s>>>(ns, d_segp, d_seg, W, d_spp, d_spc,
                                                                     d_spv, M);
        AMG_CUDA_TRY(cudaGetLastError());
        ok = invert_dense(ns, M, S, s);
    }
    DissDesc& d = out.host[0];
    d.nI = nI;
    d.ns = ns;
    d.nblk = (int32_t)(blk.size() / kDissBlk);
    d.longest = longest;
    d.most_adj = most_adj;
    d.segp = d_segp;
    d.seg = d_seg;
    d.W = W;
    d.S = S;
    d.blk = to_device(arena, blk, s);
    d.adj = to_device(arena, adj_all, s);
    d.B = B;
    d.WT = WT;
    d.y = arena.alloc<double>(nI);
    d.t = arena.alloc<double>(ns);
    d.xs = arena.alloc<double>(ns);
    DissDesc* dev = arena.alloc<DissDesc>(1);
    AMG_CUDA_TRY(cudaMemcpyAsync(dev, &d, sizeof(DissDesc), cudaMemcpyHostToDevice, s));
    out.desc[0] = dev;
    out.grow = d_grow;
    out.part_ptr = P.ptr;
    out.nW = nW;
    out.nB = b0[np];
    out.n_seg = ng;
    out.adj_ptr = adj_ptr;
    out.entries = 2 * nW + b0[np] + (int64_t)ns * ns;
    out.on = true;
    AMG_CUDA_TRY(cudaStreamSynchronize(s));
    return ok;
}

void dissect_scaled(Dissected& o, const double* diag, DevArena& arena, cudaStream_t s) {
    DissDesc& d = o.host[1];
    d = o.host[0];
    double* W = arena.alloc<double>((size_t)o.nW);
    double* S = arena.alloc<double>((size_t)d.ns * d.ns);
    double* B = arena.alloc<double>((size_t)o.nB);
    double* WT = arena.alloc<double>((size_t)o.nW);
    if (o.n_seg > 0) k_diss_scale_w<<<o.n_seg, 128, 0, s>>>(d.nI, d.seg, o.grow, diag, d.W, W);
    if (d.ns > 0) {
        const int64_t m = (int64_t)d.ns * d.ns;
        k_diss_scale_dense<<<blocks_for(m), kBlock, 0, s>>>(m, d.nI, d.ns, diag, d.S, S);
    }
    int64_t at = 0, wt = 0;
    for (size_t k = 0; k + 1 < o.part_ptr.size(); ++k) {
        const int len = o.part_ptr[k + 1] - o.part_ptr[k], na = o.adj_ptr[k + 1] - o.adj_ptr[k];
        const int64_t m = (int64_t)len * len, w = (int64_t)len * na;
        k_diss_scale_dense<<<blocks_for(m), kBlock, 0, s>>>(m, o.part_ptr[k], len, diag, d.B + at, B + at);
        if (w > 0)
            k_diss_scale_wt<<<blocks_for(w), kBlock, 0, s>>>(w, o.part_ptr[k], na, d.nI, d.adj + o.adj_ptr[k],
                                                             diag, d.WT + wt, WT + wt);
        at += m;
        wt += w;
    }
    AMG_CUDA_TRY(cudaGetLastError());
    d.W = W;
    d.S = S;
    d.B = B;
    d.WT = WT;
    DissDesc* dev = arena.alloc<DissDesc>(1);
    AMG_CUDA_TRY(cudaMemcpyAsync(dev, &d, sizeof(DissDesc), cudaMemcpyHostToDevice, s));
    o.desc[1] = dev;
}

__global__ void k_to_float_padded(int n, int ld, const double* __restrict__ in, float* __restrict__ out) {
    const size_t count = (size_t)n * ld;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < count;
         t += (size_t)gridDim.x * blockDim.x) {
        const size_t i = t / ld, j = t % ld;
        out[t] = j < (size_t)n ? (float)in[i * n + j] : 0.f;
    }
}

void to_float_padded_device(int n, int ld, const double* in, float* out, cudaStream_t s) {
    const int64_t count = (int64_t)n * ld;
    k_to_float_padded<<<std::max(1, (int)std::min<int64_t>(blocks_for(count), 1216 * 4)), kBlock, 0, s>>>(
        n, ld, in, out);
    AMG_CUDA_TRY(cudaGetLastError());
}

void scale_inverse_device(int n, const double* diag, const double* Minv, double* Minv_s,
                          cudaStream_t s) {
    k_scale_inverse<<<blocks_for((int64_t)n * n), kBlock, 0, s>>>(n, diag, Minv, Minv_s);
    AMG_CUDA_TRY(cudaGetLastError());
}

void build_level_fp32(DevLevel& L, const double* coarse_diag, DevArena& arena, cudaStream_t s) {
    const int n = L.n;
    L.sval32 = arena.alloc<float>(L.padded);
    L.diag32 = arena.alloc<float>(n);
    L.dinv32 = arena.alloc<float>(n);
    L.t32 = coarse_diag ? arena.alloc<float>(n) : nullptr;
    L.x32 = arena.alloc<float>(n);
    L.b32 = arena.alloc<float>(n);
    L.r32 = arena.alloc<float>(n);
    k_level_fp32<<<blocks_for(n), kBlock, 0, s>>>(n, L.width, L.scol, L.sval, L.diag, L.agg, coarse_diag,
                                                  L.sval32, L.diag32, L.dinv32, L.t32);
    AMG_CUDA_TRY(cudaGetLastError());
    if (L.soff) {
        const int64_t ce = L.stage_entries;
        L.cval32 = arena.alloc<float>(ce);
        AMG_CUDA_TRY(cudaMemsetAsync(L.cval32, 0, sizeof(float) * ce, s));
        k_sell_own_width<float><<<blocks_for(n), kBlock, 0, s>>>(n, L.width, L.rlow, L.soff, nullptr,
                                                                  L.sval32, nullptr, L.cval32);
        AMG_CUDA_TRY(cudaGetLastError());
    }
}

}  // namespace amg
