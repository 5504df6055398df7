// AFT (Eq. 20, 21, 15, 16), structured Jacobian products (Eq. 22, 23), the dense
// outer Newton solve and the Lyapunov exponents (App. F).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <string>
#include <vector>

#include "fse_common.cuh"

namespace fse {

// ----------------------------------------------------------------------------
// AFT: i-DFT (Eq. 20) and DFT + rotation + residual (Eq. 21, 15, 16)
// ----------------------------------------------------------------------------

__global__ void k_idft(int N, int U, int n2, const double* __restrict__ G,
                       const double* __restrict__ Z, double* zb) {
    const int s = blockIdx.y;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += gridDim.x * blockDim.x) {
        double acc = 0.0;
        for (int c = 0; c < U; ++c) acc += G[(size_t)s * U + c] * Z[(size_t)i * U + c];
        zb[(size_t)s * n2 + i] = acc;
    }
}

// q, u (internal numbering) -> end points (N x 2n, the caller's dof order)
__global__ void k_join(int N, int n, int ni, const int* __restrict__ row_of, const double* __restrict__ q,
                       const double* __restrict__ u, double* zb) {
    const size_t total = (size_t)N * n;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t s = idx / n, i = idx % n;
        const size_t r = s * ni + row_of[i];
        zb[s * 2 * n + i] = q[r];
        zb[s * 2 * n + n + i] = u[r];
    }
}

// out[i*U + c] = sum_s RG[c][s] zb[s][i] - (subtract ? Z0[i*U + c] : 0), in two forms (the launcher chooses).
// FP64 work bounds large ones (N U 2n multiply-adds: 15 M for the 1872-dof shell, 24 us), the chain of one
// sum and the launch the small ones, so the samples of a sum are always dealt out.
//
// W warps share 32 states i and one coefficient c: lanes along i (zb coalesced, RG a broadcast), each warp a
// slice of the samples, partial sums through shared memory; the loads of four samples go out together (one
// by one a slice of 25 is a chain of 13 trips to L2: 10.8 us at 24 states, 196 x 169, now 6.5).  Against one
// warp per output with its lanes over the samples (zb with a stride of 2n): 447-dof beam (64 samples x 63)
// 30.7 -> 10.2 us, 243-dof plate (256 x 225) 90 -> 54, 72-dof plate (81 x 81) 10.7 -> 5.3.
template <int W>
__global__ void __launch_bounds__(32 * W) k_dft_warps(int N, int U, int n2, const double* __restrict__ RG,
                                                      const double* __restrict__ zb, const double* __restrict__ Z0,
                                                      double* out, int subtract) {
    __shared__ double part[W][32];
    const int tiles = (n2 + 31) / 32, c = blockIdx.x / tiles;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, i = (blockIdx.x % tiles) * 32 + lane;
    const int per = (N + W - 1) / W, s0 = warp * per, s1 = min(N, s0 + per);
    double a = 0.0, b = 0.0;
    if (i < n2) {
        const double *z = zb + i, *r = RG + (size_t)c * N;
        int s = s0;
#pragma unroll 2
        for (; s + 4 <= s1; s += 4) {   // four samples' loads at a time
            double zv[4], rv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                zv[q] = z[(size_t)(s + q) * n2];
                rv[q] = r[s + q];
            }
            a += rv[0] * zv[0];
            b += rv[1] * zv[1];
            a += rv[2] * zv[2];
            b += rv[3] * zv[3];
        }
        for (; s < s1; ++s) a += r[s] * z[(size_t)s * n2];
    }
    part[warp][lane] = a + b;
    __syncthreads();
    if (warp == 0 && i < n2) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < W; ++w) t += part[w][lane];
        const size_t o = (size_t)i * U + c;
        out[o] = t - (subtract ? Z0[o] : 0.0);
    }
}

// one warp per output, lanes over the samples: for few states, where most lanes of the form above would be
// idle (4 states, 1024 samples x 961 coefficients: 11 us against 60)
__global__ void __launch_bounds__(256) k_dft_lanes(int N, int U, int n2, const double* __restrict__ RG,
                                                   const double* __restrict__ zb, const double* __restrict__ Z0,
                                                   double* out, int subtract) {
    const int warp = (blockIdx.x * 256 + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= n2 * U) return;
    const int i = warp / U, c = warp % U;
    double acc = 0.0;
    for (int s = lane; s < N; s += 32) acc += RG[(size_t)c * N + s] * zb[(size_t)s * n2 + i];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) out[warp] = acc - (subtract ? Z0[warp] : 0.0);
}

// ----------------------------------------------------------------------------
// Jacobian products (Eq. 22, 23) from the stored tangents
// ----------------------------------------------------------------------------

// 4 values as FP64.  FP32 -> FP64 conversions run at the FP64 rate (GB300: 2 a clock and SM), as dear as
// the multiply-add that follows; moving the bits with integer instructions is exact for normal values.
// Zeros (far entries of narrow bands, most of a chain's after few steps) are selected in a branch of their
// own, since the selects cost dense tangents 2.5 %; the conversion is kept for a vector that holds a
// subnormal, an infinity or a NaN.
__device__ __forceinline__ double widen(unsigned b) {
    return __hiloint2double((((int)b >> 3) & 0x8fffffff) + 0x38000000, (int)(b << 29));
}
__device__ __forceinline__ void ld4_fp64(const float* p, double v[4]) {
    const float4 f = *reinterpret_cast<const float4*>(p);
    const unsigned b[4] = {__float_as_uint(f.x), __float_as_uint(f.y), __float_as_uint(f.z), __float_as_uint(f.w)};
    bool normal = true, plain = true;   // plain: normal or zero
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const bool nk = ((b[k] + 0x00800000u) & 0x7fffffffu) > 0x00ffffffu;
        normal = normal && nk;
        plain = plain && (nk || (b[k] & 0x7fffffffu) == 0);
    }
    if (normal) {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = widen(b[k]);
    } else if (plain) {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = (b[k] & 0x7fffffffu) ? widen(b[k]) : 0.0;
    } else {
        v[0] = f.x;
        v[1] = f.y;
        v[2] = f.z;
        v[3] = f.w;
    }
}

// zout[s][i] = sum_{j < 2n} Phi_s[i][j] zin[s][j], in two forms (launch_phi_apply chooses).
//
// G lanes take one row of X or V (B = 1), or both rows of a dof, which share each z (B = 2); z comes from
// global memory, in the panel's column order through orig_of where there are panels.  FP64 multiply-adds
// bound large ones (447-dof beam, 64 trajectories: 51 M = 81 us, 107 measured), the length of a lane's chain and
// the launch small ones: 72 dofs, 64 trajectories, FP64: 7.4 us with 32 lanes a row, 5.3 with 16, 12.5 with
// a staged z as below.
template <typename T, int G, int B>
__global__ void __launch_bounds__(256) k_phi_rows(int N, PhiView<T> F, const double* __restrict__ zin, double* zout) {
    const int n = F.n, per = B == 2 ? n : 2 * n, total = N * per;
    const int gid = (int)(((size_t)blockIdx.x * 256 + threadIdx.x) / G), l = threadIdx.x % G;
    const int id = min(gid, total - 1);   // lanes past the last row repeat it: all take part in the shuffles
    const int s = id / per, i = id % per, dof = i < n ? i : i - n;
    const double* z = zin + (size_t)s * 2 * n;
    const T* first = (B == 2 || i < n) ? F.X : F.V;
    double a = 0.0, b = 0.0;
    if (F.pan.nc == 1) {   // the caller's numbering
        const size_t o = (size_t)s * F.pan.tot + (size_t)dof * F.pan.ld[0];
        const T *x = first + o, *v = F.V + o;
        for (int j = l; j < 2 * n; j += G) {
            const double zj = z[j];
            a += (double)x[j] * zj;
            if (B == 2) b += (double)v[j] * zj;
        }
    } else {
        const int r = F.row_of[dof], g = F.panel(r), m = F.pan.n[g], row0 = F.pan.row0[g];
        const size_t o = (size_t)s * F.pan.tot + F.pan.off[g] + (size_t)(r - row0) * F.pan.ld[g];
        const T *x = first + o, *v = F.V + o;
        for (int j = l; j < 2 * m; j += G) {
            const double zj = z[F.col(g, j)];
            a += (double)x[j] * zj;
            if (B == 2) b += (double)v[j] * zj;
        }
    }
    if (B == 2) {   // halves of the group keep one sum each
        const bool up = l & (G / 2);
        const double other = __shfl_xor_sync(0xffffffffu, up ? a : b, G / 2);
        a = (up ? b : a) + other;
    }
#pragma unroll
    for (int o = G / 2 / B; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (gid < total && l % (G / B) == 0) zout[(size_t)s * 2 * n + i + (l ? n : 0)] = a;
}

// FP32 tangents of some size: a conversion at the FP64 rate for every multiply-add doubles the work, so
// values are widened by bit moves, and four dot products share each z.  A CTA takes PHI_ROWS rows of one
// panel of one trajectory: the panel's part of zin goes to shared memory in the panel's column order, a warp
// takes the X and V rows of two dofs.  Bound by the FP64 FMAs (349 M for the 1872-dof shell's 64
// trajectories = 0.55 ms) or by reading the tangents.  Converting loads and a warp per row: 1.28 ms there,
// 0.65 ms this way; 243-dof plate, 256 trajectories, 484 -> 143 us.
constexpr int PHI_ROWS = 16;
__global__ void __launch_bounds__(256) k_phi_apply(PhiView<float> F, const double* __restrict__ zin, double* zout) {
    extern __shared__ double zs[];
    int x = blockIdx.x, g = 0;
    while (x >= (F.pan.n[g] + PHI_ROWS - 1) / PHI_ROWS) x -= (F.pan.n[g++] + PHI_ROWS - 1) / PHI_ROWS;
    const int s = blockIdx.y, n = F.n, m = F.pan.n[g], ld = F.pan.ld[g], row0 = F.pan.row0[g];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double* z = zin + (size_t)s * 2 * n;
    for (int k = threadIdx.x; k < m; k += 256) {
        const int j = F.orig_of[row0 + k];
        zs[k] = z[j];
        zs[m + k] = z[n + j];
    }
    __syncthreads();
    const int ra = x * PHI_ROWS + 2 * warp, rb = ra + 1;
    if (ra >= m) return;
    const size_t base = (size_t)s * F.pan.tot + F.pan.off[g];
    const size_t oa = base + (size_t)ra * ld, ob = rb < m ? oa + ld : oa;
    const float* rows[4] = {F.X + oa, F.V + oa, F.X + ob, F.V + ob};
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const int m4 = (2 * m) & ~3;
    for (int j = 4 * lane; j < m4; j += 128) {
        double zv[4], v[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) ld4_fp64(rows[q] + j, v[q]);
#pragma unroll
        for (int k = 0; k < 4; ++k) zv[k] = zs[j + k];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[q] += v[q][k] * zv[k];
    }
    for (int j = m4 + lane; j < 2 * m; j += 32)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] += (double)rows[q][j] * zs[j];
    // sums over the lanes, six FP64 additions instead of 20: halves of the warp keep two sums each, then
    // quarters one, so that lanes 8 q .. 8 q + 7 end with sum q
    const bool up = lane & 16, up2 = lane & 8;
    double k0 = up ? acc[2] : acc[0], k1 = up ? acc[3] : acc[1];
    k0 += __shfl_xor_sync(0xffffffffu, up ? acc[0] : acc[2], 16);
    k1 += __shfl_xor_sync(0xffffffffu, up ? acc[1] : acc[3], 16);
    double t = up2 ? k1 : k0;
    t += __shfl_xor_sync(0xffffffffu, up2 ? k0 : k1, 8);
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((lane & 7) == 0) {
        const int q = lane >> 3, r = q < 2 ? ra : rb;   // X and V row of ra, of rb
        if (r < m) zout[(size_t)s * 2 * n + (q & 1) * n + F.orig_of[row0 + r]] = t;
    }
}

template <typename T>
__global__ void k_domega_col(int N, PhiView<T> F, double* zout) {
    const int n2 = 2 * F.n;
    const size_t total = (size_t)N * n2;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        int g;
        const T* row = F.row((int)(idx / n2), (int)(idx % n2), g);
        zout[idx] = (double)row[2 * F.pan.n[g]];
    }
}

// Phi_s and d zbar_s / d w_1 of trajectories s0 .. s0 + N - 1
template <typename T>
__global__ void k_phi_copy(int N, int s0, PhiView<T> F, double* Phi, double* dzdw) {
    const int n2 = 2 * F.n;
    const size_t total = (size_t)N * n2 * n2;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t s = idx / ((size_t)n2 * n2);
        const int r = (int)((idx / n2) % n2), c = (int)(idx % n2);
        if (Phi) Phi[idx] = F.at(s0 + (int)s, r, c);
        if (dzdw && c == 0) {
            int g;
            const T* row = F.row(s0 + (int)s, r, g);
            dzdw[s * n2 + r] = (double)row[2 * F.pan.n[g]];
        }
    }
}

// dense Eq. (22): J[(i,u),(j,v)] = sum_s RG[u][s] Phi_s[i][j] G[s][v] - delta
template <typename T>
__global__ void k_dense_jac(int N, int U, PhiView<T> F, const double* RG, const double* G, double* J, size_t lda) {
    const int n2 = 2 * F.n;
    const size_t m = (size_t)n2 * U;
    const size_t total = m * m;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t row = idx / m, col = idx % m;
        const int i = (int)(row / U), uu = (int)(row % U);
        const int j = (int)(col / U), vv = (int)(col % U);
        double acc = 0.0;
        for (int s = 0; s < N; ++s) acc += RG[(size_t)uu * N + s] * F.at(s, i, j) * G[(size_t)s * U + vv];
        J[row * lda + col] = acc - (row == col ? 1.0 : 0.0);
    }
}

// hyper-time form (Sec. 3.4, Eq. FSES_T): Pm = Gamma R(rho) Gamma^-1 (N x N), Pm[s][t] =
// sum_c G[s][c] RG[c][t]
__global__ void k_pmat(int N, int U, const double* __restrict__ G, const double* __restrict__ RG, double* Pm) {
    const size_t total = (size_t)N * N;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t s = idx / N, t = idx % N;
        double acc = 0.0;
        for (int c = 0; c < U; ++c) acc += G[s * U + c] * RG[(size_t)c * N + t];
        Pm[idx] = acc;
    }
}

// dense Jacobian of Eq. FSES_T: J[(s,i),(t,j)] = Pm[s][t] Phi_t[i][j] - delta (unknowns sample-major)
template <typename T>
__global__ void k_dense_jac_ht(int N, PhiView<T> F, const double* Pm, double* J) {
    const int n2 = 2 * F.n;
    const size_t m = (size_t)N * n2;
    const size_t total = m * m;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
         idx += (size_t)gridDim.x * blockDim.x) {
        const size_t row = idx / m, col = idx % m;
        const int s = (int)(row / n2), i = (int)(row % n2);
        const int t = (int)(col / n2), j = (int)(col % n2);
        J[idx] = Pm[(size_t)s * N + t] * F.at(t, i, j) - (row == col ? 1.0 : 0.0);
    }
}

// border of the pseudo-arclength system: column m = dR/dw_1, row m = (t_Z, tail)
__global__ void k_border(size_t m, const double* __restrict__ Rw, const double* __restrict__ tZ, double tail,
                         double* B) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i <= m; i += (size_t)gridDim.x * blockDim.x) {
        if (i < m) {
            B[i * (m + 1) + m] = Rw[i];
            B[m * (m + 1) + i] = tZ[i];
        } else {
            B[m * (m + 1) + m] = tail;
        }
    }
}

// Unknown base frequency w_{j+2} (Sec. 3.2, Eq. 18, 19, 23, 24), one harmonic row l of the table
// (column j: k = k~_lj) acting on each (cos, sin) coefficient pair (a, b) of the 2n states:
//   col = dR/dw_{j+2} = (2 pi / w_1) (I (x) Upsilon_j) (R + Z0), Upsilon: (a, b) -> (-k b, k a)
//         ((I (x) R(rho)) Z(2 pi) = R + Z0; the trajectories do not move with an unforced w_i);
//   row = (I (x) grad_j) Z0,                         grad:    (a, b) -> (k b, -k a)
// (the phase condition of Eq. 18 on the Newton correction).  The constant coefficient gives 0.
__global__ void k_unknown_border(size_t m, int U, int dm1, int j, const int* __restrict__ ktab, double scale,
                                 const double* __restrict__ R, const double* __restrict__ Z0, double* col,
                                 double* row) {
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < m; idx += (size_t)gridDim.x * blockDim.x) {
        const size_t i = idx / U;
        const int c = (int)(idx % U);
        if (c == 0) {
            col[idx] = 0.0;
            row[idx] = 0.0;
            continue;
        }
        const int l = (c - 1) >> 1;
        const double k = (double)ktab[l * dm1 + j];
        const size_t ci = i * U + 1 + 2 * l, si = ci + 1;
        if (((c - 1) & 1) == 0) {   // cos coefficient
            col[idx] = -scale * k * (R[si] + Z0[si]);
            row[idx] = k * Z0[si];
        } else {                    // sin coefficient
            col[idx] = scale * k * (R[ci] + Z0[ci]);
            row[idx] = -k * Z0[ci];
        }
    }
}

// border of a bordered m x m matrix with u extra columns / rows (lda = m + u): B[i][m + a] =
// cols[a][i], B[m + a][i] = rows[a][i], B[m + a][m + b] = 0
__global__ void k_border_multi(size_t m, int u, const double* __restrict__ cols, const double* __restrict__ rows,
                               double* B) {
    const size_t lda = m + u;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < m + u; i += (size_t)gridDim.x * blockDim.x)
        for (int a = 0; a < u; ++a) {
            if (i < m) {
                B[i * lda + m + a] = cols[(size_t)a * m + i];
                B[(m + a) * lda + i] = rows[(size_t)a * m + i];
            } else {
                B[(m + a) * lda + i] = 0.0;
            }
        }
}

// ----------------------------------------------------------------------------
// dense LU with partial pivoting (FP64) for the outer Newton step
// ----------------------------------------------------------------------------

// Blocked right-looking LU of A (m x m, row-major) with the right-hand side b carried along as one more
// column; L is not kept beyond its panel.  Per panel of LU_NB columns: k_lu_panel (one CTA: pivots, row
// exchanges and elimination inside the panel), k_lu_rows (the exchanges and L11^-1 on the columns to the
// right and b), k_lu_update (A22 -= L21 U12, b2 -= L21 u).  A rank-1 update of the whole matrix and three
// launches per column took 15 us a column on 540 unknowns; now the panel's chain of pivot searches sets
// the pace: 540 unknowns 8.8 -> 3.0 ms with the back substitution.
// FP64 multiply-adds (m^3 / 3) are the floor of large systems.
constexpr int LU_NB = 16;

// largest |value| and its smallest row: keys are the bits of |v| (ordered like the values; NaN as 0, so
// that it is never a pivot while another entry is not)
__device__ __forceinline__ long long lu_key(double v) {
    const long long k = __double_as_longlong(v) & 0x7fffffffffffffffll;
    return k > 0x7ff0000000000000ll ? 0 : k;
}

// panel rows k .. m - 1, columns k .. k + nb - 1; in shared memory (row pitch LU_NB + 1) when it fits
__global__ void __launch_bounds__(512) k_lu_panel(double* A, int* piv, int m, int k, int nb, int in_smem, int* flag) {
    extern __shared__ double sp[];
    __shared__ long long skey[16];
    __shared__ int srow[16];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rows = m - k;
    double* P = in_smem ? sp : A + (size_t)k * m + k;
    const size_t pitch = in_smem ? LU_NB + 1 : m;
    if (in_smem) {
        for (int e = tid; e < rows * LU_NB; e += 512) {
            const int r = e / LU_NB, c = e % LU_NB;
            if (c < nb) P[r * pitch + c] = A[(size_t)(k + r) * m + k + c];
        }
        __syncthreads();
    }
    for (int j = 0; j < nb; ++j) {
        long long best = -1;
        int bi = j;
        for (int r = j + tid; r < rows; r += 512) {
            const long long v = lu_key(P[r * pitch + j]);
            if (v > best) {
                best = v;
                bi = r;
            }
        }
        auto reduce = [&](int width) {
            for (int o = width / 2; o > 0; o >>= 1) {
                const long long v = __shfl_xor_sync(0xffffffffu, best, o);
                const int i = __shfl_xor_sync(0xffffffffu, bi, o);
                if (v > best || (v == best && i < bi)) {
                    best = v;
                    bi = i;
                }
            }
        };
        reduce(32);
        if (lane == 0) {
            skey[warp] = best;
            srow[warp] = bi;
        }
        __syncthreads();
        if (warp == 0) {
            best = lane < 16 ? skey[lane] : -1;
            bi = lane < 16 ? srow[lane] : j;
            reduce(32);
            // exchange rows j and bi of the panel: one lane a column
            if (bi != j && lane < nb) {
                const double t = P[j * pitch + lane];
                P[j * pitch + lane] = P[bi * pitch + lane];
                P[bi * pitch + lane] = t;
            }
            if (lane == 0) {
                piv[k + j] = k + bi;
                if (best <= 0) *flag = 1;
            }
        }
        __syncthreads();
        const double pv = P[j * pitch + j];
        for (int r = j + 1 + tid; r < rows; r += 512) {
            double* p = P + r * pitch;
            const double l = p[j] / pv;
            p[j] = l;
            for (int c = j + 1; c < nb; ++c) p[c] -= l * P[j * pitch + c];
        }
        __syncthreads();
    }
    if (in_smem)
        for (int e = tid; e < rows * LU_NB; e += 512) {
            const int r = e / LU_NB, c = e % LU_NB;
            if (c < nb) A[(size_t)(k + r) * m + k + c] = P[r * pitch + c];
        }
}

// columns k + nb .. m - 1 of A and b (column m): the panel's row exchanges, then L11^-1 (unit lower)
__global__ void __launch_bounds__(128) k_lu_rows(double* A, double* b, const int* __restrict__ piv, int m, int k,
                                                 int nb) {
    __shared__ double L[LU_NB][LU_NB];
    __shared__ int pr[LU_NB];
    for (int e = threadIdx.x; e < nb * nb; e += 128) L[e / nb][e % nb] = A[(size_t)(k + e / nb) * m + k + e % nb];
    if (threadIdx.x < nb) pr[threadIdx.x] = piv[k + threadIdx.x];
    __syncthreads();
    const int c = k + nb + blockIdx.x * 128 + threadIdx.x;
    if (c > m) return;
    double* col = c < m ? A + c : b;
    const size_t st = c < m ? m : 1;
    for (int j = 0; j < nb; ++j)
        if (pr[j] != k + j) {
            const double t = col[(size_t)(k + j) * st];
            col[(size_t)(k + j) * st] = col[(size_t)pr[j] * st];
            col[(size_t)pr[j] * st] = t;
        }
    double u[LU_NB];
#pragma unroll
    for (int j = 0; j < LU_NB; ++j) u[j] = j < nb ? col[(size_t)(k + j) * st] : 0.0;
#pragma unroll
    for (int j = 1; j < LU_NB; ++j) {
        if (j >= nb) break;
#pragma unroll
        for (int i = 0; i < j; ++i) u[j] -= L[j][i] * u[i];
        col[(size_t)(k + j) * st] = u[j];
    }
}

// A22 -= L21 U12, 64 x 64 tiles, 4 x 4 values a thread; the first column of tiles also updates b
__global__ void __launch_bounds__(256) k_lu_update(double* A, double* b, int m, int k, int nb) {
    __shared__ double L[LU_NB][65], U[LU_NB][64];   // L transposed
    const int r0 = k + nb + blockIdx.y * 64, c0 = k + nb + blockIdx.x * 64;
    for (int e = threadIdx.x; e < 64 * LU_NB; e += 256) {
        const int r = e / LU_NB, j = e % LU_NB;
        L[j][r] = (r0 + r < m && j < nb) ? A[(size_t)(r0 + r) * m + k + j] : 0.0;
        const int j2 = e / 64, c = e % 64;
        U[j2][c] = (c0 + c < m && j2 < nb) ? A[(size_t)(k + j2) * m + c0 + c] : 0.0;
    }
    __syncthreads();
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;   // columns tx + 16 v, rows ty + 16 u
    double acc[4][4] = {};
#pragma unroll
    for (int j = 0; j < LU_NB; ++j) {
        double l[4], u[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            l[q] = L[j][ty + 16 * q];
            u[q] = U[j][tx + 16 * q];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[q][v] += l[q] * u[v];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int r = r0 + ty + 16 * q, c = c0 + tx + 16 * v;
            if (r < m && c < m) A[(size_t)r * m + c] -= acc[q][v];
        }
    if (blockIdx.x == 0 && threadIdx.x < 64 && r0 + threadIdx.x < m) {
        double t = b[r0 + threadIdx.x];
        for (int j = 0; j < nb; ++j) t -= L[j][threadIdx.x] * b[k + j];
        b[r0 + threadIdx.x] = t;
    }
}

// U x = b in place, one CTA: blocks of 32 rows from the last up; warp 0 solves the 32 x 32 triangle (a
// row per lane, reciprocals of the diagonal formed together), then all threads subtract its columns from
// the rows above, two lanes a row
__global__ void __launch_bounds__(1024) k_back_subst(const double* __restrict__ A, double* x, int m) {
    __shared__ double xs[32], T[32][33];
    const int tid = threadIdx.x, lane = tid & 31;
    for (int k1 = m; k1 > 0; k1 -= 32) {
        const int k0 = max(0, k1 - 32), nb = k1 - k0;
        {
            const int r = tid >> 5;
            T[r][lane] = (r < nb && lane < nb) ? A[(size_t)(k0 + r) * m + k0 + lane] : (r == lane ? 1.0 : 0.0);
        }
        __syncthreads();
        if (tid < 32) {
            double v = lane < nb ? x[k0 + lane] : 0.0;
            const double inv = 1.0 / T[lane][lane];
            for (int i = 31; i >= 0; --i) {
                const double xi = __shfl_sync(0xffffffffu, v * inv, i);
                if (lane == i) v = xi;
                if (lane < i) v -= T[lane][i] * xi;
            }
            xs[lane] = v;
            if (lane < nb) x[k0 + lane] = v;
        }
        __syncthreads();
        for (int r0 = 0; r0 < k0; r0 += 512) {
            const int r = r0 + (tid >> 1);
            double t = 0.0;
            if (r < k0)
                for (int j = tid & 1; j < nb; j += 2) t += A[(size_t)r * m + k0 + j] * xs[j];
            t += __shfl_xor_sync(0xffffffffu, t, 1);
            if (r < k0 && !(tid & 1)) x[r] -= t;
        }
        __syncthreads();
    }
}

// ----------------------------------------------------------------------------
// Lyapunov exponents (App. F)
// ----------------------------------------------------------------------------

// weights w_s(phi) = sum_c H_c(phi) Gamma^-1[c][s] of the trigonometric interpolant; a warp per sample,
// its lanes share the harmonics (sine and cosine in FP64 are the work)
__global__ void __launch_bounds__(128) k_lyap_weights(int N, int U, int dm1, const int* __restrict__ ktab,
                                                      const double* __restrict__ Gi, double phi0, double phi1,
                                                      double phi2, double* wts) {
    const double ph[3] = {phi0, phi1, phi2};
    const int s = (blockIdx.x * 128 + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (s >= N) return;
    double acc = 0.0;
    for (int l = lane; 1 + 2 * l < U; l += 32) {
        double arg = 0.0, sn, cs;
        for (int j = 0; j < dm1; ++j) arg += (double)ktab[l * dm1 + j] * ph[j];
        sincos(arg, &sn, &cs);
        acc += cs * Gi[(size_t)(1 + 2 * l) * N + s] + sn * Gi[(size_t)(2 + 2 * l) * N + s];
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) wts[s] = Gi[s] + acc;
}

// A[i][c] = sum_j (sum_s w_s Psi_s[i][j]) Q[j][c],  Psi = diag(1, w) Phi diag(1, 1/w)  (Eq. F3): the
// interpolated monodromy first, then its product, 4 n^2 (N + h) multiply-adds instead of 4 n^2 N h.  A
// CTA takes LYP_R rows of X or V of one panel; LYP_C columns of the interpolated rows go to shared
// memory, then thread (row, c) adds their products with column c < h <= 64 of Q.
// 90-dof shell, 15 trajectories, h = 32: 92 -> 21 us.
constexpr int LYP_R = 4, LYP_C = 128;
template <typename T>
__global__ void __launch_bounds__(256) k_lyap_prop(int N, int h, double w, PhiView<T> F, const double* __restrict__ wts,
                                                   const double* __restrict__ Q, double* Aout) {
    __shared__ double ms[LYP_R][LYP_C + 1];
    __shared__ int cols[LYP_C];
    int x = blockIdx.x, g = 0;
    while (x >= (F.pan.n[g] + LYP_R - 1) / LYP_R) x -= (F.pan.n[g++] + LYP_R - 1) / LYP_R;
    const int n = F.n, m = F.pan.n[g], ld = F.pan.ld[g], row0 = F.pan.row0[g], r0 = x * LYP_R;
    const bool vel = blockIdx.y != 0;   // rows of V
    const T* B = (vel ? F.V : F.X) + F.pan.off[g] + (size_t)r0 * ld;
    const int tr = threadIdx.x >> 6, tc = threadIdx.x & 63;   // product: row, column of Q
    double acc = 0.0;
    for (int j0 = 0; j0 < 2 * m; j0 += LYP_C) {
        const int nj = min(LYP_C, 2 * m - j0);
        __syncthreads();
        for (int e = threadIdx.x; e < LYP_R * LYP_C; e += 256) {
            const int r = e / LYP_C, j = e % LYP_C;
            double v = 0.0;
            if (j < nj && r0 + r < m) {
                const T* p = B + (size_t)r * ld + j0 + j;
#pragma unroll 4
                for (int s = 0; s < N; ++s) v += wts[s] * (double)p[(size_t)s * F.pan.tot];
                if (j0 + j >= m) v /= w;
            }
            ms[r][j] = v;
            if (r == 0 && j < nj) cols[j] = F.col(g, j0 + j);
        }
        __syncthreads();
        if (tc < h)
#pragma unroll 8
            for (int j = 0; j < nj; ++j) acc += ms[tr][j] * Q[(size_t)cols[j] * h + tc];
    }
    if (tc < h && r0 + tr < m) {
        const int i = F.orig_of[row0 + r0 + tr];
        Aout[(size_t)(vel ? n + i : i) * h + tc] = vel ? w * acc : acc;
    }
}

// Classical Gram-Schmidt with re-orthogonalisation, Q R = A; acc[c] += ln R[c][c].  One cluster: each of
// its CTAs keeps a slice of the rows in shared memory (B, odd row pitch: a column of 32 rows and a row of
// 32 columns both hit 32 banks), Q replacing A column by column; a column needs two sums over all rows
// (the coefficients of each pass, the norm with the second), which the CTAs exchange through distributed
// shared memory, one cluster barrier a sum.  The 2 m h^2 FP64 multiply-adds at 2 a clock and SM would take
// one SM 90 us (m = 180, h = 32), so the rows are split even when few; a warp alone has a quarter of that
// rate (64 clocks an FP64 instruction), so sums are kept shallow and nothing is computed by more warps than
// need it.  With one CTA and a block-wide reduction per coefficient this took 2.3 ms; now 172 us (90-dof
// shell, h = 32, launch included).  Slices that do not fit in shared memory (beyond m h = 200 k values over
// 8 CTAs) work in place on A.
//
// Barriers between the writes and reads of each shared word: red -> the first barrier of exchange, and its
// readers are done at the cluster barrier; part -> the cluster barrier, its slot not written again before
// the cluster barrier of the next exchange; coef -> the last barrier of exchange, its readers are done at
// the barrier that ends the pass (or the norm branch); s_nrm2 = -1 -> the barriers of pass 0 (c > 0 only:
// column 0 has no passes and its branch does not ask), s_nrm2 = |a|^2 -> the barrier that ends pass 1 or
// the norm branch, its readers are done at the barrier that ends the column, as the readers of B are;
// nrms -> that barrier.
constexpr int LYQ_T = 256, LYQ_W = LYQ_T / 32;
__global__ void __launch_bounds__(LYQ_T) k_lyap_qr(int m, int h, int in_smem, double* A, double* Q, double* acc) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = cl.block_rank(), size = cl.num_blocks();   // size 1, 2, 4 or 8
    extern __shared__ double sB[];
    __shared__ double red[LYQ_W][64], coef[64], nrms[64], s_nrm2, part[2][8][64];   // part[event & 1][rank][k]
    const int per = (m + size - 1) / size, i0 = min(m, rank * per), rows = min(m, i0 + per) - i0;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, bp = in_smem ? (h | 1) : h;
    double* B = in_smem ? sB : A + (size_t)i0 * h;
    if (in_smem)
        for (int e = tid; e < rows * h; e += LYQ_T) B[(e / h) * bp + e % h] = A[(size_t)i0 * h + e];
    for (int e = tid; e < 2 * 8 * 64; e += LYQ_T) (&part[0][0][0])[e] = 0.0;   // ranks past the cluster add 0
    cl.sync();
    int event = 0;
    // v[0] + .. + v[7 stride] in pairs
    auto sum8 = [](const double* v, int stride) {
        return ((v[0] + v[stride]) + (v[2 * stride] + v[3 * stride])) +
               ((v[4 * stride] + v[5 * stride]) + (v[6 * stride] + v[7 * stride]));
    };
    // coef[k] = sum over the warps' red[.][k] of all CTAs, k < cnt
    auto exchange = [&](int cnt) {
        __syncthreads();
        if (tid < cnt) {
            const double t = sum8(&red[0][tid], 64);
            for (int r = 0; r < size; ++r) *cl.map_shared_rank(&part[event & 1][rank][tid], r) = t;
        }
        cl.sync();
        if (tid < cnt) coef[tid] = sum8(&part[event & 1][0][tid], 64);
        ++event;
        __syncthreads();
    };
    for (int c = 0; c < h; ++c) {
        if (c > 0 && tid == 0) s_nrm2 = -1.0;
        for (int pass = 0; pass < 2 && c > 0; ++pass) {
            // pass 1 also sums the square of the column itself (k = c) that it is about to correct
            for (int k = lane; k < c + pass; k += 32) {   // lanes across the columns, warps across the rows
                double d = 0.0;
                for (int i = warp; i < rows; i += LYQ_W) d += B[(size_t)i * bp + k] * B[(size_t)i * bp + c];
                red[warp][k] = d;
            }
            exchange(c + pass);
            if (pass == 1 && warp == LYQ_W - 1) {
                // |a - Q y|^2 = |a|^2 - |y|^2 for orthonormal Q; y is what the first pass left, rounding
                // as a rule, and where it is more the norm is summed again below
                double y2 = lane < c ? coef[lane] * coef[lane] : 0.0;
                if (lane + 32 < c) y2 += coef[lane + 32] * coef[lane + 32];
                for (int o = 16; o > 0; o >>= 1) y2 += __shfl_xor_sync(0xffffffffu, y2, o);
                if (lane == 0 && y2 <= 1e-8 * coef[c]) s_nrm2 = coef[c] - y2;
            }
            // four lanes a row
            for (int i0 = 0; i0 < rows; i0 += LYQ_T / 4) {
                const int i = i0 + (tid >> 2);
                double v = 0.0;
                if (i < rows)
                    for (int k = tid & 3; k < c; k += 4) v += coef[k] * B[(size_t)i * bp + k];
                if (i0 + 8 * warp < rows) {   // this warp has rows
                    v += __shfl_xor_sync(0xffffffffu, v, 1);
                    v += __shfl_xor_sync(0xffffffffu, v, 2);
                    if (i < rows && (tid & 3) == 0) B[(size_t)i * bp + c] -= v;
                }
            }
            __syncthreads();
        }
        // the same in every thread of the cluster: coef is, and column 0 does not read the flag
        if (c == 0 || s_nrm2 < 0.0) {
            double d = 0.0;
            for (int i = tid; i < rows; i += LYQ_T) d += B[(size_t)i * bp + c] * B[(size_t)i * bp + c];
            for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            if (lane == 0) red[warp][0] = d;
            exchange(1);
            if (tid == 0) s_nrm2 = coef[0];
            __syncthreads();
        }
        for (int i = tid; i < rows; i += LYQ_T) B[(size_t)i * bp + c] /= sqrt(s_nrm2);
        if (tid == LYQ_T - 1) nrms[c] = sqrt(s_nrm2);
        __syncthreads();
    }
    for (int e = tid; e < rows * h; e += LYQ_T) Q[(size_t)i0 * h + e] = B[(size_t)(e / h) * bp + e % h];
    if (rank == 0 && tid < h) acc[tid] += log(nrms[tid]);
    cl.sync();   // no CTA leaves while another may still write to its shared memory
}

// ----------------------------------------------------------------------------
// launchers
// ----------------------------------------------------------------------------

void launch_idft(fse_ctx* c, const double* Z, double* zb) {
    const Params& p = c->p;
    dim3 g((2 * p.n + 127) / 128, p.N);
    k_idft<<<g, 128, 0, c->stream>>>(p.N, p.U, 2 * p.n, c->d.G, Z, zb);
}

void launch_collect_end(fse_ctx* c) {
    const Params& p = c->p;
    const size_t tot = (size_t)p.N * p.n;
    k_join<<<nblocks(tot, 256), 256, 0, c->stream>>>(p.N, p.n, p.ni, c->d.row_of, c->d.q, c->d.u, c->d.zb);
}

void launch_dft_residual(fse_ctx* c, const double* zb, const double* Z0, double* R, int subtract) {
    const Params& p = c->p;
    const int N = p.N, U = p.U, n2 = 2 * p.n, tiles = (n2 + 31) / 32;
    // FP64 issue slots of one coefficient: a warp per output takes N / 32 and some three for the sum over
    // its lanes, a tile of 32 states N.  Few states have the shorter chains in the first form (18 states,
    // 63 x 63: 2.5 us, 2.8 for the tiles; 24: 3.0 and 2.8; with at most a sample a lane up to 48: 36 states, 25
    // x 25, 2.1 and 2.2); from 128 on its strided reads cost more than any idle lane (144 states, 1024 x 961:
    // 498 us, 263).
    if (n2 < 24 || (n2 < 48 && N <= 32) ||
        (n2 < 128 && (long long)n2 * ((N + 31) / 32 + 3) < (long long)tiles * N)) {
        const size_t lanes = (size_t)32 * n2 * U;
        k_dft_lanes<<<(unsigned)((lanes + 255) / 256), 256, 0, c->stream>>>(N, U, n2, c->d.RG, zb, Z0, R, subtract);
        return;
    }
    // eight warps a tile while the tiles are few and each warp has two samples or more (24 states, 196 x 169:
    // 5.3 us, 5.9 with four; 72 states, 16 x 15: 2.2 and 1.9; 1872-dof shell 34 and 30)
    const unsigned g = (unsigned)tiles * U;
    if (g < 2u * num_sms() && N > 16)
        k_dft_warps<8><<<g, 256, 0, c->stream>>>(N, U, n2, c->d.RG, zb, Z0, R, subtract);
    else
        k_dft_warps<4><<<g, 128, 0, c->stream>>>(N, U, n2, c->d.RG, zb, Z0, R, subtract);
}

template <typename T>
static PhiView<T> phi_view(const fse_ctx* c) {
    return {(const T*)c->d.X, (const T*)c->d.V, c->d.row_of, c->d.orig_of, c->p.n, c->p.pan};
}

template <typename T, int G, int B>
static void phi_rows(fse_ctx* c, const double* zin, double* zout) {
    const size_t lanes = (size_t)c->p.N * (B == 2 ? 1 : 2) * c->p.n * G;
    k_phi_rows<T, G, B><<<(unsigned)((lanes + 255) / 256), 256, 0, c->stream>>>(c->p.N, phi_view<T>(c), zin, zout);
}

void launch_phi_apply(fse_ctx* c, const double* zin, double* zout) {
    const Params& p = c->p;
    int tiles = 0, most = 0;
    double work = 0.0;   // multiply-adds
    for (int g = 0; g < p.pan.nc; ++g) {
        tiles += (p.pan.n[g] + PHI_ROWS - 1) / PHI_ROWS;
        most = std::max(most, p.pan.n[g]);
        work += 4.0 * p.N * p.pan.n[g] * p.pan.n[g];
    }
    const bool f32 = p.prec == FSE_MIXED_FP32, many = (long long)2 * p.n * p.N >= 1024;
    // The staged form needs enough work and enough CTAs to pay for the trip of z through shared memory
    // (FP32, us staged / by rows: 120 dofs, 32 trajectories, 1.8 M: 7.9 / 11.4; 72, 64, 1.3 M: 10.5 / 8.0; 624, 3,
    // 4.7 M: 20 / 25; 360, 3, 1.6 M: 13 / 9; 936, 1, 3.5 M: 28 / 19).
    if (f32 && ((work >= 1.5e6 && p.N >= 8) || (work >= 4e6 && p.N >= 3))) {
        static std::atomic<unsigned long long> attr{0};
        if (needs_device_setup(attr)) {
            cudaFuncSetAttribute(k_phi_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
            mark_device(attr);
        }
        k_phi_apply<<<dim3(tiles, p.N), 256, (size_t)2 * most * 8, c->stream>>>(phi_view<float>(c), zin, zout);
        return;
    }
    // By rows: 16 lanes a row while rows are short (their chains stay short) and many enough to fill the
    // GPU, else 32 (FP64, us with 16 / 32: 243 dofs, 64 trajectories 37 / 66; 200, 3: 4.3 / 3.3; FP32: 54, 16:
    // 3.2 / 4.4; 200, 9: 9.3 / 8.3).  Long FP64 rows of several trajectories in pairs: 447 dofs, 16: 30.8, 34.9 one
    // by one; 936, 16: 107 and 110 (3 trajectories: no difference; one: 11.8 and 10.1).
    if (f32) {
        if (many && 2 * most <= 256)
            phi_rows<float, 16, 1>(c, zin, zout);
        else
            phi_rows<float, 32, 1>(c, zin, zout);
    } else if (2 * most > 512 && p.N >= 9) {
        phi_rows<double, 32, 2>(c, zin, zout);
    } else if (many && 2 * most <= 512) {
        phi_rows<double, 16, 1>(c, zin, zout);
    } else {
        phi_rows<double, 32, 1>(c, zin, zout);
    }
}

void launch_domega(fse_ctx* c, double* zout) {
    const Params& p = c->p;
    const size_t tot = (size_t)p.N * 2 * p.n;
    if (p.prec == FSE_MIXED_FP32)
        k_domega_col<float><<<nblocks(tot, 256), 256, 0, c->stream>>>(p.N, phi_view<float>(c), zout);
    else
        k_domega_col<double><<<nblocks(tot, 256), 256, 0, c->stream>>>(p.N, phi_view<double>(c), zout);
}

static void phi_copy_range(fse_ctx* c, int s0, int count, double* Phi, double* dzdw) {
    const Params& p = c->p;
    const size_t tot = (size_t)count * 4 * p.n * p.n;
    if (p.prec == FSE_MIXED_FP32)
        k_phi_copy<float><<<nblocks(tot, 256), 256, 0, c->stream>>>(count, s0, phi_view<float>(c), Phi, dzdw);
    else
        k_phi_copy<double><<<nblocks(tot, 256), 256, 0, c->stream>>>(count, s0, phi_view<double>(c), Phi, dzdw);
}

void launch_phi_copy(fse_ctx* c, double* Phi, double* dzdw) { phi_copy_range(c, 0, c->p.N, Phi, dzdw); }

void launch_phi_copy_one(fse_ctx* c, int s, double* Phi, double* dzdw) { phi_copy_range(c, s, 1, Phi, dzdw); }

// dense Eq. (22) into an array of row stride lda
static void dense_jac(fse_ctx* c, double* J, size_t lda) {
    const Params& p = c->p;
    const size_t m = (size_t)2 * p.n * p.U;
    if (p.prec == FSE_MIXED_FP32)
        k_dense_jac<float><<<nblocks(m * m, 256, 64), 256, 0, c->stream>>>(p.N, p.U, phi_view<float>(c), c->d.RG,
                                                                           c->d.G, J, lda);
    else
        k_dense_jac<double><<<nblocks(m * m, 256, 64), 256, 0, c->stream>>>(p.N, p.U, phi_view<double>(c), c->d.RG,
                                                                            c->d.G, J, lda);
}

void launch_dense_jac(fse_ctx* c, double* J) { dense_jac(c, J, (size_t)2 * c->p.n * c->p.U); }

void launch_pmat(fse_ctx* c, double* Pm) {
    const Params& p = c->p;
    k_pmat<<<nblocks((size_t)p.N * p.N, 256), 256, 0, c->stream>>>(p.N, p.U, c->d.G, c->d.RG, Pm);
}

void launch_dense_jac_ht(fse_ctx* c, const double* Pm, double* J) {
    const Params& p = c->p;
    const size_t m = (size_t)2 * p.n * p.N;
    if (p.prec == FSE_MIXED_FP32)
        k_dense_jac_ht<float><<<nblocks(m * m, 256, 64), 256, 0, c->stream>>>(p.N, phi_view<float>(c), Pm, J);
    else
        k_dense_jac_ht<double><<<nblocks(m * m, 256, 64), 256, 0, c->stream>>>(p.N, phi_view<double>(c), Pm, J);
}

void launch_bordered_jac(fse_ctx* c, const double* Rw, const double* tZ, double tail, double* B) {
    const size_t m = (size_t)2 * c->p.n * c->p.U;
    dense_jac(c, B, m + 1);
    k_border<<<nblocks(m + 1, 256), 256, 0, c->stream>>>(m, Rw, tZ, tail, B);
}

void launch_unknown_border(fse_ctx* c, int j, double w, const double* R, const double* Z0, double* col,
                           double* row) {
    const Params& p = c->p;
    const size_t m = (size_t)2 * p.n * p.U;
    k_unknown_border<<<nblocks(m, 256), 256, 0, c->stream>>>(m, p.U, p.d - 1, j, c->d.ktab, 2.0 * M_PI / w, R, Z0,
                                                             col, row);
}

void launch_dense_jac_bordered(fse_ctx* c, int u, const double* cols, const double* rows, double* B) {
    const size_t m = (size_t)2 * c->p.n * c->p.U;
    dense_jac(c, B, m + u);
    k_border_multi<<<nblocks(m + u, 256), 256, 0, c->stream>>>(m, u, cols, rows, B);
}

int dense_lu_solve(fse_ctx* c, double* A, double* bvec, int m) {
    int* flag = c->d.flag + 1;   // zero-pivot flag: the context's second status word
    cudaMemsetAsync(flag, 0, sizeof(int), c->stream);
    static std::atomic<unsigned long long> attr{0};
    if (needs_device_setup(attr)) {
        cudaFuncSetAttribute(k_lu_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        mark_device(attr);
    }
    for (int k = 0; k < m; k += LU_NB) {
        const int nb = std::min(LU_NB, m - k), rest = m - k - nb;
        const size_t smem = (size_t)(m - k) * (LU_NB + 1) * 8;
        const int in_smem = smem <= 200 * 1024;
        k_lu_panel<<<1, 512, in_smem ? smem : 0, c->stream>>>(A, c->piv, m, k, nb, in_smem, flag);
        k_lu_rows<<<(rest + 1 + 127) / 128, 128, 0, c->stream>>>(A, bvec, c->piv, m, k, nb);
        if (rest > 0)
            k_lu_update<<<dim3((rest + 63) / 64, (rest + 63) / 64), 256, 0, c->stream>>>(A, bvec, m, k, nb);
    }
    k_back_subst<<<1, 1024, 0, c->stream>>>(A, bvec, m);
    int h = 0;
    cudaMemcpyAsync(&h, flag, sizeof(int), cudaMemcpyDeviceToHost, c->stream);
    const cudaError_t e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) {
        c->err = std::string("dense LU: ") + cudaGetErrorString(e);
        return FSE_ECUDA;
    }
    return h ? FSE_ENONPOS_PIVOT : FSE_OK;
}

// N_Ly steps of the propagation from Q, with scratch A (2n x h), wts (N); acc[c] += sum of ln R[c][c]
static int lyapunov_steps(fse_ctx* c, double w, int N_Ly, int h, double* Q, double* A, double* acc, double* wts) {
    const Params& p = c->p;
    const int m = 2 * p.n;
    static std::atomic<unsigned long long> attr{0};
    if (needs_device_setup(attr)) {
        cudaFuncSetAttribute(k_lyap_qr, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        mark_device(attr);
    }
    // 8 CTAs (the portable cluster size) from 64 rows on: fewer rows a CTA than that are all barrier
    int size = 1;
    while (size < 8 && m / (2 * size) >= 8) size *= 2;
    const size_t smem = (size_t)((m + size - 1) / size) * (h | 1) * 8;
    const int in_smem = smem <= 200 * 1024;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(size);
    cfg.blockDim = dim3(LYQ_T);
    cfg.dynamicSmemBytes = in_smem ? smem : 0;
    cfg.stream = c->stream;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = size;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int tiles = 0;
    for (int g = 0; g < p.pan.nc; ++g) tiles += (p.pan.n[g] + LYP_R - 1) / LYP_R;
    for (int i = 1; i <= N_Ly; ++i) {
        double ph[3] = {0, 0, 0};
        for (int j = 0; j < p.d - 1; ++j) ph[j] = 2.0 * (i - 1) * M_PI * c->rho[j];
        k_lyap_weights<<<(p.N + 3) / 4, 128, 0, c->stream>>>(p.N, p.U, p.d - 1, c->d.ktab, c->d.Gi, ph[0], ph[1],
                                                             ph[2], wts);
        if (p.prec == FSE_MIXED_FP32)
            k_lyap_prop<float><<<dim3(tiles, 2), 256, 0, c->stream>>>(p.N, h, w, phi_view<float>(c), wts, Q, A);
        else
            k_lyap_prop<double><<<dim3(tiles, 2), 256, 0, c->stream>>>(p.N, h, w, phi_view<double>(c), wts, Q, A);
        const cudaError_t e = cudaLaunchKernelEx(&cfg, k_lyap_qr, m, h, in_smem, A, Q, acc);
        if (e != cudaSuccess) {
            c->err = std::string("Lyapunov QR launch: ") + cudaGetErrorString(e);
            return FSE_ECUDA;
        }
    }
    return FSE_OK;
}

int lyapunov_run(fse_ctx* c, double w, int N_Ly, int h, double* sigma) {
    const Params& p = c->p;
    const int m = 2 * p.n;
    double *Q = nullptr, *A = nullptr, *acc = nullptr, *wts = nullptr;
    cudaError_t ea = cudaMalloc(&Q, sizeof(double) * m * h);
    if (ea == cudaSuccess) ea = cudaMalloc(&A, sizeof(double) * m * h);
    if (ea == cudaSuccess) ea = cudaMalloc(&acc, sizeof(double) * h);
    if (ea == cudaSuccess) ea = cudaMalloc(&wts, sizeof(double) * p.N);
    if (ea != cudaSuccess) {
        // nothing has been launched: free what was allocated and report before any kernel runs
        cudaGetLastError();
        for (double* q : {Q, A, acc, wts})
            if (q) cudaFree(q);
        c->err = std::string("Lyapunov scratch allocation failed: ") + cudaGetErrorString(ea);
        return FSE_ENOMEM;
    }
    std::vector<double> Q0((size_t)m * h, 0.0);
    for (int c2 = 0; c2 < h; ++c2) Q0[(size_t)c2 * h + c2] = 1.0;
    cudaMemcpyAsync(Q, Q0.data(), sizeof(double) * m * h, cudaMemcpyHostToDevice, c->stream);
    cudaMemsetAsync(acc, 0, sizeof(double) * h, c->stream);
    const int rc = lyapunov_steps(c, w, N_Ly, h, Q, A, acc, wts);
    std::vector<double> hacc(h);
    cudaMemcpyAsync(hacc.data(), acc, sizeof(double) * h, cudaMemcpyDeviceToHost, c->stream);
    cudaError_t e = cudaStreamSynchronize(c->stream);
    cudaFree(Q);
    cudaFree(A);
    cudaFree(acc);
    cudaFree(wts);
    if (rc) return rc;
    if (e != cudaSuccess) {
        c->err = std::string("Lyapunov run: ") + cudaGetErrorString(e);
        return FSE_ECUDA;
    }
    const double T1 = 2.0 * M_PI / w;
    for (int j = 0; j < h; ++j) sigma[j] = hacc[j] / (N_Ly * T1);
    return FSE_OK;
}

}  // namespace fse

// ----------------------------------------------------------------------------
// Lyapunov propagation with static device scratch (no allocation)
// ----------------------------------------------------------------------------
// Some callers must not allocate device memory while they run: a process that
// hands all of the GPU's memory to its own pool at start-up and allows no
// other allocation, or a latency-bound loop that cannot take the device-wide
// synchronisation that cudaFree implies.  For them the propagation's scratch
// (the Q and A blocks, the ln|R_jj| accumulators and the interpolation
// weights) is one fixed-size array in the library's device image: every GPU
// that loads the library holds its 4.5 MiB until the process exits.  All calls
// share it and it keeps the last call's contents, so each call sets Q and the
// accumulators before use, and calls that overlap on the GPU race on it.

namespace {

constexpr size_t kNoallocQ = FSE_NOALLOC_MAX_QH;   // doubles of Q (and of A)
constexpr size_t kNoallocAcc = 64;                  // ln|R_jj| accumulators (h <= 64)
constexpr size_t kNoallocW = FSE_NOALLOC_MAX_N;     // interpolation weights (one per trajectory)

// In host code this name is only a stand-in for the symbol, never a device
// address: the address is looked up per device with cudaGetSymbolAddress.
static __device__ __align__(256) double g_lyap_scratch[2 * kNoallocQ + kNoallocAcc + kNoallocW];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
double* g_scratch_dev[kMaxDevices] = {};   // device address of g_lyap_scratch, per device ordinal

// Q = [I_h; 0] (m x h, row-major) and acc = 0
__global__ void k_lyap_init(int m, int h, double* Q, double* acc) {
    const size_t total = (size_t)m * h;
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < total; x += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(x / h), col = (int)(x % h);
        Q[x] = (i == col) ? 1.0 : 0.0;
        if (x < (size_t)h) acc[x] = 0.0;
    }
}

}  // namespace

namespace fse {

// Device address of the static scratch on `device` (which must be current);
// looked up on the first call per device and cached.
static int noalloc_scratch(fse_ctx* c, double** out) {
    if (c->device < 0 || c->device >= kMaxDevices) {
        c->err = "static scratch: device ordinal out of range";
        return FSE_EINVAL;
    }
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_dev[c->device]) {
        void* ptr = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&ptr, g_lyap_scratch);
        if (e != cudaSuccess || !ptr) {
            c->err = std::string("static scratch: cudaGetSymbolAddress failed: ") + cudaGetErrorString(e);
            return FSE_ECUDA;
        }
        g_scratch_dev[c->device] = (double*)ptr;
    }
    *out = g_scratch_dev[c->device];
    return FSE_OK;
}

int lyapunov_run_noalloc(fse_ctx* c, double w, int N_Ly, int h, double* sigma) {
    const Params& p = c->p;
    const int m = 2 * p.n;
    if (h < 1 || (size_t)h > kNoallocAcc || (size_t)m * h > kNoallocQ || (size_t)p.N > kNoallocW) {
        c->err = "static scratch: size beyond its maximum";
        return FSE_EINVAL;
    }
    double* base = nullptr;
    const int rc = noalloc_scratch(c, &base);
    if (rc) return rc;
    double* Q = base;
    double* A = base + kNoallocQ;
    double* acc = base + 2 * kNoallocQ;
    double* wts = acc + kNoallocAcc;
    k_lyap_init<<<nblocks((size_t)m * h, 256), 256, 0, c->stream>>>(m, h, Q, acc);
    const int rs = lyapunov_steps(c, w, N_Ly, h, Q, A, acc, wts);
    if (rs) return rs;
    double hacc[kNoallocAcc];
    cudaMemcpyAsync(hacc, acc, sizeof(double) * h, cudaMemcpyDeviceToHost, c->stream);
    const cudaError_t e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) {
        c->err = std::string("static-scratch Lyapunov run: ") + cudaGetErrorString(e);
        return FSE_ECUDA;
    }
    const double T1 = 2.0 * M_PI / w;
    for (int j = 0; j < h; ++j) sigma[j] = hacc[j] / (N_Ly * T1);
    return FSE_OK;
}

}  // namespace fse

// ----------------------------------------------------------------------------
// small vector helpers of the outer solve and the continuation driver
// ----------------------------------------------------------------------------

namespace fse {

// y = a x + b y; with b = 0 what y held (nothing yet, or a NaN of an earlier call) does not take part
__global__ void k_axpby(size_t n, double a, const double* x, double b, double* y) {
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x)
        y[k] = b == 0.0 ? a * x[k] : a * x[k] + b * y[k];
}

// out[i] = a_i . b_i for i < gridDim.y, a_i = a + i sa, b_i = b + i sb.  gridDim.x blocks share a dot
// product; the last one to finish adds the partial sums in block order, so the result does not depend on
// which that is.  part: gridDim.y x gridDim.x doubles, count: gridDim.y counters, zero before and after.
__global__ void __launch_bounds__(256) k_dots(size_t n, const double* a, ptrdiff_t sa, const double* b, ptrdiff_t sb,
                                              double* part, unsigned* count, double* out) {
    __shared__ double red[8];
    __shared__ bool last;
    const int i = blockIdx.y, nb = gridDim.x;
    const double *x = a + (ptrdiff_t)i * sa, *y = b + (ptrdiff_t)i * sb;
    const size_t per = (n + nb - 1) / nb, k0 = blockIdx.x * per, k1 = min(n, k0 + per);
    double acc = 0.0;
#pragma unroll 4
    for (size_t k = k0 + threadIdx.x; k < k1; k += 256) acc += x[k] * y[k];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        part[(size_t)i * nb + blockIdx.x] = t;
        __threadfence();
        last = atomicInc(&count[i], nb - 1) == (unsigned)nb - 1;
    }
    __syncthreads();
    if (last && threadIdx.x == 0) {
        __threadfence();
        double t = 0.0;
        for (int k = 0; k < nb; ++k) t += __ldcg(part + (size_t)i * nb + k);
        out[i] = t;
    }
}

// x *= 1 / sqrt(norm2[0]) (left alone where that is not positive)
__global__ void k_normalise(size_t n, const double* norm2, double* x) {
    const double s = *norm2;
    if (!(s > 0.0)) return;
    const double f = 1.0 / sqrt(s);
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x)
        x[k] *= f;
}

// z = mean + sum_k c_k basis[k]  (basis r x nu)
__global__ void k_pod_expand(size_t nu, int r, const double* mean, const double* basis, const double* coef,
                             double* z) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < nu; x += (size_t)gridDim.x * blockDim.x) {
        double acc = mean[x];
        for (int k = 0; k < r; ++k) acc += coef[k] * basis[(size_t)k * nu + x];
        z[x] = acc;
    }
}

// coef[j][k] = basis[k] . (Z[j] - mean), one block per (j, k)
__global__ void k_pod_project(size_t nu, int r, const double* mean, const double* basis, const double* Z,
                              double* coef) {
    const int j = blockIdx.x, k = blockIdx.y;
    __shared__ double red[256];
    double acc = 0.0;
    for (size_t x = threadIdx.x; x < nu; x += blockDim.x)
        acc += basis[(size_t)k * nu + x] * (Z[(size_t)j * nu + x] - mean[x]);
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) coef[(size_t)j * r + k] = red[0];
}

// w += sign sum_{i<k} coef[i] V_i
__global__ void __launch_bounds__(128) k_mupdate(size_t n, int k, const double* __restrict__ V,
                                                 const double* __restrict__ coef, double sign, double* w) {
    __shared__ double cs[257];   // k <= restart + 1
    for (int i = threadIdx.x; i < k; i += 128) cs[i] = sign * coef[i];
    __syncthreads();
    for (size_t x = blockIdx.x * (size_t)128 + threadIdx.x; x < n; x += (size_t)gridDim.x * 128) {
        double acc = w[x];
#pragma unroll 8
        for (int i = 0; i < k; ++i) acc += cs[i] * V[(size_t)i * n + x];
        w[x] = acc;
    }
}

// One block per dot product left the GPU idle (31 us for 40 products of 26640 values, 2 us of reading):
// blocks of about 4096 values, at most FSE_DOT_BLOCKS a product (10 us, launches and caches cold).
static void dots(fse_ctx* c, size_t n, int k, const double* a, ptrdiff_t sa, const double* b, ptrdiff_t sb,
                 double* out_dev) {
    const int nb = (int)std::min<size_t>(FSE_DOT_BLOCKS, (n + 4095) / 4096);
    for (int i = 0; i < k; i += FSE_DOT_VECS) {   // the partial sums hold FSE_DOT_VECS products at a time
        const int m = std::min(FSE_DOT_VECS, k - i);
        k_dots<<<dim3(nb, m), 256, 0, c->stream>>>(n, a + i * sa, sa, b + i * sb, sb, c->d.red, c->d.redc, out_dev + i);
    }
}

void vec_mdot(fse_ctx* c, size_t n, int k, const double* V, const double* w, double* out_dev) {
    dots(c, n, k, V, (ptrdiff_t)n, w, 0, out_dev);
}

void vec_mupdate(fse_ctx* c, size_t n, int k, const double* V, const double* coef_dev, double sign, double* w) {
    k_mupdate<<<nblocks(n, 128), 128, 0, c->stream>>>(n, k, V, coef_dev, sign, w);
}

void vec_normalise(fse_ctx* c, size_t n, const double* norm2_dev, double* x) {
    k_normalise<<<nblocks(n, 256), 256, 0, c->stream>>>(n, norm2_dev, x);
}

void vec_axpby(fse_ctx* c, size_t n, double a, const double* x, double b, double* y) {
    k_axpby<<<nblocks(n, 256), 256, 0, c->stream>>>(n, a, x, b, y);
}

void vec_norms2(fse_ctx* c, size_t n, const double* x, const double* y, double* out_dev) {
    if (!y) cudaMemsetAsync(out_dev + 1, 0, 8, c->stream);
    const ptrdiff_t d = y ? ((intptr_t)y - (intptr_t)x) / 8 : 0;
    dots(c, n, y ? 2 : 1, x, d, x, d, out_dev);
}

void pod_expand(fse_ctx* c, size_t nu, int r, const double* mean, const double* basis, const double* coef,
                double* z) {
    k_pod_expand<<<nblocks(nu, 256), 256, 0, c->stream>>>(nu, r, mean, basis, coef, z);
}

void pod_project(fse_ctx* c, size_t nu, int r, int m, const double* mean, const double* basis, const double* Z,
                 double* coef) {
    k_pod_project<<<dim3(m, r), 256, 0, c->stream>>>(nu, r, mean, basis, Z, coef);
}

}  // namespace fse
