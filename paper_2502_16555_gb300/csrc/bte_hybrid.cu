// Self-consistent field, ion fluid step and the fully-implicit electron step of arXiv 2502.16555
// (Section 2.3, eqs. "hybrid_discrete", "voltage_bc", "fl_ion_bc"; Section 3.4, eqs. "fluid_step",
// "bte_semi_implicit_efield", "bte_fully_implicit", "1dbte_jac_action"), declared in include/bte.h.
//
//   field        E = L (n_i - u^T F) + V(0, t) E_1: n_e per point, then one dense Nx x Nx product
//                (L and E_1 from the Dirichlet Laplacian on the collocation points, host-assembled);
//   ion step     (I/dt + D_x (mu_i E^n .) - D_i D_x D_x) n^{n+1} = n^n/dt + n0 r_ion.F^n with the
//                outflow-only wall fluxes as the first and last rows, solved by one CTA (GEPP);
//   sc step      the semi-implicit step with E^{1/2} recomputed after the first x half step;
//   implicit     Newton with backtracking on R(F) = F - F^n + dt [A_x F D_x^T - P_O (C + E(F) A_v) P_S F]
//                (inflow rows R = F), each Newton system by restarted flexible GMRES on the Jacobian
//                action J X = X + dt [A_x X D_x^T - P_O (C + E(F) A_v) P_S X
//                + P_O A_v P_S ((L u^T X) . F)], right-preconditioned at the iterate's field by the
//                per-point solves (factors formed once per Newton iteration) followed by one full x
//                step (default), or by the semi-implicit step's map; the preconditioned vectors are
//                kept, so the update is exact for the basis GMRES built. Orthogonalisation by
//                classical Gram-Schmidt applied twice; the small Hessenberg least-squares problem on
//                the host. All vectors FP64 on the device.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "bte_handle.h"
#include "bte_kernels.h"
#include "bte_mass.cuh"
#include "bte_recip.cuh"

namespace {

constexpr int kDotBlock = 256;   // threads of the reduction kernels
constexpr int kDotGrid = 152;    // blocks of the partial dot products (at most; one per SM)
// blocks for n elements: at least four elements a thread
int dot_grid(size_t n) {
  return static_cast<int>(std::max<size_t>(1, std::min<size_t>(kDotGrid, n / (4 * kDotBlock))));
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) s += red[w];
  __syncthreads();
  return s;
}

// out[i] = w . X_i for every point i (one CTA per point): n_e with w = u, the ionisation source
// with w = r_ion.
__global__ void point_dot_kernel(const double* __restrict__ X, const double* __restrict__ w, int nv,
                                 double* __restrict__ out) {
  __shared__ double red[32];
  const double* x = X + static_cast<size_t>(blockIdx.x) * nv;
  double s = 0.0;
  for (int v = threadIdx.x; v < nv; v += blockDim.x) s = fma(__ldg(w + v), x[v], s);
  s = block_sum(s, red);
  if (threadIdx.x == 0) out[blockIdx.x] = s;
}

// E_i = sum_j L[i][j] (ni_j - ne_j) + vleft E1_i (ni NULL: no ions), one warp per row.
__global__ void field_kernel(const double* __restrict__ Lop, const double* __restrict__ E1,
                             const double* __restrict__ ni, const double* __restrict__ ne, double vleft, int nx,
                             double* __restrict__ E) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= nx) return;
  const double* l = Lop + static_cast<size_t>(warp) * nx;
  double s = 0.0;
  for (int j = lane; j < nx; j += 32) s = fma(l[j], (ni ? ni[j] : 0.0) - ne[j], s);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) E[warp] = s + vleft * E1[warp];
}

// D2 = D_x D_x, once per handle (row i per CTA).
__global__ void square_kernel(const double* __restrict__ Dx, int nx, double* __restrict__ D2) {
  const int i = blockIdx.x;
  const double* di = Dx + static_cast<size_t>(i) * nx;
  for (int j = threadIdx.x; j < nx; j += blockDim.x) {
    double dd = 0.0;
    for (int k = 0; k < nx; ++k) dd = fma(di[k], Dx[static_cast<size_t>(k) * nx + j], dd);
    D2[static_cast<size_t>(i) * nx + j] = dd;
  }
}

// The ion system of eq. "fluid_step", row i per CTA: A = I/dt + D_x diag(mu E) - d D_x D_x,
// b = ni/dt + src; the wall rows are the flux conditions J(0) = n max(0, -mu E(0)) and
// J(L) = -n max(0, mu E(L)) with J = mu E n - d D_x n (right-hand side 0).
__global__ void ion_assemble_kernel(const double* __restrict__ Dx, const double* __restrict__ D2,
                                    const double* __restrict__ E,
                                    const double* __restrict__ ni, const double* __restrict__ src, double mu,
                                    double d, double dt, int nx, double* __restrict__ A, double* __restrict__ b) {
  const int i = blockIdx.x;
  double* a = A + static_cast<size_t>(i) * nx;
  const double* di = Dx + static_cast<size_t>(i) * nx;
  const bool wall = i == 0 || i == nx - 1;
  for (int j = threadIdx.x; j < nx; j += blockDim.x) {
    double v;
    if (wall) {
      v = -d * di[j] + (i == j ? mu * E[i] : 0.0);
      if (i == j) v += i == 0 ? -fmax(0.0, -mu * E[i]) : fmax(0.0, mu * E[i]);
    } else {
      v = di[j] * mu * E[j] - d * D2[static_cast<size_t>(i) * nx + j] + (i == j ? 1.0 / dt : 0.0);
    }
    a[j] = v;
  }
  if (threadIdx.x == 0) b[i] = wall ? 0.0 : ni[i] / dt + src[i];
  if (wall) {
    // the flux rows are ~1e-9 of the interior rows (1/dt) in scale: equilibrate them (same
    // solution) so the wall values are not left to the rounding of a badly scaled system
    __shared__ double red[32];
    __syncthreads();
    double mx = 0.0;
    for (int j = threadIdx.x; j < nx; j += blockDim.x) mx = fmax(mx, fabs(a[j]));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < static_cast<int>(blockDim.x >> 5); ++w) red[0] = fmax(red[0], red[w]);
    }
    __syncthreads();
    const double sc = red[0] > 0.0 ? (1.0 / dt) / red[0] : 1.0;
    for (int j = threadIdx.x; j < nx; j += blockDim.x) a[j] *= sc;
  }
}

// x = A^-1 b by Gaussian elimination with partial pivoting, one CTA. A ([n][ld], column n holds b) is
// in shared memory for n <= kSmemSolve, in global memory above (overwritten). Rows are marked, not
// exchanged: every warp finds the pivot of a column for itself (the magnitudes as ordered integers, so
// that the FP64 units, whose rate bounds the kernel, do products only) and takes the rows i = warp,
// warp + nw, ..; one barrier a column. A zero or non-finite pivot sets kZeroPivot in status.
// A warp's FMA takes the FP64 units 16 cycles however many lanes are active, so the multipliers of 32 rows are
// formed by one instruction, and in shared memory b is A's column n and the pivot row is in registers.
// n = 100: 286 us; 406 with a multiplier and a right-hand side's FMA per row and warp, 470 with row
// exchanges, a division and FP64 comparisons per column.
constexpr int kSmemSolve = 150;
constexpr int kChunks = (kSmemSolve + 32) / 32;  // of 32 columns of [A b]
size_t ion_smem(size_t n, bool shared) {
  return (shared ? sizeof(double) * n * ((n + 1) | 1) : 0) + n * (2 * sizeof(double) + sizeof(int));
}
template <bool kShared>
__global__ void __launch_bounds__(512) dense_solve_kernel(double* __restrict__ Ag, const double* __restrict__ bg, int n,
                                                          double* __restrict__ x, unsigned* status) {
  extern __shared__ double sm[];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int ld = kShared ? (n + 1) | 1 : n;  // odd: a column's entries lie in different banks
  double* A = kShared ? sm : Ag;
  double* b = kShared ? sm + n : sm;         // n, stride bs: column n of A in shared memory
  const int bs = kShared ? ld : 1;
  double* pin = kShared ? sm + n * ld : b + n;  // n: reciprocals of the pivots
  int* slot = reinterpret_cast<int*>(pin + n);  // n: the column a row was the pivot of, -1 before
  __shared__ unsigned used_w[128];           // bit per row
  for (int i = tid; i < n; i += nt) b[i * bs] = bg[i], slot[i] = -1;
  for (int i = tid; i < 128; i += nt) used_w[i] = 0u;
  if (kShared)
    for (int i = warp; i < n; i += nw)
      for (int j = lane; j < n; j += 32) A[i * ld + j] = Ag[static_cast<size_t>(i) * n + j];
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    unsigned long long best = 0ull;
    int bi = -1;
    for (int i = lane, q = 0; i < n; i += 32, ++q) {
      if ((used_w[q] >> lane) & 1u) continue;
      const unsigned long long key =
          static_cast<unsigned long long>(__double_as_longlong(A[static_cast<size_t>(i) * ld + k]) & 0x7fffffffffffffffll) + 1ull;
      if (key > best) best = key, bi = i;
    }
    const unsigned hi = static_cast<unsigned>(best >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned lo = hi == mh ? static_cast<unsigned>(best) : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
    const unsigned row = hi == mh && static_cast<unsigned>(best) == ml && bi >= 0 ? static_cast<unsigned>(bi) : 0xffffffffu;
    const int p = static_cast<int>(__reduce_min_sync(0xffffffffu, row));
    const unsigned long long pk = (static_cast<unsigned long long>(mh) << 32) | ml;
    const double* ap = A + static_cast<size_t>(p) * ld;
    const double inv = bte::recip(ap[k]);
    if constexpr (kShared) {
      double apr[kChunks];
#pragma unroll
      for (int c = 0; c < kChunks; ++c) apr[c] = k + 1 + lane + 32 * c <= n ? ap[k + 1 + lane + 32 * c] : 0.0;
      for (int i0 = 0; warp + nw * i0 < n; i0 += 32) {  // 32 rows of the warp: a lane takes a row's multiplier
        const int il = warp + nw * (i0 + lane);
        const bool on = il < n && il != p && !((used_w[il >> 5] >> (il & 31)) & 1u);
        const double lm = on ? A[static_cast<size_t>(il) * ld + k] * inv : 0.0;
        for (unsigned rest = __ballot_sync(0xffffffffu, on); rest; rest &= rest - 1) {
          const int src = __ffs(rest) - 1;
          double* ai = A + static_cast<size_t>(warp + nw * (i0 + src)) * ld;
          const double l = __shfl_sync(0xffffffffu, lm, src);
#pragma unroll
          for (int c = 0; c < kChunks; ++c) {
            if (k + 1 + 32 * c > n) break;
            const int j = k + 1 + lane + 32 * c;
            if (j <= n) ai[j] = fma(-l, apr[c], ai[j]);
          }
        }
      }
    } else {
      const double bp = b[p];
      for (int i = warp; i < n; i += nw) {
        if (i == p || ((used_w[i >> 5] >> (i & 31)) & 1u)) continue;
        double* ai = A + static_cast<size_t>(i) * ld;
        const double l = ai[k] * inv;
        for (int j = k + 1 + lane; j < n; j += 32) ai[j] = fma(-l, ap[j], ai[j]);
        if (lane == 0) b[i] = fma(-l, bp, b[i]);
      }
    }
    __syncthreads();  // every warp has read the marks and the pivot row's marker of this column
    if (tid == 0) {
      if (pk < 2ull || pk > 0x7ff0000000000000ull) atomicOr(status, bte::kZeroPivot);
      used_w[p >> 5] |= 1u << (p & 31);
      slot[k] = p;
      pin[k] = inv;
    }
    __syncthreads();
  }
  // back substitution by columns, warp 0: x_k, then every earlier pivot row's right-hand side
  if (warp == 0) {
    for (int k = n - 1; k >= 0; --k) {
      const double xk = b[slot[k] * bs] * pin[k];
      __syncwarp();
      for (int q = lane; q < k; q += 32) {
        const int r = slot[q];
        b[r * bs] = fma(-A[static_cast<size_t>(r) * ld + k], xk, b[r * bs]);
      }
      if (lane == 0) x[k] = xk;
      __syncwarp();
    }
  }
}

// out_i = P_O M_v^-1 (c C + e_i A_v) P_S X_i per point (one CTA per point): c = 1 and e_i = E[i] for
// the velocity operator at a field, c = 0 and e_i = 1 for P_O A_v P_S alone. Banded operators as in the
// refinement residual (Algorithm 2), or, with few unknowns, the dense mass-scaled blocks (Cs not NULL): the
// Cholesky substitution is 2 nr dependent steps of one warp (25 us at nr = 64 whatever nl, on FP64 units
// that take a warp's FMA in about 70 cycles), the dense products 3 nl nr^2 FMAs over all warps (8 us at
// nl = 3); they meet near nl nr = 400. The projections by parity (Y_l(-mu) = (-1)^l Y_l(mu), symmetric
// ordinates): half their FP64 operations, which bound it.
__global__ void v_apply_kernel(const double* __restrict__ X, const double* __restrict__ E, double c, bte::ResidualOps ro,
                               const double* __restrict__ Cs, const double* __restrict__ Alo,
                               const double* __restrict__ Aup, const double* __restrict__ TO, const double* __restrict__ TS, double* __restrict__ out,
                               int nt, int nr, int nl) {
  extern __shared__ double sm[];
  const int i = blockIdx.x, nv = nt * nr, hf = nt / 2, hc = (nt + 1) / 2, w = ro.w, bw = 2 * w + 1;
  double* fold = sm;                 // 2 hc nr
  double* xS = fold + 2 * hc * nr;   // nl nr
  double* g = xS + nl * nr;          // nl nr
  const double* x = X + static_cast<size_t>(i) * nv;
  const double e = E ? E[i] : 1.0;
  for (int v = threadIdx.x; v < hc * nr; v += blockDim.x) {
    const int q = v / nr, k = v % nr;
    const double p = x[v], m = q < hf ? x[(nt - 1 - q) * nr + k] : 0.0;
    fold[v] = p + m;
    fold[hc * nr + v] = q < hf ? p - m : 0.0;
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < nl * nr; idx += blockDim.x) {
    const int l = idx / nr, k = idx % nr;
    const double* src = fold + (l & 1 ? hc * nr : 0) + k;
    double s0 = 0.0, s1 = 0.0;
    int q = 0;
    for (; q + 1 < hc; q += 2) {
      s0 = fma(__ldg(TS + l * nt + q), src[q * nr], s0);
      s1 = fma(__ldg(TS + l * nt + q + 1), src[(q + 1) * nr], s1);
    }
    if (q < hc) s0 = fma(__ldg(TS + l * nt + q), src[q * nr], s0);
    xS[idx] = s0 + s1;
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < nl * nr; idx += blockDim.x) {
    const int l = idx / nr, p = idx % nr, k0 = max(0, p - w), k1 = min(nr - 1, p + w);
    const double* z = xS + l * nr;
    double cc = 0.0, f = 0.0;
    if (Cs) {
      const size_t off = (static_cast<size_t>(l) * nr + p) * nr;
      if (c != 0.0)
        for (int k = 0; k < nr; ++k) cc = fma(__ldg(Cs + off + k), z[k], cc);
      if (l >= 1)
        for (int k = 0; k < nr; ++k) f = fma(__ldg(Alo + off + k), z[k - nr], f);
      if (l + 1 < nl)
        for (int k = 0; k < nr; ++k) f = fma(__ldg(Aup + off + k), z[k + nr], f);
      g[idx] = c * cc + e * f;
      continue;
    }
    if (c != 0.0) {
      if (l > 0) {
        const double* row = ro.band + static_cast<size_t>(p) * bw + w - p;
        for (int k = k0; k <= k1; ++k) cc = fma(__ldg(row + k), z[k], cc);
      } else {
        const double* row = ro.c0 + static_cast<size_t>(p) * nr;
        for (int k = k0; k < nr; ++k) cc = fma(__ldg(row + k), z[k], cc);
      }
    }
    if (l >= 1) {
      const double* row = ro.fband + (static_cast<size_t>(l) * nr + p) * bw + w - p;
      for (int k = k0; k <= k1; ++k) f = fma(__ldg(row + k), z[k - nr], f);
    }
    if (l + 1 < nl) {
      const double* row = ro.fband + (static_cast<size_t>(nl + l) * nr + p) * bw + w - p;
      for (int k = k0; k <= k1; ++k) f = fma(__ldg(row + k), z[k + nr], f);
    }
    g[idx] = c * cc + e * f;
  }
  __syncthreads();
  if (!Cs) {
    for (int l = threadIdx.x; l < nl; l += blockDim.x) bte::mass_solve(g + l * nr, ro.chol, ro.cinv, nr, w);
    __syncthreads();
  }
  double* o = out + static_cast<size_t>(i) * nv;
  for (int v = threadIdx.x; v < hc * nr; v += blockDim.x) {
    const int a = v / nr, p = v % nr;
    double se = 0.0, so = 0.0;
    for (int l = 0; l < nl; l += 2) {
      se = fma(__ldg(TO + a * nl + l), g[l * nr + p], se);
      if (l + 1 < nl) so = fma(__ldg(TO + a * nl + l + 1), g[(l + 1) * nr + p], so);
    }
    o[v] = se + so;
    if (a < hf) o[(nt - 1 - a) * nr + p] = se - so;
  }
}

// out = X + s0 Y0 + dt (Zx - VX) - dt El_i KAF_i  (El, KAF may be NULL), except the inflow rows of
// each ordinate (x = 0 for mu >= 0, x = L otherwise), where out = X.
__global__ void implicit_combine_kernel(const double* __restrict__ X, const double* __restrict__ Y0, double s0,
                                        const double* __restrict__ Zx, const double* __restrict__ VX,
                                        const double* __restrict__ El, const double* __restrict__ KAF,
                                        const double* __restrict__ mu, double dt, int nx, int nt, int nr,
                                        double* __restrict__ out) {
  const size_t n = static_cast<size_t>(nx) * nt * nr;
  for (size_t e = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; e < n;
       e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int i = static_cast<int>(e / (static_cast<size_t>(nt) * nr));
    const int a = static_cast<int>((e / nr) % nt);
    const bool inflow = mu[a] >= 0.0 ? i == 0 : i == nx - 1;
    double v = X[e];
    if (!inflow) {
      if (Y0) v += s0 * Y0[e];
      double r = Zx[e] - VX[e];
      if (El) r -= El[i] * KAF[e];
      v += dt * r;
    }
    out[e] = v;
  }
}

// partial[blk][j] = sum over this block's elements of V_j . w, j < k (V_j = V + j ld). blockIdx.y takes
// eight of the vectors: w is read once for them and their block sums share the barriers.
constexpr int kDotVec = 8;
static_assert(kDotVec == kDotBlock / 32, "one warp per vector");
__global__ void __launch_bounds__(kDotBlock) multi_dot_kernel(const double* __restrict__ V, size_t ld, int k,
                                                              const double* __restrict__ w, size_t n,
                                                              double* __restrict__ partial) {
  __shared__ double red[kDotVec][kDotBlock];
  const int j0 = blockIdx.y * kDotVec, nj = min(kDotVec, k - j0), lane = threadIdx.x & 31;
  const double* v = V + j0 * ld;
  double s[kDotVec];
#pragma unroll
  for (int j = 0; j < kDotVec; ++j) s[j] = 0.0;
  for (size_t e = blockIdx.x * static_cast<size_t>(kDotBlock) + threadIdx.x; e < n;
       e += static_cast<size_t>(gridDim.x) * kDotBlock) {
    const double we = w[e];
#pragma unroll
    for (int j = 0; j < kDotVec; ++j)
      if (j < nj) s[j] = fma(v[j * ld + e], we, s[j]);
  }
#pragma unroll
  for (int j = 0; j < kDotVec; ++j) red[j][threadIdx.x] = s[j];
  __syncthreads();
  // warp j sums vector j: FP64 additions bound this part, so it takes 13 of them where a shuffle tree
  // in every warp takes 40
  const int j = threadIdx.x >> 5;
  if (j < nj) {
    double t = 0.0;
#pragma unroll
    for (int q = 0; q < kDotBlock / 32; ++q) t += red[j][lane + 32 * q];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) partial[static_cast<size_t>(blockIdx.x) * k + j0 + j] = t;
  }
}

// out[j] = sum over blocks of partial[blk][j]: one CTA per j, strided partial sums then a tree
// (a fixed order, so the result is reproducible); with status its word goes to out[k]
__global__ void sum_partials_kernel(const double* __restrict__ partial, int nblk, int k, double* __restrict__ out,
                                    const unsigned* status) {
  __shared__ double red[32];
  const int j = blockIdx.x;
  double s = 0.0;
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += partial[static_cast<size_t>(b) * k + j];
  s = block_sum(s, red);
  if (threadIdx.x == 0) out[j] = s;
  if (status && j == 0 && threadIdx.x == 0) out[k] = *status;
}

// w = a w + sg sum_{j<k} c_j V_j   (c in device memory)
__global__ void multi_axpy_kernel(double* __restrict__ w, double a, const double* __restrict__ V, size_t ld, int k,
                                  const double* __restrict__ c, double sg, size_t n) {
  for (size_t e = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; e < n;
       e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    double s = 0.0;
    for (int j = 0; j < k; ++j) s = fma(c[j], V[j * ld + e], s);
    w[e] = (a == 0.0 ? 0.0 : a * w[e]) + sg * s;
  }
}

// y += a x
__global__ void axpy_kernel(double* __restrict__ y, double a, const double* __restrict__ x, size_t n) {
  for (size_t e = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; e < n;
       e += static_cast<size_t>(gridDim.x) * blockDim.x)
    y[e] = fma(a, x[e], y[e]);
}

// x *= a
__global__ void scale_kernel(double* __restrict__ x, double a, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) x[i] *= a;
}

}  // namespace

namespace bte {
namespace {

bte_status hfail(const bte_handle* h, bte_status s, const std::string& m) { return handle_fail(h, s, m); }

#define BH_CUDA(h, call)                                                                          \
  do {                                                                                            \
    cudaError_t e_ = (call);                                                                      \
    if (e_ != cudaSuccess) return hfail((h), BTE_ECUDA, std::string(#call ": ") + cudaGetErrorString(e_)); \
  } while (0)

template <typename T>
bte_status halloc(bte_handle* h, T** p, size_t count) {
  void* q = nullptr;
  const cudaError_t e = cudaMalloc(&q, std::max<size_t>(count * sizeof(T), 16));
  if (e != cudaSuccess) return hfail(h, BTE_ENOMEM, std::string("cudaMalloc failed: ") + cudaGetErrorString(e));
  h->allocs.push_back(q);
  h->bytes += count * sizeof(T);
  *p = static_cast<T*>(q);
  return BTE_OK;
}

template <typename T>
bte_status hupload(bte_handle* h, T** p, const std::vector<T>& v) {
  bte_status s = halloc(h, p, v.size());
  if (s != BTE_OK) return s;
  BH_CUDA(h, cudaMemcpyAsync(*p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, h->st));
  BH_CUDA(h, cudaStreamSynchronize(h->st));
  return BTE_OK;
}

int vec_grid(size_t n) { return static_cast<int>(std::min<size_t>((n + 255) / 256, 1216)); }

// Operators of the self-consistent parts, assembled and uploaded on first use.
bte_status hybrid_setup(bte_handle* h) {
  if (h->hybrid) return BTE_OK;
  const HostOps& o = h->ops;
  if (!o.have_v) return hfail(h, BTE_ESTATE, "set the cross sections first");
  std::vector<double> Lop, E1;
  const std::string e = assemble_field(o, Lop, E1);
  if (!e.empty()) return hfail(h, BTE_EINVAL, e);
  std::vector<double> rion(o.nv, 0.0);
  for (size_t j = 0; j < h->procs.size(); ++j)
    if (h->procs[j].kind == BTE_IONIZATION) {
      std::copy(o.mom_r.begin() + j * o.nv, o.mom_r.begin() + (j + 1) * o.nv, rion.begin());
      break;
    }
  bte_status s = BTE_OK;
  if (s == BTE_OK) s = hupload(h, &h->Lop, Lop);
  if (s == BTE_OK) s = hupload(h, &h->E1, E1);
  if (s == BTE_OK) s = hupload(h, &h->Dxd, o.Dx);
  if (s == BTE_OK) s = hupload(h, &h->DxT, o.Dx);
  if (s == BTE_OK) launch_transpose_blocks(h->DxT, o.nx, 1, h->st);
  if (s == BTE_OK) s = hupload(h, &h->mud, o.mu);
  if (s == BTE_OK) s = hupload(h, &h->lamd, o.lam);
  if (s == BTE_OK) s = hupload(h, &h->rion, rion);
  if (s == BTE_OK) s = halloc(h, &h->D2, static_cast<size_t>(o.nx) * o.nx);
  if (s == BTE_OK) square_kernel<<<o.nx, 256, 0, h->st>>>(h->Dxd, o.nx, h->D2);
  if (s == BTE_OK) s = halloc(h, &h->Esc, o.nx);
  if (s == BTE_OK) s = halloc(h, &h->ned, o.nx);
  if (s == BTE_OK) s = halloc(h, &h->Ek, o.nx);
  if (s == BTE_OK) s = halloc(h, &h->ionA, static_cast<size_t>(o.nx) * o.nx);
  if (s == BTE_OK) s = halloc(h, &h->ionb, o.nx);
  if (s != BTE_OK) return s;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(v_apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
    attr = true;
  }
  h->hybrid = true;
  return BTE_OK;
}

// Work vectors of the fully-implicit step for a GMRES basis of m + 1 vectors.
bte_status implicit_setup(bte_handle* h, int m, bool full_q) {
  bte_status s = BTE_OK;
  if (full_q && !h->Qfull) {
    // Q_ij for a full step, (I + dt lam_i mu_a D_x)^-1 with the inflow rows
    std::vector<double> Q;
    if (!assemble_q(h->ops, h->ops.dt, Q)) return hfail(h, BTE_EINVAL, "a full-step x operator is singular");
    if ((s = hupload(h, &h->Qfull, Q)) != BTE_OK) return s;
    launch_transpose_blocks(h->Qfull, h->ops.nx, static_cast<size_t>(h->ops.nt) * h->ops.nr, h->st);
  }
  if (h->gm >= m) return BTE_OK;
  const size_t D = static_cast<size_t>(h->ops.nx) * h->ops.nv;
  if (!h->Fk) {
    for (double** p : {&h->Fk, &h->Fn, &h->Rv, &h->Zx, &h->VX, &h->KAF, &h->Wv, &h->Pz, &h->Dl})
      if (s == BTE_OK) s = halloc(h, p, D);
    if (s == BTE_OK) s = halloc(h, &h->El, h->ops.nx);
  }
  if (s == BTE_OK) s = halloc(h, &h->Vb, D * (m + 1));
  if (s == BTE_OK) s = halloc(h, &h->Zb, D * m);
  if (s == BTE_OK) s = halloc(h, &h->part, static_cast<size_t>(kDotGrid) * (m + 1));
  if (s == BTE_OK) s = halloc(h, &h->dsum, 3 * (m + 1));  // two Gram-Schmidt passes and a norm
  if (s != BTE_OK) return s;
  if (h->dsum_host) cudaFreeHost(h->dsum_host);
  BH_CUDA(h, cudaMallocHost(reinterpret_cast<void**>(&h->dsum_host), 3 * (m + 1) * sizeof(double)));
  h->gm = m;
  return BTE_OK;
}

// A_x X D_x^T (per ordinate mu_a D_x X_a G^T, G = M_v^-1 G_v) through the eigen basis of G; X NULL: of
// the vector whose eigen coefficients are in Y2
void enqueue_xop(bte_handle* h, const double* X, double* out) {
  const HostOps& o = h->ops;
  cudaStream_t st = h->st;
  double *in = h->Y2, *mid = h->Y;
  if (X) {
    std::swap(in, mid);
    launch_x_to_eigen(X, h->Uinv, in, o.nx, o.nt, o.nr, h->status, st);
  }
  launch_x_matvec(h->DxT, false, h->lamd, h->mud, in, mid, o.nx, o.nt, o.nr, st);  // lam_i mu_a D_x Y
  launch_x_from_eigen(mid, h->U, out, o.nx, o.nt, o.nr, nullptr, st);
}

void enqueue_vapply(bte_handle* h, const double* X, const double* E, double c, double* out) {
  const HostOps& o = h->ops;
  const size_t smem = sizeof(double) * o.nr * (2 * ((o.nt + 1) / 2) + 2 * static_cast<size_t>(o.nl));
  v_apply_kernel<<<o.nx, 256, smem, h->st>>>(X, E, c, handle_residual_ops(h), o.nl * o.nr <= 400 ? h->Cs : nullptr, h->Alo,
                                          h->Aup, h->TO, h->TS, out, o.nt, o.nr, o.nl);
}

// out_dev[j] = V_j . w for j < k on the device (stream-ordered; no host synchronisation); with status the
// handle's status word follows as out_dev[k]
void enqueue_dots(bte_handle* h, const double* V, size_t ld, int k, const double* w, double* out_dev,
                  bool status = false) {
  const size_t D = static_cast<size_t>(h->ops.nx) * h->ops.nv;
  multi_dot_kernel<<<dim3(dot_grid(D), (k + kDotVec - 1) / kDotVec), kDotBlock, 0, h->st>>>(V, ld, k, w, D, h->part);
  sum_partials_kernel<<<k, 128, 0, h->st>>>(h->part, dot_grid(D), k, out_dev, status ? h->status : nullptr);
}

// dots[j] = V_j . w for j < k into the pinned host array (synchronises the stream)
bte_status host_dots(bte_handle* h, const double* V, size_t ld, int k, const double* w, std::vector<double>& out) {
  const size_t D = static_cast<size_t>(h->ops.nx) * h->ops.nv;
  multi_dot_kernel<<<dim3(dot_grid(D), (k + kDotVec - 1) / kDotVec), kDotBlock, 0, h->st>>>(V, ld, k, w, D, h->part);
  sum_partials_kernel<<<k, 128, 0, h->st>>>(h->part, dot_grid(D), k, h->dsum, nullptr);
  BH_CUDA(h, cudaMemcpyAsync(h->dsum_host, h->dsum, k * sizeof(double), cudaMemcpyDeviceToHost, h->st));
  BH_CUDA(h, cudaStreamSynchronize(h->st));
  out.assign(h->dsum_host, h->dsum_host + k);
  return BTE_OK;
}

}  // namespace

bte_status enqueue_field(bte_handle* h, const double* F_dev, const double* ni_dev, double t, double V0,
                         double freq, double* E_dev) {
  const HostOps& o = h->ops;
  point_dot_kernel<<<o.nx, 256, 0, h->st>>>(F_dev, h->mom_n, o.nv, h->ned);
  const double vleft = V0 * std::sin(2.0 * kPi * freq * t);
  field_kernel<<<(o.nx * 32 + 255) / 256, 256, 0, h->st>>>(h->Lop, h->E1, ni_dev, h->ned, vleft, o.nx, E_dev);
  handle_add_launches(h, 2);
  BH_CUDA(h, cudaGetLastError());
  return BTE_OK;
}

}  // namespace bte

// ---------------------------------------------------------------------------------- entry points

using bte::hfail;

extern "C" {

bte_status bte_set_ion_transport(bte_handle* h, double n0_mu_i, double n0_D_i) {
  if (!h) return hfail(nullptr, BTE_EINVAL, "handle is NULL");
  if (!(n0_mu_i >= 0.0) || !(n0_D_i > 0.0) || !std::isfinite(n0_mu_i) || !std::isfinite(n0_D_i))
    return hfail(h, BTE_EINVAL, "ion mobility must be >= 0 and ion diffusion > 0 (both finite)");
  h->n0_mu_i = n0_mu_i;
  h->n0_D_i = n0_D_i;
  return BTE_OK;
}

bte_status bte_field(bte_handle* h, const double* F_dev, const double* ni_dev, double t_s, double V0,
                     double freq_Hz, double* E_dev) {
  if (!h) return hfail(nullptr, BTE_EINVAL, "handle is NULL");
  if (!F_dev || !E_dev) return hfail(h, BTE_EINVAL, "F_dev and E_dev must not be NULL");
  {
    const bte_status ds = bte::handle_device_status(h);
    if (ds != BTE_OK) return ds;
  }
  bte_status s = bte::hybrid_setup(h);
  if (s != BTE_OK) return s;
  return bte::enqueue_field(h, F_dev, ni_dev, t_s, V0, freq_Hz, E_dev);
}

bte_status bte_ion_step(bte_handle* h, double* ni_dev, const double* F_dev, double t_s, double V0,
                        double freq_Hz) {
  if (!h) return hfail(nullptr, BTE_EINVAL, "handle is NULL");
  if (!ni_dev || !F_dev) return hfail(h, BTE_EINVAL, "ni_dev and F_dev must not be NULL");
  {
    const bte_status ds = bte::handle_device_status(h);
    if (ds != BTE_OK) return ds;
  }
  bte_status s = bte::hybrid_setup(h);
  if (s != BTE_OK) return s;
  const bte::HostOps& o = h->ops;
  cudaStream_t st = h->st;
  BH_CUDA(h, cudaMemsetAsync(h->status, 0, 2 * sizeof(unsigned), st));
  // E^n from (n_i^n, F^n) at t_n, then the source n0 r_ion . F^n, the system, its solve
  s = bte::enqueue_field(h, F_dev, ni_dev, t_s, V0, freq_Hz, h->Esc);
  if (s != BTE_OK) return s;
  point_dot_kernel<<<o.nx, 256, 0, st>>>(F_dev, h->rion, o.nv, h->ned);
  scale_kernel<<<(o.nx + 255) / 256, 256, 0, st>>>(h->ned, o.n0, o.nx);
  ion_assemble_kernel<<<o.nx, 256, 0, st>>>(h->Dxd, h->D2, h->Esc, ni_dev, h->ned, h->n0_mu_i / o.n0, h->n0_D_i / o.n0,
                                           o.dt, o.nx, h->ionA, h->ionb);
  {
    const bool fits = o.nx <= kSmemSolve;
    const size_t smem = ion_smem(o.nx, fits);
    auto solve = fits ? dense_solve_kernel<true> : dense_solve_kernel<false>;
    BH_CUDA(h, bte::set_smem_limit(solve, fits ? ion_smem(kSmemSolve, true) : ion_smem(4096, false)));  // nx <= 4096
    solve<<<1, fits ? 256 : 512, smem, st>>>(h->ionA, h->ionb, o.nx, h->ned, h->status);
  }
  bte::launch_commit(h->ned, ni_dev, o.nx, h->status, st);
  bte::handle_add_launches(h, 5);
  BH_CUDA(h, cudaGetLastError());
  return bte::handle_read_status(h);
}

bte_status bte_step_sc(bte_handle* h, double* F_dev, const double* ni_dev, double t_s, double V0, double freq_Hz,
                       double* E_out_dev) {
  if (!h) return hfail(nullptr, BTE_EINVAL, "handle is NULL");
  if (!F_dev || !ni_dev) return hfail(h, BTE_EINVAL, "F_dev and ni_dev must not be NULL");
  {
    const bte_status ds = bte::handle_device_status(h);
    if (ds != BTE_OK) return ds;
  }
  bte_status s = bte::hybrid_setup(h);
  if (s != BTE_OK) return s;
  BH_CUDA(h, cudaMemsetAsync(h->status, 0, 2 * sizeof(unsigned), h->st));
  s = bte::handle_enqueue_sc_step(h, F_dev, ni_dev, t_s, V0, freq_Hz);
  if (s != BTE_OK) return s;
  if (E_out_dev)
    BH_CUDA(h, cudaMemcpyAsync(E_out_dev, h->Esc, h->ops.nx * sizeof(double), cudaMemcpyDeviceToDevice, h->st));
  return bte::handle_read_status(h);
}

bte_status bte_step_implicit(bte_handle* h, double* F_dev, const double* ni_dev, double t_s, double V0,
                             double freq_Hz, bte_implicit_opts* opts) {
  if (!h) return hfail(nullptr, BTE_EINVAL, "handle is NULL");
  if (!F_dev || !ni_dev) return hfail(h, BTE_EINVAL, "F_dev and ni_dev must not be NULL");
  {
    const bte_status ds = bte::handle_device_status(h);
    if (ds != BTE_OK) return ds;
  }
  double rtol = 1e-10, grtol = 1e-2;
  int newton_max = 8, m = 100, gmax = 400, precond = 0;
  if (opts) {
    if (opts->newton_rtol > 0) rtol = opts->newton_rtol;
    if (opts->gmres_rtol > 0) grtol = opts->gmres_rtol;
    if (opts->newton_max > 0) newton_max = opts->newton_max;
    if (opts->gmres_restart > 0) m = opts->gmres_restart;
    if (opts->gmres_max > 0) gmax = opts->gmres_max;
    precond = opts->precond;
    opts->newton_iters = opts->gmres_iters = 0;
    opts->residual = 0.0;
  }
  if (m > 200) return hfail(h, BTE_EINVAL, "gmres_restart must be <= 200");
  if (precond != 0 && precond != 1) return hfail(h, BTE_EINVAL, "precond must be 0 or 1");
  bte_status s = bte::hybrid_setup(h);
  if (s == BTE_OK) s = bte::implicit_setup(h, m, precond == 0);
  if (s != BTE_OK) return s;
  const bte::HostOps& o = h->ops;
  const int nx = o.nx, nt = o.nt, nr = o.nr;
  const size_t D = static_cast<size_t>(nx) * o.nv;
  const double dt = o.dt, t1 = t_s + dt;
  cudaStream_t st = h->st;
  const int vg = bte::vec_grid(D);
  unsigned long long launches = 0;

  // F^n, and the initial iterate: the semi-implicit self-consistent step from F^n (F^n itself if
  // that step does not factor or converge)
  BH_CUDA(h, cudaMemsetAsync(h->status, 0, 2 * sizeof(unsigned), st));
  BH_CUDA(h, cudaMemcpyAsync(h->Fn, F_dev, D * sizeof(double), cudaMemcpyDeviceToDevice, st));
  BH_CUDA(h, cudaMemcpyAsync(h->Fk, F_dev, D * sizeof(double), cudaMemcpyDeviceToDevice, st));
  s = bte::handle_enqueue_sc_step(h, h->Fk, ni_dev, t_s, V0, freq_Hz);
  if (s != BTE_OK) return s;
  s = bte::handle_read_status(h);
  if (s == BTE_ENONFINITE || s == BTE_ECUDA) return s;
  BH_CUDA(h, cudaMemsetAsync(h->status, 0, 2 * sizeof(unsigned), st));

  auto residual = [&](const double* X, double* R) {
    bte::enqueue_field(h, X, ni_dev, t1, V0, freq_Hz, h->Esc);
    bte::enqueue_xop(h, X, h->Zx);
    bte::enqueue_vapply(h, X, h->Esc, 1.0, h->VX);
    implicit_combine_kernel<<<vg, 256, 0, st>>>(X, h->Fn, -1.0, h->Zx, h->VX, nullptr, nullptr, h->mud, dt, nx, nt,
                                                nr, R);
    launches += 7;
  };
  auto norm = [&](const double* X, double& out) -> bte_status {
    std::vector<double> d;
    const bte_status r = bte::host_dots(h, X, 0, 1, X, d);
    out = std::sqrt(d[0]);
    launches += 2;
    return r;
  };
  // the preconditioner at the frozen field Ek, from the split step's pieces with the factors of
  // this Newton iteration. precond 0: the per-point solves, then one full x step (exact when either
  // part vanishes, also for the stiffest x modes); 1: the semi-implicit step's map (x half step,
  // solves, x half step), whose x part is (I + dt/2 A_x)^-2, far from (I + dt A_x)^-1 for x modes
  // with dt |A_x| >> 1
  auto pinv = [&](const double* in, double* out) -> bte_status {
    bte_status r = BTE_OK;
    if (precond == 0) {
      r = bte::handle_enqueue_vsolve(h, in, h->VX, h->Ek, false);
      if (r == BTE_OK) {
        bte::launch_x_to_eigen(h->VX, h->Uinv, h->Y, nx, nt, nr, nullptr, st);
        bte::launch_x_apply_q(h->Qfull, h->Y, h->Y2, nx, nt, nr, st);
        bte::launch_x_from_eigen(h->Y2, h->U, out, nx, nt, nr, nullptr, st);
        launches += 3;
      }
    } else {
      r = bte::handle_enqueue_xhalf(h, in, h->Wv);
      if (r == BTE_OK) r = bte::handle_enqueue_vsolve(h, h->Wv, h->VX, h->Ek, false);
      if (r == BTE_OK) r = bte::handle_enqueue_xhalf(h, h->VX, out);
    }
    return r;
  };
  // Jacobian action at F_k (eq. "1dbte_jac_action" with the inflow rows as identity). in_eigen: X is the
  // x step's last result, whose eigen coefficients are still in Y2 (the transform there and back is left out)
  auto jac = [&](const double* X, double* out, bool in_eigen = false) {
    point_dot_kernel<<<nx, 256, 0, st>>>(X, h->mom_n, o.nv, h->ned);
    field_kernel<<<(nx * 32 + 255) / 256, 256, 0, st>>>(h->Lop, h->E1, nullptr, h->ned, 0.0, nx, h->El);
    bte::enqueue_xop(h, in_eigen ? nullptr : X, h->Zx);
    bte::enqueue_vapply(h, X, h->Ek, 1.0, h->VX);
    implicit_combine_kernel<<<vg, 256, 0, st>>>(X, nullptr, 0.0, h->Zx, h->VX, h->El, h->KAF, h->mud, dt, nx, nt,
                                                nr, out);
    launches += 7;
  };

  double fn = 0.0, rn = 0.0;
  if ((s = norm(h->Fn, fn)) != BTE_OK) return s;
  residual(h->Fk, h->Rv);
  if ((s = norm(h->Rv, rn)) != BTE_OK) return s;
  bool conv = rn <= rtol * fn;
  int newton = 0, gm_total = 0;
  std::vector<double> H(static_cast<size_t>(m + 1) * m), cs(m), sn(m), g(m + 1), y(m);
  // forcing term of the current Newton iteration: a failed line search (no sufficient decrease
  // along a direction GMRES solved only to grtol) retries the iteration with a 100x tighter
  // linear solve, at most twice, before the step gives up
  double eta = grtol;
  int retries = 0;
  while (!conv && newton < newton_max) {
    // the iterate's field, frozen for the preconditioner and the Jacobian; factors at that field
    BH_CUDA(h, cudaMemcpyAsync(h->Ek, h->Esc, nx * sizeof(double), cudaMemcpyDeviceToDevice, st));
    if ((s = bte::handle_enqueue_vsolve(h, h->Rv, h->Pz, h->Ek, true)) != BTE_OK) return s;
    bte::enqueue_vapply(h, h->Fk, nullptr, 0.0, h->KAF);
    // restarted GMRES on J delta = -R, right-preconditioned: delta accumulates in Dl; every cycle
    // solves J P^-1 y = r for the current residual r = -R - J delta
    BH_CUDA(h, cudaMemsetAsync(h->Dl, 0, D * sizeof(double), st));
    int inner = 0;
    double rc = rn;  // |r| of the current cycle
    for (int cyc = 0; inner < gmax; ++cyc) {
      if (cyc > 0) {
        jac(h->Dl, h->Vb);  // r = -R - J delta
        multi_axpy_kernel<<<vg, 256, 0, st>>>(h->Vb, -1.0, nullptr, D, 0, nullptr, 0.0, D);
        axpy_kernel<<<vg, 256, 0, st>>>(h->Vb, -1.0, h->Rv, D);
        if ((s = norm(h->Vb, rc)) != BTE_OK) return s;
        if (rc <= eta * rn) break;
        multi_axpy_kernel<<<vg, 256, 0, st>>>(h->Vb, 1.0 / rc, nullptr, D, 0, nullptr, 0.0, D);
      } else {
        BH_CUDA(h, cudaMemcpyAsync(h->Vb, h->Rv, D * sizeof(double), cudaMemcpyDeviceToDevice, st));
        multi_axpy_kernel<<<vg, 256, 0, st>>>(h->Vb, -1.0 / rn, nullptr, D, 0, nullptr, 0.0, D);
      }
      std::fill(H.begin(), H.end(), 0.0);
      std::fill(g.begin(), g.end(), 0.0);
      g[0] = rc;
      int k = 0;
      bool done = false;
      for (int j = 0; j < m && inner < gmax; ++j, ++inner) {
        double* Vj = h->Vb + static_cast<size_t>(j) * D;
        double* Vn = h->Vb + static_cast<size_t>(j + 1) * D;
        double* Zj = h->Zb + static_cast<size_t>(j) * D;
        if ((s = pinv(Vj, Zj)) != BTE_OK) return s;
        jac(Zj, Vn, precond == 0);
        // classical Gram-Schmidt twice, then the norm: the projections stay on the device (the
        // axpys read them there), so the host waits once per iteration for all three results
        const size_t stride = static_cast<size_t>(m) + 1;
        for (int pass = 0; pass < 2; ++pass) {
          double* dp = h->dsum + pass * stride;
          bte::enqueue_dots(h, h->Vb, D, j + 1, Vn, dp);
          multi_axpy_kernel<<<vg, 256, 0, st>>>(Vn, 1.0, h->Vb, D, j + 1, dp, -1.0, D);
          launches += 3;
        }
        bte::enqueue_dots(h, Vn, 0, 1, Vn, h->dsum + 2 * stride, true);
        launches += 2;
        BH_CUDA(h, cudaMemcpyAsync(h->dsum_host, h->dsum, 3 * stride * sizeof(double), cudaMemcpyDeviceToHost, st));
        BH_CUDA(h, cudaStreamSynchronize(st));
        // an expired wait: every further solve would take its 2 s too, for nothing
        if (static_cast<unsigned>(h->dsum_host[2 * stride + 1]) & bte::kTimeout) return bte::handle_read_status(h);
        for (int i = 0; i <= j; ++i) H[static_cast<size_t>(i) * m + j] += h->dsum_host[i] + h->dsum_host[stride + i];
        const double hn = std::sqrt(h->dsum_host[2 * stride]);
        H[static_cast<size_t>(j + 1) * m + j] = hn;
        if (hn > 0.0) multi_axpy_kernel<<<vg, 256, 0, st>>>(Vn, 1.0 / hn, nullptr, D, 0, nullptr, 0.0, D);
        for (int i = 0; i < j; ++i) {  // earlier rotations on the new column
          const double a = H[static_cast<size_t>(i) * m + j], b = H[static_cast<size_t>(i + 1) * m + j];
          H[static_cast<size_t>(i) * m + j] = cs[i] * a + sn[i] * b;
          H[static_cast<size_t>(i + 1) * m + j] = -sn[i] * a + cs[i] * b;
        }
        const double a = H[static_cast<size_t>(j) * m + j], b = H[static_cast<size_t>(j + 1) * m + j];
        const double r = std::hypot(a, b);
        cs[j] = r > 0.0 ? a / r : 1.0;
        sn[j] = r > 0.0 ? b / r : 0.0;
        H[static_cast<size_t>(j) * m + j] = r;
        H[static_cast<size_t>(j + 1) * m + j] = 0.0;
        g[j + 1] = -sn[j] * g[j];
        g[j] = cs[j] * g[j];
        k = j + 1;
        if (std::fabs(g[j + 1]) <= eta * rn || hn == 0.0) {
          done = true;
          ++inner;
          break;
        }
      }
      for (int i = k - 1; i >= 0; --i) {  // H y = g, upper triangular
        double v = g[i];
        for (int q = i + 1; q < k; ++q) v -= H[static_cast<size_t>(i) * m + q] * y[q];
        y[i] = v / H[static_cast<size_t>(i) * m + i];
      }
      // delta += Z y with the stored Z_j = P^-1 V_j (flexible GMRES): the Arnoldi relation
      // J Z = V H holds for whatever the preconditioner returned, so the residual the rotations
      // track is the true one even where the FP32 solves inside P^-1 are far from linear (stiff
      // velocity systems: relative rounding kappa eps_32 of order one)
      std::copy(y.begin(), y.begin() + k, h->dsum_host);
      BH_CUDA(h, cudaMemcpyAsync(h->dsum, h->dsum_host, k * sizeof(double), cudaMemcpyHostToDevice, st));
      multi_axpy_kernel<<<vg, 256, 0, st>>>(h->Dl, 1.0, h->Zb, D, k, h->dsum, 1.0, D);
      if (done) break;
    }
    gm_total += inner;
    // backtracking on |R|
    double lam = 1.0, rt = 0.0;
    bool acc = false;
    for (int ls = 0; ls < 8 && !acc; ++ls) {
      BH_CUDA(h, cudaMemcpyAsync(h->Wv, h->Fk, D * sizeof(double), cudaMemcpyDeviceToDevice, st));
      axpy_kernel<<<vg, 256, 0, st>>>(h->Wv, lam, h->Dl, D);
      residual(h->Wv, h->Rv);
      if ((s = norm(h->Rv, rt)) != BTE_OK) return s;
      if (rt <= (1.0 - 1e-4 * lam) * rn) acc = true;
      else lam *= 0.5;
    }
    if (!acc) {
      if (retries < 2 && inner > 0) {
        eta *= 1e-2;
        ++retries;
        // the residual of the iterate again (the line search overwrote Rv and the field)
        residual(h->Fk, h->Rv);
        if ((s = norm(h->Rv, rn)) != BTE_OK) return s;
        continue;
      }
      ++newton;
      break;
    }
    ++newton;
    eta = grtol;
    retries = 0;
    std::swap(h->Fk, h->Wv);
    rn = rt;
    conv = rn <= rtol * fn;
  }
  bte::handle_add_launches(h, launches);
  BH_CUDA(h, cudaGetLastError());
  if (opts) {
    opts->newton_iters = newton;
    opts->gmres_iters = gm_total;
    opts->residual = fn > 0.0 ? rn / fn : rn;
  }
  s = bte::handle_read_status(h);
  if (s != BTE_OK) return s;
  if (!conv) return hfail(h, BTE_ENOCONV, "Newton did not reach newton_rtol");
  BH_CUDA(h, cudaMemcpyAsync(F_dev, h->Fk, D * sizeof(double), cudaMemcpyDeviceToDevice, st));
  BH_CUDA(h, cudaStreamSynchronize(st));
  return BTE_OK;
}

}  // extern "C"
