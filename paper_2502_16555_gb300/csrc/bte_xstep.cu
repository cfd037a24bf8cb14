// x half step (Algorithm 1 of arXiv 2502.16555), operator formation, FP64 refinement residual
// (Algorithm 2), moments and small helpers. All FP64 unless templated on the storage type.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "bte_kernels.h"
#include "bte_mass.cuh"

namespace bte {
namespace {

constexpr int kXT = 32;  // rows (ordinate, point) per CTA in the eigen-basis transforms
constexpr int kIC = 32;  // eigen (to) or B-spline (from) indices per CTA
constexpr int kG = 4;    // output indices per thread in the transforms (one staged operand, four FMAs)

__device__ __forceinline__ bool finite(double v) { return isfinite(v); }

// The rows of both transforms are the pairs m = a nx + x, taken 32 at a time without regard to where an
// ordinate ends (a tile per ordinate and 32 points left up to 31 of 32 lanes idle in the last tile: 72
// against 47 us of FP64 work at nx = 100, nr = 128).

// Y[a][i][x] = sum_k Uinv[i][k] F[x][a][k]  (the U^-1 contraction of Algorithm 1) for the kXT
// rows and kIC eigen indices of this CTA: a thread takes kG consecutive i at one row, a warp shares
// them (the Uinv rows are broadcasts) and its lanes run over the rows. Bound by the FP64 units. Flags
// non-finite inputs (blockIdx.y == 0 only), which is where a NaN handed in by the caller is first seen.
__global__ void x_to_eigen_kernel(const double* __restrict__ F, const double* __restrict__ Uinv,
                                  double* __restrict__ Y, int nx, int nt, int nr,
                                  unsigned* status) {
  extern __shared__ double sm[];
  const int m0 = blockIdx.x * kXT, i0 = blockIdx.y * kIC;
  const int nmt = min(kXT, nx * nt - m0), nit = min(kIC, nr - i0);
  const int ld = nr + 1;  // padded row
  const bool check = status && blockIdx.y == 0;
  bool bad = false;
  for (int r = threadIdx.x >> 5; r < nmt; r += blockDim.x >> 5) {
    const int a = (m0 + r) / nx, x = (m0 + r) % nx;
    const double* f = F + (static_cast<size_t>(x) * nt + a) * nr;
    for (int k = threadIdx.x & 31; k < nr; k += 32) {
      const double v = f[k];
      bad |= !finite(v);
      sm[r * ld + k] = v;
    }
  }
  if (check && bad) atomicOr(status, kNonFiniteIn);
  __syncthreads();
  const int ngr = (nit + kG - 1) / kG, xx = threadIdx.x % kXT;
  if (xx >= nmt) return;
  const int a = (m0 + xx) / nx, x = (m0 + xx) % nx;
  double* y = Y + static_cast<size_t>(a) * nr * nx + x;
  const double* f = sm + xx * ld;
  for (int grp = threadIdx.x / kXT; grp < ngr; grp += blockDim.x / kXT) {
    const int ib = i0 + grp * kG, nu = min(kG, i0 + nit - ib);
    const double* u = Uinv + static_cast<size_t>(ib) * nr;
    double s[kG];
#pragma unroll
    for (int g = 0; g < kG; ++g) s[g] = 0.0;
    if (nu == kG) {
#pragma unroll 4
      for (int k = 0; k < nr; ++k) {
        const double fv = f[k];
#pragma unroll
        for (int g = 0; g < kG; ++g) s[g] = fma(__ldg(u + static_cast<size_t>(g) * nr + k), fv, s[g]);
      }
    } else {
      for (int k = 0; k < nr; ++k)
#pragma unroll
        for (int g = 0; g < kG; ++g)
          if (g < nu) s[g] = fma(__ldg(u + static_cast<size_t>(g) * nr + k), f[k], s[g]);
    }
#pragma unroll
    for (int g = 0; g < kG; ++g)
      if (g < nu) y[static_cast<size_t>(ib + g) * nx] = s[g];
  }
}

// Y2[b] = s_b M_b Y[b] for every (ordinate, eigen-index) pair b = a nr + i; MT holds the transposes,
// M_b^T = MT + b mstride (mstride = nx^2: the per-pair Q_ij of Algorithm 1; 0: one shared matrix),
// s_b = lam[i] mu[a] when lam is given, else 1. One CTA per pair, one thread per row: a column of M is
// one coalesced read and every FP64 instruction is an FMA of the product (with M by rows a warp spent
// a fifth of them on its transposing reduction: 105 us on the medium grid, where the FMAs take 61
// at 1.1 TFLOP/s and the 268 MB 40).
__global__ void x_matvec_kernel(const double* __restrict__ MT, size_t mstride, const double* __restrict__ lam,
                                const double* __restrict__ mu, const double* __restrict__ Y,
                                double* __restrict__ Y2, int nx, int nr) {
  extern __shared__ double ys[];
  const size_t b = blockIdx.x;
  const double* y = Y + b * nx;
  for (int i = threadIdx.x; i < nx; i += blockDim.x) ys[i] = y[i];
  __syncthreads();
  const double* Mb = MT + b * mstride;
  for (int r = threadIdx.x; r < nx; r += blockDim.x) {
    const double* q = Mb + r;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    int c = 0;
    for (; c + 16 <= nx; c += 16) {
      double v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = __ldg(q + static_cast<size_t>(c + k) * nx);
#pragma unroll
      for (int k = 0; k < 16; ++k) acc[k & 3] = fma(v[k], ys[c + k], acc[k & 3]);
    }
    for (; c < nx; ++c) acc[0] = fma(__ldg(q + static_cast<size_t>(c) * nx), ys[c], acc[0]);
    const double s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    Y2[b * nx + r] = lam ? lam[b % nr] * mu[b / nr] * s : s;
  }
}

// In-place transpose of consecutive n x n matrices: tile pair (blockIdx.x <= blockIdx.y) of matrix
// blockIdx.z + z0.
__global__ void transpose_blocks_kernel(double* __restrict__ M, int n, size_t z0) {
  if (blockIdx.x > blockIdx.y) return;
  __shared__ double a[32][33], b[32][33];
  double* m = M + (z0 + blockIdx.z) * n * n;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32, tx = threadIdx.x & 31;
  for (int ty = threadIdx.x >> 5; ty < 32; ty += blockDim.x >> 5) {
    if (r0 + ty < n && c0 + tx < n) a[ty][tx] = m[static_cast<size_t>(r0 + ty) * n + c0 + tx];
    if (c0 + ty < n && r0 + tx < n) b[ty][tx] = m[static_cast<size_t>(c0 + ty) * n + r0 + tx];
  }
  __syncthreads();
  for (int ty = threadIdx.x >> 5; ty < 32; ty += blockDim.x >> 5) {
    if (r0 + ty < n && c0 + tx < n) m[static_cast<size_t>(r0 + ty) * n + c0 + tx] = b[tx][ty];
    if (c0 + ty < n && r0 + tx < n) m[static_cast<size_t>(c0 + ty) * n + r0 + tx] = a[tx][ty];
  }
}

// F[x][a][k] = sum_i U[k][i] Y2[a][i][x] for the kXT rows and kIC B-spline indices of this CTA:
// a thread takes kG consecutive k at one row, a warp shares them (the U rows are broadcasts) and its
// lanes run over the rows (consecutive shared-memory words); flags non-finite results.
__global__ void x_from_eigen_kernel(const double* __restrict__ Y2, const double* __restrict__ U,
                                    double* __restrict__ F, int nx, int nt, int nr,
                                    unsigned* status) {
  extern __shared__ double sm[];
  const int m0 = blockIdx.x * kXT, k0 = blockIdx.y * kIC;
  const int nmt = min(kXT, nx * nt - m0), nkt = min(kIC, nr - k0), xx = threadIdx.x % kXT;
  const int a = (m0 + xx) / nx, x = (m0 + xx) % nx;
  const double* y2 = Y2 + static_cast<size_t>(a) * nr * nx + x;
  for (int i = threadIdx.x / kXT; i < nr; i += blockDim.x / kXT)
    sm[i * (kXT + 1) + xx] = xx < nmt ? y2[static_cast<size_t>(i) * nx] : 0.0;
  __syncthreads();
  if (xx >= nmt) return;
  bool bad = false;
  const int ngr = (nkt + kG - 1) / kG;
  double* f = F + (static_cast<size_t>(x) * nt + a) * nr;
  for (int grp = threadIdx.x / kXT; grp < ngr; grp += blockDim.x / kXT) {
    const int kb = k0 + grp * kG, nu = min(kG, k0 + nkt - kb);
    const double* u = U + static_cast<size_t>(kb) * nr;
    double s[kG];
#pragma unroll
    for (int g = 0; g < kG; ++g) s[g] = 0.0;
    if (nu == kG) {
#pragma unroll 4
      for (int i = 0; i < nr; ++i) {
        const double y = sm[i * (kXT + 1) + xx];
#pragma unroll
        for (int g = 0; g < kG; ++g) s[g] = fma(__ldg(u + static_cast<size_t>(g) * nr + i), y, s[g]);
      }
    } else {
      for (int i = 0; i < nr; ++i)
#pragma unroll
        for (int g = 0; g < kG; ++g)
          if (g < nu) s[g] = fma(__ldg(u + static_cast<size_t>(g) * nr + i), sm[i * (kXT + 1) + xx], s[g]);
    }
#pragma unroll
    for (int g = 0; g < kG; ++g)
      if (g < nu) {
        bad |= !finite(s[g]);
        f[kb + g] = s[g];
      }
  }
  if (status && bad) atomicOr(status, kNonFinite);
}

template <typename T>
__global__ void v_form_kernel(const double* __restrict__ KCg, const double* __restrict__ KAg, MassBand mass,
                              const double* __restrict__ E, double E_uniform, double dt,
                              T* __restrict__ fac, int nx, int nv) {
  // Per element, base = M - dt KCg and slope = -dt KAg once in FP64; per point, one FMA in the
  // factor precision, base + E_i slope (for FP32 factors an FP32 FMA: GB300's FP64 rate would bound
  // the Nx FP64 operations per element at about eight times the store time). A per-point field is
  // staged in shared memory in that precision; the uniform field takes the same arithmetic, so
  // equal fields give equal factors on both paths.
  extern __shared__ __align__(8) unsigned char vf_smem[];
  T* Es = reinterpret_cast<T*>(vf_smem);
  if (E) {
    for (int i = threadIdx.x; i < nx; i += blockDim.x) Es[i] = static_cast<T>(E[i]);
    __syncthreads();
  }
  const T Eu = static_cast<T>(E_uniform);
  const size_t nn = static_cast<size_t>(nv) * nv;
  const int nr = mass.nr, bw = 2 * mass.w + 1;
  for (size_t e = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; e < nn;
       e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const double kc = KCg[e], ka = KAg[e];
    // (I (x) M_v)[(a,p),(b,k)] = M_v[p][k] when a == b and |p - k| <= w
    const int row = static_cast<int>(e / nv), col = static_cast<int>(e % nv);
    const int p = row % nr, k = col % nr, dk = k - p;
    const double d = (row - p == col - k && dk >= -mass.w && dk <= mass.w) ? __ldg(mass.m + p * bw + dk + mass.w) : 0.0;
    const T base = static_cast<T>(d - dt * kc), slope = static_cast<T>(-dt * ka);
    if (E) {
      for (int i = 0; i < nx; ++i) fac[static_cast<size_t>(i) * nn + e] = Es[i] * slope + base;
    } else {
      const T v = Eu * slope + base;
      for (int i = 0; i < nx; ++i) fac[static_cast<size_t>(i) * nn + e] = v;
    }
  }
}

// Refinement residual of one point (CTA per point), Algorithm 2 with the structured operators:
// xS = P_S x, g = M_v^-1 (C + E_i A_v) xS, r = b - x + dt P_O g. The products with C and A_v run
// over bands (the loss part of C, the field blocks; C_0 carries the gain and the heavy-temperature
// term and is dense); M_v^-1 is a forward and a backward substitution with the banded Cholesky
// factor of M_v along the B-spline index. The point has converged when
// max|r| <= tol max|b|, or when max|r| is already at the rounding level of an FP64 product A_i x,
// max|r| <= min(kBackwardFloor, tol) (|A_i| max|x| + max|b|) with |A_i| <= 1 + dt (|K_C| +
// |E_i| |K_A|) (infinity norms): a normwise backward error no refinement can improve on. The second
// test decides only for ill-conditioned A_i, where |A_i| |x| is far above |b|.
// 256 unit roundoffs of FP64: the normwise backward error at which a residual computed in FP64 is
// rounding noise.
constexpr double kBackwardFloor = 256.0 * 1.1102230246251565e-16;

__global__ void residual_kernel(const double* __restrict__ X, const double* __restrict__ B,
                                const double* __restrict__ E, double E_uniform, double dt, ResidualOps ro,
                                const double* __restrict__ TO, const double* __restrict__ TS, double* __restrict__ R,
                                double* __restrict__ ratio, int* __restrict__ conv, double tol,
                                double kc_inf, double ka_inf, int nt, int nr, int nl,
                                unsigned* __restrict__ status) {
  extern __shared__ double sm[];
  const int i = blockIdx.x;
  // a point that has converged keeps its iterate (the solves skip it), so its residual is final
  if (conv[i]) return;
  const int nv = nt * nr;
  double* xs = sm;             // nv
  double* xS = xs + nv;        // nl*nr
  double* g = xS + nl * nr;    // nl*nr
  __shared__ double red_r[32], red_b[32], red_x[32];
  const double* x = X + static_cast<size_t>(i) * nv;
  const double* b = B + static_cast<size_t>(i) * nv;
  const double Ei = E ? E[i] : E_uniform;
  for (int v = threadIdx.x; v < nv; v += blockDim.x) xs[v] = x[v];
  __syncthreads();
  for (int idx = threadIdx.x; idx < nl * nr; idx += blockDim.x) {
    const int l = idx / nr, k = idx % nr;
    double s = 0.0;
    for (int a = 0; a < nt; ++a) s = fma(__ldg(TS + l * nt + a), xs[a * nr + k], s);
    xS[idx] = s;
  }
  __syncthreads();
  const int w = ro.w, bw = 2 * w + 1;
  for (int idx = threadIdx.x; idx < nl * nr; idx += blockDim.x) {
    const int l = idx / nr, p = idx % nr;
    const int k0 = max(0, p - w), k1 = min(nr - 1, p + w);
    double c = 0.0, f = 0.0;
    if (l > 0) {   // C_0 (dense) is added in the next stage
      const double* row = ro.band + static_cast<size_t>(p) * bw + w - p;   // row[k] = loss[p][k]
      for (int k = k0; k <= k1; ++k) c = fma(__ldg(row + k), xS[l * nr + k], c);
    }
    if (l >= 1) {
      const double* row = ro.fband + (static_cast<size_t>(l) * nr + p) * bw + w - p;   // (A_v)_{l,l-1}[p][k]
      const double* y = xS + (l - 1) * nr;
      for (int k = k0; k <= k1; ++k) f = fma(__ldg(row + k), y[k], f);
    }
    if (l + 1 < nl) {
      const double* row = ro.fband + (static_cast<size_t>(nl + l) * nr + p) * bw + w - p;   // (A_v)_{l,l+1}[p][k]
      const double* y = xS + (l + 1) * nr;
      for (int k = k0; k <= k1; ++k) f = fma(__ldg(row + k), y[k], f);
    }
    g[idx] = c + Ei * f;
  }
  __syncthreads();
  // the dense C_0 rows (l = 0): eight lanes per row, each a strided part of the dot product, summed
  // over the lane group by shuffles (every thread runs the same number of rounds)
  {
    const int sub = threadIdx.x & 7, rows = blockDim.x >> 3;
    for (int pb = 0; pb < nr; pb += rows) {
      const int p = pb + (threadIdx.x >> 3);
      double c = 0.0;
      if (p < nr) {
        const double* row = ro.c0 + static_cast<size_t>(p) * nr;
        for (int k = sub; k < nr; k += 8) c = fma(__ldg(row + k), xS[k], c);
      }
      c += __shfl_down_sync(0xffffffffu, c, 4, 8);
      c += __shfl_down_sync(0xffffffffu, c, 2, 8);
      c += __shfl_down_sync(0xffffffffu, c, 1, 8);
      if (p < nr && sub == 0) g[p] += c;
    }
  }
  __syncthreads();
  // g_l <- M_v^-1 g_l, one thread per harmonic
  for (int l = threadIdx.x; l < nl; l += blockDim.x) mass_solve(g + l * nr, ro.chol, ro.cinv, nr, w);
  __syncthreads();
  double mr = 0.0, mb = 0.0, mx = 0.0;
  for (int v = threadIdx.x; v < nv; v += blockDim.x) {
    const int a = v / nr, p = v % nr;
    double s = 0.0;
    for (int l = 0; l < nl; ++l) s = fma(__ldg(TO + a * nl + l), g[l * nr + p], s);
    const double bv = b[v];
    const double rv = bv - xs[v] + dt * s;
    R[static_cast<size_t>(i) * nv + v] = rv;
    mr = fmax(mr, fabs(rv));
    mb = fmax(mb, fabs(bv));
    mx = fmax(mx, fabs(xs[v]));
  }
  for (int o = 16; o > 0; o >>= 1) {
    mr = fmax(mr, __shfl_xor_sync(0xffffffffu, mr, o));
    mb = fmax(mb, __shfl_xor_sync(0xffffffffu, mb, o));
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) red_r[threadIdx.x >> 5] = mr, red_b[threadIdx.x >> 5] = mb, red_x[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int wi = 1; wi < static_cast<int>(blockDim.x >> 5); ++wi)
      mr = fmax(mr, red_r[wi]), mb = fmax(mb, red_b[wi]), mx = fmax(mx, red_x[wi]);
    const double q = mb > 0.0 ? mr / mb : (mr > 0.0 ? INFINITY : 0.0);
    const double nA = 1.0 + dt * (kc_inf + fabs(Ei) * ka_inf);
    ratio[i] = q;
    conv[i] = (q <= tol || mr <= fmin(kBackwardFloor, tol) * (nA * mx + mb)) ? 1 : 0;
    atomicAdd(status + 1, 1u);  // residual evaluations (refinement accounting)
  }
}

__global__ void check_field_kernel(const double* __restrict__ E, int nx, unsigned* status) {
  bool bad = false;
  for (int i = threadIdx.x; i < nx; i += blockDim.x) bad |= !isfinite(E[i]);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, kNonFiniteIn);
}

__global__ void check_conv_kernel(const int* conv, int nx, unsigned* status) {
  bool all = true;
  for (int i = threadIdx.x; i < nx; i += blockDim.x) all &= conv[i] != 0;
  if (!__syncthreads_and(all) && threadIdx.x == 0) atomicOr(status, kNoConv);
}

__global__ void commit_kernel(const double* __restrict__ src, double* __restrict__ dst, size_t n,
                              const unsigned* status) {
  if (*status != 0u) return;
  for (size_t e = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; e < n;
       e += static_cast<size_t>(gridDim.x) * blockDim.x)
    dst[e] = src[e];
}

// ne = mom_n . F_i, mean = (mom_e . F_i)/ne, rates_j = (mom_r_j . F_i)/ne; FP64 block reductions.
__global__ void moments_kernel(const double* __restrict__ F, const double* __restrict__ mn,
                               const double* __restrict__ me, const double* __restrict__ mr,
                               int n_proc, double* ne, double* mean, double* rates, int nx, int nv) {
  __shared__ double red[32];
  __shared__ double ne_s;
  const int i = blockIdx.x;
  const double* f = F + static_cast<size_t>(i) * nv;
  auto block_sum = [&](const double* w) {
    double s = 0.0;
    for (int v = threadIdx.x; v < nv; v += blockDim.x) s = fma(w[v], f[v], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
      for (int w2 = 0; w2 < static_cast<int>(blockDim.x >> 5); ++w2) t += red[w2];
    return t;  // valid on thread 0
  };
  const double n = block_sum(mn);
  if (threadIdx.x == 0) {
    ne_s = n;
    if (ne) ne[i] = n;
  }
  __syncthreads();
  const double nn = ne_s;
  const double e = block_sum(me);
  if (threadIdx.x == 0 && mean) mean[i] = nn != 0.0 ? e / nn : 0.0;
  for (int j = 0; j < n_proc; ++j) {
    const double r = block_sum(mr + static_cast<size_t>(j) * nv);
    if (threadIdx.x == 0 && rates) rates[static_cast<size_t>(j) * nx + i] = nn != 0.0 ? r / nn : 0.0;
  }
}

__global__ void fill_maxwellian_kernel(double* F, const double* ne, const double* coef, int nx,
                                       int nt, int nr) {
  const size_t n = static_cast<size_t>(nx) * nt * nr;
  for (size_t e = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; e < n;
       e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t i = e / (static_cast<size_t>(nt) * nr);
    F[e] = ne[i] * coef[e % nr];
  }
}

int grid_for(size_t n, int block) {
  size_t g = (n + block - 1) / block;
  if (g > 152 * 32) g = 152 * 32;
  return static_cast<int>(g < 1 ? 1 : g);
}

}  // namespace

// Both transforms stage nr x (kXT + 1) doubles: past 48 KB (nr > 186) they need the opt-in
// shared-memory size, which bte_create keeps them within (nr <= kMaxNr).
static void set_x_transform_smem() {
  static bool done = false;
  if (done) return;
  cudaFuncSetAttribute(x_to_eigen_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  cudaFuncSetAttribute(x_from_eigen_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  done = true;
}

void launch_x_to_eigen(const double* F, const double* Uinv, double* Y, int nx, int nt, int nr,
                       unsigned* status, cudaStream_t st) {
  set_x_transform_smem();
  dim3 grid((nx * nt + kXT - 1) / kXT, (nr + kIC - 1) / kIC);
  const size_t smem = sizeof(double) * kXT * (nr + 1);
  x_to_eigen_kernel<<<grid, 256, smem, st>>>(F, Uinv, Y, nx, nt, nr, status);
}

void launch_x_matvec(const double* MT, bool per_pair, const double* lam, const double* mu, const double* Y,
                     double* Y2, int nx, int nt, int nr, cudaStream_t st) {
  const int threads = std::min(256, (nx + 31) / 32 * 32);
  x_matvec_kernel<<<nt * nr, threads, sizeof(double) * nx, st>>>(
      MT, per_pair ? static_cast<size_t>(nx) * nx : 0, lam, mu, Y, Y2, nx, nr);
}

void launch_x_apply_q(const double* QT, const double* Y, double* Y2, int nx, int nt, int nr,
                      cudaStream_t st) {
  launch_x_matvec(QT, true, nullptr, nullptr, Y, Y2, nx, nt, nr, st);
}

void launch_transpose_blocks(double* M, int n, size_t count, cudaStream_t st) {
  const unsigned t = static_cast<unsigned>((n + 31) / 32);
  for (size_t z = 0; z < count; z += 32768)
    transpose_blocks_kernel<<<dim3(t, t, static_cast<unsigned>(std::min<size_t>(32768, count - z))), 256, 0, st>>>(M, n, z);
}

void launch_x_from_eigen(const double* Y2, const double* U, double* F, int nx, int nt, int nr,
                         unsigned* status, cudaStream_t st) {
  set_x_transform_smem();
  dim3 grid((nx * nt + kXT - 1) / kXT, (nr + kIC - 1) / kIC);
  const size_t smem = sizeof(double) * nr * (kXT + 1);
  x_from_eigen_kernel<<<grid, 256, smem, st>>>(Y2, U, F, nx, nt, nr, status);
}

void launch_check_field(const double* E, int nx, unsigned* status, cudaStream_t st) {
  check_field_kernel<<<1, 256, 0, st>>>(E, nx, status);
}

template <typename T>
void launch_v_form(const double* KCg, const double* KAg, MassBand mass, const double* E, double E_uniform,
                   double dt, T* fac, int nx, int nv, cudaStream_t st) {
  const size_t nn = static_cast<size_t>(nv) * nv;
  const size_t smem = E ? sizeof(T) * static_cast<size_t>(nx) : 0;   // nx <= 4096: at most 32 KB
  v_form_kernel<T><<<grid_for(nn, 256), 256, smem, st>>>(KCg, KAg, mass, E, E_uniform, dt, fac, nx, nv);
}
template void launch_v_form<double>(const double*, const double*, MassBand, const double*, double, double,
                                    double*, int, int, cudaStream_t);
template void launch_v_form<float>(const double*, const double*, MassBand, const double*, double, double,
                                   float*, int, int, cudaStream_t);

void launch_residual(const double* x, const double* b, const double* E, double E_uniform, double dt,
                     const ResidualOps& ro, const double* TO, const double* TS, double* r, double* ratio, int* conv,
                     double tol, double kc_inf, double ka_inf, int nx, int nt, int nr, int nl, unsigned* status,
                     cudaStream_t st) {
  const size_t smem = sizeof(double) * (static_cast<size_t>(nt) * nr + 2 * nl * nr);
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(residual_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
    attr_set = true;
  }
  residual_kernel<<<nx, 512, smem, st>>>(x, b, E, E_uniform, dt, ro, TO, TS, r, ratio, conv, tol, kc_inf, ka_inf, nt,
                                         nr, nl, status);
}

void launch_check_conv(const int* conv, int nx, unsigned* status, cudaStream_t st) {
  check_conv_kernel<<<1, 256, 0, st>>>(conv, nx, status);
}

void launch_commit(const double* src, double* dst, size_t n, const unsigned* status, cudaStream_t st) {
  commit_kernel<<<grid_for(n, 256), 256, 0, st>>>(src, dst, n, status);
}

void launch_moments(const double* F, const double* mom_n, const double* mom_e, const double* mom_r,
                    int n_proc, double* ne, double* mean, double* rates, int nx, int nv,
                    cudaStream_t st) {
  moments_kernel<<<nx, 256, 0, st>>>(F, mom_n, mom_e, mom_r, n_proc, ne, mean, rates, nx, nv);
}

void launch_fill_maxwellian(double* F, const double* ne, const double* coef, int nx, int nt, int nr,
                            cudaStream_t st) {
  const size_t n = static_cast<size_t>(nx) * nt * nr;
  fill_maxwellian_kernel<<<grid_for(n, 256), 256, 0, st>>>(F, ne, coef, nx, nt, nr);
}

}  // namespace bte
