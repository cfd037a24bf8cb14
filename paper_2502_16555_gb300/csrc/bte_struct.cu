// Structure-exploiting velocity solve. The per-point matrix of eq. "vspace_batched_system" is
// A_i = I - dt P_O B_i P_S with B_i = C + E_i A_v in the spherical-harmonic basis (arXiv 2502.16555,
// eqs. "proj_ops", "bte_1d_discrete"), where C is block diagonal in l and A_v block tridiagonal
// (couplings l -> l +- 1 only, Section 3.3). Because P_S P_O = T_S T_O = I,
//     A_i^-1 f = f + P_O ( (I - dt B_i)^-1 - I ) P_S f,
// so one dense Nv x Nv solve becomes one block-tridiagonal solve of N_l blocks of Nr x Nr.
//
// BTE_FLAG_STRUCTURED (struct_factor_kernel, struct_substitute_kernel): the system multiplied by the
// mass matrix, H_i = (I (x) M_v)(I - dt B_i), whose blocks are banded but for the gain in the block
// (0, 0). It is eliminated from the highest harmonic down, S_l = D_l - U_l S_{l+1}^-1 L_{l+1} with
// D_l = M_v - dt C_l, L_l = -dt E (A_v)_{l,l-1}, U_l = -dt E (A_v)_{l,l+1}: A_v is skew-symmetric and
// M_v - dt C_l symmetric positive definite for l >= 1, so every S_l, l >= 1, is D_l plus a positive
// semidefinite matrix and its inversion needs no pivoting; S_0 comes last. The products with L and U
// cost 7 operations an element. The inverses are kept for the refinement's solves.
//
// vsolve_struct_kernel: the mass-scaled blocks I - dt B_i, eliminated upwards and solved in one launch. In
// FP64 it is the mixed paths' escalation, for the points whose refinement has not converged; in FP32 the
// structured solve of handles with at most one refinement sweep, whose results show the solve's own accuracy
// (1.2e-7 of f; 2.1e-6 through H_i, whose elimination meets the condition of M_v).
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "bte_kernels.h"
#include "bte_async.cuh"
#include "bte_recip.cuh"

namespace bte {
namespace {

constexpr int kST = 256;  // threads per CTA
constexpr int kSubstituteRoom = 200 * 1024;  // shared memory of the substitution: bte_create's check of
                                             // struct_smem_bytes leaves it at least one stage
constexpr int kG = 4;     // elements per thread and dimension (Nr <= 16 kG)

// acc(a, b) += sum_k AT[k][ty + 16 a] B[k][tx + 16 b] over k < n: AT is the left factor stored
// transposed (AT[k][i] = A[i][k]), both n x n with leading dimension n in shared memory.
template <typename T>
__device__ __forceinline__ void grid_gemm(const T* AT, const T* B, int n, T (&acc)[kG][kG]) {
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  for (int k = 0; k < n; ++k) {
    T a[kG], b[kG];
#pragma unroll
    for (int u = 0; u < kG; ++u) {
      a[u] = ty + 16 * u < n ? AT[k * n + ty + 16 * u] : T(0);
      b[u] = tx + 16 * u < n ? B[k * n + tx + 16 * u] : T(0);
    }
#pragma unroll
    for (int u = 0; u < kG; ++u)
#pragma unroll
      for (int v = 0; v < kG; ++v) acc[u][v] += a[u] * b[v];
  }
}

// out[i] = alpha * sum_k MT[k][i] x[k] for i < n (MT the matrix stored transposed): thread i,
// consecutive threads read consecutive addresses.
template <typename T>
__device__ __forceinline__ void gemv_t(const T* MT, const T* x, T* out, int n, T alpha) {
  for (int i = threadIdx.x; i < n; i += kST) {
    T acc = T(0);
    for (int k = 0; k < n; ++k) acc += MT[k * n + i] * x[k];
    out[i] = alpha * acc;
  }
}

// In-place inverse of the block held in registers (s[a][b] = S[ty + 16 a][tx + 16 b]) by
// Gauss-Jordan elimination without pivoting. Step k reads the pivot row and column from a copy
// written in step k - 1 by the owners of row/column k (double-buffered by parity): one barrier
// per step.
template <typename T>
__device__ void grid_gauss_jordan(T (&s)[kG][kG], int n, T* prow2, T* pcol2) {
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
  for (int a = 0; a < kG; ++a)
#pragma unroll
    for (int b = 0; b < kG; ++b) {
      const int i = ty + 16 * a, j = tx + 16 * b;
      if (i == 0 && j < n) prow2[j] = s[a][b];
      if (j == 0 && i < n) pcol2[i] = s[a][b];
    }
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    const T* prow = prow2 + (k & 1) * 64;
    const T* pcol = pcol2 + (k & 1) * 64;
    T* nrow = prow2 + ((k + 1) & 1) * 64;
    T* ncol = pcol2 + ((k + 1) & 1) * 64;
    const T p = T(1) / prow[k];
    T pr[kG], fc[kG];
#pragma unroll
    for (int u = 0; u < kG; ++u) {
      pr[u] = tx + 16 * u < n ? prow[tx + 16 * u] : T(0);
      fc[u] = ty + 16 * u < n ? pcol[ty + 16 * u] * p : T(0);
    }
#pragma unroll
    for (int a = 0; a < kG; ++a)
#pragma unroll
      for (int b = 0; b < kG; ++b) {
        const int i = ty + 16 * a, j = tx + 16 * b;
        T v = s[a][b] - fc[a] * pr[b];
        if (i == k) v = pr[b] * p;
        if (j == k) v = (i == k) ? p : -fc[a];
        s[a][b] = v;
        if (i == k + 1 && j < n) nrow[j] = v;
        if (j == k + 1 && i < n) ncol[i] = v;
      }
    __syncthreads();
  }
}

template <typename T>
__global__ void __launch_bounds__(kST) vsolve_struct_kernel(const double* __restrict__ Fin, double* __restrict__ Fout,
                                                            const double* __restrict__ E, double E_uniform, double dt,
                                                            const double* __restrict__ Cs, const double* __restrict__ Alo,
                                                            const double* __restrict__ Aup, const double* __restrict__ TO,
                                                            const double* __restrict__ TS, T* __restrict__ Xg, int nt,
                                                            int nr, int nl, const int* __restrict__ conv, int accumulate,
                                                            unsigned* status) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int pt = blockIdx.x;
  if (conv && conv[pt]) return;
  const int n = nr, nn = nr * nr, nv = nt * nr;
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T* SinvT = reinterpret_cast<T*>(smraw);  // S_q^-1, transposed
  T* Xp = SinvT + nn;                      // X_{q-1} = S_{q-1}^-1 U_{q-1}, row-major
  T* Xc = Xp + nn;                         // X_q
  T* Ab = Xc + nn;                         // As_lo[q] transposed, then As_up[q] row-major
  T* y = Ab + nn;                          // nl x nr: P_S f, then w_q
  T* wq = y + nl * nr;                     // nl x nr: S_q^-1 w_q, then z
  T* tmp = wq + nl * nr;                   // nr
  T* prow2 = tmp + nr;                     // 2 x 64 pivot rows
  T* pcol2 = prow2 + 128;                  // 2 x 64 pivot columns
  const double* f = Fin + static_cast<size_t>(pt) * nv;
  const T eE = static_cast<T>(dt * (E ? E[pt] : E_uniform));
  T* X = Xg + static_cast<size_t>(pt) * nl * nn;

  // y = T_S f (per radial index)
  for (int e = threadIdx.x; e < nl * nr; e += kST) {
    const int l = e / nr, k = e % nr;
    double s = 0.0;
    for (int a = 0; a < nt; ++a) s += TS[l * nt + a] * f[a * nr + k];
    y[e] = static_cast<T>(s);
  }
  __syncthreads();
  for (int q = 0; q < nl; ++q) {
    // S_q = I - dt Cs_q + dt E As_lo[q] X_{q-1} in registers;  w_q = y_q + dt E As_lo[q] wq_{q-1}
    T s[kG][kG];
    const double* C = Cs + static_cast<size_t>(q) * nn;
#pragma unroll
    for (int a = 0; a < kG; ++a)
#pragma unroll
      for (int b = 0; b < kG; ++b) {
        const int i = ty + 16 * a, j = tx + 16 * b;
        s[a][b] = (i < n && j < n) ? (i == j ? T(1) : T(0)) - static_cast<T>(dt * C[i * n + j]) : T(0);
      }
    if (q > 0) {
      const double* Al = Alo + static_cast<size_t>(q) * nn;
      for (int e = threadIdx.x; e < nn; e += kST) Ab[(e % n) * n + e / n] = static_cast<T>(Al[e]);
      __syncthreads();
      T acc[kG][kG] = {};
      grid_gemm<T>(Ab, Xp, n, acc);
#pragma unroll
      for (int a = 0; a < kG; ++a)
#pragma unroll
        for (int b = 0; b < kG; ++b) s[a][b] += eE * acc[a][b];
      gemv_t<T>(Ab, wq + (q - 1) * nr, tmp, n, eE);
      for (int k = threadIdx.x; k < nr; k += kST) y[q * nr + k] += tmp[k];  // same thread wrote tmp[k]
    }
    grid_gauss_jordan<T>(s, n, prow2, pcol2);
#pragma unroll
    for (int a = 0; a < kG; ++a)
#pragma unroll
      for (int b = 0; b < kG; ++b) {
        const int i = ty + 16 * a, j = tx + 16 * b;
        if (i < n && j < n) SinvT[j * n + i] = s[a][b];
      }
    if (q + 1 < nl) {
      const double* Au = Aup + static_cast<size_t>(q) * nn;
      for (int e = threadIdx.x; e < nn; e += kST) Ab[e] = static_cast<T>(Au[e]);
    }
    __syncthreads();
    // wq_q = S_q^-1 w_q;  X_q = S_q^-1 U_q = -dt E S_q^-1 As_up[q]
    gemv_t<T>(SinvT, y + q * nr, wq + q * nr, n, T(1));
    if (q + 1 < nl) {
      T acc[kG][kG] = {};
      grid_gemm<T>(SinvT, Ab, n, acc);
#pragma unroll
      for (int a = 0; a < kG; ++a)
#pragma unroll
        for (int b = 0; b < kG; ++b) {
          const int i = ty + 16 * a, j = tx + 16 * b;
          if (i < n && j < n) {
            const T v = -eE * acc[a][b];
            Xc[i * n + j] = v;
            X[static_cast<size_t>(q) * nn + i * n + j] = v;
          }
        }
      T* t = Xp;
      Xp = Xc;
      Xc = t;
    }
    __syncthreads();
  }
  // back substitution: z_{L-1} = wq_{L-1}; z_q = wq_q - X_q z_{q+1}, a warp per row, lanes across k
  for (int q = nl - 2; q >= 0; --q) {
    const T* Xq = X + static_cast<size_t>(q) * nn;
    for (int r = warp; r < nr; r += kST / 32) {
      T acc = T(0);
      for (int k = lane; k < nr; k += 32) acc += Xq[r * nr + k] * wq[(q + 1) * nr + k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) wq[q * nr + r] -= acc;
    }
    __syncthreads();
  }
  // z - y with y = P_S f again (y held w_q), then f* = f + T_O (z - y)
  for (int e = threadIdx.x; e < nl * nr; e += kST) {
    const int l = e / nr, k = e % nr;
    double s = 0.0;
    for (int a = 0; a < nt; ++a) s += TS[l * nt + a] * f[a * nr + k];
    y[e] = wq[e] - static_cast<T>(s);
  }
  __syncthreads();
  bool bad = false;
  double* out = Fout + static_cast<size_t>(pt) * nv;
  for (int e = threadIdx.x; e < nv; e += kST) {
    const int a = e / nr, k = e % nr;
    double s = 0.0;
    for (int l = 0; l < nl; ++l) s += TO[a * nl + l] * static_cast<double>(y[l * nr + k]);
    const double v = f[e] + s;
    bad |= !isfinite(v);
    out[e] = accumulate ? out[e] + v : v;
  }
  if (bad && status) atomicOr(status, kNonFinite);
}

// S_l^-1 of every harmonic of one point (CTA), l = nl - 1 .. 0, into Sg[pt][l] (by columns, stride
// `stride` values). A 16 x 16 thread grid holds the block being inverted in registers, thread
// (ty, tx) the elements (ty + 16 a, tx + 16 b); the Gauss-Jordan step k reads the pivot row, column
// and reciprocal that their owners posted in step k - 1: one barrier a step. In FP32 the latency of the
// nl nr dependent steps bounds it: 128 points of 64 x 32 672 us (752 with a condition on each product of
// the band). In FP64 the units' rate does (a step is 16 FMAs and 4 products a thread; the reciprocal is
// the owner's alone), so there the blocks l >= 1, which are symmetric, are held and swept by half: 3.45 ms
// instead of 4.30, with the same errors (in FP32 it would be 738 us: as many steps, each a little longer).
template <typename T>
__global__ void __launch_bounds__(kST) struct_factor_kernel(const double* __restrict__ E, double E_uniform, double dt,
                                                            ResidualOps ro, MassBand mass, T* __restrict__ Sg,
                                                            size_t stride, int n, int nl) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr bool kSym = sizeof(T) == 8;
  const int w = mass.w, bw = 2 * w + 1;
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  // both products' operands have a zero border of the band's half width, so that they need no conditions
  const int lds = (n + 2 * w) | 1, ldy = n | 1;
  T* Sinv = reinterpret_cast<T*>(smraw) + w;  // rows of lds: [i][j], j = -w .. n - 1 + w
  T* Y = reinterpret_cast<T*>(smraw) + n * lds + w * ldy;  // rows of ldy: i = -w .. n - 1 + w
  T* Lb = Y + (n + w) * ldy;              // [bw][n]: Lb[t + w][j] = dt E (A_v)_{l+1,l}[j + t][j]
  T* Ub = Lb + n * bw;                    // [n][bw], dt E (A_v)_{l,l+1}
  T* prow2 = Ub + n * bw;                 // 2 x 64 pivot rows
  T* pcol2 = prow2 + 128;                 // 2 x 64 pivot columns
  __shared__ T pinv2[2];
  const int pt = blockIdx.x;
  const double dtE = dt * (E ? E[pt] : E_uniform);
  T* out = Sg + static_cast<size_t>(pt) * nl * stride;
  for (int e = threadIdx.x; e < n * lds + (n + 2 * w) * ldy; e += kST) reinterpret_cast<T*>(smraw)[e] = T(0);
  for (int l = nl - 1; l >= 0; --l) {
    const bool half = kSym && l > 0;  // blocks a >= b alone
    T s[kG][kG];
#pragma unroll
    for (int a = 0; a < kG; ++a)
#pragma unroll
      for (int b = 0; b < kG; ++b) {
        const int i = ty + 16 * a, j = tx + 16 * b, d = j - i + w;
        double v = i == j ? 1.0 : 0.0;  // past the block: the identity
        if (i < n && j < n) {
          const bool in = d >= 0 && d < bw;
          v = in ? __ldg(mass.m + i * bw + d) : 0.0;
          if (l == 0) v -= dt * __ldg(ro.c0 + i * n + j);
          else if (in) v -= dt * __ldg(ro.band + i * bw + d);
        }
        s[a][b] = static_cast<T>(v);
      }
    if (l + 1 < nl) {
      for (int e = threadIdx.x; e < n * bw; e += kST) {
        const int t = e / n, c = e - t * n, r = c + t - w;  // L[r][c], r = c + t - w
        Lb[e] = r >= 0 && r < n ? static_cast<T>(dtE * __ldg(ro.fband + (static_cast<size_t>(l + 1) * n + r) * bw + c - r + w)) : T(0);
        Ub[e] = static_cast<T>(dtE * __ldg(ro.fband + static_cast<size_t>(nl + l) * n * bw + e));
      }
      __syncthreads();
#pragma unroll
      for (int b = 0; b < kG; ++b) {  // Y = S_{l+1}^-1 L_{l+1} (up to sign)
        const int c = tx + 16 * b;
        if (c >= n) break;
        T acc[kG] = {T(0), T(0), T(0), T(0)};
        auto rows = [&](int a) { return ty + 16 * a < n && (!half || a >= b || (a + 1 == b && ty + w >= 16)); };
        for (int t = 0; t < bw; ++t) {
          const T lv = Lb[t * n + c];
#pragma unroll
          for (int a = 0; a < kG; ++a)
            if (rows(a)) acc[a] = fma(Sinv[(ty + 16 * a) * lds + c + t - w], lv, acc[a]);
        }
#pragma unroll
        for (int a = 0; a < kG; ++a)
          if (rows(a)) Y[(ty + 16 * a) * ldy + c] = acc[a];
      }
      __syncthreads();
#pragma unroll
      for (int a = 0; a < kG; ++a) {
        const int i = ty + 16 * a;
        if (i >= n) break;
        for (int t = 0; t < bw; ++t) {
          const T u = -Ub[i * bw + t];
#pragma unroll
          for (int b = 0; b < kG; ++b)
            if (tx + 16 * b < n && (b <= a || !half)) s[a][b] = fma(u, Y[(i + t - w) * ldy + tx + 16 * b], s[a][b]);
        }
      }
    }
    // in-place inverse; the identity beyond n needs no steps. Steps kb, 16 + kb, .. by blocks of 16, so
    // that the pivot's register index is known
    auto post = [&](int o, auto q, int buf) {  // row and column 16 q + o, and the reciprocal of the pivot
      constexpr int Q = decltype(q)::value;
      if (ty == o)
#pragma unroll
        for (int b = 0; b < kG; ++b) prow2[64 * buf + tx + 16 * b] = s[Q][b];
      if (tx == o) {
#pragma unroll
        for (int a = 0; a < kG; ++a) pcol2[64 * buf + ty + 16 * a] = s[a][Q];
        if (ty == o) pinv2[buf] = recip(s[Q][Q]);
      }
    };
    auto sweep = [&](auto q) {
      constexpr int Q = decltype(q)::value;
      const int kn = min(16, n - 16 * Q);
#pragma unroll 1
      for (int o = 0; o < kn; ++o) {
        const int c = o & 1;
        const T p = pinv2[c];
        T pr[kG], fc[kG];
#pragma unroll
        for (int u = 0; u < kG; ++u) {
          pr[u] = prow2[64 * c + tx + 16 * u];
          fc[u] = pcol2[64 * c + ty + 16 * u] * p;
        }
#pragma unroll
        for (int a = 0; a < kG; ++a)
#pragma unroll
          for (int b = 0; b < kG; ++b) s[a][b] = fma(-fc[a], pr[b], s[a][b]);
        if (tx == o)
#pragma unroll
          for (int a = 0; a < kG; ++a) s[a][Q] = -fc[a];
        if (ty == o)  // the pivot row: scaled instead
#pragma unroll
          for (int b = 0; b < kG; ++b) s[Q][b] = b == Q && tx == o ? p : pr[b] * p;
        if (o + 1 < kn) post(o + 1, q, c ^ 1);
        else if (Q + 1 < kG && kn == 16 && 16 * (Q + 1) < n) post(0, std::integral_constant<int, (Q + 1) % kG>{}, 0);
        __syncthreads();
      }
    };
    // the same on blocks a >= b alone. In place, the rows and columns already done and those still to come
    // form symmetric blocks, and the blocks between them are each other's negative: v, the pivot row up to
    // the pivot's block and the column below it, gives both the row and, with that sign, the column.
    auto post_sym = [&](int o, auto q, int buf) {
      constexpr int Q = decltype(q)::value;
      if (ty == o)
#pragma unroll
        for (int b = 0; b <= Q; ++b) prow2[64 * buf + tx + 16 * b] = s[Q][b];
      if (tx == o) {
#pragma unroll
        for (int a = Q + 1; a < kG; ++a) prow2[64 * buf + ty + 16 * a] = s[a][Q];
        if (ty == o) pinv2[buf] = recip(s[Q][Q]);
      }
    };
    auto sweep_sym = [&](auto q) {
      constexpr int Q = decltype(q)::value;
      const int kn = min(16, n - 16 * Q);
#pragma unroll 1
      for (int o = 0; o < kn; ++o) {
        const int c = o & 1;
        const T p = pinv2[c], pq = ty < o ? -p : p;
        T pr[kG], fc[kG];
#pragma unroll
        for (int u = 0; u < kG; ++u) {
          pr[u] = prow2[64 * c + tx + 16 * u];
          fc[u] = prow2[64 * c + ty + 16 * u] * (u < Q ? -p : u == Q ? pq : p);
        }
#pragma unroll
        for (int a = 0; a < kG; ++a)
#pragma unroll
          for (int b = 0; b <= a; ++b) s[a][b] = fma(-fc[a], pr[b], s[a][b]);
        if (tx == o)
#pragma unroll
          for (int a = Q; a < kG; ++a) s[a][Q] = -fc[a];
        if (ty == o)
#pragma unroll
          for (int b = 0; b <= Q; ++b) s[Q][b] = b == Q && tx == o ? p : pr[b] * p;
        if (o + 1 < kn) post_sym(o + 1, q, c ^ 1);
        else if (Q + 1 < kG && kn == 16 && 16 * (Q + 1) < n) post_sym(0, std::integral_constant<int, (Q + 1) % kG>{}, 0);
        __syncthreads();
      }
    };
    constexpr std::integral_constant<int, 0> q0{};
    constexpr std::integral_constant<int, 1> q1{};
    constexpr std::integral_constant<int, 2> q2{};
    constexpr std::integral_constant<int, 3> q3{};
    if (half) {
      post_sym(0, q0, 0);
      __syncthreads();
      sweep_sym(q0), sweep_sym(q1), sweep_sym(q2), sweep_sym(q3);
    } else {
      post(0, q0, 0);
      __syncthreads();
      sweep(q0), sweep(q1), sweep(q2), sweep(q3);
    }
    T* o = out + static_cast<size_t>(l) * stride;
#pragma unroll
    for (int a = 0; a < kG; ++a)
#pragma unroll
      for (int b = 0; b < kG; ++b) {
        const int i = ty + 16 * a, j = tx + 16 * b;
        if (i >= n || j >= n || (half && b > a)) continue;
        Sinv[i * lds + j] = s[a][b];
        if (half && b < a) Sinv[j * lds + i] = s[a][b];
      }
    __syncthreads();
    for (int c = threadIdx.x >> 5; c < n; c += kST / 32)
      for (int i = threadIdx.x & 31; i < n; i += 32) o[c * n + i] = Sinv[i * lds + c];
  }
}

// z += H^-1 rho (vectors [nx][3 nl n]: y, z, rho) through the inverses: downwards g_l = S_l^-1 r_l with
// r_l = rho_l - U_l g_{l+1}, then upwards z_l = g_l - S_l^-1 L_l z_{l-1}. Thread (part, row) takes 16
// columns of a row; the inverses are streamed twice, through a ring of shared-memory stages filled by
// bulk copies; the couplings' band and rho are read a product ahead. Bound by the latency of 2 nl - 1
// dependent products, in FP64 half by the units' rate: 128 points of 64 x 32 65 us a solve in FP32 and
// 123 in FP64 (86 and 188 with the inverses loaded by rows, one block ahead, and the band where it is
// used); the 67 MB of FP32 inverses, twice, are 20 us at the copy bandwidth. Converged points return at once.
template <typename T>
__global__ void __launch_bounds__(kST) struct_substitute_kernel(const double* __restrict__ E, double E_uniform,
                                                                double dt, ResidualOps ro, MassBand mass,
                                                                const T* __restrict__ Sg, int stride, int stages,
                                                                double* __restrict__ vec, const int* conv, int n,
                                                                int nl, unsigned* status, int probe) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int pt = blockIdx.x, tid = threadIdx.x;
  if (conv && conv[pt]) return;
  const int w = mass.w, bw = 2 * w + 1, m = nl * n, ncopy = 2 * nl - 1;
  T* ring = reinterpret_cast<T*>(smraw);  // [stages][stride]
  T* g = ring + stages * stride;          // [nl][n]
  T* r = g + m;                           // [64]
  T* part = r + 64;                       // [4][64]
  __shared__ __align__(8) uint64_t full[8], never;
  __shared__ int gave_up;
  double* z = vec + static_cast<size_t>(pt) * 3 * m + m;
  const double* rho = z + m;
  const T* S = Sg + static_cast<size_t>(pt) * nl * stride;
  const T dtE = static_cast<T>(dt * (E ? E[pt] : E_uniform));
  const uint32_t bytes = static_cast<uint32_t>(stride * sizeof(T));
  auto block_of = [&](int q) { return q < nl ? nl - 1 - q : q - nl + 1; };  // down nl - 1 .. 0, up 1 .. nl - 1
  // by thread 0, which also waits for each copy and stops when that fails
  bool quit = false;
  int issued = 0;
  auto issue = [&](int q, int st) {
    if (quit) return;
    issued = q + 1;
    expect_tx(&full[st], bytes);
    bulk_load(ring + st * stride, S + static_cast<size_t>(block_of(q)) * stride, bytes, &full[st]);
  };
  if (tid == 0) {
    for (int i = 0; i < stages; ++i) mbar_init(&full[i], 1);
    mbar_init(&never, 1);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    for (int q = 0; q < min(stages, ncopy); ++q) issue(q, q);
    if (probe) quit = !mbar_wait(&never, 0, &gave_up, status, kProbeCycles);
  }
  const int row = tid & 63, p = tid >> 6;
  if (tid < 64) r[tid] = tid < n ? static_cast<T>(rho[(nl - 1) * n + tid]) : T(0);
  __syncthreads();
  int st = 0;
  uint32_t ph = 0;
  for (int q = 0; q < ncopy; ++q) {
    const bool down = q < nl;
    const int l = block_of(q);
    // what the next vector needs of rho and of the couplings' band (w <= 3), ahead of the wait
    const bool up = !down || l == 0;
    const int dst = up ? l + 1 : l - 1;
    double fb[7] = {}, rn = 0.0;
    if (tid < n && dst < nl) {
      if (!up) rn = rho[dst * n + tid];
      const double* fr = ro.fband + (static_cast<size_t>(up ? dst : nl + dst) * n + tid) * bw + w - 3;
#pragma unroll
      for (int t = 0; t < 7; ++t) {
        const int k = tid + t - 3;
        if (t >= 3 - w && t <= 3 + w && k >= 0 && k < n) fb[t] = __ldg(fr + t);
      }
    }
    if (!mbar_wait(&full[st], ph, &gave_up, status)) quit = true;
    T a0 = T(0), a1 = T(0);
    if (row < n) {
      const T* sc = ring + st * stride + row;
#pragma unroll
      for (int c = 0; c < 16; c += 2) {
        const int j = 16 * p + c;
        if (j < n) a0 = fma(sc[j * n], r[j], a0);
        if (j + 1 < n) a1 = fma(sc[(j + 1) * n], r[j + 1], a1);
      }
    }
    part[p * 64 + row] = a0 + a1;
    __syncthreads();
    if (tid == 0 && q + stages < ncopy) issue(q + stages, st);
    if (tid < n) {
      T v = (part[tid] + part[64 + tid]) + (part[128 + tid] + part[192 + tid]);
      if (!down) v += g[l * n + tid];
      g[l * n + tid] = v;
    }
    if (tid < 64) asm volatile("bar.sync 1, 64;" ::: "memory");
    // the next vector: rho_{l-1} + dt E Aup_{l-1} g_l downwards, dt E Alo_{l+1} z_l upwards (z_0 = g_0)
    if (tid < 64) {
      T v = T(0);
#pragma unroll
      for (int t = 0; t < 7; ++t) {
        const int k = tid + t - 3;
        if (k >= 0 && k < n) v = fma(static_cast<T>(fb[t]), g[l * n + k], v);
      }
      v = tid < n ? fma(dtE, v, static_cast<T>(rn)) : T(0);
      r[tid] = v;
    }
    __syncthreads();
    if (++st == stages) st = 0, ph ^= 1u;
  }
  for (int i = tid; i < m; i += kST) z[i] += static_cast<double>(g[i]);
  if (tid == 0 && quit)
    for (int q = max(0, issued - stages); q < issued; ++q) mbar_drain(&full[q % stages], (q / stages) & 1);
}

// ---- the reduced dense system (N_l < N_theta): the same identity with I - dt B_i factored as a
// dense m x m matrix, m = N_l Nr, by the LU kernels of the full system, in its unscaled form
// (I (x) M_v)(I - dt B_i) (LU with partial pivoting on the mass-scaled form meets large element
// growth on fine speed grids). Row and column (l, k) sit at l Nr + k: block (l, l) = M_v - dt Cg_l,
// block (l, l - 1) = -dt E_i Aglo[l], block (l, l + 1) = -dt E_i Agup[l], zero elsewhere.

// (I (x) M_v) G_i, one CTA per row (point i, row (l, p)); columns in blocks of Nr.
template <typename T>
__global__ void v_form_reduced_kernel(const double* __restrict__ Cg, const double* __restrict__ Aglo,
                                      const double* __restrict__ Agup, MassBand mass, const double* __restrict__ E,
                                      double E_uniform, double dt, T* __restrict__ G, int nr, int nl) {
  const int m = nl * nr;
  const size_t rowg = blockIdx.x;  // i * m + row
  const int i = static_cast<int>(rowg / m), row = static_cast<int>(rowg % m);
  const int l = row / nr, p = row % nr;
  const double Ei = E ? E[i] : E_uniform;
  const size_t off = (static_cast<size_t>(l) * nr + p) * nr;
  T* out = G + rowg * m;
  const int bw = 2 * mass.w + 1;
  for (int lc = 0; lc < nl; ++lc) {
    const double* src = lc == l ? Cg : lc == l - 1 ? Aglo : lc == l + 1 ? Agup : nullptr;
    const double w = lc == l ? 1.0 : Ei;
    for (int k = threadIdx.x; k < nr; k += blockDim.x) {
      const double b = src ? w * __ldg(src + off + k) : 0.0;
      const int dk = k - p;
      const double d = lc == l && dk >= -mass.w && dk <= mass.w ? __ldg(mass.m + p * bw + dk + mass.w) : 0.0;
      out[lc * nr + k] = static_cast<T>(d - dt * b);
    }
  }
}

// y_i = P_S f_i: y[l][k] = sum_a T_S[l][a] f[a][k], skipping converged points.
__global__ void reduce_project_kernel(const double* __restrict__ F, const double* __restrict__ TS,
                                      double* __restrict__ Yr, const int* __restrict__ conv, int nt, int nr,
                                      int nl) {
  const int i = blockIdx.x;
  if (conv && conv[i]) return;
  const int m = nl * nr;
  const double* f = F + static_cast<size_t>(i) * nt * nr;
  for (int idx = threadIdx.x; idx < m; idx += blockDim.x) {
    const int l = idx / nr, k = idx % nr;
    double s = 0.0;
    for (int a = 0; a < nt; ++a) s = fma(__ldg(TS + l * nt + a), f[a * nr + k], s);
    Yr[static_cast<size_t>(i) * m + idx] = s;
  }
}

// out_i (+)= f_i + P_O (z_i - y_i): out[a][k] = f[a][k] + sum_l T_O[a][l] (z[l][k] - y[l][k]),
// skipping converged points.
__global__ void reduce_lift_kernel(const double* __restrict__ F, const double* __restrict__ Yr,
                                   const double* __restrict__ Zr, const double* __restrict__ TO,
                                   double* __restrict__ out, const int* __restrict__ conv, int accumulate, int nt,
                                   int nr, int nl) {
  const int i = blockIdx.x;
  if (conv && conv[i]) return;
  const int m = nl * nr, nv = nt * nr;
  const size_t base = static_cast<size_t>(i) * nv;
  const double* y = Yr + static_cast<size_t>(i) * m;
  const double* z = Zr + static_cast<size_t>(i) * m;
  for (int v = threadIdx.x; v < nv; v += blockDim.x) {
    const int a = v / nr, k = v % nr;
    double s = F[base + v];
    for (int l = 0; l < nl; ++l) s = fma(__ldg(TO + a * nl + l), z[l * nr + k] - y[l * nr + k], s);
    out[base + v] = accumulate ? out[base + v] + s : s;
  }
}

}  // namespace

template <typename T>
void launch_v_form_reduced(const double* Cg, const double* Aglo, const double* Agup, MassBand mass, const double* E,
                           double E_uniform, double dt, T* G, int nx, int nr, int nl, cudaStream_t st) {
  const unsigned rows = static_cast<unsigned>(nx) * nl * nr;
  v_form_reduced_kernel<T><<<rows, nr >= 128 ? 128 : 64, 0, st>>>(Cg, Aglo, Agup, mass, E, E_uniform, dt, G, nr, nl);
}
template void launch_v_form_reduced<float>(const double*, const double*, const double*, MassBand, const double*,
                                           double, double, float*, int, int, int, cudaStream_t);
template void launch_v_form_reduced<double>(const double*, const double*, const double*, MassBand, const double*,
                                            double, double, double*, int, int, int, cudaStream_t);

void launch_reduce_project(const double* F, const double* TS, double* Yr, const int* conv, int nx, int nt, int nr,
                           int nl, cudaStream_t st) {
  reduce_project_kernel<<<nx, 256, 0, st>>>(F, TS, Yr, conv, nt, nr, nl);
}

void launch_reduce_lift(const double* F, const double* Yr, const double* Zr, const double* TO, double* out,
                        const int* conv, int accumulate, int nx, int nt, int nr, int nl, cudaStream_t st) {
  reduce_lift_kernel<<<nx, 256, 0, st>>>(F, Yr, Zr, TO, out, conv, accumulate, nt, nr, nl);
}

size_t struct_smem_bytes(int nr, int nl, size_t tsize) {
  return (4ull * nr * nr + 2ull * nl * nr + nr + 4ull * 64) * tsize;
}

template <typename T>
void launch_vsolve_struct(const double* Fin, double* Fout, const double* E, double E_uniform, double dt,
                          const double* Cs, const double* Alo, const double* Aup, const double* TO, const double* TS,
                          T* Xscratch, int nx, int nt, int nr, int nl, const int* conv, int accumulate,
                          unsigned* status, cudaStream_t st) {
  const size_t smem = struct_smem_bytes(nr, nl, sizeof(T));
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(vsolve_struct_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    attr_set = true;
  }
  vsolve_struct_kernel<T><<<nx, kST, smem, st>>>(Fin, Fout, E, E_uniform, dt, Cs, Alo, Aup, TO, TS, Xscratch, nt, nr, nl,
                                                 conv, accumulate, status);
}

template void launch_vsolve_struct<float>(const double*, double*, const double*, double, double, const double*,
                                          const double*, const double*, const double*, const double*, float*, int,
                                          int, int, int, const int*, int, unsigned*, cudaStream_t);
template void launch_vsolve_struct<double>(const double*, double*, const double*, double, double, const double*,
                                           const double*, const double*, const double*, const double*, double*, int,
                                           int, int, int, const int*, int, unsigned*, cudaStream_t);

size_t struct_stride(int nr) { return (static_cast<size_t>(nr) * nr + 3) / 4 * 4; }

template <typename T>
cudaError_t launch_struct_factor(const double* E, double E_uniform, double dt, const ResidualOps& ro, MassBand mass,
                                 T* S, int nx, int nr, int nl, cudaStream_t st) {
  auto values = [w2 = 2 * mass.w](int n) { return n * ((n + w2) | 1) + (n + w2) * (n | 1) + 2 * n * (w2 + 1) + 4 * 64; };
  const int smem = static_cast<int>(sizeof(T)) * values(nr);
  const cudaError_t e = set_smem_limit(struct_factor_kernel<T>, sizeof(T) * values(16 * kG));  // nr <= 64
  if (e != cudaSuccess) return e;
  struct_factor_kernel<T><<<nx, kST, smem, st>>>(E, E_uniform, dt, ro, mass, S, struct_stride(nr), nr, nl);
  return cudaGetLastError();
}
template cudaError_t launch_struct_factor<float>(const double*, double, double, const ResidualOps&, MassBand, float*,
                                                 int, int, int, cudaStream_t);
template cudaError_t launch_struct_factor<double>(const double*, double, double, const ResidualOps&, MassBand, double*,
                                                  int, int, int, cudaStream_t);

template <typename T>
cudaError_t launch_struct_substitute(const double* E, double E_uniform, double dt, const ResidualOps& ro, MassBand mass,
                                     const T* S, double* vec, const int* conv, int nx, int nr, int nl, unsigned* status,
                                     int probe, cudaStream_t st) {
  const int stride = static_cast<int>(struct_stride(nr)), fixed = static_cast<int>(sizeof(T)) * (nl * nr + 64 + 256);
  const int sb = stride * static_cast<int>(sizeof(T));
  const int stages = std::max(1, std::min(8, (kSubstituteRoom - fixed) / sb));
  const int smem = fixed + stages * sb;
  const cudaError_t e = set_smem_limit(struct_substitute_kernel<T>, kSubstituteRoom);
  if (e != cudaSuccess) return e;
  struct_substitute_kernel<T><<<nx, kST, smem, st>>>(E, E_uniform, dt, ro, mass, S, stride, stages, vec, conv, nr, nl, status,
                                                      probe);
  return cudaGetLastError();
}
template cudaError_t launch_struct_substitute<float>(const double*, double, double, const ResidualOps&, MassBand,
                                                     const float*, double*, const int*, int, int, int,
                                                     unsigned*, int, cudaStream_t);
template cudaError_t launch_struct_substitute<double>(const double*, double, double, const ResidualOps&, MassBand,
                                                      const double*, double*, const int*, int, int, int,
                                                      unsigned*, int, cudaStream_t);

}  // namespace bte
