// The per-point velocity solves of eq. "vspace_batched_system" (arXiv 2502.16555) through a windowed
// LU with partial pivoting, one CTA per collocation point from formation to the last factor.
//
// The system. With P_S P_O = T_S T_O = I, A_i^-1 f = f + P_O (G_i^-1 - I) P_S f, G_i = I - dt B_i in the
// harmonic basis (Section 3.3), and H_i = (I (x) M_v) G_i = I (x) M_v - dt (C + E_i A_v) has the same
// solutions. Its blocks are banded in the speed index (cubic B-splines couple |p - k| <= 3) and couple
// only l and l +- 1; the one exception is the gain of the inelastic processes, which reaches from row
// (p, l = 0) to columns (k, l = 0) far above p. Taken with the speed index slowest, H_i is a band
// matrix of half width 3 nl + 1 plus, for the l = 0 columns, entries far to the right: order
// n = nl nr, but 2 n (4 nl) (6 nl + nr) operations instead of 2 n^3 / 3 (medium grid 0.27 against
// 5.7 Gflop a point), with partial pivoting over every row that has an entry in the column, exactly as
// in a dense LU of the same matrix.
//
// The window. Columns are taken 32 at a time ("chunks": g = 32 / nlp speed indices, nlp the power of
// two >= nl, unused columns skipped). While chunk s is eliminated, the rows that can have an entry in
// it are those of chunks <= s + RC (RC = ceil(3 / g) <= 3): at most 128 live rows, held in 128 fixed
// slots; the 32 rows chosen as pivots leave their slots to the 32 rows of the chunk that enters, so
// no row is ever moved. Their columns are those of the next RS = 2 RC chunks (a ring of RS x 32) and
// the far l = 0 columns, one per speed index; when a chunk enters the ring, its l = 0 columns take over
// what the far columns held.
//
// In a panel every eliminated row keeps, in the place of the eliminated column, the running product
// of the elimination (the in-place form of Gauss elimination that carries its own inverse): after
// 32 columns a pivot row holds its row of inv(L11) left of the diagonal and of U11 from it on, and
// any other row holds t = -L21 inv(L11). The whole window is then updated by one product,
// D += T B with B the pivot rows (T's pivot rows: inv(L11) - I), and the forward substitution is
// one matrix-vector product with T per panel.
//
// Levelled rows (FP64, and mixed handles without the FP64 escalation): the rows are multiplied by powers of two that
// level the row sums of M_v (window_row_scale), which changes nothing but the choice of pivots. Without it the
// FP32 factors of fine speed grids at strong fields took the error only 1e-3 down a refinement sweep, and some steps
// that the dense LU refined in time did not converge (256 x 7, 1.1e6 V/m, FP32 LU on the host, error after each
// sweep: 2.1e-2, 8.8e-5, 3.0e-7; levelled 3.5e-5, 7.9e-9, 7.9e-13; the dense LU, harmonic slowest, 4.4e-2, 6.1e-7,
// 1.3e-11). FP64 steps of 168 small grids need 1.0 residual evaluations a point instead of 1.7, with errors 0.6 of what
// they were. Mixed handles with the escalation need it less and stay as they are: levelled they end a sweep earlier
// and further off (a batch of eight: 1.3e-12 instead of 4.6e-13).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <vector>

#include "bte_async.cuh"
#include "bte_handle.h"
#include "bte_kernels.h"
#include "bte_mass.cuh"
#include "bte_recip.cuh"
#include "bte_tf32.cuh"

namespace bte {
namespace {

constexpr int kPW = 32;      // panel (chunk) width
constexpr int kSlots = 128;  // row slots: the tensor cores' M
constexpr int kThreads = 256;
constexpr double kBackwardFloor = 256.0 * 1.1102230246251565e-16;  // as in launch_residual

__host__ __device__ inline int imin(int a, int b) { return a < b ? a : b; }
__host__ __device__ inline int imax(int a, int b) { return a > b ? a : b; }

// columns of chunk s that are unknowns of the system
__device__ __forceinline__ unsigned chunk_mask(const WindowPlan& w, int s) {
  unsigned m = 0;
  for (int i = 0; i < w.g; ++i)
    if (s * w.g + i < w.nr) m |= ((w.nl < 32 ? (1u << w.nl) : 0u) - 1u) << (i * w.nlp);
  return m;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 B apart
__device__ __forceinline__ uint64_t sdesc(uint32_t addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((addr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;
  d |= static_cast<uint64_t>(1024 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}

__device__ __forceinline__ void mma_tf32(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, 1, 0;\n"
      " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}"
      ::"r"(tmem_d), "l"(a), "l"(b), "r"(idesc));
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(bar))
               : "memory");
}

// Loads from tensor memory and their wait in one statement: the registers hold nothing before the wait, and between
// two statements the compiler may copy or spill them.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      " tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
        "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float (&v)[32]) {
  uint32_t r[32];
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(v[i]);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}

__device__ __forceinline__ float tmem_ld1(uint32_t taddr) {
  uint32_t r;
  __syncwarp();
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n tcgen05.wait::ld.sync.aligned;"
               : "=r"(r)
               : "r"(taddr)
               : "memory");
  return __uint_as_float(r);
}

__device__ __forceinline__ void tmem_st1(uint32_t taddr, float v) {
  __syncwarp();
  asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "r"(__float_as_uint(v)) : "memory");
}

__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Row r of a 32 x 32 block stored with its 16-byte pieces exchanged (piece q of row r at place
// q ^ (r & 7), so that a warp's lanes, one row each, meet different banks).
__device__ __forceinline__ void load_row(const float* block, int r, float (&v)[32]) {
  const float4* p = reinterpret_cast<const float4*>(block + r * 32);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float4 x = p[q ^ (r & 7)];
    v[4 * q] = x.x, v[4 * q + 1] = x.y, v[4 * q + 2] = x.z, v[4 * q + 3] = x.w;
  }
}
__device__ __forceinline__ void store_row(float* block, int r, const float (&v)[32]) {
  float4* p = reinterpret_cast<float4*>(block + r * 32);
#pragma unroll
  for (int q = 0; q < 8; ++q) p[q ^ (r & 7)] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}
// A template row at the field E: the columns of its own harmonic (bits of own) stand as they are, the
// others are per unit of the field.
__device__ __forceinline__ void scale_row(float (&v)[32], unsigned own, float E) {
#pragma unroll
  for (int c = 0; c < 32; ++c) v[c] = (own >> c) & 1u ? v[c] : E * v[c];
}

// Where p: the 8 values v[0 .. 7] to row, (key, inv) to rec (shared-memory addresses), without a branch.
__device__ __forceinline__ void post_row(bool p, uint32_t row, const float (&v)[32], uint32_t rec, unsigned key, float inv) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %0, 0;\n"
      " @p st.shared.v4.f32 [%1], {%2, %3, %4, %5};\n @p st.shared.v4.f32 [%1 + 16], {%6, %7, %8, %9};\n"
      " @p st.shared.v2.b32 [%10], {%11, %12};\n}"
      ::"r"(static_cast<unsigned>(p)), "r"(row), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]),
      "f"(v[6]), "f"(v[7]), "r"(rec), "r"(key), "f"(inv)
      : "memory");
}

struct FactorArgs {
  WindowPlan w;
  const void* base;    // row templates: FP64 [np 32][NW], FP32 window_blocks
  const void* slope;   // FP64 [np 32][(RS + 1) 32]
  const double* E;
  double Eu;
  void* T;             // [nx][np][32][NS]
  void* U;             // [nx][np][1024 + 32 NU]: inv(U11), then the pivot rows over the window (FP64 by
                       // rows, FP32 in 32 x 32 blocks)
  signed char* slotj;  // [nx][np][NS]: the pivot index of each slot, -1 if its row stays
  double* W;           // FP64: the window [nx][128][NU + 32]
  int* rows;           // FP64: the padded row in each slot [nx][128]
  unsigned* status;
  int probe;           // FP32: in the first panel, with its products in flight, a wait runs out
};

// Mixed path. The window D (128 slots x NU columns) lives in tensor memory in FP32; T and B are split
// into TF32 heads and remainders in shared memory (the split and the three products of the dense
// path's trailing updates) and D += T B runs as tcgen05.mma with M = 128, K = 32.
// Warps 0-3 (one thread a slot) hold the panel's 32 columns in registers and eliminate them: per
// column one warp-wide argmax, each warp's candidate row posted to shared memory, one barrier of
// the panel's warps. Warps 4-7 meanwhile finish the panel before: the pivot rows' updated window is
// written out as U, the rows of the entering chunk take the freed slots. The next panel waits only for
// the update of its own 32 columns, which is issued first.
// Bound by the latency of a panel's two chains, equally long (12.6 us a panel): the 32 dependent columns, and
// the conversion, products, rows passed on and the inverse of U11; not by the tensor cores (5000 cycles
// a panel) or memory. Medium grid (128 points, order 2048): 0.81 ms for formation and factors, where
// the dense LU took 11.6 ms. Every warp eliminating all 128 rows by itself (8 barriers a panel instead of
// 40) with a ninth warp for the inverse took 0.82 ms: the second chain slows down beside it.
__global__ void __launch_bounds__(kThreads, 2) window_lu_tc_kernel(const FactorArgs a) {
  extern __shared__ __align__(1024) unsigned char raw[];
  const WindowPlan& w = a.w;
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
  float* Thi = reinterpret_cast<float*>(sm);
  float* Tlo = Thi + kSlots * kPW;
  float* Bhi = Tlo + kSlots * kPW;
  float* Blo = Bhi + w.NU * kPW;
  float* t0 = Blo + w.NU * kPW;  // the entering rows' template of the next panel's columns
  __shared__ __align__(16) float prow[2][4][8];    // each warp's candidate row in the current sub-block
  __shared__ __align__(16) uint2 keys[2][4];       // its magnitude and lane, and 1 / its pivot
  __shared__ __align__(16) float pblk[2][8][24];   // a sub-block's pivot rows over the other columns
  __shared__ signed char slotj[2][kSlots];
  __shared__ float u11[32 * 33];
  __shared__ float ui[32 * 17];  // inverses of U11's 16 x 16 diagonal blocks
  // products of chunk s + 1, of the rest; templates of the ring and far columns, of the panel's; U11 inverted
  __shared__ __align__(8) uint64_t bar_next, bar_rest, bar_tmpl, bar_t0, bar_u;
  __shared__ __align__(8) uint64_t never;  // the probe's
  __shared__ uint32_t tmem_base;
  __shared__ int gave_up;

  const int pt = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, quad = warp & 3;
  const int slot = quad * 32 + lane, np = w.np, NS = w.NS, RS = w.RS, RC = w.RC, g = w.g;
  const int nch = RS + 1 + w.NF / 32;  // template chunks of a row: the panel's, the ring's, the far ones
  const bool panel_warp = warp < 4;
  const int npw = NS / 32;  // panel warps that hold rows
  const float* tmpl = static_cast<const float*>(a.base);
  auto block = [&](int t, int ch) { return tmpl + (static_cast<size_t>(t) * nch + ch) * 1024; };
  const float E = static_cast<float>(a.E ? a.E[pt] : a.Eu);
  float* Tg = static_cast<float*>(a.T) + static_cast<size_t>(pt) * np * 32 * NS;
  const size_t ustride = 1024 + 32 * static_cast<size_t>(w.NU);
  float* Ug = static_cast<float*>(a.U) + static_cast<size_t>(pt) * np * ustride;
  signed char* sjg = a.slotj + static_cast<size_t>(pt) * np * NS;

  if (tid == 0) {
    mbar_init(&bar_next, 1);
    mbar_init(&bar_rest, 1);
    mbar_init(&bar_tmpl, 1);
    mbar_init(&bar_t0, 1);
    mbar_init(&bar_u, 1);
    mbar_init(&never, 1);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_base)),
                 "r"(static_cast<uint32_t>(w.tmem_cols)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  // K columns of unused unknowns are never converted: they hold zeros, later rows of U or of templates, all finite,
  // and T's columns for them are zero
  for (int i = tid; i < w.NU * kPW; i += kThreads) Bhi[i] = Blo[i] = 0.f;
  for (int i = tid; i < 2 * 8 * 24; i += kThreads) (&pblk[0][0][0])[i] = 0.f;
  if (tid < 8) (&keys[0][0])[tid] = make_uint2(0u, 0u);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);  // this warp's lanes
  const int nfar = imax(0, w.nr - w.kf0);

  float v[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = 0.f;
  unsigned rep = 0;  // bit of every harmonic 0 column in a chunk
  for (int i = 0; i < g; ++i) rep |= 1u << (i * w.nlp);
  auto own = [&](int j) { return rep << (j & (w.nlp - 1)); };  // columns of row j's harmonic
  // rows of chunks 0 .. RC enter at panel 0, slot by slot
  const int t_in = slot / 32;
  const bool valid0 = slot < NS && t_in < np && ((chunk_mask(w, t_in) >> lane) & 1u);
  bool act = panel_warp && valid0;
  if (panel_warp) {
    if (act) {
      load_row(block(t_in, 0), lane, v);
      scale_row(v, own(lane), E);
    }
  } else {
    for (int ch = 1; ch < nch; ++ch) {
      float r[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) r[i] = 0.f;
      if (valid0) {
        load_row(block(t_in, ch), lane, r);
        if (ch <= RS) scale_row(r, own(lane), E);
      }
      tmem_st32(tmem + (ch <= RS ? ch % RS : ch - 1) * 32, r);
    }
    tmem_wait_st();
    tc_fence_before();
  }
  bool bad = false;
  // quit: a wait of this thread ran out, it issues nothing more; sent: it has issued, in this panel, what it
  // will wait for (threads 0: bar_next, 32: bar_t0, 160: bar_tmpl)
  bool quit = false, sent = false;
  auto wait = [&](uint64_t* b, uint32_t ph, bool mine) {
    if (mbar_wait(b, ph, &gave_up, a.status)) return;
    quit = true;
    if (mine) mbar_drain(b, ph);
  };

  for (int s = 0; s < np; ++s) {
    const int par = s & 1;
    sent = false;
    const int dmax = imin(RS, np - 1 - s);                       // ring chunks right of the panel
    const int fc0 = (s * g) / 32, nfc = s * g < nfar ? w.NF / 32 : fc0;  // far chunks [fc0, nfc)
    int pj = -1;
    if (panel_warp) {
      // ---- the panel: 32 columns in registers, one thread a row
      if (warp < npw) {
        const unsigned mask = chunk_mask(w, s);
        bool cand = act;
        int b = 0;  // posting buffer: alternates from one eliminated column to the next
        // Four sub-blocks of 8 columns. Inside one, only its 8 columns follow every pivot; the other 24
        // (T entries of earlier columns, values of later ones) take the 8 pivots at once from the
        // pivot rows as they were (D += T B again). The registers turn by one place per column and
        // by 8 per sub-block, so that the column being eliminated is always v[0] and the loops stay
        // rolled (unrolled over 32 columns they ran from instruction memory: 1600 cycles a column).
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          int pq = -1;  // this row's pivot index within the sub-block
#pragma unroll 1
          for (int c = 0; c < 8; ++c) {
            float f = 0.f, last = v[0];
            float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0;
            if ((mask >> (8 * q + c)) & 1u) {
              b ^= 1;
              // the low 5 bits of the magnitude give way to the lane: the largest entry to 2^-18. No
              // branches in a column's chain (each cost 50 to 100 cycles): the store is predicated.
              const unsigned key = cand ? (__float_as_uint(v[0]) & 0x7fffffe0u) + 32u + lane : 0u;
              const float inv = recip(v[0]);
              const unsigned best = __reduce_max_sync(0xffffffffu, key);
              post_row(best ? key == best : lane == 0, saddr(prow[b][warp]), v, saddr(&keys[b][warp]), key, inv);
              asm volatile("bar.sync 1, %0;" ::"r"(npw * 32) : "memory");
              const uint4 k01 = *reinterpret_cast<const uint4*>(&keys[b][0]), k23 = *reinterpret_cast<const uint4*>(&keys[b][2]);
              const bool s1 = k01.z > k01.x, s2 = k23.z > k23.x;
              const unsigned ka = s1 ? k01.z : k01.x, kc = s2 ? k23.z : k23.x;
              const bool s3 = kc > ka;
              const unsigned kb = s3 ? kc : ka;
              const unsigned iv = s3 ? (s2 ? k23.w : k23.y) : (s1 ? k01.w : k01.y);
              const int wb = s3 ? (s2 ? 3 : 2) : (s1 ? 1 : 0);
              r0 = *reinterpret_cast<const float4*>(&prow[b][wb][0]);
              r1 = *reinterpret_cast<const float4*>(&prow[b][wb][4]);
              const bool win = wb == warp && key == kb;
              pq = win ? c : pq;
              cand = cand && !win;
              bad |= kb < 64u || kb >= 0x7f800020u;  // zero, infinite or NaN
              f = cand ? v[0] * __uint_as_float(iv) : 0.f;
              last = cand ? -f : last;
            }
            v[0] = fmaf(-f, r0.y, v[1]), v[1] = fmaf(-f, r0.z, v[2]), v[2] = fmaf(-f, r0.w, v[3]);
            v[3] = fmaf(-f, r1.x, v[4]), v[4] = fmaf(-f, r1.y, v[5]), v[5] = fmaf(-f, r1.z, v[6]);
            v[6] = fmaf(-f, r1.w, v[7]);
            v[7] = last;
          }
          if (pq >= 0) {
            pj = 8 * q + pq;
#pragma unroll
            for (int k = 0; k < 6; ++k)
              *reinterpret_cast<float4*>(&pblk[q & 1][pq][4 * k]) =
                  make_float4(v[8 + 4 * k], v[9 + 4 * k], v[10 + 4 * k], v[11 + 4 * k]);
          }
          __syncwarp();
          asm volatile("bar.sync 1, %0;" ::"r"(npw * 32) : "memory");
          // rows eliminated before this sub-block and slots without a row do not change
          const bool live = cand || pq >= 0;
          float t[8], w8[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            w8[k] = v[k];
            t[k] = live && (pq < 0 || k < pq) && ((mask >> (8 * q + k)) & 1u) ? v[k] : 0.f;
          }
#pragma unroll
          for (int k4 = 0; k4 < 6; ++k4) {
            float4 acc = make_float4(v[8 + 4 * k4], v[9 + 4 * k4], v[10 + 4 * k4], v[11 + 4 * k4]);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const float4 r = *reinterpret_cast<const float4*>(&pblk[q & 1][k][4 * k4]);
              acc.x = fmaf(t[k], r.x, acc.x), acc.y = fmaf(t[k], r.y, acc.y);
              acc.z = fmaf(t[k], r.z, acc.z), acc.w = fmaf(t[k], r.w, acc.w);
            }
            v[4 * k4] = acc.x, v[4 * k4 + 1] = acc.y, v[4 * k4 + 2] = acc.z, v[4 * k4 + 3] = acc.w;
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) v[24 + k] = w8[k];
        }
        if (s > 0) wait(&bar_u, (s - 1) & 1, false);
        if (pj >= 0) {
#pragma unroll
          for (int k = 0; k < 32; ++k) u11[pj * 33 + k] = k >= pj ? v[k] : 0.f;
#pragma unroll
          for (int k = 0; k < 32; ++k)
            if (k >= pj) v[k] = 0.f;
        }
        if (warp == 0 && !((mask >> lane) & 1u))
          for (int k = 0; k < 32; ++k) u11[lane * 33 + k] = k == lane ? 1.f : 0.f;
        // T of this panel: global (column k of the 32, slots contiguous) and the split operand
#pragma unroll
        for (int k = 0; k < 32; ++k) Tg[(static_cast<size_t>(s) * 32 + k) * NS + slot] = v[k];
        sjg[static_cast<size_t>(s) * NS + slot] = static_cast<signed char>(pj);
      }
      slotj[par][slot] = static_cast<signed char>(pj);
      if (s > 0) wait(&bar_rest, (s - 1) & 1, false);  // T and B are free again
      if (dmax > 0) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          float4 h, l;
          split_tf32(v[4 * q], h.x, l.x);
          split_tf32(v[4 * q + 1], h.y, l.y);
          split_tf32(v[4 * q + 2], h.z, l.z);
          split_tf32(v[4 * q + 3], h.w, l.w);
          const int o = slot * 32 + ((q ^ (slot & 7)) << 2);
          *reinterpret_cast<float4*>(Thi + o) = h;
          *reinterpret_cast<float4*>(Tlo + o) = l;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
    }
    __syncthreads();  // T in place, pivots known; the window of the panel before is complete in tensor memory
    tc_fence_after();
    const int j = slotj[par][slot];
    const int tnew = s + 1 + RC;  // a row of chunk tnew takes this slot
    const bool enter = tnew < np, fresh = j >= 0 && enter && ((chunk_mask(w, tnew) >> j) & 1u);
    const unsigned mine = own(j & 31);
    if (dmax > 0) {
      if (tid == 32 && enter && !quit) {
        expect_tx(&bar_t0, 4096);
        bulk_load(t0, block(tnew, 0), 4096, &bar_t0);
        sent = true;
      }
      // the pivot rows' window, split, as the K-major B operand: chunk s + 1, which the next panel needs,
      // by the panel warps, whose product is issued at once, the others by the other half
      const int cnt = dmax + (nfc - fc0);
      auto convert = [&](int c) {
        const int col = c < dmax ? ((s + 1 + c) % RS) * 32 : (RS + fc0 + c - dmax) * 32;
        float r[32];
        tmem_ld32(tmem + col, r);
        if (j >= 0) {
          float* bh = Bhi + col * 32 + (j & 3);
          float* bl = Blo + col * 32 + (j & 3);
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            float h, l;
            split_tf32(r[i], h, l);
            const int o = i * 32 + (((j >> 2) ^ (i & 7)) << 2);
            bh[o] = h;
            bl[o] = l;
          }
        }
      };
      // warp 0 issues the first product, warp 5 the rest (not a panel warp: the tensor cores' queue holds
      // the issuing thread up). Both loops stay rolled: unrolled over k inside the rolled loop over column groups
      // the products came out wrong, the same every time; with both rolled, or both unrolled, they are right. The
      // cause was not found (the loads from tensor memory and their wait were two statements then, see
      // tmem_ld32; the form has not been run again). Speed is no reason: the queue bounds the issue.
      auto issue = [&](int col, int ncol) {
        const uint64_t dah = sdesc(saddr(Thi)), dal = sdesc(saddr(Tlo)), dbh = sdesc(saddr(Bhi)), dbl = sdesc(saddr(Blo));
        const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | (static_cast<uint32_t>(ncol >> 3) << 17) |
                               (static_cast<uint32_t>(kSlots >> 4) << 24);
        const uint64_t off = static_cast<uint64_t>(col) * 8;  // 128-byte rows in units of 16 bytes
        const uint32_t d = tmem_base + col;
        if (lane == 0 && !quit) {
#pragma unroll 1
          for (int k = 0; k < 4; ++k) {  // 8 TF32 columns = 32 bytes inside the swizzle row
            mma_tf32(d, dal + 2 * k, dbh + off + 2 * k, idesc);
            mma_tf32(d, dah + 2 * k, dbl + off + 2 * k, idesc);
            mma_tf32(d, dah + 2 * k, dbh + off + 2 * k, idesc);
          }
        }
        __syncwarp();
      };
      auto converted = [&]() {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncwarp();
      };
#pragma unroll 1
      for (int c = panel_warp ? 0 : 1; c < (panel_warp ? 1 : cnt); ++c) {
        convert(c);
        if (c == 0) {
          converted();
          asm volatile("bar.sync 3, 128;" ::: "memory");
          if (warp == 0) {
            tc_fence_after();
            issue(((s + 1) % RS) * 32, 32);
            if (lane == 0 && !quit) mma_commit(&bar_next), sent = true;
            __syncwarp();
          }
        }
      }
      if (!panel_warp) {
        converted();
        asm volatile("bar.sync 4, 128;" ::: "memory");  // the other chunks are in place
        tc_fence_after();
        if (warp == 5) {
          // the other ring chunks, slots (s + 2) % RS .. (s + dmax) % RS, wrapping, then the far columns
          // (at most 256 columns an instruction)
          const int q2 = (s + 2) % RS, m = dmax - 1, m1 = imin(m, RS - q2);
#pragma unroll 1
          for (int r = 1; r < 5; ++r) {
            int col = q2 * 32, n = m1 * 32;
            if (r == 2) col = 0, n = (m - m1) * 32;
            if (r >= 3) col = (RS + fc0) * 32 + (r - 3) * 256, n = imin(256, (nfc - fc0) * 32 - (r - 3) * 256);
            if (n > 0) issue(col, n);
          }
          if (lane == 0 && !quit) {
            mma_commit(&bar_rest);
            if (a.probe && s == 0) quit = !mbar_wait(&never, 0, &gave_up, a.status, kProbeCycles);
            wait(&bar_next, par, false);
            wait(&bar_rest, par, true);
            if (enter && !quit) {
              // the products are done: B's remainders give way to the entering rows' templates, chunk d of
              // the ring to template chunk d - 1, the chunk that enters (in the place of chunk s + 1) to RS
              const int far = nfc - fc0, last = s + 1 + RS < np ? RS + 1 : dmax;
              expect_tx(&bar_tmpl, 4096u * (last - 1 + far));
              for (int d = 2; d <= last; ++d) bulk_load(Blo + ((s + d) % RS) * 1024, block(tnew, d - 1), 4096, &bar_tmpl);
              for (int c = fc0; c < nfc; ++c) bulk_load(Blo + (RS + c) * 1024, block(tnew, RS + 1 + c), 4096, &bar_tmpl);
              sent = true;
            }
          }
          __syncwarp();
        }
      }
    }
    float* Up = Ug + s * ustride;
    if (warp == 4) {
      // inv(U11) by one warp: the two 16 x 16 diagonal blocks at once (one lane a column, the rows in
      // turning registers), then -inv(A) B inv(D)
      const float* u = u11;
      const int blk = lane >> 4, c = lane & 15;
      const float* d = u + blk * 16 * 34;
      const float rd = recip(d[c * 34]);
      float x[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) x[r] = r == c ? 1.f : 0.f;
#pragma unroll 1
      for (int k = 15; k >= 0; --k) {
        const float xk = x[15] * __shfl_sync(0xffffffffu, rd, (lane & 16) + k);
        ui[(blk * 16 + k) * 17 + c] = xk;
        const float* dk = d + (k - 16) * 33 + k;  // row k - 16 + i, column k; rows above the block are not used
#pragma unroll
        for (int i = 15; i > 0; --i) x[i] = fmaf(-dk[max(i, 16 - k) * 33], xk, x[i - 1]);
        x[0] = 0.f;
      }
      __syncwarp();
      // rows blk * 8 .. + 7 of the upper right block, column c
      float t[16], y[8];
#pragma unroll
      for (int r = 0; r < 16; ++r) t[r] = 0.f;
#pragma unroll 1
      for (int k = 0; k < 16; ++k) {
        const float z = ui[(16 + k) * 17 + c];
#pragma unroll
        for (int r = 0; r < 16; ++r) t[r] = fmaf(u[r * 33 + 16 + k], z, t[r]);
      }
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        float acc = 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) acc = fmaf(-ui[(blk * 8 + r) * 17 + k], t[k], acc);
        y[r] = acc;
      }
      // by rows, the pieces of a row exchanged like a block's
      auto at = [&](int r, int col) { return Up + r * 32 + ((((col >> 2) ^ (r & 7)) << 2) | (col & 3)); };
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        *at(r, lane) = lane < 16 ? ui[r * 17 + c] : 0.f;
        *at(16 + r, lane) = lane < 16 ? 0.f : ui[(16 + r) * 17 + c];
      }
      __syncwarp();
#pragma unroll
      for (int r = 0; r < 8; ++r) *at(blk * 8 + r, 16 + c) = y[r];
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&bar_u)) : "memory");
    }
    if (dmax == 0) break;
    if (panel_warp) {
      // the next panel's columns: updated rows from tensor memory, the entering rows from the template; the
      // pivot rows go to the place of B's heads as U, from where they are copied out below
      float r[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = 0.f;
      if (enter) {
        wait(&bar_t0, par, sent && tid == 32);
        if (fresh) {
          load_row(t0, j, v);
          scale_row(v, mine, E);
        }
      }
      wait(&bar_next, par, sent && tid == 0);
      tc_fence_after();
      tmem_ld32(tmem + ((s + 1) % RS) * 32, r);
      if (j >= 0) {
        store_row(Bhi + ((s + 1) % RS) * 1024, j, r);
        act = fresh;
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = r[i];
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      asm volatile("bar.arrive 2, %0;" ::"r"(kThreads) : "memory");
    } else {
      wait(&bar_rest, par, false);
      tc_fence_after();
      if (enter) wait(&bar_tmpl, par, sent);
      const int cnt = dmax - 1 + nfc - fc0;
#pragma unroll 1
      for (int q = 0; q < cnt; ++q) {
        const bool ring = q < dmax - 1;
        const int at = ring ? (s + 2 + q) % RS : RS + fc0 + q - (dmax - 1);
        float r[32];
        tmem_ld32(tmem + at * 32, r);
        if (j >= 0) {
          store_row(Bhi + at * 1024, j, r);
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = 0.f;
          if (fresh) {
            load_row(Blo + at * 1024, j, r);
            if (ring) scale_row(r, mine, E);
          }
        }
        tmem_st32(tmem + at * 32, r);
      }
      tmem_wait_st();
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      asm volatile("bar.sync 2, %0;" ::"r"(kThreads) : "memory");  // U is complete; chunk s + 1 has been read
      tc_fence_after();
      if (tid == 160 && !quit) {
        for (int d = 1; d <= dmax; ++d) bulk_store(Up + d * 1024, Bhi + ((s + d) % RS) * 1024, 4096);
        for (int c = fc0; c < nfc; ++c) bulk_store(Up + (1 + RS + c) * 1024, Bhi + (RS + c) * 1024, 4096);
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      }
      if (s + 1 + RS < np) {
        // chunk s + 1 + RS enters the ring in the place of chunk s + 1: the rows that stay have
        // entries only in its l = 0 columns, so far kept apart
        const int at = (s + 1) % RS;
        const uint32_t t = tmem + at * 32;
        float r[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) r[i] = 0.f;
        if (fresh) {
          load_row(Blo + at * 1024, j, r);
          scale_row(r, mine, E);
        }
        tmem_st32(t, r);
        tmem_wait_st();
        for (int i = 0; i < g; ++i) {
          if ((s + 1 + RS) * g + i >= w.nr) break;
          const uint32_t tf = tmem + RS * 32 + s * g + i;
          float x = tmem_ld1(tf);
          if (fresh) {
            const int c = i * w.nlp;
            x = Blo[at * 1024 + j * 32 + ((((c >> 2) ^ (j & 7)) << 2) | (c & 3))] * ((mine >> c) & 1u ? 1.f : E);
          } else if (j >= 0) {
            x = 0.f;
          }
          tmem_st1(t + i * w.nlp, x);
          tmem_st1(tf, 0.f);
        }
        tmem_wait_st();
      }
      // B's heads are written again after the next barrier
      if (tid == 160) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      __syncwarp();
      tc_fence_before();
    }
  }
  if (tid == 160) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  if (bad) atomicOr(a.status, kZeroPivot);
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(static_cast<uint32_t>(w.tmem_cols)));
}

// FP64 path: the same elimination as two launches per panel, the window in a global scratch that stays
// in L2 ([nx][128][NU + 32]: the ring holds one chunk more than in tensor memory, the panel's own). The
// products run on the FP64 units, whose rate bounds them (7.2 GFLOP/s an SM), so the update of a
// panel is spread over all SMs, one CTA per point and 32-column chunk, whatever the number of
// points. (One CTA per point for the whole factorisation took 1.77 ms on the 32-point small grid and
// 23.7 ms on the medium one.)
struct PanelArgs {
  FactorArgs f;
  int s;
};

__device__ __forceinline__ int ring_col(const WindowPlan& w, int chunk) { return (chunk % (w.RS + 1)) * 32; }

// Rows of chunks 0 .. RC into the window: one CTA per point and slot.
__global__ void window_f64_init_kernel(const FactorArgs a) {
  const WindowPlan& w = a.w;
  const int pt = blockIdx.y, r = blockIdx.x, ldw = w.NU + 32, NWR = (w.RS + 1) * 32;
  double* D = a.W + (static_cast<size_t>(pt) * kSlots + r) * ldw;
  const double E = a.E ? a.E[pt] : a.Eu;
  if (threadIdx.x == 0) a.rows[pt * kSlots + r] = r;
  const bool valid = r < w.NS && r / 32 < w.np && ((chunk_mask(w, r / 32) >> (r & 31)) & 1u);
  const double* base = static_cast<const double*>(a.base) + static_cast<size_t>(r) * w.NW;
  const double* slope = static_cast<const double*>(a.slope) + static_cast<size_t>(r) * NWR;
  for (int c = threadIdx.x; c < ldw; c += blockDim.x) {
    // at panel 0 ring slot d holds chunk d
    double x = 0.0;
    if (valid) x = c < NWR ? fma(E, __ldg(slope + c), __ldg(base + c)) : __ldg(base + c);
    D[c] = x;
  }
}

// The 32 columns of panel s, one thread a slot: T, U11 and the pivots. Bound by the FP64 units of one SM
// (31 FMAs a column and thread) and the latency of the columns; nothing else runs on them here: the
// pivot's checks are made on its bits and its reciprocal takes two Newton steps.
__global__ void __launch_bounds__(kSlots) window_f64_panel_kernel(const PanelArgs pa) {
  const FactorArgs& a = pa.f;
  const WindowPlan& w = a.w;
  __shared__ __align__(16) double prow[2][4][32];
  __shared__ unsigned long long kval[2][4];
  const int pt = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, s = pa.s;
  const int np = w.np, NS = w.NS, npw = NS / 32;
  for (int i = tid; i < 256; i += kSlots) (&prow[0][0][0])[i] = 0.0;
  __syncthreads();
  const unsigned mask = chunk_mask(w, s);
  int pj = -1;
  bool bad = false;
  if (warp < npw) {
    const int row = a.rows[pt * kSlots + tid];  // the padded row in this slot
    bool cand = row < np * 32 && ((chunk_mask(w, row / 32) >> (row & 31)) & 1u);
    const double* D = a.W + (static_cast<size_t>(pt) * kSlots + tid) * (w.NU + 32) + ring_col(w, s);
    double v[32];
#pragma unroll
    for (int k = 0; k < 32; k += 2) {
      const double2 x = *reinterpret_cast<const double2*>(D + k);
      v[k] = cand ? x.x : 0.0, v[k + 1] = cand ? x.y : 0.0;
    }
    int b = 0;
#pragma unroll 1
    for (int j = 0; j < 32; ++j) {  // the registers turn as in window_lu_tc_kernel
      double f = 0.0, last = v[0];
      const double* pr = prow[0][0];
      if ((mask >> j) & 1u) {
        b ^= 1;
        // |v| as an ordered integer, candidates above the rest (NaN above all: reported below)
        const unsigned long long key =
            cand ? static_cast<unsigned long long>(__double_as_longlong(v[0]) & 0x7fffffffffffffffll) + 1ull : 0ull;
        const unsigned hi = static_cast<unsigned>(key >> 32), bh = __reduce_max_sync(0xffffffffu, hi);
        const unsigned lo = hi == bh ? static_cast<unsigned>(key) : 0u, bl = __reduce_max_sync(0xffffffffu, lo);
        const int src = __ffs(__ballot_sync(0xffffffffu, hi == bh && static_cast<unsigned>(key) == bl)) - 1;
        if (lane == src) {
#pragma unroll
          for (int k = 0; k < 32; k += 2) *reinterpret_cast<double2*>(&prow[b][warp][k]) = make_double2(v[k], v[k + 1]);
          kval[b][warp] = (static_cast<unsigned long long>(bh) << 32) | bl;
        }
        __syncwarp();
        asm volatile("bar.sync 1, %0;" ::"r"(npw * 32) : "memory");
        unsigned long long kb = kval[b][0];
        int wb = 0;
        for (int q = 1; q < npw; ++q)
          if (kval[b][q] > kb) kb = kval[b][q], wb = q;
        pr = prow[b][wb];
        if (wb == warp && lane == src) {
          pj = j;
          cand = false;
          if (kb < 2ull || kb > 0x7ff0000000000000ull) bad = true;  // zero, infinite or NaN
        }
        const double m = v[0] * recip(pr[0]);
        if (cand) f = m, last = -m;
      }
#pragma unroll
      for (int k = 0; k < 32; k += 2) {
        const double2 r = *reinterpret_cast<const double2*>(pr + k);
        if (k > 0) v[k - 1] = fma(-f, r.x, v[k]);
        v[k] = fma(-f, r.y, v[k + 1]);
      }
      v[31] = last;
    }
    // U11 goes where its inverse will be (window_f64_update_kernel inverts it in place)
    double* u11 = static_cast<double*>(a.U) + (static_cast<size_t>(pt) * np + s) * (1024 + 32 * static_cast<size_t>(w.NU));
    if (pj >= 0) {
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        u11[pj * 32 + k] = k >= pj ? v[k] : 0.0;
        if (k >= pj) v[k] = 0.0;
      }
    }
    if (warp == 0 && !((mask >> lane) & 1u))
      for (int k = 0; k < 32; ++k) u11[lane * 32 + k] = k == lane ? 1.0 : 0.0;
    double* T = static_cast<double*>(a.T) + (static_cast<size_t>(pt) * np + s) * 32 * NS;
#pragma unroll
    for (int k = 0; k < 32; ++k) T[k * NS + tid] = v[k];
    a.slotj[(static_cast<size_t>(pt) * np + s) * NS + tid] = static_cast<signed char>(pj);
    if (pj >= 0) a.rows[pt * kSlots + tid] = (s + 1 + w.RC) * 32 + pj;
  }
  if (bad) atomicOr(a.status, kZeroPivot);
}

// U11 (32 x 32, row-major, upper triangular) <- its inverse, 128 threads, sm 3 x 16 x 17 values: the two
// 16 x 16 diagonal blocks at once (one lane a column, the rows in turning registers), then
// -inv(A) B inv(D) by 16 x 16 products.
__device__ void invert_u11(double* u, double* sm, int tid) {
  double* x = sm;               // [2][16][17]: the diagonal blocks' inverses
  double* t = sm + 2 * 16 * 17; // [16][17]: B inv(D)
  if (tid < 32) {
    const int blk = tid >> 4, c = tid & 15;
    const double* d = u + blk * 16 * 33;  // the block's corner
    const double rd = recip(d[c * 33]);
    double v[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = r == c ? 1.0 : 0.0;
#pragma unroll 1
    for (int k = 15; k >= 0; --k) {
      const double xk = v[15] * __shfl_sync(0xffffffffu, rd, (tid & 16) + k);
      x[(blk * 16 + k) * 17 + c] = xk;
#pragma unroll
      for (int i = 15; i > 0; --i) {
        const int r = k - 16 + i;  // the row now moving into place i
        v[i] = fma(r >= 0 ? -d[r * 32 + k] : 0.0, xk, v[i - 1]);
      }
      v[0] = 0.0;
    }
  }
  __syncthreads();
  for (int e = tid; e < 256; e += kSlots) {
    const int r = e >> 4, c = e & 15;
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 16; ++k) s = fma(u[r * 32 + 16 + k], x[(16 + k) * 17 + c], s);
    t[r * 17 + c] = s;
  }
  __syncthreads();
  for (int e = tid; e < 1024; e += kSlots) {
    const int r = e >> 5, c = e & 31;
    double s = 0.0;
    if (r >= 16 || c < 16) {
      s = (r >> 4) == (c >> 4) ? x[r * 17 + (c & 15)] : 0.0;
    } else {
#pragma unroll
      for (int k = 0; k < 16; ++k) s = fma(-x[r * 17 + k], t[k * 17 + c - 16], s);
    }
    u[r * 32 + c] = s;
  }
}

// D += T B on one chunk of the window after panel s; the pivot rows go out as U and the rows that
// enter take their slots. blockIdx.x: the ring chunks s + 1 .. s + dmax, the far chunks from the
// first that still has a live column, and last the chunk that enters the ring, whose l = 0 columns
// are the g far columns it takes over. Pivot rows that are zero on the chunk are left out of the
// product (on the outer half of the ring all but the rows that pivoting brought forward). One more CTA per
// point inverts U11 meanwhile.
__global__ void __launch_bounds__(kSlots) window_f64_update_kernel(const PanelArgs pa, int dmax, int fc0, int nfc) {
  const FactorArgs& a = pa.f;
  const WindowPlan& w = a.w;
  extern __shared__ __align__(1024) unsigned char raw[];
  double* Ts = reinterpret_cast<double*>(raw);  // [32][128], rows of T in use, in the order of ks
  double* Bs = Ts + kPW * kSlots;               // [32][32]
  __shared__ signed char slotj[kSlots];
  __shared__ int pslot[32], ks[32], nk;
  const int pt = blockIdx.y, tid = threadIdx.x, lane = tid & 31, s = pa.s;
  const int np = w.np, NS = w.NS, RS = w.RS, g = w.g, NU = w.NU, ldw = NU + 32, NWR = (RS + 1) * 32;
  const double* base = static_cast<const double*>(a.base);
  const double* slope = static_cast<const double*>(a.slope);
  const double E = a.E ? a.E[pt] : a.Eu;
  double* D = a.W + static_cast<size_t>(pt) * kSlots * ldw;
  const double* T = static_cast<const double*>(a.T) + (static_cast<size_t>(pt) * np + s) * 32 * NS;
  double* U = static_cast<double*>(a.U) + (static_cast<size_t>(pt) * np + s) * (1024 + 32 * static_cast<size_t>(NU)) + 1024;
  if (blockIdx.x == gridDim.x - 1) {
    invert_u11(U - 1024, Ts, tid);
    return;
  }
  const int bx = blockIdx.x;
  const bool ring = bx < dmax, far = !ring && bx < dmax + nfc - fc0;
  // D's column for column i of the product: a ring chunk, a far chunk without the columns already taken
  // over, or the far columns s g + i that the entering chunk takes over
  const int fc = fc0 + bx - dmax, nfar = w.nr - w.kf0;
  const int col = ring ? ring_col(w, s + 1 + bx) : NWR + (far ? fc * 32 : s * g);
  const int ilo = far ? imax(0, (s + 1) * g - fc * 32) : 0;
  const int ihi = ring ? 32 : far ? imin(32, nfar - fc * 32) : imax(0, imin(g, nfar - s * g));
  auto dcol = [&](int i) -> int { return i >= ilo && i < ihi ? col + i : -1; };
  if (tid < 32) pslot[tid] = -1;
  __syncthreads();
  {
    const int j = tid < NS ? a.slotj[(static_cast<size_t>(pt) * np + s) * NS + tid] : -1;
    slotj[tid] = static_cast<signed char>(j);
    if (j >= 0) pslot[j] = tid;
  }
  __syncthreads();
  // the pivot rows with an entry on the chunk, 32 rows by four warps
  for (int k = tid >> 5; k < 32; k += 4) {
    const int ps = pslot[k], dc = dcol(lane);
    const double x = ps >= 0 && dc >= 0 ? D[static_cast<size_t>(ps) * ldw + dc] : 0.0;
    const bool any = __any_sync(0xffffffffu, (__double_as_longlong(x) & 0x7fffffffffffffffll) != 0);
    Bs[k * 32 + lane] = x;
    if (lane == 0) ks[k] = any ? 1 : 0;
  }
  __syncthreads();
  if (tid < 32) {
    const bool has = ks[tid] != 0;
    const unsigned m = __ballot_sync(0xffffffffu, has);
    __syncwarp();
    if (has) ks[__popc(m & ((1u << tid) - 1u))] = tid;
    if (tid == 0) nk = __popc(m);
  }
  __syncthreads();
  const int cnt = nk;
  for (int q = 0; q < cnt; ++q) Ts[q * kSlots + tid] = tid < NS ? __ldg(T + ks[q] * NS + tid) : 0.0;
  // 4 rows (lane + 32 q) x 8 columns (of the warp) a thread: a warp whose columns are not in use has no
  // FP64 work
  const int c0 = 8 * (tid >> 5);
  const bool work = c0 < ihi && c0 + 8 > ilo, entering = !ring && !far;
  double acc[4][8];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const double* dr = D + static_cast<size_t>(lane + 32 * q) * ldw;
#pragma unroll
    for (int c = 0; c < 8; c += 2) {
      acc[q][c] = acc[q][c + 1] = 0.0;
      if (!work) continue;
      if (entering) {  // its far columns start anywhere
        const int d0 = dcol(c0 + c), d1 = dcol(c0 + c + 1);
        if (d0 >= 0) acc[q][c] = dr[d0];
        if (d1 >= 0) acc[q][c + 1] = dr[d1];
      } else {
        const double2 x = *reinterpret_cast<const double2*>(dr + col + c0 + c);
        acc[q][c] = x.x, acc[q][c + 1] = x.y;
      }
    }
  }
  __syncthreads();
  if (work) {
#pragma unroll 2
    for (int k = 0; k < cnt; ++k) {
      const double* b = Bs + ks[k] * 32 + c0;
      const double2 b0 = *reinterpret_cast<const double2*>(b), b1 = *reinterpret_cast<const double2*>(b + 2);
      const double2 b2 = *reinterpret_cast<const double2*>(b + 4), b3 = *reinterpret_cast<const double2*>(b + 6);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (32 * q >= NS) break;  // slots not in use
        const double t = Ts[k * kSlots + lane + 32 * q];
        acc[q][0] = fma(t, b0.x, acc[q][0]), acc[q][1] = fma(t, b0.y, acc[q][1]);
        acc[q][2] = fma(t, b1.x, acc[q][2]), acc[q][3] = fma(t, b1.y, acc[q][3]);
        acc[q][4] = fma(t, b2.x, acc[q][4]), acc[q][5] = fma(t, b2.y, acc[q][5]);
        acc[q][6] = fma(t, b3.x, acc[q][6]), acc[q][7] = fma(t, b3.y, acc[q][7]);
      }
    }
  }
  const int tnew = s + 1 + w.RC;
  const unsigned mnew = tnew < np ? chunk_mask(w, tnew) : 0u;
  const int ecol = ring_col(w, s + 1 + RS);  // where the entering chunk goes: the panel's own place
  const int uoff = ring ? bx * 32 : col - 32;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = lane + 32 * q, j = slotj[r];
    const bool fresh = j >= 0 && ((mnew >> j) & 1u);
    const size_t row = static_cast<size_t>(tnew) * 32 + (j >= 0 ? j : 0);
    double* dr = D + static_cast<size_t>(r) * ldw;
    if (entering) {
      // columns 0, nlp, 2 nlp .. of the chunk are the far columns; a fresh row brings its own values
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int i = c0 + c;
        if (dcol(i) >= 0) {
          if (j >= 0) U[static_cast<size_t>(j) * NU + uoff + i] = acc[q][c];
          else dr[ecol + i * w.nlp] = acc[q][c];
        }
        const int b = i / w.nlp;  // column i of the chunk is not a far column, or the row is fresh or gone
        if (j >= 0)
          dr[ecol + i] = fresh ? fma(E, __ldg(slope + row * NWR + RS * 32 + i), __ldg(base + row * w.NW + RS * 32 + i)) : 0.0;
        else if (i % w.nlp != 0 || b >= ihi)
          dr[ecol + i] = 0.0;
      }
    } else if (work) {
      if (j >= 0) {
        double* ur = U + static_cast<size_t>(j) * NU + uoff + c0;
#pragma unroll
        for (int c = 0; c < 8; c += 2)
          if (c0 + c >= ilo) *reinterpret_cast<double2*>(ur + c) = make_double2(acc[q][c], acc[q][c + 1]);
          else if (c0 + c + 1 >= ilo) ur[c + 1] = acc[q][c + 1];
        const double* bp = base + row * w.NW + (ring ? bx * 32 : col) + c0;
        const double* sp = slope + row * NWR + bx * 32 + c0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          acc[q][c] = 0.0;
          if (fresh) acc[q][c] = ring ? fma(E, __ldg(sp + c), __ldg(bp + c)) : __ldg(bp + c);
        }
      }
#pragma unroll
      for (int c = 0; c < 8; c += 2)
        if (c0 + c >= ilo)
          *reinterpret_cast<double2*>(dr + col + c0 + c) = make_double2(acc[q][c], acc[q][c + 1]);
        else if (c0 + c + 1 >= ilo)
          dr[col + c0 + c + 1] = acc[q][c + 1];
    }
  }
}

// ---------------------------------------------------------------- solves and refinement

struct SolveArgs {
  WindowPlan w;
  const void* T;
  const void* U;
  const signed char* slotj;
  const double* in;         // right-hand sides and results [nx][nt nr]
  double* out;
  const double* E;
  double Eu, dt;
  ResidualOps ro;
  MassBand mass;
  const double *TO, *TS;
  double ts_inf, to_inf;    // infinity norms of T_S and T_O
  double* vec;              // [nx][3 n]: y, z, rho
  double* fmax_;            // [nx] max|f|
  const double* minv;       // [nr] 1 / sum_k |M_pk|
  const double* rscale;     // [nr] the factors' row scale
  double* ratio;
  int* conv;
  double tol, kc_inf, ka_inf;
  double skip_tol, skip_floor;  // launch_window_residual
  int nt;
  int stages;
  unsigned stage_bytes;
  unsigned* status;
  int probe;                // a wait runs out behind the first copies
};

template <typename T>
struct Vec4;
template <>
struct Vec4<float> {
  static __device__ __forceinline__ float dot(const float* a, const float* b) {
    const float4 x = *reinterpret_cast<const float4*>(a), y = *reinterpret_cast<const float4*>(b);
    return fmaf(x.w, y.w, fmaf(x.z, y.z, fmaf(x.y, y.y, x.x * y.x)));
  }
  static __device__ __forceinline__ float4 load(const float* a) { return *reinterpret_cast<const float4*>(a); }
};
template <>
struct Vec4<double> {
  static __device__ __forceinline__ double dot(const double* a, const double* b) {
    const double2 x = *reinterpret_cast<const double2*>(a), y = *reinterpret_cast<const double2*>(b);
    const double2 z = *reinterpret_cast<const double2*>(a + 2), u = *reinterpret_cast<const double2*>(b + 2);
    return fma(z.y, u.y, fma(z.x, u.x, fma(x.y, y.y, x.x * y.x)));
  }
  struct Four {
    double x, y, z, w;
  };
  static __device__ __forceinline__ Four load(const double* a) {
    const double2 p = *reinterpret_cast<const double2*>(a), q = *reinterpret_cast<const double2*>(a + 2);
    return {p.x, p.y, q.x, q.y};
  }
};

constexpr int kEval = 512;  // threads of the projection and residual kernels

// Running maxima of magnitudes as ordered integers: the FP64 units, whose rate bounds these kernels, take
// no part (a NaN is above everything and stays).
using Mag = unsigned long long;
__device__ __forceinline__ Mag mag(double v) { return static_cast<Mag>(__double_as_longlong(v) & 0x7fffffffffffffffll); }
__device__ __forceinline__ Mag mag_max(Mag a, Mag b) { return a > b ? a : b; }

// Block-wide maximum of two magnitudes; every thread gets the result.
__device__ __forceinline__ void block_max2(Mag p, Mag q, Mag* red, double& pm, double& qm) {
  for (int o = 16; o > 0; o >>= 1) {
    p = mag_max(p, __shfl_xor_sync(0xffffffffu, p, o));
    q = mag_max(q, __shfl_xor_sync(0xffffffffu, q, o));
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = p, red[kEval / 32 + (threadIdx.x >> 5)] = q;
  __syncthreads();
  p = red[0], q = red[kEval / 32];
  for (int i = 1; i < kEval / 32; ++i) p = mag_max(p, red[i]), q = mag_max(q, red[kEval / 32 + i]);
  pm = __longlong_as_double(static_cast<long long>(p));
  qm = __longlong_as_double(static_cast<long long>(q));
}

// The solves run in the harmonic basis: y = P_S f, z the harmonic solution (x = f + P_O (z - y)); the
// residual of the system that was factored, rho = M (y - z) + dt (C + E A_v) z, needs only banded
// products, and r = P_O M^-1 rho is the residual of A_i x = f (P_S x = z).

// y = P_S f, z = 0, rho = M y, max|f|. By parity: Y_l(-mu) = (-1)^l Y_l(mu) and the ordinates are
// symmetric, so the sums over a half of them with f(a) +- f(nt - 1 - a) give the even and the odd
// harmonics: half the FP64 operations, which bound it.
__global__ void __launch_bounds__(kEval) window_project_kernel(const SolveArgs a) {
  extern __shared__ __align__(1024) unsigned char raw[];
  const int nr = a.w.nr, nl = a.w.nl, nt = a.nt, n = nl * nr, nv = nt * nr, hf = nt / 2, hc = (nt + 1) / 2;
  double* fold = reinterpret_cast<double*>(raw);  // 2 hc nr
  double* ys = fold + 2 * hc * nr;                // n
  __shared__ Mag red[2 * kEval / 32];
  const int pt = blockIdx.x, tid = threadIdx.x;
  const double* f = a.in + static_cast<size_t>(pt) * nv;
  double* y = a.vec + static_cast<size_t>(pt) * 3 * n;
  Mag mf = 0;
  for (int i = tid; i < hc * nr; i += kEval) {
    const int q = i / nr, k = i % nr;
    const double p = f[i], m = q < hf ? f[(nt - 1 - q) * nr + k] : 0.0;
    fold[i] = p + m;
    fold[hc * nr + i] = q < hf ? p - m : 0.0;
    mf = mag_max(mf, mag_max(mag(p), mag(m)));
  }
  double mb, unused;
  block_max2(mf, 0, red, mb, unused);
  if (tid == 0) {
    a.fmax_[pt] = mb;
    if (a.conv) a.conv[pt] = 0;
  }
  for (int i = tid; i < n; i += kEval) {
    const int l = i / nr, k = i % nr;
    const double* src = fold + (l & 1 ? hc * nr : 0) + k;
    const double* ts = a.TS + l * nt;
    double s0 = 0.0, s1 = 0.0;
    int q = 0;
    for (; q + 1 < hc; q += 2) {
      s0 = fma(__ldg(ts + q), src[q * nr], s0);
      s1 = fma(__ldg(ts + q + 1), src[(q + 1) * nr], s1);
    }
    if (q < hc) s0 = fma(__ldg(ts + q), src[q * nr], s0);
    ys[i] = s0 + s1;
    y[i] = s0 + s1;
    y[n + i] = 0.0;
  }
  __syncthreads();
  const int mw = a.mass.w, bw = 2 * mw + 1;
  for (int i = tid; i < n; i += kEval) {
    const int l = i / nr, p = i % nr;
    const double* mr = a.mass.m + static_cast<size_t>(p) * bw + mw - p;
    double s = 0.0;
    for (int k = imax(0, p - mw); k <= imin(nr - 1, p + mw); ++k) s = fma(__ldg(mr + k), ys[l * nr + k], s);
    y[2 * n + i] = s;
  }
}

// z += H^-1 rho through the window factors, one CTA per point. The factors are streamed once, panel by
// panel (the T forwards, then inv(U11) and U backwards), through a ring of shared-memory stages
// filled by bulk copies; of the far blocks only those still to come are copied. On the medium grid
// (128 points of 64 x 32, FP32) 0.40 GB a solve, 60 us at the copy bandwidth; measured 88 us, one CTA an
// SM bound by the panels' chain (a panel 1000 cycles forwards, 1200 backwards). It was 119 us with the
// stage found by a division, the ranks read one panel ahead and the far columns gathered from the
// unknowns. 256 points of 128 x 32: 274 us of 262 us at the copy bandwidth, two CTAs an SM (314 with the copy of the
// next block issued half a panel later; one CTA with twice the stages was slower by a tenth). Vectors are read and written by rows: 1.4 times the solve
// when each lane wrote a row of its own. Converged points return at once.
template <typename T>
__global__ void __launch_bounds__(kThreads, 2) window_substitute_kernel(const SolveArgs a) {
  extern __shared__ __align__(1024) unsigned char raw[];
  const WindowPlan& w = a.w;
  const int pt = blockIdx.x, tid = threadIdx.x;
  if (a.conv && a.conv[pt]) return;
  const int np = w.np, NS = w.NS, NU = w.NU, RS = w.RS, RC = w.RC, g = w.g, nl = w.nl, nr = w.nr, nlp = w.nlp;
  const int n = nl * nr, S = a.stages;
  const unsigned fbytes = 32u * NS * sizeof(T), bbytes = (1024u + 32u * NU) * sizeof(T);
  unsigned char* stage = raw;
  T* b = reinterpret_cast<T*>(raw + static_cast<size_t>(S) * a.stage_bytes);  // padded unknowns, chunk by chunk
  const int npad = (np + RS) * 32;
  // U's rows: FP64 [32][NU]; FP32 32 x 32 blocks, one per chunk of the window, as load_row reads them
  constexpr bool blocks = sizeof(T) == 4;
  T* x0 = b + npad + 64;  // [NF] the solution at the far columns
  T* bp = b + npad;       // [2][32] pivot values; the backward pass's 32 partial results
  double* z = a.vec + static_cast<size_t>(pt) * 3 * n + n;
  const double* rho = z + n;
  __shared__ __align__(8) uint64_t full[8], never;
  __shared__ int gave_up;
  const T* Tg = static_cast<const T*>(a.T) + static_cast<size_t>(pt) * np * 32 * NS;
  const size_t ustride = 1024 + 32 * static_cast<size_t>(NU);
  const T* Ug = static_cast<const T*>(a.U) + static_cast<size_t>(pt) * np * ustride;
  const signed char* sj = a.slotj + static_cast<size_t>(pt) * np * NS;
  const int nfar = imax(0, nr - w.kf0);
  // the far blocks of panel s that are still to be taken over
  auto far0 = [&](int s) { return imin((s * g) >> 5, w.NF >> 5); };
  auto far1 = [&](int s) { return s * g < nfar && s + 1 < np ? w.NF >> 5 : far0(s); };
  // the q-th copy: the T of panels 0 .. np - 1, then the U of panels np - 1 .. 0, into stage q mod S; by thread
  // 0, which also waits for each of them and stops when that fails
  bool quit = false;
  int issued = 0;
  auto issue = [&](int q, int st) {
    if (quit) return;
    issued = q + 1;
    T* dst = reinterpret_cast<T*>(stage + static_cast<size_t>(st) * a.stage_bytes);
    if (q < np) {
      expect_tx(&full[st], fbytes);
      bulk_load(dst, Tg + static_cast<size_t>(q) * 32 * NS, fbytes, &full[st]);
      return;
    }
    const int s = 2 * np - 1 - q;
    const T* src = Ug + static_cast<size_t>(s) * ustride;
    if constexpr (!blocks) {
      expect_tx(&full[st], bbytes);
      bulk_load(dst, src, bbytes, &full[st]);
    } else {  // the blocks that the panel's row reads
      const unsigned near = 4096u * (1 + imin(RS, np - 1 - s)), off = 1024u * (1 + RS + far0(s));
      const unsigned far = 4096u * (far1(s) - far0(s));
      expect_tx(&full[st], near + far);
      bulk_load(dst, src, near, &full[st]);
      if (far) bulk_load(dst + off, src + off, far, &full[st]);
    }
  };
  if (tid == 0) {
    for (int i = 0; i < S; ++i) mbar_init(&full[i], 1);
    mbar_init(&never, 1);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    for (int q = 0; q < imin(S, 2 * np); ++q) issue(q, q);
    if (a.probe) quit = !mbar_wait(&never, 0, &gave_up, a.status, kProbeCycles);
  }
  const int sh = 31 - __clz(nlp);
  for (int i = tid; i < npad + 64 + w.NF; i += kThreads) b[i] = T(0);  // unused unknowns stay zero
  __syncthreads();
  // rho and z by rows, whole lines at a time; the columns' conflicts in shared memory cost less
  for (int i = tid; i < n; i += kThreads) {
    const int l = i / nr, k = i - l * nr;
    b[(k << sh) + l] = static_cast<T>(__ldg(a.rscale + k) * rho[i]);
  }
  __syncthreads();
  // the stage and phase of the copy in use, advanced by hand (a division by S costs as much as the product)
  int st = 0;
  uint32_t ph = 0;
  auto advance = [&]() {
    if (++st == S) st = 0, ph ^= 1u;
  };
  // forward: one thread a slot
  if (tid < NS) {
    T wv = tid < npad ? b[tid] : T(0);
    // the slots' ranks are read four panels ahead: a panel is shorter than a load from memory
    auto rank_of = [&](int s) { return s < np ? static_cast<int>(sj[static_cast<size_t>(s) * NS + tid]) : -1; };
    int j1 = rank_of(0), j2 = rank_of(1), j3 = rank_of(2), j4 = rank_of(3), freed = 0;
    for (int s = 0; s < np; ++s) {
      const int j = j1;
      j1 = j2, j2 = j3, j3 = j4, j4 = rank_of(s + 4);
      T* q = bp + (s & 1) * 32;
      if (j >= 0) q[j] = wv;
      asm volatile("bar.sync 1, %0;" ::"r"(NS) : "memory");
      // every slot's thread is past panel s - 1: its stage can be filled again
      if (tid == 0 && ring_before_wait(s, np, S) >= 0) issue(ring_before_wait(s, np, S), freed);
      freed = st;
      if (!mbar_wait(&full[st], ph, &gave_up, a.status)) quit = true;
      const T* t = reinterpret_cast<const T*>(stage + static_cast<size_t>(st) * a.stage_bytes) + tid;
      T acc[4] = {wv, T(0), T(0), T(0)};
#pragma unroll
      for (int k = 0; k < 32; k += 4) {
        const auto p = Vec4<T>::load(q + k);
        acc[0] = fma(t[k * NS], p.x, acc[0]);
        acc[1] = fma(t[(k + 1) * NS], p.y, acc[1]);
        acc[2] = fma(t[(k + 2) * NS], p.z, acc[2]);
        acc[3] = fma(t[(k + 3) * NS], p.w, acc[3]);
      }
      wv = (acc[0] + acc[1]) + (acc[2] + acc[3]);
      if (j >= 0) {
        b[s * 32 + j] = wv;  // y of this panel; the chunk that enters takes the slot
        wv = s + 1 + RC < np ? b[(s + 1 + RC) * 32 + j] : T(0);
      }
      advance();
    }
  } else {
    for (int s = 0; s < np; ++s) advance();
  }
  __syncthreads();
  if (tid == 0 && ring_after_use(np - 1, np, S) >= 0) issue(ring_after_use(np - 1, np, S), st == 0 ? S - 1 : st - 1);
  // backward: eight threads a row of U. Columns past the window and far columns already taken over hold
  // zeros, their unknowns are finite: no conditions.
  const int row = tid >> 3, sub = tid & 7;
  for (int s = np - 1; s >= 0; --s) {
    const int q = 2 * np - 1 - s, nring = imin(RS, np - 1 - s);
    const int f0 = far0(s), f1 = far1(s);
    if (!mbar_wait(&full[st], ph, &gave_up, a.status)) quit = true;
    const T* ui = reinterpret_cast<const T*>(stage + static_cast<size_t>(st) * a.stage_bytes);
    const T* x = b + (s + 1) * 32;
    const int c4 = blocks ? 4 * (sub ^ (row & 7)) : 4 * sub;  // logical columns of the thread's piece
    const T* u = ui + 1024 + (blocks ? row * 32 : row * NU) + 4 * sub;
    const int cs = blocks ? 1024 : 32;  // from chunk to chunk
    T s0 = T(0), s1 = T(0);
#pragma unroll
    for (int c = 0; c < 6; ++c)  // RS <= 6
      if (c < nring) (c & 1 ? s1 : s0) += Vec4<T>::dot(u + c * cs, x + c * 32 + c4);
#pragma unroll 2
    for (int c = f0; c < f1; ++c) s0 += Vec4<T>::dot(u + (RS + c) * cs, x0 + c * 32 + c4);
    T acc = s0 + s1;
    acc += __shfl_xor_sync(0xffffffffu, acc, 4);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    T* t = bp + (s & 1) * 32;
    if (sub == 0) t[row] = b[s * 32 + row] - acc;
    __syncthreads();  // the panel's right-hand side is complete
    T e = Vec4<T>::dot(ui + row * 32 + 4 * sub, t + c4);
    e += __shfl_xor_sync(0xffffffffu, e, 4);
    e += __shfl_xor_sync(0xffffffffu, e, 2);
    e += __shfl_xor_sync(0xffffffffu, e, 1);
    if (sub == 0) {
      const int k = (s * 32 + row) >> sh, l = row & (nlp - 1);
      b[s * 32 + row] = k < nr && l < nl ? e : T(0);
      if (l == 0 && k >= w.kf0 && k < nr) x0[k - w.kf0] = e;
    }
    __syncthreads();  // the panel's stage is read
    if (tid == 0 && ring_after_use(q, np, S) >= 0) issue(ring_after_use(q, np, S), st);
    advance();
  }
  __syncthreads();
  for (int i = tid; i < n; i += kThreads) {
    const int l = i / nr, k = i - l * nr;
    z[i] += static_cast<double>(b[(k << sh) + l]);
  }
  if (tid == 0 && quit)
    for (int q = imax(0, issued - S); q < issued; ++q) mbar_drain(&full[q % S], (q / S) & 1);
}

// With check: rho of the iterate, the convergence test of launch_residual (max|r| and max|x| at the
// ordinates; ratio, conv and the count in status[1] as it writes them) and, where the test was
// made, x into out. As long as a bound that costs one reduction (|rho_p| <= sum_k |M_pk| max|M^-1 rho|
// and |M^-1 rho| <= |T_S| max|r|) already shows a point to be short of the tolerance, neither the
// Cholesky substitution nor the projections are made, except at the last sweep. Without check: x alone.
// FP64 operations bound it: 75 us with the full test for 128 points of 64 x 32, 28 with the bound alone;
// a step's evaluations 157 us, 178 with the maxima on the FP64 units and the row sums of M formed here.
__global__ void __launch_bounds__(kEval) window_residual_kernel(const SolveArgs a, int check, int last) {
  extern __shared__ __align__(1024) unsigned char raw[];
  const int nr = a.w.nr, nl = a.w.nl, nt = a.nt, n = nl * nr, nv = nt * nr, hf = nt / 2, hc = (nt + 1) / 2;
  const int pt = blockIdx.x, tid = threadIdx.x;
  if (check && a.conv[pt]) return;
  double* z = reinterpret_cast<double*>(raw);  // n
  double* dz = z + n;                          // z - y
  double* q = dz + n;                          // rho, then M^-1 rho
  __shared__ Mag red[2 * kEval / 32];
  const double* f = a.in + static_cast<size_t>(pt) * nv;
  double* out = a.out + static_cast<size_t>(pt) * nv;
  double* vec = a.vec + static_cast<size_t>(pt) * 3 * n;
  const double Ei = a.E ? a.E[pt] : a.Eu;
  for (int i = tid; i < n; i += kEval) {
    const double zi = vec[n + i];
    z[i] = zi;
    dz[i] = zi - vec[i];
  }
  __syncthreads();
  double mb = 0.0, nA = 0.0;
  const double floor_ = fmin(kBackwardFloor, a.tol);
  if (check) {
    mb = a.fmax_[pt];
    nA = 1.0 + a.dt * (a.kc_inf + fabs(Ei) * a.ka_inf);
    const int mw = a.mass.w, bw = 2 * mw + 1;
    Mag lbm = 0, mzm = 0;
    for (int i = tid; i < n; i += kEval) {
      const int l = i / nr, p = i % nr;
      const int k0 = imax(0, p - mw), k1 = imin(nr - 1, p + mw);
      const double* zl = z + l * nr;
      const double* dl = dz + l * nr;
      const double* mr = a.mass.m + static_cast<size_t>(p) * bw + mw - p;
      double m = 0.0, c = 0.0, fl = 0.0;
      for (int k = k0; k <= k1; ++k) m = fma(-__ldg(mr + k), dl[k], m);
      if (l > 0) {
        const double* row = a.ro.band + static_cast<size_t>(p) * bw + mw - p;
        const double* fr = a.ro.fband + (static_cast<size_t>(l) * nr + p) * bw + mw - p;
        for (int k = k0; k <= k1; ++k) {
          c = fma(__ldg(row + k), zl[k], c);
          fl = fma(__ldg(fr + k), zl[k - nr], fl);
        }
      } else {
        const double* row = a.ro.c0 + static_cast<size_t>(p) * nr;
        for (int k = k0; k < nr; ++k) c = fma(__ldg(row + k), zl[k], c);
      }
      if (l + 1 < nl) {
        const double* fr = a.ro.fband + (static_cast<size_t>(nl + l) * nr + p) * bw + mw - p;
        for (int k = k0; k <= k1; ++k) fl = fma(__ldg(fr + k), zl[k + nr], fl);
      }
      const double r = m + a.dt * (c + Ei * fl);
      q[i] = r;
      vec[2 * n + i] = r;
      lbm = mag_max(lbm, mag(r * __ldg(a.minv + p)));
      mzm = mag_max(mzm, mag(dl[p]));
    }
    double lb, mz;
    block_max2(lbm, mzm, red, lb, mz);
    if (tid == 0) atomicAdd(a.status + 1, 1u);  // residual evaluations
    const double least = lb / a.ts_inf;
    if (!last && least > a.skip_tol * mb && least > a.skip_floor * (nA * (mb + a.to_inf * mz) + mb)) return;
    // q_l <- M^-1 q_l by the banded Cholesky factor, one thread a harmonic
    for (int l = tid; l < nl; l += kEval) mass_solve(q + l * nr, a.ro.chol, a.ro.cinv, nr, mw);
    __syncthreads();
  }
  // x = f + P_O (z - y) and, with check, r = P_O q, both by parity
  Mag mrm = 0, mxm = 0;
  for (int i = tid; i < hc * nr; i += kEval) {
    const int o = i / nr, k = i % nr;
    const double* to = a.TO + o * nl;
    double xe = 0.0, xo = 0.0, re = 0.0, ro = 0.0;
    for (int l = 0; l < nl; l += 2) {
      const double t0 = __ldg(to + l);
      xe = fma(t0, dz[l * nr + k], xe);
      if (check) re = fma(t0, q[l * nr + k], re);
      if (l + 1 < nl) {
        const double t1 = __ldg(to + l + 1);
        xo = fma(t1, dz[(l + 1) * nr + k], xo);
        if (check) ro = fma(t1, q[(l + 1) * nr + k], ro);
      }
    }
    const double x1 = f[i] + (xe + xo);
    mrm = mag_max(mrm, mag(re + ro)), mxm = mag_max(mxm, mag(x1));
    if (o < hf) {
      const size_t i2 = static_cast<size_t>(nt - 1 - o) * nr + k;
      const double x2 = f[i2] + (xe - xo);
      out[i2] = x2;
      mrm = mag_max(mrm, mag(re - ro)), mxm = mag_max(mxm, mag(x2));
    }
    out[i] = x1;
  }
  if (!check) return;
  double mr, mx;
  block_max2(mrm, mxm, red, mr, mx);
  if (tid == 0) {
    const double ratio = mb > 0.0 ? mr / mb : (mr > 0.0 ? INFINITY : 0.0);
    a.ratio[pt] = ratio;
    a.conv[pt] = ratio <= a.tol || mr <= floor_ * (nA * mx + mb) ? 1 : 0;
  }
}

// out = A^-T in for the adjoint (FP64 factors, no refinement): the transposed passes of
// window_substitute_kernel in reverse order. A^-1 = I + P_O (H^-1 M - I) P_S, so
// A^-T g = g + P_S^T (M H^-T - I) P_O^T g (M symmetric).
__global__ void __launch_bounds__(kThreads) window_solve_t_kernel(const SolveArgs a) {
  extern __shared__ __align__(1024) unsigned char raw[];
  const WindowPlan& w = a.w;
  const int pt = blockIdx.x, tid = threadIdx.x;
  const int np = w.np, NS = w.NS, NU = w.NU, RS = w.RS, RC = w.RC, g = w.g, nl = w.nl, nr = w.nr, nlp = w.nlp, nt = a.nt;
  const int nv = nt * nr, npad = (np + RS) * 32, n = nl * nr;
  double* x = reinterpret_cast<double*>(raw);  // npad: cotangents, then pivot results, then H^-T
  double* wv = x + npad;                       // kSlots
  double* v = wv + kSlots;                     // 32
  const double* f = a.in + static_cast<size_t>(pt) * nv;
  double* out = a.out + static_cast<size_t>(pt) * nv;
  double* gh = a.vec + static_cast<size_t>(pt) * 3 * n;
  const double* Tg = static_cast<const double*>(a.T) + static_cast<size_t>(pt) * np * 32 * NS;
  const size_t ustride = 1024 + 32 * static_cast<size_t>(NU);
  const double* Ug = static_cast<const double*>(a.U) + static_cast<size_t>(pt) * np * ustride;
  const signed char* sj = a.slotj + static_cast<size_t>(pt) * np * NS;
  const int nfar = imax(0, nr - w.kf0);
  for (int i = tid; i < npad; i += kThreads) x[i] = 0.0;
  if (tid < kSlots) wv[tid] = 0.0;
  __syncthreads();
  for (int i = tid; i < n; i += kThreads) {
    const int l = i / nr, k = i % nr;
    double s = 0.0;
    for (int q = 0; q < nt; ++q) s = fma(__ldg(a.TO + q * nl + l), f[q * nr + k], s);
    gh[i] = s;
    x[k * nlp + l] = s;
  }
  __syncthreads();
  const int row = tid >> 3, sub = tid & 7;
  for (int s = 0; s < np; ++s) {
    const double* ui = Ug + s * ustride;
    double e = 0.0;
    for (int r = sub; r < 32; r += 8) e = fma(__ldg(ui + r * 32 + row), x[s * 32 + r], e);
    e += __shfl_xor_sync(0xffffffffu, e, 4);
    e += __shfl_xor_sync(0xffffffffu, e, 2);
    e += __shfl_xor_sync(0xffffffffu, e, 1);
    if (sub == 0) v[row] = e;
    __syncthreads();
    if (tid < 32) x[s * 32 + tid] = v[tid];
    const int wr = imin(RS, np - 1 - s) * 32;
    const int f0 = s * g, nf = s + 1 < np ? imax(0, nfar - f0) : 0;
    for (int c = tid; c < wr + nf; c += kThreads) {
      const double* u = ui + 1024 + (c < wr ? c : RS * 32 + f0 + c - wr);
      double t = 0.0;
#pragma unroll 8
      for (int j = 0; j < 32; ++j) t = fma(__ldg(u + static_cast<size_t>(j) * NU), v[j], t);
      x[c < wr ? (s + 1) * 32 + c : (w.kf0 + f0 + c - wr) * nlp] -= t;
    }
    __syncthreads();
  }
  for (int s = np - 1; s >= 0; --s) {
    const int j = tid < NS ? sj[static_cast<size_t>(s) * NS + tid] : -1;
    if (j >= 0) {
      const double keep = x[s * 32 + j];
      // the row that entered this slot after panel s: its cotangent is complete
      if (s + 1 + RC < np) x[(s + 1 + RC) * 32 + j] = wv[tid];
      wv[tid] = keep;
    }
    __syncthreads();
    double e = 0.0;
    for (int q = sub; q < NS; q += 8) e = fma(__ldg(Tg + (static_cast<size_t>(s) * 32 + row) * NS + q), wv[q], e);
    e += __shfl_xor_sync(0xffffffffu, e, 4);
    e += __shfl_xor_sync(0xffffffffu, e, 2);
    e += __shfl_xor_sync(0xffffffffu, e, 1);
    if (sub == 0) v[row] = e;
    __syncthreads();
    if (j >= 0) wv[tid] += v[j];
    __syncthreads();
  }
  if (tid < NS && tid < np * 32) x[tid] = wv[tid];
  __syncthreads();
  for (int i = tid; i < nr * nlp; i += kThreads) x[i] *= __ldg(a.rscale + i / nlp);  // H^T = (factors)^T / scale
  __syncthreads();
  const int mw = a.mass.w, bw = 2 * mw + 1;
  for (int i = tid; i < n; i += kThreads) {
    const int l = i / nr, p = i % nr;
    const double* mr = a.mass.m + static_cast<size_t>(p) * bw + mw - p;
    double s = 0.0;
    for (int k = imax(0, p - mw); k <= imin(nr - 1, p + mw); ++k) s = fma(__ldg(mr + k), x[k * nlp + l], s);
    gh[i] = s - gh[i];
  }
  __syncthreads();
  for (int i = tid; i < nv; i += kThreads) {
    const int q = i / nr, k = i % nr;
    double s = f[i];
    for (int l = 0; l < nl; ++l) s = fma(__ldg(a.TS + l * nt + q), gh[l * nr + k], s);
    out[i] = s;
  }
}

}  // namespace

std::vector<double> window_row_scale(const HostOps& o, bool levelled) {
  if (!levelled) return std::vector<double>(o.nr, 1.0);
  std::vector<double> s(o.nr);
  double most = 0.0;
  for (int p = 0; p < o.nr; ++p) {
    for (int k = 0; k < o.nr; ++k) s[p] += std::fabs(o.M[static_cast<size_t>(p) * o.nr + k]);
    most = std::max(most, s[p]);
  }
  for (double& v : s) v = std::exp2(std::round(std::log2(most / v)));
  return s;
}

void window_tables(const WindowPlan& w, const HostOps& o, const std::vector<double>& scale, std::vector<double>& base,
                   std::vector<double>& slope) {
  const int nr = o.nr, nl = o.nl, NWR = (w.RS + 1) * 32;
  base.assign(static_cast<size_t>(w.np) * 32 * w.NW, 0.0);
  slope.assign(static_cast<size_t>(w.np) * 32 * NWR, 0.0);
  for (int p = 0; p < nr; ++p)
    for (int l = 0; l < nl; ++l) {
      const int t = p / w.g, row = t * 32 + (p % w.g) * w.nlp + l;
      const int c0 = std::max(0, t - w.RC);  // the panel at which the row enters
      double* br = base.data() + static_cast<size_t>(row) * w.NW;
      double* sr = slope.data() + static_cast<size_t>(row) * NWR;
      // splines overlap for |p - k| <= 3 only; the gain couples l = 0 to any k above
      const int hi = l == 0 ? nr - 1 : std::min(nr - 1, p + 3);
      for (int k = std::max(0, p - 3); k <= hi; ++k) {
        const int d = k / w.g - c0, col = d <= w.RS ? d * 32 + (k % w.g) * w.nlp : -1;
        const size_t e = (static_cast<size_t>(l) * nr + p) * nr + k;
        const double m = std::abs(p - k) <= 3 ? o.M[p * nr + k] : 0.0;
        const double v = scale[p] * (m - o.dt * o.Cg[e]), f = -o.dt * scale[p];
        if (col >= 0) br[col + l] = v;
        else br[NWR + k - w.kf0] = v;
        if (k <= p + 3) {
          if (l > 0) sr[col + l - 1] = f * o.Ag_lo[e];
          if (l + 1 < nl) sr[col + l + 1] = f * o.Ag_up[e];
        }
      }
    }
}

std::vector<float> window_blocks(const WindowPlan& w, const std::vector<double>& base, const std::vector<double>& slope) {
  const int nch = w.RS + 1 + w.NF / 32, NWR = (w.RS + 1) * 32;
  std::vector<float> out(static_cast<size_t>(w.np) * nch * 1024);
  for (int t = 0; t < w.np; ++t)
    for (int ch = 0; ch < nch; ++ch)
      for (int r = 0; r < 32; ++r)
        for (int c = 0; c < 32; ++c) {
          const size_t row = static_cast<size_t>(t) * 32 + r;
          const bool ring = ch <= w.RS, mine = !ring || (c & (w.nlp - 1)) == (r & (w.nlp - 1));
          const double v = mine ? base[row * w.NW + ch * 32 + c] : slope[row * NWR + ch * 32 + c];
          out[((static_cast<size_t>(t) * nch + ch) * 32 + r) * 32 + (((c >> 2) ^ (r & 7)) << 2) + (c & 3)] = static_cast<float>(v);
        }
  return out;
}

size_t window_t_count(const WindowPlan& w) { return static_cast<size_t>(w.np) * 32 * w.NS; }
size_t window_u_count(const WindowPlan& w) { return static_cast<size_t>(w.np) * (1024 + 32 * static_cast<size_t>(w.NU)); }
size_t window_slot_count(const WindowPlan& w) { return static_cast<size_t>(w.np) * w.NS; }

static FactorArgs factor_args(const WindowBuffers& b, const double* E, double Eu, unsigned* status) {
  FactorArgs a;
  a.w = b.w, a.base = b.base, a.slope = b.slope, a.E = E, a.Eu = Eu, a.T = b.T, a.U = b.U, a.slotj = b.slotj;
  a.W = b.W, a.rows = b.rows, a.status = status, a.probe = b.probe;
  return a;
}

static SolveArgs solve_args(const WindowBuffers& b, MassBand mass, int nt) {
  SolveArgs a{};
  a.w = b.w, a.T = b.T, a.U = b.U, a.slotj = b.slotj, a.vec = b.vec, a.fmax_ = b.fmax_, a.minv = b.minv, a.rscale = b.rscale, a.mass = mass, a.nt = nt;
  return a;
}

cudaError_t launch_window_factor(const WindowBuffers& b, const double* E, double Eu, int nx, unsigned* status,
                                 cudaStream_t st) {
  const FactorArgs a = factor_args(b, E, Eu, status);
  const int smem = 1024 + 4096 + static_cast<int>(sizeof(float)) * kPW * 2 * (kSlots + b.w.NU);
  const cudaError_t e = set_smem_limit(window_lu_tc_kernel, 1024 + 4096 + sizeof(float) * kPW * 2 * (kSlots + 512));
  if (e != cudaSuccess) return e;
  window_lu_tc_kernel<<<nx, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_window_init_f64(const WindowBuffers& b, const double* E, double Eu, int nx, unsigned* status,
                                   cudaStream_t st) {
  window_f64_init_kernel<<<dim3(kSlots, nx), 128, 0, st>>>(factor_args(b, E, Eu, status));
  return cudaGetLastError();
}

cudaError_t launch_window_panel_f64(const WindowBuffers& b, int s, int nx, unsigned* status, cudaStream_t st) {
  window_f64_panel_kernel<<<nx, kSlots, 0, st>>>(PanelArgs{factor_args(b, nullptr, 0.0, status), s});
  return cudaGetLastError();
}

cudaError_t launch_window_update_f64(const WindowBuffers& b, const double* E, double Eu, int s, int nx, unsigned* status,
                                     cudaStream_t st) {
  const WindowPlan& w = b.w;
  const int dmax = std::min(w.RS, w.np - 1 - s), nfar = std::max(0, w.nr - w.kf0);
  // far columns s g .. s g + g - 1 belong to the entering chunk; the chunk after them has the next live one
  const int fc0 = ((s + 1) * w.g) / 32, nfc = (s + 1) * w.g < nfar ? w.NF / 32 : fc0;
  const int smem = static_cast<int>(sizeof(double)) * (kPW * kSlots + kPW * kPW);
  const int grid = dmax + nfc - fc0 + (s + 1 + w.RS < w.np ? 1 : 0) + 1;
  window_f64_update_kernel<<<dim3(grid, nx), kSlots, smem, st>>>(PanelArgs{factor_args(b, E, Eu, status), s}, dmax, fc0, nfc);
  return cudaGetLastError();
}

cudaError_t launch_window_project(const WindowBuffers& b, const double* in, MassBand mass, const double* TS, int* conv,
                                  int nx, int nt, cudaStream_t st) {
  SolveArgs a = solve_args(b, mass, nt);
  a.in = in, a.TS = TS, a.conv = conv;
  const int smem = static_cast<int>(sizeof(double)) * (2 * ((nt + 1) / 2) + b.w.nl) * b.w.nr;
  // (nt + 1 + nl) nr values, nl <= nt, nr <= 544
  const cudaError_t e = set_smem_limit(window_project_kernel, sizeof(double) * (2 * kMaxNv + 544));
  if (e != cudaSuccess) return e;
  window_project_kernel<<<nx, kEval, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_window_substitute(const WindowBuffers& b, const int* conv, int nx, unsigned* status, cudaStream_t st) {
  SolveArgs a = solve_args(b, MassBand{}, 0);
  a.conv = const_cast<int*>(conv), a.status = status, a.probe = b.probe;
  const WindowRing ring = window_ring(b.w, b.fp64 ? sizeof(double) : sizeof(float), nx, sm_count());
  a.stage_bytes = static_cast<unsigned>(ring.stage_bytes), a.stages = ring.stages;
  const int smem = static_cast<int>(ring.smem);
  auto k = b.fp64 ? window_substitute_kernel<double> : window_substitute_kernel<float>;
  const cudaError_t e = set_smem_limit(k, kRingRoom);
  if (e != cudaSuccess) return e;
  k<<<nx, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_window_residual(const WindowBuffers& b, const double* in, double* out, const double* E, double Eu,
                                   double dt, const ResidualOps& ro, MassBand mass, const double* TO, double ts_inf,
                                   double to_inf, double* ratio, int* conv, double tol, double kc_inf, double ka_inf,
                                   int nx, int nt, bool check, bool last, unsigned* status, cudaStream_t st) {
  SolveArgs a = solve_args(b, mass, nt);
  a.in = in, a.out = out, a.E = E, a.Eu = Eu, a.dt = dt, a.ro = ro, a.TO = TO, a.ts_inf = ts_inf, a.to_inf = to_inf;
  // A point whose bound is above these goes on without the full test. Levelled FP32 factors are near the tolerance one
  // sweep before they are below it: with a point or two of a launch tested in full for nothing there, 100 points of
  // 128 x 3 took 182 us of residuals a step, with what is within 256 of it (down to rounding) going on unasked 131,
  // as with rows as they come. A point that goes on ends at 1e-14, not just below 1e-12.
  const double fl = std::min(kBackwardFloor, tol), part = b.levelled && !b.fp64 ? 1.0 / 256 : 1.0;
  a.skip_tol = std::max(tol * part, fl), a.skip_floor = std::min(fl, std::max(fl * part, kBackwardFloor / 256));
  a.ratio = ratio, a.conv = conv, a.tol = tol, a.kc_inf = kc_inf, a.ka_inf = ka_inf, a.status = status;
  const int smem = static_cast<int>(sizeof(double)) * 3 * b.w.nl * b.w.nr;
  const cudaError_t e = set_smem_limit(window_residual_kernel, sizeof(double) * 3 * kMaxNv);
  if (e != cudaSuccess) return e;
  window_residual_kernel<<<nx, kEval, smem, st>>>(a, check ? 1 : 0, last ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_window_solve_t(const WindowBuffers& b, const double* in, double* out, MassBand mass,
                                  const double* TO, const double* TS, int nx, int nt, cudaStream_t st) {
  SolveArgs a = solve_args(b, mass, nt);
  a.in = in, a.out = out, a.TO = TO, a.TS = TS;
  const int smem = static_cast<int>(sizeof(double)) * ((b.w.np + b.w.RS) * 32 + kSlots + 32);
  // np <= 327 (one speed index a chunk), RS <= 6
  const cudaError_t e = set_smem_limit(window_solve_t_kernel, sizeof(double) * ((327 + 6) * 32 + kSlots + 32));
  if (e != cudaSuccess) return e;
  window_solve_t_kernel<<<nx, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace bte
