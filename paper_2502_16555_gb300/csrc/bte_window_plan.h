// Shapes of the windowed LU (bte_window.cu) and the order of its solves' copies: plain C++ without CUDA.
#pragma once

#include <algorithm>
#include <cstddef>

#ifdef __CUDACC__
#define BTE_HD __host__ __device__
#else
#define BTE_HD
#endif

namespace bte {

// The window for nl harmonics and nr B-splines; ok = false where it does not apply (nl > 32, or a window
// wider than the 512 columns of tensor memory: nr up to 544 with one harmonic, 496 with 2, 472 with 3 and
// 4, 460 with 5 to 8, 394 with 9 to 16, 327 with 17 to 32).
struct WindowPlan {
  int nr = 0, nl = 0;
  int nlp = 0, g = 0;   // power of two >= nl; speed indices per 32-column chunk
  int np = 0;           // chunks (panels)
  int RC = 0, RS = 0;   // chunks that enter ahead of the panel; ring chunks right of it
  int NS = 0;           // row slots in use, 32 (1 + RC)
  int kf0 = 0, NF = 0;  // first speed index kept as a far column; far columns (a multiple of 32)
  int NU = 0, NW = 0;   // window columns RS 32 + NF; row template length (RS + 1) 32 + NF
  int tmem_cols = 0;
  bool ok = false;
};

inline WindowPlan window_plan(int nr, int nl) {
  WindowPlan w;
  w.nr = nr, w.nl = nl;
  if (nl < 1 || nl > 32) return w;
  w.nlp = 1;
  while (w.nlp < nl) w.nlp *= 2;
  w.g = 32 / w.nlp;
  w.np = (nr + w.g - 1) / w.g;
  w.RC = (3 + w.g - 1) / w.g;
  w.RS = 2 * w.RC;
  w.NS = 32 * (1 + w.RC);
  w.kf0 = (w.RS + 1) * w.g;
  w.NF = nr > w.kf0 ? (nr - w.kf0 + 31) / 32 * 32 : 0;
  w.NU = w.RS * 32 + w.NF;
  w.NW = (w.RS + 1) * 32 + w.NF;
  w.tmem_cols = 32;
  while (w.tmem_cols < w.NU) w.tmem_cols *= 2;
  w.ok = w.NU <= 512;
  return w;
}

// The substitution's shared memory: a ring of stages, each one panel's T or U block, and the vectors.
struct WindowRing {
  size_t stage_bytes = 0, fixed = 0;
  int stages = 0;
  size_t smem = 0;
};
constexpr size_t kRingRoom = 224 * 1024;

// ts: bytes of a factor's value. One CTA an SM takes up to 8 stages; with more points than SMs two CTAs
// share one where both can have two stages (256 points of 128 x 32: 315 us instead of 352, now 274). FP64 factors
// of fine speed grids (nr >= 136 with 17 to 32 harmonics) leave room for one stage.
inline WindowRing window_ring(const WindowPlan& w, size_t ts, int nx, int sms) {
  WindowRing r;
  const size_t fb = ts * 32 * w.NS, bb = ts * (1024 + 32 * static_cast<size_t>(w.NU));
  r.stage_bytes = (std::max(fb, bb) + 127) / 128 * 128;
  r.fixed = ts * ((static_cast<size_t>(w.np + w.RS) * 32 + 64) + w.NF);
  size_t room = r.fixed < kRingRoom ? kRingRoom - r.fixed : 0;
  if (nx > sms && r.fixed + 2 * r.stage_bytes <= kRingRoom / 2) room = kRingRoom / 2 - r.fixed;
  r.stages = static_cast<int>(std::min<size_t>(8, room / r.stage_bytes));
  r.smem = r.stages * r.stage_bytes + r.fixed;
  return r;
}

// The substitution uses 2 np copies in order, the T of panels 0 .. np - 1 and the U of panels np - 1 .. 0, copy
// q in stage q mod S. Copies 0 .. S - 1 are issued first; after that copy q + S takes the stage of copy q
// as soon as every thread is past copy q: forwards that is known at the barrier before the wait for copy
// q + 1, backwards (and for the last T) at the barrier that ends panel q. Each function gives the copy to
// issue at its place, -1 for none. With S = 1 a panel's copy is issued where its predecessor is released.
BTE_HD inline int ring_before_wait(int q, int np, int S) {
  return q > 0 && q < np && q - 1 + S < 2 * np ? q - 1 + S : -1;
}
BTE_HD inline int ring_after_use(int q, int np, int S) { return q >= np - 1 && q + S < 2 * np ? q + S : -1; }

}  // namespace bte
