// Block-wide complex64 128 x 128 FFT in four shared-memory passes per propagation step, two of the
// four hand-overs inside a warp; and the pass sequences of the fused kernels per tile size (end of
// this file).
//
// Each 1-D transform uses the two-stage Cooley-Tukey split of fft_block.cuh (stages S1..S4 defined
// there), with different radices per axis so that two of the six passes of a propagation step merge:
//   y: 128 = 16 * 8   (NY1 = 16: S1/S4 radix 16, stride 8;  NY2 = 8:  S2/S3 radix 8, contiguous)
//   x: 128 = 4 * 32   (NX1 = 4:  S1/S4 radix 4, stride 32;  NX2 = 32: S2/S3 radix 32, contiguous)
// With 512 threads per CTA the passes are
//   A  (x, t < 8), two tasks per thread:  y-S4 | spatial op | y-S1    samples y = 8 k + t, k < 16
//   B  (ty < 16, tx < 32):                y-S2, then x-S1             rows 8 ty + iy (iy < 8) x
//                                                                     columns 32 ix + tx (ix < 4)
//   C  (row r, t < 4):                    x-S2 | frequency op | x-S3  32 contiguous columns 32 t + i
//   B3 (ty, tx):                          x-S4, then y-S3             the slots of B
// Pass A, which carries the global traffic of the pointwise ops (transmission, checkpoints,
// object-gradient atomics), keeps 16 values per task; the 32-value passes B, C and B3 touch only
// shared memory, except C's frequency ops at a position's first and last transform.  After B,
// shared row r holds y-frequency r / 8 + 16 (r % 8); in C the x-frequency of element i of task t
// is t + 4 i.
//
// B, C and B3 work on the same eight rows in the same warp: warp w has rows 8 w .. 8 w + 7 (tasks
// ty = w of B and B3; rows 8 w + (lane & 7), t = lane >> 3 of C), so B -> C -> B3 needs only
// __syncwarp and a step has two CTA barriers (around A) instead of four.  Between them the sixteen
// warps run apart, one's shared-memory accesses beside another's arithmetic: with a barrier after
// every pass all of them waited on the same unit at the same time (FMA pipe 44 % busy).  128-position
// multislice loss and gradient 1.306 -> 1.230 ms, 256-position forward 0.796 -> 0.723 ms.
// Shared layout: column c of a row at c + 8 (c / 32), row pitch 153 float2.  The 16 lanes of a
// half-warp access of C (rows g < 8, t and t + 1) then sit at 9 g + 8 t mod 16, one per 8-byte bank
// pair; A and B read 32 consecutive columns of one group, conflict-free at any pitch.  Two tables are not
// conflict-free: C's hy (frequencies w + 16 g of the eight rows, all on one bank pair) and B's tw[2 tx]
// (two to a bank pair).  The whole kernel counts 5.4 M conflicts in 122 M shared-memory wavefronts.
//
// Twiddles W_N^m = exp(-2 pi i m / N) come from the FP64-built table; every stage's twiddle index
// t k stays below N.  C reads its own (t, k) table two entries per 128-bit load.
#pragma once
#include "fft_block.cuh"

namespace adorym {
struct G128 {
  static constexpr int N = 128, NT = 512;
  static constexpr int NY1 = 16, NY2 = 8, NX1 = 4, NX2 = 32;
  static constexpr int GP = NX2 + 8, LD = 153;   // pitch of a 32-column group, of a row
  static constexpr int TWC = NX2 + 2;            // row pitch of C's twiddle table (four rows on distinct banks)
  __device__ static __forceinline__ int col(int c) { return c + 8 * (c / NX2); }
  // y-frequency held by shared row r after pass B
  __device__ static __forceinline__ int row_freq(int r) { return r / NY2 + NY1 * (r % NY2); }
};

// Staggered start after a CTA barrier: each next group of four warps (one per scheduler) begins D
// cycles later.  Released together, all sixteen warps load, compute and store in the same order at the
// same time, and the shared-memory and FMA pipes take turns (each about half busy); apart, one
// group's loads run under another's transforms.  128-position multislice loss and gradient, cycles
// after the barriers of A / B: 0/0 1.219 ms, 200/0 1.212, 0/200 1.201, 200/200 1.179, 300/300 1.172,
// 400/400 1.168, 600/400 1.177, 1000/200 1.206; 256-position forward 0.739 ms at 0/0, 0.679 at 300/300.
template <int D>
__device__ __forceinline__ void stagger() {
  const unsigned n = (threadIdx.x >> 7) * D, t0 = (unsigned)clock();
  while ((unsigned)clock() - t0 < n) {
  }
}

// Pass A: tasks (x, t < NY2), v[k] <-> sample y = NY2 k + t of column x; two tasks per thread, one
// after the other (their pointwise ops keep three 16-value arrays each).
//   pre(pa, pb, x, t): issues a task's global loads (before its shared loads and y-S4).  Issued earlier
//                      (ahead of the barrier, or of the first task's y-S1) they cost more in
//                      registers than they hide: 1.28 and 1.32 against 1.23 ms, multislice batch
//   op(v, pa, pb, x, t): spatial pointwise op on natural samples
//   LOAD = false: the samples come from op (no shared read, no y-S4)
//   S1 != 0: y-S1 and store; S1 == 0: store natural samples; STORE = false: no store
template <int S4, int S1, bool LOAD, bool STORE, class Pre, class Op>
__device__ __forceinline__ void pass4_a(float2* A, const float2* tw, Pre pre, Op op) {
  using G = G128;
  constexpr int N = G::N, LD = G::LD, NY1 = G::NY1, NY2 = G::NY2, Q = (N * NY2) / G::NT;
  static_assert(Q == 2, "two tasks per thread");
  const int x = threadIdx.x % N, xs = G::col(x);
  __syncthreads();
  stagger<320>();
#pragma unroll 1
  for (int q = 0; q < Q; ++q) {
    const int t = threadIdx.x / N + q * (G::NT / N);
    float2 pa[NY1], pb[NY1], v[NY1];
    pre(pa, pb, x, t);
    if (LOAD) {
#pragma unroll
      for (int i = 0; i < NY1; ++i) v[i] = A[(NY2 * i + t) * LD + xs];
      if (S4) dft<NY1, S4>(v);
    }
    op(v, pa, pb, x, t);
    if (STORE) {
      if (S1) {
        dft<NY1, S1>(v);
        twiddle<S1>(v, tw, t);
      }
#pragma unroll
      for (int i = 0; i < NY1; ++i) A[(NY2 * i + t) * LD + xs] = v[i];
    }
  }
}

// Pass B: y-S2 (sign SY) then x-S1 (sign SX, with its twiddles).  Task (ty = warp, tx = lane)
// holds u[iy][ix] = row NY2 ty + iy, column NX2 ix + tx.
template <int SY, int SX>
__device__ __noinline__ void pass4_b(float2* __restrict__ A, const float2* __restrict__ tw) {
  using G = G128;
  constexpr int LD = G::LD, GP = G::GP, NY2 = G::NY2, NX1 = G::NX1, NX2 = G::NX2;
  static_assert((G::N / NY2) * NX2 == G::NT && NX2 == 32, "one task per thread, one group of rows per warp");
  stagger<320>();
  const int tx = threadIdx.x % NX2, ty = threadIdx.x / NX2;
  float2 u[NY2][NX1];
#pragma unroll
  for (int iy = 0; iy < NY2; ++iy)
#pragma unroll
    for (int ix = 0; ix < NX1; ++ix) u[iy][ix] = A[(NY2 * ty + iy) * LD + GP * ix + tx];
#pragma unroll
  for (int ix = 0; ix < NX1; ++ix) {
    float2 c[NY2];
#pragma unroll
    for (int iy = 0; iy < NY2; ++iy) c[iy] = u[iy][ix];
    dft<NY2, SY>(c);
#pragma unroll
    for (int iy = 0; iy < NY2; ++iy) u[iy][ix] = c[iy];
  }
#pragma unroll
  for (int iy = 0; iy < NY2; ++iy) {
    dft<NX1, SX>(u[iy]);
    twiddle<SX>(u[iy], tw, tx);
  }
#pragma unroll
  for (int iy = 0; iy < NY2; ++iy)
#pragma unroll
    for (int ix = 0; ix < NX1; ++ix) A[(NY2 * ty + iy) * LD + GP * ix + tx] = u[iy][ix];
}

// Pass B3: x-S4 (sign SX) then y-S3 (sign SY, with its twiddles), on the slots of pass B.
template <int SX, int SY>
__device__ __noinline__ void pass4_b3(float2* __restrict__ A, const float2* __restrict__ tw) {
  using G = G128;
  constexpr int LD = G::LD, GP = G::GP, NY2 = G::NY2, NX1 = G::NX1, NX2 = G::NX2;
  const int tx = threadIdx.x % NX2, ty = threadIdx.x / NX2;
  float2 u[NY2][NX1];
#pragma unroll
  for (int iy = 0; iy < NY2; ++iy)
#pragma unroll
    for (int ix = 0; ix < NX1; ++ix) u[iy][ix] = A[(NY2 * ty + iy) * LD + GP * ix + tx];
#pragma unroll
  for (int iy = 0; iy < NY2; ++iy) dft<NX1, SX>(u[iy]);
#pragma unroll
  for (int ix = 0; ix < NX1; ++ix) {
    float2 c[NY2];
#pragma unroll
    for (int iy = 0; iy < NY2; ++iy) c[iy] = u[iy][ix];
    dft<NY2, SY>(c);
    twiddle<SY>(c, tw, ty);
#pragma unroll
    for (int iy = 0; iy < NY2; ++iy) u[iy][ix] = c[iy];
  }
#pragma unroll
  for (int iy = 0; iy < NY2; ++iy)
#pragma unroll
    for (int ix = 0; ix < NX1; ++ix) A[(NY2 * ty + iy) * LD + GP * ix + tx] = u[iy][ix];
}

// Pass C: task (row r, t < NX1), one per thread, the rows of a warp those of its B and B3 tasks;
// v[i] = column NX2 t + i.  twc: C's twiddle table.
//   S2 != 0: shared read + x-S2; S2 == 0: the values come from op
//   op(v, ky, t): frequency-domain op, x-frequency of v[i] is t + NX1 i
//   S3 != 0: x-S3 and store in place; S3 == 0: no store
template <int S2, int S3, class Op>
__device__ __forceinline__ void pass4_c(float2* __restrict__ A, const float2* __restrict__ twc, Op op) {
  using G = G128;
  constexpr int LD = G::LD, GP = G::GP, NX2 = G::NX2;
  const int r = (int)(threadIdx.x / 32) * G::NY2 + (int)(threadIdx.x & 7), t = (int)(threadIdx.x & 31) >> 3;
  float2 v[NX2];
  if (S2) {
#pragma unroll
    for (int i = 0; i < NX2; ++i) v[i] = A[r * LD + GP * t + i];
    dft<NX2, S2>(v);
  }
  op(v, G::row_freq(r), t);
  if (S3) {
    dft<NX2, S3>(v);
    twiddle_row<S3, NX2>(v, twc + t * G::TWC);
#pragma unroll
    for (int i = 0; i < NX2; ++i) A[r * LD + GP * t + i] = v[i];
  }
}

}  // namespace adorym

namespace adorym {

// The pass sequence of the fused kernels, per tile size.  Values per spatial-pass task CY at
// y = YS k + t (k < CY); values per frequency-pass task RX at x-frequency t + KXS i (i < RX).
//   c14<S4, S1, LOAD, STORE>(A, tw, pre, op)   CTA barrier | y-S4 | spatial op | y-S1
//   fwd_pair<S>(A, tw)                         y-S2 then x-S1 (with a barrier between them
//                                              where they are separate passes)
//   r23<S2, S3>(A, tw, op)                     x-S2 | frequency op | x-S3
//   inv_pair<S>(A, tw)                         x-S4 then y-S3
//   row_sync()                                 between fwd_pair and r23, and between r23 and inv_pair
// The caller puts a CTA barrier after c14; the one before it is inside (N <= 64: after the pass's
// global loads are issued, so that they fly while the pass before it finishes).  Shared memory: FIELD
// values at A (slot(y, x) for sample or row y, x), then TW twiddles filled by fill_twiddles.
// N <= 32: the six-pass scheme of fft_block.cuh; N = 64: its column passes with the row passes in
// a warp (below); N = 128: the four-pass scheme above.
template <int N>
struct SixPass {
  using F = Field<N>;
  static constexpr int CY = F::N1, YS = F::N2, RX = F::N2, KXS = F::N1;
  static constexpr int FIELD = N * F::LD, TW = N;
  __device__ static __forceinline__ int slot(int y, int x) { return y * F::LD + x; }
  __device__ static __forceinline__ void fill_twiddles(float2* tw, const float2* __restrict__ twg) {
    for (int i = threadIdx.x; i < N; i += F::NT) tw[i] = twg[i];
  }
  __device__ static __forceinline__ void row_sync() { __syncthreads(); }
  template <int S4, int S1, bool LOAD, bool STORE, class Pre, class Op>
  __device__ static __forceinline__ void c14(float2* A, const float2* tw, Pre pre, Op op) {
    pass_c14<N, S4, S1, LOAD, STORE>(A, tw, pre, op);
  }
  template <int S>
  __device__ static __forceinline__ void fwd_pair(float2* A, const float2* tw) {
    pass_c23<N, false, S>(A, tw);
    __syncthreads();
    pass_r14<N, true, S>(A, tw);
  }
  template <int S2, int S3, class Op>
  __device__ static __forceinline__ void r23(float2* A, const float2* tw, Op op) {
    pass_r23<N, S2, S3>(A, tw, op);
  }
  template <int S>
  __device__ static __forceinline__ void inv_pair(float2* A, const float2* tw) {
    pass_r14<N, false, S>(A, tw);
    __syncthreads();
    pass_c23<N, true, S>(A, tw);
  }
};

template <int N>
struct PathFFT : SixPass<N> {};

template <>
struct PathFFT<128> {
  using G = G128;
  static_assert(Geo<128>::NT == G::NT, "the four-pass scheme sets the CTA's thread count");
  static constexpr int CY = G::NY1, YS = G::NY2, RX = G::NX2, KXS = G::NX1;
  static constexpr int FIELD = G::N * G::LD, TW = G::N + G::NX1 * G::TWC;
  static_assert(FIELD % 2 == 0, "C's twiddle table is read in 16-byte pieces");
  __device__ static __forceinline__ int slot(int y, int x) { return y * G::LD + G::col(x); }
  __device__ static __forceinline__ void fill_twiddles(float2* tw, const float2* __restrict__ twg) {
    for (int i = threadIdx.x; i < G::N; i += G::NT) {
      tw[i] = twg[i];
      tw[G::N + (i / G::NX2) * G::TWC + i % G::NX2] = twg[(i / G::NX2) * (i % G::NX2)];
    }
  }
  __device__ static __forceinline__ void row_sync() { __syncwarp(); }
  template <int S4, int S1, bool LOAD, bool STORE, class Pre, class Op>
  __device__ static __forceinline__ void c14(float2* A, const float2* tw, Pre pre, Op op) {
    pass4_a<S4, S1, LOAD, STORE>(A, tw, pre, op);
  }
  template <int S>
  __device__ static __forceinline__ void fwd_pair(float2* A, const float2* tw) {
    pass4_b<S, S>(A, tw);
  }
  template <int S2, int S3, class Op>
  __device__ static __forceinline__ void r23(float2* A, const float2* tw, Op op) {
    pass4_c<S2, S3>(A, tw + G::N, op);
  }
  template <int S>
  __device__ static __forceinline__ void inv_pair(float2* A, const float2* tw) {
    pass4_b3<S, S>(A, tw);
  }
};

// N = 64: the column passes as in the six-pass scheme, the x transforms of a step in one row pass.
// The eight tasks of a row (t < 8) are eight lanes of one warp, so the slot exchange between a
// row's two radix-8 stages (S1 -> S2 forward, S3 -> S4 inverse) goes through a per-warp scratch
// area with warp-level synchronisation instead of a shared-memory pass and a CTA barrier:
//   C14 | C2 | R (x-S1 | exchange | x-S2 | frequency op | x-S3 | exchange | x-S4) | C3
// with the same stages, twiddles and order as the six-pass scheme (the same values).  The spatial
// pass keeps the six-pass thread mapping (consecutive x across a warp: coalesced global accesses).
// C2, R and C3 of the eight rows 8 p .. 8 p + 7 belong to the warps 2 p and 2 p + 1 (64 consecutive
// columns in C2 and C3; rows 4 w + g, lane 8 g + t, in R of warp w), so those two meet at a barrier of
// their own between the passes and a step has two CTA barriers (around C14) instead of four:
// tomography loss and gradient 1.180 -> 1.104 ms.  (A staggered start as at N = 128 costs here, 1.157 ms:
// the passes are too short.)  At a row pitch of 72 the two rows of a half-warp access of R differ by 8
// modulo 16, so its 64-bit accesses cover all 32 banks.
// Exchange: lane (g, a) stores its value k at scratch[72 g + a + 9 k]; lane (g, b) reads its
// value i from scratch[72 g + i + 9 b] (both conflict-free).

// per-warp exchange scratch of the row pass: one array per CTA
__device__ __forceinline__ float2* row64_scratch() {
  __shared__ float2 scratch[(Geo<64>::NT / 32) * 288];
  return scratch;
}

template <int S>
__device__ __forceinline__ void row64_line(float2 (&v)[8], const float2 (&wt)[8], float2* ws, int g, int a) {
  dft<8, S>(v);
#pragma unroll
  for (int k = 1; k < 8; ++k) v[k] = S < 0 ? cmul(v[k], wt[k]) : cmulc(v[k], wt[k]);   // twiddle<S>
  __syncwarp();   // the previous exchange of this warp has read its slots
#pragma unroll
  for (int k = 0; k < 8; ++k) ws[72 * g + a + 9 * k] = v[k];
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = ws[72 * g + i + 9 * a];
  dft<8, S>(v);
}

template <>
struct PathFFT<64> {
  using F = Field<64>;
  static_assert(F::N1 == 8 && F::N2 == 8 && F::NT == 512, "row pass layout");
  static constexpr int CY = F::N1, YS = F::N2, RX = F::N2, KXS = F::N1;
  static constexpr int FIELD = 64 * F::LD, TW = 64;
  __device__ static __forceinline__ int slot(int y, int x) { return y * F::LD + x; }
  __device__ static __forceinline__ void fill_twiddles(float2* tw, const float2* __restrict__ twg) {
    for (int i = threadIdx.x; i < 64; i += F::NT) tw[i] = twg[i];
  }
  // the two warps that share eight rows
  __device__ static __forceinline__ void row_sync() {
    asm volatile("bar.sync %0, 64;" ::"r"(1 + (int)(threadIdx.x >> 6)) : "memory");
  }
  template <int S4, int S1, bool LOAD, bool STORE, class Pre, class Op>
  __device__ static __forceinline__ void c14(float2* A, const float2* tw, Pre pre, Op op) {
    pass_c14<64, S4, S1, LOAD, STORE>(A, tw, pre, op);
  }
  template <int S>
  __device__ static __forceinline__ void fwd_pair(float2* A, const float2* tw) {
    pass_c23<64, false, S>(A, tw);
  }
  // row r (y-frequency row_freq(r)): S2 != 0 reads samples x = 8 i + t and runs x-S1, x-S2; op
  // sees x-frequencies t + 8 i; S3 != 0 runs x-S3, x-S4 and stores samples in place
  template <int S2, int S3, class Op>
  __device__ static __forceinline__ void r23(float2* A, const float2* tw, Op op) {
    constexpr int LD = F::LD;
    const int lane = (int)(threadIdx.x & 31), w = (int)(threadIdx.x >> 5), g = lane >> 3, t = lane & 7;
    const int r = 4 * w + g;
    float2* ws = row64_scratch() + w * 288;
    float2 v[8], wt[8];
#pragma unroll
    for (int k = 1; k < 8; ++k) wt[k] = tw[t * k];
    if (S2) {
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = A[r * LD + 8 * i + t];
      row64_line<S2>(v, wt, ws, g, t);
    }
    op(v, F::row_freq(r), t);
    if (S3) {
      row64_line<S3>(v, wt, ws, g, t);
#pragma unroll
      for (int k = 0; k < 8; ++k) A[r * LD + 8 * k + t] = v[k];
    }
  }
  template <int S>
  __device__ static __forceinline__ void inv_pair(float2* A, const float2* tw) {
    pass_c23<64, true, S>(A, tw);
  }
};

}  // namespace adorym
