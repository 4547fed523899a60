// Launchers of the fused kernel without per-gap propagators, and the per-call probe kernels
// around it (probe DFT, probe-gradient reduction, slice-gap gradient reduction).
#include <algorithm>
#include <type_traits>

#include "k_path.cuh"

namespace adorym {

// ---------------------------------------------------------------------------- probe DFT
// The probe's spectrum enters every transform that follows, so its stages stay 8 x 16 at N = 128: the
// four-pass radices round differently, and the object and probe gradients of a 32-slice batch moved by
// 6e-6 of their norm.
template <int N>
using ProbeFFT = std::conditional_t<N == 128, SixPass<N>, PathFFT<N>>;

template <int N>
__global__ void __launch_bounds__(Geo<N>::NT) k_probe_hat(const float2* __restrict__ probe, float2* __restrict__ phat,
                                                        const float2* __restrict__ twg) {
  using X = ProbeFFT<N>;
  constexpr int CY = X::CY, YS = X::YS, RX = X::RX, KXS = X::KXS;
  extern __shared__ float2 sm[];
  float2* A = sm;
  float2* tw = A + X::FIELD;
  allow_next();
  X::fill_twiddles(tw, twg);
  after_previous();
  const float2* p = probe + (size_t)blockIdx.x * N * N;
  float2* o = phat + (size_t)blockIdx.x * N * N;
  using V1 = float2[CY];
  using V2 = float2[RX];
  X::template c14<0, -1, false, true>(A, tw, [&](V1&, V1& pb, int x, int t) {
#pragma unroll
    for (int k = 0; k < CY; ++k) pb[k] = __ldg(p + (YS * k + t) * N + x);
  }, [&](V1& v, V1&, V1& pb, int, int) {
#pragma unroll
    for (int k = 0; k < CY; ++k) v[k] = pb[k];
  });
  __syncthreads();
  X::template fwd_pair<-1>(A, tw);
  X::row_sync();
  X::template r23<-1, 0>(A, tw, [&](V2& v, int ky, int t) {
#pragma unroll
    for (int i = 0; i < RX; ++i) o[ky * N + t + KXS * i] = v[i];
  });
}

// ---------------------------------------------------------------------------- probe gradient
// qsum[m][p] = sum_b qacc[b][m][p], fixed order
// Block of 256 threads = 32 consecutive elements x 8 batch chunks; each thread sums its chunk
// Kahan-compensated in FP32 (loads issued four at a time), then the 8 partials of an element are
// added in FP64 in chunk order (deterministic).
__global__ void __launch_bounds__(256) k_qsum(const float2* qacc, float2* __restrict__ qsum, int B,
                                              size_t MNN) {
  allow_next();
  after_previous();
  __shared__ double2 part[8][32];
  const int e = threadIdx.x & 31, c = threadIdx.x >> 5;
  const size_t i = (size_t)blockIdx.x * 32 + e;
  const int b0 = (B * c) / 8, b1 = (B * (c + 1)) / 8;
  Kahan sr, si;
  if (i < MNN) {
#pragma unroll 4
    for (int b = b0; b < b1; ++b) {
      const float2 v = __ldcg(qacc + (size_t)b * MNN + i);
      sr.add(v.x);
      si.add(v.y);
    }
  }
  part[c][e] = make_double2(sr.value(), si.value());
  __syncthreads();
  if (c == 0 && i < MNN) {
    double r = 0.0, im = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      r += part[k][e].x;
      im += part[k][e].y;
    }
    qsum[i] = make_float2((float)r, (float)im);
  }
}

// Running complex sum held as s + e + f: what an addition to s rounds off goes to e, what that addition rounds
// off to f, both exactly (Knuth's TwoSum), so a sum of n terms is off by at most n^3 2^-72 of their sizes (an
// FP64 sum: n 2^-53), whatever their order and signs.  A Kahan sum drops the low part of the running sum
// when the next term is larger, which an element whose terms cancel shows in full (4 to 13 % of the worst
// among 10^6 sums of eight normal terms).
__device__ __forceinline__ void two_sum(float2 a, float2 b, float2& s, float2& e) {   // s + e == a + b
  s = cadd(a, b);
  const float2 bb = csub(s, a);
  e = cadd(csub(a, csub(s, bb)), csub(b, bb));
}
struct Sum3 {
  float2 s, e = {0.f, 0.f}, f = {0.f, 0.f};
  __device__ __forceinline__ explicit Sum3(float2 first) : s(first) {}
  __device__ __forceinline__ void add(float2 x) {
    float2 r, q;
    two_sum(s, x, s, r);
    two_sum(e, r, e, q);
    f = cadd(f, q);
  }
  // the sum rounded once, within 2^-24 of an ulp: e (which exceeds s where s cancels) and f are moved up
  // exactly until each part is below half an ulp of the one above
  __device__ __forceinline__ float2 value() const {
    float2 s1, e1, e2, f2, s2, e3;
    two_sum(s, e, s1, e1);
    two_sum(e1, f, e2, f2);
    two_sum(s1, e2, s2, e3);
    return cadd(s2, cadd(e3, f2));
  }
};

// The same for a batch of at most eight, whose chunks would hold one value or none: a thread per element, the
// batch in its own order, to the accuracy of the FP64 sum over chunks of one value (Sum3).  FP32 adds: a
// call on 8 holograms of 1024 x 1024 at two distances takes 428 us, with the sum on the FP64 pipe 452, with
// a Kahan sum 426.
__global__ void __launch_bounds__(256) k_qsum_few(const float2* qacc, float2* __restrict__ qsum, int B,
                                                  size_t MNN) {
  allow_next();
  after_previous();
  const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= MNN) return;
  Sum3 t(__ldcg(qacc + i));
#pragma unroll 4
  for (int b = 1; b < B; ++b) t.add(__ldcg(qacc + (size_t)b * MNN + i));
  qsum[i] = t.value();
}

// g_gap[j] = sum of gap j's partials over the positions and column CTAs, one CTA per gap, threads strided
// over the partials, then a fixed tree.  (Gaps walked by the threads of one CTA, one after the other over
// the batch, took 40 us for 7 gaps and 100 positions.)
__global__ void __launch_bounds__(128) k_gap_final(const double* gapp, int B, int ngap, int parts,
                                                   float* __restrict__ g) {
  __shared__ double red[4];
  allow_next();
  after_previous();
  const int j = blockIdx.x;
  double s = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x; i < B * parts; i += 128)
    s += __ldcg(gapp + ((size_t)(i / parts) * ngap + j) * parts + i % parts);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) g[j] = (float)(((red[0] + red[1]) + red[2]) + red[3]);
}

// Per-angle position offset of ptychotomography (Sec. 2.3.2): one correction vector shifts every
// position of an angle, so its gradient is the sum of that batch's position gradients.  One warp:
// lane l adds positions l, l + 32, ... in FP64, then a fixed shuffle tree (deterministic).
__global__ void k_offset_sum(const double* gposd, int B, float* __restrict__ g_off) {
  allow_next();
  after_previous();
  double sy = 0.0, sx = 0.0;
  for (int b = threadIdx.x; b < B; b += 32) {
    sy += __ldcg(gposd + 2 * (size_t)b);
    sx += __ldcg(gposd + 2 * (size_t)b + 1);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sy += __shfl_xor_sync(0xffffffffu, sy, o);
    sx += __shfl_xor_sync(0xffffffffu, sx, o);
  }
  if (threadIdx.x == 0) {
    g_off[0] = (float)sy;
    g_off[1] = (float)sx;
  }
}

cudaError_t launch_offset_sum(const double* gposd, int B, float* g_off, Chain& s) {
  return s.launch(k_offset_sum, 1, 32, 0, gposd, B, g_off);
}

cudaError_t launch_gap_final(const double* gapp, int B, int ngap, int parts, float* g_gap, Chain& s) {
  return s.launch(k_gap_final, ngap, 128, 0, gapp, B, ngap, parts, g_gap);
}

cudaError_t launch_qsum(const float2* qacc, float2* qsum, int B, size_t MNN, Chain& s) {
  // up to 8 positions the eight batch chunks of k_qsum hold one value or none (21 us for 2 x 512 x 512)
  if (B <= 8) return s.launch(k_qsum_few, (unsigned)((MNN + 255) / 256), 256, 0, qacc, qsum, B, MNN);
  return s.launch(k_qsum, (unsigned)((MNN + 31) / 32), 256, 0, qacc, qsum, B, MNN);
}

// far field: g_probe[m] += IDFT_-{qsum[m]};  near field: g_probe[m] += qsum[m]
template <int N, int FAR>
__global__ void __launch_bounds__(Geo<N>::NT) k_probe_grad(const float2* qsum, float2* __restrict__ g,
                                                         const float2* __restrict__ twg, const double* lossp,
                                                         int B, double inv_npix, double* __restrict__ loss_out) {
  using X = PathFFT<N>;
  constexpr int CY = X::CY, YS = X::YS, RX = X::RX, KXS = X::KXS, NT = Geo<N>::NT;
  constexpr size_t NN = (size_t)N * N;
  extern __shared__ float2 sm[];
  float2* A = sm;
  float2* tw = A + X::FIELD;
  allow_next();
  if (FAR && g) X::fill_twiddles(tw, twg);
  after_previous();
  if (loss_out && blockIdx.x == 0 && threadIdx.x < 32) {
    // FP64 sum of the per-position partials in a fixed order: lane l adds positions l, l + 32, ...
    // in turn, then a fixed xor tree over the lanes (one warp keeps B / 32 loads in flight instead of
    // one thread walking all B partials)
    double s = 0.0;
    for (int b = (int)threadIdx.x; b < B; b += 32) s += __ldcg(lossp + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) *loss_out = s * inv_npix;
  }
  if (!g) return;
  const float2* q = qsum + blockIdx.x * NN;
  float2* o = g + blockIdx.x * NN;
  if (!FAR) {
    for (size_t i = threadIdx.x; i < NN; i += NT) o[i] = cadd(o[i], __ldcg(q + i));
    return;
  }
  __syncthreads();
  const float invNN = 1.0f / (float)NN;
  using V1 = float2[CY];
  using V2 = float2[RX];
  X::template r23<0, +1>(A, tw, [&](V2& v, int ky, int t) {
#pragma unroll
    for (int i = 0; i < RX; ++i) v[i] = cscale(__ldcg(q + ky * N + t + KXS * i), invNN);
  });
  X::row_sync();
  X::template inv_pair<+1>(A, tw);
  X::template c14<+1, 0, true, false>(A, tw, [&](V1& pa, V1&, int x, int t) {
#pragma unroll
    for (int k = 0; k < CY; ++k) pa[k] = o[(YS * k + t) * N + x];
  }, [&](V1& v, V1& pa, V1&, int x, int t) {
#pragma unroll
    for (int k = 0; k < CY; ++k) o[(YS * k + t) * N + x] = cadd(pa[k], v[k]);
  });
}

// ---------------------------------------------------------------------------- launchers
int path_smem_bytes(int N) {
  switch (N) {
    case 8: return path_smem_bytes_t<8>();
    case 16: return path_smem_bytes_t<16>();
    case 32: return path_smem_bytes_t<32>();
    case 64: return path_smem_bytes_t<64>();
    case 128: return path_smem_bytes_t<128>();
    default: return 0;
  }
}

cudaError_t launch_path(const PathArgs& a, int farfield, Chain& s) {
  if (a.hyj) return launch_path_gaps(a, farfield, s);   // variable slice spacing
  if (a.pipe) return launch_path_pipe(a, farfield, s);
  if (a.helpers) return launch_path_help(a, farfield, s);
  switch (a.N) {
#define ADORYM_CASE(n)                                                                      \
  case n:                                                                                   \
    return farfield ? launch_path_t<n, 1, false>(a, s) : launch_path_t<n, 0, false>(a, s);
    ADORYM_CASE(8)
    ADORYM_CASE(16)
    ADORYM_CASE(32)
    ADORYM_CASE(64)
    ADORYM_CASE(128)
#undef ADORYM_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

template <int N>
constexpr int probe_smem_bytes() {   // field + twiddle tables
  return std::max(PathFFT<N>::FIELD + PathFFT<N>::TW, ProbeFFT<N>::FIELD + ProbeFFT<N>::TW) * (int)sizeof(float2);
}

template <int N>
static cudaError_t launch_probe_hat_t(int M, const float2* probe, float2* phat, const float2* tw, Chain& s) {
  const int smem = probe_smem_bytes<N>();
  return s.launch(k_probe_hat<N>, M, Geo<N>::NT, smem, probe, phat, tw);
}

cudaError_t launch_probe_hat(int N, int M, const float2* probe, float2* phat, const float2* tw, Chain& s) {
  switch (N) {
    case 8: return launch_probe_hat_t<8>(M, probe, phat, tw, s);
    case 16: return launch_probe_hat_t<16>(M, probe, phat, tw, s);
    case 32: return launch_probe_hat_t<32>(M, probe, phat, tw, s);
    case 64: return launch_probe_hat_t<64>(M, probe, phat, tw, s);
    case 128: return launch_probe_hat_t<128>(M, probe, phat, tw, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int N, int FAR>
static cudaError_t launch_probe_grad_t(int M, int B, const float2* qacc, float2* qsum, float2* g, const float2* tw,
                                       const double* lossp, double inv_npix, double* loss_out, Chain& s) {
  const size_t MNN = (size_t)M * N * N;
  if (g) {
    const cudaError_t e = launch_qsum(qacc, qsum, B, MNN, s);
    if (e != cudaSuccess) return e;
  }
  const int smem = probe_smem_bytes<N>();
  return s.launch(k_probe_grad<N, FAR>, M, Geo<N>::NT, smem, qsum, g, tw, lossp, B, inv_npix, loss_out);
}

cudaError_t launch_probe_grad(int N, int M, int B, int farfield, const float2* qacc, float2* qsum, float2* g_probe,
                              const float2* tw, const double* lossp, double inv_npix, double* loss_out,
                              Chain& s) {
  switch (N) {
#define ADORYM_CASE(n)                                                                                     \
  case n:                                                                                                  \
    return farfield ? launch_probe_grad_t<n, 1>(M, B, qacc, qsum, g_probe, tw, lossp, inv_npix, loss_out, s) \
                    : launch_probe_grad_t<n, 0>(M, B, qacc, qsum, g_probe, tw, lossp, inv_npix, loss_out, s);
    ADORYM_CASE(8)
    ADORYM_CASE(16)
    ADORYM_CASE(32)
    ADORYM_CASE(64)
    ADORYM_CASE(128)
#undef ADORYM_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

template <int N, int FAR>
static cudaError_t prepare_t() {
  cudaError_t e = prepare_path_t<N, FAR, false>();
  if (e == cudaSuccess) e = prepare_path_gaps(N, FAR);
  if (e == cudaSuccess) e = prepare_path_pipe(N, FAR);
  if (e == cudaSuccess) e = prepare_path_help(N, FAR);
  const int small = probe_smem_bytes<N>();
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_probe_hat<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, small);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_probe_grad<N, FAR>, cudaFuncAttributeMaxDynamicSharedMemorySize, small);
  return e;
}

cudaError_t prepare_path(int N, int farfield) {
  // idempotent; called by every entry point before it enqueues (never inside a stream capture)
  static std::atomic<bool> done[kMaxDevices][11][2] = {};
  const int dev = current_device();
  int l = 0;
  while ((1 << l) < N) ++l;
  if (dev >= 0 && l < 11 && done[dev][l][farfield ? 1 : 0].load(std::memory_order_acquire)) return cudaSuccess;
  cudaError_t e = cudaErrorInvalidValue;
  switch (N) {
#define ADORYM_CASE(n) \
  case n:              \
    e = farfield ? prepare_t<n, 1>() : prepare_t<n, 0>(); \
    break;
    ADORYM_CASE(8)
    ADORYM_CASE(16)
    ADORYM_CASE(32)
    ADORYM_CASE(64)
    ADORYM_CASE(128)
#undef ADORYM_CASE
    default:
      return cudaErrorInvalidValue;
  }
  if (e == cudaSuccess && dev >= 0 && l < 11) done[dev][l][farfield ? 1 : 0].store(true, std::memory_order_release);
  return e;
}

}  // namespace adorym
