// Regularizers of Table regularizers in the refractive-index form, added to the data term as in
// Eq. tikhonov:
//   R = (1/N_o) [ sum a_d W_d |delta| + a_b W_b |beta| + gamma sum_axes (|grad delta| + |grad beta|) ]
// with forward differences (no term past the last index), subgradient 0 at 0, and optional
// reweighting W = max|C| / (|C| + eps) from a snapshot.  Dense volume work, HBM-bound: one pass
// reads delta, beta (and W), each voxel gathers its own TV subgradient from its neighbours (no
// atomics), per-CTA FP64 partial sums are added in a fixed order.
#include <algorithm>
#include <cstdint>
#include <type_traits>
#include <utility>

#include "numerics.cuh"
#include "kernels.cuh"

namespace adorym {

__device__ __forceinline__ float sgn(float v) { return (v > 0.f) - (v < 0.f); }

// V consecutive floats of a row (V = 4: one 128-bit access, p 16-byte aligned)
template <int V>
__device__ __forceinline__ void load_v(float (&o)[V], const float* __restrict__ p) {
  if constexpr (V == 4) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
  } else {
    o[0] = *p;
  }
}
template <int V>
__device__ __forceinline__ void store_v(float* __restrict__ p, const float (&o)[V]) {
  if constexpr (V == 4) *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
  else *p = o[0];
}

// Value and gradient, any alignment and row length.  z (stride sz) is the axis that is walked and y (stride sy) the
// other one, whichever the volume calls them.  A CTA's eight warps are RY rows times 8 / RY stretches of zc planes: a
// warp walks zc planes of 32 columns of a row.  The planes z - 1, z, z + 1 of delta and beta stay in registers, the x
// neighbours come from the lanes beside (the tile's ends from one load), the y neighbours from L1 where
// the tile holds them.  One CTA per row with every neighbour read took 98 us for 32 x 512 x 509 and 52
// for 33 x 300 x 301, this 88 and 38; eight rows for every volume took 35 us for 2000 x 1 x 301 (of which one
// row is there), one CTA per row 16.6, this 16.4.  Item indices in 32 bits: in 64 their divisions were 6 %
// (297 -> 284 us for 31 x 1025 x 1023).
template <bool TV, int RY>
__global__ void __launch_bounds__(256) k_regularize(const float* __restrict__ d, const float* __restrict__ b,
                                                    const float* __restrict__ wd, const float* __restrict__ wb,
                                                    int Lz, int Ly, int Lx, size_t sz, size_t sy, float ad, float ab,
                                                    float gam, float invNo, float* __restrict__ gd,
                                                    float* __restrict__ gb, double* __restrict__ part, int zc) {
  __shared__ double red[8];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, ty = (threadIdx.x >> 5) % RY, tz = (threadIdx.x >> 5) / RY;
  const int pz = 8 / RY * zc;   // planes of a tile
  const unsigned gx = (Lx + 31) / 32, gy = (Ly + RY - 1) / RY, gz = (Lz + pz - 1) / pz;
  const unsigned items = gx * gy * gz;   // (below 2^30 for any volume that fits the card: 128 voxels and more each)
  Kahan acc;
  for (unsigned item = blockIdx.x; item < items; item += gridDim.x) {
    const unsigned row = item / gx;
    const int ix = (int)(item - row * gx), iz = (int)(row / gy), iy = (int)(row - (unsigned)iz * gy);
    const int x = ix * 32 + lane, y = iy * RY + ty, z0 = iz * pz + tz * zc, z1 = min(z0 + zc, Lz);
    const bool in = x < Lx && y < Ly && z0 < Lz;
    size_t i = in ? z0 * sz + y * sy + x : 0;
    float cd = 0.f, cb = 0.f, pd = 0.f, pb = 0.f, nd = 0.f, nb = 0.f;   // this plane, the one before, the next
    if (in) {
      cd = d[i];
      cb = b[i];
      if (TV && z0 > 0) {
        pd = d[i - sz];
        pb = b[i - sz];
      }
    }
    for (int z = z0; z < z1; ++z, i += sz) {
      float w1 = 1.f, w2 = 1.f, od = 0.f, ob = 0.f, ud = 0.f, ub = 0.f, vd = 0.f, vb = 0.f;
      float ld = 0.f, lb = 0.f, rd = 0.f, rb = 0.f;   // x neighbours
      if (in) {
        if (z + 1 < (TV ? Lz : z1)) {
          nd = d[i + sz];
          nb = b[i + sz];
        }
        if (TV) {
          if (y + 1 < Ly) {
            ud = d[i + sy];
            ub = b[i + sy];
          }
          if (y > 0) {
            vd = d[i - sy];
            vb = b[i - sy];
          }
          if (lane == 0 && x > 0) {
            ld = d[i - 1];
            lb = b[i - 1];
          }
          if (lane == 31 && x + 1 < Lx) {
            rd = d[i + 1];
            rb = b[i + 1];
          }
        }
        if (wd) w1 = wd[i];
        if (wb) w2 = wb[i];
        if (gd) {
          od = gd[i];
          ob = gb[i];
        }
      }
      if (TV) {
        const float a = __shfl_up_sync(full, cd, 1), c = __shfl_up_sync(full, cb, 1);
        const float f = __shfl_down_sync(full, cd, 1), g = __shfl_down_sync(full, cb, 1);
        if (lane > 0) {
          ld = a;
          lb = c;
        }
        if (lane < 31) {
          rd = f;
          rb = g;
        }
      }
      if (in) {
        float term = ad * w1 * fabsf(cd) + ab * w2 * fabsf(cb);
        float g1 = ad * w1 * sgn(cd), g2 = ab * w2 * sgn(cb);
        if (TV) {
          auto ahead = [&](float hd, float hb) {   // forward difference of this voxel
            const float fd = hd - cd, fb = hb - cb;
            term += gam * (fabsf(fd) + fabsf(fb));
            g1 -= gam * sgn(fd);
            g2 -= gam * sgn(fb);
          };
          auto behind = [&](float hd, float hb) {   // forward difference of the voxel before
            g1 += gam * sgn(cd - hd);
            g2 += gam * sgn(cb - hb);
          };
          if (x + 1 < Lx) ahead(rd, rb);
          if (x > 0) behind(ld, lb);
          if (y + 1 < Ly) ahead(ud, ub);
          if (y > 0) behind(vd, vb);
          if (z + 1 < Lz) ahead(nd, nb);
          if (z > 0) behind(pd, pb);
        }
        acc.add(term);
        od += g1 * invNo;
        ob += g2 * invNo;
        if (gd) {
          gd[i] = od;
          gb[i] = ob;
        }
      }
      pd = cd;
      pb = cb;
      cd = nd;
      cb = nb;
    }
  }
  double v = acc.value();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < 8; ++k) s += red[k];
    part[blockIdx.x] = s;
  }
}

// The same with four consecutive voxels of a row per thread, over the flat volume (Lx % 4 == 0 and
// 16-byte aligned arrays): 128-bit loads of delta, beta, the weights, the neighbour rows and
// planes and the gradients, the x neighbours across the group from two scalar loads.  Same
// per-voxel arithmetic and order as k_regularize, whose tiles with four voxels a thread were slower
// (73.7 against 71.5 us for 32 x 512 x 512, 43.0 against 36.8 for 8 x 700 x 700).
template <bool TV>
__global__ void __launch_bounds__(256) k_regularize4(const float* __restrict__ d, const float* __restrict__ b,
                                                     const float* __restrict__ wd, const float* __restrict__ wb,
                                                     int Lz, int Ly, int Lx, float ad, float ab, float gam,
                                                     float invNo, float* __restrict__ gd, float* __restrict__ gb,
                                                     double* __restrict__ part) {
  __shared__ double red[8];
  const int Lx4 = Lx >> 2;
  const size_t sy = Lx, sz = (size_t)Lx * Ly;
  const size_t n4 = (size_t)Ly * Lz * Lx4;
  const float4 one4 = make_float4(1.f, 1.f, 1.f, 1.f);
  Kahan acc;
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < n4; q += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(q / Lx4), x0 = 4 * (int)(q - (size_t)r * Lx4);
    const int z = r / Ly, y = r - z * Ly;
    const size_t i = (size_t)r * Lx + x0;
    const float4 vd = *reinterpret_cast<const float4*>(d + i), vb = *reinterpret_cast<const float4*>(b + i);
    const float4 w1 = wd ? *reinterpret_cast<const float4*>(wd + i) : one4;
    const float4 w2 = wb ? *reinterpret_cast<const float4*>(wb + i) : one4;
    const float cd[4] = {vd.x, vd.y, vd.z, vd.w}, cb[4] = {vb.x, vb.y, vb.z, vb.w};
    const float cw1[4] = {w1.x, w1.y, w1.z, w1.w}, cw2[4] = {w2.x, w2.y, w2.z, w2.w};
    float term[4], g1[4], g2[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      term[e] = ad * cw1[e] * fabsf(cd[e]) + ab * cw2[e] * fabsf(cb[e]);
      g1[e] = ad * cw1[e] * sgn(cd[e]);
      g2[e] = ab * cw2[e] * sgn(cb[e]);
    }
    if (TV) {
      // x neighbours: within the group, and one scalar on each side
      float nd[6], nb[6];   // nd[e + 1] = delta at x0 + e, e = -1..4
      nd[0] = x0 > 0 ? d[i - 1] : 0.f;
      nb[0] = x0 > 0 ? b[i - 1] : 0.f;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        nd[e + 1] = cd[e];
        nb[e + 1] = cb[e];
      }
      nd[5] = x0 + 4 < Lx ? d[i + 4] : 0.f;
      nb[5] = x0 + 4 < Lx ? b[i + 4] : 0.f;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int x = x0 + e;
        if (x + 1 < Lx) {
          const float fd = nd[e + 2] - cd[e], fb = nb[e + 2] - cb[e];
          term[e] += gam * (fabsf(fd) + fabsf(fb));
          g1[e] -= gam * sgn(fd);
          g2[e] -= gam * sgn(fb);
        }
        if (x > 0) {
          g1[e] += gam * sgn(cd[e] - nd[e]);
          g2[e] += gam * sgn(cb[e] - nb[e]);
        }
      }
      // y and z neighbours: whole groups of the adjacent rows and planes
      const int pos[2] = {y, z}, lim[2] = {Ly, Lz};
      const size_t st[2] = {sy, sz};
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        if (pos[a] + 1 < lim[a]) {
          const float4 ud = *reinterpret_cast<const float4*>(d + i + st[a]);
          const float4 ub = *reinterpret_cast<const float4*>(b + i + st[a]);
          const float qd[4] = {ud.x, ud.y, ud.z, ud.w}, qb[4] = {ub.x, ub.y, ub.z, ub.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float fd = qd[e] - cd[e], fb = qb[e] - cb[e];
            term[e] += gam * (fabsf(fd) + fabsf(fb));
            g1[e] -= gam * sgn(fd);
            g2[e] -= gam * sgn(fb);
          }
        }
        if (pos[a] > 0) {
          const float4 ud = *reinterpret_cast<const float4*>(d + i - st[a]);
          const float4 ub = *reinterpret_cast<const float4*>(b + i - st[a]);
          const float qd[4] = {ud.x, ud.y, ud.z, ud.w}, qb[4] = {ub.x, ub.y, ub.z, ub.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            g1[e] += gam * sgn(cd[e] - qd[e]);
            g2[e] += gam * sgn(cb[e] - qb[e]);
          }
        }
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) acc.add(term[e]);
    if (gd) {
      float4 od = *reinterpret_cast<float4*>(gd + i), ob = *reinterpret_cast<float4*>(gb + i);
      od.x += g1[0] * invNo; od.y += g1[1] * invNo; od.z += g1[2] * invNo; od.w += g1[3] * invNo;
      ob.x += g2[0] * invNo; ob.y += g2[1] * invNo; ob.z += g2[2] * invNo; ob.w += g2[3] * invNo;
      *reinterpret_cast<float4*>(gd + i) = od;
      *reinterpret_cast<float4*>(gb + i) = ob;
    }
  }
  double v = acc.value();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < 8; ++k) s += red[k];
    part[blockIdx.x] = s;
  }
}

// R = invNo * sum of the per-CTA partials: 256 threads, each adds a strided subset in order, then
// a fixed shuffle tree and a fixed order over the warps (deterministic)
__global__ void __launch_bounds__(256) k_reg_final(const double* __restrict__ part, int nparts, double invNo,
                                                   double* __restrict__ out) {
  __shared__ double red[8];
  double v = 0.0;
  for (int k = threadIdx.x; k < nparts; k += blockDim.x) v += part[k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += red[k];
    *out = s * invNo;
  }
}

// max |C| of delta (blockIdx.y = 0) and beta (1): per-CTA maxima (NaNs are passed over, as by fmaxf)
template <int V>
__global__ void __launch_bounds__(256) k_absmax(const float* __restrict__ cd, const float* __restrict__ cb, size_t n,
                                                float* __restrict__ part) {
  __shared__ float red[8];
  const float* __restrict__ c = blockIdx.y ? cb : cd;
  constexpr int U = 4;   // loads in flight per thread
  const size_t nv = n / V, step = (size_t)gridDim.x * blockDim.x;
  float m = 0.f;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += U * step) {
    float v[U][V];
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int e = 0; e < V; ++e) v[u][e] = 0.f;
      if (i + u * step < nv) load_v<V>(v[u], c + (i + u * step) * V);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int e = 0; e < V; ++e) m = fmaxf(m, fabsf(v[u][e]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) m = fmaxf(m, red[k]);
    part[blockIdx.y * gridDim.x + blockIdx.x] = m;
  }
}

// W = max|C| / (|C| + eps) of both volumes.  Every CTA takes the maximum of the nparts partials with
// all of its threads: walked by one thread it was 30 of the 37 us of a 512 x 512 x 32 volume.
template <int V>
__global__ void __launch_bounds__(256) k_l1_weights(const float* __restrict__ cd, const float* __restrict__ cb, size_t n,
                                                    const float* __restrict__ part, int nparts, float eps,
                                                    float* __restrict__ wd, float* __restrict__ wb) {
  __shared__ float red[8];
  const float* __restrict__ c = blockIdx.y ? cb : cd;
  float* __restrict__ w = blockIdx.y ? wb : wd;
  float m = 0.f;
  for (int k = threadIdx.x; k < nparts; k += 256) m = fmaxf(m, part[blockIdx.y * nparts + k]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  float mx = red[0];
#pragma unroll
  for (int k = 1; k < 8; ++k) mx = fmaxf(mx, red[k]);
  constexpr int U = 4;
  const size_t nv = n / V, step = (size_t)gridDim.x * blockDim.x;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += U * step) {
    float v[U][V];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i + u * step < nv) load_v<V>(v[u], c + (i + u * step) * V);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (i + u * step >= nv) break;
#pragma unroll
      for (int e = 0; e < V; ++e) v[u][e] = mx / (fabsf(v[u][e]) + eps);
      store_v<V>(w + (i + u * step) * V, v[u]);
    }
  }
}

static unsigned reg_grid(size_t n) { return (unsigned)std::min<size_t>((n + 255) / 256, 152 * 8); }

int reg_parts(size_t n) { return (int)reg_grid(n); }

static bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

cudaError_t launch_regularize(const float* d, const float* b, const float* wd, const float* wb, int Lz, int Ly, int Lx,
                              double ad, double ab, double gam, float* gd, float* gb, double* part, double* loss,
                              cudaStream_t s) {
  const size_t n = (size_t)Lz * Ly * Lx;
  const float invNo = (float)(1.0 / (double)n);
  const bool vec = Lx % 4 == 0 && aligned16(d) && aligned16(b) && aligned16(wd) && aligned16(wb) && aligned16(gd) && aligned16(gb);
  auto final_sum = [&](unsigned grid) {
    if (loss) (k_reg_final<<<1, 256, 0, s>>>(part, (int)grid, 1.0 / (double)n, loss), note_launch());
    return cudaGetLastError();
  };
  if (vec) {
    const unsigned grid = reg_grid(n);
    if (gam != 0.0)
      (k_regularize4<true><<<grid, 256, 0, s>>>(d, b, wd, wb, Lz, Ly, Lx, (float)ad, (float)ab, (float)gam, invNo, gd,
                                                gb, part), note_launch());
    else
      (k_regularize4<false><<<grid, 256, 0, s>>>(d, b, wd, wb, Lz, Ly, Lx, (float)ad, (float)ab, 0.f, invNo, gd, gb,
                                                 part), note_launch());
    return final_sum(grid);
  }
  // One plane is walked along y (1 x 3000 x 3001: 120 us as a walk of one plane, 90 so; one CTA per row 98).
  int Lw = Lz, Lr = Ly;
  size_t sw = (size_t)Lx * Ly, sr = Lx;
  if (Lz == 1) {
    std::swap(Lw, Lr);
    std::swap(sw, sr);
  }
  // Rows per tile: a divisor of a small row count, so that no warp is without a row (4096 x 2 x 255: 59 -> 29 us,
  // 100 x 5 x 1001 17.4 -> 16.7).
  int ry = 8;
  while (Lr < 8 && Lr % ry) ry /= 2;
  // planes per walk: as many as leave the chip eight CTAs per SM (fewer planes re-read more of their neighbours)
  const long long tiles = (long long)((Lx + 31) / 32) * ((Lr + ry - 1) / ry);
  auto items = [&](int zc) { return tiles * ((Lw + 8 / ry * zc - 1) / (8 / ry * zc)); };
  int zc = 16;
  while (zc > 2 && items(zc) < 152 * 8) zc /= 2;
  const unsigned grid = (unsigned)std::min<long long>(items(zc), reg_grid(n));
  auto run = [&](auto kernel, float g) {
    (kernel<<<grid, 256, 0, s>>>(d, b, wd, wb, Lw, Lr, Lx, sw, sr, (float)ad, (float)ab, g, invNo, gd, gb, part, zc), note_launch());
  };
  auto rows = [&](auto r) {
    gam != 0.0 ? run(k_regularize<true, decltype(r)::value>, (float)gam) : run(k_regularize<false, decltype(r)::value>, 0.f);
  };
  switch (ry) {
    case 8: rows(std::integral_constant<int, 8>()); break;
    case 4: rows(std::integral_constant<int, 4>()); break;
    case 2: rows(std::integral_constant<int, 2>()); break;
    default: rows(std::integral_constant<int, 1>());
  }
  return final_sum(grid);
}

cudaError_t launch_l1_weights(const float* d, const float* b, size_t n, float eps, float* part, float* wd, float* wb,
                              cudaStream_t s) {
  const bool vec = n % 4 == 0 && aligned16(d) && aligned16(b) && aligned16(wd) && aligned16(wb);
  const unsigned grid = std::min(reg_grid(n), 152u * 4);   // per volume
  auto run = [&](unsigned volumes, const float* c0, float* w0) {
    const dim3 g(grid, volumes);
    if (vec) {
      (k_absmax<4><<<g, 256, 0, s>>>(c0, b, n, part), note_launch());
      (k_l1_weights<4><<<g, 256, 0, s>>>(c0, b, n, part, (int)grid, eps, w0, wb), note_launch());
    } else {
      (k_absmax<1><<<g, 256, 0, s>>>(c0, b, n, part), note_launch());
      (k_l1_weights<1><<<g, 256, 0, s>>>(c0, b, n, part, (int)grid, eps, w0, wb), note_launch());
    }
  };
  auto overlap = [n](const float* p, const float* q) { return p < q + n && q < p + n; };
  if (overlap(wd, wb) || overlap(wd, b) || overlap(wb, d)) {   // one volume after the other (one buffer for both, say)
    run(1, d, wd);
    run(1, b, wb);
  } else {
    run(2, d, wd);
  }
  return cudaGetLastError();
}

}  // namespace adorym
