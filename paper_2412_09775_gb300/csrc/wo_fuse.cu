// wo_fuse.cu - multi-channel fusion: one property from C data channels, each
// seen through its own transfer function (9-aperture fusion, Results; C x 1
// multi-channel Tikhonov, Eq. recon with a C-element column H):
//   F(nu) = sum_c conj(H_c) D~_c / (sum_c |H_c|^2 + eta)
// per 3D frequency, or per transverse frequency with the sums also over the
// axial bins (the 2D phase-from-defocus model; Parseval over z).
//
// The z pass streams the channels: for each channel it loads its z columns,
// transforms them along z and adds conj(H_c) D_c and |H_c|^2 into two
// accumulators; after the last channel it forms F, transforms it back (3D) or
// reduces it over k (2D), and stores one output volume.  The columns and the
// accumulators sit in registers where the plane count divides among a few
// lanes (k_z_fuse_reg), else in shared memory (k_z_fuse).
#include "wo_fft.cuh"
#include "wo_internal.h"
#include "wo_regfft.cuh"
#include "wo_zops.cuh"

namespace wo {

namespace {

template <int N>
struct FuseGeom {
  using G = ZGeom<N, 3>;  // data tile, numerator, denominator
  static constexpr int B = G::B, NT = G::NT, MINB = G::MINB;
  static constexpr size_t SMEM = G::SMEM + (size_t)NT * 3 * sizeof(float);
};

// Per tile: max over 3D frequencies of sum_c |H_c|^2 and max over transverse
// frequencies of sum_k sum_c |H_c|^2 (the relative regulariser's scales in
// 3D and 2D).  Bound by the loads' latency: a lane takes one (y, x) column of
// 32, G warps share the 32 columns (warp g the planes g, g + G, ...), and a
// thread has 16 loads in flight: up to CM channels of 16 / CM planes.  (One thread a
// column left the chip waiting on its 288 loads in turn: 4 tiles x 9 channels
// of 32x128x128 66 us, now 21.)  A CTA takes column groups in turn and ends
// in one atomic per statistic: one per warp and 32 columns, all on a few
// words, bound banks of few channels and planes (one channel, 61 tiles of
// 8x128x128: 93 us, now 14; 512 of 16x64x64: 212, now 32).
constexpr int kStatsLoads = 16;
static_assert(kStatsLoads >= kMaxFuseChannels, "a plane's channels in one batch of loads");

template <int CM>
__global__ void __launch_bounds__(256) k_fuse_stats(const float2* __restrict__ tf, int C, int Z, int Y, int Xh, int G,
                                                    float* __restrict__ stats) {
  constexpr int U = kStatsLoads / CM;
  __shared__ float part[8][32], red[2][8];
  const int t = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x / 32;
  const int g = warp % G;
  const long long plane = (long long)Y * Xh;
  const float2* tile = tf + (long long)t * C * Z * plane;
  float m3 = 0.f, m2 = 0.f;
  for (long long c0 = (long long)blockIdx.x * (256 / G); c0 < plane; c0 += (long long)gridDim.x * (256 / G)) {
    const long long col = c0 + warp / G * 32 + lane;
    float s2 = 0.f;
    if (col < plane) {
      const float2* h = tile + col;
      for (int k0 = g; k0 < Z; k0 += U * G) {
        float2 v[U][CM];
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
          for (int c = 0; c < CM; ++c)
            v[u][c] = (k0 + u * G < Z && c < C) ? __ldg(h + ((long long)c * Z + k0 + u * G) * plane)
                                                : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          float s = 0.f;
#pragma unroll
          for (int c = 0; c < CM; ++c) s += cabs2(v[u][c]);
          m3 = fmaxf(m3, s);
          s2 += s;
        }
      }
    }
    if (G > 1) {  // the column's sum over its warps
      part[warp][lane] = s2;
      __syncthreads();
      s2 = 0.f;
      if (g == 0) {
        for (int q = 0; q < G; ++q) s2 += part[warp + q][lane];
      }
      __syncthreads();
    }
    m2 = fmaxf(m2, s2);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    m3 = fmaxf(m3, __shfl_xor_sync(0xffffffffu, m3, off));
    m2 = fmaxf(m2, __shfl_xor_sync(0xffffffffu, m2, off));
  }
  if (lane == 0) {
    red[0][warp] = m3;
    red[1][warp] = m2;
  }
  __syncthreads();
  if (threadIdx.x < 2) {  // values are >= 0: integer order equals float order
    float m = 0.f;
    for (int q = 0; q < 8; ++q) m = fmaxf(m, red[threadIdx.x][q]);
    if (m > 0.f) atomicMax(reinterpret_cast<int*>(stats) + 2 * t + threadIdx.x, __float_as_int(m));
  }
}

template <int N>
__global__ void __launch_bounds__(FuseGeom<N>::NT, FuseGeom<N>::MINB)
    k_z_fuse(const float2* __restrict__ in, float2* __restrict__ out, const float2* __restrict__ tf, FuseOp op,
             int Y, int Xh) {
  using G = FuseGeom<N>;
  constexpr int B = G::B, NT = G::NT;
  extern __shared__ float2 sm[];
  float2* tw = sm;
  float2* dbuf = sm + N;
  float2* num = dbuf + N * B;
  float* den = reinterpret_cast<float*>(num + N * B);
  float* red = den + 2 * N * B;  // [NT][3] (2D reduction)
  const int t = blockIdx.z, y = blockIdx.y, x0 = blockIdx.x * B;
  const int w = min(B, Xh - x0);
  const long long zs = (long long)Y * Xh;
  const long long vol = (long long)N * zs;
  const long long col = (long long)y * Xh + x0;
  const int C = op.C;
  make_twiddles<N>(tw);
  for (int e = threadIdx.x; e < N * B; e += NT) {
    num[e] = make_float2(0.f, 0.f);
    den[e] = 0.f;
  }
  for (int c = 0; c < C; ++c) {
    load_zcols<N, 1, B, NT>(dbuf, in + ((long long)t * C + c) * vol + col, 1, vol, zs, w);
    cp_async_wait_all();
    __syncthreads();
    fft_smem<N, B, NT, false, 1>(dbuf, B, 1, tw);
    const float2* h = tf + ((long long)t * C + c) * vol + col;
    for (int e = threadIdx.x; e < N * B; e += NT) {
      const int k = e / B, b = e % B;
      if (b >= w) continue;
      float2 d = dbuf[e];
      if (k == 0 && y == 0 && x0 + b == 0) d = op.zero_dc ? make_float2(0.f, 0.f) : make_float2(d.x - op.bg_dc[c], d.y);
      const float2 hv = __ldg(h + (long long)k * zs + b);
      num[e] = cadd(num[e], cmulc(hv, d));
      den[e] += cabs2(hv);
    }
    __syncthreads();  // dbuf is reloaded for the next channel
  }
  const float* st = op.stats + 2LL * t;
  if (op.mode == WO_MODE_3D) {
    const float lam = op.eta_relative ? op.eta * st[0] : op.eta;
    for (int e = threadIdx.x; e < N * B; e += NT) {
      const float q = den[e] + lam;
      dbuf[e] = q > 0.f ? cscale(num[e], 1.0f / q) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    fft_smem<N, B, NT, true, 1>(dbuf, B, 1, tw);
    store_zcols<N, 1, B, NT>(dbuf, out + (long long)t * vol + col, 1, vol, zs, w);
    return;
  }
  // 2D: sum over k of both accumulators, per column b (fixed per thread)
  const int b = threadIdx.x % B;
  float sr = 0.f, si = 0.f, sd = 0.f;
  for (int e = threadIdx.x; e < N * B; e += NT) {
    sr += num[e].x;
    si += num[e].y;
    sd += den[e];
  }
  red[3 * threadIdx.x] = sr;
  red[3 * threadIdx.x + 1] = si;
  red[3 * threadIdx.x + 2] = sd;
  __syncthreads();
  if (threadIdx.x < B && b < w) {
    float2 a = make_float2(0.f, 0.f);
    float dd = 0.f;
    for (int q = threadIdx.x; q < NT; q += B) {
      a = cadd(a, make_float2(red[3 * q], red[3 * q + 1]));
      dd += red[3 * q + 2];
    }
    // per-plane sums are 1/Z of the sums over k, so eta enters as Z eta
    const float lam = op.eta_relative ? op.eta * st[1] : op.eta * (float)N;
    const float q = dd + lam;
    out[(long long)t * zs + col + b] = q > 0.f ? cscale(a, 1.0f / q) : make_float2(0.f, 0.f);
  }
}

template <int N>
cudaError_t launch_z_fuse(const float2* in, float2* out, const float2* tf, const FuseOp& op, int n_tiles, int Y,
                          int Xh, cudaStream_t s) {
  using G = FuseGeom<N>;
  const cudaError_t attr = allow_smem(k_z_fuse<N>, G::SMEM);
  if (attr != cudaSuccess) return attr;
  dim3 grid((unsigned)((Xh + G::B - 1) / G::B), (unsigned)Y, (unsigned)n_tiles);
  WO_LAUNCH("z_fuse", s, (k_z_fuse<N><<<grid, G::NT, G::SMEM, s>>>(in, out, tf, op, Y, Xh)));
  return cudaGetLastError();
}

// The same pass with the z columns in registers (the column transforms of
// wo_regfft.cuh): T lanes of a warp own one (y, x) column, lane l the points
// l + T m, and keep its numerator and denominator over the channels; the next
// channel's data are on their way while the present one is transformed.  The
// shared-memory tiles above wait for each channel's copy in turn and pass
// every point through shared memory nine times: 4 tiles x 9 channels of
// 32x128x128 120.9 -> 33.9 us.
template <class P>
struct FuseRegGeom {
  static constexpr int NT = 128, CPC = NT / P::T;  // columns per CTA
  static constexpr size_t SMEM = ((size_t)P::TW + (size_t)CPC * P::SLICE) * sizeof(float2);
};

template <class P>
__global__ void __launch_bounds__(FuseRegGeom<P>::NT) k_z_fuse_reg(const float2* __restrict__ in,
                                                                  float2* __restrict__ out,
                                                                  const float2* __restrict__ tf, FuseOp op,
                                                                  long long plane) {
  using G = FuseRegGeom<P>;
  constexpr int N = P::N, T = P::T, E = P::E;
  extern __shared__ float2 sm[];
  float2* tw = sm;
  const int l = threadIdx.x % T, cl = threadIdx.x / T;
  float2* S = sm + P::TW + cl * P::SLICE;
  const int t = blockIdx.y, C = op.C;
  const long long cg = (long long)blockIdx.x * G::CPC + cl;
  const bool live = cg < plane;
  const long long col = live ? cg : plane - 1;  // tail lanes compute, store nothing
  const long long vol = N * plane;
  const long long base = (long long)t * C * vol + col + l * plane, step = T * plane;
#if defined(WO_CHECK) && WO_CHECK
  {  // the CTA's last elements in the input and TF volumes and in the output (3D, or one plane a tile)
    const long long end = min((long long)(blockIdx.x + 1) * G::CPC, plane) - 1, nt = gridDim.y;
    const long long planes = op.mode == WO_MODE_3D ? N : 1;
    if (!WO_IN((long long)t * C * vol + (C - 1) * vol + (N - 1) * plane + end, nt * C * vol, 6) ||
        !WO_IN(((long long)t * planes + planes - 1) * plane + end, nt * planes * plane, 6))
      return;  // uniform across the CTA
  }
#endif
  float2 v[E], nx[E], num[E];
  float den[E];
#pragma unroll
  for (int m = 0; m < E; ++m) {
    nx[m] = __ldg(in + base + m * step);
    num[m] = make_float2(0.f, 0.f);
    den[m] = 0.f;
  }
  P::twiddles(tw);  // while the loads are in flight
  __syncthreads();
#pragma unroll 1
  for (int c = 0; c < C; ++c) {
    float2 H[E];
#pragma unroll
    for (int m = 0; m < E; ++m) {
      v[m] = nx[m];
      H[m] = __ldg(tf + base + c * vol + m * step);
    }
    if (c + 1 < C) {
#pragma unroll
      for (int m = 0; m < E; ++m) nx[m] = __ldg(in + base + (c + 1) * vol + m * step);
    }
    P::template fft<false>(v, tw, S, l);
    if (l == 0 && cg == 0) v[0] = op.zero_dc ? make_float2(0.f, 0.f) : make_float2(v[0].x - op.bg_dc[c], v[0].y);
#pragma unroll
    for (int m = 0; m < E; ++m) {
      num[m] = cadd(num[m], cmulc(H[m], v[m]));
      den[m] += cabs2(H[m]);
    }
  }
  const float* st = op.stats + 2LL * t;
  if (op.mode == WO_MODE_3D) {
    const float lam = op.eta_relative ? op.eta * st[0] : op.eta;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const float q = den[m] + lam;
      v[m] = q > 0.f ? cscale(num[m], 1.0f / q) : make_float2(0.f, 0.f);
    }
    P::template fft<true>(v, tw, S, l);
    if (live) {
      float2* o = out + (long long)t * vol + col + l * plane;
#pragma unroll
      for (int m = 0; m < E; ++m) o[m * step] = v[m];
    }
    return;
  }
  // 2D: sum over k of both accumulators, over the column's lanes
  float2 a = make_float2(0.f, 0.f);
  float dd = 0.f;
#pragma unroll
  for (int m = 0; m < E; ++m) {
    a = cadd(a, num[m]);
    dd += den[m];
  }
#pragma unroll
  for (int o = 1; o < T; o <<= 1) {
    a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
    a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
    dd += __shfl_xor_sync(0xffffffffu, dd, o);
  }
  if (live && l == 0) {
    // per-plane sums are 1/Z of the sums over k, so eta enters as Z eta
    const float lam = op.eta_relative ? op.eta * st[1] : op.eta * (float)N;
    const float q = dd + lam;
    out[(long long)t * plane + col] = q > 0.f ? cscale(a, 1.0f / q) : make_float2(0.f, 0.f);
  }
}

template <class P>
cudaError_t launch_z_fuse_reg(const float2* in, float2* out, const float2* tf, const FuseOp& op, int n_tiles, int Y,
                              int Xh, cudaStream_t s) {
  using G = FuseRegGeom<P>;
  const cudaError_t attr = allow_smem(k_z_fuse_reg<P>, G::SMEM);
  if (attr != cudaSuccess) return attr;
  const long long plane = (long long)Y * Xh;
  dim3 grid((unsigned)((plane + G::CPC - 1) / G::CPC), (unsigned)n_tiles);
  WO_LAUNCH("z_fuse", s, (k_z_fuse_reg<P><<<grid, G::NT, G::SMEM, s>>>(in, out, tf, op, plane)));
  return cudaGetLastError();
}

}  // namespace

cudaError_t fuse_stats(const float2* tf, int n_tiles, int C, int Z, int Y, int Xh, float* stats, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(stats, 0, (size_t)n_tiles * 2 * sizeof(float), s);
  if (e != cudaSuccess) return e;
  const long long plane = (long long)Y * Xh;
  // warps a column: enough planes each to fill a thread's loads; CTAs: about
  // two waves of eight an SM over the batch (more only add atomics)
  const int cm = C == 1 ? 1 : C <= 4 ? 4 : kStatsLoads;
  int G = 8;
  while (G > 1 && G * (kStatsLoads / cm) > Z) G /= 2;
  const long long groups = (plane + 256 / G - 1) / (256 / G), want = (2 * 8 * 152 + n_tiles - 1) / n_tiles;
  dim3 grid((unsigned)(groups < want ? groups : want), (unsigned)n_tiles);
  auto run = [&](auto kernel) {
    WO_LAUNCH("fuse_stats", s, (kernel<<<grid, 256, 0, s>>>(tf, C, Z, Y, Xh, G, stats)));
  };
  if (cm == 1) run(k_fuse_stats<1>);
  else if (cm == 4) run(k_fuse_stats<4>);
  else run(k_fuse_stats<kStatsLoads>);
  return cudaGetLastError();
}

cudaError_t z_fuse(int Z, const float2* in, float2* out, const float2* tf, const FuseOp& op, int n_tiles, int Y,
                   int Xh, cudaStream_t s) {
  switch (Z) {
    // even divisions into at most eight lanes of 4 to 16 points
    case 12: return launch_z_fuse_reg<Row2<12, 6>>(in, out, tf, op, n_tiles, Y, Xh, s);
    case 16: return launch_z_fuse_reg<Row2<16, 4>>(in, out, tf, op, n_tiles, Y, Xh, s);
    case 24: return launch_z_fuse_reg<Row2<24, 12>>(in, out, tf, op, n_tiles, Y, Xh, s);
    case 32: return launch_z_fuse_reg<Row2<32, 8>>(in, out, tf, op, n_tiles, Y, Xh, s);
    case 48: return launch_z_fuse_reg<Row2<48, 12>>(in, out, tf, op, n_tiles, Y, Xh, s);
    case 64: return launch_z_fuse_reg<Row2<64, 8>>(in, out, tf, op, n_tiles, Y, Xh, s);
    case 128: return launch_z_fuse_reg<Row2<128, 16>>(in, out, tf, op, n_tiles, Y, Xh, s);
#define WO_CASE(n) \
  case n:          \
    return launch_z_fuse<n>(in, out, tf, op, n_tiles, Y, Xh, s);
    WO_CASE(1) WO_CASE(2) WO_CASE(3) WO_CASE(4) WO_CASE(6) WO_CASE(8) WO_CASE(96) WO_CASE(192) WO_CASE(256)
    WO_CASE(384) WO_CASE(512) WO_CASE(768) WO_CASE(1024) WO_CASE(1536) WO_CASE(2048)
#undef WO_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace wo
