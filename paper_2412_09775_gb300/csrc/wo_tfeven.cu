// wo_tfeven.cu - the arm pass and the PSF-row pass of the TF build for an
// unaberrated detection pupil, which is even in k_x and in k_y.
//
// The detection-side arms B_j = P (i/eta) e^{i phi_j} and P_j = P e^{i phi_j}
// depend on |k_x| and |k_y| alone, phi_j = 2 pi eta z_j:
//   - their columns k_x and -k_x are the same: only the columns 0 .. k_max of
//     the detection band are generated, transformed along y and stored, and
//     the row pass reads column |k_x| (k_max reaches X/2 at critical sampling,
//     where the rounding of k / (X p) can leave that column inside the pupil);
//   - the source-side arm A_j = S P e^{i phi_j} needs only the columns
//     the source reaches (the range kCntLo .. kCntHi of the pupil record), and
//     column -k_x takes the phase factors of k_x.
// Neither changes a value: the columns left out are the same or zero.
//   - p = IDFT2(P_j) is even in y: only its rows 0 .. Y/2 are stored, and the
//     rows y and Y - y of |p|^2 are one row;
//   - with the illumination on axis A is even as well: a and b are stored and
//     transformed for the rows 0 .. Y/2 and each row of the TF serves twice.
// (With a tilted source b is still even, but sharing its rows would lose
// accuracy: near zero frequency the phase TF is what remains of sums
// conj(a) b that cancel, and their rounding cancels too only while a and b
// go through the same transforms.)
//
// On 48 x 192 x 192 tiles (detection band 87 columns, source about 60) this is
// 104 column transforms a plane instead of 174 and 44 columns of phase factors
// instead of 87; on axis five row transforms per row pair instead of nine
// (all three kinds).  256 such tiles, tilted, phase: arms 1.64 -> 1.05 ms, row
// pass 2.08 -> 2.05 ms (the same transforms, half the bytes of b).  96 x 512 x
// 512 on axis, all kinds: arms 0.152 -> 0.083 ms, row pass 0.270 -> 0.187 ms.
#include <type_traits>

#include "wo_fft.cuh"
#include "wo_internal.h"
#include "wo_regfft.cuh"
#include "wo_tf.cuh"

namespace wo {

namespace {

// ------------------------------------------------------------------- arms
template <class P>
struct EvenArmGeom {
  static constexpr int N = P::N, T = P::T, E = P::E;
  static constexpr int NT = T <= 8 ? 128 : 256;
  static constexpr int CPC = NT / T;             // columns |k_x| per CTA
  static constexpr int CH = E % 8 == 0 ? 8 : 4;  // points per load batch
  // the strip tile [N][PITCH] of a transformed arm shares its space with the
  // transposes' slices; PITCH puts a half-warp's writes (T lanes of 16/T
  // columns, or 16 lanes of one column) on distinct 8-byte bank pairs
  static constexpr int PITCH = CPC + (T < 16 ? 16 / T : 1);
  static constexpr size_t SHARED =
      (size_t)N * PITCH > (size_t)CPC * P::SLICE ? (size_t)N * PITCH : (size_t)CPC * P::SLICE;
  // plus the phase factors of the strip, [E][NT]
  static constexpr size_t SMEM = ((size_t)P::TW + SHARED + (size_t)E * NT) * sizeof(float2);
  static constexpr int MINB = NT == 128 ? 4 : 2;
  static_assert(E % CH == 0, "whole load batches");
};

// Bound by latency and issue (record loads, the phase factors, one register
// transform per column); four CTAs of 128 threads per SM by registers.  The
// factors wait in shared memory because the registers hold the transform.
//
// CTA: CPC columns |k_x| of plane j of tile t.  T lanes own a column, lane l
// the points l + T m, as in wo_armsreg.cu.  The phase factors e^{i phi} of the
// column are formed once into the lane's own shared-memory slots; then, arm
// by arm, the values (al + i be) e^{i phi} go into the registers of the
// transform, the amplitudes read from the record (hits in L1 and L2).  A
// transformed arm leaves through a strip tile in shared memory so that every
// warp store writes whole rows of the strip.  Rows outside the detection
// band (|k_y| > k_max of y) are zero in every arm and are not loaded.
template <class P>
__global__ void __launch_bounds__(EvenArmGeom<P>::NT, EvenArmGeom<P>::MINB) k_arms_even(TfArgs a) {
  using G = EvenArmGeom<P>;
  constexpr int N = G::N, T = G::T, E = G::E, NT = G::NT, CPC = G::CPC, CH = G::CH;
  extern __shared__ float2 sm[];
  float2* tw = sm;
  float2* slices = sm + P::TW;        // [CPC][SLICE]: the columns' transposes
  float2* tile = slices;              // [N][PITCH]: an arm's strip on its way out
  float2* phase = slices + G::SHARED;  // [E][NT]: e^{i phi}, zero outside the pupil
  const int X = a.X, Z = a.Z;
  const int t = blockIdx.z, j = blockIdx.y, c0 = blockIdx.x * CPC;
  const int* cnt = a.counts + kCounts * t;
  const int kxm = cnt[kCntKx], kym = cnt[kCntKy];
  if (c0 > kxm) return;  // the strip lies outside the detection band: uniform across the CTA
  const int lo = max(cnt[kCntLo], -kxm), hi = min(cnt[kCntHi], kxm);
  const bool axial = cnt[kCntAxial] != 0;
  const int c1 = min(c0 + CPC - 1, kxm);  // last column of the strip inside the band
#if defined(WO_CHECK) && WO_CHECK
  {  // the columns +-c1 of the records and of the last arm's plane
    const long long nt = gridDim.z;
    if (!WO_IN(c1, X / 2 + 1, 8) || !WO_IN((long long)t * N * X + (long long)(N - 1) * X + X - 1, nt * N * X, 8) ||
        !WO_IN((((long long)t * a.n_arms + a.n_arms - 1) * Z + j) * (long long)N * X + (long long)(N - 1) * X + X - 1,
               nt * a.n_arms * Z * (long long)N * X, 8))
      return;
  }
#endif
  P::twiddles(tw);
  // the plane's focal displacement as a float pair, formed in float64 by one
  // lane of each warp (float64 is slow on this part) and broadcast
  float zh = 0.f, zl = 0.f;
  if ((threadIdx.x & 31) == 0) {
    const double zj = __dadd_rn(__dmul_rn((double)fft_index(j, Z), a.optics[t].z_step_um), a.optics[t].defocus_um);
    zh = __double2float_rn(zj);
    zl = __double2float_rn(__dsub_rn(zj, (double)zh));
  }
  zh = __shfl_sync(0xffffffffu, zh, 0);
  zl = __shfl_sync(0xffffffffu, zl, 0);
  const int l = threadIdx.x % T, cl = threadIdx.x / T;
  const int c = c0 + cl;
  const bool live = c <= c1;
  const bool pos = live && c >= lo && c <= hi;              // the source reaches column c
  const bool neg = live && c > 0 && -c >= lo && -c <= hi;   // and column -c
  const float4* rec = a.rec + (long long)t * N * X + (live ? c : 0);
  const float4* recn = a.rec + (long long)t * N * X + (neg ? X - c : 0);
#pragma unroll
  for (int m0 = 0; m0 < E; m0 += CH) {
    float4 q[CH];
#pragma unroll
    for (int i = 0; i < CH; ++i) {  // the batch's loads first
      const int n = l + T * (m0 + i);
      q[i] = (live && (2 * (m0 + i) < E ? n : N - n) <= kym) ? __ldg(rec + (long long)n * X) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      float s = 0.f, co = 0.f;
      if (q[i].z != 0.f) unit_phasor(phase_frac(q[i].x, q[i].y, zh, zl), &s, &co);
      phase[(m0 + i) * NT + threadIdx.x] = make_float2(co, s);
    }
  }
  __syncthreads();  // the twiddles
  // steps: A at +k_x, A at -k_x (off axis), B, P
  const int first = a.lf_props ? 0 : 3, last = a.want_fl ? 3 : 2;
#pragma unroll 1
  for (int st = first; st <= last; ++st) {
    const bool minus = st == 1, source = st < 2;  // (uniform)
    const bool even = st == 3 || axial;  // rows above Y/2 repeat the rows below: not stored
    if (minus && axial) continue;
    if (source) {  // no column of the strip reached by the source
      const int s0 = minus ? max(c0, 1) : c0;
      if (minus ? (-s0 < lo || -c1 > hi || s0 > c1) : (s0 > hi || c1 < lo)) continue;
    }
    const int slot = source ? 0 : st == 2 ? 1 : (a.lf_props ? 2 : 0);
    const bool mine = source ? (minus ? neg : pos) : live;
    float2 v[E];
#pragma unroll
    for (int m0 = 0; m0 < E; m0 += CH) {
      float w[CH];
#pragma unroll
      for (int i = 0; i < CH; ++i) {
        const int n = l + T * (m0 + i);
        const bool in = mine && (2 * (m0 + i) < E ? n : N - n) <= kym;
        const float4* r = (minus ? recn : rec) + (long long)n * X;
        if (st == 3) w[i] = in ? 1.f : 0.f;
        else if (source) w[i] = in ? __ldg(&r->w) : 0.f;
        else w[i] = in ? __ldg(&r->z) : 0.f;
      }
#pragma unroll
      for (int i = 0; i < CH; ++i) {  // A = S e, P = e (zero outside the pupil), B = i (1/eta) e
        const float2 e = phase[(m0 + i) * NT + threadIdx.x];
        v[m0 + i] = st == 2 ? make_float2(-w[i] * e.y, w[i] * e.x) : make_float2(w[i] * e.x, w[i] * e.y);
      }
    }
    P::template fft<true>(v, tw, slices + cl * P::SLICE, l);
    __syncthreads();  // every column's transposes are done with the slices
#pragma unroll
    for (int m = 0; m < E; ++m) tile[(l + T * m) * G::PITCH + cl] = v[m];
    __syncthreads();
    float2* dst = a.arms + (((long long)t * a.n_arms + slot) * Z + j) * (long long)N * X;
    const int b = threadIdx.x % CPC, cb = c0 + b;  // this thread's column (NT is a multiple of CPC)
    const int kb = minus ? -cb : cb;
    if (cb <= c1 && (!source || (kb >= lo && kb <= hi && !(minus && cb == 0)))) {
      float2* d = dst + (kb < 0 ? X + kb : kb);
      const int rows = even ? N / 2 + 1 : N;
      for (int n = threadIdx.x / CPC; n < rows; n += NT / CPC) d[(long long)n * X] = tile[n * G::PITCH + b];
    }
    __syncthreads();  // the tile's reads are done before the next transform
  }
}

template <class P>
cudaError_t launch_arms_even(const TfArgs& a, cudaStream_t s) {
  using G = EvenArmGeom<P>;
  dim3 grid((unsigned)((a.X / 2 + G::CPC) / G::CPC), (unsigned)a.Z, (unsigned)a.n_tiles);  // columns 0 .. X/2
  const cudaError_t attr = allow_smem(k_arms_even<P>, G::SMEM);
  if (attr != cudaSuccess) return attr;
  WO_LAUNCH("tf_arms", s, (k_arms_even<P><<<grid, G::NT, G::SMEM, s>>>(a)));
  return cudaGetLastError();
}

// --------------------------------------------------------------- PSF rows
constexpr int kPsfThreads = 128;

// Row of an arm, points lane_t + T m: the columns k_x in [lo, hi] from their
// own place, or (even arms) |k_x| <= hi from column |k_x|; zero elsewhere.
template <class P>
__device__ __forceinline__ void load_row(float2 (&v)[P::E], const float2* row, int lo, int hi, bool even, int lane_t) {
  constexpr int N = P::N, N1 = P::E, T = P::T;
#pragma unroll
  for (int m = 0; m < N1; ++m) {
    const int n = lane_t + T * m;
    const int k = 2 * m < N1 ? n : n - N;
    const int col = (2 * m >= N1 && even) ? N - n : n;
    v[m] = (k >= lo && k <= hi) ? __ldg(row + col) : make_float2(0.f, 0.f);
  }
}

// Register index holding W(N - k) in the lane that owns it (wo_psf.cu).
template <int N1>
__device__ __forceinline__ float2 mirror_value(const float2 (&v)[N1], int m, bool lane0) {
  return lane0 ? v[(N1 - m) % N1] : v[N1 - 1 - m];
}

template <class P>
struct EvenPsfGeom {
  static constexpr int RPC = kPsfThreads / P::T;  // row pairs per CTA
  // held-row pitch = T mod 32: the rows of one warp start on distinct banks
  static constexpr int HP = P::N + (((P::T - P::N) % 32) + 32) % 32;
  static constexpr size_t SMEM =
      ((size_t)P::TW + (size_t)RPC * P::SLICE) * sizeof(float2) + (size_t)RPC * HP * sizeof(float);
};

// Bound by issue: the register transforms with their shared-memory exchanges
// and shuffles; four CTAs of 128 threads per SM at every row length (the
// 24-point rows then spill about 70 bytes a thread, as in k_psf_rows_pair).
//
// A lane group (T lanes) takes two rows of one plane: the label-free arms'
// rows 2p and 2p + 1, or with the illumination on axis p and Y - p (0 and Y/2
// for p = 0), p = 0 .. Y/2 - 1; the fluorescence rows always the latter pair.
// The row products and the sharing of real rows' transforms are those of
// k_psf_rows_pair and k_psf_rows_reg (wo_psf.cu):
//   LF == 1: the real rows of the one label-free kind, h0 + i h1 in one
//     transform; LF == 2: each row's complex g gives both kinds' rows;
//   fluorescence: |p|^2 is the same real row for p and Y - p (p > 0).
// Where every group of a warp has two equal rows (on axis, p > 0) the second
// is not transformed; otherwise every lane transforms both, so that the warp
// stays together.  ZK > 0: kx-major bank of ZK planes, [tile][kind][k][j][y].
template <class P, int LF, int ZK>
__global__ void __launch_bounds__(kPsfThreads, 4) k_psf_even(TfArgs a) {
  using G = EvenPsfGeom<P>;
  constexpr int N = P::N, N1 = P::E, T = P::T, RPC = G::RPC, HP = G::HP;
  extern __shared__ float2 sm[];
  float2* tw = sm;
  float2* slices = sm + P::TW;
  float* held = reinterpret_cast<float*>(slices + RPC * P::SLICE);
  const int lt = threadIdx.x % T, r = threadIdx.x / T;
  const int lane = threadIdx.x & 31;
  const int partner = (lane - lt) + (T - lt) % T;  // lane owning N - k
  const bool lane0 = lt == 0;
  float2* S = slices + r * P::SLICE;
  float* Hs = held + r * HP + lt;  // this lane's points lt + T m at Hs[T m]
  const int Y = a.Y, Z = a.Z, hy = Y / 2;
  const long long npairs = (long long)a.n_tiles * Z * hy;
  const long long idx = (long long)blockIdx.x * RPC + r;
  bool live = idx < npairs;
  const long long ii = live ? idx : npairs - 1;  // tails compute, store nothing
  const long long tj = ii / hy;                  // t Z + j
  int p = (int)(ii - tj * hy);
  long long t = tj / Z;
  int j = (int)(tj - t * Z);
  const int Xh = N / 2 + 1;
  const long long kstride = (long long)Z * Y * Xh;
  const bool fl = a.want_fl != 0;
#if defined(WO_CHECK) && WO_CHECK
  {  // the tile's last arm row and last TF bin inside their arrays
    const long long arms_end = (long long)a.n_tiles * a.n_arms * Z * Y * N;
    const long long tf_end = (long long)a.n_tiles * a.n_kinds * kstride;
    if (!WO_IN(t, a.n_tiles, 9) ||
        !WO_IN((((t * a.n_arms + a.n_arms - 1) * Z + j) * (long long)Y + Y - 1) * N + N - 1, arms_end, 9) ||
        !WO_IN((t * a.n_kinds + a.n_kinds - 1) * kstride + ((long long)j * Y + Y - 1) * Xh + N / 2, tf_end, 9)) {
      live = false;
      t = 0;
      j = 0;
      p = 0;
    }
  }
#endif
  const int* cnt = a.counts + kCounts * t;
  const int kxm = cnt[kCntKx];
  const bool axial = cnt[kCntAxial] != 0;
  // the source's range, symmetric (lo = -hi) on axis
  const int lo = max(cnt[kCntLo], -kxm), hi = min(cnt[kCntHi], kxm);
  const int yf = p == 0 ? hy : Y - p;                    // the row that pairs with p
  const int y0 = axial ? p : 2 * p, y1 = axial ? yf : 2 * p + 1;
  const int s1 = (axial && p > 0) ? p : y1;              // the stored row of a and b that stands for y1
  const bool same = __all_sync(0xffffffffu, s1 == y0);   // every group of the warp has two equal rows
  const long long arm_plane = (long long)Y * N;
  const float2* arm0 = a.arms + ((t * a.n_arms) * Z + j) * arm_plane;  // arm q: + q Z planes
  auto row_of = [&](int q, int y) { return arm0 + (long long)q * Z * arm_plane + (long long)y * N; };
  float2 va[N1];
  // the first arm is on its way while the block forms its twiddles
  if constexpr (LF > 0) load_row<P>(va, row_of(0, y0), lo, hi, axial, lt);
  else load_row<P>(va, row_of(0, p), -kxm, kxm, true, lt);
  float sc = 0.f, scf = 0.f;  // float64 set-up: the group's first lane, broadcast
  if (lt == 0) {
    if (LF > 0) sc = lf_scale(a, (int)t);
    if (fl) scf = fl_scale(a, (int)t);
  }
  sc = __shfl_sync(0xffffffffu, sc, lane - lt);
  scf = __shfl_sync(0xffffffffu, scf, lane - lt);
  P::twiddles(tw);
  __syncthreads();
  float2* plane0 = a.tf + t * a.n_kinds * kstride + (long long)j * Y * Xh;  // slot 0 of this plane

  // the partner's conj(W(N - k)) of register m
  auto mirror = [&](const float2(&w)[N1], int m) {
    const float2 mv = mirror_value<N1>(w, m, lane0);
    float2 c;
    c.x = __shfl_sync(0xffffffffu, mv.x, partner);
    c.y = -__shfl_sync(0xffffffffu, mv.y, partner);
    return c;
  };
  // one forward transform of w = h(ya) + i h(yb) into TF slot `slot` of both rows
  auto store_pair = [&](float2(&w)[N1], int slot, int ya, int yb) {
    P::template fft<false>(w, tw, S, lt);
    const long long db = ((t * a.n_kinds + slot) * Xh * (long long)Z + j) * Y;  // kx-major: bin k at db + k Z Y + y
    float2* da = plane0 + slot * kstride + (long long)ya * Xh;
    float2* dbr = plane0 + slot * kstride + (long long)yb * Xh;
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      if (T * m > N / 2) continue;  // no lane stores a bin of this register
      const float2 c = mirror(w, m);
      const int k = lt + T * m;
      if (k > N / 2 || !live) continue;
      const float2 h0 = make_float2(0.5f * (w[m].x + c.x), 0.5f * (w[m].y + c.y));
      const float2 h1 = make_float2(0.5f * (w[m].y - c.y), -0.5f * (w[m].x - c.x));
      if constexpr (ZK > 0) {
        if (!WO_IN(db + (long long)k * (ZK * N) + Y - 1, (long long)a.n_tiles * a.n_kinds * kstride, 9)) continue;
        float2* d = a.tf + db + (long long)k * (ZK * N);
        if (yb == ya + 1 && LF > 0) {  // ya even: one 16-byte store
          *reinterpret_cast<float4*>(d + ya) = make_float4(h0.x, h0.y, h1.x, h1.y);
        } else {
          d[ya] = h0;
          d[yb] = h1;
        }
      } else {
        da[k] = h0;
        dbr[k] = h1;
      }
    }
  };

  if constexpr (LF == 1) {
    float2 vb[N1];
    P::template fft<true>(va, tw, S, lt);
    load_row<P>(vb, row_of(1, y0), -kxm, kxm, true, lt);
    P::template fft<true>(vb, tw, S, lt);
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      const float2 g = cmulc(va[m], vb[m]);
      Hs[T * m] = sc * (a.want_phase ? g.x : -g.y);  // one kind: Re g (phase) or -Im g (absorption)
    }
    if (same) {
#pragma unroll
      for (int m = 0; m < N1; ++m) va[m] = make_float2(Hs[T * m], Hs[T * m]);
    } else {
      load_row<P>(va, row_of(0, s1), lo, hi, axial, lt);
      P::template fft<true>(va, tw, S, lt);
      load_row<P>(vb, row_of(1, s1), -kxm, kxm, true, lt);
      P::template fft<true>(vb, tw, S, lt);
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        const float2 g = cmulc(va[m], vb[m]);
        va[m] = make_float2(Hs[T * m], sc * (a.want_phase ? g.x : -g.y));
      }
    }
    store_pair(va, 0, y0, y1);
  }
  if constexpr (LF == 2) {
#pragma unroll 1
    for (int q = 0; q < 2; ++q) {
      if (q == 1 && same) break;
      const int y = q ? s1 : y0;
      float2 vb[N1];
      if (q == 1) load_row<P>(va, row_of(0, y), lo, hi, axial, lt);
      P::template fft<true>(va, tw, S, lt);
      load_row<P>(vb, row_of(1, y), -kxm, kxm, true, lt);
      P::template fft<true>(vb, tw, S, lt);
#pragma unroll
      for (int m = 0; m < N1; ++m) va[m] = cscale(cmulc(va[m], vb[m]), sc);
      P::template fft<false>(va, tw, S, lt);
      float2* d0 = plane0 + (long long)(q ? y1 : y0) * Xh;
      float2* d1 = plane0 + (long long)y1 * Xh;
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        if (T * m > N / 2) continue;
        const float2 c = mirror(va, m);
        const int k = lt + T * m;
        if (k > N / 2 || !live) continue;
        const float2 hr = make_float2(0.5f * (va[m].x + c.x), 0.5f * (va[m].y + c.y));
        const float2 hm = make_float2(-0.5f * (va[m].y - c.y), 0.5f * (va[m].x - c.x));
        d0[k] = hr;
        d0[kstride + k] = hm;
        if (same) {
          d1[k] = hr;
          d1[kstride + k] = hm;
        }
      }
    }
  }
  if (fl) {
    constexpr int fl_arm = LF > 0 ? 2 : 0;
    if (LF > 0) load_row<P>(va, row_of(fl_arm, p), -kxm, kxm, true, lt);
    P::template fft<true>(va, tw, S, lt);
#pragma unroll
    for (int m = 0; m < N1; ++m) va[m].x = scf * cabs2(va[m]);
    if (__any_sync(0xffffffffu, p == 0)) {  // the rows 0 and Y/2 differ
#pragma unroll
      for (int m = 0; m < N1; ++m) Hs[T * m] = va[m].x;
      load_row<P>(va, row_of(fl_arm, p == 0 ? hy : p), -kxm, kxm, true, lt);
      P::template fft<true>(va, tw, S, lt);
#pragma unroll
      for (int m = 0; m < N1; ++m) va[m] = make_float2(Hs[T * m], scf * cabs2(va[m]));
    } else {
#pragma unroll
      for (int m = 0; m < N1; ++m) va[m].y = va[m].x;
    }
    store_pair(va, LF, p, yf);
  }
}

template <class P, int LF, int ZK>
cudaError_t launch_psf_even(const TfArgs& a, cudaStream_t s) {
  using G = EvenPsfGeom<P>;
  constexpr size_t smem = G::SMEM;
  const cudaError_t attr = allow_smem(k_psf_even<P, LF, ZK>, smem);
  if (attr != cudaSuccess) return attr;
  const long long pairs = (long long)a.n_tiles * a.Z * (a.Y / 2);
  const unsigned grid = (unsigned)((pairs + G::RPC - 1) / G::RPC);
  WO_LAUNCH("tf_psf_rows", s, (k_psf_even<P, LF, ZK><<<grid, kPsfThreads, smem, s>>>(a)));
  return cudaGetLastError();
}

template <class P>
cudaError_t launch_psf_even_any(const TfArgs& a, cudaStream_t s) {
  if (a.kxm) {  // one kind, Y = X, Z 32 or 48 (16 with X = 64) (checked by the caller)
    if constexpr (P::N == 64 || P::N == 128 || P::N == 192) {
      if (a.Y != P::N) return cudaErrorInvalidValue;
      auto go = [&](auto zk) {
        constexpr int ZK = decltype(zk)::value;
        return a.lf_props == 0 ? launch_psf_even<P, 0, ZK>(a, s) : launch_psf_even<P, 1, ZK>(a, s);
      };
      if (a.Z == 48) return go(std::integral_constant<int, 48>{});
      if (a.Z == 32) return go(std::integral_constant<int, 32>{});
      if constexpr (P::N == 64) {
        if (a.Z == 16) return go(std::integral_constant<int, 16>{});
      }
    }
    return cudaErrorInvalidValue;
  }
  switch (a.lf_props) {
    case 0: return launch_psf_even<P, 0, 0>(a, s);
    case 1: return launch_psf_even<P, 1, 0>(a, s);
    default: return launch_psf_even<P, 2, 0>(a, s);
  }
}

template <class F>
cudaError_t arms_even_dispatch(int Y, F f) {
  switch (Y) {
    case 32: return f(Row2<32, 8>{});
    case 48: return f(Row2<48, 12>{});
    case 64: return f(Row2<64, 8>{});
    case 96: return f(Row2<96, 24>{});
    case 128: return f(Row2<128, 16>{});
    case 192: return f(Row2<192, 24>{});
    case 256: return f(Row2<256, 16>{});
    case 512: return f(Row512{});
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

// The rule: an unaberrated pupil, no derivative bank (their arm and row passes
// keep four or seven arms) and the register transforms' lengths along both
// axes (all even).  Everything else runs the general passes.
bool tf_even_supported(const TfArgs& a) {
  if (a.n_zern > 0 || a.want_dz || a.want_grad) return false;
  auto len = [](int n) {
    return n == 32 || n == 48 || n == 64 || n == 96 || n == 128 || n == 192 || n == 256 || n == 512;
  };
  return len(a.X) && len(a.Y);
}

cudaError_t tf_arms_even(const TfArgs& a, cudaStream_t s) {
  return arms_even_dispatch(a.Y, [&](auto p) { return launch_arms_even<decltype(p)>(a, s); });
}

cudaError_t tf_psf_rows_even(const TfArgs& a, cudaStream_t s) {
  return arms_even_dispatch(a.X, [&](auto p) { return launch_psf_even_any<decltype(p)>(a, s); });
}

}  // namespace wo
