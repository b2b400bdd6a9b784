// Step (a): point-source coherency prediction.
//
// C_pq(t,f) = sum_s S_s(f) exp(-2 pi i f/c (u l_s + v m_s + w (n_s - 1))), the
// coherency of a cluster of unpolarised point sources (SAGECal's sky model,
// one cluster = one calibration direction, paper §2).
//
// Mixed path: the (u,v,w) of baseline pq is uvw_p - uvw_q, so the phasor of a
// baseline is the product of two station phasors, e_p conj(e_q).  One kernel
// forms e_p(t,f,s) from a float64 argument reduced to [-1/2, 1/2] turns before
// a float32 sincospi (N phasors per (t,f,s) instead of B), the other contracts
// them, C_pq = sum_s (S_s e_p,s) conj(e_q,s), with 64x64 station tiles in
// shared memory and float32 accumulation.  k_w_splits sums w_pq = sum |C_pq|^2
// over (t,f), the only data the Gauss-Newton matrix needs.
//
// Plain FP64 path: every (source, baseline, timeslot, channel) phase and
// sincos in float64, one thread per (t, b).
#include <algorithm>

#include "sc_common.cuh"

namespace sc {

__device__ __forceinline__ double n_minus_1(double l, double m) {
  double r2 = l * l + m * m;
  return -r2 / (1.0 + sqrt(1.0 - r2));
}

// E[(tf * S + s) * N + p] = exp(-2 pi i f/c uvw_p . (l, m, n-1)), Sf[f*S + s] = S_s(f)
//
// Bound by the float64 pipes (2 FMAs a cycle per SM).  A block takes one
// source and a range of timeslots, a thread one station: n-1 (a square root
// and a division) and the channels' f/c (a division each) are formed once a
// block, the path once a (timeslot, station), which leaves four float64
// instructions per phasor (one thread per phasor formed all of them: about
// 40).  512 stations x 10 timeslots x 4 channels x 100 sources: 142 -> 32 us.
constexpr int kPhasorThreads = 128;
constexpr int kPhasorChannels = 32;  // channels whose f/c a block holds at a time

__global__ void __launch_bounds__(kPhasorThreads) k_station_phasors(
    int N, int T, int F, int S, int t_per, const double* __restrict__ uvw, const double* __restrict__ freqs,
    const double* __restrict__ l, const double* __restrict__ m, const double* __restrict__ flux,
    const double* __restrict__ alpha, double f0, float2* __restrict__ E, float* __restrict__ Sf) {
  __shared__ double s_fc[kPhasorChannels], s_nm1;
  const int p = blockIdx.x * kPhasorThreads + threadIdx.x, s = blockIdx.y;
  const int t0 = blockIdx.z * t_per, t1 = min(T, t0 + t_per);
  const double ls = l[s], ms = m[s];
  if (threadIdx.x == kPhasorThreads - 1) s_nm1 = n_minus_1(ls, ms);
  // the last warp also forms the source's fluxes, once
  if (blockIdx.x == 0 && blockIdx.z == 0 && threadIdx.x >= kPhasorThreads - 32) {
    const double al = alpha[s], fl = flux[s];
    for (int f = threadIdx.x - (kPhasorThreads - 32); f < F; f += 32)
      Sf[f * S + s] = (float)(fl * (al == 0.0 ? 1.0 : pow(freqs[f] / f0, al)));
  }
  for (int fb = 0; fb < F; fb += kPhasorChannels) {
    const int nf = min(kPhasorChannels, F - fb);
    __syncthreads();
    if (threadIdx.x < nf) s_fc[threadIdx.x] = freqs[fb + threadIdx.x] / kCLight;
    __syncthreads();
    if (p >= N) continue;
    const double nm1 = s_nm1;
    for (int t = t0; t < t1; ++t) {
      const double* x = uvw + ((size_t)t * N + p) * 3;
      const double path = fma(x[0], ls, fma(x[1], ms, x[2] * nm1));  // metres
      float2* e = E + ((size_t)(t * F + fb) * S + s) * N + p;
#pragma unroll 4
      for (int f = 0; f < nf; ++f) {
        const double turns = path * s_fc[f];
        const float y = (float)(turns - rint(turns));  // [-1/2, 1/2] turns
        float sn, cs;
        sincospif(2.0f * y, &sn, &cs);
        e[(size_t)f * S * N] = make_float2(cs, -sn);
      }
    }
  }
}

cudaError_t launch_station_phasors(const Shape& s, const double* uvw, const double* freqs,
                                   const double* l, const double* m, const double* flux,
                                   const double* alpha, double f0, int S, float2* E, float* Sf,
                                   cudaStream_t st) {
  if (S <= 0) return cudaSuccess;
  // as many timeslot ranges as give the GPU about four blocks per SM of
  // GB300: more would repeat a block's square root and divisions
  const int nb = (s.N + kPhasorThreads - 1) / kPhasorThreads;
  const long long blocks = (long long)nb * S;
  const int ranges = (int)std::max<long long>(1, std::min<long long>(s.T, (4 * 152 + blocks - 1) / blocks));
  const int t_per = (s.T + ranges - 1) / ranges;
  dim3 grd(nb, S, (s.T + t_per - 1) / t_per);
  k_station_phasors<<<grd, kPhasorThreads, 0, st>>>(s.N, s.T, s.F, S, t_per, uvw, freqs, l, m, flux, alpha, f0, E, Sf);
  return cudaGetLastError();
}

// ---- float32 contraction over sources --------------------------------------------------------

// A block takes a 64x64 station tile and a range of (timeslot, channel)
// pairs, a thread 8x4 baselines.  What bounds it is the float32 pipes (four
// FMAs per source and baseline) and the path from shared memory to the
// registers: 8x4 baselines read 24 floats per 128 FMAs; 4x4, as before, 16 per
// 64, which kept that path as busy as the FMA pipes.  The phasors of the next
// eight sources go to registers before the current ones are summed and to the
// other buffer after them, so that a block waits for global memory once, not
// at every step; eight, not sixteen, keep the registers at 128 and four blocks
// on an SM.  The ranges are short, which evens out the blocks' share of the
// SMs (36 tiles of 512 stations in 9 ranges left a third of them idle at the
// end): w, whose sums follow longer ranges, is formed from C (k_w_splits).
// 512 stations x 10 timeslots x 4 channels x 100 sources: 211 -> 162 us, the
// FMAs' own time being 52; 128 x 20 x 8 x 25: 30 -> 26.
constexpr int kCT = 64;          // stations per tile edge
constexpr int kCS = 8;           // sources staged per step
constexpr int kTX = 16;          // threads along a row of the tile
constexpr int kCThreads = 8 * kTX;

__global__ void __launch_bounds__(kCThreads, 4) k_coherency_f32(int N, int T, int F, int S, int64_t B, int nt,
                                                                int per, const float2* __restrict__ E,
                                                                const float* __restrict__ Sf,
                                                                float2* __restrict__ C) {
  __shared__ __align__(16) float2 sa[2][kCS][kCT];  // S_s(f) e_p,s
  __shared__ __align__(16) float2 se[2][kCS][kCT];  // e_q,s
  // tile (tp, tq), tp <= tq, from the linear block index
  int L = blockIdx.x, tp = 0;
  while (L >= nt - tp) { L -= nt - tp; ++tp; }
  const int tq = tp + L;
  const int p0 = tp * kCT, q0 = tq * kCT;
  const int tf0 = blockIdx.y * per, tf1 = min(T * F, tf0 + per);
  // rows 2 ty + 16 i, + 1 (i = 0..3) and columns 2 tx + 32 j, + 1 (j = 0, 1)
  const int tx = threadIdx.x % kTX, ty = threadIdx.x / kTX;

  constexpr int kPer = kCS * kCT / kCThreads;
  const int c = threadIdx.x % kCT, ss0 = threadIdx.x / kCT;
  float2 va[kPer], ve[kPer];
  float fl[kPer];
  auto fetch = [&](int tf, int s0) {
    const int f = tf % F;
    const float2* Et = E + (size_t)tf * S * N;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int sidx = s0 + ss0 + u * (kCThreads / kCT);
      const bool in = tf < tf1 && sidx < S;
      va[u] = ve[u] = make_float2(0.f, 0.f);
      fl[u] = in ? __ldg(Sf + f * S + sidx) : 0.f;
      if (in && p0 + c < N) va[u] = __ldg(Et + (size_t)sidx * N + p0 + c);
      if (in && q0 + c < N) ve[u] = __ldg(Et + (size_t)sidx * N + q0 + c);
    }
  };
  auto put = [&](int b) {
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int ss = ss0 + u * (kCThreads / kCT);
      sa[b][ss][c] = make_float2(va[u].x * fl[u], va[u].y * fl[u]);
      se[b][ss][c] = ve[u];
    }
  };

  int n = 0;
  fetch(tf0, 0);
  put(0);
  for (int tf = tf0; tf < tf1; ++tf) {
    const int t = tf / F, f = tf % F;
    float ar[8][4], ai[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) ar[i][j] = ai[i][j] = 0.f;
    for (int s0 = 0; s0 < S; s0 += kCS, ++n) {
      __syncthreads();  // step n is staged, and the other buffer is free
      if (s0 + kCS < S) fetch(tf, s0 + kCS);
      else fetch(tf + 1, 0);
      const int ns = min(kCS, S - s0);
#pragma unroll 2
      for (int ss = 0; ss < ns; ++ss) {
        float4 a[4], e[2];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(&sa[n & 1][ss][2 * ty + 16 * i]);
#pragma unroll
        for (int j = 0; j < 2; ++j) e[j] = *reinterpret_cast<const float4*>(&se[n & 1][ss][2 * tx + 32 * j]);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float ax = i & 1 ? a[i >> 1].z : a[i >> 1].x, ay = i & 1 ? a[i >> 1].w : a[i >> 1].y;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float ex = j & 1 ? e[j >> 1].z : e[j >> 1].x, ey = j & 1 ? e[j >> 1].w : e[j >> 1].y;
            // a * conj(e)
            ar[i][j] = fmaf(ax, ex, fmaf(ay, ey, ar[i][j]));
            ai[i][j] = fmaf(ay, ex, fmaf(-ax, ey, ai[i][j]));
          }
        }
      }
      put((n + 1) & 1);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int p = p0 + 2 * ty + 16 * (i >> 1) + (i & 1);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int q = q0 + 2 * tx + 32 * (j >> 1) + (j & 1);
        if (p < q && q < N) C[((size_t)t * B + bl_index(p, q, N)) * F + f] = make_float2(ar[i][j], ai[i][j]);
      }
    }
  }
}

cudaError_t launch_coherency_f32(const Shape& s, int S, const float2* E, const float* Sf, float2* C,
                                 cudaStream_t st) {
  // an empty cluster predicts zero coherencies
  if (S <= 0) return cudaMemsetAsync(C, 0, sizeof(float2) * (size_t)s.T * s.B * s.F, st);
  const int nt = (s.N + kCT - 1) / kCT, tiles = nt * (nt + 1) / 2, TF = s.T * s.F;
  // ranges of (timeslot, channel) pairs: about eight blocks per SM of GB300
  const int ranges = std::max(1, std::min(TF, (8 * 152 + tiles - 1) / tiles)), per = (TF + ranges - 1) / ranges;
  const dim3 grd(tiles, (TF + per - 1) / per);
  k_coherency_f32<<<grd, kCThreads, 0, st>>>(s.N, s.T, s.F, S, s.B, nt, per, E, Sf, C);
  return cudaGetLastError();
}

// w_pq = sum_{t,f} |C_pq(t,f)|^2 of one cluster in float32: the sums of
// `splits` equal ranges of the (t, f) pairs, added in order.  A warp sums a
// range of 32 baselines, a block's warps the next kWRanges ranges (one thread
// per baseline over all of them leaves a chain of T F loads: 50 us at 128
// stations x 20 timeslots x 8 channels).
constexpr int kWRanges = 16;

__global__ void __launch_bounds__(32 * kWRanges) k_w_splits(int T, int F, int64_t B, int splits,
                                                            const float2* __restrict__ C, float* __restrict__ w) {
  __shared__ float s_part[kWRanges][32];
  const int lane = threadIdx.x % 32, r = threadIdx.x / 32;
  const int64_t b = (int64_t)blockIdx.x * 32 + lane;
  const int TF = T * F;
  float acc = 0.f;
  for (int i0 = 0; i0 < splits; i0 += kWRanges) {
    const int i = i0 + r;
    if (i < splits && b < B) {
      const int tf0 = (int)((int64_t)TF * i / splits), tf1 = (int)((int64_t)TF * (i + 1) / splits);
      int t = tf0 / F, f = tf0 % F;
      float part = 0.f;
#pragma unroll 4
      for (int tf = tf0; tf < tf1; ++tf) {
        const float2 c = __ldg(C + ((size_t)t * B + b) * F + f);
        part += c.x * c.x + c.y * c.y;
        if (++f == F) f = 0, ++t;
      }
      s_part[r][lane] = part;
    }
    __syncthreads();
    if (r == 0)
      for (int u = 0; u < kWRanges && i0 + u < splits; ++u) acc += s_part[u][lane];
    __syncthreads();
  }
  if (r == 0 && b < B) w[b] = acc;
}

cudaError_t launch_w_splits(const Shape& s, int splits, const float2* C, float* w, cudaStream_t st) {
  k_w_splits<<<(unsigned)((s.B + 31) / 32), 32 * kWRanges, 0, st>>>(s.T, s.F, s.B, splits, C, w);
  return cudaGetLastError();
}

// ---- plain float64 path --------------------------------------------------------------------

__global__ void k_predict_f64(int N, int T, int F, int S, int64_t B, const double* __restrict__ uvw,
                              const double* __restrict__ freqs, const double* __restrict__ l,
                              const double* __restrict__ m, const double* __restrict__ flux,
                              const double* __restrict__ alpha, double f0, double2* __restrict__ C) {
  int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)T * B) return;
  int t = (int)(idx / B);
  int64_t b = idx % B;
  int p, q;
  bl_pair(b, N, p, q);
  const double* xp = uvw + ((size_t)t * N + p) * 3;
  const double* xq = uvw + ((size_t)t * N + q) * 3;
  double u = xp[0] - xq[0], v = xp[1] - xq[1], w = xp[2] - xq[2];
  for (int f = 0; f < F; ++f) {
    double fr = freqs[f];
    double re = 0.0, im = 0.0;
    for (int s = 0; s < S; ++s) {
      double ls = __ldg(l + s), ms = __ldg(m + s);
      double path = u * ls + v * ms + w * n_minus_1(ls, ms);
      double turns = path * (fr / kCLight);
      double sn, cs;
      sincospi(2.0 * (turns - rint(turns)), &sn, &cs);
      double S_f = __ldg(flux + s) * pow(fr / f0, __ldg(alpha + s));
      re += S_f * cs;
      im -= S_f * sn;
    }
    C[((size_t)t * B + b) * F + f] = make_double2(re, im);
  }
}

cudaError_t launch_predict_f64(const Shape& s, const double* uvw, const double* freqs,
                               const double* l, const double* m, const double* flux,
                               const double* alpha, double f0, int S, double2* C,
                               cudaStream_t st) {
  int64_t n = (int64_t)s.T * s.B;
  k_predict_f64<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(s.N, s.T, s.F, S, s.B, uvw, freqs, l, m,
                                                              flux, alpha, f0, C);
  return cudaGetLastError();
}

// w_pq = sum_{t,f} |C_pq(t,f)|^2
template <typename R>
__global__ void k_w_from_C(int T, int F, int64_t B, const R* __restrict__ C, R* __restrict__ w) {
  int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  R acc = 0;
  for (int t = 0; t < T; ++t)
    for (int f = 0; f < F; ++f) {
      cx<R> c = ld_c(C + 2 * (((size_t)t * B + b) * F + f));
      acc += norm2(c);
    }
  w[b] = acc;
}

template <typename R>
cudaError_t launch_w_from_C(const Shape& s, const R* C, R* w, cudaStream_t st) {
  k_w_from_C<R><<<(unsigned)((s.B + 255) / 256), 256, 0, st>>>(s.T, s.F, s.B, C, w);
  return cudaGetLastError();
}
template cudaError_t launch_w_from_C<float>(const Shape&, const float*, float*, cudaStream_t);
template cudaError_t launch_w_from_C<double>(const Shape&, const double*, double*, cudaStream_t);

}  // namespace sc
