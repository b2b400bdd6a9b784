// After calibration: the residual of the whole sky model, optionally
// corrected for the gains of one direction c,
//     R = V - sum_k c_k(t,f) G_k,      G_k = J_kp J_kq^H
//     R <- J_cp^{-1} R J_cq^{-H}
// in one streaming pass.  Every visibility of V is read once, the coherency
// of every cluster once, and R written once: (8K + 64) bytes per visibility
// in SC_MIXED (complex64), twice that in SC_FP64.  Subtracting one cluster
// at a time would stream V and R through HBM K times.
//
// Work item: one baseline and a slab of NV consecutive (timeslot, channel)
// pairs.  Consecutive threads take consecutive baselines of the same slab, so
// a warp's loads of V, C and R cover contiguous [F][2][2] and [F] blocks.
// The NV accumulators stay in registers through the cluster loop; per
// cluster and item the thread loads J_kp and J_kq (a few hundred KB for all
// clusters, L2-resident, rounded to R once by k_gain_prep) and forms G_k once
// for its NV visibilities.  (Channel-major items, one (baseline, channel)
// pair per thread with fully contiguous warp accesses, measured slower: each
// of the F threads of a baseline forms G_k again.)
#include <algorithm>

#include "sc_common.cuh"

namespace sc {

// Jr [K][N][8]: every cluster's Jones rounded to R.  Jinv [N][8]: the
// inverses of cluster corr's Jones, adjugate over determinant in float64,
// then rounded.  A station with |det J|^2 <= 1e-24 |J|_F^4 (that is
// |det J| <= 1e-12 |J|_F^2) gets Jinv = 0, which zeroes its baselines, and
// raises SC_STATUS_SINGULAR.
template <typename R>
__global__ void k_gain_prep(int K, int N, int corr, const double* __restrict__ J,
                            R* __restrict__ Jr, R* __restrict__ Jinv,
                            uint32_t* __restrict__ status) {
  const int KN = K * N;
  const int n = KN + (corr >= 0 ? N : 0);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (i < KN) {
#pragma unroll
      for (int e = 0; e < 8; ++e) Jr[8 * (size_t)i + e] = (R)J[8 * (size_t)i + e];
      continue;
    }
    const int s = i - KN;
    const double* g = J + 8 * ((size_t)corr * N + s);
    const cx<double> a{g[0], g[1]}, b{g[2], g[3]}, c{g[4], g[5]}, d{g[6], g[7]};
    const cx<double> det = a * d - b * c;
    const double fro2 = norm2(a) + norm2(b) + norm2(c) + norm2(d);
    R* o = Jinv + 8 * (size_t)s;
    if (norm2(det) <= 1e-24 * fro2 * fro2) {
#pragma unroll
      for (int e = 0; e < 8; ++e) o[e] = (R)0;
      atomicOr(status, SC_STATUS_SINGULAR);
      continue;
    }
    // 1/det = conj(det) / |det|^2
    const cx<double> r = scale(conj(det), 1.0 / norm2(det));
    const cx<double> nb{-b.re, -b.im}, nc{-c.re, -c.im};
    const cx<double> v[4] = {d * r, nb * r, nc * r, a * r};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      o[2 * e] = (R)v[e].re;
      o[2 * e + 1] = (R)v[e].im;
    }
  }
}

// one visibility by coherent (not read-only-path) vector loads, since R may
// be V
__device__ __forceinline__ m22<float> ld_vis_rw(const float* p) {
  const float4 u = reinterpret_cast<const float4*>(p)[0], v = reinterpret_cast<const float4*>(p)[1];
  return {{u.x, u.y}, {u.z, u.w}, {v.x, v.y}, {v.z, v.w}};
}
__device__ __forceinline__ m22<double> ld_vis_rw(const double* p) {
  const double2* q = reinterpret_cast<const double2*>(p);
  const double2 a = q[0], b = q[1], c = q[2], d = q[3];
  return {{a.x, a.y}, {b.x, b.y}, {c.x, c.y}, {d.x, d.y}};
}

// Per data type: NV visibilities per work item, the unroll of the cluster
// loop and the blocks per SM the register budget is cut for.  For complex64,
// 4 visibilities with the loop unrolled 4 times keep 16 coherency loads of
// each thread in flight at 128 registers, 2 blocks of 256 per SM (64 KB of
// loads per SM; an HBM stream needs about half that).  The float64 path, kept
// for comparison, uses 1 block per SM without spills.
template <typename R> struct SlabOf;
template <> struct SlabOf<float> {
  static constexpr int NV = 4, UNROLL = 4, MINB = 2;
};
template <> struct SlabOf<double> {
  static constexpr int NV = 4, UNROLL = 1, MINB = 1;
};

// IX: index type of a visibility or coherency element; uint32_t when
// 2 K T B F < 2^31 (every index into C fits), else size_t.
template <typename R, int NV, typename IX>
__global__ void __launch_bounds__(256, SlabOf<R>::MINB) k_residual_all(int N, int T, int F, int64_t B, int K,
                                                      int nslab, const R* V,
                                                      const R* __restrict__ C,
                                                      const R* __restrict__ Jr,
                                                      const R* __restrict__ Jinv, R* Rout,
                                                      double* __restrict__ part) {
  const int TF = T * F;
  const int64_t n_items = (int64_t)nslab * B;
  const IX per_cluster = (IX)TF * (IX)B;  // T*B*F coherencies
  double cost = 0.0;
  // grid-stride over (slab, baseline) items; the grid is sized to the
  // resident blocks
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n_items;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int slab = (int)(idx / B);
    const int64_t b = idx - (int64_t)slab * B;
    int p, q;
    bl_pair(b, N, p, q);
    const int r0 = slab * NV;
    const int nv = min(NV, TF - r0);
    // visibility index (t*B + b)*F + f of the slab's pairs r0 .. r0+NV-1
    IX off[NV];
    {
      int t = r0 / F, f = r0 - t * F;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        off[i] = ((IX)t * (IX)B + (IX)b) * (IX)F + (IX)f;
        if (++f == F) {
          f = 0;
          ++t;
        }
      }
    }
    m22<R> acc[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      acc[i] = i < nv ? ld_vis_rw(V + 8 * off[i]) : mzero<R>();
    }
#pragma unroll(SlabOf<R>::UNROLL)
    for (int k = 0; k < K; ++k) {
      const m22<R> G = mul_h(ld_vis(Jr + 8 * ((size_t)k * N + p)), ld_vis(Jr + 8 * ((size_t)k * N + q)));
      const R* Ck = C + (IX)2 * (IX)k * per_cluster;
#pragma unroll
      for (int i = 0; i < NV; ++i)
        if (i < nv) acc[i] = acc[i] - smul(ld_c(Ck + 2 * off[i]), G);
    }
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (i < nv) cost += (double)frob2(acc[i]);
    if (Jinv != nullptr) {
      const m22<R> Ip = ld_vis(Jinv + 8 * (size_t)p), Iq = ld_vis(Jinv + 8 * (size_t)q);
#pragma unroll
      for (int i = 0; i < NV; ++i) acc[i] = mul_h(mul(Ip, acc[i]), Iq);
    }
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (i < nv) st_vis(Rout + 8 * off[i], acc[i]);
  }
  if (part == nullptr) return;
  // block sum of the cost, in a fixed order for a fixed grid
  __shared__ double sh[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cost += __shfl_xor_sync(0xffffffffu, cost, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = cost;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
    part[blockIdx.x] = t;
  }
}

// ---- complex64: coherencies staged through a shared-memory ring ------------------------
//
// The register kernel above keeps one cluster's NV coherency loads of each
// thread in flight: about 16 KB per SM, well short of what HBM latency
// needs.  Here every thread streams its own (item, cluster) sequence
// through a ring of S stages in shared memory filled by cp.async, with a
// prefetch cursor S steps ahead of the arithmetic (crossing item
// boundaries), so S x NV x 8 B of each thread are in flight without holding
// registers.  The visibilities of an item arrive with its first stage.  A
// thread reads only slots it filled itself, so cp.async.wait_group alone
// orders the data (no block barrier).  Slots are laid out [stage][i][thread]
// so a warp's 8-byte reads are conflict-free.  Requires K >= S: the
// visibility slot of an item is refilled only after its first stage has
// been consumed.
//
// What bounds it is the issue of instructions at 16 warps per SM (HBM runs at
// 0.7 of its rate), so they are what is saved: an item is five timeslots of a
// (baseline, channel) pair, whose loads are contiguous across a warp and need
// no addresses of their own, and the products run on pairs of floats (three
// instructions per entry instead of six).  512 stations x 10 timeslots x 4
// channels, 40 clusters: 545 us with items of four channels, 443 with
// timeslots, 405 with pairs.

namespace {
__device__ __forceinline__ void ra_cp8(void* dst, const void* src) {
  unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void ra_cp16(void* dst, const void* src) {
  unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void ra_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int W>
__device__ __forceinline__ void ra_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(W) : "memory"); }
}  // namespace

constexpr int kPipeThreads = 256;
constexpr int kPipeStages = 4;
constexpr int kPipeMaxNV = 5;  // timeslots per item at most

template <int NV>
constexpr size_t pipe_smem_bytes() {
  return (size_t)kPipeStages * NV * kPipeThreads * 8 + (size_t)NV * 2 * kPipeThreads * 16;
}

// Pairs of float32 in one register pair; each half rounds like the scalar
// instruction.
namespace {
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
}  // namespace

// An item: nt x nf = NV timeslots x channels of a baseline, in nslab slabs of
// the timeslots and ngrp groups of the channels.
struct PipeSplit {
  int nt, nf, nslab, ngrp;
};

template <typename IX, int NV>
__global__ void __launch_bounds__(kPipeThreads, 2) k_residual_all_pipe(
    int N, int T, int F, int64_t B, int K, PipeSplit sp, const float* V, const float* __restrict__ C,
    const float* __restrict__ Jr, const float* __restrict__ Jinv, float* Rout,
    double* __restrict__ part) {
  constexpr int S = kPipeStages;
  extern __shared__ __align__(16) unsigned char ra_smem[];
  float2* ring = reinterpret_cast<float2*>(ra_smem);                                  // [S][NV][T]
  float4* vslot = reinterpret_cast<float4*>(ra_smem + (size_t)S * NV * kPipeThreads * 8);  // [2NV][T]
  const int tid = threadIdx.x;
  const IX BF = (IX)B * (IX)F;  // elements of one timeslot
  // five elements are five timeslots: constants here leave the registers
  constexpr bool kTimes = NV == kPipeMaxNV;
  const IX cols = kTimes ? BF : (IX)B * (IX)sp.ngrp, n_items = (IX)sp.nslab * cols;
  const IX stride = (IX)gridDim.x * kPipeThreads;
  const size_t per_cluster = (size_t)T * (size_t)BF;
  const int nf = kTimes ? 1 : sp.nf, nt = kTimes ? NV : sp.nt;
  IX steps[NV];  // from an item's first element to its others
#pragma unroll
  for (int i = 0; i < NV; ++i) steps[i] = (IX)(i / nf) * BF + (IX)(i % nf);
  auto step = [&](int i) -> size_t { return kTimes ? (size_t)((IX)i * BF) : (size_t)steps[i]; };

  // item idx: its baseline, its first element and which of its elements exist
  auto has = [](unsigned live, int i) { return kTimes ? i < (int)live : (bool)(live >> i & 1); };
  auto locate = [&](IX idx, IX& b, IX& off, unsigned& live) {
    const IX slab = idx / cols, col = idx - slab * cols;
    const int t0 = (int)slab * nt;
    if (kTimes) {
      b = col / (IX)F;
      off = (IX)t0 * BF + col;
      live = min(NV, T - t0);
      return;
    }
    b = col / (IX)sp.ngrp;
    const int f0 = (int)(col - b * (IX)sp.ngrp) * nf;
    off = (IX)t0 * BF + b * (IX)F + (IX)f0;
    live = (1u << NV) - 1;
    if (t0 + nt > T || f0 + nf > F) {
      live = 0;
      for (int i = 0; i < NV; ++i)
        if (t0 + i / nf < T && f0 + i % nf < F) live |= 1u << i;
    }
  };

  // prefetch cursor: (pf_idx, pf_k), S steps ahead of the arithmetic
  IX pf_idx = (IX)blockIdx.x * kPipeThreads + tid;
  int pf_k = 0, pf_stage = 0;
  unsigned pf_live = 0;
  IX pf_off = 0;
  const float* pf_c = C;
  auto seek = [&]() {
    pf_live = 0;
    if (pf_idx < n_items) {
      IX b;
      locate(pf_idx, b, pf_off, pf_live);
      pf_c = C + 2 * (size_t)pf_off;
    }
  };
  seek();
  auto issue = [&]() {
    float2* dst = ring + pf_stage * NV * kPipeThreads + tid;
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (has(pf_live, i)) ra_cp8(dst + i * kPipeThreads, pf_c + 2 * step(i));
    if (pf_k == 0) {
      const float* Vi = V + 8 * (size_t)pf_off;
#pragma unroll
      for (int i = 0; i < NV; ++i)
        if (has(pf_live, i)) {
          ra_cp16(&vslot[(2 * i) * kPipeThreads + tid], Vi + 8 * step(i));
          ra_cp16(&vslot[(2 * i + 1) * kPipeThreads + tid], Vi + 8 * step(i) + 4);
        }
    }
    ra_commit();
    pf_stage = pf_stage + 1 == S ? 0 : pf_stage + 1;
    pf_c += 2 * per_cluster;
    if (++pf_k == K) {
      pf_k = 0;
      pf_idx += stride;
      seek();
    }
  };
#pragma unroll 1
  for (int s = 0; s < S; ++s) issue();

  double cost = 0.0;
  int stage = 0;
#pragma unroll 1
  for (IX idx = (IX)blockIdx.x * kPipeThreads + tid; idx < n_items; idx += stride) {
    IX off, b;
    unsigned live;
    locate(idx, b, off, live);
    int p, q;
    bl_pair((int64_t)b, N, p, q);
    f32x2 acc[NV][4];
    unsigned jp = p, jq = q;  // rows of Jr
    m22<float> Jp = ld_vis(Jr + 8 * (size_t)jp), Jq = ld_vis(Jr + 8 * (size_t)jq);
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
      const m22<float> G = mul_h(Jp, Jq);
      // c G = (cr gr - ci gi, cr gi + ci gr) as cr (gr, gi) + ci (-gi, gr)
      const f32x2 g[4] = {pack2(G.a.re, G.a.im), pack2(G.b.re, G.b.im), pack2(G.c.re, G.c.im), pack2(G.d.re, G.d.im)};
      const f32x2 h[4] = {pack2(-G.a.im, G.a.re), pack2(-G.b.im, G.b.re), pack2(-G.c.im, G.c.re),
                          pack2(-G.d.im, G.d.re)};
      if (k + 1 < K) {
        jp += N;
        jq += N;
        Jp = ld_vis(Jr + 8 * (size_t)jp);
        Jq = ld_vis(Jr + 8 * (size_t)jq);
      }
      ra_wait<S - 1>();
      if (k == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          const float4 u = vslot[(2 * i) * kPipeThreads + tid], w = vslot[(2 * i + 1) * kPipeThreads + tid];
          acc[i][0] = pack2(u.x, u.y), acc[i][1] = pack2(u.z, u.w);
          acc[i][2] = pack2(w.x, w.y), acc[i][3] = pack2(w.z, w.w);
        }
      }
      const float2* src = ring + stage * NV * kPipeThreads + tid;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const float2 c = src[i * kPipeThreads];
        const f32x2 nr = pack2(-c.x, -c.x), ni = pack2(-c.y, -c.y);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][e] = add2(acc[i][e], fma2(nr, g[e], mul2(ni, h[e])));
      }
      stage = stage + 1 == S ? 0 : stage + 1;
      issue();
    }
    m22<float> r[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const float2 e0 = unpack2(acc[i][0]), e1 = unpack2(acc[i][1]), e2 = unpack2(acc[i][2]), e3 = unpack2(acc[i][3]);
      r[i] = {{e0.x, e0.y}, {e1.x, e1.y}, {e2.x, e2.y}, {e3.x, e3.y}};
      if (has(live, i)) cost += (double)frob2(r[i]);
    }
    if (Jinv != nullptr) {
      const m22<float> Ip = ld_vis(Jinv + 8 * (size_t)p), Iq = ld_vis(Jinv + 8 * (size_t)q);
#pragma unroll
      for (int i = 0; i < NV; ++i) r[i] = mul_h(mul(Ip, r[i]), Iq);
    }
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (has(live, i)) st_vis(Rout + 8 * ((size_t)off + step(i)), r[i]);
  }
  ra_wait<0>();
  if (part == nullptr) return;
  __shared__ double sh[kPipeThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cost += __shfl_xor_sync(0xffffffffu, cost, o);
  if ((tid & 31) == 0) sh[tid >> 5] = cost;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < kPipeThreads / 32; ++w) t += sh[w];
    part[blockIdx.x] = t;
  }
}

template <typename R>
cudaError_t launch_gain_prep(const Shape& s, const double* J, int corr, R* Jr, R* Jinv,
                             uint32_t* status, cudaStream_t st) {
  const int n = s.K * s.N + (corr >= 0 ? s.N : 0);
  k_gain_prep<R><<<(n + 255) / 256, 256, 0, st>>>(s.K, s.N, corr, J, Jr, Jinv, status);
  return cudaGetLastError();
}

// resident blocks of a kernel at the given block size and dynamic shared memory
template <typename Kern>
static int resident_blocks(Kern kern, int threads, size_t smem) {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem);
  return std::max(1, sms * std::max(per, 1));
}

template <typename IX, int NV>
static cudaError_t go_pipe(const Shape& s, const PipeSplit& sp, const float* V, const float* C, const float* Jr,
                           const float* Jinv, float* Rout, double* part, int max_parts, int* n_parts,
                           cudaStream_t st) {
  constexpr size_t smem = pipe_smem_bytes<NV>();
  const auto kern = k_residual_all_pipe<IX, NV>;
  // per device and cheap: set on every launch
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  static const int resident = resident_blocks(kern, kPipeThreads, smem);
  const int64_t n_items = (int64_t)sp.nslab * sp.ngrp * s.B;
  const int grid = (int)std::min<int64_t>(
      std::min<int64_t>((n_items + kPipeThreads - 1) / kPipeThreads, resident), max_parts);
  kern<<<grid, kPipeThreads, smem, st>>>(s.N, s.T, s.F, s.B, s.K, sp, V, C, Jr, Jinv, Rout, part);
  *n_parts = grid;
  return cudaGetLastError();
}

// The split with the most visibilities per item, since an item forms its
// baseline's G once per cluster: five timeslots, or up to four as timeslots x
// channels.  Timeslots alone, whose loads are contiguous across a warp, unless
// channels give a tenth more (2 x 2 of 2 timeslots x 4 channels: 73 us, 2 x 1:
// 99, at 512 stations and 20 clusters); items of three count less (6 x 4 in
// items of 2 x 2: 167 us, of 3 x 1: 220).
static PipeSplit pipe_split(int T, int F) {
  auto even = [](int n, int cap, int& parts) { parts = (n + cap - 1) / cap; return (n + parts - 1) / parts; };
  PipeSplit best{};
  double most = 0.0;
  for (int c = 0; c <= std::min(F, kPipeMaxNV - 1); ++c) {
    PipeSplit p;
    p.nf = even(F, std::max(c, 1), p.ngrp);
    p.nt = even(T, c == 0 ? kPipeMaxNV : (kPipeMaxNV - 1) / p.nf, p.nslab);
    const double vis = (double)T * F / ((double)p.nslab * p.ngrp) * (p.nf > 1 ? 0.9 : 1.0) *
                       (p.nt * p.nf == 3 ? 0.85 : 1.0);
    if (vis > most) most = vis, best = p;
  }
  return best;
}

template <typename IX>
static cudaError_t pick_pipe(const Shape& s, const float* V, const float* C, const float* Jr,
                             const float* Jinv, float* Rout, double* part, int max_parts, int* n_parts,
                             cudaStream_t st) {
  const PipeSplit sp = pipe_split(s.T, s.F);
  switch (sp.nt * sp.nf) {
    case 1: return go_pipe<IX, 1>(s, sp, V, C, Jr, Jinv, Rout, part, max_parts, n_parts, st);
    case 2: return go_pipe<IX, 2>(s, sp, V, C, Jr, Jinv, Rout, part, max_parts, n_parts, st);
    case 3: return go_pipe<IX, 3>(s, sp, V, C, Jr, Jinv, Rout, part, max_parts, n_parts, st);
    case 4: return go_pipe<IX, 4>(s, sp, V, C, Jr, Jinv, Rout, part, max_parts, n_parts, st);
    default: return go_pipe<IX, 5>(s, sp, V, C, Jr, Jinv, Rout, part, max_parts, n_parts, st);
  }
}

template <typename R>
cudaError_t launch_residual_all(const Shape& s, const R* V, const R* C, const R* Jr,
                                const R* Jinv, R* Rout, double* part, int max_parts, int* n_parts,
                                cudaStream_t st) {
  constexpr int NV = SlabOf<R>::NV;
  const uint64_t top_ = (uint64_t)s.T * s.F * (uint64_t)s.B * (uint64_t)std::max(8, 2 * s.K);
  if constexpr (sizeof(R) == 4) {
    if (s.K >= kPipeStages) {
      return top_ < (1ull << 31)
                 ? pick_pipe<uint32_t>(s, V, C, Jr, Jinv, Rout, part, max_parts, n_parts, st)
                 : pick_pipe<size_t>(s, V, C, Jr, Jinv, Rout, part, max_parts, n_parts, st);
    }
  }
  static const int resident = [] {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_residual_all<R, NV, uint32_t>, 256, 0);
    return std::max(1, sms * std::max(per, 1));
  }();
  const int nslab = (s.T * s.F + NV - 1) / NV;
  const int64_t n_items = (int64_t)nslab * s.B;
  const int grid =
      (int)std::min<int64_t>(std::min<int64_t>((n_items + 255) / 256, resident), max_parts);
  // largest index: 8 T B F (V, R) or 2 K T B F (C)
  const uint64_t top = (uint64_t)s.T * s.F * (uint64_t)s.B * (uint64_t)std::max(8, 2 * s.K);
  if (top < (1ull << 31))
    k_residual_all<R, NV, uint32_t><<<grid, 256, 0, st>>>(s.N, s.T, s.F, s.B, s.K, nslab, V, C, Jr,
                                                          Jinv, Rout, part);
  else
    k_residual_all<R, NV, size_t><<<grid, 256, 0, st>>>(s.N, s.T, s.F, s.B, s.K, nslab, V, C, Jr,
                                                        Jinv, Rout, part);
  *n_parts = grid;
  return cudaGetLastError();
}

#define SC_INST(R)                                                                              \
  template cudaError_t launch_gain_prep<R>(const Shape&, const double*, int, R*, R*, uint32_t*, \
                                           cudaStream_t);                                       \
  template cudaError_t launch_residual_all<R>(const Shape&, const R*, const R*, const R*,       \
                                              const R*, R*, double*, int, int*, cudaStream_t);
SC_INST(float)
SC_INST(double)
#undef SC_INST

}  // namespace sc
