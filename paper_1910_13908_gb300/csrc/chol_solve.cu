// Triangular solves with one float32 factor on one thread-block cluster.
//
// The substitution is a chain of 2 nT dependent 64x64 tile-vector products,
// and what bounds it is the way from one product to the next: through global
// memory (k_chol_solve) a solved block takes a store, polled loads and three
// block barriers.  Here the blocks of a job are the CTAs of one cluster.  A
// solved block goes from the registers of the warps that formed it straight to
// the shared memory of every CTA, which holds a NaN pattern no instruction
// returns until then: the values are their own flags.  What is left per tile
// row, about 950 cycles, is half of the way from one block over the product
// before last (a product, a barrier, Linv_ii's product) and M's product, and
// the store to the next CTA.
//
// CTA c takes the tile rows c, c + NC, ... forward and then the same rows
// backward.  Three groups of warps:
//   warps 0..7    the substitution, one row at a time, with the products, the
//                 orders of their sums and the roundings of k_chol_solve;
//   warps 8..15   the rows' M = Linv_ii L_{i,i-1} (forward) and
//                 N = L_{i+1,i} Linv_ii (backward), up to kSlots rows ahead;
//   warps 16..19  the copies of the tiles, in the order of their use.
//
// k_chol_solve -> here, us a solve: order 200 16.6 -> 14.5, 512 23.9 -> 18.3,
// 1024 34.7 -> 26.4, 1600 46.4 -> 43.5, 2408 66 -> 74, 4096 104 -> 160: sixteen
// SMs stream the tiles of the large orders more slowly than all of them, so
// the cluster takes up to kMaxRows tile rows.
#include <atomic>

#include "chol_tiles.cuh"

namespace sc {

namespace {

constexpr int kChain = 256, kBuild = 256, kCopy = 128;  // threads of the three groups
constexpr int kThreads = kChain + kBuild + kCopy;
constexpr int kSlots = 3;     // (Linv_ii, M or N) pairs in flight
constexpr int kRing = 4;      // streamed tiles in flight
constexpr int kMaxRows = 24;  // tile rows up to which the cluster is the faster way
constexpr int LD = Pitch<float>::value;
constexpr uint32_t kAbsent = 0xffffffffu;  // a word of a block that has not come: a NaN no instruction returns
constexpr int kTile = kNB * LD;  // floats of a tile in shared memory

struct Bars {
  uint64_t loaded[kSlots], built[kSlots], freed[kSlots];
  uint64_t full[kRing], empty[kRing];
};

constexpr size_t kSmem = sizeof(float) * ((size_t)(2 * kSlots + kRing) * kTile + 2 * kMaxRows * kNB + 2 * kNB) + sizeof(Bars);

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("{\n .reg .b64 s;\n mbarrier.arrive.shared::cta.b64 s, [%0];\n}\n" ::"r"(tc::saddr(bar)) : "memory");
}
// One arrival of `bar` once this thread's asynchronous copies so far have landed.
__device__ __forceinline__ void copies_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(tc::saddr(bar)) : "memory");
}
// The four values of a half-warp to every CTA, first to the one of row `next`,
// which is waiting for them.
__device__ __forceinline__ void send_block(float* dst, int next, int NC, float4 v) {
  auto word = [](float f) { return __float_as_uint(f) == kAbsent ? 0x7fffffffu : __float_as_uint(f); };  // any NaN
  const int l = threadIdx.x & 15, cta = (next + l) & (NC - 1);
  uint32_t d;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(tc::saddr(dst)), "r"(cta));
  auto put = [&]() {
    asm volatile("st.relaxed.cluster.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(d), "r"(word(v.x)),
                 "r"(word(v.y)), "r"(word(v.z)), "r"(word(v.w))
                 : "memory");
  };
  if (l == 0) put();
  __syncwarp();
  if (l > 0 && l < NC) put();
}
// Bounded wait of a warp for all 64 values of a block, two a lane.
__device__ __forceinline__ void block_wait(const float* y, bool& ok) {
  const uint32_t a = tc::saddr(y + 2 * (threadIdx.x & 31));
  for (long it = 0; ok; ++it) {
    uint32_t u, v;
    asm volatile("ld.relaxed.cluster.shared::cta.v2.b32 {%0, %1}, [%2];" : "=r"(u), "=r"(v) : "r"(a) : "memory");
    if (__all_sync(0xffffffffu, u != kAbsent && v != kAbsent)) break;
    if (it >= kSpinLimit) ok = false;
    if (it >= 4096) __nanosleep(64);
  }
  __syncwarp();
}
// Bounded wait of a warp for phase `parity` of a barrier; after one wait has
// run out the warp waits no more.
__device__ __forceinline__ void bar_wait(uint64_t* bar, uint32_t parity, bool& ok) {
  if (ok) ok = __all_sync(0xffffffffu, tc::mbar_wait(bar, parity));
  __syncwarp();
}
__device__ __forceinline__ void chain_bar() { asm volatile("bar.sync 1, %0;" ::"n"(kChain) : "memory"); }
__device__ __forceinline__ void build_bar() { asm volatile("bar.sync 2, %0;" ::"n"(kBuild) : "memory"); }

// mv_rows with the thread's part of the tile already in registers.
struct RowPart {
  float4 t[4];
};
__device__ __forceinline__ RowPart row_part(const float* Tm) {
  const int r = threadIdx.x >> 2, part = threadIdx.x & 3, rot = 3 * (r & 1);
  RowPart p;
#pragma unroll
  for (int u = 0; u < 4; ++u) p.t[u] = *reinterpret_cast<const float4*>(Tm + r * LD + 4 * ((part + 4 * u + rot) & 15));
  return p;
}
__device__ __forceinline__ float mv_row_part(const RowPart& p, const float* v) {
  const int r = threadIdx.x >> 2, part = threadIdx.x & 3, rot = 3 * (r & 1);
  float s = 0.f;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const float4 w = *reinterpret_cast<const float4*>(v + 4 * ((part + 4 * u + rot) & 15)), t = p.t[u];
    s = fmaf(t.x, w.x, fmaf(t.y, w.y, fmaf(t.z, w.z, fmaf(t.w, w.w, s))));
  }
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  return s;
}

// mv_cols likewise.  Every sum has mv_cols' order, but a lane keeps two and
// then one of its four sums through the butterfly (5 shuffles, not 16): lane
// e of group g ends with entry 4 g + col_entry(e).
__device__ __forceinline__ int col_entry(int e) { return 2 * (e & 1) + (e >> 1 & 1); }
struct ColPart {
  float4 t[4];
};
__device__ __forceinline__ ColPart col_part(const float* Tm) {
  const int g = threadIdx.x >> 4, mr = threadIdx.x & 15;
  ColPart p;
#pragma unroll
  for (int k = 0; k < 4; ++k) p.t[k] = *reinterpret_cast<const float4*>(Tm + (mr + 16 * k) * LD + 4 * g);
  return p;
}
__device__ __forceinline__ float mv_col_part(const ColPart& p, const float* v) {
  const int mr = threadIdx.x & 15;
  float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float w = v[mr + 16 * k];
    a0 = fmaf(p.t[k].x, w, a0), a1 = fmaf(p.t[k].y, w, a1), a2 = fmaf(p.t[k].z, w, a2), a3 = fmaf(p.t[k].w, w, a3);
  }
  const bool b0 = mr & 1, b1 = mr & 2;
  float c0 = b0 ? a2 : a0, c1 = b0 ? a3 : a1;
  c0 += __shfl_xor_sync(0xffffffffu, b0 ? a0 : a2, 1);
  c1 += __shfl_xor_sync(0xffffffffu, b0 ? a1 : a3, 1);
  float d = b1 ? c1 : c0;
  d += __shfl_xor_sync(0xffffffffu, b1 ? c0 : c1, 2);
  d += __shfl_xor_sync(0xffffffffu, d, 4);
  d += __shfl_xor_sync(0xffffffffu, d, 8);
  return d;
}

// C = A B of 64x64 tiles by the kBuild threads, 4x4 outputs each, every sum
// in ascending order of the contraction index; C may be A or B.
__device__ __forceinline__ void build_product(float* C, const float* A, const float* B) {
  const int t = threadIdx.x - kChain, tx = t & 15, ty = t >> 4;
  float acc[4][4] = {};
#pragma unroll 2
  for (int m = 0; m < kNB; m += 4) {
    float4 a[4], b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) a[u] = *reinterpret_cast<const float4*>(A + (ty + 16 * u) * LD + m);
#pragma unroll
    for (int e = 0; e < 4; ++e) b[e] = *reinterpret_cast<const float4*>(B + (m + e) * LD + 4 * tx);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float av[4] = {a[u].x, a[u].y, a[u].z, a[u].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        acc[u][0] = fmaf(av[e], b[e].x, acc[u][0]);
        acc[u][1] = fmaf(av[e], b[e].y, acc[u][1]);
        acc[u][2] = fmaf(av[e], b[e].z, acc[u][2]);
        acc[u][3] = fmaf(av[e], b[e].w, acc[u][3]);
      }
    }
  }
  build_bar();  // every thread has read A and B
#pragma unroll
  for (int u = 0; u < 4; ++u)
    *reinterpret_cast<float4*>(C + (ty + 16 * u) * LD + 4 * tx) =
        make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
}

// The rows of CTA c in the order it takes them: q = 0..R-1 forward,
// ascending, q = R..2R-1 backward, descending.
struct Row {
  int i, crit, other;  // tile row; row of the block that arrives last, or -1; tiles before it
  bool fwd;
};
__device__ __forceinline__ Row row_of(int q, int R, int c, int NC, int nT) {
  Row w;
  w.fwd = q < R;
  w.i = c + NC * (w.fwd ? q : 2 * R - 1 - q);
  w.crit = w.fwd ? w.i - 1 : (w.i + 1 < nT ? w.i + 1 : -1);
  w.other = w.crit < 0 ? 0 : w.fwd ? w.i - 1 : nT - 2 - w.i;
  return w;
}

}  // namespace

__global__ void __launch_bounds__(kThreads, 1) k_chol_solve_cluster(const float* __restrict__ A, int lda, int nT,
                                                                    const float* __restrict__ Linv,
                                                                    const double* __restrict__ b,
                                                                    double* __restrict__ x, int accumulate,
                                                                    uint32_t* status, const LMState* lm, size_t js) {
  dep_sync(js == 0);
  const int NC = gridDim.x, c = blockIdx.x, job = blockIdx.y;  // one cluster per job
  lm = job_ptr(lm, js, job);
  if (lm != nullptr && (lm->done | lm->notpd)) return;  // the whole cluster alike
  A = job_ptr(A, js, job);
  Linv = job_ptr(Linv, js, job);
  b = job_ptr(b, js, job);
  x = job_ptr(x, js, job);
  status = job_ptr(status, js, job);

  extern __shared__ __align__(16) unsigned char smraw[];
  float* slot = reinterpret_cast<float*>(smraw);       // [kSlots][2] tiles: Linv_ii, then L tile -> M or N
  float* ring = slot + 2 * kSlots * kTile;             // [kRing] tiles
  float* Y = ring + kRing * kTile;                     // [kMaxRows][64] forward blocks
  float* X = Y + kMaxRows * kNB;                       // [kMaxRows][64] backward blocks
  float* vin = X + kMaxRows * kNB;                     // [2][64]
  Bars* bar = reinterpret_cast<Bars*>(vin + 2 * kNB);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int R = c < nT ? (nT - 1 - c) / NC + 1 : 0;

  for (int k = tid; k < kSlots; k += kThreads) {
    tc::mbar_init(&bar->loaded[k], kCopy);
    tc::mbar_init(&bar->built[k], kBuild / 32);
    tc::mbar_init(&bar->freed[k], kChain / 32);
  }
  for (int k = tid; k < kRing; k += kThreads) {
    tc::mbar_init(&bar->full[k], kCopy);
    tc::mbar_init(&bar->empty[k], kChain / 32);
  }
  for (int k = tid; k < nT * kNB; k += kThreads) {
    reinterpret_cast<uint32_t*>(Y)[k] = kAbsent;
    reinterpret_cast<uint32_t*>(X)[k] = kAbsent;
  }
  // every CTA's barriers and blocks are ready before any block is sent
  asm volatile("barrier.cluster.arrive;\n barrier.cluster.wait;" ::: "memory");

  // After a wait that ran out (ok), a group goes on without waiting: every
  // thread meets every barrier, and the kernel ends.
  bool ok = true;
  if (warp < kChain / 32) {
    // ---- the substitution ----
    // Every part of a tile is in registers before the block it meets is
    // waited for: between two blocks lie one product, its shuffles and the
    // way to the next CTA.
    int rk = 0;  // streamed tiles consumed
    auto next_tile = [&]() -> const float* {
      bar_wait(&bar->full[rk % kRing], (rk / kRing) & 1, ok);
      return ring + (rk % kRing) * kTile;
    };
    auto done_tile = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar->empty[rk % kRing]);
      ++rk;
    };
    int q = 0;
    for (; q < R; ++q) {  // forward: quad r = tid / 4 owns entry r
      const Row w = row_of(q, R, c, NC, nT);
      const int i = w.i, s = q % kSlots, h = lane & 16;
      float acc = (float)b[i * kNB + (tid >> 2)];
      RowPart t, tinv, tm;
      auto slot_parts = [&]() {
        bar_wait(&bar->built[s], (q / kSlots) & 1, ok);
        tinv = row_part(slot + 2 * s * kTile);
        tm = row_part(slot + (2 * s + 1) * kTile);
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar->freed[s]);
      };
      for (int n = 0; n < w.other; ++n) {
        t = row_part(next_tile());
        done_tile();
        if (n == w.other - 1) slot_parts();
        block_wait(Y + n * kNB, ok);
        acc -= mv_row_part(t, Y + n * kNB);
      }
      if (w.other <= 0) slot_parts();
      float* vz = vin + (q & 1) * kNB;  // two rows later every thread has passed another barrier
      if ((tid & 3) == 0) vz[tid >> 2] = acc;
      chain_bar();
      float o = mv_row_part(tinv, vz);  // z = Linv_ii acc
      if (w.crit >= 0) {
        block_wait(Y + w.crit * kNB, ok);
        o -= mv_row_part(tm, Y + w.crit * kNB);
      }
      // rows 8 warp .. + 7, one per quad: lanes 16 h .. hold rows 4 h .. + 3
      float4 v;
      v.x = __shfl_sync(0xffffffffu, o, h);
      v.y = __shfl_sync(0xffffffffu, o, h + 4);
      v.z = __shfl_sync(0xffffffffu, o, h + 8);
      v.w = __shfl_sync(0xffffffffu, o, h + 12);
      send_block(Y + i * kNB + 8 * warp + (h >> 2), i + 1, NC, v);
    }
    for (; q < 2 * R; ++q) {  // backward: lane e of group tid / 16 owns entry `en`
      const Row w = row_of(q, R, c, NC, nT);
      const int i = w.i, s = q % kSlots, h = lane & 16, e = lane & 15, en = 4 * (tid >> 4) + col_entry(e);
      block_wait(Y + i * kNB, ok);
      float acc = Y[i * kNB + en];
      ColPart t, tinv, tm;
      auto slot_parts = [&]() {
        bar_wait(&bar->built[s], (q / kSlots) & 1, ok);
        tinv = col_part(slot + 2 * s * kTile);
        tm = col_part(slot + (2 * s + 1) * kTile);
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar->freed[s]);
      };
      for (int n = 0; n < w.other; ++n) {
        const float* xj = X + (nT - 1 - n) * kNB;
        t = col_part(next_tile());
        done_tile();
        if (n == w.other - 1) slot_parts();
        block_wait(xj, ok);
        acc -= mv_col_part(t, xj);
      }
      if (w.other <= 0) slot_parts();
      float* vz = vin + (q & 1) * kNB;
      if (e < 4) vz[en] = acc;
      chain_bar();
      float o = mv_col_part(tinv, vz);  // z = Linv_ii^T acc
      if (w.crit >= 0) {
        block_wait(X + w.crit * kNB, ok);
        o -= mv_col_part(tm, X + w.crit * kNB);
      }
      float4 v;
      v.x = __shfl_sync(0xffffffffu, o, h);
      v.y = __shfl_sync(0xffffffffu, o, h + 2);
      v.z = __shfl_sync(0xffffffffu, o, h + 1);
      v.w = __shfl_sync(0xffffffffu, o, h + 3);
      send_block(X + i * kNB + 4 * (tid >> 4), i + NC - 1, NC, v);
      if (e < 4 && ok) x[i * kNB + en] = accumulate ? x[i * kNB + en] + (double)o : (double)o;
    }
  } else if (warp < (kChain + kBuild) / 32) {
    // ---- M and N ----
    for (int q = 0; q < 2 * R; ++q) {
      const Row w = row_of(q, R, c, NC, nT);
      const int s = q % kSlots;
      float *Tinv = slot + 2 * s * kTile, *Tm = Tinv + kTile;
      bar_wait(&bar->loaded[s], (q / kSlots) & 1, ok);
      if (w.crit >= 0) {
        if (w.fwd) build_product(Tm, Tinv, Tm);
        else build_product(Tm, Tm, Tinv);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar->built[s]);
    }
  } else {
    // ---- copies: each instruction of the group takes eight rows of a tile ----
    auto tile = [&](float* dst, const float* src, int ld) {
      const int r = (tid - kChain - kBuild) >> 4, ch = 4 * (lane & 15);
#pragma unroll
      for (int u = 0; u < kNB; u += kCopy / 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::saddr(dst + (u + r) * LD + ch)),
                     "l"(src + (size_t)(u + r) * ld + ch)
                     : "memory");
    };
    auto tile_at = [&](int r, int col) { return A + (size_t)r * kNB * lda + (size_t)col * kNB; };
    int qs = 0, rk = 0;  // slots and streamed tiles issued
    auto fill_slot = [&]() {
      const Row w = row_of(qs, R, c, NC, nT);
      const int s = qs % kSlots;
      if (qs >= kSlots) bar_wait(&bar->freed[s], (qs / kSlots - 1) & 1, ok);
      if (!ok) return;
      float* Tinv = slot + 2 * s * kTile;
      tile(Tinv, Linv + (size_t)w.i * kNB * kNB, kNB);
      if (w.crit >= 0) tile(Tinv + kTile, w.fwd ? tile_at(w.i, w.crit) : tile_at(w.crit, w.i), lda);
      copies_arrive(&bar->loaded[s]);
      ++qs;
    };
    for (int q = 0; q < kSlots && q < 2 * R; ++q) fill_slot();
    for (int q = 0; q < 2 * R && ok; ++q) {
      const Row w = row_of(q, R, c, NC, nT);
      for (int n = 0; n < w.other; ++n, ++rk) {
        const int j = w.fwd ? n : nT - 1 - n, rs = rk % kRing;
        if (rk >= kRing) bar_wait(&bar->empty[rs], (rk / kRing - 1) & 1, ok);
        if (!ok) break;
        tile(ring + rs * kTile, w.fwd ? tile_at(w.i, j) : tile_at(j, w.i), lda);
        copies_arrive(&bar->full[rs]);
      }
      // the slot of the row before this one, whose tiles are all consumed by now or soon
      if (ok && q >= 1 && qs < 2 * R) fill_slot();
    }
    async_wait_all();  // no copy is in flight when the block ends
  }
  if (!ok) atomicOr(status, SC_STATUS_TIMEOUT);
  // no CTA's shared memory goes before every block sent to it has landed
  __syncwarp();
  asm volatile("barrier.cluster.arrive;\n barrier.cluster.wait;" ::: "memory");
}

namespace {
// Clusters of `nc` CTAs that are resident at once on the current device.
int resident_clusters(int nc) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nc, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nc;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaFuncSetAttribute(k_chol_solve_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem) != cudaSuccess ||
      cudaFuncSetAttribute(k_chol_solve_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, k_chol_solve_cluster, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}
}  // namespace

// 8 CTAs up to 8 tile rows, else 16 where the device takes such clusters (one
// row per CTA keeps a block's products ahead of the chain).  A batch goes to
// k_chol_solve once its clusters would not all be resident: its rows then fill
// the GPU without them.
//
// Beside other work a cluster is slow to start: it waits until 8 or 16 SMs of
// one GPC have 187 KB of shared memory free at the same time, while
// factorisations of other streams come and go, and launched early it keeps
// those SMs from them.  So a job whose factorisation the caller caps, which
// says that other jobs share the device, goes to k_chol_solve; jobs on 16
// streams, against clusters and against clusters launched the plain way: 32
// jobs of 64 stations 29 ms, 37 and 30, 24 of 128 stations 52, 89 and 61.  The
// bands of a consensus, which one host thread enqueues, leave SMs free: clusters
// there too, those of 16 CTAs launched the plain way.  16 bands of 128 stations
// and 10 clusters (16 CTAs) 221 ms, 296 launched early, 374 in k_chol_solve; of
// 64 stations and 12 clusters (8 CTAs) 228, 216 and 314.
int solve_cluster_size(int nT, int G, Beside beside) {
  if (beside == Beside::jobs || nT < 2 || nT > kMaxRows) return 0;
  // per device: 1 + the resident clusters of 8 and of 16 CTAs (0: not asked yet)
  constexpr int kDevs = 64;
  static std::atomic<int> cache[2][kDevs];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevs) return 0;
  auto resident = [&](int nc) {
    std::atomic<int>& v = cache[nc == 16][dev];
    if (v.load(std::memory_order_relaxed) == 0) v.store(1 + resident_clusters(nc), std::memory_order_relaxed);
    return v.load(std::memory_order_relaxed) - 1;
  };
  if (nT > 8 && resident(16) >= G) return 16;
  return resident(8) >= G ? 8 : 0;
}

cudaError_t launch_chol_solve_cluster(const float* A, int lda, int nT, int nc, const float* Linv, const double* b,
                                      double* x, int accumulate, uint32_t* status, const LMState* lm, cudaStream_t st,
                                      bool early, const Batch& bt) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nc, bt.G, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nc;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_dep
  at[1].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k_chol_solve_cluster, A, lda, nT, Linv, b, x, accumulate, status, lm, bt.js);
}

}  // namespace sc
