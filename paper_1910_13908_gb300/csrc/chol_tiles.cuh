// Pieces shared by the factorisation and solve kernels (cholesky.cu, chol_solve.cu,
// chol_f64.cu): the counters of the task graph and the bounded waits on
// them, 64x64 tile moves and products, and the factorisation of a diagonal
// tile by one block.
#pragma once

#include <type_traits>

#include "sc_common.cuh"

namespace sc {

enum TaskType { T_POTRF = 0, T_TRSM = 1, T_UPD = 2, T_FWD = 3, T_BWD = 4 };

// sync area (ints): [0] factor task counter, [1] solve task counter (during a
// factorisation LeaveWalkerSm's word), upd[nT*nT], potrf_done[nT],
// trsm_done[nT*nT].  The solves pass their blocks as tagged words instead.
struct SyncView {
  int* fctr;
  int* sctr;
  int* upd;
  int* pdone;
  int* tdone;
  __host__ __device__ SyncView(int* s, int nT)
      : fctr(s), sctr(s + 1), upd(s + 2), pdone(s + 2 + nT * nT), tdone(s + 2 + nT * nT + nT) {}
};

// ---- synchronisation primitives -----------------------------------------------------------

constexpr long kSpinLimit = 1L << 22;  // ~1 s of polling with the back-off below

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Publishes a counter.  Callers reach it through a __syncthreads() after
// the block's stores of the tile; a release store is cumulative, so those
// stores of every thread of the block become visible before the counter.
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_status(const uint32_t* p) {
  return *reinterpret_cast<const volatile uint32_t*>(p);
}

__device__ __forceinline__ int ld_relaxed(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Waits until *p >= v (the counters only grow).  The first read is an
// acquire load, which settles the common case of a dependency finished long
// ago in one round trip.  Otherwise it polls with relaxed loads (an acquire
// load on every poll would invalidate this SM's L1 each time and stall the
// load/store path of the other CTAs sharing the SM) and confirms with one
// acquire load once the value is seen.  An acquire load, unlike a fence,
// does not wait for this thread's earlier stores and atomics to complete.
// Gives up (returns false) after kSpinLimit polls or as soon as another
// CTA has recorded a timeout.
static __device__ bool wait_ge(const int* p, int v, uint32_t* status) {
  if (ld_acquire(p) >= v) return true;
  for (long it = 0; it < kSpinLimit; ++it) {
    __nanosleep(it < 16 ? 32 : 200);
    if (ld_relaxed(p) >= v) return ld_acquire(p) >= v;
    if ((it & 63) == 63 && (ld_status(status) & SC_STATUS_TIMEOUT)) return false;
  }
  atomicOr(status, SC_STATUS_TIMEOUT);
  return false;
}

// Blocks of a factorisation that share the walker's SM leave it to the
// walker, which runs the critical path.  Not all of them may: every block can
// land on that SM (the caller caps them to a few; or kernels of other streams
// hold the rest of the GPU, and queued blocks come in one after another
// through the slot the last one left), and the walker waits for tasks that
// the others run.  So at most half of them leave, which is more than ever
// share an SM with the walker when the blocks fill the GPU.
__host__ __device__ constexpr int max_leavers(int blocks) { return (blocks - 1) / 2; }
// Asked by one thread of a block before each claim.  `word`, the solve counter,
// idle during a factorisation: the walker's SM + 1 (low half, stored once by
// the walker) and the blocks that have asked to leave (high half).
struct LeaveWalkerSm {
  int state = 0;  // 1 stays, 2 leaves, 0 not known yet
  __device__ __forceinline__ static int sm() {
    int v;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(v));
    return v;
  }
  __device__ __forceinline__ static void publish(int* word) { st_release(word, sm() + 1); }
  __device__ __forceinline__ bool ask(int* word, int blocks) {
    if (state == 0) {
      const int w = ld_relaxed(word) & 0xffff;
      if (w != 0) state = w == sm() + 1 && (atomicAdd(word, 1 << 16) >> 16) < max_leavers(blocks) ? 2 : 1;
    }
    return state == 2;
  }
};

// mbarriers in shared memory
namespace tc {

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(saddr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for phase `parity` of an mbarrier; false after kSpinLimit
// polls.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  for (long it = 0; it < kSpinLimit; ++it) {
    if (mbar_test(bar, parity)) return true;
    if (it >= 8) __nanosleep(64);
  }
  return false;
}

}  // namespace tc

// ---- tile helpers --------------------------------------------------------------------------

// Shared-memory row pitch: 64 elements + 16 bytes, so that rows stay 16-byte
// aligned for vector loads and consecutive rows start 4 banks apart.
template <typename R>
struct Pitch {
  static constexpr int value = kNB + 16 / (int)sizeof(R);
};

// 64x64 tile moves between global memory (through L2 only) and shared
// memory in 16-byte vectors: each thread issues 4 (float) or 8 (double)
// independent requests instead of 16.
template <typename R>
__device__ __forceinline__ void load_tile(R* sm, const R* g, int lda) {
  constexpr int LD = Pitch<R>::value;
  constexpr int V = 16 / (int)sizeof(R);  // elements per vector
  constexpr int PER_ROW = kNB / V;
  for (int e = threadIdx.x; e < kNB * PER_ROW; e += blockDim.x) {
    int r = e / PER_ROW, c = (e - r * PER_ROW) * V;
    float4 v = __ldcg(reinterpret_cast<const float4*>(g + (size_t)r * lda + c));
    *reinterpret_cast<float4*>(sm + r * LD + c) = v;
  }
}
// The same copy issued as 16-byte cp.async requests (L2 only); the caller
// commits the group.
template <typename R>
__device__ __forceinline__ void copy_tile_async(R* sm, const R* g, int lda) {
  constexpr int LD = Pitch<R>::value;
  constexpr int PER_ROW = kNB * (int)sizeof(R) / 16;
  for (int e = threadIdx.x; e < kNB * PER_ROW; e += blockDim.x) {
    int r = e / PER_ROW, ch = e - r * PER_ROW;
    const char* src = reinterpret_cast<const char*>(g + (size_t)r * lda) + 16 * ch;
    unsigned dst = (unsigned)__cvta_generic_to_shared(reinterpret_cast<char*>(sm + r * LD) + 16 * ch);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  }
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void async_wait_prev() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

template <typename R>
__device__ __forceinline__ void store_tile(R* g, int lda, const R* sm) {
  constexpr int LD = Pitch<R>::value;
  constexpr int V = 16 / (int)sizeof(R);
  constexpr int PER_ROW = kNB / V;
  for (int e = threadIdx.x; e < kNB * PER_ROW; e += blockDim.x) {
    int r = e / PER_ROW, c = (e - r * PER_ROW) * V;
    __stcg(reinterpret_cast<float4*>(g + (size_t)r * lda + c), *reinterpret_cast<const float4*>(sm + r * LD + c));
  }
}

// acc[a][b] = sum_m X[ty+16a][m] Y[tx+16b][m]   (X Y^T on 64x64 tiles); the
// contraction index is contiguous in both operands, so each thread reads
// 16-byte vectors along it.
__device__ __forceinline__ void gemm_nt(float acc[4][4], const float* X, const float* Y) {
  constexpr int L = Pitch<float>::value;
  int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
#pragma unroll
  for (int m = 0; m < kNB; m += 4) {
    float4 x[4], y[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) x[a] = *reinterpret_cast<const float4*>(X + (ty + 16 * a) * L + m);
#pragma unroll
    for (int b = 0; b < 4; ++b) y[b] = *reinterpret_cast<const float4*>(Y + (tx + 16 * b) * L + m);
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        float t = acc[a][b];
        t = fmaf(x[a].x, y[b].x, t);
        t = fmaf(x[a].y, y[b].y, t);
        t = fmaf(x[a].z, y[b].z, t);
        t = fmaf(x[a].w, y[b].w, t);
        acc[a][b] = t;
      }
  }
}

// Reciprocal of an elimination pivot: the hardware approximation (relative
// error below 2^-22).
__device__ __forceinline__ float pivot_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Compile-time loops: every step below is instantiated with constant
// indices, so the per-lane rows stay in registers.
template <int I, int N>
struct Static {
  template <typename F>
  __device__ __forceinline__ static void each(F&& f) {
    f(std::integral_constant<int, I>());
    Static<I + 1, N>::each(f);
  }
};
template <int N>
struct Static<N, N> {
  template <typename F>
  __device__ __forceinline__ static void each(F&&) {}
};

// gemm_nt restricted to the terms that can be nonzero, for the walker's
// chain products:
//   TRI_Y: Y is lower triangular (Y[c][m] = 0 for m > c, as Linv_jj is
//          stored), so output column block b sums only m < 16 (b + 1);
//   SYM:   X Y^T is symmetric and only its lower part is read, so only the
//          16x16 blocks a >= b are formed (the others are left unset).
// The skipped terms are exact zeros, and the kept ones are added in gemm_nt's
// order, so every formed entry has gemm_nt's value.
template <bool TRI_Y, bool SYM>
__device__ __forceinline__ void gemm_nt_part(float acc[4][4], const float* X, const float* Y) {
  constexpr int L = Pitch<float>::value;
  int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
  Static<0, 4>::each([&](auto mc_) {  // contraction chunk m = 16 mc .. 16 mc + 15
    constexpr int mc = decltype(mc_)::value;
#pragma unroll
    for (int m = 16 * mc; m < 16 * mc + 16; m += 4) {
      float4 x[4], y[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) x[a] = *reinterpret_cast<const float4*>(X + (ty + 16 * a) * L + m);
      Static<0, 4>::each([&](auto b_) {
        constexpr int b = decltype(b_)::value;
        if constexpr (!TRI_Y || b >= mc) y[b] = *reinterpret_cast<const float4*>(Y + (tx + 16 * b) * L + m);
      });
      Static<0, 4>::each([&](auto a_) {
        constexpr int a = decltype(a_)::value;
        Static<0, 4>::each([&](auto b_) {
          constexpr int b = decltype(b_)::value;
          if constexpr ((!TRI_Y || b >= mc) && (!SYM || a >= b)) {
            float t = acc[a][b];
            t = fmaf(x[a].x, y[b].x, t);
            t = fmaf(x[a].y, y[b].y, t);
            t = fmaf(x[a].z, y[b].z, t);
            t = fmaf(x[a].w, y[b].w, t);
            acc[a][b] = t;
          }
        });
      });
    }
  });
}

// 16 consecutive values at a 16-byte aligned shared-memory address.
__device__ __forceinline__ void ld16(const float* p, float (&v)[16]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    float4 t = reinterpret_cast<const float4*>(p)[u];
    v[4 * u] = t.x;
    v[4 * u + 1] = t.y;
    v[4 * u + 2] = t.z;
    v[4 * u + 3] = t.w;
  }
}
__device__ __forceinline__ void st16(float* p, const float (&v)[16]) {
#pragma unroll
  for (int u = 0; u < 4; ++u)
    reinterpret_cast<float4*>(p)[u] = make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
}

// In-place Cholesky of the 64x64 SPD tile in sm (pitch of the tile, lower
// part read), writing L (upper part zeroed) to sm and L^-1 to sv
// (potrf_tile_w below).
//
// Gaussian elimination in LDL^T form over the rows of [A | Y], Y = I at the
// start, W columns per step.  With A = L' D L'^T (L' unit lower,
// D = diag(p)), L = L' D^1/2 and L^-1 = D^-1/2 L'^-1; the elimination turns
// Y into L'^-1.  Step k eliminates columns K = k..k+W-1 at once: with
// V = A[:, K] and Z = Y[K, :] as they stand before the step, and the W x W
// pivot block V[K, :] = L_D P L_D^T factorised by every thread, row i gets
//   u_i = V[i, :] L_D^-T          (A[i][k+m] at step k+m: final for column k+m)
//   g_i[m] = u_i[m] / p_m         (zero unless i > k+m)
//   c_i = g_i L_D^-1
//   A[i][j] -= c_i . V[j, :]      (j > k+W-1)
//   Y[i][:] -= c_i . Z            (equals the W single-column steps)
// Afterwards L[i][j] = A[i][j] / sqrt(p_j) for j < i, L[j][j] = sqrt(p_j),
// (L^-1)[i][c] = Y[i][c] / sqrt(p_i).  A non-positive pivot is replaced by
// 1 and sets *bad.
//
// Thread layout: warp w owns column block q = w % 4 (columns 16q..16q+15)
// of rows 32 (w / 4) .. +31, one row per lane, 16 entries of A and 16 of Y
// in registers.  Each step reads the published columns K of A and rows K of
// Y from shared memory (double-buffered, one barrier per step); the owners
// of the next W columns and rows publish them.  Once k >= 32 the rows 0..31
// are final (their multipliers c are zero), so their warps skip the row
// work and only take part in the pivots and the barriers; warp w runs on
// scheduler w % 4 of the SM, so each scheduler keeps one working warp.
template <typename R>
__device__ __forceinline__ R pivot_guard(R p, int* bad) {
  if (!(p > (R)0)) {
    if (threadIdx.x == 0) *bad = 1;
    return (R)1;
  }
  return p;
}

// Columns per elimination step of potrf_tile.  8 halves the steps (and
// barriers) of 4, each a longer chain of pivots; measured at order 4096 on
// GB300 it was no faster (1237 against 1233 us per factorisation), so 4.
#ifndef SC_POTRF_W
#define SC_POTRF_W 4
#endif

// The elimination above, W columns per step (W = 4 or 8).  The pivot
// block V[K, :] (W x W) is factorised by every thread in LDL^T form by
// right-looking elimination; a row's u, g and c follow the formulas above
// with W terms; the updates add the W rank-one terms in column order.
// aux: [2][W][64] published columns, [2][W][64] published rows of Y, [64]
// pivots (4 W 64 + 64 values).
template <int W, typename R>
__device__ void potrf_tile_w(R* sm, R* sv, R* aux, int* bad) {
  static_assert(W == 4 || W == 8, "4 or 8 columns per step");
  constexpr int LD = Pitch<R>::value;
  constexpr int S = 16 / W;  // steps per 16-column block
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int q = warp & 3, h = warp >> 2, i = 32 * h + lane, cb = 16 * q;
  R* colb = aux;               // [2][W][64]: colb[m][j] = A[j][k+m]
  R* rowb = aux + 2 * W * 64;  // [2][W][64]: rowb[m][c] = Y[k+m][c]
  R* piv = aux + 4 * W * 64;   // [64] pivots
  R a[16], y[16];
  ld16(sm + i * LD + cb, a);
  Static<0, 16>::each([&](auto tt) {
    constexpr int t = decltype(tt)::value;
    y[t] = (cb + t == i) ? (R)1 : (R)0;
  });
  if (q == 0) {
#pragma unroll
    for (int m = 0; m < W; ++m) colb[64 * m + i] = a[m];
  }
  if (i < W) st16(rowb + 64 * i + cb, y);
  __syncthreads();
  for (int kb = 0; kb < 4; ++kb) {
    Static<0, S>::each([&](auto kq_) {
      constexpr int kq = decltype(kq_)::value;
      constexpr int bsel = kq & 1;  // parity of the step index S kb + kq (S = 2 or 4, so S kb is even)
      constexpr int t0 = W * kq;    // first column of K inside block q == kb
      const int k = 16 * kb + t0;
      const R* col = colb + W * 64 * bsel;
      const R* row = rowb + W * 64 * bsel;
      R* coln = colb + W * 64 * (bsel ^ 1);
      R* rown = rowb + W * 64 * (bsel ^ 1);
      // pivot block E = V[K, :] (lower part), eliminated in place: L, p
      R E[W][W], L[W][W], p[W], r[W];
#pragma unroll
      for (int m = 0; m < W; ++m)
#pragma unroll
        for (int n = 0; n <= m; ++n) E[m][n] = col[64 * n + k + m];
#pragma unroll
      for (int n = 0; n < W; ++n) {
        p[n] = pivot_guard(E[n][n], bad);
        r[n] = pivot_rcp(p[n]);
#pragma unroll
        for (int m = n + 1; m < W; ++m) L[m][n] = E[m][n] * r[n];
#pragma unroll
        for (int m = n + 1; m < W; ++m)
#pragma unroll
          for (int o = n + 1; o <= m; ++o) E[m][o] = fma(-L[m][n], E[o][n], E[m][o]);
      }
      if (threadIdx.x == 0) {
#pragma unroll
        for (int m = 0; m < W; ++m) piv[k + m] = p[m];
      }
      // every row of this warp is at most k: c = 0, the row work is a no-op
      if (32 * h + 31 <= k) {
        __syncthreads();
        return;
      }
      // this row: u = V[i,:] L_D^-T, g = masked u / p, c = g L_D^-1
      R u[W], c[W];
#pragma unroll
      for (int m = 0; m < W; ++m) {
        u[m] = col[64 * m + i];
#pragma unroll
        for (int n = 0; n < m; ++n) u[m] = fma(-L[m][n], u[n], u[m]);
      }
#pragma unroll
      for (int m = W - 1; m >= 0; --m) {
        c[m] = i > k + m ? u[m] * r[m] : (R)0;
#pragma unroll
        for (int n = m + 1; n < W; ++n) c[m] = fma(-c[n], L[n][m], c[m]);
      }
      // A[i][j] -= c . V[j,:] for the columns j > k+W-1 of this block
      if (q >= kb) {
        if (q == kb) {
#pragma unroll
          for (int m = 0; m < W; ++m) a[t0 + m] = u[m];
        }
#pragma unroll
        for (int m = 0; m < W; ++m) {
          R v[16];
          ld16(col + 64 * m + cb, v);
          if (q > kb) {
            Static<0, 16>::each([&](auto tt) {
              constexpr int t = decltype(tt)::value;
              a[t] = fma(-c[m], v[t], a[t]);
            });
          } else {
            Static<t0 + W, 16>::each([&](auto tt) {
              constexpr int t = decltype(tt)::value;
              a[t] = fma(-c[m], v[t], a[t]);
            });
          }
        }
      }
      // Y[i][:] -= c . W; W[m][col] is zero right of column k+m
      if (q <= kb) {
#pragma unroll
        for (int m = 0; m < W; ++m) {
          R w[16];
          ld16(row + 64 * m + cb, w);
          Static<0, 16>::each([&](auto tt) {
            constexpr int t = decltype(tt)::value;
            y[t] = fma(-c[m], w[t], y[t]);
          });
        }
      }
      // publish the next W columns of A and rows of Y
      if (k + W < 64) {
        if constexpr (kq < S - 1) {
          if (q == kb) {
#pragma unroll
            for (int m = 0; m < W; ++m) coln[64 * m + i] = a[t0 + W + m];
          }
        } else {
          if (q == kb + 1) {
#pragma unroll
            for (int m = 0; m < W; ++m) coln[64 * m + i] = a[m];
          }
        }
        if (i >= k + W && i < k + 2 * W) st16(rown + 64 * (i - k - W) + cb, y);
      }
      __syncthreads();
    });
  }
  R pj[16];
  ld16(piv + cb, pj);
  const R ri = rsqrt(piv[i]);
  Static<0, 16>::each([&](auto tt) {
    constexpr int t = decltype(tt)::value;
    const int j = cb + t;
    const R rj = rsqrt(pj[t]);
    a[t] = j < i ? a[t] * rj : (j == i ? pj[t] * rj : (R)0);
    y[t] = j <= i ? y[t] * ri : (R)0;
  });
  st16(sm + i * LD + cb, a);
  st16(sv + i * LD + cb, y);
  __syncthreads();
}

template <typename R>
__device__ __forceinline__ void potrf_tile(R* sm, R* sv, R* aux, int* bad) {
  potrf_tile_w<SC_POTRF_W>(sm, sv, aux, bad);
}

// Tile-vector products on a 64x64 tile in shared memory (pitch 64 + 16
// bytes), laid out so that each quarter-warp's 16-byte loads hit all 32
// banks once.
//
// mv_rows: out[r] = sum_m T[r][m] v[m].  The quad of lanes 4r..4r+3 owns
// row r; lane `part` reads the row's 16-byte chunks part + 4u, rotated by
// three chunks on odd rows (odd rows start 4 banks further on, so the two
// rows of a quarter-warp then cover distinct banks).  Two shuffles combine
// the quad; every lane of it returns the row total.
__device__ __forceinline__ float mv_rows(const float* Tm, const float* v) {
  constexpr int LD = Pitch<float>::value;
  const int r = threadIdx.x >> 2, part = threadIdx.x & 3, rot = 3 * (r & 1);
  float s = 0.f;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int ch = (part + 4 * u + rot) & 15;
    const float4 t = *reinterpret_cast<const float4*>(Tm + r * LD + 4 * ch);
    const float4 w = *reinterpret_cast<const float4*>(v + 4 * ch);
    s = fmaf(t.x, w.x, fmaf(t.y, w.y, fmaf(t.z, w.z, fmaf(t.w, w.w, s))));
  }
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  return s;
}

// mv_cols: out[c] = sum_m T[m][c] v[m] for the columns c = 4g..4g+3 of lane
// group g = tid / 16.  Lane mr of the group takes rows m = mr + 16k: a
// quarter-warp reads eight consecutive rows (4 banks apart) at one column
// offset.  Four butterfly rounds combine the group; every lane of it
// returns the four totals.
template <typename R>
__device__ __forceinline__ void mv_cols(const R* Tm, const R* v, R (&o)[4]) {
  constexpr int LD = Pitch<R>::value;
  const int g = threadIdx.x >> 4, mr = threadIdx.x & 15;
  R a0 = 0, a1 = 0, a2 = 0, a3 = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int m = mr + 16 * k;
    const R* t = Tm + m * LD + 4 * g;
    const R w = v[m];
    const float4 q = *reinterpret_cast<const float4*>(t);
    a0 = fma((R)q.x, w, a0), a1 = fma((R)q.y, w, a1), a2 = fma((R)q.z, w, a2), a3 = fma((R)q.w, w, a3);
  }
#pragma unroll
  for (int d = 1; d < 16; d <<= 1) {
    a0 += __shfl_xor_sync(0xffffffffu, a0, d);
    a1 += __shfl_xor_sync(0xffffffffu, a1, d);
    a2 += __shfl_xor_sync(0xffffffffu, a2, d);
    a3 += __shfl_xor_sync(0xffffffffu, a3, d);
  }
  o[0] = a0, o[1] = a1, o[2] = a2, o[3] = a3;
}

}  // namespace sc
