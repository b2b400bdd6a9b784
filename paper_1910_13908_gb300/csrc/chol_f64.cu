// The float64 factorisation and solves (SC_FP64).
//
// Float64 runs at two FMAs a cycle per SM here, one warp instruction per 64
// cycles on each scheduler, whatever its number of active lanes, and that
// is also its latency.  So work is measured in warp instructions, and every
// one on the diagonal chain counts.  A 64x64 tile (131,000 cycles a product
// on one SM) is far too coarse for that: the chain of 64-wide panels took
// 210 us each.  Here tiles are 16x16, and the chain of a panel is 16 column
// steps of about 420 cycles (one reciprocal, one multiplier, one update
// instruction), a triangular product and a symmetric one.
//
// A job's blocks: one runs the diagonal chain (the walker), the
// others take tasks as they open:
//   P(i, j)     i >= j+2: L_ij = A_ij Linv_jj^T, then A_i,j+1 -= L_ij L_j+1,j^T
//   B(I, K, j)  the 32x32 block of tile rows 2I, 2I+1 and tile columns 2K,
//               2K+1: A_ik -= L_ij L_kj^T for its tiles with i >= k >= j+2
// P(., j) opens when POTRF(j) is published and the first column pair of
// B(., ., j-1), which holds column j+1, is claimed; B(., ., j) opens when
// P(., j) is wholly claimed; tasks are claimed panel by panel, in order.
// So every tile a claimed task waits for is written by a task claimed
// before it or by the walker, and the walker waits only for tasks that
// open once what it has published is published: some claimed task can
// always run, with one block beside the walker or more (the host launches two
// at least, and at most half of the others leave the walker's SM,
// LeaveWalkerSm).  Every wait is bounded and reports SC_STATUS_TIMEOUT.
//
// A batch of G jobs is one launch of G such sets of blocks.  A tile is
// formed by the same operations whichever block forms it, so a job's factor
// has the same bits alone and in a batch.
#include <algorithm>
#include <cstddef>

#include "chol_tiles.cuh"

namespace sc {

constexpr int kNB64 = 16;
// tiles a side of a float64 matrix padded to nT tiles of 64
static int tiles64(int nT) { return nT * (kNB / kNB64); }
int chol64_sync_ints(int nT) {
  const int n = tiles64(nT);
  return 2 + 2 * n * n + 3 * n;
}

namespace {

// The counters of SyncView, then the claim counters of the two kinds of task, one of each per panel.
struct Sync64 : SyncView {
  int *pclaim, *bclaim;
  __device__ Sync64(int* s, int n) : SyncView(s, n), pclaim(tdone + n * n), bclaim(pclaim + n) {}
};

constexpr int kThr = 128;            // compute threads of a block
constexpr int kBlock64 = kThr + 64;  // and the walker's loading and publishing warps

// named barriers: 1 the compute threads; the rest the walker's
enum { BAR_START = 2, BAR_LOADED = 3, BAR_STORED = 4 };  // BAR_STORED + 2 (j % 2): Linv_jj; + 1: L_j+1,j
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void csync() { bar_sync(1, kThr); }
__device__ __forceinline__ bool csync_and(bool v) {
  int r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n bar.red.and.pred q, 1, %2, p;\n selp.s32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((int)v), "r"(kThr)
      : "memory");
  return r != 0;
}
constexpr int kTurnBlocks = 16;  // blocks per job up to which the walkers' places go round
constexpr int kTLD = kNB64 + 2;  // row pitch of a tile in shared memory: consecutive rows start 4 banks apart

// ---- the 136 entries of a lower triangle on 128 threads ----------------------------------
//
// Rows p and 15 - p together hold 17 entries: the 16 threads 16p .. 16p+15
// take row 15 - p, then columns 0 .. p-1 of row p; (p, p) is left over.
__device__ __forceinline__ void tri_entry(int t, int& r, int& c) {
  const int p = t >> 4, q = t & 15;
  if (q < 16 - p) r = 15 - p, c = q;
  else r = p, c = q - (16 - p);
}

// u / p for a pivot p > 0.  The reciprocal is the hardware's approximation
// (about 2^-20) and one step of Halley's iteration, 1 / p = r / (1 - e) with
// e = 1 - p r, taken as r (1 + e + e^2): off by e^3, below the roundings.  The
// approximation flushes subnormal pivots and subnormal reciprocals to zero, so
// below 2^-1022 and from 2^1022 on both numbers are first scaled by a power of
// two (u <= sqrt(p A_rr) keeps the product in range; what underflows of u has
// an underflowing quotient).
__device__ __forceinline__ double over_pivot(double u, double p) {
  const unsigned field = (unsigned)(__double2hiint(p) >> 20);  // the biased exponent; on the bits, off the float64 pipe
  if (field - 1u >= 2044u) {
    if (field == 0x7ff) return u * 0.0;  // p infinite
    const double s = field == 0 ? 0x1p600 : 0x1p-600;
    u *= s;
    p *= s;
  }
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(p));
  const double e = fma(-p, r, 1.0);
  return u * fma(r, fma(e, e, e), r);
}

struct Potrf64 {
  double col[2][kNB64], row[2][kNB64];  // column k of A (rows >= k), row k of Y (columns < k)
  double piv[kNB64], rs[kNB64];
  double u[kNB64][kTLD];  // columns of L times the pivots
};

// POTRF of the 16x16 tile in sm (lower part): L to sm and L^-1 to sv, upper
// parts zeroed.  Gaussian elimination in LDL^T form with the inverse formed in
// the place of the columns that are done: at step k entry (r, c), r > k, is
// A[r][c] if c > k and Y[r][c] if c < k, and changes by -c_r times A[c][k] or
// Y[k][c], c_r = A[r][k] / p_k; at c = k it becomes Y[r][k] = -c_r.  One
// update instruction a step covers every entry.  True if a pivot was not
// positive.
__device__ bool potrf64(double* sm, double* sv, Potrf64& S) {
  const int t = threadIdx.x, pe = t >> 4;
  int r, c;
  tri_entry(t, r, c);
  const bool extra = (t & 15) == 0;  // this thread also has (pe, pe)
  double x = sm[r * kTLD + c], xe = extra ? sm[pe * kTLD + pe] : 0.0;
  bool bad = false;
  if (c == 0) S.col[0][r] = x;
  if (t == 0) S.col[0][0] = xe;
  csync();
  const int lane = t & 31, row_lane = (lane & 16) | (pe > 0 ? 16 - pe : 0);  // a lane with an entry of row pe
#pragma unroll 1
  for (int k = 0; k < kNB64; ++k) {
    const double *col = S.col[k & 1], *row = S.row[k & 1];
    double *coln = S.col[(k + 1) & 1], *rown = S.row[(k + 1) & 1];
    double p = col[k];
    const double ur = col[r], val = c > k ? col[c] : c < k ? row[c] : 1.0;
    // p > 0 on the bits: a float64 comparison would take the float64 pipe's 64 cycles
    if ((unsigned long long)(__double_as_longlong(p) - 1) >= 0x7ff0000000000000ull) {
      p = 1.0;
      bad = true;
    }
    const double cr = over_pivot(ur, p);
    const double ce = __shfl_sync(0xffffffffu, cr, row_lane);
    if (c == k && r > k) {
      S.u[r][k] = ur;
      x = 0.0;
    }
    if (r > k) x = fma(-cr, val, x);
    if (extra && pe > k) xe = fma(-ce, col[pe], xe);
    if (t == 0) S.piv[k] = p;
    // the next column and row
    if (c == k + 1) coln[r] = x;
    if (extra && pe == k + 1) coln[pe] = xe;
    if (r == k + 1 && c <= k) rown[c] = x;
    csync();
  }
  if (t < kNB64) S.rs[t] = rsqrt(S.piv[t]);
  csync();
  // (r, c), r > c, except that row 15 - p also holds its diagonal entry
  if (r > c) {
    sm[r * kTLD + c] = S.u[r][c] * S.rs[c];
    sv[r * kTLD + c] = x * S.rs[r];
    sm[c * kTLD + r] = 0.0;
    sv[c * kTLD + r] = 0.0;
  } else {
    sm[r * kTLD + r] = S.piv[r] * S.rs[r];
    sv[r * kTLD + r] = S.rs[r];
  }
  if (extra) {
    sm[pe * kTLD + pe] = S.piv[pe] * S.rs[pe];
    sv[pe * kTLD + pe] = S.rs[pe];
  }
  csync();
  return bad;
}

// ---- tile products ---------------------------------------------------------------------------
//
// Thread t has row t / 8 and columns t % 8 and t % 8 + 8 of a tile; operands
// are read along the contraction index in 16-byte vectors.

__device__ __forceinline__ double2 ldd2(const double* p) { return *reinterpret_cast<const double2*>(p); }

// acc = X Y^T on row-major tiles; Y lower triangular if TRI (the terms left
// out are exact zeros).  An update sums its panel's products from zero and
// subtracts once: one rounding at the size of the matrix per panel, not per
// term.
template <bool TRI>
__device__ __forceinline__ void product64(double (&acc)[2], const double* X, const double* Y) {
  acc[0] = acc[1] = 0.0;
  const double *x = X + (threadIdx.x >> 3) * kTLD, *y0 = Y + (threadIdx.x & 7) * kTLD, *y1 = y0 + 8 * kTLD;
#pragma unroll
  for (int m = 0; m < kNB64; m += 2) {
    const double2 xv = ldd2(x + m);
    if (!TRI || m < 8) {
      const double2 v = ldd2(y0 + m);
      acc[0] = fma(xv.y, v.y, fma(xv.x, v.x, acc[0]));
    }
    const double2 v = ldd2(y1 + m);
    acc[1] = fma(xv.y, v.y, fma(xv.x, v.x, acc[1]));
  }
}

// a 16x16 tile between global (through L2) and shared memory, 16 bytes a thread
__device__ __forceinline__ void tile_in(double* sm, const double* g, size_t lda) {
  const int r = threadIdx.x >> 3, c = 2 * (threadIdx.x & 7);
  *reinterpret_cast<double2*>(sm + r * kTLD + c) = __ldcg(reinterpret_cast<const double2*>(g + r * lda + c));
}
__device__ __forceinline__ void tile_out(double* g, size_t lda, const double* sm) {
  const int r = threadIdx.x >> 3, c = 2 * (threadIdx.x & 7);
  __stcg(reinterpret_cast<double2*>(g + r * lda + c), ldd2(sm + r * kTLD + c));
}

// ---- tasks --------------------------------------------------------------------------------------

// Panel j of n tiles: n - 2 - j tasks P; B for column pairs K from (j + 2) / 2 and rows pairs I >= K.
__host__ __device__ __forceinline__ int p_count64(int n, int j) { return n - 2 - j; }
__host__ __device__ __forceinline__ int b_first64(int n, int j) { return n / 2 - (j + 2) / 2; }
__host__ __device__ __forceinline__ int b_count64(int n, int j) {
  const int m = b_first64(n, j);
  return m * (m + 1) / 2;
}
// B task idx of panel j: pairs (I, K), column pair by column pair
__device__ __forceinline__ void b_task64(int n, int j, int idx, int& I, int& K) {
  const int m = b_first64(n, j);
  // pairs before x hold x m - x (x - 1) / 2 tasks
  const float h = m + 0.5f;
  int x = (int)(h - sqrtf(fmaxf(h * h - 2.0f * (float)idx, 0.f)));
  if (x < 0) x = 0;
  if (x > m - 1) x = m - 1;
  while (x > 0 && x * m - x * (x - 1) / 2 > idx) --x;
  while (x + 1 < m && (x + 1) * m - (x + 1) * x / 2 <= idx) ++x;
  K = (j + 2) / 2 + x;
  I = K + (idx - (x * m - x * (x - 1) / 2));
}

struct Claim {
  int kind;  // 0: P(i, j), 1: B(I, K, j), -1: none left, -2: gave up
  int i, K, j;
};

// by one warp: claims the next open task, of panel jp on (P) or jb on (B)
__device__ Claim claim64(int n, const Sync64& sv, uint32_t* status, int& jp, int& jb) {
  const int lane = threadIdx.x & 31, jend = n - 2;
  for (long it = 0;; ++it) {
    int v = 1;
    if (lane == 0 && jp < jend) v = ld_relaxed(sv.pdone + jp);
    if (lane == 1 && jp < jend && jp > 0) v = ld_relaxed(sv.bclaim + jp - 1) >= b_first64(n, jp - 1);
    if (lane == 2 && jb < jend) v = ld_relaxed(sv.pclaim + jb) >= p_count64(n, jb);
    const unsigned open = __ballot_sync(0xffffffffu, v);
    int idx = 0;
    if (jp < jend && (open & 3) == 3) {
      if (lane == 0) idx = atomicAdd(sv.pclaim + jp, 1);
      idx = __shfl_sync(0xffffffffu, idx, 0);
      if (idx < p_count64(n, jp)) return {0, jp + 2 + idx, 0, jp};
      ++jp;
      continue;
    }
    if (jb < jend && (open & 4)) {
      if (lane == 0) idx = atomicAdd(sv.bclaim + jb, 1);
      idx = __shfl_sync(0xffffffffu, idx, 0);
      if (idx < b_count64(n, jb)) {
        Claim c{1, 0, 0, jb};
        b_task64(n, jb, idx, c.i, c.K);
        return c;
      }
      ++jb;
      continue;
    }
    if (jp >= jend && jb >= jend) return {-1, 0, 0, 0};
    __nanosleep(40);
    int stop = 0;
    if (lane == 0 && (it & 63) == 63) {
      stop = (ld_status(status) & SC_STATUS_TIMEOUT) != 0;
      if (it > kSpinLimit / 4) {
        atomicOr(status, SC_STATUS_TIMEOUT);
        stop = 1;
      }
    }
    if (__shfl_sync(0xffffffffu, stop, 0)) return {-2, 0, 0, 0};
  }
}

// The diagonal chain of one job; its SM is left to it (see k_chol64).  The
// compute warps factorise and multiply.  One more warp fetches the next two
// tiles while the diagonal tile is factorised, and another publishes: a
// release store waits about 1000 cycles for the stores before it.  Neither
// uses the float64 pipes.  A barrier is arrived at again two panels on, by
// when BAR_START has shown that its waiters have passed it.
struct Walker64 {
  double diag[2][kNB64 * kTLD];  // A_jj (buffer j % 2) and A_j+1,j+1
  double linv[kNB64 * kTLD], panel[kNB64 * kTLD];
  Potrf64 S;
  int ok, failed;
};
__device__ void walker64_loads(const double* A, size_t lda, int n, const Sync64& sv, uint32_t* status, Walker64& W) {
  const int lane = threadIdx.x & 31;
  for (int j = 0; j < n; ++j) {
    bar_sync(BAR_START, kBlock64);
    if (W.failed || j + 1 == n) return;
    bool ok = true;
    if (lane < 2) ok = wait_ge(sv.upd + (j + 1) * n + j + lane, j, status);
    ok = __all_sync(0xffffffffu, ok);
    __syncwarp();  // a vote orders no memory: the other lanes' reads come after the acquire loads of lanes 0 and 1
    if (ok) {
      const double* Ap = A + ((size_t)(j + 1) * lda + j) * kNB64;
      double* d = W.diag[(j + 1) & 1];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = 4 * u + (lane >> 3), c = 2 * (lane & 7);
        const double2 v = __ldcg(reinterpret_cast<const double2*>(Ap + r * lda + c));
        const double2 w = __ldcg(reinterpret_cast<const double2*>(Ap + kNB64 + r * lda + c));
        *reinterpret_cast<double2*>(W.panel + r * kTLD + c) = v;
        *reinterpret_cast<double2*>(d + r * kTLD + c) = w;
      }
    }
    if (lane == 0) W.ok = ok;
    bar_arrive(BAR_LOADED, kThr + 32);
    if (!ok) return;
  }
}
__device__ void walker64_publishes(int n, const Sync64& sv, Walker64& W) {
  const bool lead = (threadIdx.x & 31) == 0;
  for (int j = 0; j < n; ++j) {
    bar_sync(BAR_START, kBlock64);
    if (W.failed) return;
    bar_sync(BAR_STORED + 2 * (j & 1), kThr + 32);
    if (lead) st_release(sv.pdone + j, 1);
    if (j + 1 == n) return;
    bar_sync(BAR_STORED + 2 * (j & 1) + 1, kThr + 32);
    if (W.failed) return;
    if (lead) st_release(sv.tdone + (j + 1) * n + j, 1);
  }
}
__device__ void walker64(double* A, size_t lda, int n, double* Linv, uint32_t* status, LMState* lm, Walker64& W) {
  const int tid = threadIdx.x, r = tid >> 3, c = tid & 7;
  tile_in(W.diag[0], A, lda);
  csync();
  for (int j = 0; j < n; ++j) {
    double *Ajj = A + ((size_t)j * lda + j) * kNB64, *T0 = W.diag[j & 1], *Tn = W.diag[(j + 1) & 1], *T2 = W.panel;
    bar_arrive(BAR_START, kBlock64);
    const bool bad = potrf64(T0, W.linv, W.S);
    tile_out(Linv + (size_t)j * kNB64 * kNB64, kNB64, W.linv);
    tile_out(Ajj, lda, T0);
    if (bad && tid == 0) {
      atomicOr(status, SC_STATUS_NOTPD);
      if (lm != nullptr) lm->notpd = 1;
    }
    bar_arrive(BAR_STORED + 2 * (j & 1), kThr + 32);
    if (j + 1 == n) return;
    bar_sync(BAR_LOADED, kThr + 32);
    if (!W.ok) {
      if (tid == 0) {
        W.failed = 1;
        if (lm != nullptr) lm->notpd = 1;
      }
      csync();
      bar_arrive(BAR_STORED + 2 * (j & 1) + 1, kThr + 32);
      return;
    }
    // L_j+1,j, and the next diagonal tile
    double* Ap = Ajj + lda * kNB64;
    double acc[2];
    product64<true>(acc, T2, W.linv);
    csync();
    T2[r * kTLD + c] = acc[0];
    T2[r * kTLD + c + 8] = acc[1];
    csync();
    tile_out(Ap, lda, T2);
    bar_arrive(BAR_STORED + 2 * (j & 1) + 1, kThr + 32);
    // lower part only: the 128 entries of tri_entry, and (p, p), p < 8, each
    // by four lanes of warp 3
    int er, ec;
    tri_entry(tid, er, ec);
    double a = 0.0, e = 0.0;
    const int q = (tid & 31) >> 2, part = 4 * (tid & 3);
#pragma unroll
    for (int m = 0; m < kNB64; m += 2) {
      const double2 v = ldd2(T2 + er * kTLD + m), w = ldd2(T2 + ec * kTLD + m);
      a = fma(v.y, w.y, fma(v.x, w.x, a));
    }
    if (tid >= 96) {
#pragma unroll
      for (int m = 0; m < 4; ++m) e = fma(T2[q * kTLD + part + m], T2[q * kTLD + part + m], e);
      e += __shfl_xor_sync(0xffffffffu, e, 1);
      e += __shfl_xor_sync(0xffffffffu, e, 2);
    }
    Tn[er * kTLD + ec] -= a;
    if (tid >= 96 && part == 0) Tn[q * kTLD + q] -= e;
    csync();
  }
}

__global__ void __launch_bounds__(kBlock64) k_chol64(double* __restrict__ A0, int lda_, int n,
                                                    double* __restrict__ Linv0, int per_job, int sms, size_t js, int* sync0,
                                                    uint32_t* status0, LMState* lm0) {
  const int job = blockIdx.x / per_job;
  LMState* lm = job_ptr(lm0, js, job);
  if (lm != nullptr && lm->done) return;
  double* A = job_ptr(A0, js, job);
  double* Linv = job_ptr(Linv0, js, job);
  uint32_t* status = job_ptr(status0, js, job);
  const Sync64 sv(job_ptr(sync0, js, job), n);
  const size_t lda = lda_;
  // a worker's four tiles lie over the walker's
  __shared__ __align__(16) Walker64 W;
  double(*T)[kNB64 * kTLD] = reinterpret_cast<double(*)[kNB64 * kTLD]>(&W);
  static_assert(offsetof(Walker64, S) >= 4 * kNB64 * kTLD * sizeof(double), "four tiles");
  __shared__ Claim s_claim;
  __shared__ int s_first;
  const int tid = threadIdx.x, warp = tid >> 5;
  if (tid == 0) {
    // The walker: the first block to arrive; of jobs with few blocks, which go
    // round the SMs, another place in each round: with the first of every job
    // and an even number of SMs, half of them or a quarter had the walkers and
    // the others the work (304 jobs of 64 stations, two blocks each: 25.8 ms a
    // factorisation, 20.0; 4 jobs, 152 blocks each, are faster the first way).
    s_first = per_job > kTurnBlocks ? atomicAdd(sv.fctr, 1) == 0
                                    : (int)blockIdx.x - job * per_job == job * per_job / sms % per_job;
    if (s_first) LeaveWalkerSm::publish(sv.sctr);
    W.failed = 0;
  }
  __syncthreads();
  if (s_first) {
    if (warp < kThr / 32) walker64(A, lda, n, Linv, status, lm, W);
    else if (warp == kThr / 32) walker64_loads(A, lda, n, sv, status, W);
    else walker64_publishes(n, sv, W);
    return;
  }
  if (warp >= kThr / 32) return;
  // With blocks on several SMs, those that share the walker's leave it, up to
  // half of them: one warp instruction of theirs is 64 cycles of its.
  const bool yield = per_job > 16 && (int)gridDim.x == per_job;
  LeaveWalkerSm leave;
  int jp = 0, jb = 0;
  for (;;) {
    if (warp == 0) {
      Claim c = {-1, 0, 0, 0};
      const int stay = __shfl_sync(0xffffffffu, !(yield && tid == 0 && leave.ask(sv.sctr, per_job)), 0);
      if (stay) c = claim64(n, sv, status, jp, jb);
      if (tid == 0) s_claim = c;
    }
    csync();
    const Claim tk = s_claim;
    if (tk.kind < 0) {
      if (tk.kind == -2 && tid == 0 && lm != nullptr) lm->notpd = 1;
      return;
    }
    const int j = tk.j;
    bool ok = true;
    if (tk.kind == 0) {
      const int i = tk.i, r = tid >> 3, c = tid & 7;
      double* Ap = A + ((size_t)i * lda + j) * kNB64;
      if (tid == 0) ok = ld_acquire(sv.pdone + j) != 0;
      if (tid == 32) ok = wait_ge(sv.upd + i * n + j, j, status);
      ok = csync_and(ok);
      if (ok) {
        tile_in(T[0], Ap, lda);
        tile_in(T[1], Linv + (size_t)j * kNB64 * kNB64, kNB64);
        csync();
        double acc[2];
        product64<true>(acc, T[0], T[1]);
        csync();
        T[0][r * kTLD + c] = acc[0];
        T[0][r * kTLD + c + 8] = acc[1];
        csync();
        tile_out(Ap, lda, T[0]);
        if (tid == 64) ok = wait_ge(sv.tdone + (j + 1) * n + j, 1, status);
        if (tid == 96) ok = wait_ge(sv.upd + i * n + j + 1, j, status);
        ok = csync_and(ok);
        if (tid == 0) st_release(sv.tdone + i * n + j, 1);
      }
      if (ok) {
        tile_in(T[1], A + ((size_t)(j + 1) * lda + j) * kNB64, lda);
        double* Out = Ap + kNB64 + r * lda + c;
        const double old0 = __ldcg(Out), old1 = __ldcg(Out + 8);
        csync();
        double acc[2];
        product64<false>(acc, T[0], T[1]);
        __stcg(Out, old0 - acc[0]);
        __stcg(Out + 8, old1 - acc[1]);
        csync();
        if (tid == 32) st_release(sv.upd + i * n + j + 1, j + 1);
      }
    } else {
      // tile rows i0, i0 + 1, tile columns k0, k0 + 1; active: i >= k >= j + 2
      const int i0 = 2 * tk.i, k0 = 2 * tk.K;
      const bool left = k0 >= j + 2, diag = i0 == k0;
      // tile q: row i0 + q / 2, column k0 + q % 2
      auto active = [&](int q) { return (q & 1 || left) && !(diag && q == 1) && !(q == 0 && i0 < j + 2); };
      if (tid < 4) {
        if (active(tid)) ok = wait_ge(sv.upd + (i0 + (tid >> 1)) * n + k0 + (tid & 1), j, status);
      } else if (tid >= 32 && tid < 34) {
        if (i0 + tid - 32 >= j + 2) ok = wait_ge(sv.tdone + (i0 + tid - 32) * n + j, 1, status);
      } else if (tid >= 64 && tid < 66) {
        if (k0 + tid - 64 >= j + 2) ok = wait_ge(sv.tdone + (k0 + tid - 64) * n + j, 1, status);
      }
      ok = csync_and(ok);
      if (ok) {
        const double *L0 = A + ((size_t)i0 * lda + j) * kNB64, *L1 = A + ((size_t)k0 * lda + j) * kNB64;
        tile_in(T[0], L0, lda);
        tile_in(T[1], L0 + lda * kNB64, lda);
        tile_in(T[2], L1, lda);
        tile_in(T[3], L1 + lda * kNB64, lda);
        const int r = tid >> 3, c = tid & 7;
        double* Out = A + ((size_t)i0 * lda + k0) * kNB64 + r * lda + c;
        double old[4][2];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const double* o = Out + (size_t)(q >> 1) * kNB64 * lda + (q & 1) * kNB64;
          old[q][0] = active(q) ? __ldcg(o) : 0.0;
          old[q][1] = active(q) ? __ldcg(o + 8) : 0.0;
        }
        csync();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (!active(q)) continue;
          double* o = Out + (size_t)(q >> 1) * kNB64 * lda + (q & 1) * kNB64;
          double acc[2];
          product64<false>(acc, T[q >> 1], T[2 + (q & 1)]);
          __stcg(o, old[q][0] - acc[0]);
          __stcg(o + 8, old[q][1] - acc[1]);
        }
        csync();
        if (tid == 32) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (active(q)) st_release(sv.upd + (i0 + (q >> 1)) * n + k0 + (q & 1), j + 1);
        }
      }
    }
    if (!ok) {
      if (tid == 0 && lm != nullptr) lm->notpd = 1;
      return;
    }
    csync();  // the tiles and s_claim are free
  }
}

// ---- triangular solves ---------------------------------------------------------------------
//
// One block per 32 rows and direction, y_i = Linv_ii (b_i - sum_{j<i} L_ij y_j),
// x_i = Linv_ii^T (y_i - sum_{j>i} L_ji^T x_j), as k_chol_solve (cholesky.cu)
// with the solved blocks passed as tagged words.  32 rows balance the
// passing of a block (about 700 cycles) against its two products (512 cycles
// each, the float64 rate); each thread keeps its share of a row's sum over
// all the tiles, so that a product ends in two shuffle steps only where a
// block is finished.  The inverse of the 32x32 diagonal block comes from
// those of its 16x16 tiles.
constexpr int kSB = 32, kSLD = kSB + 2;

__device__ __forceinline__ void put_tagged64(uint64_t* w, double v, uint32_t tag) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const ulonglong2 p = make_ulonglong2(((unsigned long long)tag << 32) | (b >> 32),
                                       ((unsigned long long)tag << 32) | (b & 0xffffffffull));
  __stcg(reinterpret_cast<unsigned long long*>(w), p.x);
  __stcg(reinterpret_cast<unsigned long long*>(w) + 1, p.y);
}
__device__ __forceinline__ unsigned long long ld_word64(const uint64_t* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ bool get_tagged64(const uint64_t* w, uint32_t tag, double& v, uint32_t* status) {
  for (long it = 0; it < kSpinLimit; ++it) {
    const unsigned long long w0 = ld_word64(w), w1 = ld_word64(w + 1);
    if ((uint32_t)(w0 >> 32) == tag && (uint32_t)(w1 >> 32) == tag) {
      v = __longlong_as_double((long long)((w0 << 32) | (w1 & 0xffffffffull)));
      return true;
    }
    if ((it & 63) == 63 && (ld_status(status) & SC_STATUS_TIMEOUT)) return false;
    if (it >= 32) __nanosleep(64);
  }
  atomicOr(status, SC_STATUS_TIMEOUT);
  return false;
}

// a 32x32 tile into shared memory as one cp.async group
__device__ __forceinline__ void tile32_async(double* sm, const double* g, size_t lda) {
  for (int e = threadIdx.x; e < kSB * kSB / 2; e += kThr) {
    const int r = e >> 4, c = 2 * (e & 15);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::saddr(sm + r * kSLD + c)), "l"(g + r * lda + c)
                 : "memory");
  }
  async_commit();
}

__global__ void __launch_bounds__(kThr) k_solve64(const double* __restrict__ A0, int lda_, int nS,
                                                 const double* __restrict__ Linv0, int* sync0,
                                                 const double* __restrict__ b0, uint64_t* __restrict__ yw0,
                                                 double* __restrict__ x0, int accumulate, uint32_t tag_fwd,
                                                 uint32_t* status0, const LMState* lm0, int G, size_t js) {
  dep_sync(js == 0);
  const uint32_t tag_bwd = tag_fwd + 1;
  __shared__ __align__(16) double D[kSB * kSLD], B[2][kSB * kSLD];
  __shared__ double vin[kSB];
  __shared__ int s_task, s_ok;
  const int tid = threadIdx.x, row = tid >> 2, part = tid & 3;
  const size_t lda = lda_;
  int* const counter = sync0 + 1;  // the solve counter (SyncView::sctr)
  const int n_tasks = 2 * nS;
  for (;;) {
    __syncthreads();
    if (tid == 0) {
      s_task = atomicAdd(counter, 1);
      s_ok = 1;
    }
    __syncthreads();
    const int tg = s_task;
    if (tg >= n_tasks * G) break;
    const int job = tg % G, t = tg / G;
    const LMState* lm = job_ptr(lm0, js, job);
    if (lm != nullptr && (lm->done | lm->notpd)) continue;
    const double* A = job_ptr(A0, js, job);
    const double* Linv = job_ptr(Linv0, js, job);
    const double* b = job_ptr(b0, js, job);
    uint64_t* yw = job_ptr(yw0, js, job);
    double* x = job_ptr(x0, js, job);
    uint32_t* status = job_ptr(status0, js, job);
    const bool fwd = t < nS;
    const int i = fwd ? t : 2 * nS - 1 - t;
    const int cnt = fwd ? i : nS - 1 - i;  // off-diagonal tiles, in the order their blocks are solved
    auto other = [&](int m) { return fwd ? m : nS - 1 - m; };
    auto tile = [&](int m) {
      const int o = other(m);
      return fwd ? A + ((size_t)i * lda + o) * kSB : A + ((size_t)o * lda + i) * kSB;
    };
    auto fetch = [&](int blk, uint32_t tag) {
      if (tid < kSB) {
        double v = 0.0;
        if (!get_tagged64(yw + 2 * (size_t)(blk * kSB + tid), tag, v, status)) s_ok = 0;
        vin[tid] = v;
      }
    };
    if (cnt > 0) tile32_async(B[0], tile(0), lda);
    else async_commit();
    // the inverse of the diagonal block: its tiles' inverses V0, V1, and
    // -V1 L10 V0 below the diagonal, through B[1]
    {
      const double* V = Linv + (size_t)2 * i * kNB64 * kNB64;
      const double* L10 = A + ((size_t)(i * kSB + kNB64)) * lda + i * kSB;
      const int r = tid >> 3, c = 2 * (tid & 7);
      const double2 zero = make_double2(0.0, 0.0);
      *reinterpret_cast<double2*>(D + r * kSLD + c) = __ldcg(reinterpret_cast<const double2*>(V + r * kNB64 + c));
      *reinterpret_cast<double2*>(D + r * kSLD + kNB64 + c) = zero;
      *reinterpret_cast<double2*>(D + (r + kNB64) * kSLD + kNB64 + c) =
          __ldcg(reinterpret_cast<const double2*>(V + kNB64 * kNB64 + r * kNB64 + c));
      *reinterpret_cast<double2*>(B[1] + r * kSLD + c) = __ldcg(reinterpret_cast<const double2*>(L10 + r * lda + c));
      __syncthreads();
      double w0 = 0.0, w1 = 0.0;  // L10 V0
#pragma unroll 4
      for (int m = 0; m < kNB64; ++m) {
        const double l = B[1][r * kSLD + m];
        w0 = fma(l, D[m * kSLD + c], w0);
        w1 = fma(l, D[m * kSLD + c + 1], w1);
      }
      B[1][(r + kNB64) * kSLD + c] = w0;
      B[1][(r + kNB64) * kSLD + c + 1] = w1;
      __syncthreads();
      double e0 = 0.0, e1 = 0.0;
#pragma unroll 4
      for (int m = 0; m < kNB64; ++m) {
        const double l = -D[(r + kNB64) * kSLD + kNB64 + m];
        e0 = fma(l, B[1][(m + kNB64) * kSLD + c], e0);
        e1 = fma(l, B[1][(m + kNB64) * kSLD + c + 1], e1);
      }
      D[(r + kNB64) * kSLD + c] = e0;
      D[(r + kNB64) * kSLD + c + 1] = e1;
      __syncthreads();
    }
    double acc = 0.0;  // this thread's share of entry `row`
    if (fwd) {
      if (part == 0) acc = b[i * kSB + row];
    } else {
      fetch(i, tag_fwd);  // y_i
      __syncthreads();
      if (part == 0) acc = vin[row];
    }
    for (int m = 0; m < cnt; ++m) {
      const double* cur = B[m & 1];
      __syncthreads();  // every thread is done with vin and with the buffer refilled next
      if (m + 1 < cnt) tile32_async(B[(m + 1) & 1], tile(m + 1), lda);
      else async_commit();
      fetch(other(m), fwd ? tag_fwd : tag_bwd);
      async_wait_prev();
      __syncthreads();
      if (!s_ok) break;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = part + 4 * u;
        acc = fma(-(fwd ? cur[row * kSLD + k] : cur[k * kSLD + row]), vin[k], acc);
      }
    }
    async_wait_all();
    __syncthreads();
    if (!s_ok) break;
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    if (part == 0) vin[row] = acc;
    __syncthreads();
    double o = 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = part + 4 * u;
      o = fma(fwd ? D[row * kSLD + k] : D[k * kSLD + row], vin[k], o);
    }
    o += __shfl_xor_sync(0xffffffffu, o, 1);
    o += __shfl_xor_sync(0xffffffffu, o, 2);
    if (part == 0) {
      const int e = i * kSB + row;
      put_tagged64(yw + 2 * (size_t)e, o, fwd ? tag_fwd : tag_bwd);
      if (!fwd) x[e] = accumulate ? x[e] + o : o;
    }
  }
  async_wait_all();
}

}  // namespace

cudaError_t launch_chol64(double* A, int lda, int nT, double* Linv, int* sync, uint32_t* status, LMState* lm,
                          int max_ctas, cudaStream_t st, bool zeroed, const Batch& bt) {
  // up to four blocks per SM: the float64 pipes take about one, the others
  // cover claims, waits and loads (one block of four groups per SM with
  // blocks kept for P was 4% slower at order 1200 and 15% at 4096)
  static const int sms = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return std::max(1, v);
  }();
  static const int resident = [] {
    int per = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_chol64, kBlock64, 0);
    return std::max(2, sms * std::min(std::max(per, 1), 4));
  }();
  const int n = tiles64(nT);
  const size_t row = sizeof(int) * chol64_sync_ints(nT);
  cudaError_t e = zeroed      ? cudaSuccess
                  : bt.G == 1 ? cudaMemsetAsync(sync, 0, row, st)
                              : cudaMemset2DAsync(sync, bt.js, 0, row, bt.G, st);
  if (e != cudaSuccess) return e;
  // per job: the walker and as many blocks as the first panel has tasks, at
  // least one, within what is resident at once; of a large batch three, even if
  // its last jobs then start when others are done: a job's walker keeps an SM
  // little busy, and its one worker waits as much as it multiplies (64 stations,
  // 304 jobs 18.2 ms with two workers, 14.6 with three; 400 jobs 26.7 with one,
  // 17.5; 64x64 tiles in one list for all jobs, as before, took 14.3 and 18.8)
  const long long tasks = (long long)p_count64(n, 0) + b_count64(n, 0);
  const int total = max_ctas > 0 ? std::min(resident, max_ctas) : resident;
  const int share = std::max(total / bt.G, max_ctas > 0 ? 2 : 4);
  const int per_job = (int)std::max<long long>(2, std::min<long long>(1 + tasks, share));
  if ((long long)per_job * bt.G > (1LL << 30)) return cudaErrorInvalidValue;
  // not by launch_dep: blocks that come in while the assembly still runs crowd
  // on the SMs it has left, the walker among them (64 stations: 4.58 ms, 3.81)
  k_chol64<<<per_job * bt.G, kBlock64, 0, st>>>(A, lda, n, Linv, per_job, sms, bt.js, sync, status, lm);
  return cudaGetLastError();
}

cudaError_t launch_solve64(const double* A, int lda, int nT, const double* Linv, int* sync, const double* b,
                           uint64_t* bwork, double* x, int accumulate, uint32_t tag, uint32_t* status,
                           const LMState* lm, cudaStream_t st, const Batch& bt) {
  const int nS = nT * (kNB / kSB);
  if ((long long)2 * nS * bt.G > (1LL << 30)) return cudaErrorInvalidValue;
  const cudaError_t e = cudaMemsetAsync(sync + 1, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  return launch_dep(bt.js == 0, k_solve64, 2 * nS * bt.G, kThr, 0, st, A, lda, nS, Linv, sync, b, bwork, x, accumulate, tag, status,
                    lm, bt.G, bt.js);
}

}  // namespace sc
