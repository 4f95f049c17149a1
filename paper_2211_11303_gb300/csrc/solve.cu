// The triangular solve of Algorithm 1 step III (sm_103a): one persistent
// launch runs the solve DAG of one or several problems, the preconditioner
// application x = U^-1 (L^-1 P b) with up to 16 right-hand sides at a time.
//
// Every task is a narrow product: PROJ t (+)= Y^T z over a range of rows, or
// ROWMV, one unit of at most 64 rows (mostly at most 32) receiving sum_t A_t B_t (dense tiles,
// low-rank X factors, or a row panel of an inverted diagonal block).  The
// work is one pass over the factor; what bounds it is the chain through the
// solve blocks, three dependent tasks (panel, projection, update) per block
// and direction.  So the kernel is built for the latency of one such link:
//
// - Tasks are numbered in the order in which a simulated list schedule starts
//   them and handed out by one counter per problem, so a CTA holds its task
//   long before the task is ready.  It loads the task's records, builds the
//   table of its columns, loads the first 32 columns of each warp into registers
//   and asks L2 for the others, and only then waits for the predecessors' counter.
// - A finished task decrements its successors' counters with reductions after
//   one fence (no queue, no reply to wait for).
// - Lanes own rows (or, for PROJ, the summed index) and carry 4 or 8
//   right-hand sides in registers; the eight warps split the columns and meet
//   in shared memory.  The sums' order depends on neither the number of
//   right-hand sides carried nor the CTA, so batched results equal single ones.
//
// Tickets cannot deadlock: a problem's tickets are claimed in topological
// order, so all predecessors of the smallest unfinished ticket are finished
// and its CTA, which holds nothing else, runs it; no two CTAs need to be
// resident together.  Every wait is bounded by the launch's limit
// (%globaltimer); one that runs out records HLU_ERR_TIMEOUT and all CTAs stop.
//
// One apply of 8 columns at n = 24 (N = 91,656): 7.8 ms, against 54.8 ms for
// the tile-by-tile chain through the factorisation's executor.
#include <cuda_runtime.h>

#include <cstdint>

#include "launch_count.h"

#include "exec.h"
#include "hlu_internal.h"

namespace hlu {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kCols = 512;   // columns (or summed rows of a PROJ) staged at a time
constexpr int kTerms = 32;   // terms staged at a time

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ int32_t ld_acquire_s32(const int32_t* p) {
  int32_t v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void red_dec(int32_t* p) {
  asm volatile("red.relaxed.gpu.global.add.s32 [%0], -1;" ::"l"(p) : "memory");
}

template <class T, int KC>
struct SolveSmem {
  T b[kCols * KC];           // staged right operand, KC per column; then the warps' partial sums
  T red[64 * KC];            // PROJ: partial sums of the splits
  int64_t col_a[kCols];      // arena offset of tile row 0 of a column of A
  int64_t col_b[kCols];      // arena offset of a row of B
  int32_t col_ld[kCols];     // column stride of that row of B
  int32_t col_r[kCols];      // rows the column covers: lo | hi << 8
  Term tm[kTerms];
  int32_t pre[kTerms + 1];   // first column of each staged term
  Task t;
  int64_t succ[2];
  int64_t task;
  int32_t prob;
  uint64_t start;            // trace: when the wait ended
};

// the KC values of a staged row
template <int KC>
__device__ __forceinline__ void row_of(const float* p, float (&v)[KC]) {
#pragma unroll
  for (int q = 0; q < KC / 4; ++q) {
    const float4 x = reinterpret_cast<const float4*>(p)[q];
    v[4 * q] = x.x, v[4 * q + 1] = x.y, v[4 * q + 2] = x.z, v[4 * q + 3] = x.w;
  }
}
template <int KC>
__device__ __forceinline__ void row_of(const double* p, double (&v)[KC]) {
#pragma unroll
  for (int q = 0; q < KC / 2; ++q) {
    const double2 x = reinterpret_cast<const double2*>(p)[q];
    v[2 * q] = x.x, v[2 * q + 1] = x.y;
  }
}

// Sums each of the V values over the warp, pairs 16, 8, 4, 2, 1 lanes apart;
// while values are left to split, each step sends the half the partner keeps.
// Returns the value whose index the lane's high bits spell (bit 16 first).
template <class T, int V>
__device__ __forceinline__ T warp_halve(T (&v)[V], int lane) {
  int w = V;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (w > 1) {
      w >>= 1;
      const bool hi = (lane & o) != 0;
#pragma unroll
      for (int q = 0; q < V / 2; ++q)
        if (q < w) {
          const T keep = hi ? v[q + w] : v[q], send = hi ? v[q] : v[q + w];
          v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
  return v[0];
}

// b[c][j] <- *at(c, j), c < n, j < kc (zero up to KC); neighbouring threads
// take the KC values of a row, so the shared stores are conflict-free
template <class T, int KC, class At>
__device__ __forceinline__ void stage_rows(T* b, int n, int kc, const At& at) {
  constexpr int U = KC * kCols / kThreads < 12 ? KC * kCols / kThreads : 12;
  for (int e0 = threadIdx.x; e0 < n * KC; e0 += U * kThreads) {
    T v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * kThreads, c = e / KC, j = e % KC;
      v[u] = (e < n * KC && j < kc) ? __ldcg(at(c, j)) : T(0);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (e0 + u * kThreads < n * KC) b[e0 + u * kThreads] = v[u];
  }
}

// Waits until the task's predecessors are finished; false when the launch is
// aborted.  Thread 0 polls, the barrier passes its acquire on.
template <class T, int KC>
__device__ __forceinline__ bool wait_ready(SolveSmem<T, KC>& s, const SolveProb& P, const SolveArgs& a) {
  if (threadIdx.x == 0) {
    const int32_t* cnt = P.indeg + s.task;
    volatile int32_t* abort_flag = (volatile int32_t*)a.status + 3;
    if (ld_acquire_s32(cnt) > 0) {
      const uint64_t t0 = now_ns();
      for (int spin = 1;; ++spin) {
        if (ld_acquire_s32(cnt) <= 0) break;
        if ((spin & 15) == 0) {
          if (*abort_flag) {
            s.task = -1;
            break;
          }
          if (now_ns() - t0 > a.wait_limit_ns) {
            atomicCAS(a.status, 0, 5);
            atomicCAS(a.status + 1, -1, (int32_t)s.task);
            *abort_flag = 1;
            s.task = -1;
            break;
          }
        }
      }
    }
    if (a.trace) s.start = now_ns();
  }
  __syncthreads();
  return s.task >= 0;
}

// Stages terms [q0, q0 + kTerms) of the task and their column prefix; returns
// the columns of the group.
template <class T, int KC>
__device__ __forceinline__ int stage_terms(SolveSmem<T, KC>& s, const SolveProb& P, int q0) {
  const int nq = min(kTerms, s.t.list_count - q0);
  const int words = nq * (int)(sizeof(Term) / 4);
  const int32_t* src = reinterpret_cast<const int32_t*>(P.terms + s.t.list_begin + q0);
  int32_t* dst = reinterpret_cast<int32_t*>(s.tm);
  for (int w = threadIdx.x; w < words; w += kThreads) dst[w] = __ldg(src + w);
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    int p = lane < nq ? __ldg(P.term_p + s.t.list_begin + q0 + lane) : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, p, o);
      if (lane >= o) p += x;
    }
    s.pre[lane + 1] = p;
    if (lane == 0) s.pre[0] = 0;
  }
  __syncthreads();
  return s.pre[kTerms];
}
// The table of columns [base, base + kCols) of the staged group.
template <class T, int KC>
__device__ __forceinline__ void fill_columns(SolveSmem<T, KC>& s, int q0, int base) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nq = min(kTerms, s.t.list_count - q0);
  for (int q = warp; q < nq; q += kWarps) {
    const Term& m = s.tm[q];
    const int lo = m.roff, hi = m.roff + m.A.rows;
    for (int l = lane; l < s.pre[q + 1] - s.pre[q]; l += 32) {
      const int c = s.pre[q] + l - base;
      if (c < 0 || c >= kCols) continue;
      s.col_a[c] = m.A.off + (int64_t)l * m.A.cs - lo;
      s.col_b[c] = m.B.off + l;
      s.col_ld[c] = m.B.cs;
      s.col_r[c] = lo | (hi << 8);
    }
  }
  __syncthreads();
}

// One ROWMV task: unit rows r (lane r, and r + 32 when NR is 2) of c, KC columns
// at a time.  NR is a template parameter because a test of it between the
// loads kept them from being in flight together (n = 24: 12.3 instead of
// 8.4 ms an apply).
template <class T, int KC, int NR>
__device__ __forceinline__ bool run_rowmv(SolveSmem<T, KC>& s, const SolveProb& P, const SolveArgs& a) {
  constexpr int U = sizeof(T) == 4 ? 16 : 8;  // columns of a warp in one register buffer
  constexpr int kOut = 64 * KC / kThreads;    // outputs of a thread: row e % 64, column e / 64
  constexpr int kLines = 64 * (int)sizeof(T) / 128;  // cache lines of a column
  T* arena = reinterpret_cast<T*>(P.arena);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rows = s.t.c.rows, k = P.nrhs;
  const bool over = (s.t.flags & TF_OVERWRITE) != 0;
  const T sign = T(s.t.sign);
  bool waited = false;
  for (int j0 = 0; j0 < k; j0 += KC) {
    const int kc = min(KC, k - j0);
    T* out = arena + s.t.c.off + (int64_t)j0 * s.t.c.cs;
    T acc[NR][KC], old[kOut];
#pragma unroll
    for (int i = 0; i < NR; ++i)
#pragma unroll
      for (int j = 0; j < KC; ++j) acc[i][j] = T(0);
    bool have_old = false;
    auto load_old = [&]() {
#pragma unroll
      for (int o = 0; o < kOut; ++o) {
        const int e = threadIdx.x + o * kThreads, r = e & 63, j = e >> 6;
        old[o] = (!over && r < rows && j < kc) ? __ldcg(out + r + (int64_t)j * s.t.c.cs) : T(0);
      }
      have_old = true;
    };
    for (int q0 = 0; q0 < s.t.list_count; q0 += kTerms) {
      const int total = stage_terms(s, P, q0);
      for (int base = 0; base < total; base += kCols) {
        const int n = min(kCols, total - base);
        fill_columns(s, q0, base);
        // buffer g holds columns warp + 8 (g U + u) of the chunk; lanes and
        // columns outside repeat an element inside and count it as zero, so
        // that no branch comes between the loads
        T x[NR][U], y[NR][U];
        auto load = [&](T(&v)[NR][U], int g) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int c = warp + kWarps * (g * U + u), cc = min(c, n - 1);
            const int r = s.col_r[cc], lo = r & 255, hi = r >> 8;
            const T* p = arena + s.col_a[cc];
#pragma unroll
            for (int i = 0; i < NR; ++i) {
              const int row = lane + 32 * i;
              const T q = __ldg(p + min(max(row, lo), hi - 1));
              v[i][u] = c < n && row >= lo && row < hi ? q : T(0);
            }
          }
        };
        auto fma = [&](const T(&v)[NR][U], int g) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int c = warp + kWarps * (g * U + u);
            if (sizeof(T) == 8 && c >= n) continue;  // FP64 is bound by its FMAs
            T w[KC];
            row_of<KC>(s.b + min(c, n - 1) * KC, w);
#pragma unroll
            for (int i = 0; i < NR; ++i)
#pragma unroll
              for (int j = 0; j < KC; ++j) acc[i][j] += v[i][u] * w[j];
          }
        };
        const int groups = (n + kWarps * U - 1) / (kWarps * U);
        load(x, 0);
        if (groups > 1) load(y, 1);
        // the columns behind the registers come from L2 then, not from memory
        for (int e = threadIdx.x; e < (n - 2 * kWarps * U) * kLines; e += kThreads) {
          const int c = 2 * kWarps * U + e / kLines, r = s.col_r[c], lo = r & 255, hi = r >> 8;
          const int row = lo + (e % kLines) * (128 / (int)sizeof(T));
          if (row < hi) prefetch_l2(arena + s.col_a[c] + row);
        }
        if (!waited) {
          if (!wait_ready(s, P, a)) return false;
          waited = true;
        }
        if (!have_old) load_old();
        stage_rows<T, KC>(s.b, n, kc, [&](int c, int j) { return arena + s.col_b[c] + (int64_t)(j0 + j) * s.col_ld[c]; });
        __syncthreads();
        for (int g = 0; g < groups; g += 2) {
          fma(x, g);
          if (g + 2 < groups) load(x, g + 2);
          if (g + 1 < groups) fma(y, g + 1);
          if (g + 3 < groups) load(y, g + 3);
        }
        __syncthreads();  // the table and the staged rows are free again
      }
      __syncthreads();  // (also when the group had no columns)
    }
    if (!waited) {  // no columns at all (every rank zero)
      if (!wait_ready(s, P, a)) return false;
      waited = true;
    }
    if (!have_old) load_old();
    // the warps' partial sums: [warp][j][row]
#pragma unroll
    for (int j = 0; j < KC; ++j) {
#pragma unroll
      for (int i = 0; i < NR; ++i) s.b[(warp * KC + j) * 64 + lane + 32 * i] = acc[i][j];
    }
    __syncthreads();
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
      const int e = threadIdx.x + o * kThreads, r = e & 63, j = e >> 6;
      T sum = T(0);
      if (r < rows)
#pragma unroll
        for (int w = 0; w < kWarps; ++w) sum += s.b[w * KC * 64 + e];
      if (r < rows && j < kc) __stcg(out + r + (int64_t)j * s.t.c.cs, old[o] + sign * sum);
    }
    __syncthreads();
  }
  return true;
}

// One PROJ task: c (r x k) (+)= a^T b over a.rows summed rows.  A warp takes
// pairs of A's columns (lanes along the summed rows); when there are fewer
// pairs than warps, the warps of a pair split the rows.
template <class T, int KC>
__device__ bool run_proj(SolveSmem<T, KC>& s, const SolveProb& P, const SolveArgs& a) {
  constexpr int U = sizeof(T) == 4 ? 16 : 8;  // 32-row steps in the register buffer
  constexpr int kOut = 64 * KC / kThreads;
  T* arena = reinterpret_cast<T*>(P.arena);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m = s.t.a.rows, k = P.nrhs;
  const int r = s.t.a.slot < 0 ? s.t.a.cols : __ldcg(P.ranks + s.t.a.slot);
  if (r == 0) return wait_ready(s, P, a);
  const int npairs = (r + 1) / 2;
  const int split = npairs >= kWarps ? 1 : kWarps / npairs;
  const int pair0 = split == 1 ? warp : warp % npairs, sub = split == 1 ? 0 : warp / npairs;
  const bool busy = sub < split;
  const T* A = arena + s.t.a.off;
  const int64_t lda = s.t.a.cs;
  T x[2][U];
  // rows 32 (s0 + split u) + lane of columns 2 pr, 2 pr + 1, row limit m
  auto load = [&](T(&v)[2][U], int pr, int m0, int st) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int row = m0 + 32 * (st + split * u) + lane;
      const bool in = row < m && row < m0 + kCols;
      v[0][u] = in ? __ldg(A + row + (int64_t)(2 * pr) * lda) : T(0);
      v[1][u] = in && 2 * pr + 1 < r ? __ldg(A + row + (int64_t)(2 * pr + 1) * lda) : T(0);
    }
  };
  if (busy && pair0 < npairs) load(x, pair0, 0, sub);
  bool preloaded = true;
  {
    const int lines = (m * (int)sizeof(T) + 127) / 128, per = 128 / (int)sizeof(T);
    for (int e = threadIdx.x; e < r * lines; e += kThreads)
      if (e / lines >= 2 * kWarps || (e % lines) * per >= 32 * U * split)
        prefetch_l2(A + (int64_t)(e / lines) * lda + (e % lines) * per);
  }
  if (!wait_ready(s, P, a)) return false;
  for (int j0 = 0; j0 < k; j0 += KC) {
    const int kc = min(KC, k - j0);
    T* out = arena + s.t.c.off + (int64_t)j0 * s.t.c.cs;
    const T* B = arena + s.t.b.off + (int64_t)j0 * s.t.b.cs;
    T old[kOut];
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
      const int e = threadIdx.x + o * kThreads, i = e % 64, j = e / 64;
      old[o] = ((s.t.flags & TF_ADD) && i < r && j < kc) ? __ldcg(out + i + (int64_t)j * s.t.c.cs) : T(0);
    }
    for (int m0 = 0; m0 < m; m0 += kCols) {
      const int n = min(kCols, m - m0);
      if (m0 > 0) __syncthreads();
      stage_rows<T, KC>(s.b, n, kc, [&](int c, int j) { return B + m0 + c + (int64_t)j * s.t.b.cs; });
      __syncthreads();
      const int steps = (n + 31) / 32;
      for (int pr = pair0; busy && pr < npairs; pr += kWarps) {
        T acc[2 * KC];
#pragma unroll
        for (int q = 0; q < 2 * KC; ++q) acc[q] = T(0);
        for (int st = sub; st < steps; st += split * U) {
          if (!preloaded) load(x, pr, m0, st);
          preloaded = false;
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int c = 32 * (st + split * u) + lane;
            if (32 * (st + split * u) < n) {
              T w[KC];
              if (c < n)
                row_of<KC>(s.b + c * KC, w);
              else
#pragma unroll
                for (int j = 0; j < KC; ++j) w[j] = T(0);
#pragma unroll
              for (int j = 0; j < KC; ++j) {
                acc[j] += x[0][u] * w[j];
                acc[KC + j] += x[1][u] * w[j];
              }
            }
          }
        }
        preloaded = false;
        const T sum = warp_halve<T, 2 * KC>(acc, lane);
        constexpr int kRep = 32 / (2 * KC);  // lanes holding the same value
        if (lane % kRep == 0) {
          const int v = lane / kRep;
          T* dst = s.red + ((sub * 2 * npairs + 2 * pr) + v / KC) * KC + v % KC;
          *dst = m0 > 0 ? *dst + sum : sum;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
      const int e = threadIdx.x + o * kThreads, i = e % 64, j = e / 64;
      if (i < r && j < kc) {
        T sum = s.red[i * KC + j];
        for (int q = 1; q < split; ++q) sum += s.red[(q * 2 * npairs + i) * KC + j];
        __stcg(out + i + (int64_t)j * s.t.c.cs, old[o] + sum);
      }
    }
    __syncthreads();
  }
  return true;
}

template <class T, int KC>
__global__ void __launch_bounds__(kThreads, 2) solve_kernel(const __grid_constant__ SolveArgs a) {
  __shared__ __align__(16) SolveSmem<T, KC> s;
  int prob = 0;
  while (prob + 1 < a.nprobs && (int)blockIdx.x >= a.probs[prob + 1].cta0) ++prob;
  int left = a.nprobs;  // problems this CTA has not seen the end of
  for (;;) {
    if (threadIdx.x == 0) {
      int64_t ti = -1;
      if (!*((volatile int32_t*)a.status + 3))
        for (; left > 0; --left) {
          ti = (int64_t)atomicAdd(a.probs[prob].ticket, 1ULL);
          if (ti < a.probs[prob].ntasks) break;
          ti = -1;
          prob = prob + 1 < a.nprobs ? prob + 1 : 0;
        }
      s.task = ti;
      s.prob = prob;
    }
    __syncthreads();
    if (s.task < 0) break;
    const SolveProb& P = a.probs[s.prob];
    const int64_t ti = s.task;
    uint64_t t_claim = 0;
    if (a.trace && threadIdx.x == 0) t_claim = now_ns();
    if (threadIdx.x < sizeof(Task) / 4)
      reinterpret_cast<int32_t*>(&s.t)[threadIdx.x] = __ldg(reinterpret_cast<const int32_t*>(P.tasks + ti) + threadIdx.x);
    if (threadIdx.x >= 64 && threadIdx.x < 66) s.succ[threadIdx.x - 64] = __ldg(P.succ_ptr + ti + threadIdx.x - 64);
    __syncthreads();
    // every thread holds one of the first 256 successors
    const int64_t e0 = s.succ[0], e1 = s.succ[1];
    int32_t sx = -1;
    if (e0 + threadIdx.x < e1) sx = __ldg(P.succ_idx + e0 + threadIdx.x);
    bool ok;
    if (s.t.type == TK_PROJ)
      ok = run_proj<T, KC>(s, P, a);
    else if (s.t.type == TK_ROWMV)
      ok = s.t.c.rows <= 32 ? run_rowmv<T, KC, 1>(s, P, a) : run_rowmv<T, KC, 2>(s, P, a);
    else
      ok = wait_ready(s, P, a);
    if (!ok) break;
    __syncthreads();  // the task's stores come before the releases
    // one fence a thread, then plain reductions (a release per reduction waited
    // for the stores again every 32 successors)
    if (sx >= 0) {
      __threadfence();
      red_dec(P.indeg + sx);
      for (int64_t e = e0 + kThreads + threadIdx.x; e < e1; e += kThreads) red_dec(P.indeg + __ldg(P.succ_idx + e));
    }
    if (a.trace && threadIdx.x == 0) {
      unsigned long long* tr = a.trace + 4 * ti;
      tr[0] = ((unsigned long long)s.prob << 40) | (unsigned long long)ti;
      tr[1] = t_claim;
      tr[2] = s.start;
      tr[3] = now_ns();
    }
    __syncthreads();
  }
}

// counters, tickets and status of a launch
__global__ void k_solve_reset(const __grid_constant__ SolveArgs a) {
  const SolveProb& P = a.probs[blockIdx.y];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < P.ntasks; i += (int64_t)gridDim.x * blockDim.x)
    P.indeg[i] = P.indeg0[i];
  if (blockIdx.x == 0 && threadIdx.x == 0) *P.ticket = 0ULL;
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 8) a.status[threadIdx.x] = threadIdx.x == 1 ? -1 : 0;
}

template <class T, int KC>
cudaError_t launch(const SolveArgs& a, int64_t total, int sms, cudaStream_t s) {
  note_launch();
  k_solve_reset<<<dim3((unsigned)(1 + total / (8192 * a.nprobs)), a.nprobs), kThreads, 0, s>>>(a);
  note_launch();
  const int grid = (int)(total < 2 * sms ? total : 2 * sms);
  solve_kernel<T, KC><<<grid, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

// Right-hand sides carried in registers: 8 in FP32 (4 when no problem has
// more), 4 in FP64, whose accumulators take twice the registers.
template <class T>
cudaError_t solve_launch(SolveArgs& a, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  int64_t total = 0, before = 0;
  int32_t nrhs = 0;
  for (int i = 0; i < a.nprobs; ++i) {
    total += a.probs[i].ntasks;
    nrhs = a.probs[i].nrhs > nrhs ? a.probs[i].nrhs : nrhs;
  }
  if (total == 0) return cudaSuccess;
  // CTAs start on the problems in proportion to their tasks and move on when
  // a problem has none left to hand out
  const int64_t grid = total < 2 * sms ? total : 2 * sms;
  for (int i = 0; i < a.nprobs; ++i) {
    a.probs[i].cta0 = (int32_t)(before * grid / total);
    before += a.probs[i].ntasks;
  }
  if (sizeof(T) == 4 && nrhs > 4) return launch<T, sizeof(T) == 4 ? 8 : 4>(a, total, sms, s);
  return launch<T, 4>(a, total, sms, s);
}
template cudaError_t solve_launch<float>(SolveArgs&, cudaStream_t);
template cudaError_t solve_launch<double>(SolveArgs&, cudaStream_t);

}  // namespace hlu
