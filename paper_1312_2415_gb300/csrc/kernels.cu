// FP64 kernels of the two-site sweep (sm_103a).  Every launch executes a table built
// by the host planner; no kernel waits on another block or on another launch.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <limits>
#include <memory>
#include <mutex>
#include <new>
#include <stdexcept>
#include <string>
#include <type_traits>
#include <unordered_map>

#include "device.hpp"
#include "plans.hpp"

namespace dmrg {

namespace {

thread_local std::string g_err;
int64_t g_launches = 0;  // kernels launched by this library (all contexts)

inline cudaStream_t S(Stream s) { return (cudaStream_t)s; }

inline void ck(cudaError_t e, const char* what) {
  if (e != cudaSuccess) {
    g_err = std::string(what) + ": " + cudaGetErrorString(e);
    throw std::runtime_error(g_err);
  }
}

inline int nblk(int64_t n, int t) { return (int)std::min<int64_t>((n + t - 1) / t, 65535 * 8); }

}  // namespace

// ------------------------------------------------------------------ memory

// Device bytes the library holds (all contexts), and an optional cap on them: an
// allocation that would pass the cap fails on the host with std::bad_alloc (reported as
// DMRG_ENOMEM) before any CUDA call is made.
namespace {
std::mutex g_mem_mu;
std::unordered_map<void*, size_t> g_mem_live;
size_t g_mem_in_use = 0, g_mem_cap = 0;
}  // namespace

void* dev_alloc(size_t bytes, Stream s) {
  void* p = nullptr;
  if (bytes == 0) bytes = 16;
  {
    std::lock_guard<std::mutex> lk(g_mem_mu);
    if (g_mem_cap && g_mem_in_use + bytes > g_mem_cap) throw std::bad_alloc();
    g_mem_in_use += bytes;  // reserved before the call, released if it fails
  }
  cudaError_t e = cudaMallocAsync(&p, bytes, S(s));
  std::lock_guard<std::mutex> lk(g_mem_mu);
  if (e != cudaSuccess) {
    g_mem_in_use -= bytes;
    ck(e, "cudaMallocAsync");
  }
  g_mem_live[p] = bytes;
  return p;
}
void dev_free(void* p, Stream s) {
  if (!p) return;
  {
    std::lock_guard<std::mutex> lk(g_mem_mu);
    auto it = g_mem_live.find(p);
    if (it != g_mem_live.end()) {
      g_mem_in_use -= it->second;
      g_mem_live.erase(it);
    }
  }
  ck(cudaFreeAsync(p, S(s)), "cudaFreeAsync");
}
bool no_room(const std::exception& e) {
  if (dynamic_cast<const std::bad_alloc*>(&e)) return true;
  if (std::string(e.what()).find("out of memory") == std::string::npos) return false;
  cudaGetLastError();
  return true;
}
size_t dev_bytes_in_use() {
  std::lock_guard<std::mutex> lk(g_mem_mu);
  return g_mem_in_use;
}
void dev_set_cap(size_t bytes) {
  std::lock_guard<std::mutex> lk(g_mem_mu);
  g_mem_cap = bytes;
}
void dev_h2d(void* d, const void* h, size_t b, Stream s) {
  if (b) ck(cudaMemcpyAsync(d, h, b, cudaMemcpyHostToDevice, S(s)), "h2d");
}
void dev_d2h(void* h, const void* d, size_t b, Stream s) {
  if (b) ck(cudaMemcpyAsync(h, d, b, cudaMemcpyDeviceToHost, S(s)), "d2h");
}
void dev_d2d(void* d, const void* x, size_t b, Stream s) {
  if (b) ck(cudaMemcpyAsync(d, x, b, cudaMemcpyDeviceToDevice, S(s)), "d2d");
}
void dev_zero(void* p, size_t b, Stream s) {
  if (b) ck(cudaMemsetAsync(p, 0, b, S(s)), "memset");
}
void dev_sync(Stream s) { ck(cudaStreamSynchronize(S(s)), "stream sync"); }
int64_t kernel_launches() { return g_launches; }
void note_launches(int64_t k) { g_launches += k; }
int dev_check(const char** msg) {
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) return 0;
  g_err = cudaGetErrorString(e);
  if (msg) *msg = g_err.c_str();
  return (int)e;
}
void* host_pinned_alloc(size_t b) {
  void* p = nullptr;
  ck(cudaMallocHost(&p, b ? b : 16), "cudaMallocHost");
  return p;
}
void host_pinned_free(void* p) {
  if (p) cudaFreeHost(p);
}
void* event_create() {
  cudaEvent_t e;
  ck(cudaEventCreate(&e), "cudaEventCreate");
  return (void*)e;
}
void event_destroy(void* e) {
  if (e) cudaEventDestroy((cudaEvent_t)e);
}
void event_record(void* e, Stream s) { ck(cudaEventRecord((cudaEvent_t)e, S(s)), "cudaEventRecord"); }
Stream stream_create() {
  cudaStream_t s;
  ck(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking), "cudaStreamCreate");
  return (Stream)s;
}
void stream_destroy(Stream s) {
  if (s) cudaStreamDestroy(S(s));
}
void stream_wait(Stream s, void* ev) { ck(cudaStreamWaitEvent(S(s), (cudaEvent_t)ev, 0), "cudaStreamWaitEvent"); }
void event_sync(void* ev) { ck(cudaEventSynchronize((cudaEvent_t)ev), "cudaEventSynchronize"); }
float event_elapsed_ms(void* a, void* b) {
  float ms = 0.f;
  ck(cudaEventSynchronize((cudaEvent_t)b), "cudaEventSynchronize");
  ck(cudaEventElapsedTime(&ms, (cudaEvent_t)a, (cudaEvent_t)b), "cudaEventElapsedTime");
  return ms;
}

// ------------------------------------------------------------------ batched copies
//
// The vectors of a batch of small instances (some 14 KB each) are bound by the calls: a
// cudaMemcpyAsync each costs the host 7 us.  Up to 64 of them go with one launch, whose
// parameters are the table.  Measured (six Hubbard L=8 problems, whole call): 300 us with
// twelve copies, 263 us with two launches.

namespace {
struct CopyTable {
  CopyJob job[64];
};

__global__ void __launch_bounds__(256) k_copy_batched(const __grid_constant__ CopyTable t) {
  const CopyJob J = t.job[blockIdx.y];
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < J.n; i += (int64_t)gridDim.x * 256) J.dst[i] = J.src[i];
}

// One launch may do the jobs if the caller's pointers are aligned device memory and no job
// writes what another one reads or writes (an instance given twice, buffers of the batch
// passed as vectors): the launch has no order between jobs.
bool one_launch(const std::vector<CopyJob>& jobs) {
  struct Range {
    uintptr_t lo, hi;
    bool write;
  };
  std::vector<Range> r;
  for (const CopyJob& j : jobs) {
    if (((uintptr_t)j.dst | (uintptr_t)j.src) % sizeof(double)) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, j.user) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    if (a.type != cudaMemoryTypeDevice) return false;
    const uintptr_t d = (uintptr_t)j.dst, q = (uintptr_t)j.src, b = sizeof(double) * (size_t)j.n;
    r.push_back({d, d + b, true});
    r.push_back({q, q + b, false});
  }
  std::sort(r.begin(), r.end(), [](const Range& x, const Range& y) { return x.lo < y.lo; });
  uintptr_t read = 0, written = 0;  // ends of the ranges so far
  for (const Range& x : r) {
    if (x.lo < written || (x.write && x.lo < read)) return false;
    uintptr_t& end = x.write ? written : read;
    end = std::max(end, x.hi);
  }
  return true;
}
}  // namespace

void copy_batched(const std::vector<CopyJob>& jobs, Stream s) {
  if (!one_launch(jobs)) {
    for (const CopyJob& j : jobs) dev_d2d(j.dst, j.src, sizeof(double) * (size_t)j.n, s);
    return;
  }
  for (size_t b = 0; b < jobs.size(); b += 64) {
    CopyTable t{};
    const size_t n = std::min<size_t>(64, jobs.size() - b);
    int64_t most = 1;
    for (size_t i = 0; i < n; ++i) {
      t.job[i] = jobs[b + i];
      most = std::max(most, t.job[i].n);
    }
    const int grid = (int)std::min<int64_t>((most + 1023) / 1024, 1024);
    k_copy_batched<<<dim3(grid, (unsigned)n), 256, 0, S(s)>>>(t);
    ++g_launches;
  }
  ck(cudaGetLastError(), "batched copies");
}

// ------------------------------------------------------------------ grouped GEMM
//
// C_g += sum_t alpha_t op(A_t) op(B_t) over tables of thousands of small blocks (1 to ~150
// rows, tens to thousands of tasks per output).  An SM retires two FP64 FMAs per cycle, 16
// cycles for one warp's FMA, while L1 serves a warp's operand in 1 to 4: below about 160 rows
// neither register tiling nor staging in shared memory buys anything, but every idle lane,
// every wait on a chain of tasks and every further FP64 operation does cost.  So the output
// elements of a group are laid on lanes without padding to a tile: a lane owns R rows of one
// column (R = 1, 2 or 4, chosen per group so that the fewest lanes idle), the operands come
// straight from L1 / L2 with no barrier anywhere in the sum, and groups with long task lists
// are shared by 2 to 8 warps of a CTA, whose partial sums are added in a fixed order
// (deterministic, no atomics).  Larger groups go in staged tiles, short tables of long ordered
// lists in rounds (below).  Measured against staged tiles for every size (H_eff x, whole call):
// Hubbard L=8, D=64 769 -> 98 us; random L=12, D=500 17.4 -> 1.2 ms; random L=28, D=1500
// 281 -> 128 ms (0.90 TFLOP/s; cuBLAS DGEMM reaches 1.10 on large squares).  Four
// CTAs of 64 registers per SM against two of 128: phase 1 95 -> 83 ms, phase 2 39 -> 43 ms
// there.  The last one to three columns of a task are loaded together, not one at a time:
// phase 2 50 -> 39 ms.

namespace {
constexpr int kGemmWarps = 8, kGemmMinCtas = 4;

struct Remap {
  const char* lo[4];
  const char* hi[4];
  char* to[4];
};

__device__ __forceinline__ const double* remap_ptr(const double* p, const Remap& m) {
  const char* c = (const char*)p;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (c >= m.lo[k] && c < m.hi[k]) return (const double*)(m.to[k] + (c - m.lo[k]));
  return p;
}

// acc[r] = sum over tasks [t0, t1) of the element (row i0 + r, column j); rows past the
// group's last one read row i0 again (their sums are dropped by the caller).
//
// kOrdered: one chain of FMAs per element over the tasks and columns in table order with
// alpha multiplied into A first, whatever the job table: the products that steer a Davidson
// run (an unconverged one amplifies a rounding difference about a hundredfold per
// iteration) keep their bits when the work split changes.  alpha = +-1 needs no multiply;
// otherwise the warp scales each distinct element of A once, four columns at a time,
// through buf (its 128 doubles of shared memory), instead of once per lane that reads it.
// Otherwise each task is summed on its own and alpha applied to the sum.
template <int R, bool kRemap, bool kOrdered>
__device__ __forceinline__ void gemm_sum(const GemmTask* __restrict__ tasks, int t0, int t1, int i0, int j, int m,
                                         const Remap& rm, double* buf, double (&acc)[R]) {
  const int lane = threadIdx.x & 31;
  // rows the warp's lanes read: first row, count, and this lane's rows among them
  const int row0 = __reduce_min_sync(0xffffffffu, i0);
  const int nrow = kOrdered ? min(__reduce_max_sync(0xffffffffu, i0) + R, m) - row0 : 0;
  int ro[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    ro[r] = i0 + r < m ? i0 + r : i0;
    acc[r] = 0.0;
  }
  GemmTask T = tasks[t0 < t1 ? t0 : 0];
  for (int t = t0; t < t1; ++t) {
    const GemmTask cur = T;
    if (t + 1 < t1) T = tasks[t + 1];  // the next descriptor is in flight while this task runs
    const double* B = kRemap ? remap_ptr(cur.B, rm) : cur.B;
    if (cur.A == nullptr) {  // op(A) = identity
      const int64_t si = cur.transB ? 1 : cur.ldb, sj = cur.transB ? cur.ldb : 1;
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = fma(cur.alpha, B[ro[r] * si + j * sj], acc[r]);
      continue;
    }
    const double* A = kRemap ? remap_ptr(cur.A, rm) : cur.A;
    const int64_t sai = cur.transA ? 1 : cur.lda, sak = cur.transA ? cur.lda : 1;
    const int64_t sbk = cur.transB ? 1 : cur.ldb, sbj = cur.transB ? cur.ldb : 1;
    const double* pb = B + j * sbj;
    const bool unit = fabs(cur.alpha) == 1.0;
    if (kOrdered && !unit && nrow * 4 <= 128) {
      const int per = nrow > 0 ? nrow : 1;
      int k = cur.k;
      for (; k > 0; k -= 4) {
        double b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) b[u] = u < k ? pb[u * sbk] : 0.0;
        __syncwarp();
        for (int e = lane; e < nrow * 4; e += 32) {
          const int u = cur.transA ? e / per : e & 3, r = cur.transA ? e - u * per : e >> 2;
          if (u < k) buf[r * 4 + u] = A[(row0 + r) * sai + u * sak] * cur.alpha;
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (u < k) {
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fma(buf[(ro[r] - row0) * 4 + u], b[u], acc[r]);
          }
        pb += 4 * sbk;
        A += 4 * sak;
      }
      continue;
    }
    const double* pa[R];
    double s[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      pa[r] = A + ro[r] * sai;
      s[r] = kOrdered ? acc[r] : 0.0;
    }
    // What multiplies an element of A (ordered sums): alpha, or its sign moved to B.  The two
    // are separate loops: a multiplication behind a test inside the loop is issued whether it
    // is wanted or not, and costs as much as the FMA.  Measured (one loop / two): tables of
    // 16 to 150 rows with alpha = +-1 380..520 / 740..1210 GFLOP/s (shared sums the same);
    // phase 1 of random L=28, D=2500, sites 13, 14 after a step 231 / 105 ms, phase 2 174 / 77
    // ms (32 x 32 tiles staged in shared memory: 155 and 155 ms).
    const long long fb = kOrdered && unit && cur.alpha < 0.0 ? (long long)(1ull << 63) : 0ll;
    auto flip = [&](double v) { return __longlong_as_double(__double_as_longlong(v) ^ fb); };
    auto sum = [&](auto scale) {
      constexpr bool kScale = decltype(scale)::value;
      int k = cur.k;
      for (; k >= 4; k -= 4) {
        double b[4], a[R][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          b[u] = kOrdered && !kScale ? flip(pb[u * sbk]) : pb[u * sbk];
#pragma unroll
          for (int r = 0; r < R; ++r) a[r][u] = kScale ? pa[r][u * sak] * cur.alpha : pa[r][u * sak];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int r = 0; r < R; ++r) s[r] = fma(a[r][u], b[u], s[r]);
        pb += 4 * sbk;
#pragma unroll
        for (int r = 0; r < R; ++r) pa[r] += 4 * sak;
      }
      if (k > 0) {  // the last one to three columns, their loads in flight together
        double b[3], a[R][3];
#pragma unroll
        for (int u = 0; u < 3; ++u)
          if (!kOrdered || u < k) {
            const int o = kOrdered || u < k ? u : 0;  // shared sums: a repeated load for a branch
            b[u] = kOrdered && !kScale ? flip(pb[o * sbk]) : pb[o * sbk];
#pragma unroll
            for (int r = 0; r < R; ++r) a[r][u] = kScale ? pa[r][o * sak] * cur.alpha : pa[r][o * sak];
          }
#pragma unroll
        for (int u = 0; u < 3; ++u)
          if (u < k) {
#pragma unroll
            for (int r = 0; r < R; ++r) s[r] = fma(a[r][u], b[u], s[r]);
          }
      }
    };
    if (kOrdered && !unit) sum(std::true_type{});
    else sum(std::false_type{});
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = kOrdered ? s[r] : fma(cur.alpha, s[r], acc[r]);
  }
}

// The same ordered sum for long lists of small tasks, which are chains of FMAs (66 cycles
// each) behind trips to L2 and address arithmetic of some 2000 cycles per task when one warp
// does everything.  One CTA per 32-element slice, one row per lane: in each round
// kRoundWarps - 1 warps fetch one chunk each (up to four columns of one task; A scaled by
// alpha on the way) into shared memory while the last warp sums the previous round's chunks
// in order.  The chunks' table (task, first column) is made at upload.  Measured (phase 2, lanes
// / rounds): Hubbard L=8, D=64 165 / 47 us; random L=12, D=350 443 / 288 us, L=12, D=500 1.26 / 0.53
// ms.  Short lists (phase 1, one task per sum) start faster the other way (25 / 41 us), and so do
// tables that fill the SMs (OrderedCost).
constexpr int kRoundWarps = 8;

template <bool kRemap>
__global__ void __launch_bounds__(kRoundWarps * 32, 4)
    k_gemm_rounds(const GemmTask* __restrict__ tasks, const GemmGroup* __restrict__ groups,
                  const GemmChunk* __restrict__ chunks, const GemmJob* __restrict__ jobs, bool over, Remap rm) {
  constexpr int kF = kRoundWarps - 1;
  __shared__ double as[2][kF][4][32], bs[2][kF][4][32];
  __shared__ int ks[2][kF];       // columns of the chunk; 0: identity task
  __shared__ double al[2][kF];    // identity: alpha
  // the summing warp (number kF) sits on another SM sub-partition in every fourth CTA: its FMAs
  // are what fills an FP64 pipe
  const int warp = ((threadIdx.x >> 5) + blockIdx.x) % kRoundWarps, lane = threadIdx.x & 31;
  const GemmJob J = jobs[blockIdx.x];
  const GemmGroup g = groups[J.group];
  const int c0 = chunks[J.group].begin, nc = chunks[J.group].end - c0;  // the group's chunks
  const GemmChunk* list = chunks + c0;
  const int q = min(J.w0 * 32 + lane, g.m * g.n - 1), i = q / g.n, j = q % g.n;
  const int row0 = __reduce_min_sync(0xffffffffu, i), nrow = __reduce_max_sync(0xffffffffu, i) + 1 - row0;
  const int lr = i - row0, nr = (nc + kF - 1) / kF;
  double s = 0.0;
  GemmChunk cn{};  // this warp's chunk of the next round, fetched a round ahead
  GemmTask T{};
  if (warp < kF) {
    if (warp < nc) {
      cn = list[warp];
      T = tasks[cn.task];
    }
  }
  for (int r = 0; r <= nr; ++r) {
    const int buf = r & 1;
    if (warp < kF) {
      const int c = r * kF + warp;
      if (c < nc) {
        const int k0 = cn.k0;
        const GemmTask Q = T;
        if (c + kF < nc) {
          cn = list[c + kF];
          T = tasks[cn.task];
        }
        const double* B = kRemap ? remap_ptr(Q.B, rm) : Q.B;
        if (Q.A == nullptr) {
          bs[buf][warp][0][lane] = Q.transB ? B[j * (int64_t)Q.ldb + i] : B[i * (int64_t)Q.ldb + j];
          if (lane == 0) {
            ks[buf][warp] = 0;
            al[buf][warp] = Q.alpha;
          }
        } else {
          const double* A = kRemap ? remap_ptr(Q.A, rm) : Q.A;
          const int64_t sai = Q.transA ? 1 : Q.lda, sak = Q.transA ? Q.lda : 1;
          const int64_t sbk = Q.transB ? 1 : Q.ldb, sbj = Q.transB ? Q.ldb : 1;
          const double* pa = A + (row0 + min(lane, nrow - 1)) * sai + k0 * sak;
          const double* pb = B + j * sbj + k0 * sbk;
          const int k = min(4, Q.k - k0);
          double av[4], bv[4];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (u < k) {
              av[u] = pa[u * sak];
              bv[u] = pb[u * sbk];
            }
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (u < k) {
              as[buf][warp][u][lane] = __dmul_rn(av[u], Q.alpha);
              bs[buf][warp][u][lane] = bv[u];
            }
          if (lane == 0) ks[buf][warp] = k;
        }
      }
    } else if (r > 0) {
      const int pb = buf ^ 1, n = min(kF, nc - (r - 1) * kF);
      for (int c = 0; c < n; ++c) {
        const int k = ks[pb][c];
        if (k == 0) {
          s = fma(al[pb][c], bs[pb][c][0][lane], s);
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (u < k) s = fma(as[pb][c][u][lr], bs[pb][c][u][lane], s);
        }
      }
    }
    __syncthreads();
  }
  if (warp == kF && J.w0 * 32 + lane < g.m * g.n) {
    double* C = (kRemap ? (double*)remap_ptr(g.C, rm) : g.C) + (size_t)i * g.ldc + j;
    *C = over ? s : *C + s;
  }
}

// The same sums (one chain per element, alpha multiplied into A first) of large blocks: a CTA
// per 32 x 32 tile of C, the operands staged in shared memory sixteen columns at a time, 2 x 2
// elements per thread.  Lanes read a block of 200 rows and columns (some 0.4 MB) through L1 once
// per four rows of C; a tile reads it once per 32.  Padding to the tile is what it costs: by the
// rule at kTileMin few groups come here.  Measured (lanes / tiles, Hubbard L=16, D=2500 after a
// step, blocks of up to 245 rows): phase 1 677 / 585 ms, in Davidson 617 / 565 ms, the operator
// update 697 / 631 ms.
constexpr int kTileM = 32, kTileN = 32, kTileK = 16;

template <bool kRemap>
__global__ void __launch_bounds__(256)
    k_gemm_tiles(const GemmTask* __restrict__ tasks, const GemmGroup* __restrict__ groups, const GemmJob* __restrict__ jobs,
                 bool over, Remap rm) {
  __shared__ double As[kTileK][kTileM + 1];
  __shared__ double Bs[kTileK][kTileN + 1];
  const GemmJob J = jobs[blockIdx.x];
  const GemmGroup g = groups[J.group];
  const int tn = (g.n + kTileN - 1) / kTileN;
  const int row0 = (J.w0 / tn) * kTileM, col0 = (J.w0 % tn) * kTileN;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int t = g.task_begin; t < g.task_end; ++t) {
    const GemmTask T = tasks[t];
    const double* B = kRemap ? remap_ptr(T.B, rm) : T.B;
    if (T.A == nullptr) {  // op(A) = identity
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int r = row0 + ty + 16 * i, c = col0 + tx + 16 * j;
          if (r < g.m && c < g.n)
            acc[i][j] = fma(T.alpha, T.transB ? B[(size_t)c * T.ldb + r] : B[(size_t)r * T.ldb + c], acc[i][j]);
        }
      continue;
    }
    const double* A = kRemap ? remap_ptr(T.A, rm) : T.A;
    for (int k0 = 0; k0 < T.k; k0 += kTileK) {
#pragma unroll
      for (int u = 0; u < kTileM * kTileK / 256; ++u) {
        const int e = tid + 256 * u;
        const int kk = T.transA ? e / kTileM : e % kTileK, r = T.transA ? e % kTileM : e / kTileK;
        const int gr = row0 + r, gk = k0 + kk;
        double v = 0.0;
        if (gr < g.m && gk < T.k) v = T.transA ? A[(size_t)gk * T.lda + gr] : A[(size_t)gr * T.lda + gk];
        As[kk][r] = v * T.alpha;
      }
#pragma unroll
      for (int u = 0; u < kTileN * kTileK / 256; ++u) {
        const int e = tid + 256 * u;
        const int kk = T.transB ? e % kTileK : e / kTileN, c = T.transB ? e / kTileK : e % kTileN;
        const int gc = col0 + c, gk = k0 + kk;
        double v = 0.0;
        if (gc < g.n && gk < T.k) v = T.transB ? B[(size_t)gc * T.ldb + gk] : B[(size_t)gk * T.ldb + gc];
        Bs[kk][c] = v;
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < kTileK; ++kk) {
        const double a0 = As[kk][ty], a1 = As[kk][ty + 16];
        const double b0 = Bs[kk][tx], b1 = Bs[kk][tx + 16];
        acc[0][0] = fma(a0, b0, acc[0][0]);
        acc[0][1] = fma(a0, b1, acc[0][1]);
        acc[1][0] = fma(a1, b0, acc[1][0]);
        acc[1][1] = fma(a1, b1, acc[1][1]);
      }
      __syncthreads();
    }
  }
  double* C = kRemap ? (double*)remap_ptr(g.C, rm) : g.C;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = row0 + ty + 16 * i, c = col0 + tx + 16 * j;
      if (r < g.m && c < g.n) {
        double* p = C + (size_t)r * g.ldc + c;
        *p = over ? acc[i][j] : *p + acc[i][j];
      }
    }
}

// buf: 128 doubles per warp of the CTA
template <int R, bool kRemap, bool kOrdered>
__device__ __forceinline__ void gemm_job(const GemmTask* __restrict__ tasks, const GemmGroup& g, const GemmJob& J,
                                         const Remap& rm, double* buf, bool lead_only, bool over) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int slots = ((g.m + R - 1) / R) * g.n;
  const int nt = g.task_end - g.task_begin;
  const int t0 = g.task_begin + (int)((int64_t)nt * J.sidx / J.ns);
  const int t1 = g.task_begin + (int)((int64_t)nt * (J.sidx + 1) / J.ns);
  double* C = kRemap ? (double*)remap_ptr(g.C, rm) : g.C;
  // a shared sum's partial sums: R x 32 of every warp
  auto part = [&](int w) { return buf + w * 128; };
  for (int w = J.w0; w < J.w0 + J.nw; ++w) {
    const int slot = w * 32 + lane;
    const bool valid = slot < slots;
    const int q = valid ? slot : slots - 1;
    const int i0 = (q / g.n) * R, j = q % g.n;
    double acc[R];
    if (lead_only) {  // second call of a shared sum: this warp adds the other warps' parts
#pragma unroll
      for (int r = 0; r < R; ++r) {
        acc[r] = part(warp)[r * 32 + lane];
        for (int o = 1; o < J.ns; ++o) acc[r] += part(warp + o)[r * 32 + lane];
      }
    } else {
      gemm_sum<R, kRemap, kOrdered>(tasks, t0, t1, i0, j, g.m, rm, buf + warp * 128, acc);
      if (!kOrdered && J.ns > 1) {
#pragma unroll
        for (int r = 0; r < R; ++r) part(warp)[r * 32 + lane] = acc[r];
        return;
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (valid && i0 + r < g.m) {
        double* c = C + (size_t)(i0 + r) * g.ldc + j;
        *c = over ? acc[r] : *c + acc[r];
      }
  }
}

// one warp per job; the ns jobs of a shared sum are consecutive and never straddle CTAs
// (ordered sums are never shared)
template <bool kRemap, bool kOrdered>
__global__ void __launch_bounds__(kGemmWarps * 32, kGemmMinCtas)
    k_grouped_gemm(const GemmTask* __restrict__ tasks, const GemmGroup* __restrict__ groups,
                   const GemmJob* __restrict__ jobs, int njobs, bool over, Remap rm) {
  __shared__ double gemm_smem[kGemmWarps * 128];
  const int id = blockIdx.x * kGemmWarps + (threadIdx.x >> 5);
  GemmJob J{-1, 0, 0, 0, 0};
  GemmGroup g{};
  if (id < njobs) {
    J = jobs[id];
    g = groups[J.group];
  }
  for (int pass = 0; pass < (kOrdered ? 1 : 2); ++pass) {
    if (pass == 1) __syncthreads();
    if (J.group >= 0 && (pass == 0 || (J.ns > 1 && J.sidx == 0))) {
      if (g.rpl == 4) gemm_job<4, kRemap, kOrdered>(tasks, g, J, rm, gemm_smem, pass == 1, over);
      else if (g.rpl == 2) gemm_job<2, kRemap, kOrdered>(tasks, g, J, rm, gemm_smem, pass == 1, over);
      else gemm_job<1, kRemap, kOrdered>(tasks, g, J, rm, gemm_smem, pass == 1, over);
    }
  }
}

// Rows per lane of a group: the choice that leaves the fewest lanes idle, with a preference
// for more rows (fewer operand loads per FMA), stronger when lanes of neighbouring columns
// read B with a stride.
int rows_per_lane(int m, int n, bool strided_b) {
  int best = 1;
  double score = -1.0;
  for (int R : {4, 2, 1}) {
    const int64_t slots = (int64_t)((m + R - 1) / R) * n, warps = (slots + 31) / 32;
    const double eff = (double)m * n / ((double)warps * 32 * R);
    const double s = eff * (R == 4 ? 1.0 : R == 2 ? (strided_b ? 0.8 : 0.95) : (strided_b ? 0.5 : 0.85));
    if (s > score) { score = s; best = R; }
  }
  return best;
}

// Jobs of a table.  A job's work is counted in warp FMAs (plus a task's fixed cost); the
// target is what gives every SM about 40 jobs, at least kGemmMinWork so that a job is worth
// its start.  Groups above it are shared by up to max_ns warps, groups below it give one
// warp several of their 32-lane slices.  Longest jobs first.
constexpr int64_t kGemmMinWork = 48, kGemmJobsTarget = 152 * 40;
// Ordered sums in rounds: lists of at least kGemmRoundTasks tasks in the mean, in tables of at
// most kGemmMaxChunks chunks (their table costs the host 8 bytes and a pass each; the operator
// updates' lists, two to ten tasks in the mean, keep the FP64 pipes busy as they are: 10 ms in
// rounds, 6 ms without for one of random L=28, D=700), and of those the ones that the
// estimates below find shorter in rounds.  Rounds shorten the longest chain four- to tenfold but
// scale every chunk of A, so that they retire FMAs at half the rate of the lanes: they are for
// tables too small to fill the SMs.
constexpr int64_t kGemmRoundTasks = 12, kGemmMaxChunks = 1 << 21;

// Time of a table of ordered sums (cycles): what the FP64 pipes need for all of it (16 cycles
// of an SM per warp FMA) and the longest chain, which the start of the last CTAs and uneven
// SMs stretch.  Fitted to phase 2 of 30 tables, within 30 % but for the smallest; measured, lanes
// / rounds: Hubbard L=8, D=64 165 / 47 us, L=12, D=300 3.2 / 1.9 ms, L=16, D=200 0.97 / 0.50 ms,
// L=16, D=1000 15.7 / 28.5 ms and, a step on, 61 / 136 ms (staged tiles: 110 ms); random L=12,
// D=500 1.26 / 0.53 ms, L=16, D=600 0.88 / 1.01 ms and 1.49 / 1.08 ms, L=16, D=1500 2.3 / 2.9 ms,
// L=28, D=700 12.5 / 5.2 ms, L=28, D=1500 32 / 40 ms.
struct OrderedCost {
  double lane_fmas = 0.0, lane_chain = 0.0, round_fmas = 0.0, round_chain = 0.0;
  // slices: 32-lane slices of the group, in lanes (rpl rows each) and in rounds
  void add(int64_t lane_slices, int64_t slices, int rpl, int64_t tasks, int64_t columns, int64_t chunks) {
    lane_fmas += (double)lane_slices * rpl * columns;
    lane_chain = std::max(lane_chain, 1300.0 * tasks + 145.0 * rpl * columns);
    round_fmas += 8.0 * slices * chunks;  // four FMAs and the scaling of four columns of A
    round_chain = std::max(round_chain, 520.0 * chunks);
  }
  bool rounds() const {
    constexpr double kPipe = 16.0 / 152;
    return 1.35 * kPipe * round_fmas + round_chain < kPipe * lane_fmas + 1.3 * lane_chain;
  }
};

// Staged tiles: groups of at least kTileMin rows and columns of which padding to the tile (32 x
// 32, 16 columns of A) leaves at least kTileEff, in tables with at least kTileCount such tiles, four
// to five per place on the SMs.  Measured (none / from 160 / from 192 / from 224 rows): phase 1 of
// Hubbard L=16, D=2500 674 / 589 / 645 / 676 ms, its update 696 / 632 / 632 / 638 ms, the energy of
// swept random L=28, D=2500 677 / 656 / 675 ms; from 96 rows on the same within 2 %, but up to 6 %
// more for updates of Hubbard L=24, D=4000.  In tables of one product per symmetry sector (the
// refined eigensolver's, up to 202 rows) tiles are too few CTAs: dmrg_truncate of random L=28,
// D=1500 21.4 / 22.4 ms.
constexpr int kTileMin = 160;
constexpr double kTileEff = 0.8;
constexpr int64_t kTileCount = 152 * 32;

// ks: columns of a group's tasks in all; rpl: its rows per lane; max_ns: warps that may share a
// sum; max_nw: slices that a job may take.
std::vector<GemmJob> gemm_jobs(const std::vector<GemmGroup>& g, const std::vector<int64_t>& ks, const std::vector<int>& rpl,
                               int max_ns, int max_nw) {
  std::vector<int64_t> work(g.size(), 0);
  int64_t total = 0;
  for (size_t q = 0; q < g.size(); ++q) {
    const GemmGroup& G = g[q];
    if (ks[q] == 0) continue;
    work[q] = rpl[q] * ks[q] + 4 * (int64_t)(G.task_end - G.task_begin);
    total += work[q] * (((int64_t)((G.m + rpl[q] - 1) / rpl[q]) * G.n + 31) / 32);
  }
  const int64_t target = std::max(kGemmMinWork, total / kGemmJobsTarget);
  // buckets: by sharing warps (8, 4, 2, 1), then by decreasing powers of two of the work
  std::vector<GemmJob> bucket[4][48];
  for (size_t q = 0; q < g.size(); ++q) {
    const GemmGroup& G = g[q];
    if (work[q] == 0) continue;
    const int nt = G.task_end - G.task_begin;
    const int64_t slices = ((int64_t)((G.m + rpl[q] - 1) / rpl[q]) * G.n + 31) / 32;
    int ns = 1, b = 3;
    while (ns < max_ns && work[q] > ns * target && 2 * ns <= nt) { ns *= 2; --b; }
    const int64_t nw = ns > 1 ? 1 : std::min<int64_t>(max_nw, std::max<int64_t>(1, target / work[q]));
    int64_t w = work[q] * nw / ns;
    int lg = 0;
    while (w > 1) { w >>= 1; ++lg; }
    auto& out = bucket[b][47 - std::min(lg, 47)];
    for (int64_t s = 0; s < slices; s += nw)
      for (int i = 0; i < ns; ++i)
        out.push_back({(int)q, (int)s, (short)std::min<int64_t>(nw, slices - s), (unsigned char)i, (unsigned char)ns});
  }
  std::vector<GemmJob> jobs;
  for (auto& row : bucket)
    for (auto& v : row) jobs.insert(jobs.end(), v.begin(), v.end());
  return jobs;
}
}  // namespace

namespace {
// *rounds: the plan sums in rounds (also where the upload fails)
GemmPlan* plan_upload(const std::vector<GemmTask>& t, std::vector<GemmGroup>& g, Stream s, int sums, bool* rounds) {
  auto drop = [s](GemmPlan* q) {  // what there is of the plan, on every way out but the last
    try {
      gemm_plan_free(q, s);
    } catch (...) {
    }
  };
  std::unique_ptr<GemmPlan, decltype(drop)> hold(new GemmPlan, drop);
  GemmPlan* p = hold.get();
  p->ntasks = (int64_t)t.size();
  p->kinds = sums & (GEMM_ORDERED | GEMM_SHARED);
  p->overwrite = (sums & GEMM_OVERWRITE) != 0;
  // per group: columns and chunks in all, rows per lane, staged tiles (0: none)
  std::vector<int64_t> ks(g.size(), 0), chunk(g.size(), 0), tile(g.size(), 0);
  std::vector<int> rpl(g.size(), 1);
  const int forced = sums & (GEMM_LANES | GEMM_ROUNDS | GEMM_TILES);
  int64_t ntiles = 0;
  for (size_t q = 0; q < g.size(); ++q) {
    GemmGroup& G = g[q];
    if (G.m <= 0 || G.n <= 0) continue;
    bool strided = false;
    int64_t padded = 0;
    for (int k = G.task_begin; k < G.task_end; ++k) {
      const int cols = t[k].A ? t[k].k : 1;
      ks[q] += cols;
      chunk[q] += (cols + 3) / 4;
      padded += t[k].A ? (cols + kTileK - 1) / kTileK * kTileK : 1;
      strided = strided || (t[k].A && t[k].transB);
    }
    if (ks[q] == 0) continue;
    G.rpl = rpl[q] = rows_per_lane(G.m, G.n, strided);
    const int64_t nt = (int64_t)((G.m + kTileM - 1) / kTileM) * ((G.n + kTileN - 1) / kTileN);
    const bool large = G.m >= kTileMin && G.n >= kTileMin &&
                       (double)G.m * G.n * ks[q] >= kTileEff * kTileM * kTileN * nt * padded;
    if (forced ? forced == GEMM_TILES : large) ntiles += tile[q] = nt;
  }
  if (!forced && ntiles < kTileCount) ntiles = 0;
  // what goes where: tiles by decreasing powers of two of their columns; the other groups'
  // totals decide on rounds
  std::vector<GemmJob> tile_bucket[48];
  int64_t chunks = 0, live = 0, tasks = 0;
  OrderedCost cost;
  for (size_t q = 0; q < g.size(); ++q) {
    if (ks[q] == 0) continue;
    const GemmGroup& G = g[q];
    if (ntiles > 0 && tile[q] > 0) {
      int lg = 0;
      while (ks[q] >> (lg + 1)) ++lg;
      for (int64_t w = 0; w < tile[q]; ++w) tile_bucket[47 - std::min(lg, 47)].push_back({(int)q, (int)w, 1, 0, 1});
      ks[q] = 0;  // not in the job tables
      continue;
    }
    const int R = rpl[q];
    cost.add(((int64_t)((G.m + R - 1) / R) * G.n + 31) / 32, ((int64_t)G.m * G.n + 31) / 32, R,
             G.task_end - G.task_begin, ks[q], chunk[q]);
    chunks += chunk[q];
    tasks += G.task_end - G.task_begin;
    ++live;
  }
  std::vector<GemmJob> tiles;
  for (auto& v : tile_bucket) tiles.insert(tiles.end(), v.begin(), v.end());
  if (tiles.size() > (size_t)std::numeric_limits<int>::max())
    throw std::runtime_error("block-product table exceeds 2^31 jobs");
  p->rounds = (sums & GEMM_ORDERED) && tasks >= kGemmRoundTasks * live && chunks <= kGemmMaxChunks && cost.rounds();
  if (forced) p->rounds = forced == GEMM_ROUNDS;
  *rounds = p->rounds;
  const std::vector<int> one(p->rounds ? g.size() : 0, 1);  // rows per lane of the rounds
  for (int kind = 0; kind < 2; ++kind) {
    if (!(sums & (kind == 0 ? GEMM_ORDERED : GEMM_SHARED))) continue;
    const std::vector<GemmJob> jobs =
        gemm_jobs(g, ks, kind == 0 && p->rounds ? one : rpl, kind == 0 ? 1 : kGemmWarps,
                  kind == 0 && p->rounds ? 1 : 32767);
    if (jobs.size() > (size_t)std::numeric_limits<int>::max() - kGemmWarps)
      throw std::runtime_error("block-product table exceeds 2^31 jobs");
    p->njobs[kind] = (int)jobs.size();
    if (jobs.empty()) continue;
    p->jobs[kind] = (GemmJob*)dev_alloc(jobs.size() * sizeof(GemmJob), s);
    dev_h2d(p->jobs[kind], jobs.data(), jobs.size() * sizeof(GemmJob), s);
  }
  if (!tiles.empty()) {
    p->ntiles = (int)tiles.size();
    p->tiles = (GemmJob*)dev_alloc(tiles.size() * sizeof(GemmJob), s);
    dev_h2d(p->tiles, tiles.data(), tiles.size() * sizeof(GemmJob), s);
  }
  if (p->rounds) {
    // the groups' chunk ranges (begin, end), then the chunks (task, first column); the
    // ranges are relative to the table
    std::vector<GemmChunk> ch(g.size());
    for (size_t q = 0; q < g.size(); ++q) {
      ch[q].begin = (int)ch.size();
      if (ks[q] > 0)
        for (int k = g[q].task_begin; k < g[q].task_end; ++k)
          for (int k0 = 0; k0 < (t[k].A ? t[k].k : 1); k0 += 4) ch.push_back(GemmChunk{{k}, {k0}});
      ch[q].end = (int)ch.size();
    }
    p->chunks = (GemmChunk*)dev_alloc(std::max<size_t>(ch.size(), 1) * sizeof(GemmChunk), s);
    dev_h2d(p->chunks, ch.data(), ch.size() * sizeof(GemmChunk), s);
  }
  if (!t.empty()) {
    p->tasks = (GemmTask*)dev_alloc(t.size() * sizeof(GemmTask), s);
    dev_h2d(p->tasks, t.data(), t.size() * sizeof(GemmTask), s);
  }
  if (!g.empty()) {
    p->groups = (GemmGroup*)dev_alloc(g.size() * sizeof(GemmGroup), s);
    dev_h2d(p->groups, g.data(), g.size() * sizeof(GemmGroup), s);
  }
  return hold.release();
}
}  // namespace

GemmPlan* gemm_plan_upload(const std::vector<GemmTask>& t, std::vector<GemmGroup>& g, Stream s, int sums) {
  bool rounds = false;
  try {
    return plan_upload(t, g, s, sums, &rounds);
  } catch (const std::exception& e) {
    if (!rounds || (sums & GEMM_ROUNDS) || !no_room(e)) throw;
  }
  return plan_upload(t, g, s, sums | GEMM_LANES, &rounds);  // no room for the chunks (same bits)
}

namespace {
template <bool kRemap>
void gemm_launch(const GemmPlan* p, const Remap& rm, int sums, Stream s) {
  const int kind = sums == GEMM_ORDERED ? 0 : 1;
  if (p && !(p->kinds & sums)) throw std::logic_error("block products run with sums they were not uploaded for");
  if (!p) return;
  if (p->ntiles > 0) {
    k_gemm_tiles<kRemap><<<p->ntiles, 256, 0, S(s)>>>(p->tasks, p->groups, p->tiles, p->overwrite, rm);
    ++g_launches;
  }
  const int n = p->njobs[kind], grid = (n + kGemmWarps - 1) / kGemmWarps;
  const GemmJob* jobs = p->jobs[kind];
  if (n > 0) {
    if (kind == 0 && p->rounds)
      k_gemm_rounds<kRemap><<<n, kRoundWarps * 32, 0, S(s)>>>(p->tasks, p->groups, p->chunks, jobs, p->overwrite, rm);
    else if (kind == 0)
      k_grouped_gemm<kRemap, true><<<grid, kGemmWarps * 32, 0, S(s)>>>(p->tasks, p->groups, jobs, n, p->overwrite, rm);
    else
      k_grouped_gemm<kRemap, false><<<grid, kGemmWarps * 32, 0, S(s)>>>(p->tasks, p->groups, jobs, n, p->overwrite, rm);
    ++g_launches;
  }
  ck(cudaGetLastError(), "grouped_gemm launch");
}
}  // namespace

void gemm_plan_run(const GemmPlan* p, Stream s, int sums) { gemm_launch<false>(p, Remap{}, sums, s); }

void gemm_plan_free(GemmPlan* p, Stream s) {
  if (!p) return;
  dev_free(p->tasks, s);
  dev_free(p->groups, s);
  dev_free(p->jobs[0], s);
  dev_free(p->jobs[1], s);
  dev_free(p->chunks, s);
  dev_free(p->tiles, s);
  delete p;
}

int64_t gemm_plan_tasks(const GemmPlan* p) { return p ? p->ntasks : 0; }

// ------------------------------------------------------------------ combine

namespace {
// One warp per destination block (most have 4 to 150 elements), its sources four at a time:
// descriptors first, then their elements, so that a chain of sources is not a chain of
// loads.  The sum itself stays in source order.  Measured (W sums of random L=12, D=500: 0.33
// million blocks; L=16, D=600: 1.1 million): a 128-thread CTA per block 250 / 661 us, now
// 129 / 315 us.
constexpr int kCombWarps = 8;

template <bool kRemap>
__global__ void __launch_bounds__(kCombWarps * 32) k_combine(const CombSrc* __restrict__ src, const CombDst* __restrict__ dst,
                                                            int ndst, int wpd, Remap rm) {
  const int w = blockIdx.x * kCombWarps + (threadIdx.x >> 5), id = w / wpd;
  if (id >= ndst) return;
  const CombDst d = dst[id];
  double* out = kRemap ? (double*)remap_ptr(d.dst, rm) : d.dst;
  const int n = d.rows * d.cols;
  for (int e = (w - id * wpd) * 32 + (threadIdx.x & 31); e < n; e += 32 * wpd) {
    const int r = e / d.cols, c = e - r * d.cols;
    double v = d.accumulate ? out[(size_t)r * d.ld + c] : 0.0;
    int s = d.src_begin;
    for (; s + 4 <= d.src_end; s += 4) {
      CombSrc q[4];
      double x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) q[u] = src[s + u];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = (kRemap ? remap_ptr(q[u].src, rm) : q[u].src)[(size_t)r * q[u].ld + c];
#pragma unroll
      for (int u = 0; u < 4; ++u) v += q[u].alpha * x[u];
    }
    for (; s < d.src_end; ++s) {
      const CombSrc q = src[s];
      v += q.alpha * (kRemap ? remap_ptr(q.src, rm) : q.src)[(size_t)r * q.ld + c];
    }
    out[(size_t)r * d.ld + c] = v;
  }
}

template <bool kRemap>
void combine_launch(const CombPlan* p, const Remap& rm, Stream s) {
  if (!p || p->ndst == 0) return;
  // warps per block: one where the blocks fill the GPU, a CTA's eight for short tables
  const int wpd = p->ndst >= 152 * 64 ? 1 : kCombWarps;
  const int64_t grid = ((int64_t)p->ndst * wpd + kCombWarps - 1) / kCombWarps;
  k_combine<kRemap><<<(unsigned)grid, kCombWarps * 32, 0, S(s)>>>(p->src, p->dst, p->ndst, wpd, rm);
  ++g_launches;
  ck(cudaGetLastError(), "combine launch");
}
}  // namespace

CombPlan* comb_plan_upload(const std::vector<CombSrc>& s, const std::vector<CombDst>& d, Stream st) {
  CombPlan* p = new CombPlan;
  p->ndst = (int)d.size();
  if (!s.empty()) {
    p->src = (CombSrc*)dev_alloc(s.size() * sizeof(CombSrc), st);
    dev_h2d(p->src, s.data(), s.size() * sizeof(CombSrc), st);
  }
  if (!d.empty()) {
    p->dst = (CombDst*)dev_alloc(d.size() * sizeof(CombDst), st);
    dev_h2d(p->dst, d.data(), d.size() * sizeof(CombDst), st);
  }
  return p;
}

void comb_plan_run(const CombPlan* p, Stream s) { combine_launch<false>(p, Remap{}, s); }

void comb_plan_free(CombPlan* p, Stream s) {
  if (!p) return;
  dev_free(p->src, s);
  dev_free(p->dst, s);
  delete p;
}

// ------------------------------------------------------------------ diagonal

namespace {
__global__ void k_diag(const DiagTerm* __restrict__ t, const DiagOut* __restrict__ o) {
  const DiagOut d = o[blockIdx.x];
  const int64_t n = (int64_t)d.dL * d.dR;
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {
    int a = (int)(e / d.dR), b = (int)(e % d.dR);
    double v = d.out[e];
    for (int s = d.term_begin; s < d.term_end; ++s)
      v += t[s].coef * t[s].C[(size_t)a * t[s].ldc + a] * t[s].D[(size_t)b * t[s].ldd + b];
    d.out[e] = v;
  }
}
}  // namespace

DiagPlan* diag_plan_upload(const std::vector<DiagTerm>& t, const std::vector<DiagOut>& o, Stream s) {
  DiagPlan* p = new DiagPlan;
  p->n = (int)o.size();
  if (!t.empty()) {
    p->t = (DiagTerm*)dev_alloc(t.size() * sizeof(DiagTerm), s);
    dev_h2d(p->t, t.data(), t.size() * sizeof(DiagTerm), s);
  }
  if (!o.empty()) {
    p->o = (DiagOut*)dev_alloc(o.size() * sizeof(DiagOut), s);
    dev_h2d(p->o, o.data(), o.size() * sizeof(DiagOut), s);
  }
  return p;
}

void diag_plan_run(const DiagPlan* p, Stream s) {
  if (!p || p->n == 0) return;
  for (int off = 0; off < p->n; off += 65535) {
    int n = std::min(65535, p->n - off);
    k_diag<<<n, 128, 0, S(s)>>>(p->t, p->o + off);
    ++g_launches;
  }
  ck(cudaGetLastError(), "diag launch");
}

void diag_plan_free(DiagPlan* p, Stream s) {
  if (!p) return;
  dev_free(p->t, s);
  dev_free(p->o, s);
  delete p;
}

// ------------------------------------------------------------------ grouped Frobenius products

namespace {
// one CTA per group: the threads stride over every element of every task of the group,
// then a block reduction; the group's output is written by this CTA only
__global__ void __launch_bounds__(256) k_dot_grouped(const DotTask* __restrict__ t,
                                                    const DotGroup* __restrict__ g) {
  const DotGroup G = g[blockIdx.x];
  double s = 0.0;
  for (int k = G.task_begin; k < G.task_end; ++k) {
    const DotTask T = t[k];
    const int64_t ne = (int64_t)T.rows * T.cols;
    double u = 0.0;
    for (int64_t e = threadIdx.x; e < ne; e += blockDim.x) {
      const int r = (int)(e / T.cols), c = (int)(e % T.cols);
      u = fma(T.A[(size_t)r * T.lda + c], T.B[(size_t)r * T.ldb + c], u);
    }
    s = fma(T.alpha, u, s);
  }
  __shared__ double sh[256];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *G.out += sh[0];
}

// Gamma_ijkl = 2 x mean of dg over (ijkl), (jilk), (klij), (lkji), (kjil), (ilkj), (lijk), (jkli)
__global__ void k_rdm2(const double* __restrict__ dg, int L, double* __restrict__ Gamma) {
  const int64_t L4 = (int64_t)L * L * L * L;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < L4; e += (int64_t)gridDim.x * blockDim.x) {
    const int l = (int)(e % L), k = (int)(e / L % L), j = (int)(e / L / L % L), i = (int)(e / L / L / L);
    auto at = [&](int a, int b, int c, int d) { return dg[(((int64_t)a * L + b) * L + c) * L + d]; };
    const double s = at(i, j, k, l) + at(j, i, l, k) + at(k, l, i, j) + at(l, k, j, i) + at(k, j, i, l) +
                     at(i, l, k, j) + at(l, i, j, k) + at(j, k, l, i);
    Gamma[e] = 0.25 * s;
  }
}

__global__ void k_rdm1(const double* __restrict__ Gamma, int L, int N, double* __restrict__ gamma) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= L * L) return;
  const int i = e / L, k = e % L;
  double s = 0.0;
  for (int j = 0; j < L; ++j) s += Gamma[(((int64_t)i * L + j) * L + k) * L + j];
  gamma[e] = s / (N - 1);
}
}  // namespace

void dot_grouped(const std::vector<DotTask>& t, const std::vector<DotGroup>& g, Stream s) {
  if (g.empty()) return;
  DotTask* dt = (DotTask*)dev_alloc(std::max<size_t>(t.size(), 1) * sizeof(DotTask), s);
  DotGroup* dgp = (DotGroup*)dev_alloc(g.size() * sizeof(DotGroup), s);
  if (!t.empty()) dev_h2d(dt, t.data(), t.size() * sizeof(DotTask), s);
  dev_h2d(dgp, g.data(), g.size() * sizeof(DotGroup), s);
  for (size_t off = 0; off < g.size(); off += 65535) {
    const int n = (int)std::min<size_t>(65535, g.size() - off);
    k_dot_grouped<<<n, 256, 0, S(s)>>>(dt, dgp + off);
    ++g_launches;
  }
  ck(cudaGetLastError(), "dot launch");
  dev_free(dt, s);
  dev_free(dgp, s);
}

void rdm_finish(const double* dg, int L, int N, double* gamma, double* Gamma, Stream s) {
  const int64_t L4 = (int64_t)L * L * L * L;
  k_rdm2<<<(int)std::min<int64_t>((L4 + 255) / 256, 4096), 256, 0, S(s)>>>(dg, L, Gamma);
  k_rdm1<<<(L * L + 255) / 256, 256, 0, S(s)>>>(Gamma, L, N, gamma);
  g_launches += 2;
  ck(cudaGetLastError(), "rdm launch");
}

// ------------------------------------------------------------------ vector kernels

namespace {
constexpr int kDotChunk = 4096;
constexpr int kMaxChunks = 512;

__global__ void k_multidot_partial(const double* __restrict__ V, int64_t ldv,
                                   const double* __restrict__ w, int64_t n, int nch,
                                   double* __restrict__ part) {
  __shared__ double sh[256];
  const int j = blockIdx.y, c = blockIdx.x;
  const double* v = V + (size_t)j * ldv;
  double s = 0.0;
  for (int64_t i = (int64_t)c * 256 + threadIdx.x; i < n; i += (int64_t)nch * 256) s += v[i] * w[i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[(size_t)j * nch + c] = sh[0];  // the result itself when nch == 1
}

__global__ void k_multidot_final(const double* __restrict__ part, int nch, int m, double* out) {
  const int j = blockIdx.x;
  __shared__ double sh[256];
  double s = 0.0;
  for (int c = threadIdx.x; c < nch; c += 256) s += part[(size_t)j * nch + c];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[j] = sh[0];
}

__global__ void k_vec_combine(const double* __restrict__ V, int64_t ldv, int m,
                              const double* __restrict__ c, double beta, double* __restrict__ y,
                              int64_t n) {
  __shared__ double cs[128];
  for (int j = threadIdx.x; j < m; j += blockDim.x) cs[j] = c[j];
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double s = beta == 0.0 ? 0.0 : beta * y[i];
    for (int j = 0; j < m; ++j) s += cs[j] * V[(size_t)j * ldv + i];
    y[i] = s;
  }
}

__global__ void k_axpby(double a, const double* __restrict__ x, double b, double* __restrict__ y,
                        int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] = a * x[i] + (b == 0.0 ? 0.0 : b * y[i]);
}

__global__ void k_normalize(double* __restrict__ y, const double* __restrict__ nrm2, int64_t n) {
  double s = *nrm2 > 0.0 ? 1.0 / sqrt(*nrm2) : 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] *= s;
}

// One Davidson iteration's elementwise work, fused (each was three to five launches of 2 to 3
// us over vectors that fit in L2; the same operations per element in the same order).
// x = sum_j c_j V_j, r = sum_j c_j AV_j - theta x, t = r / (theta - d), the denominator floored
__global__ void k_ritz(const double* __restrict__ V, const double* __restrict__ AV, int64_t ldv, int m,
                       const double* __restrict__ c, const double* __restrict__ theta, const double* __restrict__ d,
                       double* __restrict__ x, double* __restrict__ r, double* __restrict__ t, int64_t n) {
  __shared__ double cs[128];
  for (int j = threadIdx.x; j < m; j += blockDim.x) cs[j] = c[j];
  __syncthreads();
  const double th = *theta;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double xs = 0.0, rs = 0.0;
#pragma unroll 4
    for (int j = 0; j < m; ++j) {
      xs += cs[j] * V[(size_t)j * ldv + i];
      rs += cs[j] * AV[(size_t)j * ldv + i];
    }
    x[i] = xs;
    rs = fma(-th, xs, rs);
    r[i] = rs;
    double den = th - d[i];
    if (fabs(den) < 1e-12) den = den < 0 ? -1e-12 : 1e-12;
    t[i] = rs / den;
  }
}

// t -= sum_j c_j V_j
__global__ void k_project_out(const double* __restrict__ V, int64_t ldv, int m, const double* __restrict__ c,
                              double* __restrict__ t, int64_t n) {
  __shared__ double cs[128];
  for (int j = threadIdx.x; j < m; j += blockDim.x) cs[j] = c[j];
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
#pragma unroll 4
    for (int j = 0; j < m; ++j) s += cs[j] * V[(size_t)j * ldv + i];
    t[i] = t[i] - s;
  }
}

// a = b = t / sqrt(*nrm2)
__global__ void k_normalize2(const double* __restrict__ t, const double* __restrict__ nrm2, double* __restrict__ a,
                             double* __restrict__ b, int64_t n) {
  const double s = *nrm2 > 0.0 ? 1.0 / sqrt(*nrm2) : 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double v = t[i] * s;
    a[i] = v;
    b[i] = v;
  }
}

__device__ inline void sym_schur2(double app, double aqq, double apq, double& c, double& s) {
  if (apq == 0.0) { c = 1.0; s = 0.0; return; }
  double th = (aqq - app) / (2.0 * apq);
  double t = (th >= 0 ? 1.0 : -1.0) / (fabs(th) + sqrt(1.0 + th * th));
  c = 1.0 / sqrt(1.0 + t * t);
  s = t * c;
}

// round-robin pairing of np (even) indices: pair r of a step
__device__ __forceinline__ void rr_pair(int r, int step, int np, int& p, int& q) {
  const int b = np - 1 - r;
  p = r == 0 ? 0 : 1 + (r - 1 + step) % (np - 1);
  q = 1 + (b - 1 + step) % (np - 1);
  if (p > q) { const int t = p; p = q; q = t; }
}

// ---- one sweep of cyclic FP64 Jacobi on a matrix in shared memory, by a CTA of 256 threads
//
// A step's rotations are a chain of three divisions and two square roots (3000 cycles), its
// row and column updates 6 n^2 FP64 operations (3 n^2 cycles of an SM).  The two overlap: a
// step first updates the 2 x 2 blocks J_r^T A J_u that hold the next step's pairs, then one
// warp computes the next rotations while the others update the rest of A and Q.  Every
// element sees the same operations in the same order as with one barrier between rotations,
// rows and columns, so the results are the same to the bit.
struct JacobiBuf {
  double cs[2][32], sn[2][32];
  int pp[2][32], qq[2][32];
  unsigned crit[32];  // per row pair: the column pairs whose block is updated first
};

// pair of element x in a step's round-robin pairing
__device__ __forceinline__ int rr_pair_of(int x, int step, int np) {
  int pos = 0;
  if (x > 0) {
    pos = x - 1 - step % (np - 1);
    pos = 1 + (pos < 0 ? pos + np - 1 : pos);
  }
  return pos < np / 2 ? pos : np - 1 - pos;
}

// rot(p, q, next, c, s): the rotation of pair (p, q), p < q; next: of the following sweep
template <class Rot>
__device__ __forceinline__ void jacobi_rotations(JacobiBuf& S, int buf, int step, int np, int r, bool next, Rot rot) {
  int p, q;
  rr_pair(r, step, np, p, q);
  double c = 1.0, s = 0.0;
  rot(p, q, next, c, s);
  S.cs[buf][r] = c;
  S.sn[buf][r] = s;
  S.pp[buf][r] = p;
  S.qq[buf][r] = q;
}

// A (np x np, np even, at most 64), Q (m rows, np columns), row stride ld; the rotations of
// step 0 are in S[buf] on entry, those of the next sweep's step 0 on return (if `more`).
// Called by all 256 threads, a barrier behind the rotations; ends with a barrier.
template <class Rot>
__device__ void jacobi_sweep(double* A, double* Q, int ld, int np, int m, JacobiBuf& S, int& buf, bool more, Rot rot) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nr = np / 2, ns = np - 1;
  const bool early = nr >= 4;  // below, two pairs can share a block
  for (int step = 0; step < ns; ++step) {
    const bool last = step + 1 == ns;
    const int next = last ? 0 : step + 1;
    const double* cs = S.cs[buf];
    const double* sn = S.sn[buf];
    const int* pp = S.pp[buf];
    const int* qq = S.qq[buf];
    if (tid < nr) S.crit[tid] = 0u;
    __syncthreads();
    // the blocks of the next step's pairs: the diagonal ones and the one holding (p', q'),
    // four lanes per block (one element each)
    if (early && tid < 8 * nr) {
      const int b = tid >> 2, o = tid & 3;
      int r = b, u = b;
      if (b >= nr) {
        int p, q;
        rr_pair(b - nr, next, np, p, q);
        r = rr_pair_of(p, step, np);
        u = rr_pair_of(q, step, np);
      }
      const double cr = cs[r], sr = sn[r], cu = cs[u], su = sn[u];
      const int p = pp[r] * ld, q = qq[r] * ld, v = pp[u], w = qq[u];
      const double a0 = A[p + v], a1 = A[p + w], b0 = A[q + v], b1 = A[q + w];
      double x0, x1;  // row p or q after the row rotation
      if (o < 2) {
        x0 = cr * a0 - sr * b0;
        x1 = cr * a1 - sr * b1;
      } else {
        x0 = sr * a0 + cr * b0;
        x1 = sr * a1 + cr * b1;
      }
      const double z = (o & 1) ? su * x0 + cu * x1 : cu * x0 - su * x1;
      __syncwarp(0xfu << (lane & ~3));  // the block's four lanes have all read before one writes
      A[(o < 2 ? p : q) + ((o & 1) ? w : v)] = z;
      if (o == 0) atomicOr(&S.crit[r], 1u << u);
    }
    __syncthreads();
    if (early && warp == 0 && lane < nr && (more || !last)) jacobi_rotations(S, buf ^ 1, next, np, lane, last, rot);
    // the other blocks and Q (an FP64 instruction costs the same for one lane as for 32):
    // up to 16 pairs packed onto the lanes of the warps on the other sub-partitions, more
    // with lane = column pair on every warp but the rotating one
    auto block = [&](int r, int u) {
      const double cr = cs[r], sr = sn[r], cu = cs[u], su = sn[u];
      if (((S.crit[r] >> u) & 1u) || (sr == 0.0 && su == 0.0)) return;
      const int p = pp[r] * ld, q = qq[r] * ld, v = pp[u], w = qq[u];
      const double a0 = A[p + v], a1 = A[p + w], b0 = A[q + v], b1 = A[q + w];
      const double x0 = cr * a0 - sr * b0, x1 = cr * a1 - sr * b1;
      const double y0 = sr * a0 + cr * b0, y1 = sr * a1 + cr * b1;
      A[p + v] = cu * x0 - su * x1;
      A[p + w] = su * x0 + cu * x1;
      A[q + v] = cu * y0 - su * y1;
      A[q + w] = su * y0 + cu * y1;
    };
    auto column = [&](int i, int u) {
      const double c = cs[u], t = sn[u];
      if (t == 0.0) return;
      double* row = Q + i * ld;
      const int v = pp[u], w = qq[u];
      const double a0 = row[v], a1 = row[w];
      row[v] = c * a0 - t * a1;
      row[w] = t * a0 + c * a1;
    };
    if (nr <= 16) {
      if (!early || (warp & 3) != 0) {
        const int nt = early ? 192 : 256, t0 = (early ? (warp < 4 ? warp - 1 : warp - 2) : warp) * 32 + lane;
        const unsigned inv = 65536u / nr + 1;  // e / nr = e * inv >> 16 for e < 65536 / nr
        for (int e = t0; e < nr * nr; e += nt) {
          const int r = (int)(e * inv >> 16);
          block(r, e - r * nr);
        }
        for (int e = t0; e < nr * m; e += nt) {
          const int i = (int)(e * inv >> 16);
          column(i, e - i * nr);
        }
      }
    } else if (warp > 0 && lane < nr) {
      for (int r = warp - 1; r < nr; r += 7) block(r, lane);
      for (int i = warp - 1; i < m; i += 7) column(i, lane);
    }
    __syncthreads();
    if (!early && (more || !last)) {
      if (tid < nr) jacobi_rotations(S, buf ^ 1, next, np, tid, last, rot);
      __syncthreads();
    }
    buf ^= 1;
  }
}

// Lowest k eigenpairs of the m x m Rayleigh matrix (m <= kSeMax) by cyclic Jacobi, one CTA
// of 256 threads.  Measured (mean call of a Hubbard L=8, D=32 solve): phase by phase 339 us,
// overlapped 215 us.
constexpr int kSeMax = 48, kSeLd = 49;

struct SmallEigMem {
  double A[kSeMax * kSeLd], Q[kSeMax * kSeLd], red[16];
  JacobiBuf j;
  int order[kSeMax], tie;
};

__device__ void small_eig_block(const double* __restrict__ G, int gld, int m, int k, double* __restrict__ theta,
                                double* __restrict__ C) {
  __shared__ SmallEigMem S;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int np = (m + 1) & ~1, nr = np / 2;
  for (int e = tid; e < np * np; e += blockDim.x) {
    const int i = e / np, j = e % np;
    const bool in = i < m && j < m;
    S.A[i * kSeLd + j] = !in ? 0.0 : i >= j ? G[(size_t)i * gld + j] : G[(size_t)j * gld + i];  // lower triangle
    S.Q[i * kSeLd + j] = (i == j) ? 1.0 : 0.0;
  }
  __syncthreads();
  auto rot = [&](int p, int q, bool, double& c, double& s) {
    if (q < m) sym_schur2(S.A[p * kSeLd + p], S.A[q * kSeLd + q], S.A[p * kSeLd + q], c, s);
  };
  int buf = 0;
  if (tid < nr) jacobi_rotations(S.j, 0, 0, np, tid, false, rot);
  __syncthreads();
  for (int sweep = 0; sweep < 60 && m > 1; ++sweep) {
    // off-diagonal against total
    double off = 0.0, tot = 0.0;
    for (int e = tid; e < m * m; e += blockDim.x) {
      const int i = e / m, j = e % m;
      const double v = S.A[i * kSeLd + j];
      tot += v * v;
      if (i != j) off += v * v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if (lane == 0) {
      S.red[warp] = off;
      S.red[8 + warp] = tot;
    }
    __syncthreads();
    off = tot = 0.0;
    for (int w = 0; w < 8; ++w) {
      off += S.red[w];
      tot += S.red[8 + w];
    }
    if (off <= 1e-30 * tot || off == 0.0) break;  // the same sums in every thread
    jacobi_sweep(S.A, S.Q, kSeLd, np, m, S.j, buf, true, rot);
  }
  __syncthreads();
  // ascending order of the diagonal; equal and unordered values (NaN) as an exchange sort
  // leaves them, so that `order` is a permutation whatever the matrix holds
  if (tid == 0) S.tie = 0;
  __syncthreads();
  if (tid < m) {
    const double vi = S.A[tid * kSeLd + tid];
    int rank = 0;
    for (int j = 0; j < m; ++j) {
      const double vj = S.A[j * kSeLd + j];
      rank += vj < vi;
      if (!(vj < vi) && !(vj > vi) && j != tid) S.tie = 1;
    }
    S.order[rank] = tid;
  }
  __syncthreads();
  if (S.tie && tid == 0) {
    auto d = [&](int i) { return S.A[S.order[i] * kSeLd + S.order[i]]; };
    for (int i = 0; i < m; ++i) S.order[i] = i;
    for (int i = 0; i < m; ++i)
      for (int j = i + 1; j < m; ++j)
        if (d(j) < d(i)) {
          const int t = S.order[i];
          S.order[i] = S.order[j];
          S.order[j] = t;
        }
  }
  __syncthreads();
  for (int e = tid; e < k * m; e += blockDim.x) C[(size_t)(e / m) * m + e % m] = S.Q[(e % m) * kSeLd + S.order[e / m]];
  if (tid < k) theta[tid] = S.A[S.order[tid] * kSeLd + S.order[tid]];
}

__global__ void k_small_eig(const double* __restrict__ G, int gld, int m, int k,
                            double* __restrict__ theta, double* __restrict__ C) {
  small_eig_block(G, gld, m, k, theta, C);
}

// ---- grouped Davidson kernels: one launch per operation over all instances of a batch
// (blockIdx.y or blockIdx.x = instance); instances with act[i] == 0 are skipped.

__device__ __forceinline__ double* bd_pick(const BdSlot& s, int which, int col) {
  switch (which) {
    case BD_V: return s.V + (int64_t)col * s.n;
    case BD_AV: return s.AV + (int64_t)col * s.n;
    case BD_R: return s.r;
    case BD_T: return s.t;
    case BD_X: return s.x;
    case BD_X0: return s.x0;
    case BD_TMP: return s.tmp + (int64_t)col * s.n;
    case BD_BX: return s.bx;
    default: return s.by;
  }
}

// part[(j nch + c)] = partial sums of <A col (a_col + j), B>, j < m (grid: nch x m x count)
__global__ void k_bd_dots_partial(const BdSlot* __restrict__ sl, const int* __restrict__ act, int aw, int a_col,
                                  int bw, int b_col, int nch) {
  __shared__ double sh[256];
  const int i = blockIdx.z, j = blockIdx.y, c = blockIdx.x;
  if (!act[i]) return;
  const BdSlot s = sl[i];
  const double* a = bd_pick(s, aw, a_col + j);
  const double* b = bd_pick(s, bw, b_col);
  double v = 0.0;
  for (int64_t e = (int64_t)c * 256 + threadIdx.x; e < s.n; e += (int64_t)nch * 256) v += a[e] * b[e];
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) s.part[(size_t)j * nch + c] = sh[0];
}

// out[j] = sum of the partials; out = G + row * mmax (to_g) or dots (grid: m x count)
__global__ void k_bd_dots_final(const BdSlot* __restrict__ sl, const int* __restrict__ act, int nch, int to_g,
                                int row, int mmax) {
  __shared__ double sh[256];
  const int i = blockIdx.y, j = blockIdx.x;
  if (!act[i]) return;
  const BdSlot s = sl[i];
  double v = 0.0;
  for (int c = threadIdx.x; c < nch; c += 256) v += s.part[(size_t)j * nch + c];
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) (to_g ? s.G + (size_t)row * mmax : s.dots)[j] = sh[0];
}

// y = beta y + sum_j c[j] V col j, c = C + cv * m (from_c) or dots
__global__ void k_bd_combine(const BdSlot* __restrict__ sl, const int* __restrict__ act, int vw, int m, int from_c,
                             int cv, double beta, int yw, int y_col) {
  __shared__ double cs[64];
  const int i = blockIdx.y;
  if (!act[i]) return;
  const BdSlot s = sl[i];
  const double* c = from_c ? s.C + (size_t)cv * m : s.dots;
  for (int j = threadIdx.x; j < m; j += blockDim.x) cs[j] = c[j];
  __syncthreads();
  const double* V = bd_pick(s, vw, 0);
  double* y = bd_pick(s, yw, y_col);
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < s.n; e += (int64_t)gridDim.x * blockDim.x) {
    double v = beta == 0.0 ? 0.0 : beta * y[e];
    for (int j = 0; j < m; ++j) v += cs[j] * V[(size_t)j * s.n + e];
    y[e] = v;
  }
}

// y = a x + b y; a = -theta[0] when a_theta
__global__ void k_bd_axpby(const BdSlot* __restrict__ sl, const int* __restrict__ act, int a_theta, double a, int xw,
                           int x_col, double b, int yw, int y_col) {
  const int i = blockIdx.y;
  if (!act[i]) return;
  const BdSlot s = sl[i];
  const double av = a_theta ? -s.th[0] : a;
  const double* x = bd_pick(s, xw, x_col);
  double* y = bd_pick(s, yw, y_col);
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < s.n; e += (int64_t)gridDim.x * blockDim.x)
    y[e] = av * x[e] + (b == 0.0 ? 0.0 : b * y[e]);
}

// y /= sqrt(dots[0])
__global__ void k_bd_normalize(const BdSlot* __restrict__ sl, const int* __restrict__ act, int yw, int y_col) {
  const int i = blockIdx.y;
  if (!act[i]) return;
  const BdSlot s = sl[i];
  const double sc = s.dots[0] > 0.0 ? 1.0 / sqrt(s.dots[0]) : 0.0;
  double* y = bd_pick(s, yw, y_col);
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < s.n; e += (int64_t)gridDim.x * blockDim.x)
    y[e] *= sc;
}

// t = r / (theta[0] - diag), |denominator| floored as in the single-instance kernel
__global__ void k_bd_precondition(const BdSlot* __restrict__ sl, const int* __restrict__ act) {
  const int i = blockIdx.y;
  if (!act[i]) return;
  const BdSlot s = sl[i];
  const double th = s.th[0];
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < s.n; e += (int64_t)gridDim.x * blockDim.x) {
    double den = th - s.diag[e];
    if (fabs(den) < 1e-12) den = den < 0 ? -1e-12 : 1e-12;
    s.t[e] = s.r[e] / den;
  }
}

__global__ void k_bd_small_eig(const BdSlot* __restrict__ sl, const int* __restrict__ act, int mmax, int m, int k) {
  const int i = blockIdx.x;
  if (!act[i]) return;
  const BdSlot s = sl[i];
  small_eig_block(s.G, mmax, m, k, s.th, s.C);
}

// restart: G = diag(theta[0..k)) (zero elsewhere)
__global__ void k_bd_restart_g(const BdSlot* __restrict__ sl, const int* __restrict__ act, int mmax, int k) {
  const int i = blockIdx.x;
  if (!act[i]) return;
  const BdSlot s = sl[i];
  for (int e = threadIdx.x; e < mmax * mmax; e += blockDim.x) {
    const int r = e / mmax, c = e % mmax;
    s.G[e] = (r == c && r < k) ? s.th[r] : 0.0;
  }
}

__global__ void k_bd_gather(const BdSlot* __restrict__ sl, int count, double* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    out[2 * i] = sl[i].th[0];
    out[2 * i + 1] = sl[i].dots[0];
  }
}

// x = -x where <x, x0> (dots[0]) < 0
__global__ void k_bd_sign(const BdSlot* __restrict__ sl, const int* __restrict__ act) {
  const int i = blockIdx.y;
  if (!act[i]) return;
  const BdSlot s = sl[i];
  if (!(s.dots[0] < 0.0)) return;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < s.n; e += (int64_t)gridDim.x * blockDim.x)
    s.x[e] = -s.x[e];
}

__device__ inline uint64_t splitmix(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

__global__ void k_noise(double* x, int64_t n, double amp, uint64_t seed) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t u = splitmix(seed + (uint64_t)i) >> 11;
    double r = (double)u * (2.0 / 9007199254740992.0) - 1.0;
    x[i] += amp * r;
  }
}
}  // namespace

void vec_multidot(const double* V, int64_t ldv, int m, const double* w, int64_t n, double* out,
                  double* scratch, Stream s) {
  if (m <= 0) return;
  int nch = (int)std::min<int64_t>(kMaxChunks, std::max<int64_t>(1, (n + kDotChunk - 1) / kDotChunk));
  dim3 grid(nch, m);
  k_multidot_partial<<<grid, 256, 0, S(s)>>>(V, ldv, w, n, nch, nch == 1 ? out : scratch);
  ++g_launches;
  if (nch > 1) {
    k_multidot_final<<<m, 256, 0, S(s)>>>(scratch, nch, m, out);
    ++g_launches;
  }
  ck(cudaGetLastError(), "multidot");
}

void vec_combine(const double* V, int64_t ldv, int m, const double* c, double beta, double* y,
                 int64_t n, Stream s) {
  k_vec_combine<<<nblk(n, 256), 256, 0, S(s)>>>(V, ldv, m, c, beta, y, n);
  ++g_launches;
  ck(cudaGetLastError(), "vec_combine");
}

void vec_axpby(double a, const double* x, double b, double* y, int64_t n, Stream s) {
  k_axpby<<<nblk(n, 256), 256, 0, S(s)>>>(a, x, b, y, n);
  ++g_launches;
  ck(cudaGetLastError(), "axpby");
}

void vec_normalize(double* y, const double* nrm2, int64_t n, Stream s) {
  k_normalize<<<nblk(n, 256), 256, 0, S(s)>>>(y, nrm2, n);
  ++g_launches;
  ck(cudaGetLastError(), "normalize");
}

void vec_ritz(const double* V, const double* AV, int64_t ldv, int m, const double* c, const double* theta, const double* d,
              double* x, double* r, double* t, int64_t n, Stream s) {
  k_ritz<<<nblk(n, 128), 128, 0, S(s)>>>(V, AV, ldv, m, c, theta, d, x, r, t, n);
  ++g_launches;
  ck(cudaGetLastError(), "ritz");
}

void vec_project_out(const double* V, int64_t ldv, int m, const double* c, double* t, int64_t n, Stream s) {
  k_project_out<<<nblk(n, 128), 128, 0, S(s)>>>(V, ldv, m, c, t, n);
  ++g_launches;
  ck(cudaGetLastError(), "project out");
}

void vec_normalize2(const double* t, const double* nrm2, double* a, double* b, int64_t n, Stream s) {
  k_normalize2<<<nblk(n, 256), 256, 0, S(s)>>>(t, nrm2, a, b, n);
  ++g_launches;
  ck(cudaGetLastError(), "normalize2");
}

namespace {
inline int bd_blocks(int64_t nmax, int count) {
  // enough CTAs per instance to fill the GPU a few times over, no more than the data needs
  const int per = (int)std::max<int64_t>(1, std::min<int64_t>((nmax + 255) / 256, std::max(1, 2048 / std::max(count, 1))));
  return per;
}
}  // namespace

void bd_dots(const BdSlot* sl, const int* act, int count, int64_t nmax, int aw, int a_col, int m, int bw, int b_col,
             int to_g, int row, int mmax, Stream s) {
  if (m <= 0 || count <= 0) return;
  const int nch = (int)std::min<int64_t>(kBdChunks, std::max<int64_t>(1, (nmax + 256 * 8 - 1) / (256 * 8)));
  k_bd_dots_partial<<<dim3(nch, m, count), 256, 0, S(s)>>>(sl, act, aw, a_col, bw, b_col, nch);
  ++g_launches;
  k_bd_dots_final<<<dim3(m, count), 256, 0, S(s)>>>(sl, act, nch, to_g, row, mmax);
  ++g_launches;
  ck(cudaGetLastError(), "grouped dots");
}

void bd_combine(const BdSlot* sl, const int* act, int count, int64_t nmax, int vw, int m, int from_c, int cv,
                double beta, int yw, int y_col, Stream s) {
  if (count <= 0) return;
  k_bd_combine<<<dim3(bd_blocks(nmax, count), count), 256, 0, S(s)>>>(sl, act, vw, m, from_c, cv, beta, yw, y_col);
  ++g_launches;
  ck(cudaGetLastError(), "grouped combine");
}

void bd_axpby(const BdSlot* sl, const int* act, int count, int64_t nmax, int a_theta, double a, int xw, int x_col,
              double b, int yw, int y_col, Stream s) {
  if (count <= 0) return;
  k_bd_axpby<<<dim3(bd_blocks(nmax, count), count), 256, 0, S(s)>>>(sl, act, a_theta, a, xw, x_col, b, yw, y_col);
  ++g_launches;
  ck(cudaGetLastError(), "grouped axpby");
}

void bd_normalize(const BdSlot* sl, const int* act, int count, int64_t nmax, int yw, int y_col, Stream s) {
  if (count <= 0) return;
  k_bd_normalize<<<dim3(bd_blocks(nmax, count), count), 256, 0, S(s)>>>(sl, act, yw, y_col);
  ++g_launches;
  ck(cudaGetLastError(), "grouped normalize");
}

void bd_precondition(const BdSlot* sl, const int* act, int count, int64_t nmax, Stream s) {
  if (count <= 0) return;
  k_bd_precondition<<<dim3(bd_blocks(nmax, count), count), 256, 0, S(s)>>>(sl, act);
  ++g_launches;
  ck(cudaGetLastError(), "grouped precondition");
}

void bd_small_eig(const BdSlot* sl, const int* act, int count, int mmax, int m, int k, Stream s) {
  if (count <= 0) return;
  k_bd_small_eig<<<count, 256, 0, S(s)>>>(sl, act, mmax, m, k);
  ++g_launches;
  ck(cudaGetLastError(), "grouped small eig");
}

void bd_restart_g(const BdSlot* sl, const int* act, int count, int mmax, int k, Stream s) {
  if (count <= 0) return;
  k_bd_restart_g<<<count, 256, 0, S(s)>>>(sl, act, mmax, k);
  ++g_launches;
  ck(cudaGetLastError(), "grouped restart");
}

void bd_gather(const BdSlot* sl, int count, double* out, Stream s) {
  if (count <= 0) return;
  k_bd_gather<<<(count + 127) / 128, 128, 0, S(s)>>>(sl, count, out);
  ++g_launches;
  ck(cudaGetLastError(), "grouped gather");
}

void bd_sign(const BdSlot* sl, const int* act, int count, int64_t nmax, Stream s) {
  if (count <= 0) return;
  k_bd_sign<<<dim3(bd_blocks(nmax, count), count), 256, 0, S(s)>>>(sl, act);
  ++g_launches;
  ck(cudaGetLastError(), "grouped sign");
}

void small_eig(const double* G, int gld, int m, int k, double* theta, double* C, Stream s) {
  k_small_eig<<<1, 256, 0, S(s)>>>(G, gld, m, k, theta, C);
  ++g_launches;
  ck(cudaGetLastError(), "small_eig");
}

void vec_add_noise(double* x, int64_t n, double amp, uint64_t seed, Stream s) {
  k_noise<<<nblk(n, 256), 256, 0, S(s)>>>(x, n, amp, seed);
  ++g_launches;
  ck(cudaGetLastError(), "noise");
}

// ------------------------------------------------------------------ batched Jacobi

namespace {
// device arrays of one call, released on every way out of it
struct DevScratch {
  Stream s;
  std::vector<void*> p;
  explicit DevScratch(Stream st) : s(st) {}
  DevScratch(const DevScratch&) = delete;
  template <class T>
  T* get(size_t n) {
    p.push_back(nullptr);
    p.back() = dev_alloc(sizeof(T) * n, s);
    return (T*)p.back();
  }
  ~DevScratch() {
    for (void* q : p) {
      try {
        dev_free(q, s);
      } catch (...) {
      }
    }
  }
};

constexpr int kEigSmemN = 64;  // blocks up to this size are diagonalised in shared memory

// Cyclic Jacobi (round-robin pairing, n/2 rotations per step) on one symmetric block per
// CTA, the matrix and the eigenvectors in shared memory.  Measured (135 blocks, 63 of 64 rows
// the largest, random L=28, D=700): phase by phase 35.2 ms, overlapped (jacobi_sweep) 22.4 ms.
// A pair is rotated only while |a_pq| exceeds
// 1e-16 sqrt(|a_pp a_qq|) plus an absolute floor; the loop ends after a sweep without
// rotations (at most 40 sweeps).  Output: eigenvalues descending, eigenvectors as
// columns of J.Q.
template <int NT>
__global__ void __launch_bounds__(NT) k_eig_batched(const EigJob* __restrict__ jobs) {
  static_assert(NT == 256, "jacobi_sweep");
  const EigJob J = jobs[blockIdx.x];
  const int n = J.n, tid = threadIdx.x;
  extern __shared__ double sm[];
  const int np = (n + 1) & ~1, ld = np + 1;
  double* A = sm;
  double* Q = sm + (size_t)np * ld;
  double* wtmp = Q + (size_t)np * ld;
  __shared__ JacobiBuf S;
  __shared__ int nrot[2];
  for (int e = tid; e < np * np; e += NT) {
    const int i = e / np, j = e % np;
    A[i * ld + j] = i < n && j < n ? J.A[(size_t)i * n + j] : 0.0;
    Q[i * ld + j] = i == j ? 1.0 : 0.0;
  }
  if (tid < 2) nrot[tid] = 0;
  __syncthreads();
  double scale = 0.0;
  for (int i = 0; i < n; ++i) scale = fmax(scale, fabs(A[(size_t)i * ld + i]));
  const double floor_abs = 1e-300 + 1e-18 * scale;
  int cur = 0, buf = 0;  // the current sweep's counter
  auto rot = [&](int p, int q, bool next, double& c, double& s) {
    if (q >= n) return;
    const double app = A[p * ld + p], aqq = A[q * ld + q], apq = A[p * ld + q];
    if (fabs(apq) > 1e-16 * sqrt(fabs(app * aqq)) + floor_abs) {
      sym_schur2(app, aqq, apq, c, s);
      atomicAdd(&nrot[next ? cur ^ 1 : cur], 1);
    }
  };
  if (n > 1) {
    if (tid < np / 2) jacobi_rotations(S, 0, 0, np, tid, false, rot);
    __syncthreads();
    for (int sweep = 0; sweep < 40; ++sweep) {
      jacobi_sweep(A, Q, ld, np, n, S, buf, sweep < 39, rot);
      if (nrot[cur] == 0) break;
      __syncthreads();
      if (tid == 0) nrot[cur] = 0;
      cur ^= 1;
      __syncthreads();
    }
  }
  // eigenpairs sorted descending (ties by index)
  for (int i = tid; i < n; i += NT) wtmp[i] = A[(size_t)i * ld + i];
  __syncthreads();
  const double* Qs = Q;
  for (int i = tid; i < n; i += NT) {
    double vi = wtmp[i];
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      double vj = wtmp[j];
      if (vj > vi || (vj == vi && j < i)) ++rank;
    }
    J.w[rank] = vi;
    for (int rr = 0; rr < n; ++rr) J.Q[(size_t)rr * n + rank] = Qs[(size_t)rr * ld + i];
  }
}
}  // namespace

// ------------------------------------------------------------------ parallel block Jacobi

namespace {
// Cyclic Jacobi in FP32 on the np x np matrix A (np even, at most 64, row stride ld) in
// shared memory, the rotations accumulated into Q, by a CTA of 256 threads: at most `sweeps`
// sweeps, ended by one without an off-diagonal above floor_abs (pairs are rotated from a
// tenth of that on).  A step has two barriers: one warp computes the
// rotations, then every thread updates whole 2 x 2 blocks J_r^T A J_u (lane = pair u, warps
// stride over r, four blocks' loads in flight) and columns of Q.
__device__ void jacobi_f32(float* A, float* Q, int np, int ld, int sweeps, float floor_abs, float* cs, float* sn, int* pp,
                           int* qq, int* flag) {
  const int tid = threadIdx.x, nr = np / 2, lane = tid & 31, warp = tid >> 5;
  for (int sweep = 0; sweep < sweeps; ++sweep) {
    if (tid == 0) *flag = 0;
    __syncthreads();
    for (int step = 0; step < np - 1; ++step) {
      if (tid < nr) {
        int p, q;
        rr_pair(tid, step, np, p, q);
        const float app = A[p * ld + p], aqq = A[q * ld + q], apq = A[p * ld + q];
        float c = 1.0f, s = 0.0f;
        if (fabsf(apq) > 0.1f * floor_abs) {
          const float th = __fdividef(aqq - app, 2.0f * apq), at = fabsf(th);
          const float t = copysignf(at < 1e18f ? __fdividef(1.0f, at + sqrtf(fmaf(at, at, 1.0f))) : 0.0f, th);
          c = rsqrtf(fmaf(t, t, 1.0f));
          s = t * c;
          if (fabsf(apq) > floor_abs) *flag = 1;
        }
        cs[tid] = c; sn[tid] = s; pp[tid] = p; qq[tid] = q;
      }
      __syncthreads();
      if (lane < nr) {
        const float cu = cs[lane], su = sn[lane];
        const int v = pp[lane], w = qq[lane];
#pragma unroll 4
        for (int r = warp; r < nr; r += 8) {
          const float cr = cs[r], sr = sn[r];
          const int p = pp[r] * ld, q = qq[r] * ld;
          const float a0 = A[p + v], a1 = A[p + w], b0 = A[q + v], b1 = A[q + w];
          const float x0 = cr * a0 - sr * b0, x1 = cr * a1 - sr * b1, y0 = sr * a0 + cr * b0, y1 = sr * a1 + cr * b1;
          A[p + v] = cu * x0 - su * x1;
          A[p + w] = r == lane ? 0.0f : su * x0 + cu * x1;
          A[q + v] = r == lane ? 0.0f : cu * y0 - su * y1;
          A[q + w] = su * y0 + cu * y1;
        }
#pragma unroll 8
        for (int i = warp; i < np; i += 8) {  // columns of Q
          float* row = Q + i * ld;
          const float a0 = row[v], a1 = row[w];
          row[v] = cu * a0 - su * a1;
          row[w] = su * a0 + cu * a1;
        }
      }
      __syncthreads();
    }
    if (!*flag) break;
    __syncthreads();
  }
}
}  // namespace

namespace {
// Symmetric eigensolver for the large Gram blocks (n above the shared-memory limit): a
// two-sided block Jacobi.  Rows and columns are grouped in blocks of 32; each step of
// a round-robin tournament pairs the blocks, and for every pair (I, J) the 64 x 64
// diagonal sub-block G[I+J, I+J] is diagonalised in shared memory (cyclic Jacobi),
// giving V.  One launch applies V^T to the rows I+J of every pair (the pairs' rows are
// disjoint), the next applies V to the columns I+J of G and of Q (disjoint columns):
// together G <- W^T G W with W the block rotation of the step.  At convergence the
// eigenvalues are the diagonal of G and the eigenvectors the columns of Q; the
// absolute accuracy is ~eps |G|, that of the Gram route.
constexpr int kOB = 32;   // rows per block
constexpr int kOP = 64;   // rows per pair
constexpr int kOL = 65;   // shared-memory row stride (doubles)

template <class T>
struct BjJob {
  T* A;           // n x n symmetric (the Gram matrix), diagonalised in place
  T* Q;           // n x n accumulated rotations (eigenvectors as columns)
  double* w;      // n eigenvalues (output, descending)
  int n, nb;      // nb = number of row blocks, even
  int pair_begin; // first CTA of this job in a step launch
  int pad;
};

// cyclic Jacobi on a 64 x 64 symmetric matrix A (shared memory, stride kOL),
// eigenvectors accumulated into V (identity on entry), all 256 threads; a pair is
// rotated while |a_pq| > 1e-16 sqrt|a_pp a_qq| + floor_abs, for one sweep: the outer
// iteration returns to every pair until it is diagonal, and inner sweeps beyond the first
// cost more than they save (measured: 1 sweep 1.4-1.9x faster than 3, 2.1-2.7x than 5,
// at the same accuracy)
__device__ void cta_jacobi64(double* A, double* V, JacobiBuf& S, double floor_abs) {
  auto rot = [&](int p, int q, bool, double& c, double& s) {
    const double app = A[p * kOL + p], aqq = A[q * kOL + q], apq = A[p * kOL + q];
    if (fabs(apq) > 1e-16 * sqrt(fabs(app * aqq)) + floor_abs) sym_schur2(app, aqq, apq, c, s);
  };
  int buf = 0;
  if (threadIdx.x < kOP / 2) jacobi_rotations(S, 0, 0, kOP, threadIdx.x, false, rot);
  __syncthreads();
  jacobi_sweep(A, V, kOL, kOP, kOP, S, buf, false, rot);
}

// out(64 x 64 tile) = op(X) op(Y) with a 4 x 4 register tile per thread; X, Y in shared
// memory with stride kOL; tx / ty: transpose flags
template <bool TX, bool TY, class T>
__device__ __forceinline__ void tile64(const T* X, const T* Y, T (&acc)[4][4]) {
  const int ti = threadIdx.x >> 4, tj = threadIdx.x & 15;
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = T(0);
  for (int k = 0; k < kOP; ++k) {
    T x[4], y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      x[u] = TX ? X[k * kOL + ti * 4 + u] : X[(ti * 4 + u) * kOL + k];
      y[u] = TY ? Y[(tj * 4 + u) * kOL + k] : Y[k * kOL + tj * 4 + u];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[u][v] = fma(x[u], y[v], acc[u][v]);
  }
}

template <class T>
__device__ __forceinline__ int find_job(const BjJob<T>* jobs, int njobs) {
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].pair_begin <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

template <class T>
__device__ __forceinline__ void pair_rows(const BjJob<T>& J, int r, int step, int* idx) {
  const int a = r, b = J.nb - 1 - r;
  const int p = a == 0 ? 0 : 1 + (a - 1 + step) % (J.nb - 1);
  const int q = b == 0 ? 0 : 1 + (b - 1 + step) % (J.nb - 1);
  if (threadIdx.x < kOP) {
    const int blk = threadIdx.x < kOB ? p : q, row = blk * kOB + (threadIdx.x % kOB);
    idx[threadIdx.x] = row < J.n ? row : -1;
  }
}

// Q = identity, and the largest |diagonal| of A per job (the noise scale eps |G|)
__global__ void k_bj_prep(const BjJob<double>* __restrict__ jobs, double* __restrict__ gmax) {
  const BjJob<double> J = jobs[blockIdx.x];
  const int n = J.n;
  for (int64_t e = threadIdx.x; e < (int64_t)n * n; e += blockDim.x) J.Q[e] = (e / n == e % n) ? 1.0 : 0.0;
  double best = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) best = fmax(best, fabs(J.A[(size_t)i * n + i]));
  __shared__ double red[256];
  red[threadIdx.x] = best;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]);
    __syncthreads();
  }
  if (threadIdx.x == 0) gmax[blockIdx.x] = red[0];
}

// What the two element types ask of a pair: an off-diagonal above rel sqrt|g_ii g_jj| +
// abs |G| sends it to the inner solver (|G| = the largest diagonal entry).  FP64: below that
// it is rounding noise of the rotations (~eps sqrt(64) |G|) and moves the eigenvalues only at
// second order; the absolute part must stay above the inner solver's floor, or pairs of
// null-space directions would be sent back to it forever.  FP32 (passes whose result is
// refined): the pass's floor alone.
template <class T>
struct BjTol;
template <>
struct BjTol<double> {
  static constexpr double rel = 1e-14, abs = 1e-14;
};
template <>
struct BjTol<float> {
  static constexpr double rel = 0.0, abs = 1.0;  // gmax carries the pass's floor
};

__device__ __forceinline__ void bj_inner(double* S, double* V, JacobiBuf& B, int*, double gmax) {
  cta_jacobi64(S, V, B, 1e-16 * gmax);  // floor below the outer one
}
__device__ __forceinline__ void bj_inner(float* S, float* V, JacobiBuf& B, int* nrot, double gmax) {
  jacobi_f32(S, V, kOP, kOL, 1, (float)(BjTol<float>::abs * gmax), (float*)B.cs, (float*)B.sn, B.pp[0], B.qq[0], nrot);
}

// step, part 1: V of every pair from its diagonal sub-block (one CTA per pair)
template <class T>
__global__ void __launch_bounds__(256) k_bj_rows(const BjJob<T>* __restrict__ jobs, int njobs, int step,
                                                 const double* __restrict__ gmax, T* __restrict__ vbuf,
                                                 int* __restrict__ flag, int* __restrict__ nrot) {
  extern __shared__ double bsm[];
  T* S = reinterpret_cast<T*>(bsm);  // sub-block, then diagonalised
  T* V = S + kOP * kOL;              // its eigenvectors
  __shared__ JacobiBuf jb;
  __shared__ int idx[kOP], inner_rot, need;
  const int lo = find_job(jobs, njobs);
  const BjJob<T> J = jobs[lo];
  const int r = blockIdx.x - J.pair_begin, tid = threadIdx.x, n = J.n;
  if (r >= J.nb / 2 || step >= J.nb - 1) {
    if (tid == 0) flag[blockIdx.x] = 0;
    return;
  }
  pair_rows(J, r, step, idx);
  if (tid == 0) need = 0;
  __syncthreads();
  const T rel = (T)BjTol<T>::rel, fl = (T)(BjTol<T>::abs * gmax[lo]);
  for (int e = tid; e < kOP * kOP; e += 256) {
    const int i = e >> 6, j = e & 63;
    S[i * kOL + j] = (idx[i] >= 0 && idx[j] >= 0) ? J.A[(size_t)idx[i] * n + idx[j]] : T(0);
  }
  __syncthreads();
  for (int e = tid; e < kOP * kOP; e += 256) {
    const int i = e >> 6, j = e & 63;
    if (i < j && fabs(S[i * kOL + j]) > rel * sqrt(fabs(S[i * kOL + i] * S[j * kOL + j])) + fl) need = 1;
  }
  __syncthreads();
  if (!need) {
    if (tid == 0) flag[blockIdx.x] = 0;
    return;
  }
  for (int e = tid; e < kOP * kOL; e += 256) V[e] = ((e / kOL) == (e % kOL)) ? T(1) : T(0);
  __syncthreads();
  bj_inner(S, V, jb, &inner_rot, gmax[lo]);
  __syncthreads();
  // one Newton-Schulz step V <- V (3 I - V^T V) / 2 against the rounding of the rotations
  {
    T acc[4][4];
    tile64<true, false, T>(V, V, acc);  // V^T V
    __syncthreads();
    const int ti = tid >> 4, tj = tid & 15;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int i = ti * 4 + u, j = tj * 4 + v;
        S[i * kOL + j] = (i == j ? T(1.5) : T(0)) - T(0.5) * acc[u][v];
      }
    __syncthreads();
    tile64<false, false, T>(V, S, acc);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) V[(ti * 4 + u) * kOL + tj * 4 + v] = acc[u][v];
    __syncthreads();
  }
  T* vg = vbuf + (size_t)blockIdx.x * kOP * kOP;
  for (int e = tid; e < kOP * kOP; e += 256) vg[e] = V[(e >> 6) * kOL + (e & 63)];
  if (tid == 0) {
    flag[blockIdx.x] = 1;
    atomicAdd(&nrot[lo], 1);
  }
}

// step, part 2: rows I+J of A <- V^T rows I+J, one 64-column chunk per CTA (grid.y)
template <class T>
__global__ void __launch_bounds__(256) k_bj_rowapply(const BjJob<T>* __restrict__ jobs, int njobs, int step,
                                                     const T* __restrict__ vbuf, const int* __restrict__ flag) {
  extern __shared__ double bsm[];
  T* V = reinterpret_cast<T*>(bsm);
  T* buf = V + kOP * kOL;
  __shared__ int idx[kOP];
  if (!flag[blockIdx.x]) return;
  const int lo = find_job(jobs, njobs);
  const BjJob<T> J = jobs[lo];
  const int r = blockIdx.x - J.pair_begin, tid = threadIdx.x, n = J.n;
  const int c0 = blockIdx.y * kOP;
  if (c0 >= n) return;
  pair_rows(J, r, step, idx);
  const T* vg = vbuf + (size_t)blockIdx.x * kOP * kOP;
  for (int e = tid; e < kOP * kOP; e += 256) V[(e >> 6) * kOL + (e & 63)] = vg[e];
  __syncthreads();
  for (int e = tid; e < kOP * kOP; e += 256) {
    const int i = e >> 6, k = e & 63;
    buf[i * kOL + k] = (idx[i] >= 0 && c0 + k < n) ? J.A[(size_t)idx[i] * n + c0 + k] : T(0);
  }
  __syncthreads();
  T acc[4][4];
  tile64<true, false, T>(V, buf, acc);
  const int ti = tid >> 4, tj = tid & 15;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int row = idx[ti * 4 + u];
    if (row < 0) continue;
#pragma unroll
    for (int v = 0; v < 4; ++v)
      if (c0 + tj * 4 + v < n) J.A[(size_t)row * n + c0 + tj * 4 + v] = acc[u][v];
  }
}

// step, part 3: columns I+J of A (grid.z = 0) and of Q (grid.z = 1) <- columns times V,
// one 64-row chunk per CTA (grid.y)
template <class T>
__global__ void __launch_bounds__(256) k_bj_cols(const BjJob<T>* __restrict__ jobs, int njobs, int step,
                                                 const T* __restrict__ vbuf, const int* __restrict__ flag) {
  extern __shared__ double bsm[];
  T* V = reinterpret_cast<T*>(bsm);
  T* buf = V + kOP * kOL;
  __shared__ int idx[kOP];
  if (!flag[blockIdx.x]) return;
  const int lo = find_job(jobs, njobs);
  const BjJob<T> J = jobs[lo];
  const int r = blockIdx.x - J.pair_begin, tid = threadIdx.x, n = J.n;
  pair_rows(J, r, step, idx);
  const T* vg = vbuf + (size_t)blockIdx.x * kOP * kOP;
  for (int e = tid; e < kOP * kOP; e += 256) V[(e >> 6) * kOL + (e & 63)] = vg[e];
  __syncthreads();
  const int ti = tid >> 4, tj = tid & 15;
  T* M = blockIdx.z == 0 ? J.A : J.Q;
  const int r0 = blockIdx.y * kOP;
  if (r0 >= n) return;
  for (int e = tid; e < kOP * kOP; e += 256) {
    const int rr = e >> 6, k = e & 63;
    buf[rr * kOL + k] = (idx[k] >= 0 && r0 + rr < n) ? M[(size_t)(r0 + rr) * n + idx[k]] : T(0);
  }
  __syncthreads();
  T acc[4][4];
  tile64<false, false, T>(buf, V, acc);
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int rr = r0 + ti * 4 + u;
    if (rr >= n) continue;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int col = idx[tj * 4 + v];
      if (col >= 0) M[(size_t)rr * n + col] = acc[u][v];
    }
  }
}

// eigenvalues = diagonal of the rotated A, sorted descending (ties by index) with the
// normalised columns of Q; A is scratch for the unsorted eigenvectors
__global__ void k_bj_finish(const BjJob<double>* __restrict__ jobs) {
  const BjJob<double> J = jobs[blockIdx.x];
  const int n = J.n, tid = threadIdx.x;
  extern __shared__ double wn[];
  double* qn = wn + n;
  for (int i = tid; i < n; i += blockDim.x) {
    wn[i] = J.A[(size_t)i * n + i];
    double q2 = 0.0;
    for (int j = 0; j < n; ++j) q2 += J.Q[(size_t)j * n + i] * J.Q[(size_t)j * n + i];
    qn[i] = 1.0 / sqrt(q2);
  }
  __syncthreads();
  for (int64_t e = tid; e < (int64_t)n * n; e += blockDim.x) J.A[e] = J.Q[e] * qn[e % n];
  __syncthreads();
  for (int i = tid; i < n; i += blockDim.x) {
    const double vi = wn[i];
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      const double vj = wn[j];
      if (vj > vi || (vj == vi && j < i)) ++rank;
    }
    J.w[rank] = vi;
    for (int rr = 0; rr < n; ++rr) J.Q[(size_t)rr * n + rank] = J.A[(size_t)rr * n + i];
  }
}

// Block-Jacobi sweeps over the jobs (A and Q in place) until no pair needs one, at most
// `sweeps`; gmax: the largest diagonal entry of every job (device).
template <class T>
void bj_sweeps(std::vector<BjJob<T>>& bj, const double* gmax, int sweeps, Stream s) {
  if (bj.empty()) return;
  int pairs = 0, nbmax = 0, nmax = 0;
  for (auto& j : bj) {
    j.nb = (j.n + kOB - 1) / kOB;
    j.nb += j.nb & 1;
    j.pair_begin = pairs;
    pairs += j.nb / 2;
    nbmax = std::max(nbmax, j.nb);
    nmax = std::max(nmax, j.n);
  }
  const int nj = (int)bj.size();
  const int nch = (nmax + kOP - 1) / kOP;  // 64-wide chunks of the largest matrix
  DevScratch mem(s);
  BjJob<T>* d = mem.get<BjJob<T>>(nj);
  dev_h2d(d, bj.data(), sizeof(BjJob<T>) * nj, s);
  T* vbuf = mem.get<T>((size_t)pairs * kOP * kOP);
  int* flag = mem.get<int>(pairs);
  int* nrot = mem.get<int>(nj);
  std::vector<int> hrot(nj);
  const size_t sh = sizeof(T) * 2 * kOP * kOL;
  static bool attr = false;  // per element type
  if (!attr) {
    ck(cudaFuncSetAttribute(k_bj_rows<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh), "bj smem");
    ck(cudaFuncSetAttribute(k_bj_cols<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh), "bj smem");
    ck(cudaFuncSetAttribute(k_bj_rowapply<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh), "bj smem");
    attr = true;
  }
  for (int sweep = 0; sweep < sweeps; ++sweep) {
    ck(cudaMemsetAsync(nrot, 0, sizeof(int) * nj, S(s)), "bj counters");
    for (int step = 0; step < nbmax - 1; ++step) {
      k_bj_rows<T><<<pairs, 256, sh, S(s)>>>(d, nj, step, gmax, vbuf, flag, nrot);
      k_bj_rowapply<T><<<dim3(pairs, nch), 256, sh, S(s)>>>(d, nj, step, vbuf, flag);
      k_bj_cols<T><<<dim3(pairs, nch, 2), 256, sh, S(s)>>>(d, nj, step, vbuf, flag);
      g_launches += 3;
    }
    ck(cudaGetLastError(), "bj step");
    dev_d2h(hrot.data(), nrot, sizeof(int) * nj, s);
    dev_sync(s);
    bool any = false;
    for (int v : hrot) any = any || v > 0;
    if (!any) break;
  }
}

}  // namespace

static void eig_block_jacobi(const std::vector<EigJob>& jobs, Stream s) {
  if (jobs.empty()) return;
  std::vector<BjJob<double>> bj;
  int nmax = 0;
  for (const EigJob& j : jobs) {
    bj.push_back({j.A, j.Q, j.w, j.n, 0, 0, 0});
    nmax = std::max(nmax, j.n);
  }
  const int nj = (int)bj.size();
  const size_t shf = sizeof(double) * 2 * nmax;
  if (shf > 220 * 1024) throw std::runtime_error("eig_batched: block too large");
  DevScratch mem(s);
  BjJob<double>* d = mem.get<BjJob<double>>(nj);
  dev_h2d(d, bj.data(), sizeof(BjJob<double>) * nj, s);
  double* gmax = mem.get<double>(nj);
  k_bj_prep<<<nj, 256, 0, S(s)>>>(d, gmax);
  ++g_launches;
  bj_sweeps(bj, gmax, 40, s);
  if (shf > 48 * 1024)
    ck(cudaFuncSetAttribute(k_bj_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shf), "bj finish smem");
  k_bj_finish<<<nj, 256, shf, S(s)>>>(d);
  ++g_launches;
  ck(cudaGetLastError(), "bj finish");
}

void eig_batched(const std::vector<EigJob>& jobs, Stream s) {
  if (jobs.empty()) return;
  std::vector<EigJob> small, large;
  int nmax_s = 1, nmax_l = 1;
  for (auto& j : jobs) {
    if (j.n <= kEigSmemN) { small.push_back(j); nmax_s = std::max(nmax_s, j.n); }
    else { large.push_back(j); nmax_l = std::max(nmax_l, j.n); }
  }
  DevScratch mem(s);
  EigJob* d = mem.get<EigJob>(jobs.size());
  if (!small.empty()) {
    dev_h2d(d, small.data(), small.size() * sizeof(EigJob), s);
    const int np = (nmax_s + 1) & ~1;
    size_t shm = sizeof(double) * ((size_t)2 * np * (np + 1) + nmax_s) + 64;
    ck(cudaFuncSetAttribute(k_eig_batched<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm), "eig smem");
    k_eig_batched<256><<<(int)small.size(), 256, shm, S(s)>>>(d);
    ++g_launches;
    ck(cudaGetLastError(), "eig_batched (shared)");
  }
  if (!large.empty()) eig_block_jacobi(large, s);
}

// ------------------------------------------------------------------ refined eigensolver
//
// The same eigenproblems, mostly in FP32.  FP64 Jacobi costs about 50 n^3 FP64 operations
// and a chain of n - 1 rotations (3000 cycles each) per sweep; an SM does two FP64 FMAs
// per cycle and 128 FP32 ones.  So three passes of: FP32 Jacobi on the current matrix S
// (scaled by its largest diagonal entry) -> Q; X <- X Q, orthonormalised by a Newton-Schulz
// step X (3 I - X^T X) / 2; T = M^T X (or M X), S = T^T T, all of these FP64 products of the
// whole GPU (S from M itself, G = M M^T or M^T M, has errors of eps sigma_i sigma_j, where
// X^T G X has eps |G|).  Each pass resolves eigenvectors to FP32 accuracy within blocks of
// similar eigenvalues, so the unresolved part of S falls from |G| to 1e-7, 1e-14 |G| and
// rounding (the floors below which a pass leaves an off-diagonal alone).  Then one step of
// the iterative refinement of T. Ogita and K. Aishima (Japan J. Indust. Appl. Math. 35, 2018):
// with R = I - X^T X, lambda_i = S_ii / (1 - R_ii), X <- X + X E, E_ij = (S_ij + lambda_j
// R_ij) / (lambda_j - lambda_i), R_ij / 2 where that is not small, and a last Newton-Schulz
// step.  Measured (dmrg_truncate, against the Jacobi solver): Hubbard L=16, D=200 (sectors up
// to 114 rows) 37.1 -> 8.1 ms, random L=28, D=1500 (up to 202) 116 -> 22.4 ms, the error of the
// truncated state against an SVD 6.5e-15 -> 2.3e-15 and 1.5e-14 -> 3.5e-15.  A job that still
// has an
// off-diagonal above rounding whose rotation is not negligible (a relative gap below FP32's
// resolution) is handed to the FP64 solver.

namespace {
struct ReJob {
  const double* G;
  double *X, *S, *R, *w, *Q;
  float *A32, *Q32;
  int n, pad;
};

// A32 = S / max diagonal, Q32 = I
__global__ void __launch_bounds__(256) k_re_start(const ReJob* __restrict__ jobs, int first) {
  const ReJob J = jobs[blockIdx.x];
  const double* S = first ? J.G : J.S;
  const int n = J.n, tid = threadIdx.x;
  __shared__ double red[256];
  double best = 0.0;
  for (int i = tid; i < n; i += 256) best = fmax(best, fabs(S[(size_t)i * n + i]));
  red[tid] = best;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (tid < o) red[tid] = fmax(red[tid], red[tid + o]);
    __syncthreads();
  }
  const double inv = red[0] > 0.0 ? 1.0 / red[0] : 0.0;
  for (int64_t e = tid; e < (int64_t)n * n; e += 256) {
    const int i = (int)(e / n), j = (int)(e % n);
    J.A32[e] = (float)(S[i <= j ? e : (int64_t)j * n + i] * inv);  // symmetric to the bit
    J.Q32[e] = i == j ? 1.0f : 0.0f;
  }
}

// FP32 Jacobi of the blocks up to kEigSmemN rows, one CTA each
__global__ void __launch_bounds__(256) k_re_small(const ReJob* __restrict__ jobs, const int* __restrict__ which,
                                                  int sweeps, float floor_abs) {
  const ReJob J = jobs[which[blockIdx.x]];
  const int n = J.n, np = (n + 1) & ~1, ld = np + 1, tid = threadIdx.x;
  extern __shared__ float fsm[];
  float* A = fsm;
  float* Q = A + np * ld;
  __shared__ float cs[kEigSmemN / 2], sn[kEigSmemN / 2];
  __shared__ int pp[kEigSmemN / 2], qq[kEigSmemN / 2], flag;
  for (int e = tid; e < np * np; e += 256) {
    const int i = e / np, j = e % np;
    const bool in = i < n && j < n;
    A[i * ld + j] = in ? J.A32[(size_t)i * n + j] : 0.0f;
    Q[i * ld + j] = i == j ? 1.0f : 0.0f;
  }
  __syncthreads();
  if (np > 1) jacobi_f32(A, Q, np, ld, sweeps, floor_abs, cs, sn, pp, qq, &flag);
  __syncthreads();
  for (int e = tid; e < n * n; e += 256) J.Q32[e] = Q[(e / n) * ld + e % n];
}

// out = (double)Q32 (to X on the first pass, to S, as scratch, afterwards)
__global__ void k_re_widen(const ReJob* __restrict__ jobs, int first) {
  const ReJob J = jobs[blockIdx.x];
  double* out = first ? J.X : J.S;
  for (int64_t e = threadIdx.x + (int64_t)blockIdx.y * blockDim.x; e < (int64_t)J.n * J.n; e += (int64_t)gridDim.y * blockDim.x)
    out[e] = (double)J.Q32[e];
}

__global__ void k_re_identity(const ReJob* __restrict__ jobs) {  // R = I
  const ReJob J = jobs[blockIdx.x];
  for (int64_t e = threadIdx.x + (int64_t)blockIdx.y * blockDim.x; e < (int64_t)J.n * J.n; e += (int64_t)gridDim.y * blockDim.x)
    J.R[e] = e / J.n == e % J.n ? 1.0 : 0.0;
}

__global__ void k_re_half(const ReJob* __restrict__ jobs) {  // R <- R / 2 (Newton-Schulz)
  const ReJob J = jobs[blockIdx.x];
  for (int64_t e = threadIdx.x + (int64_t)blockIdx.y * blockDim.x; e < (int64_t)J.n * J.n; e += (int64_t)gridDim.y * blockDim.x)
    J.R[e] *= 0.5;
}

// May the refinement step take E = g / gap for a pair (gm: the largest eigenvalue)?  The step
// is of first order: it leaves an off-diagonal of about g E, and an error of E^2 in the
// eigenvectors.  So E is small and g E below the rounding of the Gram route (which has errors
// of eps gm / gap in such a pair's vectors too); a pass that stopped at its sweep limit with
// more than that left goes to the FP64 solver.
__host__ __device__ inline bool refine_accepts(double g, double gap, double gm) {
  return fabs(g) < 1e-5 * fabs(gap) && fabs(g) * fabs(g) <= 1e-16 * gm * fabs(gap);
}

// R <- E; bad[job] = 1 where the refinement cannot be trusted
__global__ void __launch_bounds__(256) k_re_correct(const ReJob* __restrict__ jobs, int* __restrict__ bad) {
  const ReJob J = jobs[blockIdx.x];
  const int n = J.n, tid = threadIdx.x;
  extern __shared__ double lam[];
  __shared__ double gm;
  __shared__ int fail;
  if (tid == 0) { fail = 0; gm = 0.0; }
  for (int i = tid; i < n; i += 256) lam[i] = J.S[(size_t)i * n + i] / (1.0 - J.R[(size_t)i * n + i]);
  __syncthreads();
  if (tid < 32) {
    double m = 0.0;
    for (int i = tid; i < n; i += 32) m = fmax(m, fabs(lam[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (tid == 0) gm = m;
  }
  __syncthreads();
  for (int64_t e = tid; e < (int64_t)n * n; e += 256) {
    const int i = (int)(e / n), j = (int)(e % n);
    const double r = J.R[e];
    double v = 0.5 * r;
    if (!(fabs(r) <= 1e-9)) fail = 1;  // also not finite
    if (i != j) {
      const double g = J.S[e] + lam[j] * r, gap = lam[j] - lam[i];
      if (refine_accepts(g, gap, gm)) v = g / gap;
      else if (!(fabs(g) <= 1e-14 * gm)) fail = 1;
    }
    J.R[e] = v;
  }
  for (int i = tid; i < n; i += 256) J.w[i] = lam[i];
  __syncthreads();
  if (tid == 0) bad[blockIdx.x] = fail;
}

// eigenvalues (in w) sorted descending (ties by index) with the columns of X, into w and Q
__global__ void __launch_bounds__(256) k_re_finish(const ReJob* __restrict__ jobs) {
  const ReJob J = jobs[blockIdx.x];
  const int n = J.n, tid = threadIdx.x;
  extern __shared__ double lam[];
  int* rank = reinterpret_cast<int*>(lam + n);
  for (int i = tid; i < n; i += 256) lam[i] = J.w[i];
  __syncthreads();
  for (int i = tid; i < n; i += 256) {
    int r = 0;
    for (int j = 0; j < n; ++j) r += lam[j] > lam[i] || (lam[j] == lam[i] && j < i);
    rank[i] = r;
    J.w[r] = lam[i];
  }
  __syncthreads();
  for (int64_t e = tid; e < (int64_t)n * n; e += 256) J.Q[(e / n) * n + rank[e % n]] = J.X[e];
}
}  // namespace

bool eig_refine_accepts(double g, double gap, double gm) { return refine_accepts(g, gap, gm); }

namespace {
// the jobs that have to go to eig_batched (their Gram matrices are as they were)
std::vector<EigJob> refined_passes(const std::vector<EigJob>& jobs, const std::vector<EigSource>& src, int nmax, Stream s) {
  std::vector<int64_t> off(1, 0), toff(1, 0);
  for (size_t k = 0; k < jobs.size(); ++k) {
    off.push_back(off.back() + (int64_t)jobs[k].n * jobs[k].n);
    toff.push_back(toff.back() + (int64_t)src[k].inner * jobs[k].n);
  }
  const int64_t tot = off.back();
  const int nj = (int)jobs.size();
  // X, X2, S, R, T (FP64), A32, Q32 (FP32)
  const int64_t ttot = toff.back();
  DevScratch mem(s);
  double* buf = mem.get<double>((size_t)(tot * 5 + ttot));
  double *X = buf, *X2 = X + tot, *Sm = X2 + tot, *R = Sm + tot, *T = R + tot;
  float *A32 = (float*)(T + ttot), *Q32 = A32 + tot;
  std::vector<int> hbad(nj, 0);
  struct Plans {
    Stream s;
    GemmPlan *pq = nullptr, *pr = nullptr, *pn = nullptr, *pt = nullptr, *ps = nullptr;
    ~Plans() {
      for (GemmPlan* p : {pq, pr, pn, pt, ps}) {
        try {
          gemm_plan_free(p, s);
        } catch (...) {
        }
      }
    }
  } g{s};
  GemmPlan *&pq = g.pq, *&pr = g.pr, *&pn = g.pn, *&pt = g.pt, *&ps = g.ps;
  std::vector<ReJob> re;
  std::vector<int> small;
  std::vector<BjJob<float>> big;
  int nsm = 1;
  for (int k = 0; k < nj; ++k) {
    const EigJob& j = jobs[k];
    const int64_t o = off[k];
    re.push_back({j.A, X + o, Sm + o, R + o, j.w, j.Q, A32 + o, Q32 + o, j.n, 0});
    if (j.n <= kEigSmemN) {
      small.push_back(k);
      nsm = std::max(nsm, j.n);
    } else {
      big.push_back({A32 + o, Q32 + o, nullptr, j.n, 0, 0, 0});
    }
  }
  ReJob* d = mem.get<ReJob>(nj);
  dev_h2d(d, re.data(), sizeof(ReJob) * nj, s);
  int* dsmall = mem.get<int>(small.size() + 1);
  dev_h2d(dsmall, small.data(), sizeof(int) * small.size(), s);
  int* dbad = mem.get<int>(nj);
  // the three passes: floor (of the largest diagonal entry, scaled to 1: a little above
  // what FP32 rounding leaves of the part that the pass resolves), sweeps at most, and
  // Newton-Schulz steps (FP32 rotations leave Q orthonormal to 1e-5 where they are large)
  constexpr double kFloor[3] = {1e-6, 5e-13, 5e-16};
  constexpr int kSweeps[3] = {10, 8, 4}, kSchulz[3] = {2, 2, 1};
  const size_t nb = big.size();
  double* gbig = mem.get<double>(std::max<size_t>(3 * nb, 1));
  std::vector<double> fl;
  for (double f : kFloor) fl.insert(fl.end(), nb, f);
  dev_h2d(gbig, fl.data(), sizeof(double) * fl.size(), s);
  // one n-column product per job: C (m x n) += alpha op(A) B
  auto plan = [&](auto task) {
    std::vector<GemmTask> t;
    std::vector<GemmGroup> g;
    for (int k = 0; k < nj; ++k) {
      double* c = nullptr;
      int m = jobs[k].n;
      t.push_back(task(k, c, m));
      g.push_back({c, jobs[k].n, m, jobs[k].n, k, k + 1, 0});
    }
    return gemm_plan_upload(t, g, s, GEMM_SHARED);
  };
  pq = plan([&](int k, double*& c, int&) {  // X2 = X Q (Q widened into S)
    const int n = jobs[k].n;
    c = X2 + off[k];
    return GemmTask{X + off[k], Sm + off[k], n, n, n, 0, 0, 1.0};
  });
  pr = plan([&](int k, double*& c, int&) {  // R -= X^T X
    const int n = jobs[k].n;
    c = R + off[k];
    return GemmTask{X + off[k], X + off[k], n, n, n, 1, 0, -1.0};
  });
  pn = plan([&](int k, double*& c, int&) {  // X2 += X R
    const int n = jobs[k].n;
    c = X2 + off[k];
    return GemmTask{X + off[k], R + off[k], n, n, n, 0, 0, 1.0};
  });
  pt = plan([&](int k, double*& c, int& m) {  // T = M^T X or M X
    const int n = jobs[k].n;
    c = T + toff[k];
    m = src[k].inner;
    return GemmTask{src[k].M, X + off[k], src[k].ld, n, n, src[k].trans, 0, 1.0};
  });
  ps = plan([&](int k, double*& c, int&) {  // S = T^T T
    const int n = jobs[k].n;
    c = Sm + off[k];
    return GemmTask{T + toff[k], T + toff[k], n, n, src[k].inner, 1, 0, 1.0};
  });
  const size_t bytes = sizeof(double) * (size_t)tot;
  const dim3 grid(nj, std::max(1, std::min(64, nmax * nmax / 4096)));
  const int np = (nsm + 1) & ~1;
  const size_t shs = sizeof(float) * 2 * (size_t)np * (np + 1), shc = sizeof(double) * 2 * (size_t)nmax;
  if (shc > 48 * 1024) {
    ck(cudaFuncSetAttribute(k_re_correct, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shc), "eig smem");
    ck(cudaFuncSetAttribute(k_re_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shc), "eig smem");
  }
  // X <- X2 + ... where X2 holds a copy of X, then X = X2
  auto residual = [&]() {  // R = I - X^T X
    k_re_identity<<<grid, 256, 0, S(s)>>>(d);
    gemm_plan_run(pr, s, GEMM_SHARED);
    ++g_launches;
  };
  auto add_correction = [&]() {  // X <- X + X R
    dev_d2d(X2, X, bytes, s);
    gemm_plan_run(pn, s, GEMM_SHARED);
    dev_d2d(X, X2, bytes, s);
  };
  auto schulz = [&]() {  // X <- X (3 I - X^T X) / 2
    residual();
    k_re_half<<<grid, 256, 0, S(s)>>>(d);
    ++g_launches;
    add_correction();
  };
  for (int pass = 0; pass < 3; ++pass) {
    k_re_start<<<nj, 256, 0, S(s)>>>(d, pass == 0);
    if (!small.empty()) k_re_small<<<(int)small.size(), 256, shs, S(s)>>>(d, dsmall, kSweeps[pass], (float)kFloor[pass]);
    bj_sweeps(big, gbig + pass * nb, kSweeps[pass], s);
    k_re_widen<<<grid, 256, 0, S(s)>>>(d, pass == 0);
    g_launches += 3;
    if (pass > 0) {
      dev_zero(X2, bytes, s);
      gemm_plan_run(pq, s, GEMM_SHARED);
      dev_d2d(X, X2, bytes, s);
    }
    for (int u = 0; u < kSchulz[pass]; ++u) schulz();
    dev_zero(T, sizeof(double) * (size_t)ttot, s);
    gemm_plan_run(pt, s, GEMM_SHARED);
    dev_zero(Sm, bytes, s);
    gemm_plan_run(ps, s, GEMM_SHARED);
  }
  residual();
  k_re_correct<<<nj, 256, shc, S(s)>>>(d, dbad);
  add_correction();
  schulz();
  ck(cudaGetLastError(), "refined eig");
  dev_d2h(hbad.data(), dbad, sizeof(int) * nj, s);
  k_re_finish<<<nj, 256, shc, S(s)>>>(d);
  g_launches += 2;
  ck(cudaGetLastError(), "refined eig");
  dev_sync(s);
  std::vector<EigJob> again;
  for (int k = 0; k < nj; ++k)
    if (hbad[k]) again.push_back(jobs[k]);
  return again;
}
}  // namespace

void eig_refined(const std::vector<EigJob>& jobs, const std::vector<EigSource>& src, Stream s) {
  if (jobs.empty()) return;
  int nmax = 1;
  for (const EigJob& j : jobs) nmax = std::max(nmax, j.n);
  // Small blocks: the passes' launches and tables cost some 0.7 ms whatever the sizes.  Whole
  // call, Hubbard chains, Jacobi / refined: largest block 11 rows 0.59 / 0.84 ms, 20 rows 0.89 /
  // 1.02, 26 rows 1.37 / 1.16, 49 rows 4.5 / 2.1.
  constexpr int kRefineRows = 23;
  if (nmax < kRefineRows || sizeof(double) * 2 * (size_t)nmax > 200 * 1024) return eig_batched(jobs, s);
  std::vector<EigJob> again;
  try {
    again = refined_passes(jobs, src, nmax, s);
  } catch (const std::exception& e) {
    if (!no_room(e)) throw;
    again = jobs;  // the workspace has been released: the solver in place
  }
  eig_batched(again, s);
}

// ------------------------------------------------------------------ selection

namespace {
// rank of every value (descending, ties by position) over all n values: one thread per
// value, many CTAs; keep[i] = rank < D and above the zero threshold
__global__ void k_select_rank(const double* __restrict__ v, int n, const double* __restrict__ vmax,
                              int D, double zero_rel, int* __restrict__ keep) {
  // non-negative doubles order like their bit patterns: integer comparisons (an FP64 one
  // costs a warp 16 cycles of the SM: 0.82 ms for 6,000 values, now 0.10)
  __shared__ long long tile[1024];
  auto bits = [](double x) { return x > 0.0 ? __double_as_longlong(x) : 0ll; };
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const double vd = i < n ? fmax(v[i], 0.0) : 0.0;
  const long long vi = bits(vd);
  int rank = 0;
  for (int j0 = 0; j0 < n; j0 += 1024) {
    for (int t = threadIdx.x; t < 1024; t += blockDim.x) tile[t] = (j0 + t < n) ? bits(v[j0 + t]) : -1ll;
    __syncthreads();
    const int jn = min(1024, n - j0);
    for (int t = 0; t < jn; ++t) {
      const long long vj = tile[t];
      rank += (vj > vi || (vj == vi && j0 + t < i)) ? 1 : 0;
    }
    __syncthreads();
  }
  if (i < n) keep[i] = (rank < D && vd > zero_rel * zero_rel * (*vmax)) ? 1 : 0;
}

__global__ void k_select_max(const double* __restrict__ v, int n, double* __restrict__ vmax) {
  __shared__ double red[256];
  double mx = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) mx = fmax(mx, v[i]);
  red[threadIdx.x] = mx;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) { if (threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]); __syncthreads(); }
  if (threadIdx.x == 0) *vmax = red[0];
}

// per-group kept counts and the weighted sums (norm^2, discarded) in a fixed order
__global__ void k_select_sums(const double* __restrict__ v, int n, const int* __restrict__ gid,
                              const int* __restrict__ wgt, const int* __restrict__ keep, int* kept,
                              double* sums) {
  __shared__ double red[2][256];
  double nrm = 0.0, disc = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) {
    const double w = (double)wgt[gid[i]] * fmax(v[i], 0.0);
    nrm += w;
    if (keep[i]) atomicAdd(&kept[gid[i]], 1); else disc += w;
  }
  red[0][threadIdx.x] = nrm;
  red[1][threadIdx.x] = disc;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) { red[0][threadIdx.x] += red[0][threadIdx.x + o]; red[1][threadIdx.x] += red[1][threadIdx.x + o]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) { sums[0] = red[0][0]; sums[1] = red[1][0]; }
}
}  // namespace

void select_largest(const double* vals, const std::vector<int>& goff, const std::vector<int>& wgt,
                    int D, double zero_rel, std::vector<int>& kept, double* norm2, double* disc,
                    Stream s) {
  const int G = (int)wgt.size();
  const int n = goff.back();
  std::vector<int> gid(n);
  for (int g = 0; g < G; ++g)
    for (int i = goff[g]; i < goff[g + 1]; ++i) gid[i] = g;
  int* d_gid = (int*)dev_alloc(sizeof(int) * (n + 1), s);
  int* d_w = (int*)dev_alloc(sizeof(int) * (G + 1), s);
  int* d_k = (int*)dev_alloc(sizeof(int) * (G + 1), s);
  int* d_keep = (int*)dev_alloc(sizeof(int) * (n + 1), s);
  double* d_s = (double*)dev_alloc(sizeof(double) * 3, s);
  dev_h2d(d_gid, gid.data(), sizeof(int) * n, s);
  dev_h2d(d_w, wgt.data(), sizeof(int) * G, s);
  dev_zero(d_k, sizeof(int) * (G + 1), s);
  k_select_max<<<1, 256, 0, S(s)>>>(vals, n, d_s + 2);
  ++g_launches;
  if (n > 0) {
    k_select_rank<<<(n + 255) / 256, 256, 0, S(s)>>>(vals, n, d_s + 2, D, zero_rel, d_keep);
    ++g_launches;
  }
  k_select_sums<<<1, 256, 0, S(s)>>>(vals, n, d_gid, d_w, d_keep, d_k, d_s);
  ++g_launches;
  ck(cudaGetLastError(), "select");
  kept.assign(G, 0);
  double sums[2];
  dev_d2h(kept.data(), d_k, sizeof(int) * G, s);
  dev_d2h(sums, d_s, sizeof(double) * 2, s);
  dev_sync(s);
  *norm2 = sums[0];
  *disc = sums[1];
  dev_free(d_gid, s);
  dev_free(d_w, s);
  dev_free(d_k, s);
  dev_free(d_keep, s);
  dev_free(d_s, s);
}

// ------------------------------------------------------------------ scatter

namespace {
__device__ inline double scl(const double* v, int i, int mode) {
  if (mode == 0) return 1.0;
  double x = v[i];
  return mode == 1 ? sqrt(x) : 1.0 / sqrt(x);
}

__global__ void k_scatter(const ScatterJob* __restrict__ jobs) {
  const ScatterJob J = jobs[blockIdx.x];
  const int64_t n = (int64_t)J.rows * J.cols;
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {
    int i = (int)(e / J.cols), j = (int)(e % J.cols);
    double v = J.trans ? J.src[(size_t)j * J.lds + i] : J.src[(size_t)i * J.lds + j];
    J.dst[(size_t)i * J.ldd + j] = J.a * scl(J.rs, i, J.rmode) * scl(J.cs, j, J.cmode) * v;
  }
}
}  // namespace

void scatter_batched(const std::vector<ScatterJob>& jobs, Stream s) {
  if (jobs.empty()) return;
  ScatterJob* d = (ScatterJob*)dev_alloc(jobs.size() * sizeof(ScatterJob), s);
  dev_h2d(d, jobs.data(), jobs.size() * sizeof(ScatterJob), s);
  for (size_t off = 0; off < jobs.size(); off += 65535) {
    int n = (int)std::min<size_t>(65535, jobs.size() - off);
    k_scatter<<<n, 128, 0, S(s)>>>(d + off);
    ++g_launches;
  }
  ck(cudaGetLastError(), "scatter");
  dev_free(d, s);
}

// ------------------------------------------------------------------ allocation-free matvec
//
// For callers that cannot allocate device memory at the time of the call (inside a
// region where cudaMalloc is not allowed, or on a budget that forbids growth): the
// matvec's scratch (the right-operator products Z and the weighted sums W) is placed in
// this fixed array instead of the context's own buffers.  The array exists once per
// device that loads the library and stays allocated until the process exits.

namespace {

constexpr int64_t kNoAllocScratchDoubles = (int64_t)8 << 20;  // 64 MiB
static __device__ __align__(256) double g_noalloc_scratch[kNoAllocScratchDoubles];

std::mutex g_noalloc_mu;
double* g_noalloc_ptr[64] = {nullptr};  // device address of the array, per device ordinal

// Device address of the static array on the current device (looked up once per device).
double* noalloc_scratch(int* err) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 64) { *err = 1; return nullptr; }
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    double* p = nullptr;
    e = cudaGetSymbolAddress((void**)&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) { *err = 2; return nullptr; }
    g_noalloc_ptr[dev] = p;
  }
  *err = 0;
  return g_noalloc_ptr[dev];
}

}  // namespace

int64_t noalloc_scratch_capacity() { return kNoAllocScratchDoubles; }

void noalloc_matvec_run(const GemmPlan* p1, const CombPlan* pc, const GemmPlan* p2,
                        const double* xin, const double* yout, int64_t n, const double* Z,
                        int64_t zsize, const double* Wb, int64_t wsize, const double* x,
                        double* y, Stream s) {
  if (zsize + wsize > kNoAllocScratchDoubles)
    throw std::invalid_argument("scratch needed exceeds the 64 MiB static maximum of the allocation-free matvec");
  int err = 0;
  double* scratch = noalloc_scratch(&err);
  if (!scratch) throw std::runtime_error("cuda: cudaGetSymbolAddress of the static scratch failed");
  Remap rm;
  rm.lo[0] = (const char*)xin;  rm.hi[0] = (const char*)(xin + n);     rm.to[0] = (char*)x;
  rm.lo[1] = (const char*)yout; rm.hi[1] = (const char*)(yout + n);    rm.to[1] = (char*)y;
  rm.lo[2] = (const char*)Z;    rm.hi[2] = (const char*)(Z + zsize);   rm.to[2] = (char*)scratch;
  rm.lo[3] = (const char*)Wb;   rm.hi[3] = (const char*)(Wb + wsize);  rm.to[3] = (char*)(scratch + zsize);
  // phase 2 accumulates into y, which starts at zero; Z and W are overwritten
  if (n) ck(cudaMemsetAsync(y, 0, sizeof(double) * n, S(s)), "memset y");
  gemm_launch<true>(p1, rm, GEMM_SHARED, s);
  combine_launch<true>(pc, rm, s);
  gemm_launch<true>(p2, rm, GEMM_SHARED, s);
  ck(cudaGetLastError(), "allocation-free matvec launch");
}

}  // namespace dmrg
