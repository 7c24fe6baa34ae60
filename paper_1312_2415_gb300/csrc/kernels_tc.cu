// Mixed-precision H_eff matvec on the 5th-generation tensor cores (tcgen05, sm_103a).
//
// The effective Hamiltonian of Eq. 9, written with the renormalised and complementary
// operators of Sec. 2.5, acts on an output block y_X' as a sum of terms
//   y_X' += C W,   W = sum_s coef_s x_s D_s^T,
// C a left-operator block, x_s blocks of the two-site vector and D_s right-operator
// blocks (the combined operators of the left / right environments).  An output tile (up to
// 128 rows x 128 columns of one block) is cut into runs of terms; a CTA computes a run and
// leaves its partial sums, which are added in term order afterwards (nothing is added with
// atomics and the summation order is fixed).  The launch is persistent (one to four CTAs per
// SM by tile size, taking runs from a work queue), so the pipeline runs on from one run into
// the next (tiles of at most 4 x 4 outputs go to a CUDA-core kernel, k_tc_tiny, instead):
//   product 1: W^T = D_s x_s^T per source, into tensor-memory accumulators of at most
//              two 32-column K chunks each (M = 128 output columns, N = x rows of the
//              term, K = the right sector);
//   the converter warps add coef_s times each accumulator into FP32 registers, split the
//              sum into TF32 head and tail and store it as the A operand of
//   product 2: y^T += W^T C^T (M = 128 output columns, N = output rows, K = x rows),
//              restarted per term and drained into FP32 registers, stored every few
//              terms (the partial sums, added to y in FP64).  The tensor core's own FP32
//              accumulation loses accuracy over long runs of products, hence the short
//              accumulators.
// Every product uses split TF32: v = hi + lo with hi = rna_tf32(v), lo = rna_tf32(v - hi),
// and the three leading products hi*hi + hi*lo + lo*hi (about 2^-21 relative).  The
// second operand's hi and lo tiles sit one above the other in shared memory, so one MMA
// of twice the N gives A_hi B_hi^T and A_hi B_lo^T side by side in the accumulator and a
// second one adds A_lo B_hi^T to the first half: two instructions per K step instead of
// three.  An M = 128 tf32 MMA costs the issuing thread about 40-50 cycles whatever its N
// up to 64, so fewer, wider instructions are what the small blocks of this method need;
// products 1 and 2 are issued by two threads.
//
// Operands live in global memory already split and tiled in the K-major core-matrix
// order the MMA reads (see device.hpp), so a warp-specialised pipeline moves them with
// cp.async.bulk into shared memory (completion counted in bytes on mbarriers): a producer
// thread fills the product-1 ring, the product-2 thread loads the C tiles itself; only
// W^T passes through registers.  The shared-memory operand descriptors are K-major
// without swizzle: core matrices of 8 rows x 16 bytes, 128 bytes apart along K (LBO) and
// 1024 bytes apart along M/N (SBO), for 32-column chunks.
//
// Every wait is bounded: a CTA that gives up records an error, stops issuing work, waits
// (bounded) for its own copies and products in flight, frees its tensor memory and
// returns; the host reads and clears the error flag.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <limits>
#include <unordered_map>
#include <stdexcept>
#include <string>

#include "device.hpp"
#include "plans.hpp"

namespace dmrg {

namespace {

constexpr long long kSpinLimit = 1ll << 22;  // polls of an mbarrier before giving up (seconds)
constexpr int kRowsF = 128 * 32;             // floats an M = 128 product reads of its first operand (16 KB)
constexpr int kMaxS1 = 8;                    // slots of the product-1 operand ring, at most
constexpr int kMaxB2 = 2;                    // C slots, at most
constexpr int kMaxW = 3;                     // W^T accumulators, at most
constexpr int kTileQ = 4;                    // tiles taken from the work queue ahead of the slowest role
constexpr int kSegChunks = 2;   // K chunks per product-1 accumulator (then added in registers)
constexpr int kFlushTerms = 16; // terms summed in FP32 registers per partial sum of y

// Three builds of the kernel by tile size.  A tile's terms form a chain (product 1, the
// conversion of W^T, product 2: about 3.5 us a term, mostly handoffs between the roles), so
// what counts for small blocks is how many chains an SM runs at once: four CTAs for tiles of
// at most 32 x 32, two up to 64 x 64, one up to 128 x 128, each with its share of shared
// memory (KB), tensor memory (columns) and only the converter warps whose rows exist.  NQ:
// 32-column quarters of the output (tensor-memory lanes); NH: converter warps per quarter,
// which split the x rows of W^T and the output rows.
template <int NQ, int NH, int A2KB, int S1KB, int B2KB, int TMEM, int YCOLS, int CTAS>
struct TileClass {
  static constexpr int kA2F = A2KB * 256, kS1F = S1KB * 256, kB2F = B2KB * 256;
  static constexpr int kTmem = TMEM, kWReg = TMEM - YCOLS, kCtas = CTAS;
  static constexpr int kSmemF = kA2F + kS1F + kB2F;
  static constexpr int kMaxM = YCOLS, kMaxN = 32 * NQ, kMaxKdl = 32 * NH;
  static constexpr int kYR = YCOLS / NH;  // output rows per converter thread
  // warps: a converter of quarter q is a warp with index q mod 4 (tensor-memory lanes)
  static constexpr int kProducerWarp = NQ == 1 ? 1 : NQ == 2 ? 2 : 8;
  static constexpr int kMma1Warp = NQ == 1 ? 2 : NQ == 2 ? 3 : 9;
  static constexpr int kMma2Warp = NQ == 1 ? 3 : NQ == 2 ? 6 : 10;
  static constexpr int kThreads = NQ == 1 ? 128 : NQ == 2 ? 224 : 352;
  static constexpr int kConvThreads = NQ * NH * 32;
};
using TileS = TileClass<1, 1, 8, 32, 8, 128, 32, 4>;
using TileM = TileClass<2, 2, 24, 62, 24, 256, 64, 2>;
using TileL = TileClass<4, 2, 64, 96, 64, 512, 128, 1>;

__device__ int g_tc_error = 0;
__device__ int g_tc_inject = 0;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ float tf32_round(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// float index of element (row, k) of a K-major no-swizzle tile with 32 columns
__device__ __forceinline__ int kmo(int row, int k) {
  return (row >> 3) * 256 + (k >> 2) * 32 + (row & 7) * 4 + (k & 3);
}

__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  // start >> 4 | LBO (128 B) >> 4 << 16 | SBO (1024 B) >> 4 << 32 | descriptor version 1 << 46
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) |
         ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46);
}

// instruction descriptor: D f32, A and B tf32, both K-major, M = 128, N = n (multiple of 16)
__device__ __forceinline__ uint32_t idesc_tf32(int n) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint64_t* mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(mbar))
               : "memory");
}

__device__ __forceinline__ void mbar_init_n(uint64_t* mbar, int n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(n));
}

__device__ __forceinline__ void mbar_arrive(uint64_t* mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(mbar)) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t* mbar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}\n"
      : "=r"(done)
      : "r"(smem_u32(mbar)), "r"(parity)
      : "memory");
  return done != 0;
}

// bounded wait that also gives up once another thread has flagged an abort; on its own
// timeout it records the error and flags the abort
__device__ __forceinline__ bool wait_or_abort(uint64_t* mbar, uint32_t parity, volatile int* abort_flag,
                                              long long limit = kSpinLimit) {
  for (long long it = 0; it < limit; ++it) {
    if (mbar_test(mbar, parity)) return true;
    if ((it & 1023) == 1023 && *abort_flag) return false;
  }
  atomicExch(&g_tc_error, 1);
  *abort_flag = 1;
  return false;
}

// bounded wait that ignores the abort flag (draining work in flight before exit)
__device__ __forceinline__ void wait_drain(uint64_t* mbar, uint32_t parity) {
  for (long long it = 0; it < kSpinLimit; ++it)
    if (mbar_test(mbar, parity)) return;
  atomicExch(&g_tc_error, 1);
}

// global -> shared bulk copy counted on mbar (16-byte aligned, size a multiple of 16)
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(mbar))
               : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
               "r"(cols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}

__device__ __forceinline__ void tmem_free(uint32_t tmem, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols));
}

// 32 consecutive accumulator columns of this warp's 32 lanes
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// the three split products of one K step, unstacked: A_hi B_hi^T + A_hi B_lo^T +
// A_lo B_hi^T into the same columns; nst steps of K = 8
__device__ __forceinline__ void mma_triple_steps(uint32_t tmem, uint64_t ah, uint64_t al, uint64_t bh, uint64_t bl,
                                                 uint32_t id, int nst, bool fresh) {
  for (int st = 0; st < nst; ++st) {
    const uint64_t o = (uint64_t)(16 * st);
    mma_tf32(tmem, ah + o, bh + o, id, (fresh && st == 0) ? 0u : 1u);
    mma_tf32(tmem, ah + o, bl + o, id, 1u);
    mma_tf32(tmem, al + o, bh + o, id, 1u);
  }
}

struct Bars {
  uint64_t s1_full[kMaxS1], s1_empty[kMaxS1];
  uint64_t b2_full[kMaxB2];
  uint64_t w_full[kMaxW], w_empty[kMaxW];
  uint64_t a2_full, mma2_done;
  uint64_t drain1, drain2, never;
  uint64_t tile_full[kTileQ], tile_empty[kTileQ];
};

// the two split products of one K step stacked along N: A_hi [B_hi; B_lo]^T (N = 2 kp)
// into accumulator columns [0, 2 kp) and A_lo B_hi^T (N = kp) into [0, kp); nst steps of
// K = 8 (8 columns = 256 bytes = 16 in the descriptor's address field), the first
// product restarting the accumulator when `fresh`
__device__ __forceinline__ void mma_pair_steps(uint32_t tmem, uint64_t ah, uint64_t al, uint64_t b, uint32_t id2,
                                               uint32_t id1, int nst, bool fresh) {
  mma_tf32(tmem, ah, b, id2, fresh ? 0u : 1u);
  mma_tf32(tmem, al, b, id1, 1u);
  if (nst > 1) {
    mma_tf32(tmem, ah + 16, b + 16, id2, 1u);
    mma_tf32(tmem, al + 16, b + 16, id1, 1u);
  }
  if (nst > 2) {
    mma_tf32(tmem, ah + 32, b + 32, id2, 1u);
    mma_tf32(tmem, al + 32, b + 32, id1, 1u);
  }
  if (nst > 3) {
    mma_tf32(tmem, ah + 48, b + 48, id2, 1u);
    mma_tf32(tmem, al + 48, b + 48, id1, 1u);
  }
}

// Geometry of one output tile in its class.  kp: x rows of a term rounded up to 16 (x hi
// and x lo are stacked kp rows apart; kpm for the widest term); mp: output rows rounded up to
// 16 (C hi and C lo are stacked mp rows apart).  Product-1 slots are sized for the tile (its
// output columns and its widest term), as many as fit: small blocks keep more copies in
// flight; the D tiles of the last slot must leave room for an M = 128 product's reads.  C
// slots hold the chunks of the tile's widest term.  A segment's slots are released together,
// so there are at least kSegChunks of them.  wc, nw: tensor-memory columns and number
// of the W^T accumulators.
__host__ __device__ constexpr int term_rows(int kdl) { return (kdl + 15) & ~15; }

template <class K>
struct TileGeom {
  int T, nvg, mg, mp, kpm, slot_f, nslots, b2_f, nb2, a2_f, wc, nw;
  bool fits;  // the class can run the tile
  __host__ __device__ explicit TileGeom(const TfTile& t) {
    T = t.t_end - t.t_begin;
    nvg = (t.nv + 7) >> 3;
    mg = (t.m + 7) >> 3;
    mp = (t.m + 15) & ~15;
    kpm = term_rows(t.kdg * 8);
    a2_f = nvg * 256;  // one W^T tile: nvg * 8 rows x 32 columns
    slot_f = (2 * nvg + kpm / 4) * 256;
    const int room = (K::kSmemF - K::kA2F - kRowsF - nvg * 256) / slot_f + 1, fit = K::kS1F / slot_f;
    nslots = room < fit ? room : fit;
    if (nslots > kMaxS1) nslots = kMaxS1;
    b2_f = 2 * mp * 32 * (kpm > 32 ? 2 : 1);
    nb2 = K::kB2F / b2_f;
    if (nb2 > kMaxB2) nb2 = kMaxB2;
    wc = 2 * kpm;
    nw = K::kWReg / wc;
    if (nw > kMaxW) nw = kMaxW;
    fits = t.m <= K::kMaxM && t.nv <= K::kMaxN && t.kdg * 8 <= K::kMaxKdl && nslots >= kSegChunks && nb2 >= 1 && nw >= 1 &&
           a2_f * 2 * (kpm > 32 ? 2 : 1) <= K::kA2F;
  }
};

// Persistent: K::kCtas CTAs per SM take tiles from a work queue (a counter in global
// memory, zeroed before the launch, handing out the tiles in the planner's order) until it
// is empty, so the pipeline runs on from one tile into the next.  A tile here is a run of
// the terms of one output tile, a multiple of kFlushTerms long (tc_plan_build); the FP32
// sum of every kFlushTerms terms goes to `part`, and k_tc_reduce adds an output tile's
// partial sums to y in FP64 in term order: the same additions in the same order whatever
// the split.  The producer thread takes each tile and passes its index to the other roles
// through a small ring in shared memory (tile_full / tile_empty); -1 ends the list.  Ring
// phases are kept per slot across tiles (bit masks of parities), and a tile whose product-1
// slot or W^T accumulator layout differs from the last one's waits for the last one's to be
// released first.
template <class K>
__global__ void __launch_bounds__(K::kThreads, K::kCtas)
    k_tc_matvec(const TfTile* __restrict__ tiles, const TfTask* __restrict__ tasks, const TfSrc* __restrict__ srcs,
                float* __restrict__ part, int* __restrict__ queue, const int* __restrict__ active, int ntiles) {
  extern __shared__ unsigned char smem_dyn[];
  float* sm = (float*)(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
  float* a2 = sm;                      // W^T: chunk 0 hi, lo, chunk 1 hi, lo (a2_f floats each)
  float* s1 = sm + K::kA2F;            // product-1 slots: D hi, D lo (nvg KB each), x hi, x lo (kp rows each)
  float* b2 = s1 + K::kS1F;            // C slots: per K chunk C hi (mp rows) then C lo (mp rows)
                                       // (an M = 128 product reads 16 KB from a D or W^T tile's start,
                                       // past its rows: rows of the result nobody uses)
  __shared__ __align__(8) Bars bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;
  __shared__ int tile_q[kTileQ];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == K::kMma1Warp) tmem_alloc(&tmem_slot, K::kTmem);
  if (tid == 0) {
    for (int s = 0; s < kMaxS1; ++s) {
      mbar_init_n(&bar.s1_full[s], 1);
      mbar_init_n(&bar.s1_empty[s], 1);
    }
    for (int s = 0; s < kMaxB2; ++s) {
      mbar_init_n(&bar.b2_full[s], 1);
    }
    for (int q = 0; q < kMaxW; ++q) {
      mbar_init_n(&bar.w_full[q], 1);
      mbar_init_n(&bar.w_empty[q], K::kConvThreads);
    }
    mbar_init_n(&bar.a2_full, K::kConvThreads);
    mbar_init_n(&bar.mma2_done, 1);
    mbar_init_n(&bar.drain1, 1);
    mbar_init_n(&bar.drain2, 1);
    mbar_init_n(&bar.never, 1);
    for (int r = 0; r < kTileQ; ++r) {
      mbar_init_n(&bar.tile_full[r], 1);
      mbar_init_n(&bar.tile_empty[r], 2 + K::kConvThreads);
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
    abort_flag = 0;
  }
  // stale shared memory past the rows a copy fills must be finite: it meets zeros in
  // padded products
  for (int e = tid * 4; e < K::kSmemF; e += K::kThreads * 4)
    *reinterpret_cast<float4*>(sm + e) = make_float4(0.f, 0.f, 0.f, 0.f);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_slot;
  if (tid == K::kMma1Warp * 32 && g_tc_inject) {
    // test hook: a wait on a barrier that nothing completes, with a short limit
    wait_or_abort(&bar.never, 0, &abort_flag, 4096);
  }
  __syncthreads();

  // the k-th tile of this CTA for the roles other than the producer (-1: none left, or
  // the CTA gave up)
  auto next_tile = [&](int k) -> int {
    const int r = k % kTileQ;
    if (!wait_or_abort(&bar.tile_full[r], (k / kTileQ) & 1, &abort_flag)) return -1;
    const int ti = tile_q[r];
    mbar_arrive(&bar.tile_empty[r]);
    return ti;
  };
  if (warp == K::kProducerWarp) {
    // ---- producer: takes the tiles; product-1 operands in the order the MMA thread
    // consumes them
    if (lane == 0 && !abort_flag) {
      uint32_t emp = 0, pend = 0, fpar = 0;  // per slot: release parity, fill not yet released, fill parity
      int last_slot_f = -1;
      bool ok = true;
      for (int k = 0; ok; ++k) {
        // take the next tile and pass it on
        const int r = k % kTileQ;
        if (k >= kTileQ && !wait_or_abort(&bar.tile_empty[r], (k / kTileQ - 1) & 1, &abort_flag)) break;
        int ti = atomicAdd(queue, 1);
        if (ti >= ntiles) ti = -1;
        tile_q[r] = ti;
        mbar_arrive(&bar.tile_full[r]);
        if (ti < 0) break;
        const TfTile tile = tiles[ti];
        if (!active[tile.inst]) continue;
        const TileGeom<K> g(tile);
        if (g.slot_f != last_slot_f) {
          // a new slot layout overlaps the old slots: all of them are released first
          for (int s = 0; s < kMaxS1 && ok; ++s)
            if ((pend >> s) & 1u) {
              ok = wait_or_abort(&bar.s1_empty[s], (emp >> s) & 1u, &abort_flag);
              emp ^= 1u << s;
              pend &= ~(1u << s);
            }
          last_slot_f = g.slot_f;
        }
        int slot = 0;
        for (int t = 0; t < g.T && ok; ++t) {
          const TfTask tk = tasks[tile.t_begin + t];
          const int kdg = (tk.kdl + 7) >> 3, kp = term_rows(tk.kdl);
          const uint32_t bytes = 2u * (g.nvg + kdg) * 1024u;
          for (int si = tk.s_begin; si < tk.s_end && ok; ++si) {
            const TfSrc S = srcs[si];
            for (int kk = 0; kk < S.nkc; ++kk) {
              if ((pend >> slot) & 1u) {
                if (!wait_or_abort(&bar.s1_empty[slot], (emp >> slot) & 1u, &abort_flag)) {
                  ok = false;
                  break;
                }
                emp ^= 1u << slot;
              }
              float* dst = s1 + slot * g.slot_f;
              const float* d = S.d + (int64_t)kk * S.d_cs;
              const float* x = S.x + (int64_t)kk * S.x_cs;
              mbar_expect_tx(&bar.s1_full[slot], bytes);
              bulk_g2s(dst, d, g.nvg * 1024u, &bar.s1_full[slot]);
              bulk_g2s(dst + g.nvg * 256, d + tile.dlo, g.nvg * 1024u, &bar.s1_full[slot]);
              bulk_g2s(dst + 2 * g.nvg * 256, x, kdg * 1024u, &bar.s1_full[slot]);
              bulk_g2s(dst + 2 * g.nvg * 256 + kp * 32, x + tile.xlo, kdg * 1024u, &bar.s1_full[slot]);
              pend |= 1u << slot;
              fpar ^= 1u << slot;
              if (++slot == g.nslots) slot = 0;
            }
          }
        }
      }
      // copies still in flight land before the CTA can exit: wait for the last fill of
      // every slot not yet released (a completed phase keeps testing complete while no
      // newer one starts)
      for (int s = 0; s < kMaxS1; ++s)
        if ((pend >> s) & 1u) wait_drain(&bar.s1_full[s], ((fpar >> s) & 1u) ^ 1u);
    }
  } else if (warp == K::kMma1Warp) {
    // ---- product 1: W^T = D x^T per source, segments of up to two K chunks per
    // accumulator
    if (lane == 0 && !abort_flag) {
      uint32_t ful = 0;              // per slot: parity of the next fill
      uint32_t wemp = 0, wpend = 0;  // per accumulator: release parity, written and not yet released
      int last_wc = -1;
      bool ok = true;
      for (int k = 0; ok; ++k) {
        const int ti = next_tile(k);
        if (ti < 0) break;
        const TfTile tile = tiles[ti];
        if (!active[tile.inst]) continue;
        const TileGeom<K> g(tile);
        if (g.wc != last_wc) {
          for (int q = 0; q < kMaxW && ok; ++q)
            if ((wpend >> q) & 1u) {
              ok = wait_or_abort(&bar.w_empty[q], (wemp >> q) & 1u, &abort_flag);
              wemp ^= 1u << q;
              wpend &= ~(1u << q);
            }
          last_wc = g.wc;
        }
        int slot = 0, q = 0;
        for (int t = 0; t < g.T && ok; ++t) {
          const TfTask tk = tasks[tile.t_begin + t];
          const int kp = term_rows(tk.kdl);
          const uint32_t id2 = idesc_tf32(2 * kp), id1 = idesc_tf32(kp);
          for (int si = tk.s_begin; si < tk.s_end && ok; ++si) {
            const TfSrc S = srcs[si];
            for (int k0 = 0; k0 < S.nkc; k0 += kSegChunks) {
              if ((wpend >> q) & 1u) {
                if (!wait_or_abort(&bar.w_empty[q], (wemp >> q) & 1u, &abort_flag)) {
                  ok = false;
                  break;
                }
                wemp ^= 1u << q;
              }
              const uint32_t wq = tmem + (uint32_t)(q * g.wc);
              const int k1 = min(S.nkc, k0 + kSegChunks);
              for (int kk = k0; kk < k1; ++kk) {
                if (!wait_or_abort(&bar.s1_full[slot], (ful >> slot) & 1u, &abort_flag)) {
                  ok = false;
                  break;
                }
                ful ^= 1u << slot;
                asm volatile("tcgen05.fence::after_thread_sync;");
                const int kv = kk == S.nkc - 1 ? S.klast : 32;
                const float* base = s1 + slot * g.slot_f;
                mma_pair_steps(wq, smem_desc(smem_u32(base)), smem_desc(smem_u32(base + g.nvg * 256)),
                               smem_desc(smem_u32(base + 2 * g.nvg * 256)), id2, id1, (kv + 7) >> 3, kk == k0);
                if (++slot == g.nslots) slot = 0;
              }
              if (!ok) break;
              mma_commit(&bar.w_full[q]);
              wpend |= 1u << q;
              if (++q == g.nw) q = 0;
            }
          }
        }
      }
      // every product issued has finished before tensor memory is released
      mma_commit(&bar.drain1);
      wait_drain(&bar.drain1, 0);
    }
  } else if (warp == K::kMma2Warp) {
    // ---- product 2: y^T = W^T C^T per term, fresh accumulator; this thread also loads
    // the C tiles (slot u % nb2 of the tile; the next fill of a slot waits for the
    // product that read it, and a tile starts once the last one's products have finished)
    if (lane == 0 && !abort_flag) {
      uint32_t bf = 0, lf = 0, filled = 0;  // per C slot: fill parity to wait, last fill, ever filled
      int gt = 0;                                    // terms of the CTA's earlier tiles
      int tiles_done = 0;
      bool ok = true;
      for (int k = 0; ok; ++k) {
        const int ti = next_tile(k);
        if (ti < 0) break;
        const TfTile tile = tiles[ti];
        if (!active[tile.inst]) continue;
        const TileGeom<K> g(tile);
        auto load_c = [&](int u) {
          const TfTask tk = tasks[tile.t_begin + u];
          const int nch = (tk.kdl + 31) >> 5, s = u % g.nb2;
          float* dst = b2 + s * g.b2_f;
          mbar_expect_tx(&bar.b2_full[s], 2u * nch * g.mg * 1024u);
          for (int c = 0; c < nch; ++c) {
            const float* src = tk.c + (int64_t)c * tk.c_cs;
            bulk_g2s(dst + c * 2 * g.mp * 32, src, g.mg * 1024u, &bar.b2_full[s]);
            bulk_g2s(dst + c * 2 * g.mp * 32 + g.mp * 32, src + tile.dlo, g.mg * 1024u, &bar.b2_full[s]);
          }
          lf ^= 1u << s;
          filled |= 1u << s;
        };
        for (int u = 0; u < min(g.nb2, g.T); ++u) load_c(u);
        const uint32_t idm = idesc_tf32(g.mp);
        for (int t = 0; t < g.T; ++t) {
          const int s = t % g.nb2;
          const TfTask tk = tasks[tile.t_begin + t];
          if (!wait_or_abort(&bar.a2_full, (gt + t) & 1, &abort_flag) ||
              !wait_or_abort(&bar.b2_full[s], (bf >> s) & 1u, &abort_flag)) {
            ok = false;
            break;
          }
          bf ^= 1u << s;
          asm volatile("tcgen05.fence::after_thread_sync;");
          const float* cb = b2 + s * g.b2_f;
          for (int c = 0; c * 32 < tk.kdl; ++c) {
            const int kv = min(32, tk.kdl - 32 * c);
            mma_triple_steps(tmem + K::kWReg, smem_desc(smem_u32(a2 + (2 * c) * g.a2_f)),
                             smem_desc(smem_u32(a2 + (2 * c + 1) * g.a2_f)), smem_desc(smem_u32(cb + c * 2 * g.mp * 32)),
                             smem_desc(smem_u32(cb + c * 2 * g.mp * 32 + g.mp * 32)), idm, (kv + 7) >> 3, c == 0);
          }
          mma_commit(&bar.mma2_done);
          if (t + g.nb2 < g.T) {
            if (!wait_or_abort(&bar.mma2_done, (gt + t) & 1, &abort_flag)) {
              ok = false;
              break;
            }
            load_c(t + g.nb2);
          }
        }
        gt += g.T;
        // the next tile's C layout may overlap this one's slots: its products finish first
        mma_commit(&bar.drain2);
        wait_drain(&bar.drain2, tiles_done & 1);
        ++tiles_done;
      }
      // every C copy has landed before the CTA exits (the last fill of every slot)
      for (int s = 0; s < kMaxB2; ++s)
        if ((filled >> s) & 1u) wait_drain(&bar.b2_full[s], ((lf >> s) & 1u) ^ 1u);
      if (tiles_done == 0) {
        mma_commit(&bar.drain2);
        wait_drain(&bar.drain2, 0);
      }
    }
  } else {
    // ---- converters: warp w reads tensor-memory lanes 32 (w % 4) .. (its output
    // columns); half h holds x rows 32 h .. of W^T and output rows kYR h .. of y.  A W^T
    // accumulator holds the hi part in columns [0, kp) and the stacked lo part in
    // [kp, 2 kp); their sum is the product.
    const int quarter = warp & 3, half = warp >> 2;
    const int n = quarter * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    uint32_t wful = 0;  // per accumulator: parity of the next fill
    int gt = 0;
    bool ok = !abort_flag;
    for (int k = 0; ok; ++k) {
      const int ti = next_tile(k);
      if (ti < 0) break;
      const TfTile tile = tiles[ti];
      if (!active[tile.inst]) continue;
      const TileGeom<K> g(tile);
      const int T = g.T;
      int q = 0, slot = 0;
      float* pp = part + tile.part;  // the partial sums of this run: m x nv values each
      float yacc[K::kYR];
#pragma unroll
      for (int j = 0; j < K::kYR; ++j) yacc[j] = 0.0f;
      auto drain_y = [&]() {
        asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
        for (int i = 0; i < K::kYR / 32; ++i) {
          if (K::kYR * half + 32 * i < tile.m) {
            float v[32];
            tmem_ld32(lane_base + (uint32_t)(K::kWReg + K::kYR * half + 32 * i), v);
#pragma unroll
            for (int j = 0; j < 32; ++j) yacc[32 * i + j] += v[j];
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
      };
      auto flush_y = [&]() {
        if (abort_flag) return;
#pragma unroll
        for (int j = 0; j < K::kYR; ++j) {
          const int r = K::kYR * half + j;
          if (r < tile.m && n < tile.nv) pp[r * tile.nv + n] = yacc[j];
          yacc[j] = 0.0f;
        }
        pp += tile.m * tile.nv;
      };
      for (int t = 0; t < T && ok; ++t) {
        const TfTask tk = tasks[tile.t_begin + t];
        const int kp = term_rows(tk.kdl);
        float wsum[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) wsum[j] = 0.0f;
        for (int si = tk.s_begin; si < tk.s_end && ok; ++si) {
          const float coef = srcs[si].coef;
          const int nseg = (srcs[si].nkc + kSegChunks - 1) / kSegChunks;
          for (int sg = 0; sg < nseg; ++sg) {
            if (!wait_or_abort(&bar.w_full[q], (wful >> q) & 1u, &abort_flag)) {
              ok = false;
              break;
            }
            wful ^= 1u << q;
            // the segment's products have finished, so its operand slots are free: a plain
            // arrival here costs a few cycles, a commit per slot 150 to 200 of the MMA
            // thread's
            for (int c = min(srcs[si].nkc - sg * kSegChunks, kSegChunks); c > 0; --c) {
              if (tid == 0) mbar_arrive(&bar.s1_empty[slot]);
              if (++slot == g.nslots) slot = 0;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            if (32 * half < tk.kdl) {
              const uint32_t wa = lane_base + (uint32_t)(q * g.wc + 32 * half);
              float v[32];
              tmem_ld32(wa, v);
#pragma unroll
              for (int j = 0; j < 32; ++j) wsum[j] = fmaf(coef, v[j], wsum[j]);
              tmem_ld32(wa + (uint32_t)kp, v);
#pragma unroll
              for (int j = 0; j < 32; ++j) wsum[j] = fmaf(coef, v[j], wsum[j]);
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            mbar_arrive(&bar.w_empty[q]);
            if (++q == g.nw) q = 0;
          }
        }
        if (!ok) break;
        // product 2 of the previous term has finished: its result is added to the
        // registers, and W^T in shared memory and y^T may be overwritten (the first term
        // of a tile follows the drain of the CTA's previous tile)
        if (t >= 1) {
          if (!wait_or_abort(&bar.mma2_done, (gt + t - 1) & 1, &abort_flag)) {
            ok = false;
            break;
          }
          drain_y();
          if (t % kFlushTerms == 0) flush_y();
        }
        if (n < g.nvg * 8 && 32 * half < kp) {
          float* ah = a2 + (2 * half) * g.a2_f;
          float* al = ah + g.a2_f;
#pragma unroll
          for (int gg = 0; gg < 8; ++gg) {
            float4 h, l;
            float* hv = &h.x;
            float* lv = &l.x;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float v = (32 * half + 4 * gg + e < tk.kdl) ? wsum[4 * gg + e] : 0.0f;
              hv[e] = tf32_round(v);
              lv[e] = tf32_round(v - hv[e]);
            }
            *reinterpret_cast<float4*>(ah + kmo(n, 4 * gg)) = h;
            *reinterpret_cast<float4*>(al + kmo(n, 4 * gg)) = l;
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(&bar.a2_full);
      }
      if (ok && T >= 1) {
        if (wait_or_abort(&bar.mma2_done, (gt + T - 1) & 1, &abort_flag)) drain_y();
        else ok = false;
      }
      flush_y();
      gt += T;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == K::kMma1Warp) tmem_free(tmem, K::kTmem);
}

// y of one output tile: its partial sums, in term order, in FP64 (one CTA per tile)
struct TfReduce { double* y; int64_t part; int ldy, m, nv, count, inst, pad; };

__global__ void __launch_bounds__(256) k_tc_reduce(const TfReduce* __restrict__ red, const float* __restrict__ part,
                                                  const int* __restrict__ active) {
  const TfReduce R = red[blockIdx.x];
  if (!active[R.inst]) return;
  const int mn = R.m * R.nv;
  for (int e = threadIdx.x; e < mn; e += 256) {
    const float* p = part + R.part + e;
    double v = (double)p[0];
    int f = 1;
    for (; f + 8 <= R.count; f += 8) {  // eight loads in flight ahead of the chain of additions
      float q[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) q[u] = p[(int64_t)(f + u) * mn];
#pragma unroll
      for (int u = 0; u < 8; ++u) v += (double)q[u];
    }
    for (; f < R.count; ++f) v += (double)p[(int64_t)f * mn];
    R.y[(int64_t)(e / R.nv) * R.ldy + e % R.nv] = v;
  }
}

// ------------------------------------------------------------------ tiny tiles

// four consecutive columns (col0 a multiple of 4, < 32) of a row of a tiled hi / lo operand
// (chunk 0) as hi + lo in FP64; hi + lo has at most 23 significant bits, so the FP32 sum is
// exact and one conversion per element is enough
__device__ __forceinline__ void tiled_val4(const float* __restrict__ p, int64_t lo, int row, int col0, double (&v)[4]) {
  const int64_t e = (int64_t)kmo(row, col0);
  const float4 h = *reinterpret_cast<const float4*>(p + e), l = *reinterpret_cast<const float4*>(p + e + lo);
  v[0] = (double)(h.x + l.x);
  v[1] = (double)(h.y + l.y);
  v[2] = (double)(h.z + l.z);
  v[3] = (double)(h.w + l.w);
}

// Output tiles of at most 4 x 4 elements whose terms have at most 4 x rows and whose
// sources are one K chunk (tile.tiny): the same sum y += C (sum_s coef_s x_s D_s^T) on
// CUDA cores in FP64 from the FP32 operand tiles (tensor-core products would be nearly all
// padding and the pipeline's per-term handoffs would dominate).  One CTA of four warps per
// tile.  The terms are dealt to 32 chains (chain l sums the terms l, l + 32, ... in order);
// of the next 4 x 32 terms warp w forms W of the w-th 32, one term per lane, and then warp i
// adds row i of C W of all four to the chains, lane = chain.  The chains are reduced in a
// fixed order and written once: deterministic, no atomics, the same sums as one warp per
// tile gives.  FP64 is what bounds it (a warp's FMA holds a sub-partition for 64 cycles):
// each element is converted once per use in a 4 x 4 product, and the tiles, far fewer than
// the sub-partitions, spread over four of them.  Measured (one matvec, random L=28, D=700):
// one warp per tile converting per product 3.33 ms, now 0.48 ms.
constexpr int kTinyWarps = 4;

__global__ void __launch_bounds__(kTinyWarps * 32) k_tc_tiny(const TfTile* __restrict__ tiles,
                                                             const TfTask* __restrict__ tasks,
                                                             const TfSrc* __restrict__ srcs,
                                                             const int* __restrict__ active) {
  __shared__ double Ws[kTinyWarps][16][32];  // W (k, j) of every lane's term
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const TfTile tile = tiles[blockIdx.x];
  if (!active[tile.inst]) return;
  double y[4] = {0.0, 0.0, 0.0, 0.0};  // row `warp` of the chain `lane`
  for (int t0 = tile.t_begin; t0 < tile.t_end; t0 += 32 * kTinyWarps) {
    const int t = t0 + 32 * warp + lane;
    if (t < tile.t_end) {
      const TfTask tk = tasks[t];
      double W[4][4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) W[k][j] = 0.0;
      for (int si = tk.s_begin; si < tk.s_end; ++si) {
        const TfSrc S = srcs[si];
        const double coef = (double)S.coef;
        double acc[4][4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[k][j] = 0.0;
        for (int r0 = 0; r0 < S.klast; r0 += 4) {
          double dv[4][4];
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < tile.nv) tiled_val4(S.d, tile.dlo, j, r0, dv[j]);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (k >= tk.kdl) break;
            double xv[4];
            tiled_val4(S.x, tile.xlo, k, r0, xv);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              if (r0 + r >= S.klast) break;
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (j < tile.nv) acc[k][j] = fma(xv[r], dv[j][r], acc[k][j]);
            }
          }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (k >= tk.kdl) break;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (j >= tile.nv) break;
            W[k][j] = fma(coef, acc[k][j], W[k][j]);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (k < tk.kdl && j < tile.nv) Ws[warp][4 * k + j][lane] = W[k][j];
    }
    __syncthreads();
    if (warp < tile.m) {
      for (int u = 0; u < kTinyWarps; ++u) {
        const int tu = t0 + 32 * u + lane;
        if (tu >= tile.t_end) break;
        const TfTask tk = tasks[tu];
        double cv[4];
        tiled_val4(tk.c, tile.dlo, warp, 0, cv);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (k >= tk.kdl) break;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < tile.nv) y[j] = fma(cv[k], Ws[u][4 * k + j][lane], y[j]);
        }
      }
    }
    __syncthreads();
  }
  if (warp >= tile.m) return;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    double v = y[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0 && j < tile.nv) tile.y[(int64_t)warp * tile.ldy + j] = v;
  }
}

// ------------------------------------------------------------------ conversions

// FP64 blocks -> tiled hi / lo (one CTA per block); identity blocks write their diagonal
__global__ void k_tiled_convert(const TfConv* __restrict__ m) {
  const TfConv M = m[blockIdx.x];
  const int n = M.identity ? M.rows : M.rows * M.cols;
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    int r, c;
    double v;
    if (M.identity) {
      r = c = e;
      v = 1.0;
    } else {
      r = e / M.cols;
      c = e - r * M.cols;
      v = M.src[e];
    }
    const int64_t off = ((int64_t)(c >> 5) * M.nrg + (r >> 3)) * 256 + ((c & 31) >> 2) * 32 + (r & 7) * 4 + (c & 3);
    const float f = (float)v;
    const float hi = tf32_round(f);
    M.dst[off] = hi;
    M.dst[off + M.lo] = tf32_round(f - hi);
  }
}

inline void ck(cudaError_t e, const char* what) {
  if (e != cudaSuccess) throw std::runtime_error(std::string(what) + ": " + cudaGetErrorString(e));
}

template <typename T>
T* upload(const std::vector<T>& v, Stream s) {
  if (v.empty()) return nullptr;
  T* p = (T*)dev_alloc(v.size() * sizeof(T), s);
  dev_h2d(p, v.data(), v.size() * sizeof(T), s);
  return p;
}

template <class K>
size_t smem_bytes() {
  return sizeof(float) * (size_t)K::kSmemF + 1024;
}

}  // namespace

// Output tiles whose partial sums are in memory together: their runs of terms by class (S, M,
// L; ranges of TcPlan::tiles) and their sums (a range of TcPlan::red).
struct TcPass {
  int nclass[3] = {0, 0, 0}, first[3] = {0, 0, 0}, grid[3] = {0, 0, 0};
  int red = 0, nred = 0;
};

struct TcPlan {
  TfTile* tiles = nullptr;     // runs of terms by pass and class, in queue order
  TfTask* tasks = nullptr;
  TfSrc* srcs = nullptr;
  TfConv* xb = nullptr;
  TfTile* tiny = nullptr;      // tiles for k_tc_tiny
  TfReduce* red = nullptr;     // output tiles and their partial sums
  float* part = nullptr;
  std::vector<TcPass> passes;  // one, unless the partial sums do not fit
  int ntiny = 0;
  int* queue = nullptr;        // the persistent kernels' tile counters, one per class
  int* active = nullptr;       // per instance: 0 = skip its tiles
  int ninst = 0;
  int nxb = 0;
  int launches = 0;  // kernels of one launch sequence
};

namespace {

int sm_count() {
  int dev = 0, n = 0;
  ck(cudaGetDevice(&dev), "device");
  ck(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev), "SM count");
  return std::max(n, 1);
}

}  // namespace

namespace {
// part_max: partial sums (floats) that may be in memory together (the largest tile's may be
// more); *part_need: how many there are at most
TcPlan* plan_build(const std::vector<const TcHost*>& inst, int64_t part_max, int64_t* part_need, Stream st) {
  TcPlan* P = new TcPlan;
  try {
    std::vector<TfSrc> s;
    std::vector<TfTask> t;
    std::vector<TfTile> tl;
    std::vector<TfConv> xb;
    const bool single = inst.size() == 1;
    int64_t inst_id = 0;
    for (const TcHost* H : inst) {
      if (single) break;  // one instance: its tables are uploaded as they are
      const int s0 = (int)s.size(), t0 = (int)t.size();
      s.insert(s.end(), H->s.begin(), H->s.end());
      for (TfTask q : H->t) {
        q.s_begin += s0;
        q.s_end += s0;
        t.push_back(q);
      }
      for (TfTile q : H->tiles) {
        q.t_begin += t0;
        q.t_end += t0;
        q.group += inst_id << 32;  // groups never span instances
        q.inst = (int)inst_id;
        tl.push_back(q);
      }
      ++inst_id;
      xb.insert(xb.end(), H->xb.begin(), H->xb.end());
    }
    const std::vector<TfTile>& tiles0 = single ? inst[0]->tiles : tl;
    // Tiles of output blocks with the same right sector read the same right-operator
    // blocks: they run together (so that those blocks stay in L2), groups in decreasing
    // order of their largest tile and tiles in decreasing order of work within a group
    // (the hardware starts CTAs in launch order, so the longest work does not finish last)
    std::unordered_map<int64_t, int64_t> gmax;
    for (const TfTile& q : tiles0) {
      int64_t& g = gmax[q.group];
      g = std::max(g, q.cost);
    }
    std::vector<int> order(tiles0.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
      const TfTile &A = tiles0[a], &B = tiles0[b];
      const int64_t ga = gmax[A.group], gb = gmax[B.group];
      if (ga != gb) return ga > gb;
      if (A.group != B.group) return A.group < B.group;
      return A.cost > B.cost;
    });
    std::vector<TfTile> sorted, tiny;
    sorted.reserve(tiles0.size());
    for (size_t i = 0; i < order.size(); ++i) (tiles0[order[i]].tiny ? tiny : sorted).push_back(tiles0[order[i]]);
    P->tiny = upload(tiny, st);
    P->ntiny = (int)tiny.size();
    // Classes, and runs of terms.  A run is long enough to pay for its pipeline fill (about
    // two terms' time) and short enough that every resident CTA gets several: 16 terms up
    // to kMaxRun.
    const int sms = sm_count();
    constexpr int kMaxRun = 64;
    auto cls = [](const TfTile& q) {
      return TileGeom<TileS>(q).fits ? 0 : TileGeom<TileM>(q).fits ? 1 : 2;
    };
    int64_t terms[3] = {0, 0, 0};
    std::vector<char> cl(sorted.size());
    for (size_t i = 0; i < sorted.size(); ++i) {
      cl[i] = (char)cls(sorted[i]);
      terms[(int)cl[i]] += sorted[i].t_end - sorted[i].t_begin;
    }
    const int ctas[3] = {sms * TileS::kCtas, sms * TileM::kCtas, sms * TileL::kCtas};
    int64_t run[3];
    for (int c = 0; c < 3; ++c) {
      run[c] = terms[c] / ((int64_t)8 * ctas[c]);
      run[c] = std::min<int64_t>(kMaxRun, std::max<int64_t>(kFlushTerms, run[c] / kFlushTerms * kFlushTerms));
    }
    std::vector<TfTile> runs[3], all;
    std::vector<TfReduce> red;
    red.reserve(sorted.size());
    int64_t part = 0, need = 0;  // of the current pass, of the largest
    auto close = [&]() {  // ends a pass
      TcPass ps;
      for (int c = 0; c < 3; ++c) {
        ps.first[c] = (int)all.size();
        ps.nclass[c] = (int)runs[c].size();
        ps.grid[c] = (int)std::min<size_t>(runs[c].size(), (size_t)ctas[c]);
        all.insert(all.end(), runs[c].begin(), runs[c].end());
        runs[c].clear();
        P->launches += ps.nclass[c] > 0;
      }
      ps.red = P->passes.empty() ? 0 : P->passes.back().red + P->passes.back().nred;
      ps.nred = (int)red.size() - ps.red;
      P->launches += ps.nred > 0;
      P->passes.push_back(ps);
      need = std::max(need, part);
      part = 0;
    };
    for (size_t i = 0; i < sorted.size(); ++i) {
      const TfTile& q = sorted[i];
      const int T = q.t_end - q.t_begin, nf = std::max(1, (T + kFlushTerms - 1) / kFlushTerms);
      const int64_t mn = (int64_t)q.m * q.nv, step = run[(int)cl[i]];
      if (part > 0 && part + nf * mn > part_max) close();
      red.push_back({q.y, part, q.ldy, q.m, q.nv, nf, q.inst, 0});
      int64_t t = 0;
      do {
        TfTile u = q;
        u.t_begin = q.t_begin + (int)t;
        u.t_end = q.t_begin + (int)std::min<int64_t>(T, t + step);
        u.part = part + t / kFlushTerms * mn;
        runs[(int)cl[i]].push_back(u);
        t += step;
      } while (t < T);
      part += nf * mn;
    }
    if (!red.empty()) close();
    *part_need = need;
    P->queue = (int*)dev_alloc(3 * sizeof(int), st);
    P->part = (float*)dev_alloc(sizeof(float) * std::max<int64_t>(need, 1), st);
    // a CTA that gives up leaves its partial sums as they are, and the reduction reads them
    // before the host sees the error: they hold numbers from the start
    dev_zero(P->part, sizeof(float) * std::max<int64_t>(need, 1), st);
    P->ninst = (int)inst.size();
    P->active = upload(std::vector<int>(inst.size(), 1), st);
    P->tiles = upload(all, st);
    P->red = upload(red, st);
    P->tasks = upload(single ? inst[0]->t : t, st);
    P->srcs = upload(single ? inst[0]->s : s, st);
    P->xb = upload(single ? inst[0]->xb : xb, st);
    P->nxb = (int)(single ? inst[0]->xb.size() : xb.size());
    P->launches += (P->nxb > 0) + (P->ntiny > 0);
  } catch (...) {
    tc_plan_free(P, st);
    throw;
  }
  return P;
}

}  // namespace

// The partial sums of all output tiles take some 8 % of a large plan (random L=28, D=2500: 0.25
// of 3.2 GB).  Where they do not fit, the tiles go in passes that share a smaller array: the
// same sums in the same order, with shorter queues.
TcPlan* tc_plan_build(const std::vector<const TcHost*>& inst, Stream st) {
  int64_t max = std::numeric_limits<int64_t>::max(), last = max;
  for (;;) {
    int64_t need = 0;
    try {
      return plan_build(inst, max, &need, st);
    } catch (const std::exception& e) {
      if (!no_room(e) || need == 0 || need >= last) throw;  // one tile's partial sums are the least
    }
    last = need;
    max = need / 2;
  }
}

int* tc_plan_active(TcPlan* p) { return p ? p->active : nullptr; }

void tc_plan_free(TcPlan* p, Stream s) {
  if (!p) return;
  dev_free(p->tiles, s);
  dev_free(p->tasks, s);
  dev_free(p->srcs, s);
  dev_free(p->xb, s);
  dev_free(p->queue, s);
  dev_free(p->tiny, s);
  dev_free(p->red, s);
  dev_free(p->part, s);
  dev_free(p->active, s);
  delete p;
}

namespace {

void tc_set_attributes() {
  static bool attr = false;
  if (attr) return;
  auto set = [](const void* f, size_t bytes) {
    ck(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes), "tc matvec smem");
  };
  set((const void*)k_tc_matvec<TileS>, smem_bytes<TileS>());
  set((const void*)k_tc_matvec<TileM>, smem_bytes<TileM>());
  set((const void*)k_tc_matvec<TileL>, smem_bytes<TileL>());
  attr = true;
}

template <class K>
void tc_run(const TcPlan* p, const TcPass& q, int c, cudaStream_t cs) {
  if (q.nclass[c] > 0)
    k_tc_matvec<K><<<q.grid[c], K::kThreads, smem_bytes<K>(), cs>>>(p->tiles + q.first[c], p->tasks, p->srcs, p->part,
                                                                    p->queue + c, p->active, q.nclass[c]);
}

void tc_enqueue(const TcPlan* p, void* const* ev, cudaStream_t cs) {
  if (ev) event_record(ev[0], cs);
  if (p->nxb > 0) k_tiled_convert<<<p->nxb, 256, 0, cs>>>(p->xb);
  if (ev) event_record(ev[1], cs);
  if (p->ntiny > 0)
    k_tc_tiny<<<p->ntiny, kTinyWarps * 32, 0, cs>>>(p->tiny, p->tasks, p->srcs, p->active);
  for (const TcPass& q : p->passes) {
    ck(cudaMemsetAsync(p->queue, 0, 3 * sizeof(int), cs), "tile queue reset");
    tc_run<TileL>(p, q, 2, cs);
    tc_run<TileM>(p, q, 1, cs);
    tc_run<TileS>(p, q, 0, cs);
    k_tc_reduce<<<q.nred, 256, 0, cs>>>(p->red + q.red, p->part, p->active);
  }
  if (ev) event_record(ev[2], cs);
  ck(cudaGetLastError(), "tc matvec launch");
}

struct TcGraph {
  cudaGraph_t g = nullptr;
  cudaGraphExec_t ex = nullptr;
  int launches = 0;
};

}  // namespace

void tc_plan_launch(const TcPlan* p, void* const* ev, Stream s) {
  tc_set_attributes();
  tc_enqueue(p, ev, (cudaStream_t)s);
  note_launches(p->launches);
}

void* tc_graph_create(const TcPlan* p) {
  tc_set_attributes();
  cudaStream_t cs;
  ck(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking), "graph stream");
  TcGraph* G = new TcGraph;
  G->launches = p->launches;
  cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    tc_enqueue(p, nullptr, cs);
    e = cudaStreamEndCapture(cs, &G->g);
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(&G->ex, G->g, 0);
  cudaStreamDestroy(cs);
  if (e != cudaSuccess) {
    if (G->g) cudaGraphDestroy(G->g);
    delete G;
    throw std::runtime_error(std::string("cuda graph of the batched matvec: ") + cudaGetErrorString(e));
  }
  return G;
}

void tc_graph_launch(void* g, Stream s) {
  TcGraph* G = (TcGraph*)g;
  ck(cudaGraphLaunch(G->ex, (cudaStream_t)s), "graph launch");
  note_launches(G->launches);
}

void tc_graph_free(void* g) {
  TcGraph* G = (TcGraph*)g;
  if (!G) return;
  if (G->ex) cudaGraphExecDestroy(G->ex);
  if (G->g) cudaGraphDestroy(G->g);
  delete G;
}

void tc_convert(const std::vector<TfConv>& m, Stream s) {
  if (m.empty()) return;
  TfConv* d = upload(m, s);
  k_tiled_convert<<<(int)m.size(), 256, 0, (cudaStream_t)s>>>(d);
  note_launches(1);
  ck(cudaGetLastError(), "tc convert launch");
  dev_free(d, s);
}

int tc_error_flag(Stream s) {
  int h = 0;
  ck(cudaMemcpyFromSymbolAsync(&h, g_tc_error, sizeof(int), 0, cudaMemcpyDeviceToHost, (cudaStream_t)s),
     "tc error flag");
  ck(cudaStreamSynchronize((cudaStream_t)s), "tc error flag");
  if (h) {
    const int zero = 0;
    ck(cudaMemcpyToSymbolAsync(g_tc_error, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, (cudaStream_t)s),
       "tc error flag");
    ck(cudaStreamSynchronize((cudaStream_t)s), "tc error flag");
  }
  return h;
}

void tc_inject_timeout(int on) {
  const int v = on ? 1 : 0;
  ck(cudaMemcpyToSymbol(g_tc_inject, &v, sizeof(int)), "tc inject");
}

}  // namespace dmrg
