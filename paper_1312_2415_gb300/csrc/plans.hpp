// Device-side plan tables shared by the FP64 and tensor-core kernels (internal).
#pragma once
#include "device.hpp"

namespace dmrg {

void note_launches(int64_t k);  // adds to the count kernel_launches() reports

// what one warp of the grouped GEMM does: nw 32-lane slices of a group's output from slice
// w0 on, or (ns > 1) the sidx-th of ns parts of the task list for one slice
struct GemmJob {
  int group, w0;
  short nw;
  unsigned char sidx, ns;
};

// ordered sums in rounds: a chunk (task, first column), or a group's range of chunks
struct GemmChunk {
  union { int task, begin; };
  union { int k0, end; };
};

struct GemmPlan {
  GemmTask* tasks = nullptr;
  GemmGroup* groups = nullptr;
  GemmJob* jobs[2] = {nullptr, nullptr};  // ordered sums, shared sums
  GemmChunk* chunks = nullptr;
  GemmJob* tiles = nullptr;  // groups in staged tiles, for either kind: (group, tile)
  int njobs[2] = {0, 0}, ntiles = 0;
  int kinds = 0;           // GEMM_ORDERED, GEMM_SHARED: the job tables it has
  bool overwrite = false;  // C = sum instead of C += sum
  bool rounds = false;  // ordered sums by k_gemm_rounds
  int64_t ntasks = 0;
};

struct CombPlan {
  CombSrc* src = nullptr;
  CombDst* dst = nullptr;
  int ndst = 0;
};

struct DiagPlan {
  DiagTerm* t = nullptr;
  DiagOut* o = nullptr;
  int n = 0;
};

}  // namespace dmrg
