// Launch parameters of the arbitrated-transfer simulation for 33 to 256
// accelerators (gmgsim_arbw.cu).  Private to the library: shared by the host
// translation unit (gmgsim_host.cu) and gmgsim_arbw.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gmg_layout.h"

namespace gsim {

struct ArbWParams {
  SimParams P;            // the full simulation's parameters (slot offsets inside P too)
  const uint16_t* link;   // [D*D] link id of each ordered accelerator pair (< D*D)
  const int32_t* pre_status;  // [K] optional: a nonzero entry is the candidate's status, not simulated
  int32_t shared_links;   // 1 if two ordered pairs share a link id
  int32_t xcap;           // transfers per candidate (sum over ops of min(successors, D-1))
  int32_t smem_arb;       // shared bytes of the arbitration state per warp
  int32_t few;            // 1: the instance with more registers and fewer blocks per SM
  int64_t smem_std;       // shared bytes of the simulation state of all warps of a block
  // byte offsets inside a warp's scratch slot
  int64_t off_cnt;        // int32 [N]  inputs present (joins)
  int64_t off_rmax;       // time  [N]  latest input arrival so far
  int64_t off_refs;       // int32 [N]  holds left on an op's own output copy
  int64_t off_nextop;     // int32 [N]  next started op of the same accelerator with intents to come
  int64_t off_xent;       // uint32 [E] arrived intent: producer << 8 | destination
  int64_t off_xnext;      // int32 [E]  next intent of the same accelerator
  int64_t off_lb;         // uint32 [ceil(D*D/32)] busy links (shared_links)
};

cudaError_t set_arbw_smem_limit();
const void* arbw_kernel_ptr(const DevGmg& g, bool few);
cudaError_t launch_arbw(const ArbWParams& A, int grid, int block, size_t smem,
                        cudaStream_t st);

}  // namespace gsim
