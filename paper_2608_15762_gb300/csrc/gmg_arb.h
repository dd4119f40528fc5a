// Launch parameters of the arbitrated-transfer simulation (sim_batch with
// transfer_mode = GMG_TRANSFER_ARBITRATED).  Private to the library: shared
// by the host translation unit (gmgsim_host.cu) and gmgsim_arb.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gmg_layout.h"

namespace gsim {

// An arbitrated base snapshot keeps, beside the simulation state of every
// checkpoint (DevBase), the arbiter's state at that instant in one arena per
// checkpoint: the per-op input counters, latest arrivals, holds, remote sets,
// list links and hold times, every lane's sending transfer and list ends, and
// the receiving endpoints and links in use.
struct ArbCk {
  uint8_t* arena;         // [nck][bytes]
  int64_t bytes;          // per checkpoint
  int64_t off_cnt, off_rmax, off_refs, off_rmask, off_nextop, off_hold;  // per op (times as int64)
  int64_t off_lanes;      // [32][7] int64: xd, xdp, ah, al, uh, lt, fu
  int64_t off_warp;       // int64 xev, recvm; then uint32 lbits[32]
};

struct ArbParams {
  SimParams P;            // the full simulation's parameters (slot offsets inside P too)
  const uint16_t* link;   // [D*D] link id of each ordered accelerator pair (< D*D)
  int32_t shared_links;   // 1 if two ordered pairs share a link id (else the sender check covers links)
  int32_t xcap;           // transfers per candidate (sum over ops of min(successors, D-1))
  int32_t smem_arb;       // shared bytes of the arbitration state per warp
  int32_t blocks;         // blocks per SM of the instance that sim_batch launches (kArbBlocks and more)
  int64_t smem_std;       // shared bytes of the simulation state of all warps of a block
  // byte offsets inside a warp's scratch slot
  int64_t off_cnt;        // int32 [N]  inputs present (joins)
  int64_t off_rmax;       // time  [N]  latest input arrival so far
  int64_t off_refs;       // int32 [N]  holds left on an op's own output copy
  int64_t off_rmask;      // uint32 [N] destinations left of an op's transfers
  int64_t off_nextop;     // int32 [N]  next op of the accelerator's list (ops with transfers to come)
  const int32_t* pre_status;  // [K] optional: a nonzero entry is the candidate's status, not simulated
  ArbCk ck;               // arbitrated base snapshot (base and resumed incremental launches)
};

// Incremental candidates under arbitrated transfers: row k = the base row with
// candidate k's moves applied (rows [K][ld]); status[k] = the move list's
// GMG_SIM_* code (GMG_SIM_BADBASE for every candidate if *base_status is not OK).
cudaError_t launch_expand_moves(const uint8_t* base_row, const int32_t* base_status, int32_t ld, int32_t n,
                                int32_t D, const int32_t* off, const int32_t* op, const uint8_t* dev, int32_t K,
                                uint8_t* rows, int32_t* status, cudaStream_t st);

// Blocks per SM of the arbitrated kernels on at most 32 accelerators; how many ops
// and accelerators a graph may have that takes 7.
constexpr int kArbBlocks = 5;
constexpr int kArbSevenOps = 1024, kArbSevenDevices = 12;

// Kernel entry of one instance (for occupancy queries) and the launcher.
const void* arb_kernel_ptr(const DevGmg& g, int blocks);
cudaError_t launch_arb(const ArbParams& A, int grid, int block, size_t smem, cudaStream_t st);

// The arbitrated base snapshot (one warp) and the incremental candidates
// resumed from it (at most 32 accelerators).
const void* arb_base_kernel_ptr(bool types);
const void* arb_inc_kernel_ptr(const DevGmg& g);
cudaError_t launch_arb_base(bool types, const ArbParams& A, size_t smem, cudaStream_t st);
cudaError_t launch_arb_inc(const ArbParams& A, int grid, int block, size_t smem, cudaStream_t st);

}  // namespace gsim
