// What the kernels of every translation unit share: the call's parameters, and the kernels' templates in a namespace per
// block size.  Included by ersd.cu, which instantiates the streaming kernel's builds, and by ersd_cluster_bf16.cu and
// ersd_cluster_f32.cu, which instantiate the cluster kernels'.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include <type_traits>

#include "ersd.h"
#include "ersd_math.cuh"

namespace ersd {

constexpr int kPerThread = 8;  // consecutive vocabulary indices a thread owns in a tile
constexpr int kPartCap = 64;                  // partial-list entries per (row, role) in the workspace
constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

struct Entry {  // one arrival: race key (natural-log units) and token id
  double key;
  int32_t idx;
  int32_t pad;
};

// Workspace layout: one slot per logit row, whatever the call's sizes, so that a counter field
// is never reused as a partial-list field by a later call with other sizes (counters must be
// zero when a call starts; partial lists are always rewritten before they are read).
struct Slot {
  int counter;  // arrivals of the group whose first row this is; reset to 0 by the last arrival
  unsigned tau_code[2];  // per role: best threshold published so far (0 = none), see code_of_tau
  int pad;
  Entry part[2][kPartCap];  // per role: S partial lists of c entries each
};

struct TreeDesc {  // draft tree of one call, passed by value in kernel parameter space
  int16_t parent[ERSD_MAX_ROWS];
  int16_t first_child[ERSD_MAX_ROWS];
  int16_t next_sib[ERSD_MAX_ROWS];
  uint8_t rank[ERSD_MAX_ROWS];
  uint8_t nchild[ERSD_MAX_ROWS];
  uint8_t order[ERSD_MAX_ROWS];  // launch order of rows: rows with a draft row first
};

// The 16 bytes that start `a` bytes (0 < a < 16) into the 32 bytes lo, hi.  (`a` is the same for a
// whole row: the switch does not diverge.)
__device__ __forceinline__ uint4 bytes_from(const uint4& lo, const uint4& hi, unsigned a) {
  uint32_t w[5];
  switch (a >> 2) {
    case 0: w[0] = lo.x; w[1] = lo.y; w[2] = lo.z; w[3] = lo.w; w[4] = hi.x; break;
    case 1: w[0] = lo.y; w[1] = lo.z; w[2] = lo.w; w[3] = hi.x; w[4] = hi.y; break;
    case 2: w[0] = lo.z; w[1] = lo.w; w[2] = hi.x; w[3] = hi.y; w[4] = hi.z; break;
    default: w[0] = lo.w; w[1] = hi.x; w[2] = hi.y; w[3] = hi.z; w[4] = hi.w; break;
  }
  const unsigned bits = (a & 3) * 8;
  return make_uint4(__funnelshift_r(w[0], w[1], bits), __funnelshift_r(w[1], w[2], bits),
                    __funnelshift_r(w[2], w[3], bits), __funnelshift_r(w[3], w[4], bits));
}

// Programmatic dependent launch: a kernel launched with the attribute starts while the kernel before
// it on the stream still runs; everything it reads or writes in global memory comes after this wait,
// which ends when that kernel has completed and its stores are visible.
__device__ __forceinline__ void wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel start once every block of this one has come here (without it: when this one has
// ended, which still spares it most of a launch's latency).  Called past the wait, so that at most one
// launch waits on the device.
__device__ __forceinline__ void let_next_kernel_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

enum Mode { kSample = 0, kVerify = 1 };

struct Params {
  const void* target;  // target logits (race_sample: the logits)
  const void* draft;
  const int32_t* given_tok;  // [B, k] drafted tokens when they are given instead of draft rows
  int64_t ld_t, ld_d;
  const uint64_t* seeds;
  const uint32_t* seq_ids;
  const uint32_t* pos_offsets;
  const float* temps;
  int64_t ts_b, ts_r;
  float T;
  int B, rows, V;
  int S, per_chunk;
  int threads;  // threads per block of the kernel variant this call launches (128 or 256)
  int mode;
  int c_sample;          // arrivals per row in sample mode
  int draft_rows;        // draft rows per sequence (k, or N + 1 for trees)
  int depth;             // columns of out_tokens - 1
  int chain_outputs;     // 1: out_draft_* are [B, k] indexed by position (sequence variant)
  int aligned_t, aligned_d;
  int32_t* out_tokens;
  int32_t* out_accept_len;
  int32_t* out_path;
  int32_t* out_draft_tok;
  float* out_draft_key;
  int32_t* out_target_tok;
  float* out_target_key;
  float* out_key;        // sample mode
  uint32_t* near_tie;    // count of races with two consecutive arrivals closer than 1e-5 (nullable)
  int extra;             // 1 when near-ties are counted: every race is run for one more arrival
  int top_picks;         // its short way: groups a warp screens for races of three arrivals and more
  int top_cmax;          // cluster kernel for several arrivals: most arrivals any race of the call wants
  int top_split;         // the same kernel: 0, or 1 + the number of nodes with children when every row gets its own cluster
  int early;             // cluster kernels: let the next kernel on the stream start early
  Slot* slots;
};

// ---------------------------------------------------------------------------------------------
// The kernel, compiled for two block sizes: many rows are raced by 128-thread blocks (seven per
// SM: more, smaller work items and a shorter last wave), few rows by 256-thread blocks (four per
// SM: a row's thresholds are shared by more warps, half as many blocks to set up).
// ---------------------------------------------------------------------------------------------
namespace b256 {
constexpr int kThreads = 256, kMinBlocks = 4;
constexpr bool kMany = false;
#include "ersd_kernel.inc"
}  // namespace b256
namespace b128 {
constexpr int kThreads = 128, kMinBlocks = 7;
constexpr bool kMany = false;
#include "ersd_kernel.inc"
}  // namespace b128
// The same two for calls of few rows with races that want several arrivals (tree and batch
// drafting, top_c > 1) and for every call with a race of more than 32 arrivals: see launch().
namespace b256m {
constexpr int kThreads = 256, kMinBlocks = 4;
constexpr bool kMany = true;
#include "ersd_kernel.inc"
}  // namespace b256m
namespace b128m {
constexpr int kThreads = 128, kMinBlocks = 7;
constexpr bool kMany = true;
#include "ersd_kernel.inc"
}  // namespace b128m
namespace b128 {
#include "ersd_cluster.inc"
}  // namespace b128
namespace b256 {
#include "ersd_cluster.inc"
#include "ersd_cluster_top.inc"
}  // namespace b256

// The build of the cluster kernels for a call, see ersd_cluster_select.inc.
__attribute__((visibility("hidden"))) const void* cluster_kernel_bf16(bool aligned, bool verify, int cmax, int roles, bool staged, bool small, int short_way);
__attribute__((visibility("hidden"))) const void* cluster_kernel_f32(bool aligned, bool verify, int cmax, int roles, bool staged, bool small, int short_way);

}  // namespace ersd
