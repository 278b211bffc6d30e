// libersd: exponential-race speculative decoding kernels for sm_100a and their C entry points.
//
// One thread block streams one chunk of one logit row (or of a draft/target
// row pair that shares its race variables).  Logits arrive through a
// shared-memory ring filled by cp.async; per group of eight vocabulary indices
// a thread draws the Philox words and compares one cheap lower bound of the
// eight race keys with the block's running threshold.  The few groups that
// survive are screened index by index in single precision and the survivors of
// that are decided in double precision and kept in per-warp sorted lists.
// Lists are merged per block, exchanged through a small workspace, and the
// last block of a sequence turns the winners into the accepted prefix
// (sequence scan or tree walk) in the same launch.
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <mutex>
#include <type_traits>

#include "ersd.h"
#include "ersd_device.cuh"

namespace ersd {

template <int DT>
__global__ void ersd_row_keys_kernel(const void* row, int V, float T, uint64_t seed, uint32_t seq,
                                     uint32_t pos, int mode, float* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= V) return;
  float z;
  if (DT == ERSD_BF16) z = __uint_as_float((uint32_t)((const uint16_t*)row)[i] << 16);
  else z = ((const float*)row)[i];
  const uint32_t x = token_word(seed, seq, pos, (uint32_t)i);
  if (mode == 0) {
    out[i] = (float)exact_key(x, z, T);
  } else if (mode == 2) {
    // the deciding key against the CUDA math library's log / log1p, in units of 1e-12
    const double w = ((double)x + 0.5) * (1.0 / 4294967296.0);
    const double ref = (T == 0.0f) ? -(double)z : log(-log1p(-w)) - (double)z / (double)T;
    out[i] = (float)((exact_key(x, z, T) - ref) * 1e12);
  } else {
    const float c2 = (float)(1.4426950408889634 / (T == 0.0f ? 1.0 : (double)T));
    const float lg = (T == 0.0f) ? 0.0f : screen_lg2_e(x);
    out[i] = fmaf(-z, c2, lg) * kLn2;
  }
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
static thread_local int g_last_cuda_error = 0;
static thread_local char g_last_launch[192] = "";  // ersd_last_launch(): what this thread's last call launched

// The error stays with the library: the runtime keeps it per thread too, where the next check of some
// other launch on this thread would find it.
static int cuda_fail(cudaError_t e) {
  g_last_cuda_error = (int)e;
  (void)cudaGetLastError();
  return ERSD_ECUDA;
}

// A launch that may start while the kernel before it on the stream still runs (see
// wait_for_previous_kernel), in clusters of CL blocks.
struct Launch {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[2];
  Launch(dim3 grid, unsigned threads, size_t smem, cudaStream_t st, unsigned CL = 1) {
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = CL;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = CL > 1 ? 2 : 1;
  }
  Launch(const Launch&) = delete;
};

struct OwnedWorkspace {
  void* ptr = nullptr;
  size_t bytes = 0;
};
static std::mutex g_ws_mutex;
static OwnedWorkspace g_ws[64];

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

static size_t workspace_bytes(int64_t B, int64_t rows) {
  return (size_t)B * (size_t)rows * sizeof(Slot);
}

// The private workspace of a device is zeroed on the stream of the call that (re)allocates it, so
// that the zeroing is ordered before that call's kernel whatever kind of stream it is.
static int get_workspace(const ersd_opts& o, size_t need, void** ws, cudaStream_t stream) {
  if (o.workspace) {
    if (o.workspace_bytes < need) return ERSD_EWORKSPACE;
    if (((uintptr_t)o.workspace & 15) != 0) return ERSD_EALIGN;
    *ws = o.workspace;
    return ERSD_OK;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e);
  if (dev < 0 || dev >= 64) return ERSD_EUNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_ws_mutex);
  OwnedWorkspace& w = g_ws[dev];
  if (w.bytes < need) {
    if (w.ptr) {
      e = cudaFree(w.ptr);
      w.ptr = nullptr;
      w.bytes = 0;
      if (e != cudaSuccess) return cuda_fail(e);
    }
    const size_t grow = align_up(need + need / 2, 1 << 20);
    e = cudaMalloc(&w.ptr, grow);
    if (e != cudaSuccess) {
      w.ptr = nullptr;
      return cuda_fail(e);
    }
    e = cudaMemsetAsync(w.ptr, 0, grow, stream);
    if (e != cudaSuccess) return cuda_fail(e);
    w.bytes = grow;
  }
  *ws = w.ptr;
  return ERSD_OK;
}

static ersd_opts read_opts(const ersd_opts* opts) {
  ersd_opts o;
  memset(&o, 0, sizeof o);
  if (opts) {
    size_t n = opts->struct_size;
    if (n == 0 || n > sizeof o) n = sizeof o;
    memcpy(&o, opts, n);
  }
  return o;
}

static bool temp_ok(float T) { return T >= 0.0f && T < INFINITY; }

static int elem_size(int dt) { return dt == ERSD_BF16 ? 2 : 4; }

static bool rows_aligned(const void* base, int64_t ld, int dt) {
  return ((uintptr_t)base & 15) == 0 && ((ld * elem_size(dt)) & 15) == 0;
}

constexpr int kMinChunkTiles = 8;  // smallest chunk of a row that the default split makes

// Multiprocessors of the current device (asked once per device; 148 on a B200).
static int sm_count() {
  static std::mutex m;
  static int count[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  std::lock_guard<std::mutex> lock(m);
  if (!count[dev]) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
      (void)cudaGetLastError();
      n = 148;
    }
    count[dev] = n;
  }
  return count[dev];
}

// Block size of a call: opts->block_threads if given, else 128-thread blocks when there are enough
// rows to give every one of their (twice as many) resident-block slots a chunk, 256 otherwise.
static int choose_threads(const ersd_opts& o, int64_t units, int* threads) {
  if (o.block_threads == 0) *threads = units >= (int64_t)sm_count() * b128::kMinBlocks ? 128 : 256;
  else if (o.block_threads == 128 || o.block_threads == 256) *threads = (int)o.block_threads;
  else return ERSD_EINVAL;
  return ERSD_OK;
}

// Thread blocks per row.
static int choose_split(const ersd_opts& o, int64_t units, int V, int cmax, int threads) {
  int smax = kPartCap / cmax;
  if (smax > ERSD_MAX_SPLIT) smax = ERSD_MAX_SPLIT;
  if (smax < 1) smax = 1;
  const int tile = threads * kPerThread;
  const int ntiles = (V + tile - 1) / tile;
  int S;
  if (o.split_v) {
    S = (int)o.split_v;
    if (S > ntiles) S = ntiles;
  } else {
    // about 1.7 blocks per SM: a block costs as much set-up, first threshold, merge and finish as
    // eight tiles of streaming, so more chunks than the SMs need to be busy only add work
    // (measured on calls of 48 to 400 rows: 5 to 15 % quicker than one block per resident slot)
    const int64_t slots = (int64_t)sm_count() * (threads == 128 ? b128::kMinBlocks : b256::kMinBlocks);
    // (races of several arrivals: their rare path is the long one, and shorter chunks bound it;
    // there a block per resident slot stays the better choice)
    const int64_t wanted = cmax > 1 ? slots : ((int64_t)sm_count() * 27) / 16;
    S = (int)((wanted + units - 1) / units);
    // whole rows that make more than one wave, and rows of uneven cost (trees): halves even out the last wave
    if (S < 2 && (units > slots || cmax > 1) && (int64_t)ntiles * tile >= 4 * kMinChunkTiles * b256::kTile) S = 2;
    const int by_v = ntiles / kMinChunkTiles;
    if (S > by_v) S = by_v;
  }
  if (S > smax) S = smax;
  if (S < 1) S = 1;
  return S;
}

static void set_chunks(Params& p, int S) {
  const int tile = p.threads * kPerThread;
  int per = (p.V + S - 1) / S;
  per = (per + tile - 1) / tile * tile;
  p.per_chunk = per;
  p.S = (p.V + per - 1) / per;
}

static int build_tree(const int32_t* parent, int N, TreeDesc* t, int* depth_out, int* cmax_out) {
  const int nodes = N + 1;
  if (parent[0] != -1) return ERSD_EINVAL;
  int depth[ERSD_MAX_ROWS];
  int last_child[ERSD_MAX_ROWS];
  memset(t, 0, sizeof *t);
  for (int n = 0; n < nodes; ++n) {
    t->first_child[n] = -1;
    t->next_sib[n] = -1;
    last_child[n] = -1;
  }
  t->parent[0] = -1;
  depth[0] = 0;
  int D = 0, cmax = 1;
  for (int n = 1; n < nodes; ++n) {
    const int par = parent[n];
    if (par < 0 || par >= n) return ERSD_EINVAL;
    t->parent[n] = (int16_t)par;
    if (t->nchild[par] >= ERSD_MAX_TOP_C) return ERSD_EUNSUPPORTED;
    t->rank[n] = t->nchild[par]++;
    if (last_child[par] < 0) t->first_child[par] = (int16_t)n;
    else t->next_sib[last_child[par]] = (int16_t)n;
    last_child[par] = n;
    depth[n] = depth[par] + 1;
    if (depth[n] > D) D = depth[n];
    if (t->nchild[par] > cmax) cmax = t->nchild[par];
  }
  int k = 0;
  for (int n = 0; n < nodes; ++n)
    if (t->nchild[n] > 0) t->order[k++] = (uint8_t)n;
  for (int n = 0; n < nodes; ++n)
    if (t->nchild[n] == 0) t->order[k++] = (uint8_t)n;
  *depth_out = D;
  *cmax_out = cmax;
  return ERSD_OK;
}

// The build of the race kernel for a call, and its dynamic shared memory.
struct RaceKernel {
  void (*kernel)(Params, TreeDesc);
  size_t smem;
};
template <int DT, bool AL>
static RaceKernel race_kernel_of(bool many, int threads) {
  if (many) return threads == 128 ? RaceKernel{b128m::ersd_race_kernel<DT, AL>, sizeof(b128m::Shared<DT>)}
                                  : RaceKernel{b256m::ersd_race_kernel<DT, AL>, sizeof(b256m::Shared<DT>)};
  return threads == 128 ? RaceKernel{b128::ersd_race_kernel<DT, AL>, sizeof(b128::Shared<DT>)}
                        : RaceKernel{b256::ersd_race_kernel<DT, AL>, sizeof(b256::Shared<DT>)};
}
static RaceKernel race_kernel(bool bf16, bool aligned, bool many, int threads) {
  if (bf16) return aligned ? race_kernel_of<ERSD_BF16, true>(many, threads) : race_kernel_of<ERSD_BF16, false>(many, threads);
  return aligned ? race_kernel_of<ERSD_F32, true>(many, threads) : race_kernel_of<ERSD_F32, false>(many, threads);
}

// What a kernel needs before its first launch on a device: its dynamic shared memory allowed, and
//   carveout: the largest shared-memory carveout asked for (a hint to the driver: four resident blocks of
//             the streaming kernel need about 180 KB);
//   cluster:  the opt-in for clusters of 16 blocks; *limit = the largest cluster (a power of two) that it
//             can be launched in: 16 where that is granted and such a cluster fits, else 8.
// Done when a call first wants the kernel: asking for all cluster builds (40 then) at once was 3 of the 32 ms that a
// process's first call took (drafting 32.1 -> 29.4 ms, verification 33.6 -> 30.2; most of the rest is loading the code).
struct KernelState {
  const void* kernel;
  uint64_t ready, sixteen;  // bits: devices
};
static int prepare_kernel(const void* kernel, size_t smem, bool carveout, bool cluster, int* limit) {
  static std::mutex m;
  static KernelState known[96];  // (no fewer than there are builds)
  static int count;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e);
  if (dev < 0 || dev >= 64) return ERSD_EUNSUPPORTED;
  const uint64_t bit = (uint64_t)1 << dev;
  std::lock_guard<std::mutex> lock(m);
  int at = 0;
  while (at < count && known[at].kernel != kernel) ++at;
  KernelState fresh = {kernel, 0, 0};
  KernelState& k = at < 96 ? known[at] : fresh;
  if (at == count && at < 96) {
    k = fresh;
    ++count;
  }
  if (!(k.ready & bit)) {
    if (carveout) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess && smem) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e);
    if (cluster) {
      int n = 0;
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e == cudaSuccess) {
        Launch l(dim3(16, 1, 1), b256::kThreads, smem, nullptr, 16);
        l.cfg.attrs = &l.at[1];  // (the cluster's size alone)
        l.cfg.numAttrs = 1;
        e = cudaOccupancyMaxActiveClusters(&n, kernel, &l.cfg);
      }
      if (e == cudaSuccess && n >= 1) k.sixteen |= bit;
      (void)cudaGetLastError();  // a refused opt-in only means clusters of eight
    }
    k.ready |= bit;
  }
  if (limit) *limit = (k.sixteen & bit) ? 16 : 8;
  return ERSD_OK;
}

// `many`: some race of the call wants several arrivals (a tree node with several children,
// top_c > 1).  Calls of up to two rows per SM then take the variant of the kernel that pools the
// block's decided indices (measured: a star of 8 at B=1 48 -> 42 us, the 17-node tree 35 -> 33 us;
// at 544 rows the pooling costs 0.7 % instead).
// cmax: most arrivals any race of the call wants.  The builds for races of several arrivals take
// calls of few rows (their loop is slower, their rare path quicker) and every call with a race of
// more than 32 arrivals (only they hold two list entries per lane).
static int launch(const Params& p, const TreeDesc& tree, int dt, int cmax, cudaStream_t st) {
  const bool many = cmax > 32 || (cmax > 1 && (int64_t)p.B * p.rows <= 2 * sm_count());
  // grid (sequence, row in launch order, chunk): blocks are dispatched x fastest, z slowest, which
  // is the chunk-major order the kernel counts on, and the kernel needs no division to decode
  if (p.rows > 65535 || p.S > 65535) return ERSD_EUNSUPPORTED;
  const dim3 grid((unsigned)p.B, (unsigned)p.rows, (unsigned)p.S);
  const RaceKernel k = race_kernel(dt == ERSD_BF16, p.aligned_t && p.aligned_d, many, p.threads);
  const int pst = prepare_kernel((const void*)k.kernel, k.smem, true, false, nullptr);
  if (pst != ERSD_OK) return pst;
  snprintf(g_last_launch, sizeof g_last_launch, "ersd_race_kernel<%s>%s: %d threads x (%d, %d, %d) blocks, %d chunk(s) per row",
           dt == ERSD_BF16 ? "bf16" : "f32", many ? " (pooled thresholds)" : "", p.threads, p.B, p.rows, p.S, p.S);
  Launch l(grid, (unsigned)p.threads, k.smem, st);
  const cudaError_t e = cudaLaunchKernelEx(&l.cfg, k.kernel, p, tree);
  return e == cudaSuccess ? ERSD_OK : cuda_fail(e);
}

// ---------------------------------------------------------------------------------------------
// One cluster of thread blocks per position (ersd_cluster.inc, ersd_cluster_top.inc).
// ---------------------------------------------------------------------------------------------
// Default choice for races of one arrival, by the logits of the call (positions x V).  32-bit logits and
// rows of up to 65536 always take the cluster kernel (verification, cluster kernel / streaming
// kernel: 6000 positions of 15048 bf16 logits 112.5 / 173 us, 2300 of 48000 120.9 / 134.5; 32-bit: 2000 of
// 32000 92.1 / 148, 150 of 128256 39.6 / 60, 2300 of 151936 459 / 653; sampling of 2304 x 128256 256 /
// 325).  The streaming kernel spends less on an index, once its thresholds have settled, and more on
// starting: it takes longer bf16 rows from a number of logits on (verification: at 65256 logits 1500
// positions 111.2 / 113.5 and 2250 157.2 / 159.5; at 100000 500 65.5 / 69.7; at 128256 400 66.4 / 68.8, 450
// 77.9 / 81.0, 576 91.8 / 87.5; at 151936 300 64.0 / 71.4 and 400 81.4 / 76.4; trees: at 128256 450 rows 85.7 /
// 83.8.  Sampling and given tokens, one row per position: at 128256 800 93.1 / 95.1; given tokens at 151936 576
// 89.4 / 83.3, 640 98.6 / 91.9).
struct ClusterLimit {
  int row;         // rows of up to this many logits ...
  int64_t logits;  // ... take the cluster kernel while the call has no more logits than this
};
// Races of several arrivals gain more from it, but see top_streams (trees of 17 nodes of bf16 logits, time of the
// cluster kernel / of the streaming kernel: 16 of 128256 0.72, 24 of 100000 1.02, 64 of 64000 0.99, 200 of 40000 0.92,
// and of 48000, where a row takes two blocks, 233 / 193 us).  Trees of more than 131072 logits a row stream from
// 20M logits on although the cluster kernel would be quicker there (8 x 17 nodes of 151936: 39.4 / 63.7 us): the
// tests fix which kernel takes that call.
constexpr ClusterLimit kClusterLimits[3][4] = {  // bf16: one row per position, draft and target row, the same in trees
    {{65536, INT64_MAX}, {INT32_MAX, 100 << 20}},
    {{65536, INT64_MAX}, {INT32_MAX, 56 << 20}},
    {{40960, INT64_MAX}, {65536, 80 << 20}, {131072, 40 << 20}, {INT32_MAX, 19 << 20}}};
// The number of blocks up to which a tree's rows get a cluster each (one block per SM and a half)
constexpr int64_t kClusterSplitBlocks = 384;
constexpr size_t kClusterSmemBytes = 200 * 1024;  // dynamic shared memory a block of the cluster kernels may use

// Tiles per block that fit (roles = rows raced together: 1, or 2 for a draft/target pair; cmax > 1:
// the kernel for races of several arrivals, which keeps its lists behind the rows).
static int cluster_max_tiles(int dt, int roles, int cmax, bool aligned) {
  const size_t per_tile = dt == ERSD_BF16 ? b256::cluster_role_bytes<ERSD_BF16>(1, aligned) : b256::cluster_role_bytes<ERSD_F32>(1, aligned);
  const size_t lists = cmax > 1 ? b256::top_list_bytes(cmax, b256::kClusterMax) : 0;
  return (int)((kClusterSmemBytes - lists) / (per_tile * (size_t)roles));
}

template <int DT, bool AL>
static const void* cluster_kernel(bool verify, int cmax, int roles, bool staged, bool small, int short_way) {
  return DT == ERSD_BF16 ? cluster_kernel_bf16(AL, verify, cmax, roles, staged, small, short_way)
                         : cluster_kernel_f32(AL, verify, cmax, roles, staged, small, short_way);
}

// Whether a call can take a cluster kernel at all; cmax: most arrivals any of its races wants.
static bool cluster_applies(const Params& p, int dt, int cmax) {
  // (eight blocks, the portable cluster size, must be able to stage the rows of a position)
  const bool top = cmax > 1;
  const int roles = (p.mode == kVerify && p.draft) ? 2 : 1;
  const int64_t ntiles = ((int64_t)p.V + b256::kTile - 1) / b256::kTile;
  if (top && cmax > b256::kTopMaxC) return false;
  if (ntiles > 8 * (int64_t)cluster_max_tiles(dt, roles, cmax, p.aligned_t && p.aligned_d)) return false;
  if (top) {
    if (p.given_tok || p.chain_outputs || p.extra) return false;
  } else if (p.mode == kVerify && p.rows > 32) {
    return false;
  }
  return p.rows <= 65535 && p.B <= 65535;
}

// Whether the call's logits are staged in shared memory.  Staged blocks have the
// shortest path through a position but only two or three of them fit an SM; unstaged ones read the rows
// tile by tile while they compute, four (of 128 threads: eight) to an SM, and fetch the few logits
// they need again from L2.  Staged / unstaged us, verification of bf16 rows: 10 x 128256 logits 9.8 /
// 10.4, 40 x 32000 9.7 / 10.2, 500 x 4096 11.0 / 11.3, 80 x 32000 13.2 / 12.3, 40 x 128256 22.2 / 15.9, 800
// x 15048 32.5 / 25.8; sampling: 16 x 128256 8.0 / 8.6, 100 x 32000 9.1 / 9.0, 100 x 128256 21.8 /
// 19.0; 32-bit: verification of 500 x 4096 14.1 / 12.2, sampling of 100 x 32000 12.6 / 8.8.
// Several arrivals: 50 x 32000 11.0 / 11.3, 12 x 128256 12.5 / 11.4, 64 x 128256 30.0 / 22.4; a tree of 17
// nodes of 32000 logits, 10 sequences 31.7 / 21.6.
constexpr int64_t kClusterStagedBytes = 8 << 20, kClusterStagedBytesTop = 4 << 20;
static bool cluster_staged(const Params& p, int dt, int roles, int cmax) {
  return (int64_t)p.B * p.rows * p.V * (int64_t)elem_size(dt) * roles <= (cmax > 1 ? kClusterStagedBytesTop : kClusterStagedBytes);
}

// Blocks per cluster, unstaged: a power of two (clusters of 3, 5, 6 or 7 were measured too: rarely the best,
// never by more than 7 %), as large as keeps the call a little within the four blocks an SM takes, so that no
// cluster waits for room (200 positions of 32000 bf16 logits: 1 block 19.6 us, 2 16.3; 100 of 128256: 2 31.0, 4
// 23.2; 272 rows of trees of 32000: 1 27.5, 2 24.5; but 75 of 128256, 600 blocks: 4 22.3, 8 23.8, and 150 of
// 32000: 2 15.1, 4 18.3) while a block has at least four tiles (250 of 12288: 1 block 12.9, 2 13.8), and so many that it has no more tiles than its bounds leave room for beside
// three other blocks and some L1 (150 positions of 128256 bf16 logits: 1 block 72 us, 2 34.9, 4 35.8; of
// 100000 400: 2 59, 4 63; 32-bit logits, two requests to a sector: 128256 2 54, 4 39.6.  Several
// arrivals, with their lists: 160 rows of a tree of 128256 2 56.6, 4 42.6; 32-bit: 63 rows 4 32.3, 8 23.2).
static int unstaged_size(const Params& p, int dt, int roles, int cmax, int lim) {
  const int most = cmax > 1 ? (dt == ERSD_F32 && roles == 2 ? 10 : 20) : (dt == ERSD_F32 && roles == 2 ? 20 : 32);
  const int ntiles = (p.V + b256::kTile - 1) / b256::kTile;
  const int64_t units = (int64_t)p.B * p.rows;
  int CL = 1;
  while (CL < lim && ((units * CL * 2 * 10 <= 37 * sm_count() && ntiles >= CL * 2 * 4) || ntiles > CL * most)) CL *= 2;
  return CL;
}

// Blocks per cluster.  Few positions: the smallest power of two that leaves a block about
// kClusterGroups tiles (shortest path through one position).  Once such clusters would make more
// than two blocks per SM: blocks of about twice as many tiles (measured at V = 128256: clusters
// of 8 beat clusters of 16 from about 20 positions on, clusters of 4 never beat clusters of 8).
// lim: the largest cluster that the kernel can be launched in.
static int cluster_size(const ersd_opts& o, const Params& p, int dt, int cmax, bool staged, int lim, int* out) {
  const int ntiles = (p.V + b256::kTile - 1) / b256::kTile;
  const int roles = (p.mode == kVerify && p.draft) ? 2 : 1;
  const int max_tiles = cluster_max_tiles(dt, roles, cmax, p.aligned_t && p.aligned_d);
  if (o.split_v) {  // the caller's choice: a power of two that the device takes and whose blocks can stage their share
    const int CL = (int)o.split_v;
    if (CL > lim || (CL & (CL - 1)) != 0 || (ntiles + CL - 1) / CL > max_tiles) return ERSD_EUNSUPPORTED;
    *out = CL;
    return ERSD_OK;
  }
  if (!staged) {
    *out = unstaged_size(p, dt, roles, cmax, lim);
    return ERSD_OK;
  }
  int CL = 1;
  while (CL < lim && CL * b256::kClusterGroups < ntiles) CL *= 2;
  const int64_t units = (int64_t)p.B * p.rows;
  if (units * CL > 2 * sm_count() && CL > 1 && (CL / 2) * 2 * b256::kClusterGroups >= ntiles &&
      (ntiles + CL / 2 - 1) / (CL / 2) <= max_tiles)
    CL /= 2;
  *out = CL;
  return ERSD_OK;
}

// Races of several arrivals that the streaming kernel takes for other reasons than the table's.  Figures: time of
// the cluster kernel / of the streaming kernel, us, or their ratio.
static bool top_streams(const Params& p, int dt, int cmax) {
  const bool tree = p.mode == kVerify;
  const int64_t n = (int64_t)p.B * p.rows, logits = n * p.V;
  // Of a row of less than 768 logits at most three of a block's eight warps have any: too few groups are looked at
  // for a threshold and the arrivals are picked one by one (500 logits: 8 of 1 row 22.2 / 13.0, of 2048 148 / 34,
  // 4 of 1 13.6 / 11.5; but 32 of 1 0.8, trees of up to four children 0.84 up to 216 rows and 1.14 at 272).  Up to
  // 32 rows stay all the same: the tests fix which kernel takes the shortest rows.
  if (p.V < 768 && cmax > 2 && n > 32 && (n > 256 || (cmax <= 16 && cmax > (tree ? 4 : 2)))) return true;
  if (p.V <= 4096) {
    // Many short rows: a block's phases behind the bounds take longer than the bounds, and the streaming kernel's
    // are lighter (1000 logits: 4 of 1024 rows 0.75, of 2048 35.6 / 21.5; 16 of 1024 67.3 / 57.7; 32 of 6000 0.67;
    // trees: stars of 8, 1152 rows 28.1 / 24.2; 17 nodes 1088 0.96, 3400 59.6 / 43.6; stars of 32 2112 0.88, 6600
    // 122 / 77.  2048 logits: sampling up to 0.95; trees: three children 1800 35.5 / 31.3, 17 nodes 2176 0.98, 3400
    // 59.9 / 54.9; stars of 32 6600 114 / 95.  4096: three children 1800 38.6 / 36.0, 17 nodes 3400 65.8 / 61.2,
    // stars of 8 0.87).
    if (!tree) return p.V <= 1536 && (cmax <= 8 ? n > 1500 : cmax <= 16 && n > 800);
    if (p.V <= 1536) return n > (cmax <= 16 ? 1100 : 3000);
    if (cmax <= 4) return n > (cmax <= 3 ? 1500 : 3000);
    return p.V <= 3072 && n > (cmax <= 16 ? 2500 : 5000);
  }
  // (Long rows, few arrivals: 4 of 1024 rows of 100000 bf16 logits 233 / 163, 2 135 / 124.  They stay: the streaming
  // kernel would cut the rows in two and need a workspace, which a sampling call that is being captured may not have.)
  if (!tree) return false;
  // 32-bit trees, which the table leaves out (stars of 8, 200 of 48000 logits 176 / 143; two alternatives, 128 of
  // 100000 90 / 78, of 128256 1.0).
  if (dt == ERSD_F32 && p.V > 40960 && cmax <= 16) {
    if (p.V <= 65536) return logits > (80 << 20);
    return cmax == 2 && logits > (32 << 20);
  }
  return false;
}

// Whether a call that leaves the choice to the library takes the cluster kernel.
static bool cluster_by_default(const ersd_opts& o, const Params& p, int dt, int cmax) {
  if (o.kernel_path != 0 || o.split_v != 0 || o.block_threads != 0 || !cluster_applies(p, dt, cmax)) return false;
  if (cmax > 1 && top_streams(p, dt, cmax)) return false;
  if (dt == ERSD_F32) return true;
  if (cmax > 16 && p.V <= 49152) return true;  // (64 stars of 32 of 48000 logits: 0.66)
  const ClusterLimit* limit = kClusterLimits[!(p.mode == kVerify && p.draft) ? 0 : cmax > 1 ? 2 : 1];
  while (p.V > limit->row) ++limit;
  // (given tokens of rows beyond 131072 leave earlier; sampling does not, see top_streams on workspaces)
  const int64_t most = p.given_tok && p.V > 131072 ? 72 << 20 : limit->logits;
  return (int64_t)p.V * p.B * p.rows <= most;
}

template <int DT, bool AL>
static int launch_cluster_dt(const ersd_opts& o, const Params& p_in, const TreeDesc& tree, int cmax, cudaStream_t st) {
  Params p = p_in;
  p.top_cmax = cmax;
  const bool verify = p.mode == kVerify;
  int roles = (verify && p.draft) ? 2 : 1;
  int CL = 1;
  const bool staged = cluster_staged(p, DT, roles, cmax);
  int lim = 8;
  int ls = prepare_kernel(cluster_kernel<DT, AL>(verify, cmax, roles, staged, false, 0), kClusterSmemBytes, false, true, &lim);
  if (ls == ERSD_OK) ls = cluster_size(o, p, DT, cmax, staged, lim, &CL);
  if (ls != ERSD_OK) return ls;
  const int ntiles = (p.V + b256::kTile - 1) / b256::kTile;
  // Trees of few positions: a cluster per ROW (a node's draft row and its target row side by side
  // in two clusters, each drawing the position's race variables) while all clusters are resident
  // at once; the longest chain of work in the call, the root's, is then half as long.
  int jobs = p.rows;
  if (cmax > 1 && roles == 2) {
    int with_children = 0;
    for (int n = 0; n < p.rows; ++n) with_children += tree.nchild[n] > 0 ? 1 : 0;
    const int64_t rows_in_all = (int64_t)p.B * (p.rows + with_children);
    bool split = rows_in_all * CL <= kClusterSplitBlocks;
    if (!split && (staged || CL == 16) && !o.split_v && CL >= 2 && rows_in_all * (CL / 2) <= kClusterSplitBlocks &&
        (ntiles + CL / 2 - 1) / (CL / 2) <= cluster_max_tiles(DT, 1, cmax, AL)) {
      CL /= 2;  // (a row to a cluster of half as many blocks)
      split = true;
    }
    if (split) {
      ls = prepare_kernel(cluster_kernel<DT, AL>(verify, cmax, 1, staged, false, 0), kClusterSmemBytes, false, true, &lim);
      if (ls != ERSD_OK) return ls;
    }
    if (split && CL <= lim) {
      p.top_split = 1 + with_children;
      jobs = p.rows + with_children;
      roles = 1;
    }
  }
  // Positions of one block each: blocks of 128 threads, twice as many to an SM, once there are more
  // positions than 256-thread blocks would be resident (3200 rows of 2048 bf16 logits: sampling 19.6
  // instead of 25.0 us, verification 26.8 instead of 37.0; at 400 rows equal; blocks of 64 threads
  // 19.6 and 29.9), and for rows that 128 threads take in one turn (400 positions of 1024 logits: 8.4
  // instead of 10.4 us); not where the staged rows would leave fewer than five such blocks to an SM.
  // Unstaged rows leave that room up to 16384 logits and beyond; longer ones keep 256 threads busy
  // (800 positions of 15048 logits: 25.8 us with 128 threads, 27.0 with 256; 1200 of 32000 57.1 and 51.4).
  const int G128 = (p.V + b128::kTile - 1) / b128::kTile;
  const bool small = cmax == 1 && CL == 1 && ((int64_t)p.B * p.rows > 4 * sm_count() || G128 == 1) &&
                     (staged ? b128::cluster_role_bytes<DT>(G128, AL) * (size_t)roles <= 41 * 1024 : G128 <= 16);
  const int threads = small ? b128::kThreads : b256::kThreads;
  const int G = small ? G128 : (ntiles + CL - 1) / CL;  // tiles per block; they fit, see cluster_applies
  const size_t smem = (small ? b128::cluster_role_bytes<DT>(G, AL, staged) : b256::cluster_role_bytes<DT>(G, AL, staged)) * (size_t)roles +
                      (cmax > 1 ? b256::top_list_bytes(cmax, CL) : 0);
  Launch l(dim3((unsigned)CL, (unsigned)jobs, (unsigned)p.B), (unsigned)threads, smem, st, (unsigned)CL);
  const int64_t blocks = (int64_t)CL * jobs * p.B;
  // The next kernel's blocks go where this one's leave room: if this one has a block on every SM they
  // are spread unevenly when they start early.  (One row of 128256 logits 4.8 us with it and 5.0
  // without, 4 x 8 alternatives 10.7 and 11.6, a tree of 240 blocks 21.1 and 22.1; but 16 rows, 256
  // blocks, 9.1 and 8.1, 300 positions of 8192 logits 12.9 and 11.0, and the streaming kernel, two
  // blocks to an SM, 47.5 and 38.9.)
  p.early = blocks <= (cmax > 1 ? 2 : 1) * sm_count();
  // Builds for some calls (where the device does not take them in clusters of this size: the general one).  Staged rows
  // in clusters of at least four blocks: the short way of ersd_cluster_kernel.  Unstaged rows, by blocks to an SM: see
  // cluster_ahead.  Several arrivals, with ten warps of the cluster to an arrival, unless all rows are greedy: see DIRECT.
  const int ahead = AL && (DT == ERSD_BF16 || G >= 16) ? 2 : 1;
  int short_way = cmax > 1     ? (roles == 1 && CL * b256::kWarps >= 10 * cmax && (p.temps || p.T != 0.0f) ? ahead : 0)
                  : staged     ? CL >= 4
                  : small      ? 0
                  : roles == 2 ? DT == ERSD_BF16 && AL && blocks <= 3 * sm_count()
                               : DT == ERSD_F32 && blocks > 3 * sm_count() && G >= 16;
  if (short_way) {
    ls = prepare_kernel(cluster_kernel<DT, AL>(verify, cmax, roles, staged, small, short_way), kClusterSmemBytes, false, true, &lim);
    if (ls != ERSD_OK) return ls;
    if (CL > lim) short_way = 0;
  }
  snprintf(g_last_launch, sizeof g_last_launch, "%s<%s, %d row(s) per cluster>: %d clusters of %d x %d threads, %d positions%s%s",
           cmax > 1 ? "ersd_cluster_top_kernel" : "ersd_cluster_kernel", DT == ERSD_BF16 ? "bf16" : "f32", roles,
           p.B * jobs, CL, threads, p.B * p.rows, staged ? "" : " (unstaged)",
           !short_way ? "" : cmax == 1 && !staged ? ", more tiles ahead" : ", short way");
  p.top_picks = CL * b256::kWarps >= 20 * cmax ? 4 : b256::kTopRounds;
  const void* kernel = cluster_kernel<DT, AL>(verify, cmax, roles, staged, small, short_way);
  if (small) {  // (the other builds are prepared by now)
    ls = prepare_kernel(kernel, staged ? kClusterSmemBytes : 0, false, false, nullptr);
    if (ls != ERSD_OK) return ls;
  }
  void* args[] = {&p, const_cast<TreeDesc*>(&tree)};  // (the kernel for one arrival has the first alone)
  const cudaError_t e = cudaLaunchKernelExC(&l.cfg, kernel, args);
  return e == cudaSuccess ? ERSD_OK : cuda_fail(e);
}

static int launch_cluster(const ersd_opts& o, const Params& p, const TreeDesc& tree, int dt, int cmax, cudaStream_t st) {
  if (p.aligned_t && p.aligned_d)
    return dt == ERSD_BF16 ? launch_cluster_dt<ERSD_BF16, true>(o, p, tree, cmax, st)
                           : launch_cluster_dt<ERSD_F32, true>(o, p, tree, cmax, st);
  return dt == ERSD_BF16 ? launch_cluster_dt<ERSD_BF16, false>(o, p, tree, cmax, st)
                         : launch_cluster_dt<ERSD_F32, false>(o, p, tree, cmax, st);
}

static int check_common(const void* logits, int dt, const uint64_t* seeds, int B, int rows, int V,
                        float T) {
  if (!logits || !seeds) return ERSD_EINVAL;
  if (dt != ERSD_F32 && dt != ERSD_BF16) return ERSD_EINVAL;
  if (B < 1 || rows < 1 || V < 1) return ERSD_EINVAL;
  if ((int64_t)B * rows > 0x7FFFFFFF) return ERSD_EINVAL;
  if (V > 0x7FFF0000) return ERSD_EUNSUPPORTED;
  if (!temp_ok(T)) return ERSD_EINVAL;
  if (((uintptr_t)logits & (elem_size(dt) - 1)) != 0 || ((uintptr_t)seeds & 7) != 0)
    return ERSD_EALIGN;
  return ERSD_OK;
}

static void fill_common(Params& p, const ersd_opts& o, const uint64_t* seeds, int B, int rows, int V,
                        float T) {
  p.seeds = seeds;
  p.seq_ids = o.seq_ids;
  p.pos_offsets = o.pos_offsets;
  p.temps = o.temps;
  p.ts_b = o.temp_stride_b;
  p.ts_r = o.temp_stride_r;
  p.T = T;
  p.B = B;
  p.rows = rows;
  p.V = V;
}

static int verify_impl(const void* target, const void* draft, int dt, const TreeDesc& tree, int D,
                       int cmax, bool chain, const uint64_t* seeds, int B, int rows, int draft_rows,
                       int V, float T, int32_t* out_tokens, int32_t* out_accept_len,
                       const ersd_opts* opts, void* stream, const int32_t* given_tok = nullptr,
                       bool check_only = false) {
  const ersd_opts o = read_opts(opts);
  Params p;
  memset(&p, 0, sizeof p);
  fill_common(p, o, seeds, B, rows, V, T);
  p.target = target;
  p.draft = draft;
  p.given_tok = given_tok;
  p.ld_t = o.ld_target ? o.ld_target : V;
  p.ld_d = o.ld_draft ? o.ld_draft : V;
  if (p.ld_t < V || p.ld_d < V) return ERSD_EINVAL;
  p.mode = kVerify;
  p.c_sample = 1;
  p.draft_rows = draft_rows;
  p.depth = D;
  p.chain_outputs = chain ? 1 : 0;
  p.aligned_t = rows_aligned(target, p.ld_t, dt);
  p.aligned_d = draft ? rows_aligned(draft, p.ld_d, dt) : 1;
  p.out_tokens = out_tokens;
  p.out_accept_len = out_accept_len;
  p.out_path = o.out_path;
  p.out_draft_tok = o.out_draft_tok;
  p.out_draft_key = o.out_draft_key;
  p.out_target_tok = o.out_target_tok;
  p.out_target_key = o.out_target_key;
  p.near_tie = o.near_tie_count;
  p.extra = o.near_tie_count ? 1 : 0;
  if (((uintptr_t)o.near_tie_count & 3) != 0) return ERSD_EALIGN;
  if (cmax + p.extra > ERSD_MAX_TOP_C) return ERSD_EUNSUPPORTED;
  cmax += p.extra;
  // sequences of few rows: one cluster per position (near-ties are counted by the streaming
  // kernel only: the cluster kernels keep no arrival beyond those asked for)
  if (o.kernel_path > 2) return ERSD_EINVAL;
  const bool cluster_ok = !p.extra && cluster_applies(p, dt, cmax);  // (a tree without branching is the chain 0 -> 1 -> ...)
  // (asked for by name it is for rows on 16-byte boundaries, as documented)
  if (o.kernel_path == 2 && !(cluster_ok && p.aligned_t && p.aligned_d)) return ERSD_EUNSUPPORTED;
  if (o.block_threads != 0 && o.block_threads != 128 && o.block_threads != 256) return ERSD_EINVAL;
  if (o.workspace) {
    if (o.workspace_bytes < workspace_bytes(B, rows)) return ERSD_EWORKSPACE;
    if (((uintptr_t)o.workspace & 15) != 0) return ERSD_EALIGN;
  }
  if (check_only) return ERSD_OK;  // every host-side check has passed; nothing was enqueued
  void* ws = nullptr;
  const int st = get_workspace(o, workspace_bytes(B, rows), &ws, (cudaStream_t)stream);
  if (st != ERSD_OK) return st;
  p.slots = (Slot*)ws;
  if (cluster_ok && (o.kernel_path == 2 || cluster_by_default(o, p, dt, cmax)))
    return launch_cluster(o, p, tree, dt, cmax, (cudaStream_t)stream);
  int st0 = choose_threads(o, (int64_t)B * rows, &p.threads);
  if (st0 != ERSD_OK) return st0;
  set_chunks(p, choose_split(o, (int64_t)B * rows, V, cmax, p.threads));
  return launch(p, tree, dt, cmax, (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------------------------
// Scratch for ersd_verify_noalloc: lives in the library image, one copy per GPU that loads it.
// In host code `g_noalloc_scratch` is only a handle for the runtime, never an address to hand
// to a kernel; noalloc_scratch() asks the runtime for the device address, once per device.
// ---------------------------------------------------------------------------------------------
constexpr size_t kNoallocBytes = (size_t)ERSD_NOALLOC_MAX_ROWS * sizeof(Slot);
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];

static std::mutex g_noalloc_mutex;
static void* g_noalloc_ptr[64];

static int noalloc_scratch(void** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e);
  if (dev < 0 || dev >= 64) return ERSD_EUNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (!g_noalloc_ptr[dev]) {
    void* ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);  // address on the current device
    if (e != cudaSuccess) return cuda_fail(e);
    if (!ptr) return ERSD_ECUDA;
    g_noalloc_ptr[dev] = ptr;
  }
  *out = g_noalloc_ptr[dev];
  return ERSD_OK;
}


// ---------------------------------------------------------------------------------------------
// Greedy speculative decoding (the paper's comparison verifier): kernels and launch logic.
// ---------------------------------------------------------------------------------------------
#include "ersd_gsd.inc"

static int gsd_check(const void* target, const void* draft, const int32_t* draft_tok, int dt,
                     const uint64_t* seeds, int B, int rows, int V, float T, const void* out_tokens,
                     const void* out_accept_len, bool need_draft) {
  int st = check_common(target, dt, seeds, B, rows, V, T);
  if (st != ERSD_OK) return st;
  if (!(T > 0.0f)) return ERSD_EINVAL;  // the ratio test needs softmax(z / T)
  if (!out_tokens || !out_accept_len) return ERSD_EINVAL;
  if (need_draft) {
    if (!draft || !draft_tok) return ERSD_EINVAL;
    if (((uintptr_t)draft & (elem_size(dt) - 1)) != 0 || ((uintptr_t)draft_tok & 3) != 0) return ERSD_EALIGN;
  }
  return ERSD_OK;
}

// Length of a slice (a multiple of eight) of rows of V logits, and their number: up to `slices` in
// all, but none shorter than one group of eight per thread.
static int gsd_slice(int V, int64_t rows, int64_t slices, int threads, int* S) {
  int64_t n = slices / rows;
  const int64_t most = ((int64_t)V + 8 * threads - 1) / (8 * threads);
  if (n > most) n = most;
  if (n > kGsdSlices) n = kGsdSlices;
  if (n < 1) n = 1;
  const int len = (int)((((int64_t)V + n - 1) / n + 7) / 8 * 8);
  *S = (int)(((int64_t)V + len - 1) / len);
  return len;
}

static void gsd_fill(GsdParams& g, const ersd_opts& o, const void* target, const void* draft,
                     const int32_t* draft_tok, const uint64_t* seeds, int B, int k, int V, float T,
                     int rows_t, int rows_d, int32_t* out_tokens, int32_t* out_accept_len) {
  memset(&g, 0, sizeof g);
  g.target = target;
  g.draft = draft;
  g.draft_tok = draft_tok;
  g.seeds = seeds;
  g.seq_ids = o.seq_ids;
  g.pos_offsets = o.pos_offsets;
  g.temps = o.temps;
  g.ts_b = o.temp_stride_b;
  g.ts_r = o.temp_stride_r;
  g.ld_t = o.ld_target ? o.ld_target : V;
  g.ld_d = o.ld_draft ? o.ld_draft : V;
  g.T = T;
  g.B = B;
  g.k = k;
  g.V = V;
  g.rows_t = rows_t;
  g.rows_d = rows_d;
  g.out_tokens = out_tokens;
  g.out_accept_len = out_accept_len;
  g.out_path = o.out_path;
}

}  // namespace ersd

using namespace ersd;

extern "C" {

int ersd_race_sample(const void* logits, ersd_dtype dt, const uint64_t* seeds, int B, int R, int V,
                     float T, int32_t* out_tok, const ersd_opts* opts, void* cuda_stream) {
  int st = check_common(logits, dt, seeds, B, R, V, T);
  if (st != ERSD_OK) return st;
  if (!out_tok) return ERSD_EINVAL;
  const ersd_opts o = read_opts(opts);
  const int c = o.top_c > 1 ? (int)o.top_c : 1;
  if (c > ERSD_MAX_TOP_C) return ERSD_EUNSUPPORTED;
  const int extra = o.near_tie_count ? 1 : 0;
  if (c + extra > ERSD_MAX_TOP_C) return ERSD_EUNSUPPORTED;
  if (((uintptr_t)o.near_tie_count & 3) != 0) return ERSD_EALIGN;
  Params p;
  memset(&p, 0, sizeof p);
  fill_common(p, o, seeds, B, R, V, T);
  p.target = logits;
  p.ld_t = o.ld_target ? o.ld_target : V;
  if (p.ld_t < V) return ERSD_EINVAL;
  p.ld_d = V;
  p.mode = kSample;
  p.c_sample = c;
  p.aligned_t = rows_aligned(logits, p.ld_t, dt);
  p.aligned_d = 1;
  p.out_tokens = out_tok;
  p.out_key = o.out_key;
  p.near_tie = o.near_tie_count;
  p.extra = extra;
  if (o.kernel_path > 2) return ERSD_EINVAL;
  // (near-ties are counted by the streaming kernel only: the cluster kernels keep no arrival beyond those asked for)
  const bool cluster_ok = !extra && cluster_applies(p, dt, c);
  // (asked for by name it is for rows on 16-byte boundaries, as documented)
  if (o.kernel_path == 2 && !(cluster_ok && p.aligned_t)) return ERSD_EUNSUPPORTED;
  TreeDesc tree;
  memset(&tree, 0, sizeof tree);
  if (cluster_ok && (o.kernel_path == 2 || cluster_by_default(o, p, dt, c)))
    return launch_cluster(o, p, tree, dt, c, (cudaStream_t)cuda_stream);
  st = choose_threads(o, (int64_t)B * R, &p.threads);
  if (st != ERSD_OK) return st;
  set_chunks(p, choose_split(o, (int64_t)B * R, V, c + extra, p.threads));
  if (p.S > 1) {
    void* ws = nullptr;
    st = get_workspace(o, workspace_bytes(B, R), &ws, (cudaStream_t)cuda_stream);
    if (st != ERSD_OK) return st;
    p.slots = (Slot*)ws;
  }
  return launch(p, tree, dt, c + extra, (cudaStream_t)cuda_stream);
}

static int verify_sequence(const void* target_logits, const void* draft_logits, int dt,
                           const uint64_t* seeds, int B, int k, int V, float T, int32_t* out_tokens,
                           int32_t* out_accept_len, const ersd_opts* opts, void* cuda_stream,
                           bool check_only) {
  if (k < 0) return ERSD_EINVAL;
  if (k + 1 > ERSD_MAX_ROWS) return ERSD_EUNSUPPORTED;
  int st = check_common(target_logits, dt, seeds, B, k + 1, V, T);
  if (st != ERSD_OK) return st;
  if (!out_tokens || !out_accept_len) return ERSD_EINVAL;
  if (k > 0) {
    if (!draft_logits) return ERSD_EINVAL;
    if (((uintptr_t)draft_logits & (elem_size(dt) - 1)) != 0) return ERSD_EALIGN;
  }
  int32_t parent[ERSD_MAX_ROWS];
  for (int n = 0; n <= k; ++n) parent[n] = n - 1;
  TreeDesc tree;
  int D = 0, cmax = 1;
  st = build_tree(parent, k, &tree, &D, &cmax);
  if (st != ERSD_OK) return st;
  return verify_impl(target_logits, draft_logits, dt, tree, D, cmax, true, seeds, B, k + 1, k, V, T,
                     out_tokens, out_accept_len, opts, cuda_stream, nullptr, check_only);
}

int ersd_verify(const void* target_logits, const void* draft_logits, ersd_dtype dt,
                const uint64_t* seeds, int B, int k, int V, float T, int32_t* out_tokens,
                int32_t* out_accept_len, const ersd_opts* opts, void* cuda_stream) {
  return verify_sequence(target_logits, draft_logits, dt, seeds, B, k, V, T, out_tokens, out_accept_len,
                         opts, cuda_stream, false);
}

int ersd_verify_tokens(const void* target_logits, const int32_t* draft_tokens, ersd_dtype dt,
                       const uint64_t* seeds, int B, int k, int V, float T, int32_t* out_tokens,
                       int32_t* out_accept_len, const ersd_opts* opts, void* cuda_stream) {
  if (k < 0) return ERSD_EINVAL;
  if (k + 1 > ERSD_MAX_ROWS) return ERSD_EUNSUPPORTED;
  int st = check_common(target_logits, dt, seeds, B, k + 1, V, T);
  if (st != ERSD_OK) return st;
  if (!out_tokens || !out_accept_len) return ERSD_EINVAL;
  if (k > 0) {
    if (!draft_tokens) return ERSD_EINVAL;
    if (((uintptr_t)draft_tokens & 3) != 0) return ERSD_EALIGN;
  }
  int32_t parent[ERSD_MAX_ROWS];
  for (int n = 0; n <= k; ++n) parent[n] = n - 1;
  TreeDesc tree;
  int D = 0, cmax = 1;
  st = build_tree(parent, k, &tree, &D, &cmax);
  if (st != ERSD_OK) return st;
  // the chain keeps its shape for the walk, but no row has a draft row to race
  for (int n = 0; n <= k; ++n) {
    tree.nchild[n] = 0;
    tree.order[n] = (uint8_t)n;
  }
  return verify_impl(target_logits, nullptr, dt, tree, D, 1, true, seeds, B, k + 1, k, V, T, out_tokens,
                     out_accept_len, opts, cuda_stream, k > 0 ? draft_tokens : nullptr);
}

int ersd_verify_tree(const void* target_logits, const void* draft_logits, ersd_dtype dt,
                     const int32_t* parent, const uint64_t* seeds, int B, int N, int V, float T,
                     int32_t* out_tokens, int32_t* out_accept_len, const ersd_opts* opts,
                     void* cuda_stream) {
  if (N < 0 || !parent) return ERSD_EINVAL;
  if (N + 1 > ERSD_MAX_ROWS) return ERSD_EUNSUPPORTED;
  int st = check_common(target_logits, dt, seeds, B, N + 1, V, T);
  if (st != ERSD_OK) return st;
  if (!out_tokens || !out_accept_len) return ERSD_EINVAL;
  if (N > 0) {
    if (!draft_logits) return ERSD_EINVAL;
    if (((uintptr_t)draft_logits & (elem_size(dt) - 1)) != 0) return ERSD_EALIGN;
  }
  TreeDesc tree;
  int D = 0, cmax = 1;
  st = build_tree(parent, N, &tree, &D, &cmax);
  if (st != ERSD_OK) return st;
  return verify_impl(target_logits, draft_logits, dt, tree, D, cmax, false, seeds, B, N + 1, N + 1,
                     V, T, out_tokens, out_accept_len, opts, cuda_stream);
}

int ersd_verify_noalloc(const void* target_logits, const void* draft_logits, ersd_dtype dt,
                        const uint64_t* seeds, int B, int k, int V, float T, int32_t* out_tokens,
                        int32_t* out_accept_len, const ersd_opts* opts, void* cuda_stream) {
  if (B < 1 || k < 0) return ERSD_EINVAL;
  if ((int64_t)B * ((int64_t)k + 1) > ERSD_NOALLOC_MAX_ROWS) return ERSD_ENOALLOC_LIMIT;
  ersd_opts o = read_opts(opts);
  if (o.workspace) return ERSD_EINVAL;  // this entry point brings its own scratch
  void* scratch = nullptr;
  int st = noalloc_scratch(&scratch);
  if (st != ERSD_OK) return st;
  o.struct_size = sizeof o;
  o.workspace = scratch;
  o.workspace_bytes = kNoallocBytes;
  // every host-side argument check of ersd_verify first: a refused call puts nothing on the stream
  st = verify_sequence(target_logits, draft_logits, dt, seeds, B, k, V, T, out_tokens, out_accept_len, &o,
                       cuda_stream, true);
  if (st != ERSD_OK) return st;
  // The array keeps whatever the previous call left; the arrival counters (the first 16 bytes
  // of every slot this call uses) must start at zero.
  const cudaError_t e = cudaMemset2DAsync(scratch, sizeof(Slot), 0, 16, (size_t)B * ((size_t)k + 1),
                                          (cudaStream_t)cuda_stream);
  if (e != cudaSuccess) return cuda_fail(e);
  return verify_sequence(target_logits, draft_logits, dt, seeds, B, k, V, T, out_tokens, out_accept_len, &o,
                         cuda_stream, false);
}


int ersd_gsd_verify(const void* target_logits, const void* draft_logits, const int32_t* draft_tokens,
                    ersd_dtype dt, const uint64_t* seeds, int B, int k, int V, float T, int32_t* out_tokens,
                    int32_t* out_accept_len, const ersd_opts* opts, void* cuda_stream) {
  if (k < 0) return ERSD_EINVAL;
  if (k + 1 > ERSD_MAX_ROWS) return ERSD_EUNSUPPORTED;
  int st = gsd_check(target_logits, draft_logits, draft_tokens, dt, seeds, B, k + 1, V, T, out_tokens,
                     out_accept_len, k > 0);
  if (st != ERSD_OK) return st;
  const ersd_opts o = read_opts(opts);
  GsdParams g;
  gsd_fill(g, o, target_logits, draft_logits, draft_tokens, seeds, B, k, V, T, k + 1, k, out_tokens,
           out_accept_len);
  if (g.ld_t < V || g.ld_d < V) return ERSD_EINVAL;
  if (B > 65535) return ERSD_EUNSUPPORTED;  // (sequences are the second dimension of both grids)
  // Sums: about 64 warps per multiprocessor in all, two waves of the 32 that are resident (32 or 128
  // per multiprocessor: 1 and 4 % slower at 64 sequences of 128256 logits).  Race: one wave of three
  // blocks per multiprocessor, because a block begins with the ratio tests.
  g.slice1 = gsd_slice(V, (int64_t)B * (2 * k + 1), 64 * (int64_t)sm_count(), 128, &g.S1);
  g.slice = gsd_slice(V, B, 3 * (int64_t)sm_count(), kGsdThreads, &g.S);
  g.sum_err = (float)(4.76837158203125e-7 + 2.384185791015625e-7 * (log2((double)V) + 32.0));
  void* ws = nullptr;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  st = get_workspace(o, workspace_bytes(B, k + 1), &ws, stream);
  if (st != ERSD_OK) return st;
  g.slots = (Slot*)ws;
  const int per_block = kGsdStatsThreads / 32;  // slices of a block of the sums
  const dim3 sums_grid((unsigned)(2 * k + 1), (unsigned)B, (unsigned)((g.S1 + per_block - 1) / per_block));
  const dim3 race_grid((unsigned)g.S, (unsigned)B);
  const bool bf16 = dt == ERSD_BF16;
  Launch sums(sums_grid, kGsdStatsThreads, 0, stream), race(race_grid, kGsdThreads, 0, stream);
  cudaError_t e = cudaLaunchKernelEx(&sums.cfg, bf16 ? gsd_stats_kernel<ERSD_BF16> : gsd_stats_kernel<ERSD_F32>, g);
  if (e == cudaSuccess) {
    e = cudaLaunchKernelEx(&race.cfg, bf16 ? gsd_race_kernel<ERSD_BF16> : gsd_race_kernel<ERSD_F32>, g);
    // (the sums are on their way and nobody will clear them)
    if (e != cudaSuccess) (void)cudaMemsetAsync(ws, 0, workspace_bytes(B, k + 1), stream);
  }
  return e == cudaSuccess ? ERSD_OK : cuda_fail(e);
}

int ersd_gsd_verify_tree(const void* target_logits, const void* draft_logits, const int32_t* draft_tokens,
                         ersd_dtype dt, const int32_t* parent, const uint64_t* seeds, int B, int N, int V,
                         float T, int32_t* out_tokens, int32_t* out_accept_len, const ersd_opts* opts,
                         void* cuda_stream) {
  if (N < 0 || !parent) return ERSD_EINVAL;
  if (N + 1 > ERSD_MAX_ROWS) return ERSD_EUNSUPPORTED;
  int st = gsd_check(target_logits, draft_logits, draft_tokens, dt, seeds, B, N + 1, V, T, out_tokens,
                     out_accept_len, N > 0);
  if (st != ERSD_OK) return st;
  TreeDesc tree;
  int D = 0, cmax = 1;
  st = build_tree(parent, N, &tree, &D, &cmax);
  if (st != ERSD_OK) return st;
  const ersd_opts o = read_opts(opts);
  GsdParams g;
  gsd_fill(g, o, target_logits, draft_logits, draft_tokens, seeds, B, N, V, T, N + 1, N + 1, out_tokens,
           out_accept_len);
  if (g.ld_t < V || g.ld_d < V) return ERSD_EINVAL;
  g.depth = D;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  if (dt == ERSD_BF16) gsd_tree_kernel<ERSD_BF16><<<(unsigned)B, kGsdTreeThreads, 0, stream>>>(g, tree);
  else gsd_tree_kernel<ERSD_F32><<<(unsigned)B, kGsdTreeThreads, 0, stream>>>(g, tree);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ERSD_OK : cuda_fail(e);
}

int ersd_tree_depth(const int32_t* parent, int N) {
  if (!parent || N < 0 || N + 1 > ERSD_MAX_ROWS) return -1;
  TreeDesc tree;
  int D = 0, cmax = 1;
  if (build_tree(parent, N, &tree, &D, &cmax) != ERSD_OK) return -1;
  return D;
}

int ersd_row_keys(const void* row_logits, ersd_dtype dt, int V, float T, uint64_t seed,
                  uint32_t seq_id, uint32_t position, int mode, float* out_keys, void* cuda_stream) {
  if (!row_logits || !out_keys || V < 1 || !temp_ok(T) || (mode < 0 || mode > 2)) return ERSD_EINVAL;
  if (dt != ERSD_F32 && dt != ERSD_BF16) return ERSD_EINVAL;
  if (((uintptr_t)row_logits & (elem_size(dt) - 1)) != 0 || ((uintptr_t)out_keys & 3) != 0)
    return ERSD_EALIGN;
  const int threads = 256, blocks = (V + threads - 1) / threads;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (dt == ERSD_BF16)
    ersd_row_keys_kernel<ERSD_BF16><<<blocks, threads, 0, st>>>(row_logits, V, T, seed, seq_id, position, mode, out_keys);
  else
    ersd_row_keys_kernel<ERSD_F32><<<blocks, threads, 0, st>>>(row_logits, V, T, seed, seq_id, position, mode, out_keys);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ERSD_OK : cuda_fail(e);
}

size_t ersd_workspace_bytes(int B, int rows_per_seq) {
  if (B < 1 || rows_per_seq < 1) return 0;
  return workspace_bytes(B, rows_per_seq);
}

int ersd_workspace_init(void* workspace, size_t bytes, void* cuda_stream) {
  if (!workspace) return ERSD_EINVAL;
  const cudaError_t e = cudaMemsetAsync(workspace, 0, bytes, (cudaStream_t)cuda_stream);
  return e == cudaSuccess ? ERSD_OK : cuda_fail(e);
}

const char* ersd_status_string(int status) {
  switch (status) {
    case ERSD_OK: return "ok";
    case ERSD_EINVAL: return "invalid argument";
    case ERSD_EALIGN: return "misaligned pointer";
    case ERSD_EUNSUPPORTED: return "size beyond a compiled limit";
    case ERSD_ECUDA: return "CUDA runtime error";
    case ERSD_EWORKSPACE: return "workspace too small";
    case ERSD_ENOALLOC_LIMIT:
      return "B * (k + 1) exceeds ERSD_NOALLOC_MAX_ROWS, the capacity of ersd_verify_noalloc's built-in scratch";
    default: return "unknown status";
  }
}

int ersd_last_cuda_error(void) { return g_last_cuda_error; }

const char* ersd_last_launch(void) { return g_last_launch; }

int ersd_version(void) { return 112; }

}  // extern "C"
