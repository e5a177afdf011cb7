// Internal declarations shared by the libbh translation units.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>

#include <atomic>
#include <cstdarg>
#include <cstdint>
#include <memory>
#include <mutex>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/bh.h"

namespace bh {

// NVTX range over a C-ABI call (precompute, cube map, render, batch, serve):
// visible in a profiler's timeline, free when no tool is attached.
struct TraceRange {
  explicit TraceRange(const char *name) { nvtxRangePushA(name); }
  ~TraceRange() { nvtxRangePop(); }
  TraceRange(const TraceRange &) = delete;
  TraceRange &operator=(const TraceRange &) = delete;
};

constexpr double kMu = 4.0 / 27.0;  // max of u^2 (1-u), photon sphere u = 2/3 (Sec. 3.3.1)
constexpr double kPi = 3.14159265358979323846;

// Sizes of the colour tables (Sec. 3.4.2 and the disc black-body table).
constexpr int kCnx = 64, kCny = 32, kCnd = 64;
constexpr int kDiscN = 1024;
constexpr int kNLambda = 95;  // 360..830 nm, 5 nm trapezoid
constexpr int kNLocus = 4096;
constexpr int kMaxUTexels = 4096;
constexpr int kMaxParticles = 256;  // animated disc: shared memory holds 32 bytes per particle

// Status word bits written by kernels (never a trap or an assert).
constexpr unsigned kStatusMbarTimeout = 1u;
constexpr unsigned kStatusBadIndex = 2u;
constexpr unsigned kStatusBarrierTimeout = 4u;  // a bounded grid-barrier wait gave up

void set_error(const char *fmt, ...);
bh_status cuda_fail(cudaError_t e, const char *what);
#define BH_CUDA(call)                                   \
  do {                                                  \
    cudaError_t e__ = (call);                           \
    if (e__ != cudaSuccess) return cuda_fail(e__, #call); \
  } while (0)

struct ServeState;

// A batched launch as a CUDA graph: the copy of the per-camera constants
// from pinned staging memory and the persistent render kernel.  Rebuilt when
// the number of cameras or the kernel changes; otherwise only the kernel's
// parameters are updated before each replay.
struct BatchGraph {
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaGraphNode_t copy = nullptr, kern = nullptr;
  int n = 0, block = 0;
  const void *func = nullptr;
  void *cam_dev = nullptr;
  void reset() {
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    exec = nullptr;
    graph = nullptr;
    copy = kern = nullptr;
    n = block = 0;
    func = nullptr;
    cam_dev = nullptr;
  }
};

struct RenderTuning {
  int warps_per_block = 8;   // block = warps * 32 threads
  int fetch = 0;             // 8 x 4 pixel warp tiles a warp takes per fetch (before the launch's
                             // tail); 0: by the launch's size
  int blocks_per_sm = 4;     // persistent grid = SMs * blocks_per_sm
};

// A served frame request on a device-resident orbit (Appendix C): advance
// *orbit by dtau of proper time in `steps` steps, then render it at
// width x height into out.
struct OrbitJob {
  bh_orbit *orbit;
  float *out;
  double dtau;
  int steps, width, height, pad;
};

// Tile-scheduler counters: every render launch takes the next pair of a ring
// (re-armed to zero by the launch's last warp), so launches in flight at once
// on different streams need distinct pairs: at most kSchedRing of them.
constexpr int kSchedRing = 1024;

// Device memory of the context's tables, cube maps and builds, kept when it is
// given back: a cudaMalloc of a 1M-star map's 277 MB and its cudaFree take 0.5
// ms, as long as building it.  At most kPoolBytes are kept, the newest; the rest
// goes back to the device at once.  bh_destroy and an allocation that fails give
// all of it back.
struct PoolBlock {
  void *p = nullptr;
  size_t bytes = 0;             // 0: stream-ordered scratch, never kept
  cudaEvent_t ready = nullptr;  // recorded behind its last use; nullptr: idle
};
constexpr size_t kPoolBytes = (size_t)512 << 20;
struct HeldBlock {
  PoolBlock b;
  unsigned long long seq;  // its number among all that were ever held
};
struct Pool {  // shared with the handles: one freed after bh_destroy finds it closed
  int device = 0;
  std::mutex mu;  // guards what follows
  std::vector<PoolBlock> kept;  // oldest first
  std::vector<HeldBlock> held;  // freed, but not known to be idle
  unsigned long long holds = 0;
  size_t bytes = 0;             // of kept and held
  size_t lent = 0;              // of scratch in use that will be kept: bytes + lent <= kPoolBytes
  size_t missed = 0;            // the largest scratch that there was no room for
  bool open = true;
};

}  // namespace bh

struct bh_ctx {
  int device = 0;
  int sm_count = 0;
  size_t budget = 0;
  cudaStream_t aux = nullptr;
  unsigned *status_dev = nullptr;     // kernel status word
  unsigned *sched_dev = nullptr;      // kSchedRing pairs of tile-scheduler counters
  std::atomic<unsigned> sched_next{0};
  std::atomic<long long> launches{0};
  // render staging: per-camera constants for batched launches
  void *cam_host = nullptr;           // pinned
  void *cam_dev = nullptr;
  int cam_cap = 0;
  bh::BatchGraph graph;               // bh_render_batch launches
  void *orb_cams_dev = nullptr;       // bh_render_orbits: per-orbit camera constants, then the tile count
  cudaEvent_t orb_done = nullptr;     // behind the last launch that reads them
  float *frame_dev = nullptr;         // bh_render_to_host frame buffer
  size_t frame_cap = 0;
  // bh_render_to_host_async: two device frames; each is copied to the host
  // on ring_copy while the next one renders
  float *ring_dev[2] = {nullptr, nullptr};
  size_t ring_cap = 0;
  cudaStream_t ring_copy = nullptr;
  cudaEvent_t ring_ready[2] = {nullptr, nullptr};  // the slot's last frame is rendered
  cudaEvent_t ring_done[2] = {nullptr, nullptr};   // ... and its copy to the host has finished
  unsigned long long ring_seq = 0;                 // frames issued (the next ticket)
  void *bloom_dev = nullptr;          // bh_bloom: mip pyramid scratch
  size_t bloom_cap = 0;
  unsigned *bloom_bar = nullptr;      // bh_bloom: grid-barrier counter
  bh::RenderTuning tuning;
  bh::ServeState *serve = nullptr;
  std::shared_ptr<bh::Pool> pool = std::make_shared<bh::Pool>();
  int inject_table_wait = 0;          // bh_inject_fault: next render's table wait never completes
  int inject_bloom_barrier = 0;       // bh_inject_fault: next bloom's first grid barrier is never complete
  std::mutex mu;
};

struct bh_tables {
  bh_ctx *ctx = nullptr;
  std::shared_ptr<bh::Pool> pool;
  bh::PoolBlock mem;  // all arrays below
  bh_table_desc desc{};
  double *D64 = nullptr, *U64 = nullptr;  // FP64 values
  void *D = nullptr, *U = nullptr;        // storage copies read by the renderer
  double *DT64 = nullptr, *UT64 = nullptr;  // regularised-time channels of D and U (FP64)
  float *DT = nullptr, *UT = nullptr;       // their FP32 copies (read by the debug render)
  float4 *C = nullptr;                    // colour shift table [k][j][i] (XYZ, pad)
  float4 *disc = nullptr;                 // ln Y, X/Y, Z/Y of black bodies, log2 T in [8, 20]
};

struct bh_particles {
  bh_ctx *ctx = nullptr;
  int n = 0;
  double *dev = nullptr;  // 8 doubles per particle, sorted by rmin: u1, u2, phi0, omega, c, rmin, rmax, 0
};

struct bh_cubemap {
  bh_ctx *ctx = nullptr;
  std::shared_ptr<bh::Pool> pool;
  bh::PoolBlock mem;  // records and mask
  int n = 0;        // face size
  int levels = 0;
  bh_dtype storage = BH_F16;
  uint2 *rec = nullptr;  // all levels
  long long records = 0;
  uint2 *mask = nullptr;     // occupancy bits by blocks of texels (mask_level_offset)
};

namespace bh {
inline long long cube_level_offset(int N, int L) {
  long long off = 0;
  for (int l = 0; l < L; ++l) off += 6LL * (N >> l) * (N >> l);
  return off;
}
// Occupancy mask layout: level-major, face, then blocks of 16 columns x 4
// rows in row-major order, one every 8 columns and 4 rows (each texel is in
// two blocks; at least one block; texels past the face are 0).  Row r of a
// block is 16 bits, the first column in the top bit: rows 0 and 1 in x (row 0
// on top), rows 2 and 3 in y.  Any 8 columns x 8 rows of a face lie in one
// block column and at most three of its blocks, so a footprint's occupancy is
// one to three loads instead of one or two per texel row.
inline long long mask_level_offset(int N, int L) {
  long long off = 0;
  for (int l = 0; l < L; ++l) {
    const long long n = N >> l;
    off += 6 * (n >= 8 ? n / 8 : 1) * (n >= 4 ? n / 4 : 1);
  }
  return off;
}
inline int cube_levels(int N) {
  int L = 0;
  while ((1 << L) < N) ++L;
  return L + 1;
}
// A block of at least `bytes`, usable by work on stream s from now on.  Scratch is
// given back behind the work on stream s (pool_put, which waits for nothing), a
// handle's memory behind all work of the device (pool_put_synced, which
// synchronises it).  From any thread.
cudaError_t pool_get(Pool &pool, size_t bytes, cudaStream_t s, PoolBlock *out, bool scratch = false);
void pool_put(Pool &pool, PoolBlock b, cudaStream_t s);
void pool_put_synced(Pool &pool, PoolBlock b);
// cudaMalloc for a context's other buffers, which takes the kept memory where
// the device has no more.
cudaError_t pool_malloc(Pool &pool, void **p, size_t bytes);
void count_launch(bh_ctx *ctx, int n = 1);
bh_status check_status(bh_ctx *ctx, cudaStream_t s);
bh_status colour_tables_launch(bh_ctx *ctx, bh_tables *t, cudaStream_t s);
void occupancy_launch(bh_ctx *ctx, const bh_cubemap *c, int first, cudaStream_t s);
bh_status cubemap_alloc_public(bh_ctx *ctx, int N, bh_dtype storage, cudaStream_t s, bh_cubemap **out);
}  // namespace bh
