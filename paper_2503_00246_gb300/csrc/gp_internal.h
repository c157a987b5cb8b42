// Internal declarations shared by the C-ABI translation units.
#pragma once

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "gp.h"
#include "gp_launch.h"
#include "gp_plan.h"

struct gp_ctx {
  gp::Plan plan;
  int device = -1;
  bool on_device = false;
  size_t elem = 8;
  int32_t* d_frows = nullptr;
  int32_t* d_lwin = nullptr;
  int32_t* d_lrow = nullptr;
  int32_t* d_lmask = nullptr;
  void* d_fac = nullptr;         // line factors (Plan::fac): FP32 mw, FP64 those of the triangular basis
  gp::LaunchForm form{};         // gp::launch_form
  int2* d_zruns = nullptr;
  void* d_tp = nullptr;          // per-face outputs W_F (scratch of the face + lift path)
  // brick path (gp_brick.cuh): tables and the partial grids of the plane nodes (scratch)
  bool use_brick = false;
  int32_t* d_bdesc = nullptr;
  int32_t* d_bcell = nullptr;
  int32_t* d_bccoord = nullptr;
  uint32_t* d_bface = nullptr;
  int32_t* d_rowtab = nullptr;
  int32_t* d_pnode = nullptr;
  int32_t* d_poff = nullptr;
  int32_t* d_pslot = nullptr;
  void* d_part = nullptr;
  bool no_scratch = false;
  void* d_xh = nullptr;          // gp_apply_host staging
  void* d_yh = nullptr;
  int2* d_truns = nullptr;       // gp_apply_host: runs (c0, len) of the touched DoFs
  int32_t ntruns = -1;           // -1: not built yet
  int host_slabs = 0;              // slabs of the last gp_apply_host
  int64_t host_bytes[2] = {0, 0};  // bytes the last gp_apply_host moved host -> device, device -> host
  // gp_apply_host with a page-locked y: a slab pipeline whose finished parts of y go back on a
  // second stream while later slabs compute (built on first use)
  bool hpipe_built = false;
  std::vector<int32_t> hslabs;   // slab table (gp::slab_table)
  std::vector<int64_t> hbounds;  // y chunk of slab s: [hbounds[s], hbounds[s + 1])
  std::vector<cudaEvent_t> hev;  // one per slab, recorded after its lift
  cudaStream_t hcopy = nullptr;  // the D2H stream
  std::vector<int2> htruns;      // host copy of d_truns
  std::vector<int32_t> hxrun;    // touched runs gathered for slab s: [hxrun[s], hxrun[s + 1])
  std::vector<cudaEvent_t> hgev; // one per slab, recorded after its gather
  cudaStream_t hin = nullptr;    // the gather stream
  gp::Tiles tiles{};             // tile shape of the face and lift launches (0: defaults)
  bool tuned = false;            // tiles was measured for the apply (the model system's face kernel keeps its default)
  std::string err;
  // tracing: one event triple per traced apply
  bool prof = false;
  std::vector<cudaEvent_t> ev;
  int64_t nprof = 0;
};

namespace gpi {

// Makes `dev` current for the lifetime of the guard and restores the caller's device.
struct DeviceGuard {
  int prev = -1;
  bool ok = true;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (dev >= 0 && dev != prev) ok = cudaSetDevice(dev) == cudaSuccess;
  }
  ~DeviceGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

// Records `m` as the last error of `c` (or of the calling thread when c is NULL).
gp_status fail(const gp_ctx* c, gp_status s, const std::string& m);

// Enqueues y = G x (add = 0) or y += G x (add = 1) for context c; `scratch` replaces the
// context's face-output buffer when given; `trace` = false never records events.
// `tiles` overrides the context's tile shape; `which` (bit 0 face, bit 1 lift) drops a
// kernel (the autotuner times them apart); `full_outputs` makes a face launch store W_F in every
// arithmetic (the model system's gather reads it).
// A slab pipeline for one launch: a slab table (SLAB ints per slab) and an event per slab.
struct SlabRun {
  const int32_t* table = nullptr;
  int n = 0;
  cudaEvent_t* events = nullptr;   // recorded after each slab's lift
  cudaEvent_t* inputs = nullptr;   // waited for before each slab's face launch (or nullptr)
};
gp_status launch(gp_ctx* c, const void* x, void* y, int add, cudaStream_t st, void* scratch = nullptr,
                 bool trace = true, const gp::Tiles* tiles = nullptr, int which = 3, const SlabRun* run = nullptr,
                 bool full_outputs = false);

// Slab pipeline of the face + lift path (gp_opts.slabs): at most MAX_SLABS slabs.
static_assert(gp::SLAB == gp::SLAB_INTS, "the plan's and the launcher's slab records differ");
constexpr int MAX_SLABS = 64;
// gp_apply_host: the device address of a page-locked host buffer (nullptr for other memory),
// the runs of touched DoFs (built on first use), and the copy of those runs of x.
const void* device_view(const void* host);
cudaError_t ensure_touched_runs(gp_ctx* c);
// The host-apply slab pipeline of c (host_slabs slabs; none when the plan has too few owners).  The
// first copy of y starts after one slab's launches, and each slab adds about 40 us of launches that are
// too small for the GPU, so that the best count grows like the square root of y's bytes: measured best
// (us at 1 / 2 / 4 / 8 / 16 slabs) for y of 4 MB 1 (72 / 77 / 99), 21 MB 2 to 3 (374 / 329 / 341 /
// 488 / 729), 88 MB 4 to 8 (842 / 703 / 650 / 664 / 767), 235 MB 8 to 12 (1733 / 1656 / 1546 / 1471 /
// 1494), 470 MB 12 (4203 / 3561 / 3137 / 2966 / 3174).
inline int host_slabs(double y_bytes) {
  return std::min(16, std::max(1, (int)(std::sqrt(y_bytes / (4 << 20)) + 0.5)));
}
cudaError_t ensure_host_pipeline(gp_ctx* c);
cudaError_t gather_runs(const void* src, void* dst, const int2* runs, int nruns, int elem, cudaStream_t st);
// Default faces per chunk of the brick kernel (about 256 threads).
int brick_default_fb(int dim, int k);
// Bytes of the brick path's partial grids (its scratch) for context c.
size_t brick_scratch_bytes(const gp_ctx* c);
// Allocates the face-output buffer W of the face + lift path if the context has none (the
// model system and the autotuner's face + lift timings need it).
gp_status ensure_face_outputs(gp_ctx* c);

// Tile-shape helpers for the context's (dimension, arithmetic).
gp::TileOps tile_ops(int dim, int precision);

// Starts a new context from the process-wide table of tuned tile shapes, if that has a shape for its kind.
void tiles_start(gp_ctx* c);

}  // namespace gpi
