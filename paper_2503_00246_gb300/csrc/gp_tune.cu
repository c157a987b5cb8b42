// Tile shapes of the face and lift launches and their autotuner.
//
// The tile shape is (faces per face CTA, owner cells per lift CTA, lift threads); on the
// brick path only the first field counts (faces per chunk of the brick kernel), and the
// autotuner times whole applies for it.
// gp_autotune times each candidate, the default among them, on the context's own tables with CUDA events,
// with the L2 flushed before every timed launch (the operator's operands are
// read from HBM in a real solve), and takes the fastest face and lift shapes if the whole apply is
// then faster than with the default, both after a flush and back to back.
// The choice is recorded in a process-wide table keyed by (device, dimension,
// degree, arithmetic) and by what the default depends on (the form of the face outputs and the size class of
// the mesh); gp_setup starts new contexts of that kind from the table, and a
// batch takes the shape of each group's first context.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "gp_internal.h"

namespace {

typedef std::tuple<int, int, int, int> Key;   // device, dimension, degree, arithmetic
struct Entry {
  bool any = false;                           // a shape for every kind (gp_tiles_record)
  gp::Tiles all{};
  std::map<int, gp::Tiles> kind;              // tuned shapes by kind_of
  gp::Tiles last{};
};
// Counted up when the kernels or their default shapes change: shapes tuned for others are not taken from a file.
constexpr int kTileVersion = 1;

std::mutex g_tiles_mu;
std::map<Key, Entry> g_tiles;                 // face + lift path
std::map<Key, gp::Tiles> g_brick_tiles;       // brick path (fb only)

// form of the face outputs and size class of a context
int kind_of(const gp_ctx* c) {
  return 16 * (c->form.compact ? 1 : 0) + gpi::tile_ops(c->plan.dim, c->plan.precision).size_class(c->plan.k, c->form);
}
Key key_of(const gp_ctx* c) { return std::make_tuple(c->device, c->plan.dim, c->plan.k, c->plan.precision); }

}  // namespace

namespace gpi {

gp::TileOps tile_ops(int dim, int precision) {
  if (precision == GP_FP64) return dim == 2 ? gp::tile_ops_f64_d2() : gp::tile_ops_f64_d3();
  if (precision == GP_FP64_FF) return dim == 2 ? gp::tile_ops_ff_d2() : gp::tile_ops_ff_d3();
  return dim == 2 ? gp::tile_ops_f32_d2() : gp::tile_ops_f32_d3();
}

void tiles_start(gp_ctx* c) {
  std::lock_guard<std::mutex> lk(g_tiles_mu);
  if (c->use_brick) {
    auto it = g_brick_tiles.find(key_of(c));
    if (it != g_brick_tiles.end()) c->tiles = it->second;
    return;
  }
  auto it = g_tiles.find(key_of(c));
  if (it == g_tiles.end()) return;
  auto own = it->second.kind.find(kind_of(c));
  c->tuned = own != it->second.kind.end();
  if (c->tuned) c->tiles = own->second;
  else if (it->second.any) c->tiles = it->second.all;
}

}  // namespace gpi

using gpi::DeviceGuard;
using gpi::fail;

namespace {

gp::Tiles from_abi(const gp_tiles& t) {
  gp::Tiles r;
  r.fb = t.faces_per_cta;
  r.lcb = t.lift_cells_per_cta;
  r.lnt = t.lift_threads;
  return r;
}

gp_tiles to_abi(const gp::Tiles& t) {
  gp_tiles r;
  r.faces_per_cta = t.fb;
  r.lift_cells_per_cta = t.lcb;
  r.lift_threads = t.lnt;
  return r;
}

int64_t ipow(int64_t b, int e) {
  int64_t r = 1;
  while (e-- > 0) r *= b;
  return r;
}

// Candidate shapes: the default; face CTAs of about 64..512 threads; lift CTAs of 64..512 threads
// with half a row to four rows per thread, or with 4..64 owners.
void candidates(const gp::Plan& p, const gp::LaunchForm& form, const gp::TileOps& ops, std::vector<gp::Tiles>& face,
                std::vector<gp::Tiles>& lift) {
  const gp::Tiles d = ops.defaults(p.k, form);
  const int L = p.L, KR = (int)ipow(p.k, p.dim - 1);
  face.assign(1, d);
  lift.assign(1, d);
  auto add_lift = [&](int owners, int threads) {
    gp::Tiles t = d;
    t.lnt = threads;
    t.lcb = std::max(1, owners);
    bool dup = false;
    for (const auto& u : lift) dup = dup || (u.lnt == t.lnt && u.lcb == t.lcb);
    if (!dup && ops.resolve(p.k, t, form)) lift.push_back(t);
  };
  for (int T : {64, 96, 128, 192, 256, 384, 512}) {
    gp::Tiles t = d;
    t.fb = std::max(1, T / L);
    bool dup = false;
    for (const auto& u : face) dup = dup || u.fb == t.fb;
    if (!dup && ops.resolve(p.k, t, form)) face.push_back(t);
  }
  for (int T : {64, 128, 256, 512}) {
    for (int halves : {1, 2, 4, 8}) add_lift(halves * T / (2 * KR), T);
    for (int owners : {4, 8, 16, 24, 32, 64})
      if (2 * owners * KR >= T && owners * KR <= 6 * T) add_lift(owners, T);
  }
}

}  // namespace

extern "C" {

gp_status gp_get_tiles(const gp_ctx* ctx, gp_tiles* out) {
  if (!ctx || !out) return fail(ctx, GP_EINVAL, "null argument");
  gp::Tiles t = ctx->tiles;
  if (!gpi::tile_ops(ctx->plan.dim, ctx->plan.precision).resolve(ctx->plan.k, t, ctx->form))
    return fail(ctx, GP_EINVAL, "the context holds an invalid tile shape");
  *out = to_abi(t);
  return GP_OK;
}

gp_status gp_set_tiles(gp_ctx* ctx, const gp_tiles* tiles) {
  if (!ctx || !tiles) return fail(ctx, GP_EINVAL, "null argument");
  gp::Tiles t = from_abi(*tiles);
  if (!gpi::tile_ops(ctx->plan.dim, ctx->plan.precision).resolve(ctx->plan.k, t, ctx->form))
    return fail(ctx, GP_EINVAL, "tile shape out of range (threads per CTA, shared memory or lift threads)");
  ctx->tiles = from_abi(*tiles);
  ctx->tuned = false;
  return GP_OK;
}

gp_status gp_tiles_record(int device, int dim, int degree, int precision, const gp_tiles* tiles) {
  if (!tiles) return fail(nullptr, GP_EINVAL, "null argument");
  if ((dim != 2 && dim != 3) || degree < 1 || degree > gp::KMAX ||
      (precision != GP_FP64 && precision != GP_FP32 && precision != GP_FP64_FF))
    return fail(nullptr, GP_EINVAL, "bad (dim, degree, precision)");
  gp::Tiles t = from_abi(*tiles);
  if (!gpi::tile_ops(dim, precision).resolve(degree, t, gp::LaunchForm{})) return fail(nullptr, GP_EINVAL, "tile shape out of range");
  std::lock_guard<std::mutex> lk(g_tiles_mu);
  Entry& e = g_tiles[std::make_tuple(device, dim, degree, precision)];
  e.kind.clear();
  e.any = true;
  e.all = e.last = from_abi(*tiles);
  return GP_OK;
}

gp_status gp_tiles_lookup(int device, int dim, int degree, int precision, gp_tiles* out) {
  if (!out) return fail(nullptr, GP_EINVAL, "null argument");
  std::lock_guard<std::mutex> lk(g_tiles_mu);
  auto it = g_tiles.find(std::make_tuple(device, dim, degree, precision));
  if (it == g_tiles.end()) return fail(nullptr, GP_EINVAL, "no entry");
  *out = to_abi(it->second.last);
  return GP_OK;
}

gp_status gp_tiles_keep(gp_ctx* ctx) {
  if (!ctx) return fail(nullptr, GP_EINVAL, "null context");
  std::lock_guard<std::mutex> lk(g_tiles_mu);
  if (ctx->use_brick) {
    g_brick_tiles[key_of(ctx)] = ctx->tiles;
  } else {
    Entry& e = g_tiles[key_of(ctx)];
    e.kind[kind_of(ctx)] = e.last = ctx->tiles;
  }
  return GP_OK;
}

gp_status gp_kernel_form(const gp_ctx* ctx, int32_t* form) {
  if (!ctx || !form) return fail(ctx, GP_EINVAL, "null argument");
  const gp::Plan& p = ctx->plan;
  form[0] = !ctx->use_brick && ctx->form.compact ? 1 : 0;
  form[1] = !ctx->use_brick && p.precision == GP_FP64 && !p.ldl.empty() ? 1 : 0;
  form[2] = ctx->use_brick ? 0 : gpi::tile_ops(p.dim, p.precision).size_class(p.k, ctx->form);
  form[3] = kTileVersion;
  return GP_OK;
}

gp_status gp_autotune(gp_ctx* ctx, int reps, gp_tiles* best, double* ms) {
  if (!ctx) return fail(nullptr, GP_EINVAL, "null context");
  if (!ctx->on_device) return fail(ctx, GP_EDEVICE, "context was built host-only (device = -1)");
  if (reps < 1) return fail(ctx, GP_EINVAL, "reps must be >= 1");
  const gp::Plan& p = ctx->plan;
  const gp::TileOps ops = gpi::tile_ops(p.dim, p.precision);
  std::vector<gp::Tiles> face, lift;
  candidates(p, ctx->form, ops, face, lift);
  gp::Tiles cur = ctx->tiles;
  if (!ops.resolve(p.k, cur, ctx->form)) cur = ops.defaults(p.k, ctx->form);
  if (p.num_faces() == 0 || face.empty() || lift.empty()) {
    if (best) *best = to_abi(cur);
    if (ms) ms[0] = ms[1] = 0.0;
    return GP_OK;
  }
  DeviceGuard dg(ctx->device);
  // operands of the timed launches and a buffer larger than the L2 to flush it
  const size_t vb = (size_t)p.n_active * ctx->elem;
  const size_t flush_bytes = (size_t)256 << 20;
  void *x = nullptr, *y = nullptr, *fl = nullptr;
  cudaStream_t st = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t e = cudaMalloc(&x, std::max<size_t>(vb, 16));
  if (e == cudaSuccess) e = cudaMalloc(&y, std::max<size_t>(vb, 16));
  if (e == cudaSuccess) e = cudaMalloc(&fl, flush_bytes);
  if (e == cudaSuccess) e = cudaMemset(x, 0, std::max<size_t>(vb, 16));
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  gp_status status = GP_OK;
  // mean time of one kernel (which = 1 face, 2 lift) or of an apply (3) over reps cold-L2 launches, or launches
  // back to back
  auto time_one = [&](const gp::Tiles& t, int which, double& out_ms, bool flush = true) -> bool {
    double total = 0;
    for (int r = -1; r < reps && e == cudaSuccess; ++r) {   // r = -1: untimed warm-up
      if (flush) e = cudaMemsetAsync(fl, r & 0xff, flush_bytes, st);
      if (e == cudaSuccess) e = cudaEventRecord(e0, st);
      if (e == cudaSuccess && gpi::launch(ctx, x, y, 0, st, nullptr, false, &t, which) != GP_OK) {
        status = GP_ECUDA;
        return false;
      }
      if (e == cudaSuccess) e = cudaEventRecord(e1, st);
      if (e == cudaSuccess) e = cudaEventSynchronize(e1);
      float m = 0;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&m, e0, e1);
      if (r >= 0) total += m;
    }
    out_ms = total / reps;
    return e == cudaSuccess;
  };
  gp::Tiles bf = cur, bl = cur;
  double tf = 1e30, tl = 1e30;
  if (ctx->use_brick) {
    // brick path: faces per chunk of the brick kernel, timed over whole applies
    for (const gp::Tiles& t : face) {
      double m;
      if (!time_one(t, 3, m)) break;
      if (m < tf) { tf = m; bf = t; }
    }
    tl = 0.0;
  }
  std::vector<double> face_ms, lift_ms;   // of the candidates; the first is the default
  for (const gp::Tiles& t : face) {
    if (ctx->use_brick) break;
    double m;
    if (!time_one(t, 1, m)) break;
    face_ms.push_back(m);
    if (m < tf) { tf = m; bf = t; }
  }
  // the lift reads the face outputs of the best face shape
  if (!ctx->use_brick && e == cudaSuccess && status == GP_OK &&
      gpi::launch(ctx, x, y, 0, st, nullptr, false, &bf, 1) != GP_OK)
    status = GP_ECUDA;
  for (const gp::Tiles& t : lift) {
    if (ctx->use_brick || e != cudaSuccess || status != GP_OK) break;
    double m;
    if (!time_one(t, 2, m)) break;
    lift_ms.push_back(m);
    if (m < tl) { tl = m; bl = t; }
  }
  // the default stays unless the whole apply gains, also with its operands in L2
  const gp::Tiles def = ops.defaults(p.k, ctx->form);
  gp::Tiles both = bf;
  both.lcb = bl.lcb;
  both.lnt = bl.lnt;
  const bool same = both.fb == def.fb && both.lcb == def.lcb && both.lnt == def.lnt;
  if (!ctx->use_brick && !same && e == cudaSuccess && status == GP_OK) {
    double m[2][2] = {};   // [default, tuned][flushed, back to back]
    bool done = true;
    for (int f = 0; f < 2 && done; ++f)
      done = time_one(def, 3, m[0][f], f == 0) && time_one(both, 3, m[1][f], f == 0);
    if (done && !(m[1][0] < m[0][0] && m[1][1] < m[0][1])) {
      bf = bl = def;
      tf = face_ms[0];
      tl = lift_ms[0];
    }
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (st) cudaStreamDestroy(st);
  if (x) cudaFree(x);
  if (y) cudaFree(y);
  if (fl) cudaFree(fl);
  if (status != GP_OK) return status;   // message set by launch
  if (e != cudaSuccess)
    return fail(ctx, e == cudaErrorMemoryAllocation ? GP_ENOMEM : GP_ECUDA,
                std::string("autotune: ") + cudaGetErrorString(e));
  gp::Tiles chosen;
  chosen.fb = bf.fb;
  chosen.lcb = bl.lcb;
  chosen.lnt = bl.lnt;
  ctx->tiles = chosen;
  ctx->tuned = true;
  gp_tiles_keep(ctx);
  if (best) *best = to_abi(chosen);
  if (ms) {
    ms[0] = tf;
    ms[1] = tl;
  }
  return GP_OK;
}

}  // extern "C"
