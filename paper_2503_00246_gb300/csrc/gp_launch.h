// Host-side launch interface between the C ABI and the templated kernels.
#pragma once

#include <cstdint>
#include <cstring>
#include <vector>
#include <cuda_runtime.h>

#include "gp_brick.cuh"
#include "gp_cell.cuh"
#include "gp_kernels.cuh"

namespace gp {

// What the default tile shapes of a launch depend on: whether FP32 stores compact outputs, the ghost faces
// of the mesh (of all segments of a batch), and whether the face kernel is the model system's, which stores W_F in
// every arithmetic (the system's gather reads it).
struct LaunchForm {
  bool compact = false;
  int64_t faces = 0;
  bool system = false;
};

struct ApplyArgs {
  int dim = 0, k = 0;
  const void* x = nullptr;   // device, n_active elements
  void* y = nullptr;         // device, n_active elements
  void* tp = nullptr;        // device scratch: face outputs, nf * (2k+1) * L values
  int add = 0;               // 0: y = Gx, 1: y += Gx
  const int32_t* frows = nullptr;
  int64_t rbase[4] = {0, 0, 0, 0};
  int32_t fstart[4] = {0, 0, 0, 0};
  LiftArgs la{};
  const int2* zruns = nullptr;
  int32_t nzruns = 0;        // zero runs to fill (0 for the add form)
  const double* g = nullptr; // host FP64: k x (2k+1)
  const double* m = nullptr; // host FP64: the lumped mass, 2 (k+1) values (Plan::lump)
  const double* w = nullptr; // host FP64: factors of the normal lines (Plan::fac)
  const void* fac = nullptr; // device: those of FP32, or of the triangular basis
  const double* s = nullptr; // host FP64: k
  const double* ldl = nullptr;  // host FP64: the triangular normal basis (Plan::ldl); nullptr: g and s as they are
  cudaEvent_t* ev = nullptr;  // optional: 3 events recorded around the two kernels
  Tiles tiles{};              // 0 fields: the defaults of default_tiles
  int which = 3;              // bit 0: face kernel, bit 1: lift kernel (the autotuner times them apart)
  LaunchForm form{};          // launch_form
  const int32_t* slabs = nullptr;  // host: SLAB ints per slab (see Plan::slabs); nslab > 1: slab pipeline
  int nslab = 0;
  cudaEvent_t* slab_events = nullptr;  // host, nslab events: recorded after each slab's lift (the
                                       // face launches then follow them in plain stream order)
  cudaEvent_t* slab_inputs = nullptr;  // host, nslab events (with slab_events): the face launch of
                                       // slab s waits for slab_inputs[s] (its part of x is in place)
  bool brick = false;         // the brick path (brick kernel + plane fixup) instead of face + lift
  BrickArgs ba{};             // brick tables (zero-run fields are filled by the launcher)
  PlaneArgs pa{};             // plane-fixup tables
};

// Whether an FP32 context stores compact face outputs.  Small W_F stays in L2, where the lift of W_F
// and its two fewer phases are the faster one for small k (us of an apply, W_F / compact: k = 2, 40^3 ball 6.4 / 7.3; k = 3, 20^3 5.7 /
// 6.6; k = 4, 12^3 7.7 / 8.7; k = 6, 32^3, 17 MB, 27 / 34); the compact form is from 10 MB of W_F at k = 3
// (64^3 21.0 / 16.4), 3 MB at k = 4 (24^3 10.2 / 9.7), 24 MB at k = 6 (64^3 81 / 72), and at any size for
// k = 5, 7 and 8 (10^3: 9.9 / 8.5, k = 7, 11^3 12.9 / 10.4, k = 8, 8^3 13.9 / 11.6).  In 2D, whose W_F is small
// always, from k = 6 on (64^2 disc, k = 4, 6.9 / 7.3; 600^2, k = 7, 11.3 / 11.0).
inline bool store_compact(int dim, int k, int64_t w_bytes) {
  const int64_t mb = (int64_t)1 << 20;
  if (dim == 2) return k >= 6;
  return k == 5 || k >= 7 || (k == 6 && w_bytes > 24 * mb) || (k == 4 && w_bytes > 3 * mb) ||
         (k == 3 && w_bytes > 10 * mb);
}
inline LaunchForm launch_form(bool fp32, int dim, int k, int64_t w_bytes, int64_t faces) {
  return LaunchForm{fp32 && store_compact(dim, k, w_bytes), faces};
}

// Default tile shapes {faces per face CTA, owners per lift CTA, lift threads}: up to four per degree, by the
// number of ghost faces.  Small meshes want many small CTAs (few faces each, a row or less per lift thread), or
// most of the GPU idles while each CTA works through its rows; large ones want what keeps most warps busy:
// FP64 and float-float face CTAs that fill the SM, lift CTAs with 32 owners, where every row type fills whole
// warps, and for the compact outputs two to four lines per thread.  Each entry is the fastest of about 30 lift
// and 10 face shapes, times taken on 15 balls (10^3 .. 96^3) and 5 gyroids per degree and 6 discs in 2D, the
// limits between them where the fastest shape changes; the same shape at every size took, against
// these, up to (us): FP32 compact k = 8, 40^3, 77 / 55, k = 7, 36^3, 50 / 34, k = 5, 64^3, 60 / 44;
// float-float k = 8, 20^3, 70 / 57, k = 5, 28^3, 39 / 26; FP64 k = 4, 25^3, 50 / 36, k = 1, 40^3, 27 / 14,
// 2D, k = 7, 300^2, 38 / 17.
struct TileRule {
  int32_t upto[3];   // faces up to which the first, the second and the third shape run
  Tiles shape[4];
};
constexpr TileRule tiles_at(Tiles a) { return {{0, 0, 0}, {a, a, a, a}}; }
constexpr TileRule tiles_at(Tiles a, int n, Tiles b) { return {{n, n, n}, {a, b, b, b}}; }
constexpr TileRule tiles_at(Tiles a, int n, Tiles b, int m, Tiles c) { return {{n, m, m}, {a, b, c, c}}; }
constexpr TileRule tiles_at(Tiles a, int n, Tiles b, int m, Tiles c, int l, Tiles d) { return {{n, m, l}, {a, b, c, d}}; }
typedef TileRule TileRules[2][8];   // [dimension - 2][degree - 1]
constexpr TileRules kTilesF64 = {
    {tiles_at({96, 256, 256}, 1000, {160, 256, 512}), tiles_at({42, 256, 512}), tiles_at({16, 16, 64}),
     tiles_at({19, 128, 512}, 1000, {6, 32, 256}), tiles_at({10, 24, 256}), tiles_at({4, 32, 256}),
     tiles_at({4, 16, 256}), tiles_at({3, 32, 512})},
    {tiles_at({128, 256, 512}), tiles_at({14, 128, 512}, 2500, {10, 64, 512}, 24000, {21, 32, 256}),
     tiles_at({2, 16, 256}, 6000, {8, 16, 256}, 70000, {24, 32, 512}), tiles_at({6, 32, 512}, 19000, {20, 32, 512}),
     tiles_at({4, 8, 256}, 6000, {7, 16, 512}),
     tiles_at({5, 1, 128}, 700, {3, 3, 256}, 3000, {7, 4, 256}, 3600, {5, 14, 512}), tiles_at({2, 8, 512}),
     tiles_at({3, 4, 256})}};
constexpr TileRules kTilesFF = {
    {tiles_at({128, 256, 512}), tiles_at({42, 128, 256}), tiles_at({24, 32, 128}), tiles_at({19, 32, 256}),
     tiles_at({10, 24, 256}), tiles_at({9, 32, 256}), tiles_at({8, 16, 256}), tiles_at({14, 32, 512})},
    {tiles_at({128, 256, 512}), tiles_at({10, 64, 256}, 15000, {14, 64, 512}, 35000, {14, 128, 512}),
     tiles_at({4, 16, 256}, 12000, {8, 28, 256}, 21000, {8, 24, 128}),
     tiles_at({5, 32, 512}, 12000, {5, 32, 256}),
     tiles_at({3, 16, 512}, 6000, {7, 24, 512}, 19000, {7, 32, 256}),
     tiles_at({2, 14, 512}, 1000, {2, 3, 128}, 2600, {3, 4, 128}, 3500, {3, 32, 512}),
     tiles_at({2, 8, 512}, 1400, {2, 16, 512}, 2800, {2, 24, 512}, 9700, {4, 32, 256}),
     tiles_at({3, 4, 256}, 2500, {3, 32, 512}, 6000, {3, 32, 256})}};
// FP32 that stores W_F, and compact outputs (a row that store_compact leaves out only serves checks of shapes
// given by hand)
constexpr TileRules kTilesF32 = {
    {tiles_at({192, 128, 256}), tiles_at({85, 128, 256}), tiles_at({48, 32, 128}), tiles_at({25, 64, 512}),
     tiles_at({21, 16, 128}), tiles_at({18, 32, 256}), tiles_at({12, 16, 256}), tiles_at({10, 32, 512})},
    {tiles_at({48, 64, 128}, 50000, {64, 128, 128}), tiles_at({21, 64, 512}, 21000, {14, 64, 512}),
     tiles_at({8, 16, 256}), tiles_at({5, 32, 512}), tiles_at({3, 8, 256}),
     tiles_at({2, 1, 64}, 2500, {3, 4, 256}), tiles_at({1, 4, 256}), tiles_at({1, 4, 256})}};
constexpr TileRules kTilesF32Compact = {
    {tiles_at({48, 64, 128}), tiles_at({85, 128, 256}), tiles_at({64, 64, 256}), tiles_at({51, 32, 128}),
     tiles_at({21, 24, 128}), tiles_at({18, 32, 256}), tiles_at({12, 32, 256}), tiles_at({14, 32, 256})},
    {tiles_at({64, 64, 128}), tiles_at({14, 64, 256}), tiles_at({6, 28, 256}, 50000, {8, 32, 128}),
     tiles_at({5, 32, 512}, 35000, {5, 32, 256}),
     tiles_at({3, 8, 256}, 3600, {3, 20, 256}, 35000, {3, 24, 256}),
     tiles_at({3, 7, 128}, 21000, {3, 14, 128}),
     tiles_at({2, 4, 256}, 2500, {1, 10, 256}, 7700, {2, 8, 128}),
     tiles_at({1, 4, 256}, 2800, {1, 6, 128}, 9700, {1, 8, 128})}};

// The model system's face kernel runs beside its cell kernel: CTAs of 110 to 260 threads are within 2 % of the
// fastest at every size (12 meshes per degree), and small ones cost up to 30 us (FP64, k = 2, 16^3 ball, 7 / 10 / 21
// faces: 56 / 25 / 24 us).  FP32, FP64, float-float in 3D; in 2D about 256 threads.
constexpr int kSystemFaces[3][8] = {{64, 14, 8, 5, 3, 3, 2, 1}, {64, 21, 16, 20, 7, 5, 4, 3}, {64, 21, 16, 5, 7, 5, 4, 3}};

template <int D, int K, typename V>
const TileRule& tile_rule(const LaunchForm& form) {
  constexpr bool F32 = std::is_same<V, float>::value, F64 = std::is_same<V, double>::value;
  return (F32 ? (form.compact ? kTilesF32Compact : kTilesF32) : F64 ? kTilesF64 : kTilesFF)[D - 2][K - 1];
}
inline int tile_class(const TileRule& r, const LaunchForm& form) {
  int c = 0;
  while (c < 3 && form.faces > r.upto[c]) ++c;
  return c;
}
template <int D, int K, typename V>
Tiles default_tiles_t(const LaunchForm& form) {
  constexpr bool F32 = std::is_same<V, float>::value, F64 = std::is_same<V, double>::value;
  const TileRule& r = tile_rule<D, K, V>(form);
  Tiles t = r.shape[tile_class(r, form)];
  if (form.system) t.fb = D == 3 ? (F32 ? kSystemFaces[0] : F64 ? kSystemFaces[1] : kSystemFaces[2])[K - 1] : Shape<D, K>::FB;
  return t;
}

// Fills zero fields of t with the defaults and checks the limits of the kernels
// (threads per CTA <= MAX_CTA_THREADS, lift threads a multiple of 32, dynamic
// shared memory <= MAX_DYN_SMEM).  Returns false if t is out of range.
template <int D, int K, typename V>
bool resolve_tiles(Tiles& t, const LaunchForm& form) {
  const Tiles d = default_tiles_t<D, K, V>(form);
  if (t.fb == 0) t.fb = d.fb;
  if (t.lcb == 0) t.lcb = d.lcb;
  if (t.lnt == 0) t.lnt = d.lnt;
  if (t.fb < 1 || t.fb * Shape<D, K>::L > MAX_CTA_THREADS || face_planes<D, K, V>(t.fb) > MAX_DYN_SMEM) return false;
  if (t.lnt < 32 || t.lnt > MAX_CTA_THREADS || t.lnt % 32 != 0) return false;
  if (t.lcb < 1 || lift_smem<D, K>(t.lcb) > MAX_DYN_SMEM) return false;
  return true;
}

// Per (arithmetic, dimension): default tiles and range check for degree k.
struct TileOps {
  Tiles (*defaults)(int k, const LaunchForm& form);
  int (*size_class)(int k, const LaunchForm& form);   // which of the rule's shapes is the default
  bool (*resolve)(int k, Tiles& t, const LaunchForm& form);
};
TileOps tile_ops_f64_d2();
TileOps tile_ops_f64_d3();
TileOps tile_ops_f32_d2();
TileOps tile_ops_f32_d3();
TileOps tile_ops_ff_d2();
TileOps tile_ops_ff_d3();

#define GP_TILE_CASE(D, A, K) \
  case K: return resolve_tiles<D, K, typename A::V>(t, form);
#define GP_CLASS_CASE(D, A, K) \
  case K: return tile_class(tile_rule<D, K, typename A::V>(form), form);
#define GP_TILE_OPS(D, A)                                                                     \
  TileOps ops;                                                                                \
  ops.size_class = [](int k, const LaunchForm& form) -> int {                                 \
    switch (k) {                                                                              \
      GP_CLASS_CASE(D, A, 1) GP_CLASS_CASE(D, A, 2) GP_CLASS_CASE(D, A, 3) GP_CLASS_CASE(D, A, 4) \
      GP_CLASS_CASE(D, A, 5) GP_CLASS_CASE(D, A, 6) GP_CLASS_CASE(D, A, 7) GP_CLASS_CASE(D, A, 8) \
      default: return 0;                                                                      \
    }                                                                                         \
  };                                                                                          \
  ops.defaults = [](int k, const LaunchForm& form) -> Tiles {                                 \
    switch (k) {                                                                              \
      case 1: return default_tiles_t<D, 1, typename A::V>(form);                              \
      case 2: return default_tiles_t<D, 2, typename A::V>(form);                              \
      case 3: return default_tiles_t<D, 3, typename A::V>(form);                              \
      case 4: return default_tiles_t<D, 4, typename A::V>(form);                              \
      case 5: return default_tiles_t<D, 5, typename A::V>(form);                              \
      case 6: return default_tiles_t<D, 6, typename A::V>(form);                              \
      case 7: return default_tiles_t<D, 7, typename A::V>(form);                              \
      default: return default_tiles_t<D, 8, typename A::V>(form);                             \
    }                                                                                         \
  };                                                                                          \
  ops.resolve = [](int k, Tiles& t, const LaunchForm& form) -> bool {                         \
    switch (k) {                                                                              \
      GP_TILE_CASE(D, A, 1) GP_TILE_CASE(D, A, 2) GP_TILE_CASE(D, A, 3) GP_TILE_CASE(D, A, 4) \
      GP_TILE_CASE(D, A, 5) GP_TILE_CASE(D, A, 6) GP_TILE_CASE(D, A, 7) GP_TILE_CASE(D, A, 8) \
      default: return false;                                                                  \
    }                                                                                         \
  };                                                                                          \
  return ops;

// One entry point per (arithmetic, dimension); each dispatches on k = 1..8.
cudaError_t apply_f64_d2(const ApplyArgs& a, cudaStream_t st);
cudaError_t apply_f64_d3(const ApplyArgs& a, cudaStream_t st);
cudaError_t apply_f32_d2(const ApplyArgs& a, cudaStream_t st);
cudaError_t apply_f32_d3(const ApplyArgs& a, cudaStream_t st);
cudaError_t apply_ff_d2(const ApplyArgs& a, cudaStream_t st);
cudaError_t apply_ff_d3(const ApplyArgs& a, cudaStream_t st);

// Faces per chunk of the brick kernel: the tile's fb, else about 256 threads.
template <int D, int K>
inline int brick_fb(const Tiles& t) {
  constexpr int L = Shape<D, K>::L;
  const int fb = t.fb > 0 ? t.fb : Shape<D, K>::FB;
  return fb * L <= MAX_CTA_THREADS ? fb : MAX_CTA_THREADS / L;
}

constexpr size_t BRICK_MAX_SMEM = 200 * 1024;   // dynamic shared memory the brick kernel may ask for

// The brick path: brick kernel (zero-fill CTAs first), then the plane fixup as its
// programmatic dependent.  Ar.ev (3 events) brackets the two kernels when given.
template <int D, int K, class A>
cudaError_t run_brick(const ApplyArgs& Ar, const Consts<typename A::V, K>& c, cudaStream_t st) {
  using V = typename A::V;
  using IO = typename A::IO;
  constexpr int L = Shape<D, K>::L;
  const int fb = brick_fb<D, K>(Ar.tiles);
  BrickArgs ba = Ar.ba;
  ba.zruns = Ar.zruns;
  ba.nzruns = Ar.nzruns;
  ba.nzblocks = (Ar.nzruns + ZGROUP - 1) / ZGROUP;
  const size_t smem = brick_smem<D, K, V>(ba.maxown, ba.maxcell, fb);
  if (smem > BRICK_MAX_SMEM) return cudaErrorInvalidConfiguration;
  // the opt-in limit covers static + dynamic shared memory: raise it once per instantiation
  // and device, whatever this launch needs
  static bool smem_raised[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 && !smem_raised[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(brick_kernel<D, K, A>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)BRICK_MAX_SMEM);
    if (e != cudaSuccess) return e;
    smem_raised[dev] = true;
  }
  const int grid = ba.nzblocks + ba.nbricks;
  if (Ar.ev) cudaEventRecord(Ar.ev[0], st);
  if (grid > 0) brick_kernel<D, K, A><<<grid, fb * L, smem, st>>>((const IO*)Ar.x, (IO*)Ar.y, Ar.add, ba, fb, c);
  if (Ar.ev) cudaEventRecord(Ar.ev[1], st);
  if (Ar.pa.nplane > 0 && ba.nbricks > 0) {
    const int nb = (Ar.pa.nplane + 255) / 256;
    if (Ar.ev) {
      plane_fixup_kernel<A><<<nb, 256, 0, st>>>((IO*)Ar.y, Ar.add, Ar.pa);
    } else {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)nb);
      cfg.blockDim = dim3(256u);
      cfg.stream = st;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[0].val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      const cudaError_t e = cudaLaunchKernelEx(&cfg, plane_fixup_kernel<A>, (IO*)Ar.y, Ar.add, Ar.pa);
      if (e != cudaSuccess) return e;
    }
  }
  if (Ar.ev) cudaEventRecord(Ar.ev[2], st);
  return cudaGetLastError();
}

// ints per slab of the slab pipeline: owner range [lo, hi), then per axis the face range [lo, hi)
constexpr int SLAB_INTS = 8;

// Launches kernel with programmatic stream serialization (it may start when its predecessor
// signals griddepcontrol.launch_dependents).
template <typename... P, typename... Args>
cudaError_t launch_pdl(void (*kernel)(P...), int grid, int threads, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Owner cells per lift CTA and dynamic shared memory of the lift kernel.
template <int D, int K, typename V>
int lift_cells(const Tiles& t, const bool compact) {
  if constexpr (StoreCompact<D, K, V>::value)
    if (compact) return lift_lines_cells<D, K, V>(t.lcb);
  return t.lcb;
}
template <int D, int K, typename V>
size_t lift_dyn_smem(int cb, const bool compact) {
  if constexpr (StoreCompact<D, K, V>::value)
    if (compact) return lift_lines_smem<D, K, V>(cb);
  return lift_smem<D, K>(cb);
}

// Launches the lift of the owners la, as a programmatic dependent of the kernel before it (pdl)
// or in plain stream order.
template <int D, int K, class A>
cudaError_t launch_lift(bool pdl, const bool compact, const Tiles& t, const typename A::V* w, typename A::IO* y,
                        int add, const LiftArgs& la, const Consts<typename A::V, K>& c, cudaStream_t st) {
  using V = typename A::V;
  const int cb = lift_cells<D, K, V>(t, compact);
  const int nlb = (la.nlift + cb - 1) / cb;
  const size_t smem = lift_dyn_smem<D, K, V>(cb, compact);
  if constexpr (StoreCompact<D, K, V>::value) {
    if (compact) {
      if (pdl) return launch_pdl(lift_lines_kernel<D, K, A>, nlb, t.lnt, smem, st, w, y, add, la, cb, c);
      lift_lines_kernel<D, K, A><<<nlb, t.lnt, smem, st>>>(w, y, add, la, cb, c);
      return cudaGetLastError();
    }
  }
  if constexpr (!StoreCompact<D, K, V>::always) {
    if (pdl) return launch_pdl(lift_kernel<D, K, A>, nlb, t.lnt, smem, st, w, y, add, la, cb);
    lift_kernel<D, K, A><<<nlb, t.lnt, smem, st>>>(w, y, add, la, cb);
    return cudaGetLastError();
  }
  return cudaErrorInvalidConfiguration;   // (launch_form gives such a context compact outputs)
}

// The face kernel of this arithmetic: with the triangular normal basis or the jump vectors, storing its
// compact outputs or W_F.
template <int D, int K, class A>
auto pick_face(const bool ldl, const bool compact) {
  using V = typename A::V;
  constexpr bool CO = StoreCompact<D, K, V>::value, LD = std::is_same<V, double>::value;
  static_assert(!(CO && LD), "compact outputs are expanded with the jump vectors");
  auto f = face_kernel<D, K, A, false, false>;
  if constexpr (CO) {
    if (compact) f = face_kernel<D, K, A, true, false>;
  }
  if constexpr (LD) {
    if (ldl) f = face_kernel<D, K, A, false, true>;
  }
  return f;
}

// The face + lift path as a pipeline of slabs along the last axis, so that the face outputs of a
// slab are still in L2 when its lift reads them: face(0), lift(0), face(1), lift(1), ...  Slab s
// holds a range of owner cells and the faces that range needs and no earlier range needed.
// lift(s) waits for face(s) before it reads W; face(s + 1) starts once every CTA of lift(s) has
// passed that wait, overlaps lift(s) (it writes other face outputs and reads only x), and waits for
// lift(s) only before it exits, so that each grid completes after all earlier ones (the last lift
// completes last).  The first face launch also zero-fills.  With slab_events, an event is
// recorded after every lift (another stream can then take the slab's finished part of y) and
// each face launch follows it in plain stream order.
template <int D, int K, class A>
cudaError_t run_slabs(const ApplyArgs& Ar, const Consts<typename A::V, K>& c, const Tiles& t, const bool ldl,
                      cudaStream_t st) {
  using S = Shape<D, K>;
  using V = typename A::V;
  using IO = typename A::IO;
  const int R[3] = {S::L, S::NP * ((D == 3) ? K + 1 : 1), S::NP * (K + 1)};   // row entries per face
  constexpr int KR = LiftShape<D, K>::KR, NW = LiftShape<D, K>::NW;
  for (int s = 0; s < Ar.nslab; ++s) {
    const int32_t* sl = Ar.slabs + (size_t)s * SLAB_INTS;
    FaceArgs fa;
    fa.frows = Ar.frows;
    fa.fac = Ar.fac;
    fa.zruns = Ar.zruns;
    fa.nzruns = s == 0 ? Ar.nzruns : 0;
    fa.tail_wait = s > 0 && !Ar.slab_events;
    for (int a = 0; a < 4; ++a) {
      const bool in = a < D;
      fa.fstart[a] = in ? sl[2 + 2 * a] : 0;
      fa.fend[a] = in ? sl[3 + 2 * a] : 0;
      fa.rbase[a] = in ? Ar.rbase[a] + (int64_t)(fa.fstart[a] - Ar.fstart[a]) * R[a] : 0;
    }
    const int nb = face_grid(fa, D, t.fb);
    if (Ar.slab_inputs) {
      const cudaError_t e = cudaStreamWaitEvent(st, Ar.slab_inputs[s], 0);
      if (e != cudaSuccess) return e;
    }
    if (nb > 0) {
      const auto face = pick_face<D, K, A>(ldl, Ar.form.compact);
      const cudaError_t e =
          (s == 0 || Ar.slab_events)
              ? (face<<<nb, t.fb * S::L, face_smem<D, K, V>(t.fb), st>>>((const IO*)Ar.x, (V*)Ar.tp, (IO*)Ar.y, fa, t.fb, c),
                 cudaGetLastError())
              : launch_pdl(face, nb, t.fb * S::L, face_smem<D, K, V>(t.fb), st, (const IO*)Ar.x, (V*)Ar.tp, (IO*)Ar.y,
                           fa, (int)t.fb, c);
      if (e != cudaSuccess) return e;
    }
    LiftArgs la = Ar.la;
    la.lwin = Ar.la.lwin + (size_t)sl[0] * NW;
    la.lrow = Ar.la.lrow + (size_t)sl[0] * KR;
    la.lmask = Ar.la.lmask ? Ar.la.lmask + sl[0] : nullptr;
    la.nlift = sl[1] - sl[0];
    if (la.nlift > 0) {
      // programmatic dependent of this slab's face launch (a plain launch after an event)
      const cudaError_t e =
          launch_lift<D, K, A>(nb > 0 || !Ar.slab_events, Ar.form.compact, t, (const V*)Ar.tp, (IO*)Ar.y, Ar.add, la, c, st);
      if (e != cudaSuccess) return e;
    }
    if (Ar.slab_events) {
      const cudaError_t e = cudaEventRecord(Ar.slab_events[s], st);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaGetLastError();
}

// Native FP64 runs the triangular normal basis where the host found one.
template <typename V>
struct UseLdl {
  static constexpr bool value = std::is_same<V, double>::value;
};
template <typename V, int K>
void ldl_consts(const double* p, Consts<V, K>& c) {
  for (int j = 0; j < K; ++j)
    for (int b = 0; b <= K; ++b) c.g[j][b] = from_host<V>(p[j * (K + 1) + b]);
}

template <int D, int K, class A>
cudaError_t run_apply(const ApplyArgs& Ar, cudaStream_t st) {
  using S = Shape<D, K>;
  using V = typename A::V;
  using IO = typename A::IO;
  Consts<V, K> c;
  for (int j = 0; j < K; ++j)
    for (int b = 0; b < 2 * K + 1; ++b) c.g[j][b] = from_host<V>(Ar.g[j * (2 * K + 1) + b]);
  for (int j = 0; j < K; ++j) {
    c.s[j] = from_host<V>(Ar.s[j]);
    for (int b = 0; b < 2 * K + 1; ++b) c.gs[j][b] = from_host<V>(Ar.s[j] * Ar.g[j * (2 * K + 1) + b]);
  }
  mass_consts<D, K, V>(Ar.m, Ar.w, c);
  // the triangular basis takes the place of g and s (the brick path runs the general form)
  constexpr bool HAS_LDL = UseLdl<V>::value;
  const bool ldl = HAS_LDL && Ar.ldl && !Ar.brick;
  if (ldl) ldl_consts<V, K>(Ar.ldl, c);
  if (Ar.brick) return run_brick<D, K, A>(Ar, c, st);
  Tiles t = Ar.tiles;
  if (!resolve_tiles<D, K, V>(t, Ar.form)) return cudaErrorInvalidConfiguration;
  if (Ar.nslab > 1 && !Ar.ev && Ar.which == 3) return run_slabs<D, K, A>(Ar, c, t, ldl, st);
  FaceArgs fa;
  fa.frows = Ar.frows;
  fa.fac = Ar.fac;
  for (int a = 0; a < 4; ++a) fa.rbase[a] = Ar.rbase[a];
  fa.zruns = Ar.zruns;
  fa.nzruns = Ar.nzruns;
  fa.tail_wait = 0;
  for (int a = 0; a < 4; ++a) fa.fstart[a] = Ar.fstart[a];
  for (int a = 0; a < 4; ++a) fa.fend[a] = a < D ? Ar.fstart[a + 1] : Ar.fstart[D];
  const int nb = face_grid(fa, D, t.fb);
  const bool faces = Ar.fstart[D] > 0;
  if (Ar.ev) cudaEventRecord(Ar.ev[0], st);
  if (nb > 0 && (Ar.which & 1)) {
    const auto face = pick_face<D, K, A>(ldl, Ar.form.compact && !Ar.form.system);
    face<<<nb, t.fb * S::L, face_smem<D, K, V>(t.fb), st>>>((const IO*)Ar.x, (V*)Ar.tp, (IO*)Ar.y, fa, t.fb, c);
  }
  if (Ar.ev) cudaEventRecord(Ar.ev[1], st);
  if (Ar.la.nlift > 0 && faces && (Ar.which & 2)) {
    // programmatic dependent launch: the lift's CTAs start while the face grid drains
    const cudaError_t e = launch_lift<D, K, A>(!Ar.ev && (Ar.which & 1), Ar.form.compact, t, (const V*)Ar.tp, (IO*)Ar.y, Ar.add,
                                               Ar.la, c, st);
    if (e != cudaSuccess) return e;
  }
  if (Ar.ev) cudaEventRecord(Ar.ev[2], st);
  return cudaGetLastError();
}

// ------------------------------------------------------------- batches --
// Host description of one batch segment (one problem, one right-hand side).
struct SegSpec {
  FaceArgs fa;          // frows, rbase, fstart, zruns, nzruns of the segment's problem
  LiftArgs la;
  void* wp = nullptr;   // the segment's face-output buffer
  const void* gs = nullptr;   // device: K x (2K+1) scaled jump vectors of the segment's problem, or its B
  double s[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // the problem's s_j
};

// Packs the segments of one (d, k, arithmetic) group into the device layouts of
// FaceSeg<V, K> and LiftSeg, with the CTA offsets of both launches.
template <int D, int K, class A>
bool pack_batch(const std::vector<SegSpec>& in, const LaunchForm& form, Tiles& t, std::vector<unsigned char>& fsegs,
                std::vector<unsigned char>& lsegs, int& face_blocks, int& lift_blocks) {
  using V = typename A::V;
  const bool compact = form.compact;
  if (!resolve_tiles<D, K, V>(t, form)) return false;
  fsegs.assign(in.size() * sizeof(FaceSeg<V, K>), 0);
  lsegs.assign(in.size() * sizeof(LiftSeg), 0);
  int fb = 0, lb = 0;
  for (size_t i = 0; i < in.size(); ++i) {
    FaceSeg<V, K> fs;
    fs.fa = in[i].fa;
    fs.fa.tail_wait = 0;
    for (int a = 0; a < 4; ++a) fs.fa.fend[a] = a < D ? fs.fa.fstart[a + 1] : fs.fa.fstart[D];
    const int nb = face_grid(fs.fa, D, t.fb);
    fs.wp = (V*)in[i].wp;
    fs.gs = (const V*)in[i].gs;
    for (int j = 0; j < K; ++j) fs.s[j] = from_host<V>(in[i].s[j]);
    fs.block0 = fb;
    fb += nb;
    LiftSeg ls;
    ls.la = in[i].la;
    ls.block0 = lb;
    const int cb = lift_cells<D, K, V>(t, compact);
    if (fs.fa.fstart[D] > 0) lb += (ls.la.nlift + cb - 1) / cb;
    std::memcpy(&fsegs[i * sizeof(FaceSeg<V, K>)], &fs, sizeof(fs));
    std::memcpy(&lsegs[i * sizeof(LiftSeg)], &ls, sizeof(ls));
  }
  face_blocks = fb;
  lift_blocks = lb;
  return true;
}

template <int D, int K, class A>
cudaError_t run_batch(const void* fsegs, const void* lsegs, const void* ptrs, int nseg, int face_blocks,
                      int lift_blocks, const double* g, const double* m, const double* w, bool ldl,
                      const LaunchForm& form, Tiles t, cudaStream_t st) {
  using V = typename A::V;
  using IO = typename A::IO;
  using S = Shape<D, K>;
  const bool compact = form.compact;
  if (!resolve_tiles<D, K, V>(t, form)) return cudaErrorInvalidConfiguration;
  Consts<V, K> c;
  for (int j = 0; j < K; ++j)
    for (int b = 0; b < 2 * K + 1; ++b) c.g[j][b] = from_host<V>(g[j * (2 * K + 1) + b]);
  mass_consts<D, K, V>(m, w, c);
  for (int j = 0; j < K; ++j) {
    c.s[j] = vzero<V>();                                          // per segment: FaceSeg::s
    for (int b = 0; b < 2 * K + 1; ++b) c.gs[j][b] = vzero<V>();  // per segment: FaceSeg::gs
  }
  using CO = StoreCompact<D, K, V>;
  if (CO::always && !compact) return cudaErrorInvalidConfiguration;   // (launch_form gives it compact outputs)
  auto face = face_kernel_batched<D, K, A, CO::always, false>;
  if constexpr (UseLdl<V>::value) {
    if (ldl) face = face_kernel_batched<D, K, A, false, true>;
  }
  if constexpr (CO::value) {
    if (compact) face = face_kernel_batched<D, K, A, true, false>;
  }
  if (face_blocks > 0)
    face<<<face_blocks, t.fb * S::L, face_smem<D, K, V>(t.fb), st>>>((const FaceSeg<V, K>*)fsegs, nseg,
                                                                   (const SegPtrs<IO>*)ptrs, t.fb, c);
  if (lift_blocks > 0) {
    const int cb = lift_cells<D, K, V>(t, compact);
    const size_t smem = lift_dyn_smem<D, K, V>(cb, compact);
    if constexpr (CO::value) {
      if (compact)
        lift_lines_kernel_batched<D, K, A><<<lift_blocks, t.lnt, smem, st>>>(
            (const LiftSeg*)lsegs, (const FaceSeg<V, K>*)fsegs, nseg, (const SegPtrs<IO>*)ptrs, cb, c);
    }
    if constexpr (!CO::always) {
      if (!compact)
        lift_kernel_batched<D, K, A><<<lift_blocks, t.lnt, smem, st>>>(
            (const LiftSeg*)lsegs, (const FaceSeg<V, K>*)fsegs, nseg, (const SegPtrs<IO>*)ptrs, cb);
    }
  }
  return cudaGetLastError();
}

// The scaled jump vectors s_j g_j[b] (k x (2k+1)) of one problem in the value type of the
// arithmetic (4 or 8 bytes per value), as the face kernels use them.
template <class A>
void scaled_jumps(int k, const double* g, const double* s, std::vector<unsigned char>& out) {
  using V = typename A::V;
  out.assign((size_t)k * (2 * k + 1) * sizeof(V), 0);
  V* o = reinterpret_cast<V*>(out.data());
  for (int j = 0; j < k; ++j)
    for (int b = 0; b < 2 * k + 1; ++b) o[j * (2 * k + 1) + b] = from_host<V>(s[j] * g[j * (2 * k + 1) + b]);
}

// Per translation unit: batch packing and launch for one (arithmetic, dimension).
struct BatchOps {
  bool (*pack)(int k, const std::vector<SegSpec>&, const LaunchForm&, Tiles&, std::vector<unsigned char>&,
               std::vector<unsigned char>&, int&, int&);
  void (*jumps)(int k, const double* g, const double* s, std::vector<unsigned char>& out);
  cudaError_t (*run)(int k, const void*, const void*, const void*, int, int, int, const double*, const double*,
                     const double*, bool, const LaunchForm&, Tiles, cudaStream_t);
};
BatchOps batch_ops_f64_d2();
BatchOps batch_ops_f64_d3();
BatchOps batch_ops_f32_d2();
BatchOps batch_ops_f32_d3();
BatchOps batch_ops_ff_d2();
BatchOps batch_ops_ff_d3();

#define GP_BATCH_OPS(D, A)                                                                              \
  BatchOps ops;                                                                                         \
  ops.jumps = scaled_jumps<A>;                                                                          \
  ops.pack = [](int k, const std::vector<SegSpec>& in, const LaunchForm& form, Tiles& t,               \
                std::vector<unsigned char>& fs,                                                         \
                std::vector<unsigned char>& ls, int& fb, int& lb) -> bool {                             \
    switch (k) {                                                                                        \
      case 1: return pack_batch<D, 1, A>(in, form, t, fs, ls, fb, lb);                                        \
      case 2: return pack_batch<D, 2, A>(in, form, t, fs, ls, fb, lb);                                        \
      case 3: return pack_batch<D, 3, A>(in, form, t, fs, ls, fb, lb);                                        \
      case 4: return pack_batch<D, 4, A>(in, form, t, fs, ls, fb, lb);                                        \
      case 5: return pack_batch<D, 5, A>(in, form, t, fs, ls, fb, lb);                                        \
      case 6: return pack_batch<D, 6, A>(in, form, t, fs, ls, fb, lb);                                        \
      case 7: return pack_batch<D, 7, A>(in, form, t, fs, ls, fb, lb);                                        \
      case 8: return pack_batch<D, 8, A>(in, form, t, fs, ls, fb, lb);                                        \
      default: return false;                                                                            \
    }                                                                                                   \
  };                                                                                                    \
  ops.run = [](int k, const void* fs, const void* ls, const void* pt, int ns, int fb, int lb,          \
               const double* g, const double* m, const double* w, bool l, const LaunchForm& form, Tiles t,    \
               cudaStream_t st) -> cudaError_t {                                                        \
    switch (k) {                                                                                        \
      case 1: return run_batch<D, 1, A>(fs, ls, pt, ns, fb, lb, g, m, w, l, form, t, st);                        \
      case 2: return run_batch<D, 2, A>(fs, ls, pt, ns, fb, lb, g, m, w, l, form, t, st);                        \
      case 3: return run_batch<D, 3, A>(fs, ls, pt, ns, fb, lb, g, m, w, l, form, t, st);                        \
      case 4: return run_batch<D, 4, A>(fs, ls, pt, ns, fb, lb, g, m, w, l, form, t, st);                        \
      case 5: return run_batch<D, 5, A>(fs, ls, pt, ns, fb, lb, g, m, w, l, form, t, st);                        \
      case 6: return run_batch<D, 6, A>(fs, ls, pt, ns, fb, lb, g, m, w, l, form, t, st);                        \
      case 7: return run_batch<D, 7, A>(fs, ls, pt, ns, fb, lb, g, m, w, l, form, t, st);                        \
      case 8: return run_batch<D, 8, A>(fs, ls, pt, ns, fb, lb, g, m, w, l, form, t, st);                        \
      default: return cudaErrorInvalidValue;                                                            \
    }                                                                                                   \
  };                                                                                                    \
  return ops;

// y (+)= (wm M_active + ws K_active) x over the active cells (cell kernel + gather; add = 1:
// onto y, 0: overwrite the nodes of active cells).  first = 1: the cell kernel is the first
// kernel of the call and is launched normally (it reads x before any dependency wait, so it must
// not start early under the previous kernel on the stream); 0: it follows the face kernel of
// the same call and starts as that kernel's programmatic dependent.
using CellsFn = cudaError_t (*)(int k, const void* x, void* y, const CellTabs& ct, const double* m, const double* s,
                                double h, double wm, double ws, int add, int first, cudaStream_t st);
CellsFn cells_f64_d2();
CellsFn cells_f64_d3();
CellsFn cells_f32_d2();
CellsFn cells_f32_d3();
CellsFn cells_ff_d2();
CellsFn cells_ff_d3();

#define GP_CELLS_CASE(D, A, K) \
  case K: return run_cells<D, K, A>(x, y, ct, m, s, h, wm, ws, add, first, st);
#define GP_CELLS_FN(D, A)                                                                                 \
  return [](int k, const void* x, void* y, const CellTabs& ct, const double* m, const double* s, double h, \
            double wm, double ws, int add, int first, cudaStream_t st) -> cudaError_t {                  \
    switch (k) {                                                                                          \
      GP_CELLS_CASE(D, A, 1) GP_CELLS_CASE(D, A, 2) GP_CELLS_CASE(D, A, 3) GP_CELLS_CASE(D, A, 4)         \
      GP_CELLS_CASE(D, A, 5) GP_CELLS_CASE(D, A, 6) GP_CELLS_CASE(D, A, 7) GP_CELLS_CASE(D, A, 8)         \
      default: return cudaErrorInvalidValue;                                                              \
    }                                                                                                     \
  };

#define GP_DISPATCH_K(D, A, Ar, st)                    \
  switch ((Ar).k) {                                    \
    case 1: return run_apply<D, 1, A>(Ar, st);         \
    case 2: return run_apply<D, 2, A>(Ar, st);         \
    case 3: return run_apply<D, 3, A>(Ar, st);         \
    case 4: return run_apply<D, 4, A>(Ar, st);         \
    case 5: return run_apply<D, 5, A>(Ar, st);         \
    case 6: return run_apply<D, 6, A>(Ar, st);         \
    case 7: return run_apply<D, 7, A>(Ar, st);         \
    case 8: return run_apply<D, 8, A>(Ar, st);         \
    default: return cudaErrorInvalidValue;             \
  }

}  // namespace gp
