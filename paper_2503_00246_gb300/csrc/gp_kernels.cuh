// Face kernels of the ghost-penalty operator y = G x on sm_103a.
//
// Per face F with normal axis a (Sec. 2.4), G_F = h^{d-2} (M^ x ... x G^) with
// G^ = sum_j c_j g_j g_j^T of rank k.  The face kernel computes the face output
//
//   t_F[j, tau] = g_j . x_F(:, tau)                    normal lines (k jump values)
//   T_F[tau, j] = s_j (M^ x M^) t_F[j, .]              tangential reference masses
//   W_F[b, tau] = sum_j g_j[b] T_F[tau, j]             normal expansion
//
// i.e. the three-step face apply of Sec. 2.5.1 with the normal step split in
// two around the tangential masses (G^ has rank k), and stores W_F as [b][tau]
// or, compact, T_F as [tau][j].  The lift kernel then adds, for every touched
// DoF, the W_F entries of the faces that contain it in a fixed order (expanding
// them from T_F in the compact form): a gather, so no atomics and bitwise
// reproducible.  For the overwrite form,
// extra CTAs of the face launch, spread over its grid, write the zeros of the untouched active DoFs.
//
// Template parameter A (gp_arith.cuh) picks the arithmetic: FP32, FP64, or
// float-float on FP64 data.
#pragma once

#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

#include "gp_arith.cuh"

namespace gp {

template <int D, int K>
struct Shape {
  static constexpr int L = (D == 2) ? (K + 1) : (K + 1) * (K + 1);  // tangential nodes per face
  static constexpr int NN = 2 * K + 1;                               // nodes on a normal line
  static constexpr int P = NN * L;                                   // patch nodes per face
  static constexpr int NP = (NN + 3) / 4 * 4;                        // row-start entries per patch column
  static constexpr int FB = (256 / L) > 0 ? (256 / L) : 1;           // default faces per CTA
};

// Tile shape of one (d, k, arithmetic) apply, picked per GPU by the autotuner:
// faces per face CTA (fb * L threads), owner cells per lift CTA and lift threads.
struct Tiles {
  int32_t fb = 0;
  int32_t lcb = 0;
  int32_t lnt = 0;
};

constexpr int MAX_CTA_THREADS = 512;
constexpr size_t MAX_DYN_SMEM = 46 * 1024;   // plus < 2 KB of static shared memory: under the 48 KB default

// dynamic shared memory of the face kernel: the k jump planes of fb faces, twice in 3D (room for
// the padded planes and the second direction's sums, see TanShape); FP32 also stages the patches of
// faces of normal x there (below 36 KB for every CTA of at most MAX_CTA_THREADS lines)
template <int D, int K, typename V>
__host__ __device__ constexpr size_t face_planes(int fb) {
  return (size_t)((D == 3) ? 2 : 1) * fb * K * Shape<D, K>::L * sizeof(V);
}
// (without compact outputs only up to k = 4: with the expansion's registers the staging spills, 128^2 disc at
// k = 5 8.2 / 7.4 us, and in the model system, where the face kernel shares the SMs with the cell kernel, it was
// slower than the plain gather at every size, 28^3 ball at k = 6 31.9 / 29.6 us, 24^3 at k = 8 45.5 / 43.7)
template <typename V, int K, bool COMPACT>
struct StagePatch {
  static constexpr bool value = std::is_same<V, float>::value && (COMPACT || K <= 4);
};
template <int D, int K, typename V>
__host__ __device__ constexpr size_t face_smem(int fb) {
  const size_t stage = StagePatch<V, K, true>::value ? (size_t)fb * Shape<D, K>::P * sizeof(V) : 0;
  const size_t planes = face_planes<D, K, V>(fb);
  // the padded planes and sums in use with the line factors of the triangular basis (FP64) behind them
  constexpr int N = K + 1, LP = (D == 3) ? (N | 1) * N : N;
  const size_t ldl = std::is_same<V, double>::value
                         ? ((size_t)fb * K * (LP + ((D == 3) ? N : 0)) + (size_t)K * Shape<D, K>::L) * sizeof(V) : 0;
  const size_t most = planes > ldl ? planes : ldl;
  return most > stage ? most : stage;
}

// Kernel constants (passed by value; they sit in the constant bank).  In FP64 and float-float
// the per-order factor s_j = c_j h^{d-2} is folded into the jump vectors of the first step
// (gs = s_j g_j), so no line multiplies by s_j; FP32 multiplies each line's k tangential results
// by s_j instead (its face kernel is bound by memory instructions, and a batch then needs no
// per-problem table).
template <typename V>
struct FoldScale {
  static constexpr bool value = !std::is_same<V, float>::value;
};
template <typename V, int K>
struct Consts {
  V g[K][2 * K + 1];   // jump of the j-th derivative of patch basis b (row j-1)
  V gs[K][2 * K + 1];  // s_j g_j[b], the jump vectors of the first step (FP64, float-float)
  V s[K];              // s_j (FP32)
  // reference mass M^ = diag(mw) (I + mc ma^T) (see tangential_mass), and the factors mw of a face's lines (3D: the
  // product of both directions')
  V ma[K + 1];
  V mc[K + 1];
  V w[(K + 1) * (K + 1)];   // 2D: the first K + 1
};

// Fills the lumped form of the reference mass from p = (ma, mc), 2 (k+1) values, and the line factors from
// fac (Plan::fac).
template <int D, int K, typename V>
void mass_consts(const double* p, const double* fac, Consts<V, K>& c) {
  constexpr int N = K + 1;
  for (int i = 0; i < N * N; ++i) c.w[i] = i < Shape<D, K>::L ? from_host<V>(fac[i]) : vzero<V>();
  for (int i = 0; i < N; ++i) {
    c.ma[i] = from_host<V>(p[i]);
    c.mc[i] = from_host<V>(p[N + i]);
  }
}

struct FaceArgs {
  const int32_t* frows;   // per-face row starts of the patch (see rbase)
  const void* fac;        // FP32: mw of a face's L lines; triangular basis: D_j mw, K rows of L (see Plan::fac)
  int64_t rbase[4];       // row entry of face fstart[a] of each axis
  int32_t fstart[4];      // first face of each axis in this launch
  int32_t fend[4];        // one past the last face of each axis in this launch
  const int2* zruns;      // (c0, len <= 256) runs of untouched active DoFs
  int32_t nzruns;         // 0 for the add form
  int32_t nzblocks;       // zero-fill CTAs
  uint64_t zstep;         // shares that spread() takes: zero-fill CTAs of the grid,
  uint64_t xstep, ystep;  // normal-x CTAs of the face CTAs, normal-y CTAs of the others
  int32_t tail_wait;      // 1: before exiting, wait for the grid this launch programmatically
                          // depends on (slab pipeline: so that this grid completes after it)
};

constexpr int ZGROUP = 16;  // zero runs per zero-fill CTA

// The kinds of CTA of a face launch are spread evenly over its grid: CTA i of n, of which m are of a
// kind, is CTA floor(i m / n) of that kind where that count steps at i, and otherwise one of the rest.
// Zero-fill CTAs write to HBM while the face CTAs compute: at the front of the grid they ran alone,
// 382 MB of zeros in an FP64 apply of the 128^3 gyroid (k = 4) with the FP64 pipe idle; spread, with
// the vector stores of zero_fill, that apply went from 1519 to 1450 us, the FP32 one from 261 to
// 240 us, and the FP32 1023^2 disc (k = 4, almost all zeros) from 12.3 to 11.0.
// The faces of each axis follow the lexicographic order of their cells, so that spread axes work on
// one region of the mesh at a time and read its x from HBM once instead of once per axis (face
// kernel of the 128^3 gyroid at k = 4: FP32 132 -> 127 us, float-float 365 -> 355 us).
inline uint64_t spread_step(const int64_t m, const int64_t n) {   // m / n in units of 2^-32, rounded up
  return n > 0 ? (((uint64_t)m << 32) + (uint64_t)n - 1) / (uint64_t)n : 0;
}
// the index of CTA i within its kind, or -1 - (its index among the rest)
__device__ __forceinline__ int spread(const int i, const uint64_t step) {
  const int k0 = (int)(((uint64_t)i * step) >> 32);
  const int k1 = (int)(((uint64_t)(i + 1) * step) >> 32);
  return k1 > k0 ? k0 : -1 - (i - k0);
}
// Fills the shares for fb faces per CTA; returns the CTAs of the launch.
inline int face_grid(FaceArgs& fa, const int dim, const int fb) {
  fa.nzblocks = (fa.nzruns + ZGROUP - 1) / ZGROUP;
  int nb[3] = {0, 0, 0}, faces = 0;
  for (int a = 0; a < dim; ++a) {
    nb[a] = (fa.fend[a] - fa.fstart[a] + fb - 1) / fb;
    faces += nb[a];
  }
  fa.zstep = spread_step(fa.nzblocks, fa.nzblocks + faces);
  fa.xstep = spread_step(nb[0], faces);
  fa.ystep = spread_step(nb[1], faces - nb[0]);
  return fa.nzblocks + faces;
}

// Zeros of the runs [ZGROUP zi, ZGROUP (zi + 1)): a warp per run, 16-byte streaming stores between
// the unaligned ends (the zeros are not read again, so they should not push x out of L2).
template <typename IO>
__device__ __forceinline__ void zero_fill(IO* __restrict__ y, const int2* __restrict__ zruns, const int nzruns,
                                          const int zi) {
  constexpr int VE = 16 / (int)sizeof(IO);
  const int lane = (int)(threadIdx.x & 31u), nt = (int)blockDim.x;
  // threads beyond the last whole warp idle (a CTA of less than a warp is one short warp)
  const int nw = max(nt >> 5, 1), step = min(nt, 32), w = (int)(threadIdx.x >> 5);
  if (w >= nw) return;
  const int r1 = min(ZGROUP * (zi + 1), nzruns);
  for (int r = ZGROUP * zi + w; r < r1; r += nw) {
    const int2 run = __ldg(zruns + r);
    IO* p = y + run.x;
    const int head = min(run.y, (int)(((16u - (unsigned)((uintptr_t)p & 15u)) & 15u) / sizeof(IO)));
    const int nv = (run.y - head) / VE;
    for (int i = lane; i < head; i += step) __stcs(p + i, IO(0));
    int4* v = reinterpret_cast<int4*>(p + head);
    for (int i = lane; i < nv; i += step) __stcs(v + i, make_int4(0, 0, 0, 0));
    for (int i = head + VE * nv + lane; i < run.y; i += step) __stcs(p + i, IO(0));
  }
}

struct LiftArgs {
  const int32_t* lwin;    // [nlift][NW] candidate face ids of each owner cell (-1 if none)
  const int32_t* lrow;    // [nlift][KR] compact index of node (ci k, cj k + q, cl k + r)
  const int32_t* lmask;   // [nlift] which nodes a ghost face reaches (see Plan::lmask)
  int32_t nlift;
  int32_t n_active;
};

// ------------------------------------------------- one normal line's steps --
// The three one-dimensional steps of the face apply for one normal line, shared by the
// face kernel and the brick kernel (gp_brick.cuh).

// Jump values t_j = g_j . v of the line (j = 1..k; row j - 1 of g).  Mirroring the patch
// about the face maps basis b to 2k - b, K- to K+ and d/dn to -d/dn, so
// g_j[2k - b] = (-1)^(j+1) g_j[b]: odd orders see v[b] + v[2k-b], even orders
// v[b] - v[2k-b], and only odd orders see the shared node b = k.
template <int K, typename V>
__device__ __forceinline__ void line_jumps(const V (&v)[2 * K + 1], const V (*g)[2 * K + 1], V (&t)[K]) {
  constexpr int NN = 2 * K + 1;
  V vp[K], vm[K];
#pragma unroll
  for (int b = 0; b < K; ++b) {
    vp[b] = vadd_loose(v[b], v[NN - 1 - b]);
    vm[b] = vsub_loose(v[b], v[NN - 1 - b]);
  }
#pragma unroll
  for (int j = 0; j < K; ++j) {
    const bool odd = (j % 2) == 0;   // order j + 1
    Dot<V> acc = dot_first(g[j][0], odd ? vp[0] : vm[0]);
#pragma unroll
    for (int b = 1; b < K; ++b) dot_fma(acc, g[j][b], odd ? vp[b] : vm[b]);
    if (odd) dot_fma(acc, g[j][K], v[K]);
    t[j] = dot_value(acc);
  }
}

// ------------------------------------------------- triangular normal basis --
// The jump vectors of one parity span the same space as r vectors in echelon form, r = number of
// orders of that parity: G^ = sum_j s_j g_j g_j^T = B diag(D) B^T, row j of B with a 1 at its pivot
// node and 0 at the pivots of the earlier rows of its parity (rows j = 0, 2, .. even in b, 1, 3, ..
// odd).  Those entries cost nothing in the jumps (t_j = B_j . v) or in the expansion: 12 + 12
// multiply-adds per line instead of 18 + 18 at k = 4, 48 + 48 instead of 68 + 68 at k = 8; D_j goes into the line factors mw (Plan::fac, rounded
// once: products of rounded D_j and mw had errors up to 1.25 times those of the jump vectors).  The host eliminates
// in 113-bit arithmetic (Plan::ldl), from the largest direction to the smallest: D is graded and
// non-negative, so x^T G x stays a sum of squares.  The pivot orders are those whose elimination
// grows least (entries below 1.2 for the default and for the factorial weights).  Native FP64 only,
// whose kernel is bound by the FP64 pipe: apply of the 128^3 gyroid at k = 4 1450 -> 1263 us, of the
// 64^3 ball at k = 3 68.9 -> 63.5 us.  Weights below 0 run the jump vectors themselves.
template <int K>
struct Pivots {
  // pivot node of row j in hexadecimal digit j
  static constexpr uint32_t CODE = K == 1 ? 0x1u : K == 2 ? 0x12u : K == 3 ? 0x122u : K == 4 ? 0x3223u :
                                   K == 5 ? 0x54133u : K == 6 ? 0x561244u : K == 7 ? 0x4276245u : 0x66187245u;
  __host__ __device__ static constexpr int at(int j) { return (int)((CODE >> (4 * j)) & 15u); }
  // node b is the pivot of an earlier row of j's parity
  __host__ __device__ static constexpr bool zero(int j, int b) {
    for (int i = j & 1; i < j; i += 2)
      if (at(i) == b) return true;
    return false;
  }
};

// t_j = B_j . v on the folded line (B in rows of g)
template <int K, typename V>
__device__ __forceinline__ void line_jumps_ldl(const V (&v)[2 * K + 1], const V (*g)[2 * K + 1], V (&t)[K]) {
  using P = Pivots<K>;
  constexpr int NN = 2 * K + 1;
  V f[2][K + 1];   // even and odd part; the middle node counts once
#pragma unroll
  for (int b = 0; b < K; ++b) {
    f[0][b] = v[b] + v[NN - 1 - b];
    f[1][b] = v[b] - v[NN - 1 - b];
  }
  f[0][K] = v[K];
#pragma unroll
  for (int j = 0; j < K; ++j) {
    V acc = f[j & 1][P::at(j)];
#pragma unroll
    for (int b = 0; b <= K; ++b)
      if (!((j & 1) && b == K) && b != P::at(j) && !P::zero(j, b)) acc = vfma(g[j][b], f[j & 1][b], acc);
    t[j] = acc;
  }
}

// w[b] = sum_j B_j[b] T[j], with w[b] = E_b + O_b and w[2k - b] = E_b - O_b
template <int K, typename V>
__device__ __forceinline__ void line_expand_ldl(const V (*g)[2 * K + 1], const V (&T)[K], V (&w)[2 * K + 1]) {
  using P = Pivots<K>;
  constexpr int NN = 2 * K + 1;
#pragma unroll
  for (int b = 0; b <= K; ++b) {
    V s[2];
#pragma unroll
    for (int par = 0; par < 2; ++par) {
      bool have = false;
      s[par] = vzero<V>();
#pragma unroll
      for (int j = par; j < K; j += 2) {
        if (P::zero(j, b)) continue;
        if (P::at(j) == b) s[par] = have ? s[par] + T[j] : T[j];
        else s[par] = have ? vfma(g[j][b], T[j], s[par]) : g[j][b] * T[j];
        have = true;
      }
    }
    if (b == K || K == 1) {
      w[b] = s[0];
      if (b < K) w[NN - 1 - b] = s[0];
    } else {
      w[b] = s[0] + s[1];
      w[NN - 1 - b] = s[0] - s[1];
    }
  }
}

// ------------------------------------------------------ tangential masses --
// Gauss-Lobatto quadrature with N = k+1 points is exact up to degree 2k - 1, and the product of
// two nodal polynomials has degree 2k, so the exact mass matrix differs from the lumped one by the
// quadrature error of x^(2k), a rank-one term in the leading coefficients a_i of the l_i:
//   M^ = diag(w) - E a a^T = diag(mw) (I + mc ma^T),   ma = a / max|a|,  mc = -E max|a| a / w
// (k = 1: diag(1/6) (I + 1 1^T), which has no cancellation).  One line costs 2 N multiply-adds
// and the N factors mw, which both directions share as one product per normal line: 2 (d-1) k + k
// multiply-adds per line.  The even / odd halves of M^ took (N^2 / 2 + 2 N) (d-1) k / N, i.e. 20
// against 34 at d = 3, k = 4 and 40 against 101 at k = 8.  Bound by the FP64 pipe: the native
// FP64 apply of the 128^3 gyroid at k = 4 went from 1780 to 1519 us and that of the 64^3 ball at
// k = 3 from 77.2 to 68.7 us; float-float 96^3 ball at k = 5 277 to 270 us; FP32 unchanged.
//
// Shared-memory layout of the tangential pass: a plane of the k jump values of a face's L lines
// (3D: line (t1, t2) at t1 + pitch t2 with an odd pitch, so that walking t1 or t2 in neighbouring
// lanes meets distinct banks; k = 3, 5, 7 had 2- to 8-way conflicts) and in 3D the N sums per
// order of the second direction.  In 3D both fit the two planes that the launch reserves.
template <int D, int K>
struct TanShape {
  static constexpr int N = K + 1;
  static constexpr int PITCH = (D == 3) ? (N | 1) : N;
  static constexpr int LP = (D == 3) ? PITCH * N : N;   // one order of one face
  __host__ __device__ static constexpr int at(int tau) { return (D == 3) ? tau % N + PITCH * (tau / N) : tau; }
};

// mc by tangential index in shared memory (a thread's index is lane-dependent: not for the constant bank)
template <int K, typename V>
__device__ __forceinline__ void fill_mc(V (&mc)[K + 1], const Consts<V, K>& c, const int t) {
  if (t <= K) mc[t] = c.mc[t];
}

// ma . u of one tangential line
template <int K, typename V>
__device__ __forceinline__ V line_dot(const Consts<V, K>& c, const V (&u)[K + 1]) {
  Dot<V> acc = dot_first(c.ma[0], u[0]);
#pragma unroll
  for (int q = 1; q <= K; ++q) dot_fma(acc, c.ma[q], u[q]);
  return dot_value(acc);
}
// u -> (I + mc ma^T) u of the line at p with stride st.  k = 1: (2 u_0 + u_1, u_0 + 2 u_1), one rounding each.  (The
// integer form of k = 2, 1/30 (4 2 -1; 2 16 2; -1 2 4), was no more accurate and in FP64 4 % slower.)
template <int K, typename V>
__device__ __forceinline__ void line_mass(const Consts<V, K>& c, const V (&u)[K + 1], V* p, const int st) {
  if constexpr (K == 1) {
    p[0] = vadd(vscale(u[0], 2.f), u[1]);
    p[st] = vadd(vscale(u[1], 2.f), u[0]);
  } else {
    const V s = line_dot<K, V>(c, u);
#pragma unroll
    for (int q = 0; q <= K; ++q) p[st * q] = vfma(c.mc[q], s, u[q]);
  }
}

// out[j] = ((M^ x M^) u_j)(tau) for the k jump values u_j of every line in `plane`.  A task is one
// (face, order j, tangential line of N values); the tasks of the CTA's fb faces are packed onto its
// first threads.  3D: pass 1 along t2 (neighbouring lanes on neighbouring t1) in place; pass 2
// along t1 only takes the dot product ma . u of each line, and every line's thread adds its own
// mc and multiplies by mw (FP32, bound by shared-memory accesses and not by arithmetic, and k = 1: pass 2 in
// place too, one access less per value).  2D: pass 1 in place.  wl[tau + WS j] is the factor of
// order j and line tau (WS = 0: one for every order; WS < 0: wt, of the thread's line), mc[t] the correction of
// tangential index t, both in shared memory.  Every thread of the CTA calls it (it synchronises, also before its first read:
// the caller has only written plane, wl and mc).
template <int D, int K, typename V, int WS = 0>
__device__ __forceinline__ void tangential_mass(V (*plane)[K][TanShape<D, K>::LP], V (*dots)[K][K + 1], const int fb,
                                                const Consts<V, K>& c, const V* wl, const V* mc, const int fl,
                                                const int tau, V (&out)[K], const V wt = vzero<V>()) {
  using T = TanShape<D, K>;
  constexpr int N = K + 1;
  constexpr int TASKS = (D == 3) ? K * N : K;     // per face and pass
  constexpr int ST = (D == 3) ? T::PITCH : 1;     // stride of pass 1
  constexpr bool DOTS = D == 3 && K > 1 && !std::is_same<V, float>::value;
  const int u = threadIdx.x;
  const bool task = u < fb * TASKS;
  const int tf = u / TASKS, w = u - tf * TASKS;
  const int j = (D == 3) ? w / N : w, tr = (D == 3) ? w % N : 0;
  __syncthreads();
  if (task) {
    V* p = &plane[tf][j][tr];
    V uu[N];
#pragma unroll
    for (int q = 0; q < N; ++q) uu[q] = p[ST * q];
    line_mass<K, V>(c, uu, p, ST);
  }
  __syncthreads();
  if constexpr (D == 3) {
    if (task) {
      V* p = &plane[tf][j][T::PITCH * tr];
      V uu[N];
#pragma unroll
      for (int q = 0; q < N; ++q) uu[q] = p[q];
      if constexpr (DOTS) {
        dots[tf][j][tr] = line_dot<K, V>(c, uu);
      } else {
        line_mass<K, V>(c, uu, p, 1);
      }
    }
    __syncthreads();
  }
  const V f = WS == 0 ? wl[tau] : wt;
  const V ct = DOTS ? mc[tau % N] : vzero<V>();
#pragma unroll
  for (int jj = 0; jj < K; ++jj) {
    V v = plane[fl][jj][T::at(tau)];
    if constexpr (DOTS) v = vfma(ct, dots[fl][jj][tau / N], v);
    out[jj] = vmul(WS > 0 ? wl[WS * jj + tau] : f, v);
  }
}

// Normal expansion w[b] = sum_j g_j[b] sj[j] (sj: the tangential results of the line):
// w[b] = E_b + O_b and w[2k-b] = E_b - O_b, with E_b (O_b) the sum over odd (even) orders of
// g_j[b] sj[j]; w[k] = E_k.
template <int K, typename V>
__device__ __forceinline__ void line_expand(const Consts<V, K>& c, const V (&sj)[K], V (&w)[2 * K + 1]) {
  constexpr int NN = 2 * K + 1;
#pragma unroll
  for (int b = 0; b <= K; ++b) {
    Dot<V> ev = dot_first(c.g[0][b], sj[0]);
#pragma unroll
    for (int j = 2; j < K; j += 2) dot_fma(ev, c.g[j][b], sj[j]);
    if (b == K || K == 1) {
      const V e = dot_value(ev);
      w[b] = e;
      if (b < K) w[NN - 1 - b] = e;
    } else {
      Dot<V> ov = dot_first(c.g[K > 1 ? 1 : 0][b], sj[K > 1 ? 1 : 0]);
#pragma unroll
      for (int j = 3; j < K; j += 2) dot_fma(ov, c.g[j][b], sj[j]);
      w[b] = dot_merge<false>(ev, ov);
      w[NN - 1 - b] = dot_merge<true>(ev, ov);
    }
  }
}

// ------------------------------------------------------- compact face outputs --
// The face kernel stores either the (2k+1) L values W_F[b][tau] of every face or only the k L
// tangential results T_F[tau][j] behind them (k padded to KP for vector accesses), which the lift
// then expands along the normal for k nodes at once (lift_lines_body): 2.25 times fewer bytes at
// k = 4 and one vector access per line instead of 2k + 1.
template <int K, typename V>
struct Compact {
  static_assert(sizeof(V) == 4, "FP32 only (StoreCompact)");
  static constexpr int KP = (K == 3) ? 4 : (K == 5) ? 6 : (K == 7) ? 8 : K;
  static constexpr int VW = KP % 4 == 0 ? 4 : 2;   // values per access
  static_assert(KP % VW == 0, "whole accesses");
  static_assert(KP <= 2 * K + 1, "compact outputs must fit the face-output buffer");
};
template <int VW, typename V>
struct alignas(VW * sizeof(V)) Chunk {
  V v[VW];
};
// FP32 stores T_F where W_F would not stay in L2 (store_compact): both of its kernels were bound by L1
// wavefronts (68% and 65% of their peak) and moved 1.11 GB per apply of the 128^3 gyroid at k = 4, 0.79 GB
// so: apply 306 -> 261 us (face kernel 187 -> 158 us, lift 117 -> 104 us).  FP64 stores W_F: the
// expansion and its FP64 adds cost the same operations either way, and W_F hides under the FP64 pipe;
// so does float-float (a lift of compact outputs took 385 us there against 283 us).
// value: some meshes of this dimension and degree store T_F; always: all do (store_compact has the sizes).
template <int D, int K, typename V>
struct StoreCompact {
  static constexpr bool value = std::is_same<V, float>::value && (D == 2 ? K >= 6 : K >= 3);
  static constexpr bool always = value && (D == 2 || K == 5 || K >= 7);
};

// ----------------------------------------------------------------- face --
// One thread per (face, normal line tau); fb faces per CTA (blockDim.x = fb L).
// `blk` is the CTA's index within its problem; `gs` holds the jump vectors of the first step
// (FP64, float-float: the scaled s_j g_j, c.gs or a batch segment's copy in shared memory;
// FP32: the plain c.g) and `sc` the k factors s_j (FP32 only); `dsm` is the
// face_smem<D, K, V>(fb) bytes of dynamic shared memory.  COMPACT: store T_F instead of W_F.  LDL: gs
// holds the rows of B.
template <int D, int K, class A, bool COMPACT, bool LDL>
__device__ __forceinline__ void face_body(const typename A::IO* __restrict__ x, typename A::V* __restrict__ wp,
                                          typename A::IO* __restrict__ y, const FaceArgs& fa,
                                          const Consts<typename A::V, K>& c, const typename A::V (*gs)[2 * K + 1],
                                          const typename A::V* sc, const int blk, const int fb, unsigned char* dsm) {
  using S = Shape<D, K>;
  using V = typename A::V;
  using IO = typename A::IO;
  constexpr int L = S::L, NN = S::NN, K1 = K + 1;
  using T = TanShape<D, K>;
  typedef V Plane[K][T::LP];
  typedef V Dots[K][K1];
  Plane* buf = reinterpret_cast<Plane*>(dsm);            // [fb][K][LP]
  Dots* dots = reinterpret_cast<Dots*>(buf + fb);         // [fb][K][N], 3D only
  __shared__ V mc[K1];
  // The lines' factors.  FP32: loaded into the thread of the line, to be used behind three barriers; the triangular
  // basis: D_j mw [K][L] behind the planes, copied there while the gather runs; else mw [L] from the constant bank.
  // (FP32 from the constant bank, 25 to 81 values for each warp in turn: 128^3 gyroid at k = 4 229.9 / 227.1 us, 49^3
  // ball at k = 8 85.3 / 83.7; float-float in registers: 50^3 ball at k = 6 123.8 / 119.7.)
  constexpr bool REG = std::is_same<V, float>::value;
  __shared__ V tw[LDL || REG ? 1 : L];
  V* wl = LDL ? reinterpret_cast<V*>(dots + ((D == 3) ? fb : 0)) : tw;
  const int nt = (int)blockDim.x;
  // the lift may start its prologue as soon as every face CTA is running (programmatic
  // dependent launch; it waits for this grid's completion before it reads W)
  asm volatile("griddepcontrol.launch_dependents;");

  const int zb = spread(blk, fa.zstep);
  if (zb >= 0) {
    // zero fill of the active DoFs outside every face patch (overwrite form only)
    zero_fill(y, fa.zruns, fa.nzruns, zb);
    return;
  }
  // axis of this CTA's faces (constant indices only: no local-memory copy of fa)
  int axis = 0, fbase = fa.fstart[0], fend = fa.fend[0], ib = spread(-1 - zb, fa.xstep);
  int64_t rbase = fa.rbase[0];
  if (ib < 0) {
    ib = spread(-1 - ib, fa.ystep);
    axis = 1; fbase = fa.fstart[1]; fend = fa.fend[1]; rbase = fa.rbase[1];
    if (D == 3 && ib < 0) {
      ib = -1 - ib;
      axis = 2; fbase = fa.fstart[2]; fend = fa.fend[2]; rbase = fa.rbase[2];
    }
  }
  const int f0 = fbase + ib * fb;
  const int t = threadIdx.x;
  const int fl = t / L, tau = t - fl * L;
  const int f = f0 + fl;
  const bool valid = f < fend;
  if constexpr (LDL) {
    for (int i = t; i < K * L; i += nt)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(wl + i)),
                   "l"(static_cast<const V*>(fa.fac) + i) : "memory");
  } else if (!REG && t < L) {
    wl[t] = c.w[t];
  }
  fill_mc<K, V>(mc, c, t);
  // ---- gather this thread's normal line (2k+1 values)
  V v[NN];
  if (StagePatch<V, K, COMPACT>::value && axis == 0) {
    // Normal x: a line is 2k+1 consecutive values, and a lane per line would touch a cache line per
    // lane in each of its 2k+1 loads (FP32's kernel is bound by L1 wavefronts).  The CTA loads the
    // patches value by value, lanes along the lines, and passes them on through shared memory (an
    // odd pitch of 2k+1: no bank conflicts).  128^3 gyroid, k = 4: face kernel 132.5 -> 127 us.
    if constexpr (StagePatch<V, K, COMPACT>::value) {
      V* st = reinterpret_cast<V*>(dsm);
      const int32_t* rows = fa.frows + rbase + (int64_t)(f0 - fbase) * L;
      const int items = min(fb, fend - f0) * S::P;
      int32_t at[NN];
#pragma unroll
      for (int u = 0; u < NN; ++u) {
        const int i = t + u * nt;
        const int line = i / NN;
        at[u] = i < items ? __ldg(rows + line) + (i - line * NN) : -1;
      }
#pragma unroll
      for (int u = 0; u < NN; ++u)
        if (at[u] >= 0) st[t + u * nt] = __ldg(x + at[u]);
      __syncthreads();
#pragma unroll
      for (int b = 0; b < NN; ++b) v[b] = valid ? st[t * NN + b] : vzero<V>();
      __syncthreads();
    }
  } else if (valid) {
    if (!StagePatch<V, K, COMPACT>::value && axis == 0) {
      const int32_t base = __ldg(fa.frows + rbase + (int64_t)(f - fbase) * L + tau);
#pragma unroll
      for (int b = 0; b < NN; ++b) v[b] = from_io(__ldg(x + base + b), (V*)nullptr);
    } else {
      // tau = tx + (K+1) tr; row b of the patch at outer tangential index tr, four starts per load
      // (one load per start: float-float apply of the 128^3 gyroid at k = 4 713 us, so 666 us)
      constexpr int NP = S::NP, R = (D == 3) ? NP * K1 : NP;
      const int tx = (D == 3) ? tau % K1 : tau;
      const int tr = (D == 3) ? tau / K1 : 0;
      const int4* rows = reinterpret_cast<const int4*>(fa.frows + rbase + (int64_t)(f - fbase) * R + NP * tr);
      int32_t at[NP];
#pragma unroll
      for (int u = 0; u < NP / 4; ++u) {
        const int4 r4 = __ldg(rows + u);
        at[4 * u] = r4.x;
        at[4 * u + 1] = r4.y;
        at[4 * u + 2] = r4.z;
        at[4 * u + 3] = r4.w;
      }
#pragma unroll
      for (int b = 0; b < NN; ++b) v[b] = from_io(__ldg(x + at[b] + tx), (V*)nullptr);
    }
  } else {
#pragma unroll
    for (int b = 0; b < NN; ++b) v[b] = vzero<V>();
  }
  if constexpr (LDL) asm volatile("cp.async.wait_all;" ::: "memory");
  // ---- contract with the k jump vectors, then the tangential reference masses
  {
    V t[K];
    if constexpr (LDL) line_jumps_ldl<K, V>(v, gs, t);
    else line_jumps<K, V>(v, gs, t);
#pragma unroll
    for (int j = 0; j < K; ++j) buf[fl][j][T::at(tau)] = t[j];
  }
  V out[K];
  tangential_mass<D, K, V, LDL ? L : REG ? -1 : 0>(buf, dots, fb, c, wl, mc, fl, tau, out,
                                                   REG ? static_cast<const V*>(fa.fac)[tau] : vzero<V>());

  if (!valid) return;
  if constexpr (!FoldScale<V>::value) {
#pragma unroll
    for (int j = 0; j < K; ++j) out[j] = vmul(sc[j], out[j]);
  }
  if constexpr (COMPACT) {
    using CP = Compact<K, V>;
    using Ch = Chunk<CP::VW, V>;
    Ch* dst = reinterpret_cast<Ch*>(wp + ((size_t)f * L + tau) * CP::KP);
#pragma unroll
    for (int i = 0; i < CP::KP / CP::VW; ++i) {
      Ch ch;
#pragma unroll
      for (int e = 0; e < CP::VW; ++e) {
        const int j = i * CP::VW + e;
        ch.v[e] = j < K ? out[j < K ? j : 0] : vzero<V>();
      }
      dst[i] = ch;
    }
  } else {
    // ---- normal expansion W_F[b, tau] = sum_j g_j[b] s_j out[j], stored at tau + L b (the
    // lanes of a face store neighbouring values)
    V* dst = wp + (size_t)f * S::P + tau;
    V w[NN];
    if constexpr (LDL) line_expand_ldl<K, V>(gs, out, w);
    else line_expand<K, V>(c, out, w);
#pragma unroll
    for (int bb = 0; bb < NN; ++bb) dst[L * bb] = w[bb];
  }
}

extern __shared__ __align__(16) unsigned char gp_dyn_smem[];

// resident CTAs of MAX_CTA_THREADS threads to compile for: FP32 is held to 32 registers, every warp
// slot of the SM (128^3 gyroid, k = 4, with 38 registers: 154 against 135 us; the compiler's choice at other degrees:
// applies of the 80^3 ball at k = 5 66.9 / 65.7 us, of the 600^2 disc at k = 7 12.1 / 11.0 us); 0: that choice
template <typename V, int K>
struct FaceCtas {
  static constexpr int value = std::is_same<V, float>::value || (std::is_same<V, ff64>::value && K == 4) ? 4 : 0;
};

template <int D, int K, class A, bool COMPACT, bool LDL>
__global__ void __launch_bounds__(MAX_CTA_THREADS, FaceCtas<typename A::V, K>::value)
face_kernel(const typename A::IO* __restrict__ x, typename A::V* __restrict__ wp,
            typename A::IO* __restrict__ y, const FaceArgs fa, const int fb,
            const __grid_constant__ Consts<typename A::V, K> c) {
  face_body<D, K, A, COMPACT, LDL>(x, wp, y, fa, c, (FoldScale<typename A::V>::value && !LDL) ? c.gs : c.g, c.s, blockIdx.x,
                                   fb, gp_dyn_smem);
  if (fa.tail_wait) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// --------------------------------------------------------------- batches --
// A batch segment is one (problem, right-hand side) pair of a group of problems
// with the same dimension, degree and arithmetic.  Its x and y pointers live in
// a separate table the host rewrites for every apply.
template <typename V, int K>
struct FaceSeg {
  FaceArgs fa;
  V* wp;           // this segment's face outputs
  const V* gs;     // FP64, float-float: K x (2K+1) scaled jump vectors s_j g_j of the problem, or the rows
                   // of its triangular basis B
  V s[K];          // FP32: s_j of the problem
  int32_t block0;  // first CTA of the segment in the group's face launch
};

struct LiftSeg {
  LiftArgs la;
  int32_t block0;  // first CTA of the segment in the group's lift launch
};

template <typename IO>
struct SegPtrs {
  const IO* x;
  IO* y;
};

// index of the segment holding CTA `blk`: the last segment whose block0 <= blk
template <typename Seg>
__device__ __forceinline__ int find_segment(const Seg* segs, const int nseg, const int blk) {
  int lo = 0, hi = nseg - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(&segs[mid].block0) <= blk) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Every segment of FP64 and float-float brings its jump vectors or its basis B (shared memory), so that
// problems of any weights share one launch: 64 FP64 balls, 24^3, k = 3, with 1, 16 or 64 sets of weights 421 us;
// with B in the constant bank and a launch per set 434, 835 and 2351 us.
template <int D, int K, class A, bool COMPACT, bool LDL>
__global__ void __launch_bounds__(MAX_CTA_THREADS, FaceCtas<typename A::V, K>::value)
face_kernel_batched(const FaceSeg<typename A::V, K>* __restrict__ segs, const int nseg,
                    const SegPtrs<typename A::IO>* __restrict__ ptrs, const int fb,
                    const __grid_constant__ Consts<typename A::V, K> c) {
  using V = typename A::V;
  __shared__ FaceSeg<V, K> seg;
  __shared__ SegPtrs<typename A::IO> sp;
  if (threadIdx.x == 0) {
    const int s = find_segment(segs, nseg, (int)blockIdx.x);
    seg = segs[s];
    sp = ptrs[s];
  }
  __syncthreads();
  if constexpr (FoldScale<V>::value) {
    __shared__ V sg[K][2 * K + 1];
    for (int i = threadIdx.x; i < K * (2 * K + 1); i += blockDim.x) sg[i / (2 * K + 1)][i % (2 * K + 1)] = seg.gs[i];
    __syncthreads();
    face_body<D, K, A, COMPACT, LDL>(sp.x, seg.wp, sp.y, seg.fa, c, sg, seg.s, (int)blockIdx.x - seg.block0, fb, gp_dyn_smem);
  } else {
    face_body<D, K, A, COMPACT, false>(sp.x, seg.wp, sp.y, seg.fa, c, c.g, seg.s, (int)blockIdx.x - seg.block0, fb, gp_dyn_smem);
  }
}

// ----------------------------------------------------------------- lift --
// Owner cell c = (ci, cj, cl) holds the lattice nodes (ci k + p, cj k + q, cl k + r),
// p, q, r in [0, k).  The faces with normal a whose patch holds such a node have
// lower cell c + (s_a - 2) e_a + (s_1 - 1) e_t1 + (s_2 - 1) e_t2 with s_a in {0,1,2}
// (0 only when p_a = 0) and s_t in {0,1} (0 only when p_t = 0); the node sits at
// normal index b = p_a + (2 - s_a) k and tangential index tau_t = p_t + (1 - s_t) k.
//
// One thread takes one x-row (q, r) of an owner cell: its k nodes p = 0..k-1 are
// contiguous in y.  Face outputs are stored as W_F[b][tau] (tau + L b, x the fastest
// tangential index), so the row's nodes read entries L apart in a face of normal x and
// contiguous entries in the other faces.  The row type
// (q == 0, r == 0) fixes at compile time which of the 36 candidate faces can reach
// the row (p = 0 is the only node on the lower x face).  Each node sums its
// contributions in the fixed order (axis, s_a, s_1, s_2): bitwise reproducible.
template <int D, int K>
struct LiftShape {
  static constexpr int KR = (D == 3) ? K * K : K;   // x-rows per owner cell
  static constexpr int CB0 = 256 / KR;
  static constexpr int CB = CB0 < 1 ? 1 : CB0;      // default owner cells per CTA
  static constexpr int NT = 256;                    // default threads per CTA
  static constexpr int NW = (D == 3) ? 36 : 12;     // candidate faces per cell
  static constexpr int NTYPE = (D == 3) ? 4 : 2;
  // rows of type m (bit 0: q == 0, bit 1: r == 0)
  __host__ __device__ static constexpr int count(int m) {
    int c = 1;
    for (int i = 0; i < D - 1; ++i)
      if (!((m >> i) & 1)) c *= (K - 1);
    return c;
  }
};

// Native FP64: the adds of a missing face are skipped (FP64 issue is the scarce
// resource on GB300; the host groups owner cells with the same candidate-face
// pattern so that the skips are warp-uniform).  FP32 and float-float: branch-free
// (a missing face reads face 0 and adds zeros), with the loads of each (axis, s_a)
// group of up to four faces issued before their adds, so they are in flight together.
// Either way each node adds its contributions in the order (axis, s_a, s_1, s_2).
template <int D, int K, class A, int M>
__device__ __forceinline__ void lift_row(const typename A::V* __restrict__ wp, const int* win, const int q,
                                         const int r, Sum<typename A::V> (&acc)[K], unsigned& found) {
  using V = typename A::V;
  constexpr int K1 = K + 1;
  constexpr int P = Shape<D, K>::P, L = Shape<D, K>::L;
  constexpr bool SKIP = std::is_same<V, double>::value;
  constexpr bool QZ = (M & 1) != 0;   // q == 0
  constexpr bool RZ = (M & 2) != 0;   // r == 0 (3D)
  constexpr unsigned ALL = (1u << K) - 1u;
  // patch position of node p = 0 of this row in the face (a, s_a, s_1, s_2), and how
  // many of the row's k nodes that face reaches
  auto where = [&](const int a, const int sa, const int s1, const int s2, int& cnt) -> int {
    if (a == 0) {             // b = p + (2 - s_a) k on the x-line (q', r') of the face (stride L)
      cnt = (sa == 0) ? 1 : K;
      const int tq = q + (1 - s1) * K;
      const int tr = (D == 3) ? r + (1 - s2) * K : 0;
      return (2 - sa) * K * L + (tq + K1 * tr);
    }
    cnt = (s1 == 0) ? 1 : K;
    if (a == 1) {             // x index p + (1 - s1) k, z index r + (1 - s2) k, b = q + (2 - s_a) k
      const int bb = q + (2 - sa) * K;
      const int tz = (D == 3) ? r + (1 - s2) * K : 0;
      return (1 - s1) * K + K1 * tz + L * bb;
    }
    const int ty = q + (1 - s2) * K;   // normal z: x index p + (1 - s1) k, y index q + (1 - s2) k
    const int bb = r + (2 - sa) * K;
    return (1 - s1) * K + K1 * ty + L * bb;
  };
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const int ps = (a == 0) ? L : 1;   // patch stride between the row's nodes
    // zero-ness of the normal coordinate and of the two tangential coordinates
    const bool nz = (a == 0) ? true : ((a == 1) ? QZ : RZ);
    const bool xz = (a == 0) ? QZ : true;         // first tangential: y (a = 0) or x
    const bool yz = (a == 0) ? RZ : ((a == 1) ? RZ : QZ);
#pragma unroll
    for (int sa = 0; sa < 3; ++sa) {
      if (a != 0 && sa == 0 && !nz) continue;
      if constexpr (SKIP) {
        // native FP64: skip the adds of a missing face (warp-uniform by the host's cell order)
#pragma unroll
        for (int s1 = 0; s1 < 2; ++s1) {
          if (s1 == 0 && !xz) continue;
#pragma unroll
          for (int s2 = 0; s2 < ((D == 3) ? 2 : 1); ++s2) {
            if (D == 3 && s2 == 0 && !yz) continue;
            const int f = win[(D == 3) ? a * 12 + sa * 4 + s1 * 2 + s2 : a * 6 + sa * 2 + s1];
            if (f < 0) continue;
            int cnt;
            const int pos = where(a, sa, s1, s2, cnt);
            const V* src = wp + (size_t)f * P + pos;
            // the first contribution of a node sets its sum (no add with zero)
#pragma unroll
            for (int p = 0; p < K; ++p)
              if (p < cnt) {
                if ((found >> p) & 1u) sum_add(acc[p], src[p * ps]);
                else sum_set(acc[p], src[p * ps]);
              }
            found |= (cnt == 1) ? 1u : ALL;
          }
        }
      } else {
        // FP32 and float-float: branch-free.  All loads of the (up to 4) faces of this
        // (a, s_a) are issued before their adds; a missing face reads face 0 and adds 0.
        V ld[4 * K];
        int n = 0;
#pragma unroll
        for (int s1 = 0; s1 < 2; ++s1) {
          if (s1 == 0 && !xz) continue;
#pragma unroll
          for (int s2 = 0; s2 < ((D == 3) ? 2 : 1); ++s2) {
            if (D == 3 && s2 == 0 && !yz) continue;
            const int f = win[(D == 3) ? a * 12 + sa * 4 + s1 * 2 + s2 : a * 6 + sa * 2 + s1];
            const bool ok = f >= 0;
            int cnt;
            const int pos = where(a, sa, s1, s2, cnt);
            const V* src = wp + (size_t)(ok ? f : 0) * P + (ok ? pos : 0);
#pragma unroll
            for (int p = 0; p < K; ++p)
              if (p < cnt) {
                const V v = src[p * ps];
                ld[n++] = ok ? v : vzero<V>();
              }
            if (ok) found |= (cnt == 1) ? 1u : ALL;
          }
        }
        n = 0;
#pragma unroll
        for (int s1 = 0; s1 < 2; ++s1) {
          if (s1 == 0 && !xz) continue;
#pragma unroll
          for (int s2 = 0; s2 < ((D == 3) ? 2 : 1); ++s2) {
            if (D == 3 && s2 == 0 && !yz) continue;
            const int cnt = (a == 0) ? ((sa == 0) ? 1 : K) : ((s1 == 0) ? 1 : K);
#pragma unroll
            for (int p = 0; p < K; ++p)
              if (p < cnt) sum_add(acc[p], ld[n++]);
          }
        }
      }
    }
  }
}

// dynamic shared memory of the lift kernel: the candidate windows of cb cells
template <int D, int K>
__host__ __device__ constexpr size_t lift_smem(int cb) {
  return (size_t)cb * (LiftShape<D, K>::NW + 1) * sizeof(int);
}

// cb owner cells per CTA; each of the blockDim.x threads takes the items g, g + nt, ...
// of the cb * KR rows.
template <int D, int K, class A>
__device__ __forceinline__ void lift_body(const typename A::V* __restrict__ wp, typename A::IO* __restrict__ y,
                                          const int add, const LiftArgs& la, const int blk, const int cb,
                                          unsigned char* dsm) {
  using S = LiftShape<D, K>;
  using V = typename A::V;
  using IO = typename A::IO;
  constexpr int NW = S::NW;
  typedef int Win[NW + 1];
  Win* win = reinterpret_cast<Win*>(dsm);                // [cb][NW + 1]
  const int cell0 = blk * cb;
  const int t = threadIdx.x, nt = (int)blockDim.x;
  for (int idx = t; idx < NW * cb; idx += nt) {
    const int ln = idx / NW, w = idx - ln * NW;
    win[ln][w] = (cell0 + ln < la.nlift) ? __ldg(la.lwin + (size_t)cell0 * NW + idx) : -1;
  }
  __syncthreads();
  // wait for the face kernel (a no-op unless launched as its programmatic dependent), and
  // let a programmatic dependent of this grid start (the cell operator of the model system)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  // one pass: item -> (row type m, cell, row of that type); items sorted by type
  const int E1 = cb * S::count(0);
  const int E2 = E1 + cb * S::count(1);
  const int E3 = E2 + cb * S::count(2);
  const int ITEMS = cb * S::KR;
  for (int g = t; g < ITEMS; g += nt) {
    int m, local;
    if (g < E1) { m = 0; local = g; }
    else if (g < E2 || S::NTYPE == 2) { m = 1; local = g - E1; }
    else if (g < E3) { m = 2; local = g - E2; }
    else { m = 3; local = g - E3; }
    const int cnt = S::count(m);
    const int ci = local / cnt;
    int rem = local - ci * cnt;
    const int cell = cell0 + ci;
    if (cell >= la.nlift) continue;
    int q = 0, r = 0;
    if constexpr (K > 1) {
      if (!(m & 1)) { q = 1 + rem % (K - 1); rem /= (K - 1); }
      if (D == 3 && !(m & 2)) { r = 1 + rem % (K - 1); }
    }
    const int row = q + (D == 3 ? K * r : 0);
    const int base = __ldg(la.lrow + (size_t)cell * S::KR + row);
    Sum<V> acc[K];
#pragma unroll
    for (int p = 0; p < K; ++p) acc[p] = sum_zero<V>();
    unsigned found = 0;
    switch (m) {
      case 0: lift_row<D, K, A, 0>(wp, win[ci], q, r, acc, found); break;
      case 1: lift_row<D, K, A, 1>(wp, win[ci], q, r, acc, found); break;
      case 2: lift_row<D, K, A, 2>(wp, win[ci], q, r, acc, found); break;
      default: lift_row<D, K, A, 3>(wp, win[ci], q, r, acc, found); break;
    }
    if (base < 0) continue;
#pragma unroll
    for (int p = 0; p < K; ++p) {
      if (!((found >> p) & 1u)) continue;
      const int idx = base + p;
      if (idx >= la.n_active) continue;
      const V sv = dot_value(acc[p]);
      const V outv = add ? vadd(from_io(y[idx], (V*)nullptr), sv) : sv;
      y[idx] = to_io(outv, (IO*)nullptr);
    }
  }
}

// ------------------------------------------------------- lift of compact outputs --
// With T_F stored, a node needs sum_j g_j[b] T_F[tau][j] of every face that holds it: k values per
// contribution, unless the k nodes of a normal line share them.  So the lift walks the owner cell's
// lines along each axis in turn: phase a gives every line (p_t1, p_t2) along a to one thread, which
// adds the T_F of the faces that share the line (up to four where p_t1 or p_t2 is 0), for the owner
// as K- (s_a = 2, b = p), K+ (s_a = 1, b = p + k) and end node (s_a = 0, b = 2k, p = 0 only), and
// expands them onto its k nodes.  The nodes' sums pass from phase to phase through shared memory;
// the last phase writes y with x-contiguous lanes.  One vector load (k = 4: 16 bytes per lane, the
// lanes of a face contiguous) replaces k loads of W_F.  Each node sums its contributions in one
// fixed order, whatever the tile shape.
template <int D, int K>
struct LineShape {
  static constexpr int KR = LiftShape<D, K>::KR;            // lines per owner and axis
  // node (p, q, r) at p + K q + PZ r: a padded plane stride keeps the lanes of a y line apart
  static constexpr int PZ = K * K + (K % 2 == 0 ? K : 0);
  static constexpr int OS = (D == 3) ? PZ * K : K * K;      // nodes' sums per owner
  // resident CTAs of 512 threads to compile for: k = 4 is held to 32 registers (0: the compiler's
  // own choice, 40 to 64 registers; holding those too makes it spill)
  static constexpr int CTAS = (K == 4) ? 4 : 0;
};
template <int D, int K, typename V>
__host__ __device__ constexpr size_t lift_lines_smem(int cb) {
  return (size_t)cb * (LiftShape<D, K>::NW + LineShape<D, K>::KR + 1) * sizeof(int) +
         (size_t)cb * LineShape<D, K>::OS * sizeof(Sum<V>);
}
// Owner cells per CTA that fit the dynamic shared memory (a tile may ask for more).
template <int D, int K, typename V>
constexpr int lift_lines_cells(int cb) {
  constexpr size_t per = (LiftShape<D, K>::NW + LineShape<D, K>::KR + 1) * sizeof(int) +
                         LineShape<D, K>::OS * sizeof(Sum<V>);
  constexpr int most = (int)(MAX_DYN_SMEM / per);
  return cb < most ? cb : most;
}

// acc[p] += the faces of normal AX on a line of an owner cell.  The line's type M (bit 0: t1 == 0,
// bit 1: t2 == 0; 3D) fixes at compile time which of the up to four candidate faces per s_a can
// share it.  `line` points at the T_F of tangential index (t1, t2) of face 0.
template <int D, int K, typename V, int AX, int M>
__device__ __forceinline__ void lift_line(const V* __restrict__ line, const int* win, const Consts<V, K>& c,
                                          Sum<V> (&acc)[K]) {
  using CP = Compact<K, V>;
  using Ch = Chunk<CP::VW, V>;
  constexpr int K1 = K + 1, L = Shape<D, K>::L, NS = (D == 3) ? 4 : 2, NCH = (K + CP::VW - 1) / CP::VW;
  // the sums over the faces that share the line, for the owner as K- (s_a = 2), K+ and end node.
  // AHEAD: every load before the first use of one (96^3 ball at k = 5: 52.6 -> 49.4 us); for small
  // k the registers of that cost more resident warps than it gains (k = 4: 104 against 108 us, with
  // the kernel held to 32 registers).
  constexpr bool AHEAD = K >= 5;
  V s[3][K];
  bool any[3] = {false, false, false};
  auto expand = [&](const int sa) {
    if (!any[sa]) return;
#pragma unroll
    for (int p = 0; p < (sa == 0 ? 1 : K); ++p) {
      // each expansion is summed before it joins the node's sum: added term by term it rounded at the
      // size of that sum (error against 64 bits, k = 5, 7, 8: 1.16 to 1.21 times that of the lift of W_F, 0.91 to
      // 0.95 so, at the same speed)
      V w = vmul(c.g[0][p + (2 - sa) * K], s[sa][0]);
#pragma unroll
      for (int j = 1; j < K; ++j) w = vfma(c.g[j][p + (2 - sa) * K], s[sa][j], w);
      sum_add(acc[p], w);
    }
  };
#pragma unroll
  for (int sa = 2; sa >= 0; --sa) {
    // the window's order (s_1, s_2): (0,0) (0,1) (1,0) (1,1); 2D: s_1 = 0, 1
    any[sa] = false;
#pragma unroll
    for (int u = NS - 1; u >= 0; --u) {
      const int s1 = (D == 3) ? u >> 1 : u, s2 = (D == 3) ? u & 1 : 1;
      if ((s1 == 0 && !(M & 1)) || (s2 == 0 && !(M & 2))) continue;
      const int f = win[AX * 3 * NS + sa * NS + u];
      const bool ok = f >= 0;
      any[sa] = any[sa] || ok;
      const Ch* src = reinterpret_cast<const Ch*>(line + (int64_t)f * (L * CP::KP) +
                                                  ((1 - s1) * K + (1 - s2) * K * K1) * CP::KP);
      Ch ch[NCH];
#pragma unroll
      for (int i = 0; i < NCH; ++i) {
#pragma unroll
        for (int e = 0; e < CP::VW; ++e) ch[i].v[e] = vzero<V>();
        if (ok) ch[i] = src[i];
      }
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const V v = ch[j / CP::VW].v[j % CP::VW];
        s[sa][j] = (u == NS - 1) ? v : vadd(s[sa][j], v);
      }
    }
    if constexpr (!AHEAD) expand(sa);
  }
  if constexpr (AHEAD) {
#pragma unroll
    for (int sa = 2; sa >= 0; --sa) expand(sa);
  }
}

// Walks the lines of type M along AX of the CTA's nc owner cells, from item g (the nc count(M) items
// of the type start at `first`) in steps of blockDim.x.  The nodes' sums are read from acc (unless
// AX == 0, the first phase) and written back, or handed to out(ci, t1, t2, sums) in the last phase.
template <int D, int K, class A, int AX, int M, class Out>
__device__ __forceinline__ void lift_lines(int& g, const int first, const typename A::V* __restrict__ tp, const int* win,
                                           const Consts<typename A::V, K>& c, Sum<typename A::V>* acc, const int nc,
                                           Out out) {
  using S = LiftShape<D, K>;
  using LS = LineShape<D, K>;
  using V = typename A::V;
  constexpr int PZ = LS::PZ, KP = Compact<K, V>::KP, CNT = S::count(M);
  // strides of the sums along the line and along its two tangential axes
  constexpr int ST = (AX == 0) ? 1 : (AX == 1) ? K : PZ;
  constexpr int S1 = (AX == 0) ? K : 1, S2 = (AX == 2) ? K : PZ;
  if constexpr (CNT > 0) {
    for (; g < first + nc * CNT; g += (int)blockDim.x) {
      const unsigned local = (unsigned)(g - first);
      const int ci = (int)(local / CNT);
      const unsigned rem = local - (unsigned)ci * CNT;
      constexpr unsigned K0 = K > 1 ? K - 1 : 1;
      const int t1 = (M & 1) ? 0 : 1 + (int)(rem % K0);
      const int t2 = (D == 2 || (M & 2)) ? 0 : 1 + (int)((M & 1) ? rem : rem / K0);
      Sum<V>* a = acc + ci * LS::OS + S1 * t1 + ((D == 3) ? S2 * t2 : 0);
      Sum<V> s[K];
#pragma unroll
      for (int p = 0; p < K; ++p) s[p] = (AX == 0) ? sum_zero<V>() : a[p * ST];
      lift_line<D, K, V, AX, M>(tp + (t1 + ((D == 3) ? (K + 1) * t2 : 0)) * KP, win + ci * S::NW, c, s);
      if constexpr (AX == D - 1) {
        out(ci, t1, t2, s);
      } else {
#pragma unroll
        for (int p = 0; p < K; ++p) a[p * ST] = s[p];
      }
    }
  }
}

// One phase: the lines along AX ordered by type, so that a warp's lanes mostly take one path (whole
// owners per warp, with the warp's own barriers, took 125 us against 104: each warp ran every path).
template <int D, int K, class A, int AX, class Out>
__device__ __forceinline__ void lift_phase(const typename A::V* __restrict__ tp, const int* win,
                                           const Consts<typename A::V, K>& c, Sum<typename A::V>* acc, const int nc,
                                           Out out) {
  using S = LiftShape<D, K>;
  int g = (int)threadIdx.x, first = 0;
  lift_lines<D, K, A, AX, 0>(g, first, tp, win, c, acc, nc, out);
  first += nc * S::count(0);
  lift_lines<D, K, A, AX, 1>(g, first, tp, win, c, acc, nc, out);
  if constexpr (D == 3) {
    first += nc * S::count(1);
    lift_lines<D, K, A, AX, 2>(g, first, tp, win, c, acc, nc, out);
    first += nc * S::count(2);
    lift_lines<D, K, A, AX, 3>(g, first, tp, win, c, acc, nc, out);
  }
}

template <int D, int K, class A>
__device__ __forceinline__ void lift_lines_body(const typename A::V* __restrict__ tp, typename A::IO* __restrict__ y,
                                                const int add, const LiftArgs& la, const Consts<typename A::V, K>& c,
                                                const int blk, const int cb, unsigned char* dsm) {
  using LS = LineShape<D, K>;
  using V = typename A::V;
  using IO = typename A::IO;
  constexpr int NW = LiftShape<D, K>::NW, KR = LS::KR, OS = LS::OS;
  Sum<V>* acc = reinterpret_cast<Sum<V>*>(dsm);                     // [cb][OS]
  int* win = reinterpret_cast<int*>(dsm + (size_t)cb * OS * sizeof(Sum<V>));   // [cb][NW]
  int* row = win + cb * NW;                                         // [cb][KR]
  int* mask = row + cb * KR;                                        // [cb]
  const int cell0 = blk * cb;
  const int nc = min(cb, la.nlift - cell0);
  const int t = threadIdx.x, nt = (int)blockDim.x;
  for (int i = t; i < nc * NW; i += nt) win[i] = __ldg(la.lwin + (size_t)cell0 * NW + i);
  for (int i = t; i < nc * KR; i += nt) row[i] = __ldg(la.lrow + (size_t)cell0 * KR + i);
  for (int i = t; i < nc; i += nt) mask[i] = __ldg(la.lmask + cell0 + i);
  __syncthreads();
  // wait for the face kernel (a no-op unless launched as its programmatic dependent), and let a
  // programmatic dependent of this grid start
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  auto none = [](int, int, int, const Sum<V>(&)[K]) {};
  lift_phase<D, K, A, 0>(tp, win, c, acc, nc, none);
  __syncthreads();
  if constexpr (D == 3) {
    lift_phase<D, K, A, 1>(tp, win, c, acc, nc, none);
    __syncthreads();
  }
  // the last axis: line (p, q) in 3D, p in 2D; its k nodes are complete
  lift_phase<D, K, A, D - 1>(tp, win, c, acc, nc, [&](const int ci, const int p, const int q, const Sum<V>(&s)[K]) {
    // bit (p > 0) + 2 (q > 0) + 4 (r > 0) of the owner's mask: a face reaches the nodes of that kind
    const int m = mask[ci] >> ((p > 0 ? 1 : 0) + ((D == 3 && q > 0) ? 2 : 0));
    constexpr int UP = (D == 3) ? 4 : 2, SR = (D == 3) ? K : 1;
    const int* rw = row + ci * KR + q;
#pragma unroll
    for (int r = 0; r < K; ++r) {
      if (!((m >> (r > 0 ? UP : 0)) & 1)) continue;
      IO* dst = y + (rw[SR * r] + p);
      const V sv = dot_value(s[r]);
      *dst = to_io(add ? vadd(from_io(*dst, (V*)nullptr), sv) : sv, (IO*)nullptr);
    }
  });
}

template <int D, int K, class A>
__global__ void __launch_bounds__(MAX_CTA_THREADS, LineShape<D, K>::CTAS)
lift_lines_kernel(const typename A::V* __restrict__ tp, typename A::IO* __restrict__ y, const int add,
                  const LiftArgs la, const int cb, const __grid_constant__ Consts<typename A::V, K> c) {
  lift_lines_body<D, K, A>(tp, y, add, la, c, blockIdx.x, cb, gp_dyn_smem);
}

template <int D, int K, class A>
__global__ void __launch_bounds__(MAX_CTA_THREADS, LineShape<D, K>::CTAS)
lift_lines_kernel_batched(const LiftSeg* __restrict__ segs, const FaceSeg<typename A::V, K>* __restrict__ fsegs,
                          const int nseg, const SegPtrs<typename A::IO>* __restrict__ ptrs, const int cb,
                          const __grid_constant__ Consts<typename A::V, K> c) {
  __shared__ LiftSeg seg;
  __shared__ typename A::V* tp;
  __shared__ typename A::IO* y;
  if (threadIdx.x == 0) {
    const int s = find_segment(segs, nseg, (int)blockIdx.x);
    seg = segs[s];
    tp = fsegs[s].wp;
    y = ptrs[s].y;
  }
  __syncthreads();
  lift_lines_body<D, K, A>(tp, y, 0, seg.la, c, (int)blockIdx.x - seg.block0, cb, gp_dyn_smem);
}

template <int D, int K, class A>
__global__ void __launch_bounds__(MAX_CTA_THREADS)
lift_kernel(const typename A::V* __restrict__ wp, typename A::IO* __restrict__ y, const int add,
            const LiftArgs la, const int cb) {
  lift_body<D, K, A>(wp, y, add, la, blockIdx.x, cb, gp_dyn_smem);
}

template <int D, int K, class A>
__global__ void __launch_bounds__(MAX_CTA_THREADS)
lift_kernel_batched(const LiftSeg* __restrict__ segs, const FaceSeg<typename A::V, K>* __restrict__ fsegs,
                    const int nseg, const SegPtrs<typename A::IO>* __restrict__ ptrs, const int cb) {
  __shared__ LiftSeg seg;
  __shared__ typename A::V* wp;
  __shared__ typename A::IO* y;
  if (threadIdx.x == 0) {
    const int s = find_segment(segs, nseg, (int)blockIdx.x);
    seg = segs[s];
    wp = fsegs[s].wp;
    y = ptrs[s].y;
  }
  __syncthreads();
  lift_body<D, K, A>(wp, y, 0, seg.la, (int)blockIdx.x - seg.block0, cb, gp_dyn_smem);
}

}  // namespace gp
