// Shifted Krylov solve for every quadrature node at once, and the weighted sum.
//
// The paper solves (z_j - H_W) y_j = b for all nodes with a shift solver seeded at
// z_seed (the shift-solver remark after Eq. 7; shifted BiCG in its numerical
// section).  For hermitian H_W, BiCG with shadow vector equal to the initial
// residual produces at step k, for every shift, the Galerkin iterate in the Krylov
// space K_k(H_W, b): y_{k,j} = V_k (z_j - T_k)^-1 e_1 ||b||, where H_W V_k = V_k T_k +
// beta_k v_{k+1} e_k^T is the hermitian Lanczos relation with real tridiagonal T_k
// (alpha_i on the diagonal, beta_i off it).  These iterates do not depend on the seed.
// We compute exactly them:
//
//   * one Lanczos process on H_W per source (kernels K1, K2 below);
//   * for every node, the LDL^T factorisation of the complex-symmetric tridiagonal
//     z_j - T_k, updated one row per step:
//       d_1 = z - alpha_1,  d_i = z - alpha_i - beta_{i-1}^2 / d_{i-1},
//       l_i = -beta_i / d_i,  omega_1 = ||b||,  omega_i = -l_{i-1} omega_{i-1},
//       zeta_i = omega_i / d_i
//     (1 / d_i is kept, so each step costs one real division per node);
//     |Im d_i| >= |Im z| > 0, so no pivot ever vanishes (no breakdown);
//   * per node the direction p_i = v_i - l_{i-1} p_{i-1} and y += zeta_i p_i, so that
//     the weighted sum of Eq. 7, s = c0 b + sum_j c_j y_j, is accumulated directly;
//   * the FOM residual of node j after step i is beta_i |zeta_i| v_{i+1}, so its norm
//     is known from scalars; a node stops updating once it is below tol ||b||.
//
// Lanczos vectors are kept unnormalised, U_i = beta_{i-1} v_i (U_1 = b), in a ring
// of three buffers; each consumer scales by 1/||U_i||.  All recurrence scalars are
// FP64 and live on the device; the last block of each kernel (per source) reduces
// the block partials in a fixed order, so reruns are bit-identical, and updates the
// scalars.  The host only reads a done counter every few iterations, and replays
// the per-iteration kernels from a CUDA graph.
//
// Links of about unit norm and |4 - m0| <= 4: the Lanczos vectors are integers of one scale per vector
// (fixed.cuh, the fx_ kernels), in the stored-basis forms and, with a ring of 32 of them, in
// the vector-space form, whose per-node FP64 vectors then advance a batch of iterations at a
// time (fx_node_update_kernel).
#include <algorithm>
#include <climits>
#include <cmath>
#include <complex>
#include <cstdio>
#include <string>
#include <cstring>
#include <functional>
#include <type_traits>
#include <vector>

#include <cooperative_groups.h>

#include "fixed.cuh"

namespace {

constexpr int NT1 = 128;  // K1: stencil + Lanczos epilogue; K3: regeneration pass
constexpr int NT2 = 256;  // K2: vector updates
// Resident blocks per SM the stencil kernels are compiled for: 4 (<= 128 registers) for
// FP64; 7 (<= 72 registers) for double-float (16^3x32, 12 sources, double-float solve:
// 467 / 421 / 457 ms at 6 / 7 / 8 blocks per SM -- at 8 the 64-register limit spills
// and the shared-memory partials leave L1 almost no room; with the link rows loaded one
// row ahead, 414 / 407.5 ms at 6 / 7).
template <typename R>
constexpr int k1_min_blocks() { return std::is_same<R, DF>::value ? 7 : 4; }
// FP64 and double-float solves read the link copy scaled by -1/2 (the hop factor of D_W) with the time
// boundary sign on the last time slice's time links, so phase 1 applies no boundary sign
// and phase 2 adds the partials to the diagonal term without a multiplication
template <typename R>
constexpr bool kHalvedLinks = std::is_same<R, double>::value || std::is_same<R, DF>::value;

// Fixed point: what the kernels of iteration i know of X_i.
struct FxVec {
  double n2, inv_n2;  // ||X_i||^2 in integer units and its reciprocal
  FX dia, gam;        // coefficients of X_i and X_{i-1} in w, unit 2^-60 (both below 2)
  int q;              // w = (H X_i / 4) 2^-q - ...
};

struct SrcState {
  double bnorm;   // ||b||
  double inv_b2;  // 1 / ||b||^2
  double n_prev;  // ||U_{i-1}||
  double n_cur;   // ||U_i||
  double alpha;   // alpha_i
  int iter;       // i
  int done;
  int status;     // OV_OK, OV_ERR_NOT_CONVERGED, OV_ERR_BREAKDOWN
  int n_act;
  double node_updates;  // sum over iterations of n_act
  int k_final;    // second pass: number of Lanczos vectors to regenerate
  int pad_;
  // derived once per iteration by the block that updates the norms (not per thread):
  double inv_n;   // 1 / ||U_i||
  double cm;      // ||U_i|| / ||U_{i-1}|| (0 at i = 1)
  double alpha_n; // alpha_i / ||U_i||: U_{i+1} = w - alpha_n U_i in one FMA per real
  float df[8];    // inv_n, cm, alpha, alpha_n as double-float (hi, lo) pairs
  // fixed-point vectors X_i (fx_* kernels); U_i = X_i up to a power of two
  FxVec vec[2];  // of X_i in slot i & 1: written by K1 of iteration i, read by K2 and the next K1
  int k[2];      // X_{i+1} = (w - a X_i) 2^k, k in slot i & 1: written by K2, read by the next K1
  int it1, it2;  // iteration K1 last ran, 0: none left to run (read by K2); iteration K1 runs
                 // next (written by K2)
  int e_in;      // X_1 = b 2^e_in
  int upd_i, upd_n;  // per-node vectors: first iteration and most iterations of the next update
};

// exact double-float split of an FP64 value: hi = rn(x), lo = rn(x - hi)
__device__ __forceinline__ void df_split(double x, float* d) {
  d[0] = __double2float_rn(x);
  d[1] = __double2float_rn(x - (double)d[0]);
}

// inv_n, cm and (double-float vectors only) their double-float forms from n_cur, n_prev
// and iter.  These run in one thread on the path between two launches, where every FP64
// instruction waits for the previous one (GB300's FP64 rate is 1/64 of FP32): the
// reciprocal is the correctly rounded one (the same value as 1.0 / n_cur), and the FP64
// solve skips the splits it does not read.
template <typename R>
__device__ __forceinline__ void set_norm_scalars(SrcState* S) {
  S->inv_n = __drcp_rn(S->n_cur);
  S->cm = (S->iter > 1) ? S->n_cur / S->n_prev : 0.0;
  if constexpr (std::is_same<R, DF>::value) {
    df_split(S->inv_n, S->df + 0);
    df_split(S->cm, S->df + 2);
  }
}

// An FP64 recurrence scalar in the vector arithmetic type; for double-float, from its
// stored split (no per-thread FP64 conversion).
template <typename R>
__device__ __forceinline__ R scal(double v, const float*) { return (R)v; }
template <>
__device__ __forceinline__ DF scal<DF>(double, const float* d) { return DF(d[0], d[1]); }

// Per-iteration scalars of the regeneration pass, in the vector arithmetic type.
template <typename R>
struct RegenRec {
  R inv_n, cm, alpha, alpha_n;
  Cx<R> g;
};

struct ShiftState {
  double2 invd, omega, zeta;  // 1 / d_i, omega_i, zeta_i of the LDL^T recurrence
  double res2;                // |beta_i zeta_i|^2 / ||b||^2 (squared relative FOM residual)
  int active;
  int last_iter;
};

struct SolveParams {
  double tol;
  int max_iter;
  int nshift;
  int vec_shifts;  // 1: per-node direction vectors and the weighted sum in K2; 0: scalars only
  int nslots;      // Lanczos vector slots per source: 3 (ring, slot i % 3) or a stored basis (slot i)
  int store;       // 1: slot i holds U_i for every i (basis kept for a later combination)
  // 1 (scalar-only forms): the per-node LDL^T rows and stopping tests run in
  // node_check_kernel every kNodeCheck iterations from the recorded alpha_i, beta_i,
  // not in the last blocks of K1 and K2 (which then only form alpha_i and beta_i)
  int defer_nodes;
  int slot_mask;  // fixed point: X_i in slot i & slot_mask
};

// Iterations between per-node stopping checks of the scalar-only forms: a source runs at
// most kNodeCheck - 1 iterations past the one where its last node met tol.
constexpr int kNodeCheck = 8;

// Per-node coefficients l_{i-1}, c_j zeta_i, zeta_i of the vector-space update, stored
// per iteration by K1's last block: FP64 for FP64 and FP32 vectors (converted where
// used), double-float splits for double-float vectors (no per-element FP64 conversion).
template <typename R>
struct Coef {
  using T = double2;
  __device__ __forceinline__ static T make(double2 v) { return v; }
  __device__ __forceinline__ static Cx<R> get(const T* p) {
    const double2 v = __ldg(p);
    return {(R)v.x, (R)v.y};
  }
};
template <>
struct Coef<DF> {
  using T = float4;
  __device__ __forceinline__ static T make(double2 v) { return Store<DF>::pack(cx_from<DF>(v.x, v.y)); }
  __device__ __forceinline__ static Cx<DF> get(const T* p) { return Store<DF>::unpack(__ldg(p)); }
};

// Device pointers of one solve (all in workspace owned by the context).
template <typename R>
struct SolveArgs {
  using T = typename Store<R>::T;
  T* ring;            // [src][3][12V]
  T* p;               // [src][nshift][12V]
  T* x;               // [src][nshift][12V] or null
  double2* sacc;      // [src][12V] weighted sum (FP64) or null
  double2* sgrp;      // [src][groups - 1][12V] its parts from K2's other node groups or null
  T* ssum;            // [src][12V] regeneration-pass sum in the vector type (double-float) or null
  const T* stencil;   // optional pre-applied H U_i for K1 ([src][12V]) or null
  SrcState* src;
  ShiftState* sh;     // [src][nshift]
  const double2* z;   // [src][nshift]
  const double2* c;   // [src][nshift]
  int* act_idx;       // [src][nshift]
  typename Coef<R>::T* act_l;   // [src][nshift] l_{i-1}
  typename Coef<R>::T* act_cz;  // [src][nshift] c_j zeta_i
  typename Coef<R>::T* act_z;   // [src][nshift] zeta_i
  double* part1;      // [src][nblk1]
  double* part2;      // [src][nblk2]
  long long* bins1;   // [src][2][kFxBins][kFxWords] fixed point: sums of K1 and of K2, slot i & 1
  long long* bins2;
  unsigned* cnt;      // [src][2]
  int* done_count;
  double* hist_a;     // [src][max_iter] or null
  double* hist_b;
  double* hist_n2;    // fixed point: ||X_i||^2
  const double2* gco; // [src][max_iter] second-pass coefficients or null
  // fixed point with a stored basis: rows of every node's LDL^T, else null
  double2* fd;        // [src][max_iter][nshift] 1 / d_i
  double2* fz;        // [src][max_iter][nshift] zeta_i
  // fixed point with per-node vectors (fx_node_update_kernel), else null
  double2* pv;        // [src][nshift][12V padded] direction vectors, in the layout of X
  double2* xv;        // [src][nshift][12V] node solutions or null
  double2* nco;       // [src][nshift][kNodeRun][3] l_{i-1}, c_j zeta_i, zeta_i of the next update
  double* nin;        // [src][kNodeRun] 1 / ||X_i||
  const RegenRec<R>* rrec;  // [src][max_iter] regeneration-pass scalars or null
  const double* tol_src;  // [src] per-source tolerance or null (then SolveParams::tol)
  const SolveParams* prm;
  const T* U;         // links
  Geom g;
  R diag;
  double diag4;       // (4 - m0) / 4 (fixed point)
};

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// Lanczos vector slot of iteration index i: a ring of three, or the stored basis.
__device__ __forceinline__ size_t lz_slot(const SolveParams* p, int i) {
  return p->store ? (size_t)i : (size_t)(i % 3);
}

// The Lanczos vector arithmetic, written with explicitly rounded operations so that
// every kernel that performs it (K1/K2 of the solve, K3 of the second pass) produces
// the same bits: the second pass of OV_MODE_FP64_2PASS regenerates the first pass's
// basis exactly.
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ DF rmul(DF a, DF b) { return a * b; }
__device__ __forceinline__ DF rfma(DF a, DF b, DF c) { return fma(a, b, c); }

// w = (H U_i) / n_i - (n_i / n_{i-1}) U_{i-1}   (second term absent at i = 1)
template <typename R>
__device__ __forceinline__ Cx<R> lz_w(Cx<R> o, Cx<R> um, R inv_n, R cm, bool first) {
  Cx<R> w = {rmul(inv_n, o.re), rmul(inv_n, o.im)};
  if (!first) {
    w.re = rfma(-cm, um.re, w.re);
    w.im = rfma(-cm, um.im, w.im);
  }
  return w;
}
// v_i = U_i / n_i
template <typename R>
__device__ __forceinline__ Cx<R> lz_v(Cx<R> u, R inv_n) {
  return {rmul(inv_n, u.re), rmul(inv_n, u.im)};
}
// U_{i+1} = w - alpha_i v_i = w - (alpha_i / ||U_i||) U_i, one FMA per real with the
// scalar alpha_n = alpha_i / ||U_i|| (the FP64 pipe bounds these kernels)
template <typename R>
__device__ __forceinline__ Cx<R> lz_next(Cx<R> w, Cx<R> u, R alpha_n) {
  return {rfma(-alpha_n, u.re, w.re), rfma(-alpha_n, u.im, w.im)};
}

// Per-thread partial of an inner product.  FP64 and FP32 vectors: an FP64 sum.
// Double-float vectors: a double-float sum (FP32 instructions only), converted to FP64
// once per thread -- per-element FP64 conversions would put the kernel on the FP64 pipe.
template <typename R>
struct Acc {
  using T = double;
  __device__ __forceinline__ static T zero() { return 0.0; }
  // FP64 vectors: two FMAs per complex (the FP64 pipe is the bound); FP32 vectors: the
  // products in FP64
  __device__ __forceinline__ static T dot(T acc, Cx<R> u, Cx<R> w) {
    if constexpr (std::is_same<R, double>::value) return fma(u.im, w.im, fma(u.re, w.re, acc));
    return acc + ((double)u.re * (double)w.re + (double)u.im * (double)w.im);
  }
  __device__ __forceinline__ static double get(T acc) { return acc; }
  template <int NT>
  __device__ __forceinline__ static double total(T acc, double* sh) { return block_sum<NT>(acc, sh); }
};
template <>
struct Acc<DF> {
  using T = DF;
  __device__ __forceinline__ static T zero() { return DF(0.f, 0.f); }
  // running sum unnormalised (renormalised by the block sum)
  __device__ __forceinline__ static T dot(T acc, Cx<DF> u, Cx<DF> w) {
    return fma_unnormalised(u.im, w.im, fma_unnormalised(u.re, w.re, acc));
  }
  __device__ __forceinline__ static double get(T acc) { return (double)acc; }
  // block sum in double-float (fixed tree), one FP64 conversion per block; sh >= NT/32 doubles
  template <int NT>
  __device__ __forceinline__ static double total(T v, double* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      v = v + DF(__shfl_down_sync(0xffffffffu, v.hi, o), __shfl_down_sync(0xffffffffu, v.lo, o));
    DF* shd = reinterpret_cast<DF*>(sh);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) shd[w] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0) {
      DF u = shd[0];
#pragma unroll
      for (int k = 1; k < NT / 32; ++k) u = u + shd[k];
      t = (double)u;
    }
    __syncthreads();
    return t;  // valid in thread 0
  }
};

// s += g v in the regeneration pass.  FP64 and FP32 vectors: into the FP64 sum.
// Double-float vectors: into a double-float sum (a.ssum), folded into the FP64 sum
// after the last iteration.  The element is read and written by this thread only.
template <typename R>
struct SumAdd {
  __device__ __forceinline__ static void add(const SolveArgs<R>& a, size_t idx, Cx<R> g, Cx<R> v) {
    double2 sv = a.sacc[idx];
    sv.x += (double)g.re * (double)v.re - (double)g.im * (double)v.im;
    sv.y += (double)g.re * (double)v.im + (double)g.im * (double)v.re;
    a.sacc[idx] = sv;
  }
};
template <>
struct SumAdd<DF> {
  __device__ __forceinline__ static void add(const SolveArgs<DF>& a, size_t idx, Cx<DF> g, Cx<DF> v) {
    const Cx<DF> sv = Store<DF>::unpack(a.ssum[idx]);
    a.ssum[idx] = Store<DF>::pack(cfma(g, v, sv));
  }
};

__device__ void mark_done(SrcState* S, int* done_count, int status) {
  S->done = 1;
  S->status = status;
  atomicAdd(done_count, 1);
}

// Block-wide ordered compaction helper: returns this thread's slot among the
// threads with flag set (in thread order) and the block total in *total.
template <int NT>
__device__ __forceinline__ int block_rank(bool flag, int* total, int* wsh) {
  const unsigned bal = __ballot_sync(0xffffffffu, flag);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) wsh[wid] = __popc(bal);
  __syncthreads();
  int off = 0, tot = 0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    if (w < wid) off += wsh[w];
    tot += wsh[w];
  }
  __syncthreads();
  *total = tot;
  return off + __popc(bal & ((1u << lane) - 1u));
}

// K1: w = H U_i / n_i - (n_i / n_{i-1}) U_{i-1};  alpha_i = Re <U_i, w> / n_i; then,
// in the last block, row i of every active node's LDL^T and the active list for K2.
// The stencil runs 4 threads per site (hw_split_*): a block covers 32 sites.
// 4 blocks per SM (<= 128 registers): an 8^4 x 4-source grid (512 blocks) fits one wave
template <typename R>
__global__ void __launch_bounds__(NT1, k1_min_blocks<R>()) lanczos_hw_kernel(SolveArgs<R> a) {
  using T = typename Store<R>::T;
  __shared__ double sh[NT1 / 32];
  __shared__ int wsh[NT1 / 32];
  __shared__ bool last;
  __shared__ double alpha_sh;
  __shared__ Cx<R> sm[4 * 12 * kSplitSites];
  // one-dimensional grid, the sources of a site tile in consecutive blocks (k1_grid)
  const int nb = (a.g.V + kSplitSites - 1) / kSplitSites;  // site tiles per source
  const int nsl = gridDim.x / nb;                           // sources in this launch
  const int r = blockIdx.x % nsl, tb = blockIdx.x / nsl;
  SrcState* S = a.src + r;
  if (S->done) return;
  const int V = a.g.V;
  const size_t n12 = (size_t)12 * V;
  const int i = S->iter;
  T* base = a.ring + (size_t)r * a.prm->nslots * n12;
  const T* Ui = base + lz_slot(a.prm, i) * n12;
  const T* Um = base + (a.prm->store ? (size_t)(i - 1) : (size_t)((i + 2) % 3)) * n12;  // U_{i-1}
  T* W = base + lz_slot(a.prm, i + 1) * n12;
  const double inv_n = S->inv_n;
  const R inv_nR = scal<R>(inv_n, S->df + 0), cmR = scal<R>(S->cm, S->df + 2);
  const int site0 = tb * kSplitSites;
  typename Acc<R>::T dot = Acc<R>::zero();
  if (a.stencil) {
    // pre-applied operator (H^2 Lanczos for the spectral gap): one thread per (site, 3 components)
    const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5, s = site0 + lane;
    if (s < V) {
      const T* Hs = a.stencil + (size_t)r * n12;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const size_t e = (3 * grp + q) * (size_t)V + s;
        const Cx<R> u = ld<R>(Ui + e);
        const Cx<R> um = (i > 1) ? ld<R>(Um + e) : Cx<R>{R(0), R(0)};
        const Cx<R> w = lz_w<R>(ld<R>(Hs + e), um, inv_nR, cmR, i == 1);
        st<R>(W + e, w);
        dot = Acc<R>::dot(dot, u, w);
      }
    }
  } else {
    hw_split_phase1<R, false, !kHalvedLinks<R>>(Ui, a.U, a.g, site0, sm);
    __syncthreads();
    Cx<R> o[3];
    int s, k0;
    if (hw_split_phase2<R, false, kHalvedLinks<R>>(Ui, a.g, site0, a.diag, sm, o, &s, &k0)) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const size_t e = (k0 + q) * (size_t)V + s;
        const Cx<R> u = ld<R>(Ui + e);
        const Cx<R> um = (i > 1) ? ld<R>(Um + e) : Cx<R>{R(0), R(0)};
        const Cx<R> w = lz_w<R>(o[q], um, inv_nR, cmR, i == 1);
        st<R>(W + e, w);
        dot = Acc<R>::dot(dot, u, w);
      }
    }
  }
  double bs = Acc<R>::template total<NT1>(dot, sh);
  if (threadIdx.x == 0) {
    a.part1[(size_t)r * nb + tb] = bs;
    __threadfence();
    last = (atomicAdd(a.cnt + 2 * r, 1u) == (unsigned)nb - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const double tot = sum_partials<NT1>(a.part1 + (size_t)r * nb, nb, sh);
  if (threadIdx.x == 0) {
    a.cnt[2 * r] = 0;
    const double alpha = tot * inv_n;
    S->alpha = alpha;
    S->alpha_n = alpha * inv_n;
    if constexpr (std::is_same<R, DF>::value) {
      df_split(alpha, S->df + 4);
      df_split(S->alpha_n, S->df + 6);
    }
    alpha_sh = alpha;
    if (a.hist_a) a.hist_a[(size_t)r * a.prm->max_iter + (i - 1)] = alpha;
    if (!isfinite(alpha)) {
      S->n_act = 0;
      mark_done(S, a.done_count, OV_ERR_BREAKDOWN);
    }
  }
  __syncthreads();
  const double alpha = alpha_sh;
  if (!isfinite(alpha) || a.prm->defer_nodes) return;
  // per-node LDL^T row i (one thread per node) and the ordered active list
  const int ns = a.prm->nshift;
  const double beta_prev = S->n_cur;  // beta_{i-1} = ||U_i|| (i >= 2)
  int na = 0;
  for (int j0 = 0; j0 < ns; j0 += NT1) {
    const int j = j0 + threadIdx.x;
    bool act = false;
    double2 lprev = make_double2(0.0, 0.0), zeta = make_double2(0.0, 0.0);
    if (j < ns) {
      ShiftState& q = a.sh[(size_t)r * ns + j];
      act = q.active != 0;
      if (act) {
        const double2 zj = a.z[(size_t)r * ns + j];
        double2 d, om;
        if (i == 1) {
          d = make_double2(zj.x - alpha, zj.y);
          om = make_double2(S->bnorm, 0.0);
        } else {
          const double2 ip = q.invd;  // 1 / d_{i-1}
          lprev = make_double2(-beta_prev * ip.x, -beta_prev * ip.y);
          const double b2 = beta_prev * beta_prev;
          d = make_double2(zj.x - alpha - b2 * ip.x, zj.y - b2 * ip.y);
          om = cmul(make_double2(-lprev.x, -lprev.y), q.omega);
        }
        const double inv = __drcp_rn(d.x * d.x + d.y * d.y);  // = 1.0 / |d|^2
        const double2 invd = make_double2(d.x * inv, -d.y * inv);
        zeta = cmul(om, invd);
        q.invd = invd;
        q.omega = om;
        q.zeta = zeta;
      }
    }
    int cnt;
    const int slot = block_rank<NT1>(act, &cnt, wsh);
    if (act) {
      const size_t o = (size_t)r * ns + na + slot;
      a.act_idx[o] = j;
      a.act_l[o] = Coef<R>::make(lprev);
      a.act_cz[o] = Coef<R>::make(cmul(a.c[(size_t)r * ns + j], zeta));
      a.act_z[o] = Coef<R>::make(zeta);
    }
    na += cnt;
  }
  if (threadIdx.x == 0) {
    S->n_act = na;
    S->node_updates += (a.prm->vec_shifts ? na : 0);
  }
}

// K2: U_{i+1} = w - alpha_i U_i / n_i (in place over w), beta_i = ||U_{i+1}||,
// per active node p = v_i - l_{i-1} p, x += zeta_i p, s += c_j zeta_i p (vec_shifts),
// then per-node residuals |beta_i zeta_i| and l_i = -beta_i / d_i in the last block.
template <typename R>
__global__ void __launch_bounds__(NT2) lanczos_update_kernel(SolveArgs<R> a) {
  using T = typename Store<R>::T;
  __shared__ double sh[NT2 / 32];
  __shared__ bool last;
  __shared__ double nrm2_sh;
  const int r = blockIdx.y;
  SrcState* S = a.src + r;
  if (S->done) return;
  const int V = a.g.V;
  const size_t n12 = (size_t)12 * V;
  const int i = S->iter;
  const int ns = a.prm->nshift;
  T* base = a.ring + (size_t)r * a.prm->nslots * n12;
  const T* Ui = base + lz_slot(a.prm, i) * n12;
  T* W = base + lz_slot(a.prm, i + 1) * n12;
  // node groups (blockIdx.z, k2_groups): group z takes the active nodes z, z + groups, ...;
  // the first one also advances the Lanczos vector, the only reader and writer of w
  const int z = blockIdx.z, nz = gridDim.z;
  const int na = a.prm->vec_shifts ? S->n_act : 0;
  const R inv_nR = scal<R>(S->inv_n, S->df + 0), anR = scal<R>(S->alpha_n, S->df + 6);
  typename Acc<R>::T nrm = Acc<R>::zero();
  double nrm_im = 0.0;  // FP64 vectors: the imaginary parts in a second, independent FMA chain
  size_t e0 = (size_t)blockIdx.x * NT2 + threadIdx.x;
  const size_t gs = (size_t)gridDim.x * NT2;
  if (z >= na && z > 0) e0 = n12;  // fewer active nodes than groups
  if constexpr (!std::is_same<R, float>::value) {
    // scalar-only forms (no per-node vectors): four elements per thread in flight, their
    // loads issued before any arithmetic (the arithmetic and HBM overlap across them)
    if (na == 0) {
      constexpr int B = 4;
      for (; e0 + (B - 1) * gs < n12; e0 += B * gs) {
        Cx<R> ub[B], wb[B];
#pragma unroll
        for (int k = 0; k < B; ++k) {
          ub[k] = ld<R>(Ui + e0 + k * gs);
          wb[k] = ld<R>(W + e0 + k * gs);
        }
#pragma unroll
        for (int k = 0; k < B; ++k) {
          const Cx<R> u = lz_next<R>(wb[k], ub[k], anR);
          st<R>(W + e0 + k * gs, u);
          if constexpr (std::is_same<R, double>::value) {
            nrm = fma(u.re, u.re, nrm);
            nrm_im = fma(u.im, u.im, nrm_im);
          } else {
            nrm = Acc<R>::dot(nrm, u, u);
          }
        }
      }
    }
  }
  // grid-stride: a few blocks per source (fewer partials and atomics than one block per chunk)
  for (size_t e = e0; e < n12; e += gs) {
    const Cx<R> ui = ld<R>(Ui + e);
    if (z == 0) {
      const Cx<R> u = lz_next<R>(ld<R>(W + e), ui, anR);
      st<R>(W + e, u);
      if constexpr (std::is_same<R, double>::value) {
        nrm = fma(u.re, u.re, nrm);
        nrm_im = fma(u.im, u.im, nrm_im);
      } else {
        nrm = Acc<R>::dot(nrm, u, u);
      }
    }
    Cx<R> v = ui;  // v_i = U_i / ||U_i||, read only by the per-node direction updates
    if (na > 0) v = lz_v<R>(ui, inv_nR);
    double sre = 0.0, sim = 0.0;      // weighted sum over nodes: FP64 (FP64, FP32 vectors)
    Cx<R> sdf = {R(0), R(0)};          // or double-float (double-float vectors)
    const int* idx = a.act_idx + (size_t)r * ns;
    const typename Coef<R>::T* al = a.act_l + (size_t)r * ns;
    const typename Coef<R>::T* acz = a.act_cz + (size_t)r * ns;
    const typename Coef<R>::T* az = a.act_z + (size_t)r * ns;
    for (int k = z; k < na; k += nz) {
      const int j = __ldg(idx + k);
      T* P = a.p + ((size_t)r * ns + j) * n12 + e;
      Cx<R> pv = v;
      if (i > 1) pv = cfma(cneg(Coef<R>::get(al + k)), ld<R>(P), v);  // v - l p
      st<R>(P, pv);
      if constexpr (std::is_same<R, DF>::value) {
        sdf = cfma(Coef<R>::get(acz + k), pv, sdf);
      } else {
        const double2 cz = __ldg(acz + k);
        sre += cz.x * (double)pv.re - cz.y * (double)pv.im;
        sim += cz.x * (double)pv.im + cz.y * (double)pv.re;
      }
      if (a.x) {
        T* X = a.x + ((size_t)r * ns + j) * n12 + e;
        const Cx<R> xo = (i > 1) ? ld<R>(X) : Cx<R>{R(0), R(0)};
        st<R>(X, cfma(Coef<R>::get(az + k), pv, xo));
      }
    }
    if (a.sacc && na > 0) {
      if constexpr (std::is_same<R, DF>::value) {
        sre = (double)sdf.re;
        sim = (double)sdf.im;
      }
      double2* Sx = (z == 0 ? a.sacc + (size_t)r * n12 : a.sgrp + ((size_t)r * (nz - 1) + z - 1) * n12) + e;
      double2 sv = *Sx;
      sv.x += sre;
      sv.y += sim;
      *Sx = sv;
    }
  }
  if constexpr (std::is_same<R, double>::value) nrm += nrm_im;
  double bs = 0.0;
  if (z == 0) bs = Acc<R>::template total<NT2>(nrm, sh);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (z == 0) a.part2[(size_t)r * gridDim.x + blockIdx.x] = bs;
    __threadfence();
    last = (atomicAdd(a.cnt + 2 * r + 1, 1u) == gridDim.x * nz - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  // ||u||^2 goes to every thread before the square root is taken: the node tests need
  // only beta^2, and sqrt sits on one thread's serial FP64 path
  const double tot = sum_partials<NT2>(a.part2 + (size_t)r * gridDim.x, gridDim.x, sh);
  if (threadIdx.x == 0) {
    a.cnt[2 * r + 1] = 0;
    nrm2_sh = tot;
    if (!isfinite(tot)) {
      if (a.hist_b) a.hist_b[(size_t)r * a.prm->max_iter + (i - 1)] = sqrt(tot);
      mark_done(S, a.done_count, OV_ERR_BREAKDOWN);
    }
  }
  __syncthreads();
  const double nrm2 = nrm2_sh;
  if (!isfinite(nrm2)) return;
  const double tol = a.tol_src ? a.tol_src[r] : a.prm->tol;
  const double tol2 = tol * tol;
  const double b2n = nrm2 * S->inv_b2;
  const bool defer = a.prm->defer_nodes != 0;
  int still = 0;
  for (int j0 = 0; j0 < ns && !defer; j0 += NT2) {
    const int j = j0 + threadIdx.x;
    bool act = false;
    if (j < ns) {
      ShiftState& q = a.sh[(size_t)r * ns + j];
      if (q.active) {
        q.res2 = b2n * (q.zeta.x * q.zeta.x + q.zeta.y * q.zeta.y);
        q.last_iter = i;
        if (q.res2 <= tol2 || nrm2 == 0.0) {
          q.active = 0;
          if (nrm2 == 0.0) q.res2 = 0.0;
        } else {
          act = true;
        }
      }
    }
    still += __syncthreads_count(act);
  }
  if (threadIdx.x != 0) return;
  const double beta = sqrt(nrm2);
  if (a.hist_b) a.hist_b[(size_t)r * a.prm->max_iter + (i - 1)] = beta;
  S->n_prev = S->n_cur;
  S->n_cur = beta;
  S->iter = i + 1;
  set_norm_scalars<R>(S);
  if (beta == 0.0) {
    mark_done(S, a.done_count, OV_OK);
  } else if (ns > 0 && still == 0 && !defer) {
    mark_done(S, a.done_count, OV_OK);
  } else if (i >= a.prm->max_iter || (a.prm->store && i + 2 >= a.prm->nslots)) {
    mark_done(S, a.done_count, ns > 0 ? OV_ERR_NOT_CONVERGED : OV_OK);
  }
}

// Per-node LDL^T rows and stopping tests of the scalar-only forms (defer_nodes), caught up
// from the recorded alpha_i, beta_i over the iterations completed since the last check:
// one thread per node, the same recurrence K1 and K2 run per iteration otherwise,
//   d_1 = z - alpha_1, omega_1 = ||b||;  l_{i-1} = -beta_{i-1} / d_{i-1},
//   d_i = z - alpha_i - beta_{i-1}^2 / d_{i-1},  omega_i = -l_{i-1} omega_{i-1};
//   zeta_i = omega_i / d_i,  node residual |beta_i zeta_i| / ||b||.
// A node stops at the first iteration that meets tol; a source whose nodes have all
// stopped is marked done (also one K2 stopped at its iteration limit in that same
// iteration: its status becomes OV_OK).  Off the per-iteration critical path: K1 and K2
// keep only their two reductions in the last block.
template <typename R>
__global__ void __launch_bounds__(NT1) node_check_kernel(SolveArgs<R> a) {
  const int r = blockIdx.y;
  SrcState* S = a.src + r;
  const int ns = a.prm->nshift;
  const int mi = a.prm->max_iter;
  const int upto = S->iter - 1;  // iterations whose alpha_i and beta_i are recorded
  const double tol = a.tol_src ? a.tol_src[r] : a.prm->tol;
  const double tol2 = tol * tol;
  const double* ha = a.hist_a + (size_t)r * mi;
  const double* hb = a.hist_b + (size_t)r * mi;
  int still = 0;
  for (int j0 = 0; j0 < ns; j0 += NT1) {
    const int j = j0 + threadIdx.x;
    bool act = false;
    if (j < ns) {
      ShiftState& q = a.sh[(size_t)r * ns + j];
      if (q.active) {
        const double2 zj = a.z[(size_t)r * ns + j];
        double2 invd = q.invd, om = q.omega, zeta = q.zeta;
        double res2 = q.res2;
        int i = q.last_iter + 1;
        act = true;
        for (; i <= upto; ++i) {
          const double alpha = ha[i - 1], beta = hb[i - 1];
          double2 d;
          if (i == 1) {
            d = make_double2(zj.x - alpha, zj.y);
            om = make_double2(S->bnorm, 0.0);
          } else {
            const double bp = hb[i - 2];  // beta_{i-1} = ||U_i||
            const double2 lprev = make_double2(-bp * invd.x, -bp * invd.y);
            const double b2 = bp * bp;
            d = make_double2(zj.x - alpha - b2 * invd.x, zj.y - b2 * invd.y);
            om = cmul(make_double2(-lprev.x, -lprev.y), om);
          }
          const double inv = __drcp_rn(d.x * d.x + d.y * d.y);
          invd = make_double2(d.x * inv, -d.y * inv);
          zeta = cmul(om, invd);
          res2 = beta * beta * S->inv_b2 * (zeta.x * zeta.x + zeta.y * zeta.y);
          if (res2 <= tol2 || beta == 0.0) {
            if (beta == 0.0) res2 = 0.0;
            act = false;
            break;
          }
        }
        q.invd = invd;
        q.omega = om;
        q.zeta = zeta;
        q.res2 = res2;
        q.last_iter = act ? upto : i;
        q.active = act ? 1 : 0;
      }
    }
    still += __syncthreads_count(act);
  }
  if (threadIdx.x == 0 && ns > 0 && still == 0) {
    if (!S->done)
      mark_done(S, a.done_count, OV_OK);
    else if (S->status == OV_ERR_NOT_CONVERGED)
      S->status = OV_OK;
  }
}

// K3 (second pass of OV_MODE_FP64_2PASS): regenerate U_{i+1} from the recorded
// alpha_i and ||U_i|| with the first pass's arithmetic, and add g_i v_i to the sum.
// One kernel per iteration; the last block advances the iteration counter.
template <typename R>
__global__ void __launch_bounds__(NT1, k1_min_blocks<R>()) lanczos_regen_kernel(SolveArgs<R> a) {
  using T = typename Store<R>::T;
  __shared__ bool last;
  __shared__ Cx<R> sm[4 * 12 * kSplitSites];
  const int r = blockIdx.y;
  SrcState* S = a.src + r;
  const int i = S->iter;
  if (i > S->k_final) return;
  const int V = a.g.V;
  const size_t n12 = (size_t)12 * V;
  const int mi = a.prm->max_iter;
  T* base = a.ring + (size_t)r * a.prm->nslots * n12;
  const T* Ui = base + (size_t)(i % 3) * n12;
  const T* Um = base + (size_t)((i + 2) % 3) * n12;
  T* W = base + (size_t)((i + 1) % 3) * n12;
  const RegenRec<R> rc = a.rrec[(size_t)r * mi + i - 1];
  const R inv_nR = rc.inv_n, cmR = rc.cm, anR = rc.alpha_n;
  const int site0 = blockIdx.x * kSplitSites;
  hw_split_phase1<R, false, !kHalvedLinks<R>>(Ui, a.U, a.g, site0, sm);
  __syncthreads();
  Cx<R> o[3];
  int s, k0;
  if (hw_split_phase2<R, false, kHalvedLinks<R>>(Ui, a.g, site0, a.diag, sm, o, &s, &k0)) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int k = k0 + q;
      const size_t e = k * (size_t)V + s;
      const Cx<R> um = (i > 1) ? ld<R>(Um + e) : Cx<R>{R(0), R(0)};
      const Cx<R> w = lz_w<R>(o[q], um, inv_nR, cmR, i == 1);
      const Cx<R> ui = ld<R>(Ui + e);
      const Cx<R> v = lz_v<R>(ui, inv_nR);
      st<R>(W + e, lz_next<R>(w, ui, anR));
      SumAdd<R>::add(a, (size_t)r * n12 + e, rc.g, v);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = (atomicAdd(a.cnt + 2 * r, 1u) == gridDim.x - 1);
    if (last) {
      a.cnt[2 * r] = 0;
      S->iter = i + 1;
    }
  }
}

// The whole Lanczos loop of the scalar-only forms (vec_shifts = 0) as one cooperative
// persistent launch.  Per iteration: stencil phase (w and <U_i, w> partials), grid
// barrier, every block reduces the same partials in the same order (so every block
// holds the same alpha_i: no serial last-block step), vector update (U_{i+1} and
// ||U_{i+1}||^2 partials), grid barrier, beta_i, and each thread of the grid advances
// at most one node's LDL^T recurrence.  A source whose nodes have all met tol is
// retired at the next barrier (it spends one extra stencil phase).  Data that other
// blocks write during the launch is read through L2 (ld.global.cg).
constexpr int kCoopMaxSrc = 16;

template <typename R>
__global__ void __launch_bounds__(NT1, 4) lanczos_coop_kernel(SolveArgs<R> a, int nsrc) {
  namespace cg = cooperative_groups;
  using T = typename Store<R>::T;
  cg::grid_group grid = cg::this_grid();
  __shared__ Cx<R> sm[4 * 12 * kSplitSites];
  __shared__ double sh[NT1 / 32];
  __shared__ double s_part[kCoopMaxSrc], s_alpha[kCoopMaxSrc], s_beta[kCoopMaxSrc];
  __shared__ double s_ncur[kCoopMaxSrc], s_nprev[kCoopMaxSrc];
  __shared__ int s_done[kCoopMaxSrc];
  __shared__ int s_stop;
  const int G = gridDim.x, b = blockIdx.x, tid = threadIdx.x;
  const int V = a.g.V;
  const size_t n12 = (size_t)12 * V;
  const int ntile = (V + kSplitSites - 1) / kSplitSites;
  const int nwork = ntile * nsrc;
  const int ns = a.prm->nshift, mi = a.prm->max_iter;
  const size_t nsl = (size_t)a.prm->nslots;
  const int lane = tid & 31, grp = tid >> 5;
  if (tid < nsrc) {
    s_ncur[tid] = a.src[tid].n_cur;
    s_nprev[tid] = a.src[tid].n_prev;
    s_done[tid] = a.src[tid].done;
  }
  __syncthreads();
  for (int i = 1;; ++i) {
    // ---- phase 1: w = H U_i / n_i - (n_i / n_{i-1}) U_{i-1}, partial <U_i, w>
    if (tid < kCoopMaxSrc) s_part[tid] = 0.0;
    __syncthreads();
    if (i <= mi) {
      for (int wk = b; wk < nwork; wk += G) {
        const int r = wk / ntile, site0 = (wk % ntile) * kSplitSites;
        if (s_done[r]) continue;
        const T* base = a.ring + (size_t)r * nsl * n12;
        const T* Ui = base + lz_slot(a.prm, i) * n12;
        const T* Um = base + (a.prm->store ? (size_t)(i - 1) : (size_t)((i + 2) % 3)) * n12;
        T* W = (T*)base + lz_slot(a.prm, i + 1) * n12;
        const double inv_n = 1.0 / s_ncur[r];
        const double cm = (i > 1) ? s_ncur[r] / s_nprev[r] : 0.0;
        const R inv_nR = (R)inv_n, cmR = (R)cm;
        hw_split_phase1<R, true, !kHalvedLinks<R>>(Ui, a.U, a.g, site0, sm);
        __syncthreads();
        Cx<R> o[3];
        int s, k0;
        typename Acc<R>::T dot = Acc<R>::zero();
        if (hw_split_phase2<R, true, kHalvedLinks<R>>(Ui, a.g, site0, a.diag, sm, o, &s, &k0)) {
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const size_t e = (k0 + q) * (size_t)V + s;
            const Cx<R> u = ld<R, true>(Ui + e);
            const Cx<R> um = (i > 1) ? ld<R, true>(Um + e) : Cx<R>{R(0), R(0)};
            const Cx<R> w = lz_w<R>(o[q], um, inv_nR, cmR, i == 1);
            st<R>(W + e, w);
            dot = Acc<R>::dot(dot, u, w);
          }
        }
        const double bs = block_sum<NT1>(Acc<R>::get(dot), sh);
        if (tid == 0) s_part[r] += bs;
        __syncthreads();
      }
    }
    if (tid < nsrc) a.part1[(size_t)tid * G + b] = s_part[tid];
    grid.sync();
    // ---- retire sources whose nodes all met tol at iteration i - 1
    if (i > 1) {
      for (int r = 0; r < nsrc; ++r) {
        if (s_done[r]) continue;
        int act = 0;
        for (int j0 = 0; j0 < ns; j0 += NT1) {
          const int j = j0 + tid;
          const int f = (j < ns) ? __ldcg(&a.sh[(size_t)r * ns + j].active) : 0;
          act += __syncthreads_count(f);
        }
        const bool beta0 = (s_ncur[r] == 0.0);
        if (act == 0 || beta0 || i > mi) {
          if (tid == 0) {
            s_done[r] = 1;
            if (b == 0) {
              SrcState* S = a.src + r;
              S->iter = i;
              S->n_cur = s_ncur[r];
              S->n_prev = s_nprev[r];
              set_norm_scalars<R>(S);
              S->status = (act > 0 && !beta0) ? OV_ERR_NOT_CONVERGED : OV_OK;
              S->done = 1;
            }
          }
        }
        __syncthreads();
      }
    }
    if (tid == 0) {
      int all = 1;
      for (int r = 0; r < nsrc; ++r) all &= s_done[r];
      s_stop = all;
    }
    __syncthreads();
    if (s_stop) break;
    // ---- alpha_i for every source (same order in every block)
    for (int r = 0; r < nsrc; ++r) {
      const double t = sum_partials<NT1>(a.part1 + (size_t)r * G, G, sh);
      if (tid == 0) s_alpha[r] = t / s_ncur[r];
    }
    __syncthreads();
    // ---- phase 2: U_{i+1} = w - alpha_i v_i (in place), partial ||U_{i+1}||^2
    if (tid < kCoopMaxSrc) s_part[tid] = 0.0;
    __syncthreads();
    for (int wk = b; wk < nwork; wk += G) {
      const int r = wk / ntile, site0 = (wk % ntile) * kSplitSites;
      if (s_done[r]) continue;
      const T* base = a.ring + (size_t)r * nsl * n12;
      const T* Ui = base + lz_slot(a.prm, i) * n12;
      T* W = (T*)base + lz_slot(a.prm, i + 1) * n12;
      const double inv_n = 1.0 / s_ncur[r];
      const int s = site0 + lane;
      typename Acc<R>::T nrm = Acc<R>::zero();
      const R anR = (R)(s_alpha[r] * inv_n);
      if (s < V) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const size_t e = (3 * grp + q) * (size_t)V + s;
          const Cx<R> u = lz_next<R>(ld<R, true>(W + e), ld<R, true>(Ui + e), anR);
          st<R>(W + e, u);
          nrm = Acc<R>::dot(nrm, u, u);
        }
      }
      const double bs = block_sum<NT1>(Acc<R>::get(nrm), sh);
      if (tid == 0) s_part[r] += bs;
      __syncthreads();
    }
    if (tid < nsrc) a.part2[(size_t)tid * G + b] = s_part[tid];
    grid.sync();
    for (int r = 0; r < nsrc; ++r) {
      const double t = sum_partials<NT1>(a.part2 + (size_t)r * G, G, sh);
      if (tid == 0) s_beta[r] = sqrt(t);
    }
    __syncthreads();
    // ---- node recurrences (one node per thread of the grid) and history
    for (int q = b * NT1 + tid; q < nsrc * ns; q += G * NT1) {
      const int r = q / ns;
      if (s_done[r]) continue;
      ShiftState& st8 = a.sh[q];
      if (!st8.active) continue;
      const double alpha = s_alpha[r], beta = s_beta[r], beta_prev = s_ncur[r];
      const double2 zj = a.z[q];
      double2 d, om;
      if (i == 1) {
        d = make_double2(zj.x - alpha, zj.y);
        om = make_double2(a.src[r].bnorm, 0.0);
      } else {
        const double2 ip = st8.invd;
        const double b2 = beta_prev * beta_prev;
        d = make_double2(zj.x - alpha - b2 * ip.x, zj.y - b2 * ip.y);
        om = cmul(make_double2(beta_prev * ip.x, beta_prev * ip.y), st8.omega);
      }
      const double inv = 1.0 / (d.x * d.x + d.y * d.y);
      const double2 invd = make_double2(d.x * inv, -d.y * inv);
      const double2 zeta = cmul(om, invd);
      st8.invd = invd;
      st8.omega = om;
      st8.zeta = zeta;
      const double tol = a.tol_src ? a.tol_src[r] : a.prm->tol;
      st8.res2 = beta * beta * a.src[r].inv_b2 * (zeta.x * zeta.x + zeta.y * zeta.y);
      st8.last_iter = i;
      if (st8.res2 <= tol * tol || beta == 0.0) {
        st8.active = 0;
        if (beta == 0.0) st8.res2 = 0.0;
      }
    }
    if (tid < nsrc && !s_done[tid]) {
      if (b == 0 && a.hist_a) {
        a.hist_a[(size_t)tid * mi + (i - 1)] = s_alpha[tid];
        a.hist_b[(size_t)tid * mi + (i - 1)] = s_beta[tid];
      }
      s_nprev[tid] = s_ncur[tid];
      s_ncur[tid] = s_beta[tid];
      if (!isfinite(s_alpha[tid]) || !isfinite(s_beta[tid])) {
        s_done[tid] = 1;
        if (b == 0) {
          a.src[tid].iter = i + 1;
          a.src[tid].status = OV_ERR_BREAKDOWN;
          a.src[tid].done = 1;
        }
      }
    }
    __syncthreads();
  }
}

// Per-iteration scalars of the regeneration pass from the recorded alpha_i, beta_i and
// the coefficients g_i, in the vector type -- with the same FP64 expressions (and
// double-float splits) as the first pass, so the regenerated basis is bit-identical.
template <typename R>
__global__ void regen_scalars_kernel(SolveArgs<R> a, RegenRec<R>* rec, int nsrc) {
  const int mi = a.prm->max_iter;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nsrc * mi; t += gridDim.x * blockDim.x) {
    const int r = t / mi, i = t % mi + 1;
    const SrcState* S = a.src + r;
    if (i > S->k_final) continue;
    const double n_i = (i == 1) ? S->bnorm : a.hist_b[(size_t)r * mi + i - 2];
    const double n_m = (i <= 2) ? S->bnorm : a.hist_b[(size_t)r * mi + i - 3];
    float d[8];
    const double inv_n = __drcp_rn(n_i), cm = (i > 1) ? n_i / n_m : 0.0, alpha = a.hist_a[(size_t)r * mi + i - 1];
    const double alpha_n = alpha * inv_n;  // as K1 forms it
    df_split(inv_n, d + 0);
    df_split(cm, d + 2);
    df_split(alpha, d + 4);
    df_split(alpha_n, d + 6);
    const double2 g = a.gco[(size_t)r * mi + i - 1];
    RegenRec<R> o;
    o.inv_n = scal<R>(inv_n, d + 0);
    o.cm = scal<R>(cm, d + 2);
    o.alpha = scal<R>(alpha, d + 4);
    o.alpha_n = scal<R>(alpha_n, d + 6);
    o.g = cx_from<R>(g.x, g.y);
    rec[t] = o;
  }
}

// Stored-basis variant of the second pass: sum[r][e] += sum_{i=1..k_r} gw[r][i-1] U_i[e],
// gw = g_i / ||U_i|| (the basis is stored unnormalised), in the arithmetic of the basis
// (FP64, or double-float with gw split into double-float pairs on the host); one read
// of the basis and one FP64 update of the sum per element.  REAL: the coefficients are
// real (a node list closed under conjugation, z_j and conj(z_j) with conj(c_j): T_k is
// real, so (conj z - T_k)^-1 e_1 = conj((z - T_k)^-1 e_1) and g = sum_j c_j y^j is real),
// two FMAs per element and basis vector instead of four.
template <typename R, bool REAL = false>
__global__ void basis_sum_kernel(const typename Store<R>::T* __restrict__ basis, int nslots,
                                 const typename Store<R>::T* __restrict__ gw, int ldg, const int* __restrict__ kr,
                                 double2* __restrict__ sum, size_t n12) {
  const int r = blockIdx.y;
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n12) return;
  const typename Store<R>::T* B = basis + (size_t)r * nslots * n12 + e;
  const typename Store<R>::T* w = gw + (size_t)r * ldg;
  Cx<R> acc = {R(0), R(0)};
  const int k = kr[r];
  for (int i = 1; i <= k; ++i) {
    const Cx<R> wi = ld<R>(w + i - 1), b = ld<R>(B + (size_t)i * n12);
    if constexpr (REAL) {
      acc.re = fma(wi.re, b.re, acc.re);
      acc.im = fma(wi.re, b.im, acc.im);
    } else {
      acc = cfma(wi, b, acc);
    }
  }
  double2 sv = sum[(size_t)r * n12 + e];
  sv.x += (double)acc.re;
  sv.y += (double)acc.im;
  sum[(size_t)r * n12 + e] = sv;
}

// Per-node solutions from a stored basis: X[r][jj][e] = sum_{i=1..k_r} Y[r][j0 + jj][i-1] U_i[e]
// for the nc nodes of a chunk (Y holds the FOM coefficients folded with 1 / ||U_i||), JT
// nodes per thread so that one read of the basis serves JT outputs; FP64 output.
template <typename R, int JT>
__global__ void basis_nodes_kernel(const typename Store<R>::T* __restrict__ basis, int nslots,
                                   const typename Store<R>::T* __restrict__ Y, int ns, int ldy,
                                   const int* __restrict__ kr, int j0, int nc, double2* __restrict__ X,
                                   size_t n12) {
  const int r = blockIdx.y, jt = blockIdx.z * JT;
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n12 || jt >= nc) return;
  const typename Store<R>::T* B = basis + (size_t)r * nslots * n12 + e;
  const typename Store<R>::T* Yr = Y + ((size_t)r * ns + j0 + jt) * ldy;
  const int k = kr[r], nj = min(JT, nc - jt);
  Cx<R> acc[JT];
#pragma unroll
  for (int q = 0; q < JT; ++q) acc[q] = {R(0), R(0)};
  for (int i = 1; i <= k; ++i) {
    const Cx<R> u = ld<R>(B + (size_t)i * n12);
#pragma unroll
    for (int q = 0; q < JT; ++q)
      if (q < nj) acc[q] = cfma(ld<R>(Yr + (size_t)q * ldy + (i - 1)), u, acc[q]);
  }
#pragma unroll
  for (int q = 0; q < JT; ++q)
    if (q < nj) X[((size_t)r * nc + jt + q) * n12 + e] = make_double2((double)acc[q].re, (double)acc[q].im);
}

// sum += (double) ssum: the double-float regeneration-pass sum into the FP64 sum
__global__ void fold_df_sum_kernel(const float4* __restrict__ ssum, double2* __restrict__ sum, size_t n) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
    const float4 v = ssum[t];
    double2 sv = sum[t];
    sv.x += (double)v.x + (double)v.y;
    sv.y += (double)v.z + (double)v.w;
    sum[t] = sv;
  }
}

// Init: U_1 = b (ring slot 1), ||b|| per source, s = c0 b, node states reset.
template <typename R>
__global__ void __launch_bounds__(NT2) lanczos_init_kernel(SolveArgs<R> a, const double2* __restrict__ b,
                                                           double2 c0) {
  using T = typename Store<R>::T;
  __shared__ double sh[NT2 / 32];
  __shared__ bool last;
  const int r = blockIdx.y;
  const size_t n12 = (size_t)12 * a.g.V;
  T* U1 = a.ring + (size_t)r * a.prm->nslots * n12 + n12;
  const size_t e = (size_t)blockIdx.x * NT2 + threadIdx.x;
  double nrm = 0.0;
  if (e < n12) {
    const double2 bv = b[(size_t)r * n12 + e];
    st<R>(U1 + e, cx_from<R>(bv.x, bv.y));
    nrm = bv.x * bv.x + bv.y * bv.y;
    if (a.sacc) a.sacc[(size_t)r * n12 + e] = make_double2(c0.x * bv.x - c0.y * bv.y, c0.x * bv.y + c0.y * bv.x);
  }
  double bs = block_sum<NT2>(nrm, sh);
  if (threadIdx.x == 0) {
    a.part2[(size_t)r * gridDim.x + blockIdx.x] = bs;
    __threadfence();
    last = (atomicAdd(a.cnt + 2 * r + 1, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double tot = sum_partials<NT2>(a.part2 + (size_t)r * gridDim.x, gridDim.x, sh);
  if (threadIdx.x != 0) return;
  a.cnt[2 * r + 1] = 0;
  SrcState* S = a.src + r;
  S->bnorm = sqrt(tot);
  S->inv_b2 = tot > 0.0 ? 1.0 / tot : 0.0;
  S->n_cur = S->bnorm;
  S->n_prev = 1.0;
  S->alpha = 0.0;
  S->iter = 1;
  set_norm_scalars<R>(S);
  S->status = OV_OK;
  S->n_act = 0;
  S->node_updates = 0.0;
  S->k_final = 0;
  S->done = 0;
  const int ns = a.prm->nshift;
  for (int j = 0; j < ns; ++j) {
    ShiftState& q = a.sh[(size_t)r * ns + j];
    q.invd = q.omega = q.zeta = make_double2(0.0, 0.0);
    q.res2 = 1.0;
    q.active = 1;
    q.last_iter = 0;
  }
  // a source whose tolerance is >= 1 needs no work (a correction right-hand side that
  // already meets tol): done before the first step, which could otherwise enlarge it
  const bool skip = a.tol_src && a.tol_src[r] >= 1.0;
  if (skip || !(S->bnorm > 0.0) || !isfinite(S->bnorm)) {
    for (int j = 0; j < ns; ++j) {
      a.sh[(size_t)r * ns + j].active = 0;
      a.sh[(size_t)r * ns + j].res2 = 0.0;
    }
    mark_done(S, a.done_count, (skip || isfinite(S->bnorm)) ? OV_OK : OV_ERR_BREAKDOWN);
  }
}

// ------------------------------------------------------ fixed-point Lanczos kernels
//
// The recurrence on integer vectors X_i (fixed.cuh), each at a power-of-two scale of its
// own.  With v_i = X_i / ||X_i||, H v_i = beta_{i-1} v_{i-1} + alpha_i v_i + beta_i v_{i+1}:
//
//   K1   w       = 2^-q H X_i / 4 - gam X_{i-1},  gam = 2^-q beta_{i-1} ||X_i|| / (4 ||X_{i-1}||)
//        a       = <X_i, w> / ||X_i||^2,          alpha_i = 4 2^q a
//   K2   X_{i+1} = 2^k (w - a X_i),               beta_i = 4 2^(q - k) ||X_{i+1}|| / ||X_i||
//
// q keeps gam at most 2 (q > 0 only while a localised source spreads); k brings
// the largest component to just below 2^58, from the bound max |w| + |a| 2^58 that K1's
// last block knows.  The inner products are sums of exact integer products (per thread),
// then FP64.
// 2^e as a double, -1022 <= e <= 1023
__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }
// floor(log2 |x|) of a normal number
__device__ __forceinline__ int exponent_of(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) - 1023; }

// Block maximum of an int; sh >= NT / 32 ints; a barrier must follow before sh is reused.
template <int NT>
__device__ __forceinline__ int block_max(int v, int* sh) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NT / 32; ++k) v = max(v, sh[k]);
  return v;
}

// Sums over a source: integers, so that atomic additions in any order give the same result.
// Blocks add into kFxBins bins (fewer collisions per address).  No block waits for the others:
// every block of the next kernel adds the bins up and forms the iteration's scalars itself,
// beside its first loads (an arrival counter, a last block's serial FP64 chain and its
// state writes took 10 us of an iteration's 21 at 8^4).  Block 0 records them.  Two slots, by
// the iteration's parity: the reader's block 0 clears the other one.
constexpr int kFxBins = 32;
constexpr int kFxWords = 6;  // K1: five words of <X, w> and the maximum; K2: four words
__device__ __forceinline__ long long* fx_bins(long long* bins, int r, int i) {
  return bins + (size_t)(2 * r + (i & 1)) * kFxBins * kFxWords;
}
__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The scalars of X_i (i >= 2) from ||X_i||^2 (K2's bins of iteration i - 1); a whole warp.
// fx_close adds what K1 does not wait for: 1 / ||X_i||^2 and, returned, beta_{i-1}.
__device__ __forceinline__ FxVec fx_vec(const SolveArgs<FX>& a, const SrcState* S, int r, int i, double* ratio, int* shift) {
  const long long* bins = fx_bins(a.bins2, r, i - 1) + (threadIdx.x & 31) * kFxWords;
  long long n[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) n[j] = warp_sum(__ldcg(bins + j));
  const FxVec p = S->vec[(i - 1) & 1];
  const int sh = p.q - S->k[(i - 1) & 1];
  FxVec v;
  v.n2 = fma((double)n[0], pow2(92), (double)n[1] * pow2(60)) + fma((double)n[2], pow2(62), (double)n[3] * pow2(30));
  *ratio = v.n2 * p.inv_n2;                // ||X_i||^2 / ||X_{i-1}||^2, 0 if beta_{i-1} is
  *shift = sh;
  const double g1 = *ratio * pow2(sh);     // beta_{i-1} ||X_i|| / (4 ||X_{i-1}||)
  v.q = max(0, exponent_of(g1));           // g1 2^-q < 2
  v.gam = fx_split(-__double2ll_rn(g1 * pow2(60 - v.q)));
  v.dia = fx_split(__double2ll_rn(a.diag4 * pow2(60 - v.q)));
  return v;
}

__device__ __forceinline__ double fx_close(FxVec* v, double ratio, int shift) {
  v->inv_n2 = __drcp_rn(v->n2);
  return sqrt(ratio) * pow2(2 + shift);
}

// What an iteration's start leaves for later kernels, by one warp per source.
__device__ __forceinline__ void fx_record(const SolveArgs<FX>& a, SrcState* S, int r, int i, FxVec v, double ratio,
                                          int shift, bool end) {
  const int lane = threadIdx.x & 31, mi = a.prm->max_iter;
  long long* z = fx_bins(a.bins2, r, i) + lane * kFxWords;
#pragma unroll
  for (int k = 0; k < kFxWords; ++k) z[k] = 0;
  if (lane != 0) return;
  if (i > 1) {
    a.hist_b[(size_t)r * mi + i - 2] = fx_close(&v, ratio, shift);
    S->vec[i & 1] = v;
    if (i <= mi) a.hist_n2[(size_t)r * mi + i - 1] = v.n2;
  }
  __threadfence();  // a check running beside this reads the history once it1 is 0
  *(volatile int*)&S->it1 = end ? 0 : i;
}

// fx_begin ahead of K1 for grids of many blocks (one warp per source)
__global__ void __launch_bounds__(32) fx_begin_kernel(const __grid_constant__ SolveArgs<FX> a) {
  SrcState* S = a.src + blockIdx.x;
  if (__any_sync(0xffffffffu, S->done)) return;
  const int i = S->it2;
  double ratio = 1.0;
  int shift = 0;
  const FxVec v = i > 1 ? fx_vec(a, S, blockIdx.x, i, &ratio, &shift) : S->vec[1];
  fx_record(a, S, blockIdx.x, i, v, ratio, shift, ratio == 0.0 || i > a.prm->max_iter);
}

// A block takes one 32-site tile of `per` sources in turn (their links then come from L1).
// Bound by the wide multiply-adds (one warp instruction per cycle and SM, 1300 per 32 sites
// for the hops and 430 for the rest, half of the time) and the L2 latency of the neighbour
// loads.  One source at 16^3 x 32: 55 us, where the FP64 kernel takes 227 us and the
// double-float one 66 us; 6 sources in one launch: 6 x 44 us (links from L1; 6 x 43 when it
// rounded down and left negations a unit short).  4 blocks per SM (64 registers): 338 ms per
// 12-source FP64 solve (with the rounding of before 334, 363 at 3, 366 at 5).  NT = 288, for small grids
// where nothing else covers it: a ninth warp forms the scalars while the others run phase 1
// (8^4, 4 sources: 8.0 -> 6.5 ms per solve against a last block's serial end); NT = 256: from
// fx_begin_kernel (formed in every block, 16^3 x 32 took 374 ms instead of 366).
template <int NT>
__global__ void __launch_bounds__(NT, NT == kFxNT ? 4 : 3) fx_lanczos_hw_kernel(const __grid_constant__ SolveArgs<FX> a,
                                                                                int nsrc, int per) {
  __shared__ int red[kFxNT / 32][kFxWords];
  __shared__ FxVec vec;
  __shared__ int stop;
  __shared__ longlong2 sm[4 * 12 * kFxTile];
  const int V = a.g.V;
  const int nb = (V + kFxTile - 1) / kFxTile, ng = gridDim.x / nb;
  const int tb = blockIdx.x / ng, r0 = blockIdx.x % ng * per;
  const size_t n12 = 12 * fx_padded(V);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int s = tb * kFxTile + lane;
  const bool in = s < V;
  const FxHops nbr = fx_hops(a.g, in ? s : 0, (wid >> 1) & 3);
  if (NT > kFxNT) cudaGridDependencySynchronize();
  for (int r = r0; r < min(nsrc, r0 + per); ++r) {
    SrcState* S = a.src + r;
    const int i = S->it2, mi = a.prm->max_iter, mask = a.prm->slot_mask, nslots = a.prm->nslots;
    // the check of earlier iterations may set `done` while this runs: one answer per block
    if (__syncthreads_or(S->done)) continue;
    FxVec next;  // the ninth warp's
    double ratio = 1.0;
    int shift = 0;
    int4* base = a.ring + (size_t)r * nslots * n12;
    const int4* Xi = base + (size_t)(i & mask) * n12;  // stored basis: slot i holds X_i
    if (NT > kFxNT && wid == kFxNT / 32) {
      next = i > 1 ? fx_vec(a, S, r, i, &ratio, &shift) : S->vec[1];
      if (lane == 0) {
        vec = next;
        stop = ratio == 0.0 || i > mi;
      }
    }
    if (NT == kFxNT && threadIdx.x == 0) {
      vec = S->vec[i & 1];
      stop = S->it1 == 0;
    }
    if (in && i <= mi && wid < kFxNT / 32) fx_phase1(Xi, a.U, wid, s, nbr, sm + (wid >> 1) * 12 * kFxTile + lane);
    __syncthreads();
    if (NT > kFxNT) cudaTriggerProgrammaticLaunchCompletion();
    if (NT > kFxNT && wid == kFxNT / 32 && tb == 0) fx_record(a, S, r, i, next, ratio, shift, stop);
    if (stop) {
      __syncthreads();
      continue;
    }
    // <X_i, w> = hh 2^62 + x1 2^30 + x2 2^32, w = wh 2^32 + wl with signed wl
    long long hh = 0, x1 = 0, x2 = 0;
    int wmax = 0;
    if (in && wid < 6) {  // components 2 wid, 2 wid + 1
      const int q = vec.q;
      const bool low = wid >= 3;
      // 2^-q diag / 4 x - gam X_{i-1} = (hh 2^60 + x 2^30) / 2^60; gamma5 = -1 on the lower spins
      const FX dg = vec.dia, nd = FX{low ? -dg.hi : dg.hi, low ? -dg.lo : dg.lo}, ngm = vec.gam;
      const size_t o = fx_index(s, 12) + 2 * wid * kFxTile;
      const int4 *xp = Xi + o, *up = base + (size_t)((i - 1) & mask) * n12 + o;
      longlong2* wp = reinterpret_cast<longlong2*>(base + (size_t)((i + 1) & mask) * n12 + o);
      int4 xb[2], ub[2];
      longlong2 t[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        xb[j] = __ldg(xp + j * kFxTile);
        ub[j] = i > 1 ? __ldg(up + j * kFxTile) : make_int4(0, 0, 0, 0);
        t[j] = fx_phase2(sm, 2 * wid + j, lane);
      }
      if (q > 0) {
        const long long rq = 1LL << (q - 1);
        for (int j = 0; j < 2; ++j) t[j] = make_longlong2((t[j].x + rq) >> q, (t[j].y + rq) >> q);
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        long long w[2] = {t[j].x, t[j].y};
        const int xv[4] = {xb[j].x, xb[j].y, xb[j].z, xb[j].w}, uv[4] = {ub[j].x, ub[j].y, ub[j].z, ub[j].w};
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          long long gh = w[c], gx = kFxHalf30;
          fx_mac(gh, gx, nd.hi, nd.lo, xv[2 * c], xv[2 * c + 1]);
          fx_mac(gh, gx, ngm.hi, ngm.lo, uv[2 * c], uv[2 * c + 1]);
          w[c] = fx_value(gh, gx);
          const int wl = (int)w[c], wh = (int)(w[c] >> 32) + (int)((unsigned)wl >> 31);
          hh += (long long)xv[2 * c] * wh;
          x1 += (long long)xv[2 * c] * wl;
          x2 += (long long)xv[2 * c + 1] * wh;
          wmax = max(wmax, abs(wh));
        }
        wp[j * kFxTile] = make_longlong2(w[0], w[1]);
      }
    } else if (wid < 6) {  // the padding of the last tile
      int4* wp = base + (size_t)((i + 1) & mask) * n12 + fx_index(s, 12) + 2 * wid * kFxTile;
      wp[0] = wp[kFxTile] = make_int4(0, 0, 0, 0);
    }
    // warp sums in words that cannot overflow 32 lanes: hh in 26 + 26 + 12 bits, the cross
    // terms (below 2^-30 of hh's weight, kept to 2^-47) in 24 + 24
    if (wid < 6) {
      const long long xs = (x2 + (x1 >> 2)) >> 16;
      int v[kFxWords];
      v[0] = __reduce_add_sync(0xffffffffu, (int)(hh & 0x3ffffff));
      v[1] = __reduce_add_sync(0xffffffffu, (int)((hh >> 26) & 0x3ffffff));
      v[2] = __reduce_add_sync(0xffffffffu, (int)(hh >> 52));
      v[3] = __reduce_add_sync(0xffffffffu, (int)(xs & 0xffffff));
      v[4] = __reduce_add_sync(0xffffffffu, (int)(xs >> 24));
      v[5] = __reduce_max_sync(0xffffffffu, wmax);
      if (lane == 0)
#pragma unroll
        for (int k = 0; k < kFxWords; ++k) red[wid][k] = v[k];
    }
    __syncthreads();
    // red is next written after the next source's first barrier
    if (wid == 0 && lane < kFxWords) {
      long long t = red[0][lane];
#pragma unroll
      for (int k = 1; k < 6; ++k) t = lane == 5 ? max(t, (long long)red[k][lane]) : t + red[k][lane];
      long long* d = fx_bins(a.bins1, r, i) + (tb % kFxBins) * kFxWords + lane;
      if (lane == 5)
        atomicMax(d, t);
      else
        atomicAdd((unsigned long long*)d, (unsigned long long)t);
    }
  }
}

// HBM-bound (576 B per site and source): two reads, one write, an exact integer norm; one
// wave of blocks, two elements in flight per thread (19.0 us for one source at 16^3 x 32).
// Warp 0 forms alpha and the scale from K1's sums beside the block's first loads.
template <>
__global__ void __launch_bounds__(NT2, 4) lanczos_update_kernel<FX>(SolveArgs<FX> a) {
  __shared__ long long red[NT2 / 32][4];
  __shared__ FX alf_sh;
  __shared__ int k_sh;
  const int r = blockIdx.y;
  SrcState* S = a.src + r;
  cudaGridDependencySynchronize();
  const int i = S->it1, mask = a.prm->slot_mask, nslots = a.prm->nslots;
  if (__syncthreads_or(S->done) || i < 1) return;
  const size_t n12 = 12 * fx_padded(a.g.V);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int4* Xi = a.ring + ((size_t)r * nslots + (i & mask)) * n12;
  int4* W = a.ring + ((size_t)r * nslots + ((i + 1) & mask)) * n12;
  const size_t e0 = (size_t)blockIdx.x * NT2 + threadIdx.x, gs = (size_t)gridDim.x * NT2;
  constexpr int B = 2;  // elements in flight per thread
  int4 xb[B], wb[B];
  auto load = [&](size_t eb) {
#pragma unroll
    for (int t = 0; t < B; ++t) {
      const bool in = eb + t * gs < n12;
      xb[t] = in ? __ldg(Xi + eb + t * gs) : make_int4(0, 0, 0, 0);
      wb[t] = in ? W[eb + t * gs] : make_int4(0, 0, 0, 0);  // int64 pair (re, im)
    }
  };
  load(e0);
  if (wid == 0) {
    const long long* bins = fx_bins(a.bins1, r, i) + lane * kFxWords;
    long long t[kFxWords];
#pragma unroll
    for (int j = 0; j < 5; ++j) t[j] = warp_sum(__ldcg(bins + j));
    const int m = __reduce_max_sync(0xffffffffu, (int)__ldcg(bins + 5));
    const double dot = fma((double)t[2], pow2(114), fma((double)t[1], pow2(88), (double)t[0] * pow2(62))) +
                       fma((double)t[4], pow2(72), (double)t[3] * pow2(48));
    const double a1 = dot * S->vec[i & 1].inv_n2;
    // |X_{i+1}| <= 2^k bound < 2^58
    const double bound = fma(fabs(a1), pow2(kFxBits), (double)(m + 1LL) * 4294967296.0);
    const int k = kFxBits - 1 - exponent_of(bound);
    if (lane == 0) {
      alf_sh = fx_split(-__double2ll_rn(a1 * pow2(59)));  // |a1| < 4 (fixed.cuh): a unit more than gam's
      k_sh = k;
    }
    if (blockIdx.x == 0) {
      long long* z = fx_bins(a.bins1, r, i + 1) + lane * kFxWords;
#pragma unroll
      for (int j = 0; j < kFxWords; ++j) z[j] = 0;
      if (lane == 0) {
        S->k[i & 1] = k;
        a.hist_a[(size_t)r * a.prm->max_iter + (i - 1)] = a1 * pow2(2 + S->vec[i & 1].q);
        S->it2 = i + 1;
      }
    }
  }
  __syncthreads();
  const FX alf = alf_sh;
  const int kl = max(k_sh, 0), kr = max(-k_sh, 0);  // below 32 both
  // 2^k y rounded, plus 2^29 (hi then comes out of a plain shift by 30)
  const long long rnd = (kr > 0 ? 1LL << (kr - 1) : 0) + (kFxHalf30 << kr);
  // ||X||^2 = n[0] 2^92 + n[1] 2^60 + n[2] 2^62 + n[3] 2^30: high and low words of the hi hi
  // products and of the rest, whose sums over the largest lattice stay within 63 bits (2^33
  // reals, one addition of at most 2^32 per four of them) however the components are correlated
  long long n[4] = {0, 0, 0, 0};
  for (size_t eb = e0; eb < n12; eb += B * gs) {
    if (eb != e0) load(eb);
    long long hh = 0, xx = 0, ll = 0;  // of up to 4 reals: hh 2^60 + xx 2^30 + ll
#pragma unroll
    for (int t = 0; t < B; ++t) {
      const int xv[4] = {xb[t].x, xb[t].y, xb[t].z, xb[t].w};
      const long long wv[2] = {(long long)(((unsigned long long)(unsigned)wb[t].y << 32) | (unsigned)wb[t].x),
                               (long long)(((unsigned long long)(unsigned)wb[t].w << 32) | (unsigned)wb[t].z)};
      FX o[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        // w - a X = w + 2 hi X.hi + (hi X.lo + lo X.hi) / 2^29
        long long ah = wv[c] + (long long)alf.hi * (2 * xv[2 * c]), ax = kFxHalf30 >> 1;
        ax += (long long)alf.hi * xv[2 * c + 1];
        ax += (long long)alf.lo * xv[2 * c];
        const long long y = fx_shr(fx_shl(ah + (ax >> 29), kl) + rnd, kr);
        o[c].hi = (int)(y >> 30);
        o[c].lo = ((int)y & 0x3fffffff) - (1 << 29);
        hh += (long long)o[c].hi * o[c].hi;
        xx += (long long)o[c].hi * (2 * o[c].lo);
        ll += (long long)o[c].lo * o[c].lo;
      }
      if (eb + t * gs < n12) W[eb + t * gs] = make_int4(o[0].hi, o[0].lo, o[1].hi, o[1].lo);
    }
    xx += ll >> 30;
    n[0] += hh >> 32;
    n[1] += (unsigned)hh;
    n[2] += xx >> 32;
    n[3] += (unsigned)xx;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    n[j] = warp_sum(n[j]);
    if (lane == 0) red[wid][j] = n[j];
  }
  __syncthreads();
  cudaTriggerProgrammaticLaunchCompletion();
  if (threadIdx.x < 4) {
    long long t = 0;
#pragma unroll
    for (int j = 0; j < NT2 / 32; ++j) t += red[j][lane];
    atomicAdd((unsigned long long*)fx_bins(a.bins2, r, i) + (blockIdx.x % kFxBins) * kFxWords + lane,
              (unsigned long long)t);
  }
}

// node_check_kernel for the fixed-point forms.  It runs beside the iterations that follow it
// (run_iterations), so that it looks at a fixed count of them: the recorded ones of whole
// check intervals.  `final` (nothing runs beside it) takes them all, with the last beta from
// K2's sums; so does a check that finds a source at the end of its Krylov space (beta = 0).
// The count of iterations a source ends with does not depend on which check finds it.
// With per-node vectors it also leaves what fx_node_update_kernel needs of these iterations,
// with a stored basis the rows of every node's factorisation, stopped ones included.
constexpr int kNodeRun = 32;   // most iterations between two updates (17: a check may run late)
constexpr int kNodeBatch = 8;  // iterations fx_node_update_kernel takes at a time
__global__ void __launch_bounds__(NT1) fx_node_check_kernel(const __grid_constant__ SolveArgs<FX> a, int final) {
  __shared__ int last_sh[NT1 / 32];
  const int r = blockIdx.y;
  SrcState* S = a.src + r;
  const bool over = S->done;  // set by this kernel only
  if (__syncthreads_or(over)) {
    if (a.pv && threadIdx.x == 0) S->upd_n = 0;
    return;
  }
  const int ns = a.prm->nshift, mi = a.prm->max_iter;
  __shared__ int it_sh;  // one answer for all threads: the iterations go on beside this
  if (threadIdx.x == 0) it_sh = *(volatile int*)&S->it2;
  __syncthreads();
  const int ran = it_sh - 1;  // iterations whose alpha is recorded; their betas but the last
  int upto = ran / kNodeCheck * kNodeCheck - 1;
  if (__syncthreads_or(*(volatile int*)&S->it1 == 0 && ran >= 1)) upto = ran;  // K1 recorded the last beta, too
  __threadfence();
  if (final) {
    upto = ran;
    if (ran >= 1 && threadIdx.x < 32) {
      double ratio;
      int shift;
      FxVec v = fx_vec(a, S, r, ran + 1, &ratio, &shift);
      if (threadIdx.x == 0) {
        a.hist_b[(size_t)r * mi + ran - 1] = fx_close(&v, ratio, shift);
        if (ran < mi) a.hist_n2[(size_t)r * mi + ran] = v.n2;
        S->iter = ran + 1;
      }
    }
    __syncthreads();
  }
  const double tol2 = a.prm->tol * a.prm->tol, inv_b2 = S->inv_b2;
  const double* ha = a.hist_a + (size_t)r * mi;
  const double* hb = a.hist_b + (size_t)r * mi;
  const int i0 = S->upd_i + S->upd_n;  // the iteration all nodes go on with
  if (a.pv) upto = min(upto, i0 + kNodeRun - 1);
  int still = 0, last = 0, run = 0;
  double updates = 0.0;
  for (int j0 = 0; j0 < ns; j0 += NT1) {
    const int j = j0 + threadIdx.x;
    bool act = false;
    if (j < ns) {
      ShiftState& q = a.sh[(size_t)r * ns + j];
      if (a.pv) a.act_idx[(size_t)r * ns + j] = 0;
      act = q.active != 0;
      if (act || !a.pv) {
        const double2 zj = a.z[(size_t)r * ns + j];
        double2* co = a.pv ? a.nco + ((size_t)r * ns + j) * kNodeRun * 3 : nullptr;
        double2 invd = q.invd, om = q.omega, zeta = q.zeta;
        double res2 = q.res2;
        int end = act ? max(upto, q.last_iter) : q.last_iter;
        for (int i = i0; i <= upto; ++i) {
          const double alpha = __ldcg(ha + i - 1), beta = __ldcg(hb + i - 1);
          double2 d, l = make_double2(0.0, 0.0);
          if (i == 1) {
            d = make_double2(zj.x - alpha, zj.y);
            om = make_double2(S->bnorm, 0.0);
          } else {
            const double bp = __ldcg(hb + i - 2);
            const double b2 = bp * bp;
            d = make_double2(zj.x - alpha - b2 * invd.x, zj.y - b2 * invd.y);
            l = make_double2(-bp * invd.x, -bp * invd.y);
            om = cmul(make_double2(bp * invd.x, bp * invd.y), om);
          }
          const double inv = __drcp_rn(d.x * d.x + d.y * d.y);
          invd = make_double2(d.x * inv, -d.y * inv);
          zeta = cmul(om, invd);
          if (co) {
            double2* p = co + 3 * (i - i0);
            p[0] = l;
            p[1] = cmul(a.c[(size_t)r * ns + j], zeta);
            p[2] = zeta;
          } else {
            const size_t o = ((size_t)r * mi + i - 1) * ns + j;
            a.fd[o] = invd;
            a.fz[o] = zeta;
          }
          if (!act) continue;
          res2 = beta * beta * inv_b2 * (zeta.x * zeta.x + zeta.y * zeta.y);
          if (res2 <= tol2 || beta == 0.0) {
            if (beta == 0.0) res2 = 0.0;
            act = false;
            end = i;
            if (co) break;
          }
        }
        q.invd = invd;
        q.omega = om;
        q.zeta = zeta;
        q.res2 = res2;
        if (co) {
          const int n = end - q.last_iter;
          a.act_idx[(size_t)r * ns + j] = n;
          // a batch's rest: p = 0 - (-1) p, nothing added
          for (int t = n; t % kNodeBatch != 0; ++t) {
            co[3 * t] = make_double2(-1.0, 0.0);
            co[3 * t + 1] = co[3 * t + 2] = make_double2(0.0, 0.0);
          }
          updates += n;
          run = max(run, n);
        }
        q.last_iter = end;
        q.active = act ? 1 : 0;
      }
      last = max(last, q.last_iter);
    }
    still += __syncthreads_count(act);
  }
  last = block_max<NT1>(last, last_sh);
  if (a.pv) {
    __syncthreads();
    run = block_max<NT1>(run, last_sh);
    if (updates > 0.0) atomicAdd(&S->node_updates, updates);  // whole numbers: exact in any order
    for (int t = threadIdx.x; t < run; t += NT1)
      a.nin[(size_t)r * kNodeRun + t] = 1.0 / sqrt(__ldcg(a.hist_n2 + (size_t)r * mi + i0 + t - 1));
    if (threadIdx.x == 0) {
      S->upd_i = i0;
      S->upd_n = run;
      if (still == 0) {
        S->iter = last + 1;
        mark_done(S, a.done_count, OV_OK);
      }
    }
    return;
  }
  if (threadIdx.x == 0) S->upd_i = max(i0, upto + 1);
  if (threadIdx.x == 0 && ns > 0 && still == 0) {
    // The next multiple of the check interval after the last node's iteration, an even count:
    // the iterates of an indefinite operator alternate, and the sum over an odd number of
    // vectors is several times further off (8^4: 2.9e-13 with 367, 3.5e-14 with 368).
    S->iter = min(ran, (last + kNodeCheck) / kNodeCheck * kNodeCheck) + 1;
    mark_done(S, a.done_count, OV_OK);
  }
}

// OV_MODE_FP64 in fixed point: p = v_i - l_{i-1} p, s += c_j zeta_i p, x_j += zeta_i p in FP64 for
// the iterations that fx_node_check_kernel has just looked at, v_i = X_i / ||X_i||.  Runs beside
// the next iterations.  Bound by the FP64 pipe (8 FMAs per node, iteration and element, 12 with
// x_j); the p of a node stay in registers over a batch of iterations, an eighth of the traffic of
// an update per iteration.  The nodes of small vectors go over the grid's third dimension as in
// K2 (k2_groups).  4^4, 1 source, 32 nodes, against K1 and K2 in FP64 with K2 in node groups:
// 6790 -> 3245 us per solve.
template <bool X>
__global__ void __launch_bounds__(256, 2) fx_node_update_kernel(const __grid_constant__ SolveArgs<FX> a) {
  const int r = blockIdx.y, z = blockIdx.z, nz = gridDim.z, V = a.g.V, ns = a.prm->nshift;
  const SrcState* S = a.src + r;
  const int run = S->upd_n, i0 = S->upd_i, mask = a.prm->slot_mask;
  const size_t np = 12 * fx_padded(V), n12 = (size_t)12 * V;
  const size_t e = (size_t)blockIdx.x * 256 + threadIdx.x;
  const size_t tk = e / kFxTile, site = tk / 12 * kFxTile + e % kFxTile, pl = tk % 12 * V + site;
  if (run == 0 || e >= np || site >= V) return;
  const int4* B = a.ring + (size_t)r * a.prm->nslots * np + e;
  const int* cnt = a.act_idx + (size_t)r * ns;
  double sre = 0.0, sim = 0.0;
  for (int b = 0; b < run; b += kNodeBatch) {
    double2 v[kNodeBatch];
#pragma unroll
    for (int t = 0; t < kNodeBatch; ++t) {
      v[t] = make_double2(0.0, 0.0);
      if (b + t < run) {
        const int4 x = __ldg(B + (size_t)((i0 + b + t) & mask) * np);
        const double in = __ldg(a.nin + (size_t)r * kNodeRun + b + t);
        v[t] = make_double2(fma((double)x.x, pow2(30), (double)x.y) * in, fma((double)x.z, pow2(30), (double)x.w) * in);
      }
    }
    for (int j = z; j < ns; j += nz) {
      if (__ldg(cnt + j) <= b) continue;
      const size_t rj = (size_t)r * ns + j;
      const double2* co = a.nco + (rj * kNodeRun + b) * 3;
      double2* P = a.pv + rj * np + e;
      double2 p = make_double2(0.0, 0.0), x = p;
      if (i0 + b > 1) p = *P;
      if (X) x = a.xv[rj * n12 + pl];
#pragma unroll
      for (int t = 0; t < kNodeBatch; ++t) {
        const double2 l = __ldg(co + 3 * t), cz = __ldg(co + 3 * t + 1);
        p = make_double2(fma(l.y, p.y, fma(-l.x, p.x, v[t].x)), fma(-l.y, p.x, fma(-l.x, p.y, v[t].y)));
        sre = fma(-cz.y, p.y, fma(cz.x, p.x, sre));
        sim = fma(cz.y, p.x, fma(cz.x, p.y, sim));
        if (X) {
          const double2 zt = __ldg(co + 3 * t + 2);
          x = make_double2(fma(-zt.y, p.y, fma(zt.x, p.x, x.x)), fma(zt.y, p.x, fma(zt.x, p.y, x.y)));
        }
      }
      *P = p;
      if (X) a.xv[rj * n12 + pl] = x;
    }
  }
  double2* s = (z == 0 ? a.sacc + (size_t)r * n12 : a.sgrp + ((size_t)r * (nz - 1) + z - 1) * n12) + pl;
  const double2 sv = *s;
  *s = make_double2(sv.x + sre, sv.y + sim);
}

// As the generic init, with the largest component of b for the scale of X_1 (written by
// fx_quantize_kernel).
template <>
__global__ void __launch_bounds__(NT2) lanczos_init_kernel<FX>(SolveArgs<FX> a, const double2* __restrict__ b,
                                                               double2 c0) {
  __shared__ double sh[NT2 / 32];
  __shared__ int shi[NT2 / 32];
  __shared__ bool last;
  __shared__ double tot_sh;
  const int r = blockIdx.y;
  const size_t n12 = (size_t)12 * a.g.V;
  const size_t e = (size_t)blockIdx.x * NT2 + threadIdx.x;
  double nrm = 0.0;
  int mx = 0;
  if (e < n12) {
    const double2 bv = b[(size_t)r * n12 + e];
    nrm = bv.x * bv.x + bv.y * bv.y;
    mx = max(__double2hiint(bv.x) & 0x7fffffff, __double2hiint(bv.y) & 0x7fffffff);  // ordered as |b|
    if (a.sacc) a.sacc[(size_t)r * n12 + e] = make_double2(c0.x * bv.x - c0.y * bv.y, c0.x * bv.y + c0.y * bv.x);
  }
  const double bs = block_sum<NT2>(nrm, sh);
  mx = block_max<NT2>(mx, shi);
  if (threadIdx.x == 0) {
    a.part2[(size_t)r * gridDim.x + blockIdx.x] = bs;
    atomicMax(fx_bins(a.bins1, r, 0) + 5, (long long)mx);
    __threadfence();
    last = (atomicAdd(a.cnt + 2 * r + 1, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const double t = sum_partials<NT2>(a.part2 + (size_t)r * gridDim.x, gridDim.x, sh);
  if (threadIdx.x == 0) tot_sh = t;
  __syncthreads();
  const double tot = tot_sh, bnorm = sqrt(tot);
  SrcState* S = a.src + r;
  const int ns = a.prm->nshift;
  const bool skip = !(bnorm > 0.0) || !isfinite(bnorm);
  for (int j = threadIdx.x; j < ns; j += NT2) {
    ShiftState& q = a.sh[(size_t)r * ns + j];
    q.invd = q.omega = q.zeta = make_double2(0.0, 0.0);
    q.res2 = skip ? 0.0 : 1.0;
    q.active = skip ? 0 : 1;
    q.last_iter = 0;
  }
  if (threadIdx.x != 0) return;
  a.cnt[2 * r + 1] = 0;
  S->bnorm = bnorm;
  S->inv_b2 = tot > 0.0 ? 1.0 / tot : 0.0;
  S->n_cur = bnorm;
  S->n_prev = 1.0;
  S->alpha = 0.0;
  S->iter = 1;
  long long* mb = fx_bins(a.bins1, r, 0) + 5;
  const int m = (int)__ldcg(mb);
  *mb = 0;
  S->e_in = kFxBits - 1 - ((m >> 20) - 1023);
  FxVec v;
  v.n2 = ldexp(tot, 2 * S->e_in);
  v.inv_n2 = 1.0 / v.n2;
  v.gam = FX{0, 0};
  v.dia = fx_split(__double2ll_rn(a.diag4 * pow2(60)));
  v.q = 0;
  S->vec[1] = v;
  S->it1 = 0;
  S->it2 = 1;
  S->upd_i = 1;
  S->upd_n = 0;
  a.hist_n2[(size_t)r * a.prm->max_iter] = v.n2;
  S->status = OV_OK;
  S->n_act = 0;
  S->node_updates = 0.0;
  S->k_final = 0;
  S->done = 0;
  if (skip) mark_done(S, a.done_count, isfinite(bnorm) ? OV_OK : OV_ERR_BREAKDOWN);
}

// X_1 = b 2^e_in, rounded to integers
__global__ void __launch_bounds__(NT2) fx_quantize_kernel(const __grid_constant__ SolveArgs<FX> a,
                                                          const double2* __restrict__ b) {
  const int r = blockIdx.y, V = a.g.V;
  const SrcState* S = a.src + r;
  if (S->done) return;
  const size_t n12 = 12 * fx_padded(V);
  const int e_in = S->e_in;
  int4* X1 = a.ring + ((size_t)r * a.prm->nslots + 1) * n12;
  for (size_t e = (size_t)blockIdx.x * NT2 + threadIdx.x; e < n12; e += (size_t)gridDim.x * NT2) {
    const size_t tk = e / kFxTile;
    const size_t site = tk / 12 * kFxTile + e % kFxTile;
    double2 v = make_double2(0.0, 0.0);
    if (site < V) v = b[((size_t)r * 12 + tk % 12) * V + site];
    const FX re = fx_split(__double2ll_rn(ldexp(v.x, e_in))), im = fx_split(__double2ll_rn(ldexp(v.y, e_in)));
    X1[e] = make_int4(re.hi, re.lo, im.hi, im.lo);
  }
}

// Coefficients y = (z_j - T_k)^-1 e_1 ||b|| of every node, one thread per node, from the rows of
// its LDL^T that the node checks left (fd, fz); rows behind the last check, at most a check
// interval of them, come first.
//   y_k = zeta_k,  y_i = zeta_i + beta_i / d_i y_{i+1};   fz[i] becomes y_i / ||X_i||
// A serial chain of two FMAs a step; rows come a batch ahead, the scalars from shared memory.
// (A factorisation from the last row up, which needs no stored rows, has a reciprocal in the
// chain: 280 us for 352 steps.)
constexpr int kCoefChunk = 512;
__global__ void __launch_bounds__(32) fx_node_coef_kernel(const __grid_constant__ SolveArgs<FX> a, int ns) {
  __shared__ double sa[kCoefChunk], sb[kCoefChunk];
  const int r = blockIdx.y, lane = threadIdx.x, j = min(blockIdx.x * 32 + lane, ns - 1);
  const bool on = blockIdx.x * 32 + lane < ns;
  const SrcState* S = a.src + r;
  const int mi = a.prm->max_iter, k = S->iter - 1;
  const double *al = a.hist_a + (size_t)r * mi, *be = a.hist_b + (size_t)r * mi, *n2 = a.hist_n2 + (size_t)r * mi;
  double2 *fd = a.fd + (size_t)r * mi * ns + j, *fz = a.fz + (size_t)r * mi * ns + j;
  const double2 z = a.z[(size_t)r * ns + j];
  for (int i = S->upd_i; i <= k; ++i) {
    double2 d = make_double2(z.x - al[i - 1], z.y), om = make_double2(S->bnorm, 0.0);
    if (i > 1) {
      const double bp = be[i - 2], b2 = bp * bp;
      const double2 g = fd[(size_t)(i - 2) * ns], zp = fz[(size_t)(i - 2) * ns];
      d = make_double2(d.x - b2 * g.x, d.y - b2 * g.y);
      om = make_double2(bp * zp.x, bp * zp.y);
    }
    const double inv = __drcp_rn(d.x * d.x + d.y * d.y);
    const double2 g = make_double2(d.x * inv, -d.y * inv);
    __syncwarp();  // lanes beyond ns share the last node's rows
    if (on) {
      fd[(size_t)(i - 1) * ns] = g;
      fz[(size_t)(i - 1) * ns] = cmul(om, g);
    }
    __syncwarp();
  }
  constexpr int B = 8;
  double2 y = make_double2(0.0, 0.0), g[B], zt[B];
  auto load = [&](int i) {  // rows i - 1, i - 2, ...
#pragma unroll
    for (int t = 0; t < B; ++t) {
      const size_t o = (size_t)max(i - 1 - t, 0) * ns;
      g[t] = fd[o];
      zt[t] = fz[o];
    }
  };
  if (k > 0) load(k);
  for (int hi = k; hi > 0; hi -= kCoefChunk) {
    const int lo = max(0, hi - kCoefChunk);
    __syncwarp();
    for (int i = lo + lane; i < hi; i += 32) {
      sa[i - lo] = rsqrt(n2[i]);
      sb[i - lo] = i + 1 < k ? be[i] : 0.0;
    }
    __syncwarp();
    for (int i0 = hi; i0 > lo; i0 -= B) {
      double2 gb[B], zb[B];
#pragma unroll
      for (int t = 0; t < B; ++t) {
        const double b = i0 - t > lo ? sb[i0 - 1 - t - lo] : 0.0;
        gb[t] = make_double2(b * g[t].x, b * g[t].y);
        zb[t] = zt[t];
      }
      load(i0 - min(B, i0 - lo));
#pragma unroll
      for (int t = 0; t < B; ++t) {
        if (i0 - t <= lo) break;
        const double rn = sa[i0 - 1 - t - lo];
        y = make_double2(fma(-gb[t].y, y.y, fma(gb[t].x, y.x, zb[t].x)), fma(gb[t].y, y.x, fma(gb[t].x, y.y, zb[t].y)));
        if (on) fz[(size_t)(i0 - 1 - t) * ns] = make_double2(y.x * rn, y.y * rn);
      }
    }
  }
}

// Coefficients of a sum over basis vectors as integers, a scale per group of vectors: up to the
// 1st, 2nd, 4th, 8th and 64th one, then 256 at a time.  G_i = g_i / ||X_i|| falls by orders of
// magnitude while a point source spreads (||X_1|| is one component, ||X_i|| as many as the source
// has reached); with one scale for all, each of the later vectors' components was rounded to
// a unit of the first one's coefficient: 2.3e-12 of a sum over the 16^4 lattice, now 8e-16 as
// with FP64 vectors.  Few groups, since each costs a conversion to FP64 per sum.
// A group's sum is one of n terms of at most 2^bits 2^58 / 2^60 (two per vector if complex)
// below 2^62: bits = 64 - log2 n, 59 at most for the cross terms' sake, one less if complex.
constexpr int kFxGroup = 256;
__host__ __device__ constexpr int fx_group_end(int g) { return g < 4 ? 1 << g : 64 + kFxGroup * (g - 4); }
constexpr int fx_groups(int k) { return 5 + (k + kFxGroup - 1) / kFxGroup; }  // at most, for k vectors

// out = w[0..k) in integers, a warp per group; scale: what undoes each group's
template <int NT, typename F>
__device__ __forceinline__ void fx_quantise(F w, int k, bool complex_sum, int4* out, double* scale) {
  const int lane = threadIdx.x & 31;
  for (int g = threadIdx.x >> 5;; g += NT / 32) {
    const int i0 = g > 0 ? fx_group_end(g - 1) : 0, end = min(k, fx_group_end(g));
    if (i0 >= k) break;
    int hi = 0;  // high word of the largest |re|, |im|
    for (int i = i0 + lane; i < end; i += 32) {
      const double2 v = w(i);
      hi = max(hi, max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff));
    }
    const int bits = min(59, 32 + __clz(end - i0 - 1)) - (complex_sum ? 1 : 0);
    const int m = __reduce_max_sync(0xffffffffu, hi) >> 20;
    const int e = m > 0 && m < 0x7ff ? bits - 1 - (m - 1023) : bits - 1;
    for (int i = i0 + lane; i < end; i += 32) {
      const double2 v = w(i);
      const FX re = fx_split(__double2ll_rn(ldexp(v.x, e))), im = fx_split(__double2ll_rn(ldexp(v.y, e)));
      out[i] = make_int4(re.hi, re.lo, im.hi, im.lo);
    }
    if (lane == 0) scale[g] = ldexp(1.0, 60 - e);
  }
}

struct FxSumInfo {
  int k, real;
};

// g[r][i] = sum_j c_j Y[r][i][j], a warp per i
__global__ void __launch_bounds__(256) fx_sum_nodes_kernel(const __grid_constant__ SolveArgs<FX> a, int ns,
                                                           const double2* __restrict__ Y, double2* __restrict__ g) {
  const int r = blockIdx.y, mi = a.prm->max_iter, k = a.src[r].iter - 1, lane = threadIdx.x & 31;
  const double2* c = a.c + (size_t)r * ns;
  for (int i = blockIdx.x * 8 + (threadIdx.x >> 5); i < k; i += gridDim.x * 8) {
    const double2* y = Y + ((size_t)r * mi + i) * ns;
    double2 t = make_double2(0.0, 0.0);
    for (int j = lane; j < ns; j += 32) {
      const double2 v = cmul(c[j], y[j]);
      t.x += v.x;
      t.y += v.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      t.x += __shfl_xor_sync(0xffffffffu, t.x, o);
      t.y += __shfl_xor_sync(0xffffffffu, t.y, o);
    }
    if (lane == 0) g[(size_t)r * mi + i] = t;
  }
}

// G = g in integers, one block per source.  Real coefficients (of unit vectors, up to rounding)
// come from a node list closed under conjugation (basis_sum_kernel).
constexpr int kCoefNT = 256;
__global__ void __launch_bounds__(kCoefNT) fx_sum_quant_kernel(const __grid_constant__ SolveArgs<FX> a,
                                                               const double2* __restrict__ g, int4* __restrict__ G,
                                                               double* __restrict__ scale, int ng,
                                                               FxSumInfo* __restrict__ info) {
  __shared__ int sh[2][kCoefNT / 32];
  const int r = blockIdx.x, mi = a.prm->max_iter, k = a.src[r].iter - 1;
  const double2* gr = g + (size_t)r * mi;
  const double* n2 = a.hist_n2 + (size_t)r * mi;
  int mr = 0, mm = 0;  // high words of the largest |re|, |im|
  for (int i = threadIdx.x; i < k; i += kCoefNT) {
    const double n = sqrt(n2[i]);
    mr = max(mr, __double2hiint(gr[i].x * n) & 0x7fffffff);
    mm = max(mm, __double2hiint(gr[i].y * n) & 0x7fffffff);
  }
  mr = block_max<kCoefNT>(mr, sh[0]);
  mm = block_max<kCoefNT>(mm, sh[1]);
  const bool real = __hiloint2double(mm, 0) <= 1e-14 * __hiloint2double(mr, 0);
  fx_quantise<kCoefNT>([&](int i) { return gr[i]; }, k, !real, G + (size_t)r * mi, scale + (size_t)r * ng);
  if (threadIdx.x == 0) info[r] = {k, real ? 1 : 0};
}

// Yq[r][j][i] = Y[r][i][j] in integers, one block per (node, source)
__global__ void __launch_bounds__(128) fx_node_quant_kernel(const __grid_constant__ SolveArgs<FX> a, int ns,
                                                            const double2* __restrict__ Y, int4* __restrict__ Yq,
                                                            double* __restrict__ scale, int ng) {
  const int r = blockIdx.y, j = blockIdx.x, mi = a.prm->max_iter, k = a.src[r].iter - 1;
  const double2* y = Y + (size_t)r * mi * ns + j;
  const size_t o = (size_t)r * ns + j;
  fx_quantise<128>([&](int i) { return y[(size_t)i * ns]; }, k, false, Yq + o * mi, scale + o * ng);
}

// K basis vectors' products, their cross terms within 63 bits, added to re and im in units of
// 2^60 over the scales.
template <bool REAL, int K>
__device__ __forceinline__ void fx_sum_group(const int4* __restrict__ w, const int4* __restrict__ B, size_t n12, int n,
                                             long long& re, long long& im) {
  long long rx = kFxHalf30, ix = kFxHalf30;
#pragma unroll
  for (int i = 0; i < K; ++i) {
    if (i < n) {
      const int4 g = __ldg(w + i), x = __ldg(B + (size_t)i * n12);
      fx_mac(re, rx, g.x, g.y, x.x, x.y);
      fx_mac(im, ix, g.x, g.y, x.z, x.w);
      if (!REAL) {
        fx_mac(re, rx, -g.z, -g.w, x.z, x.w);
        fx_mac(im, ix, g.z, g.w, x.x, x.y);
      }
    }
  }
  re += rx >> 30;
  im += ix >> 30;
}

// sum[r][e] += sum_i G_i X_i[e] (basis_sum_kernel in fixed point), G_i = g_i / ||X_i||: exact
// integer sums of a group of vectors, the groups added in FP64.  Reads 16 B per basis vector and
// element: HBM-bound.
__global__ void __launch_bounds__(256) fx_basis_sum_kernel(const int4* __restrict__ basis, int nslots,
                                                           const int4* __restrict__ G, int ldg,
                                                           const double* __restrict__ scale, int ng,
                                                           const FxSumInfo* __restrict__ info,
                                                           double2* __restrict__ sum, int V) {
  const int r = blockIdx.y;
  const size_t n12 = 12 * fx_padded(V), e = (size_t)blockIdx.x * blockDim.x + threadIdx.x, tk = e / kFxTile;
  if (e >= n12) return;
  const size_t site = tk / 12 * kFxTile + e % kFxTile;
  if (site >= V) return;
  const int4* B = basis + (size_t)r * nslots * n12 + n12 + e;
  const int4* w = G + (size_t)r * ldg;
  const double* sc = scale + (size_t)r * ng;
  const FxSumInfo f = info[r];
  constexpr int K = 8;
  double re = 0.0, im = 0.0;
  auto close = [&](int g, long long sr, long long si) {
    const double s = __ldg(sc + g);
    re = fma(s, (double)sr, re);
    im = fma(s, (double)si, im);
  };
  int g = 0, i = 0;
  if (f.k >= K) {  // the groups of 1, 1, 2 and 4, their loads together
    long long s[4][2] = {};
    fx_sum_group<false, 1>(w, B, n12, 1, s[0][0], s[0][1]);
    fx_sum_group<false, 1>(w + 1, B + n12, n12, 1, s[1][0], s[1][1]);
    fx_sum_group<false, 2>(w + 2, B + 2 * n12, n12, 2, s[2][0], s[2][1]);
    fx_sum_group<false, 4>(w + 4, B + 4 * n12, n12, 4, s[3][0], s[3][1]);
    for (; g < 4; ++g) close(g, s[g][0], s[g][1]);
    i = K;
  }
  for (; i < f.k; ++g) {
    const int end = min(f.k, fx_group_end(g));
    long long sr = 0, si = 0;
    if (f.real) {
      for (; i + K <= end; i += K) fx_sum_group<true, K>(w + i, B + (size_t)i * n12, n12, K, sr, si);
    } else {
      for (; i + K <= end; i += K) fx_sum_group<false, K>(w + i, B + (size_t)i * n12, n12, K, sr, si);
    }
    if (i < end) fx_sum_group<false, K>(w + i, B + (size_t)i * n12, n12, end - i, sr, si);
    i = end;
    close(g, sr, si);
  }
  double2* so = sum + ((size_t)r * 12 + tk % 12) * V + site;
  double2 sv = *so;
  sv.x += re;
  sv.y += im;
  *so = sv;
}

// Per-node solutions from a fixed-point basis: x_j = A + i B with A = sum_i Re(Y_i) X_i, B = sum_i
// Im(Y_i) X_i.  A node whose conjugate is also in the list needs no sums of its own: its
// coefficients are the conjugates (T_k is real), its solution A - i B.  Two nodes or pairs per
// thread (slot: node, partner or -1), Y per (source, node) with its own scales.  Bound by wide
// multiply-adds, 12 per slot, element and basis vector.  Three blocks per SM cover the FP64
// conversions between groups (8^4, 2 sources, 48 nodes, 352 vectors: 1.66 ms, 2.14 with two blocks;
// 1.89 with two and a single scale; 4.4 with every node on its own and groups of 8 summed in
// FP64).
__global__ void __launch_bounds__(256, 3) fx_basis_nodes_kernel(const int4* __restrict__ basis, int nslots,
                                                             const int4* __restrict__ Y,
                                                             const double* __restrict__ scale, int ng, int ns, int ldy,
                                                             const FxSumInfo* __restrict__ info,
                                                             const int2* __restrict__ slot, int nslot, int j0, int nc,
                                                             double2* __restrict__ X, int V) {
  constexpr int JT = 2, K = 8;
  const int r = blockIdx.y, q0 = blockIdx.z * JT;
  const size_t n12 = 12 * fx_padded(V), e = (size_t)blockIdx.x * blockDim.x + threadIdx.x, tk = e / kFxTile;
  if (e >= n12) return;
  const size_t site = tk / 12 * kFxTile + e % kFxTile;
  if (site >= V) return;
  const int4* B = basis + (size_t)r * nslots * n12 + n12 + e;
  const int k = info[r].k;
  int2 nd[JT];
  const int4* y[JT];
#pragma unroll
  for (int t = 0; t < JT; ++t) {
    nd[t] = slot[min(q0 + t, nslot - 1)];
    y[t] = Y + ((size_t)r * ns + nd[t].x) * ldy;
  }
  double s[JT][4];  // A.re, A.im, B.re, B.im
#pragma unroll
  for (int t = 0; t < JT; ++t)
#pragma unroll
    for (int c = 0; c < 4; ++c) s[t][c] = 0.0;
  long long h[JT][4] = {};
  // h += the products of vectors i .. i + n - 1 (N of them, n in a tail)
  auto add = [&](auto count, int i, int n) {
    constexpr int N = decltype(count)::value;
    long long x[JT][4];
#pragma unroll
    for (int t = 0; t < JT; ++t)
#pragma unroll
      for (int c = 0; c < 4; ++c) x[t][c] = kFxHalf30;
#pragma unroll
    for (int m = 0; m < N; ++m) {
      if (m >= n) break;
      const int4 u = __ldg(B + (size_t)(i + m) * n12);
#pragma unroll
      for (int t = 0; t < JT; ++t) {
        const int4 v = __ldg(y[t] + i + m);
        fx_mac(h[t][0], x[t][0], v.x, v.y, u.x, u.y);
        fx_mac(h[t][1], x[t][1], v.x, v.y, u.z, u.w);
        fx_mac(h[t][2], x[t][2], v.z, v.w, u.x, u.y);
        fx_mac(h[t][3], x[t][3], v.z, v.w, u.z, u.w);
      }
    }
#pragma unroll
    for (int t = 0; t < JT; ++t)
#pragma unroll
      for (int c = 0; c < 4; ++c) h[t][c] += x[t][c] >> 30;
  };
  auto close = [&](int g) {
#pragma unroll
    for (int t = 0; t < JT; ++t) {
      const double sc = __ldg(scale + ((size_t)r * ns + nd[t].x) * ng + g);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        s[t][c] = fma(sc, (double)h[t][c], s[t][c]);
        h[t][c] = 0;
      }
    }
  };
  int g = 0, i = 0;
  if (k >= K) {  // the groups of 1, 1, 2 and 4, their loads together
    add(std::integral_constant<int, 1>(), 0, 1);
    close(0);
    add(std::integral_constant<int, 1>(), 1, 1);
    close(1);
    add(std::integral_constant<int, 2>(), 2, 2);
    close(2);
    add(std::integral_constant<int, 4>(), 4, 4);
    close(3);
    g = 4;
    i = K;
  }
  for (; i < k; ++g) {
    const int end = min(k, fx_group_end(g));
    for (; i + K <= end; i += K) add(std::integral_constant<int, K>(), i, K);
    if (i < end) add(std::integral_constant<int, K>(), i, end - i);
    i = end;
    close(g);
  }
#pragma unroll
  for (int t = 0; t < JT; ++t) {
    if (q0 + t >= nslot) break;
    double2* o = X + ((size_t)r * nc * 12 + tk % 12) * V + site;
    const size_t st = (size_t)12 * V;
    o[(nd[t].x - j0) * st] = make_double2(s[t][0] - s[t][3], s[t][1] + s[t][2]);
    if (nd[t].y >= 0) o[(nd[t].y - j0) * st] = make_double2(s[t][0] + s[t][3], s[t][1] - s[t][2]);
  }
}

// second pass: U_1 = b again in ring slot 1 (the first pass overwrote the ring)
template <typename R>
__global__ void ring_reset_kernel(SolveArgs<R> a, const double2* __restrict__ b, int nsrc, int nslots) {
  using T = typename Store<R>::T;
  const size_t n12 = (size_t)12 * a.g.V;
  const size_t n = n12 * nsrc;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
    const size_t r = t / n12, e = t % n12;
    const double2 bv = b[t];
    st<R>(a.ring + r * nslots * n12 + n12 + e, cx_from<R>(bv.x, bv.y));
  }
}

// zero the per-node solution buffers (first update writes them, but a node that is
// converged at init must still read as zero)
template <typename R>
__global__ void zero_kernel(typename Store<R>::T* p, size_t n) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
    st<R>(p + t, Cx<R>{R(0), R(0)});
}

}  // namespace

// ------------------------------------------------------------------ host side

namespace {

// workspace name prefix per arithmetic type of the coefficient-space forms
template <typename R> const char* coef_tag();
template <> const char* coef_tag<double>() { return "fp64"; }
template <> const char* coef_tag<DF>() { return "df"; }
template <> const char* coef_tag<FX>() { return "fx"; }

// a complex coefficient in the storage type of the vectors (host side)
inline double2 host_store(double2 v, double2*) { return v; }
inline float4 host_store(double2 v, float4*) {
  const float rh = (float)v.x, ih = (float)v.y;
  return make_float4(rh, (float)(v.x - (double)rh), ih, (float)(v.y - (double)ih));
}

// link planes and host-side scalar conversion per arithmetic type
template <typename R> const typename Store<R>::T* solver_links(ov_ctx* ctx);
template <> const double2* solver_links<double>(ov_ctx* ctx) { return ctx->U64h; }  // -1/2 U
template <> const float2* solver_links<float>(ov_ctx* ctx) { return ctx->U32; }
template <> const float4* solver_links<DF>(ov_ctx* ctx) { return ctx->Udf; }
template <> const int4* solver_links<FX>(ov_ctx* ctx) { return ctx->Ufx; }
template <typename R> R solver_real(double x) { return (R)x; }
template <> DF solver_real<DF>(double x) {
  const float h = (float)x;
  return DF(h, (float)(x - (double)h));
}
template <> FX solver_real<FX>(double) { return FX{0, 0}; }  // SolveArgs::diag4 instead

// Elements of one Lanczos vector: 12 planes of V, padded to whole tiles in fixed point.
template <typename R> size_t vec_elems(size_t V) { return 12 * V; }
template <> size_t vec_elems<FX>(size_t V) { return 12 * fx_padded(V); }

template <typename R>
struct SolveWs {
  SolveArgs<R> a{};
  int nblk1 = 0, nblk2 = 0, nblk2u = 0;
  int ngrp = 1;  // node groups of K2 or of fx_node_update_kernel
  int slot_mask = INT_MAX;
  int nslots = 3;
  size_t nvec = 0;   // elements of one Lanczos vector (12 V, padded in fixed point)
  int nshift = 0;
  int max_iter = 0;  // row length of the per-source histories
  SolveParams* prm_dev = nullptr;
  bool defer = false;  // per-node recurrences in node_check_kernel (SolveParams::defer_nodes)
};

// The arguments of sources r0, r0 + 1, ... as a launch of their own sees them: every
// per-source array offset by r0 (kernels index sources by blockIdx.y, K1 by its
// position within a tile's group of blocks).
template <typename R>
SolveArgs<R> args_for_sources(const SolveWs<R>& w, int r0) {
  SolveArgs<R> a = w.a;
  const size_t n12 = (size_t)12 * w.a.g.V, ns = (size_t)w.nshift, r = (size_t)r0;
  a.ring += r * w.nslots * w.nvec;
  if (a.p) a.p += r * ns * n12;
  if (a.x) a.x += r * ns * n12;
  if (a.sacc) a.sacc += r * n12;
  if (a.sgrp) a.sgrp += r * (w.ngrp - 1) * n12;
  if (a.fd) a.fd += r * w.max_iter * ns;
  if (a.fz) a.fz += r * w.max_iter * ns;
  if (a.pv) a.pv += r * ns * w.nvec;
  if (a.xv) a.xv += r * ns * n12;
  if (a.nco) a.nco += r * ns * kNodeRun * 3;
  if (a.nin) a.nin += r * kNodeRun;
  if (a.ssum) a.ssum += r * n12;
  if (a.stencil) a.stencil += r * n12;
  a.src += r;
  a.sh += r * ns;
  a.z += r * ns;
  a.c += r * ns;
  a.act_idx += r * ns;
  a.act_l += r * ns;
  a.act_cz += r * ns;
  a.act_z += r * ns;
  a.part1 += r * w.nblk1;
  a.part2 += r * w.nblk2u;
  if (a.bins1) a.bins1 += r * 2 * kFxBins * kFxWords;
  if (a.bins2) a.bins2 += r * 2 * kFxBins * kFxWords;
  a.cnt += 2 * r;
  if (a.hist_a) a.hist_a += r * w.max_iter;
  if (a.hist_b) a.hist_b += r * w.max_iter;
  if (a.hist_n2) a.hist_n2 += r * w.max_iter;
  if (a.gco) a.gco += r * w.max_iter;
  if (a.rrec) a.rrec += r * w.max_iter;
  if (a.tol_src) a.tol_src += r;
  return a;
}

// Source groups of a replayed graph.  Sources are independent, so the per-iteration
// kernels of G groups can run as parallel branches of one graph: on small lattices, where
// a launch leaves SMs idle through its tail, its serial last-block step and the next
// launch's ramp, each branch fills the other's gaps; on large ones one branch's update
// kernel (bound by HBM) runs beside the other's stencil kernel (bound by the FP64 pipe or
// FP32 issue).  Auto: one group per source, at most four, when the stencil grid of all
// sources fits two waves (152 SMs x 4 blocks); else two, or six for double-float.
// (8^4, 4 sources, FP64 two-pass: 23.8 / 22.6 / 22.0 ms per apply with 1 / 2 / 4 groups;
// 16^3 x 32, 12 sources in batches of 6, 1 / 2 / 3 / 6 groups: FP64 two-pass 1385 / 1373
// / 1374 / 1375 ms, double-float 407 / 390 / 390 / 386 ms; 16^4: 533.6 / 529.8 ms.  Fixed
// point: three on large lattices -- 16^3 x 32 with 1 / 2 / 3 / 4 / 6 groups 355 / 348 / 343 / 354
// / 370 ms, 16^4 131.5 / 128.3 / 126.0 / 128.2 / 134.0 ms; 8^4 7.6 / 6.8 / 6.7 / 6.5 / 6.5 ms.)
template <typename R>
int source_groups(const ov_ctx* ctx, int nsrc, int nblk1) {
  int g = ctx->groups;
  if (g <= 0)
    g = ((size_t)nblk1 * nsrc <= (size_t)2 * 152 * 4) ? 4 : std::is_same<R, DF>::value ? 6 : std::is_same<R, FX>::value ? 3 : 2;
  return std::max(1, std::min(g, nsrc));
}

// Capture body(stream, side stream, fork and join events, args, sources) once per source group,
// each group on its own branch (forked from and joined back to the capture stream; the body
// forks and joins its side stream itself), and instantiate the graph.
template <typename R, typename F>
int capture_groups(ov_ctx* ctx, const SolveWs<R>& w, int nsrc, int G, F body, cudaGraphExec_t* exec) {
  while ((int)ctx->aux_streams.size() < 2 * G) {
    cudaStream_t st = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    if (e != cudaSuccess) return ctx_cuda(ctx, e, "cudaStreamCreate");
    ctx->aux_streams.push_back(st);
  }
  while ((int)ctx->cap_events.size() < 3 * G) {
    cudaEvent_t ev = nullptr;
    cudaError_t e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e != cudaSuccess) return ctx_cuda(ctx, e, "cudaEventCreate");
    ctx->cap_events.push_back(ev);
  }
  cudaError_t e = cudaStreamBeginCapture(ctx->cap_stream, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "cudaStreamBeginCapture");
  if (G > 1) {
    cudaEventRecord(ctx->cap_events[0], ctx->cap_stream);
    for (int g = 1; g < G; ++g) cudaStreamWaitEvent(ctx->aux_streams[g], ctx->cap_events[0], 0);
  }
  for (int g = 0; g < G; ++g) {
    const int lo = (int)((long long)nsrc * g / G), hi = (int)((long long)nsrc * (g + 1) / G);
    body(g == 0 ? ctx->cap_stream : ctx->aux_streams[g], ctx->aux_streams[G + g], ctx->cap_events[G + 2 * g],
         ctx->cap_events[G + 2 * g + 1], args_for_sources(w, lo), hi - lo);
  }
  if (G > 1) {
    for (int g = 1; g < G; ++g) {
      cudaEventRecord(ctx->cap_events[g], ctx->aux_streams[g]);
      cudaStreamWaitEvent(ctx->cap_stream, ctx->cap_events[g], 0);
    }
  }
  cudaGraph_t gph = nullptr;
  e = cudaStreamEndCapture(ctx->cap_stream, &gph);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "cudaStreamEndCapture");
  e = cudaGraphInstantiate(exec, gph, 0);
  cudaGraphDestroy(gph);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "cudaGraphInstantiate");
  return OV_OK;
}

// Node groups of K2 with per-node vectors: small vectors leave most SMs idle while each block
// runs every node through its SM's FP64 pipe.  The nodes then go over the grid's third
// dimension until it holds four blocks per SM (the parts of the weighted sum, one per group
// but the first, take at most 2.5 MB).  4^4, 1 source, 32 nodes: an iteration took 39 us with
// the 12 blocks of one group and takes 26.5 us with 32 groups.
inline int k2_groups(int nblk, int nsrc, int ns) {
  return std::max(1, std::min(ns, 4 * 152 / std::max(1, nblk * nsrc)));
}

template <typename R>
int setup_ws(ov_ctx* ctx, int nsrc, int ns, bool want_x, bool want_sacc, bool want_hist, int max_iter,
             SolveWs<R>* w, const char* tag, int nslots = 3, bool want_p = true) {
  using T = typename Store<R>::T;
  const int V = ctx->g.V;
  const size_t n12 = (size_t)12 * V;
  int st = OV_OK;
  std::string t(tag);
  w->nblk1 = (V + kSplitSites - 1) / kSplitSites;
  // K1's one-dimensional grid holds every (tile, source) pair of a launch
  if ((size_t)w->nblk1 * (size_t)nsrc > (size_t)0x7fffffff)
    return ctx_fail(ctx, OV_ERR_INVALID_ARG, "too many sources for one stencil launch at this volume");
  w->nshift = ns;
  w->max_iter = max_iter;
  // the init kernel uses the K2 partial buffer with up to ceil(12V / NT2) blocks
  w->nblk2 = (int)((n12 + NT2 - 1) / NT2);
  // K2 is a grid-stride loop: about two blocks per SM in total when the vectors are small
  // (fewer partials, short tail), up to eight (full occupancy, enough loads in flight for
  // HBM) when every thread would otherwise stride over more than 8 elements
  const size_t want = std::min<size_t>(8 * 152, std::max<size_t>(2 * 152, (size_t)nsrc * n12 / (NT2 * 8)));
  w->nblk2u = (int)std::min<size_t>(w->nblk2, std::max<size_t>(8, want / (size_t)nsrc));
  if (std::is_same<R, FX>::value)  // one wave of resident blocks at most
    w->nblk2u = (int)std::min<size_t>(w->nblk2, std::max<size_t>(8, std::min<size_t>(want, 4 * 152) / (size_t)nsrc));
  auto& a = w->a;
  w->nslots = nslots;
  w->nvec = vec_elems<R>(V);
  a.ring = (T*)ws_get(ctx, (t + ".ring").c_str(), sizeof(T) * (size_t)nslots * w->nvec * nsrc, &st);
  // per-node direction vectors: only the vector-space form (coefficient-space: none)
  a.p = (ns && want_p) ? (T*)ws_get(ctx, (t + ".p").c_str(), sizeof(T) * n12 * (size_t)nsrc * ns, &st) : nullptr;
  a.x = (want_x && ns) ? (T*)ws_get(ctx, (t + ".x").c_str(), sizeof(T) * n12 * (size_t)nsrc * ns, &st) : nullptr;
  a.sacc = want_sacc ? (double2*)ws_get(ctx, (t + ".sacc").c_str(), sizeof(double2) * n12 * nsrc, &st) : nullptr;
  w->ngrp = a.p && a.sacc ? k2_groups(w->nblk2u, nsrc, ns) : 1;
  a.sgrp = w->ngrp > 1 ? (double2*)ws_get(ctx, (t + ".sgrp").c_str(),
                                          sizeof(double2) * n12 * (size_t)nsrc * (w->ngrp - 1), &st)
                       : nullptr;
  a.src = (SrcState*)ws_get(ctx, (t + ".src").c_str(), sizeof(SrcState) * nsrc, &st);
  const size_t nsh = (size_t)nsrc * (ns > 0 ? ns : 1);
  a.sh = (ShiftState*)ws_get(ctx, (t + ".sh").c_str(), sizeof(ShiftState) * nsh, &st);
  a.z = (const double2*)ws_get(ctx, (t + ".z").c_str(), sizeof(double2) * nsh, &st);
  a.c = (const double2*)ws_get(ctx, (t + ".c").c_str(), sizeof(double2) * nsh, &st);
  a.act_idx = (int*)ws_get(ctx, (t + ".aidx").c_str(), sizeof(int) * nsh, &st);
  using CT = typename Coef<R>::T;
  a.act_l = (CT*)ws_get(ctx, (t + ".al").c_str(), sizeof(CT) * nsh, &st);
  a.act_cz = (CT*)ws_get(ctx, (t + ".acz").c_str(), sizeof(CT) * nsh, &st);
  a.act_z = (CT*)ws_get(ctx, (t + ".az").c_str(), sizeof(CT) * nsh, &st);
  a.part1 = (double*)ws_get(ctx, (t + ".part1").c_str(), sizeof(double) * (size_t)w->nblk1 * nsrc, &st);
  a.part2 = (double*)ws_get(ctx, (t + ".part2").c_str(), sizeof(double) * (size_t)w->nblk2 * nsrc, &st);
  a.bins1 = a.bins2 = nullptr;
  a.hist_n2 = nullptr;
  if (std::is_same<R, FX>::value) {
    const size_t nbins = (size_t)nsrc * 2 * kFxBins * kFxWords;
    a.bins1 = (long long*)ws_get(ctx, (t + ".bins").c_str(), sizeof(long long) * 2 * nbins, &st);
    if (a.bins1) a.bins2 = a.bins1 + nbins;
    a.hist_n2 = (double*)ws_get(ctx, (t + ".hn").c_str(), sizeof(double) * (size_t)nsrc * max_iter, &st);
  }
  a.cnt = (unsigned*)ws_get(ctx, (t + ".cnt").c_str(), sizeof(unsigned) * 2 * nsrc, &st);
  a.done_count = (int*)ws_get(ctx, (t + ".done").c_str(), sizeof(int), &st);
  if (want_hist) {
    a.hist_a = (double*)ws_get(ctx, (t + ".ha").c_str(), sizeof(double) * (size_t)nsrc * max_iter, &st);
    a.hist_b = (double*)ws_get(ctx, (t + ".hb").c_str(), sizeof(double) * (size_t)nsrc * max_iter, &st);
  } else {
    a.hist_a = a.hist_b = nullptr;
  }
  a.gco = nullptr;
  a.tol_src = nullptr;
  w->prm_dev = (SolveParams*)ws_get(ctx, (t + ".prm").c_str(), sizeof(SolveParams), &st);
  a.prm = w->prm_dev;
  a.stencil = nullptr;
  a.g = ctx->g;
  a.diag = solver_real<R>(4.0 - ctx->m0);
  a.diag4 = 0.25 * (4.0 - ctx->m0);
  a.U = solver_links<R>(ctx);
  return st;
}

// K1's grid for n sources: one dimension, the n sources of a site tile in consecutive
// blocks, so that they run side by side and the tile's links come from DRAM once for
// all of them (L2 serves the rest).  With the sources in a second grid dimension each
// source swept the whole lattice in turn and re-read the link field from DRAM (16^3 x
// 32, 6 sources: 522 MB of DRAM traffic per launch here, about 850 MB that way).  The
// time hardly moves, since neither stencil is DRAM-bound: FP64 1386 ms per 12-source
// solve either way, double-float 424.4 vs 421.7 ms.
template <typename R>
dim3 k1_grid(const SolveWs<R>& w, int n) {
  return dim3((unsigned)w.nblk1 * (unsigned)n);
}

// K1 over n sources.  Fixed point: a block takes up to kFxPerBlock sources of a tile (their
// links then come from L1), fewer while the grid would not fill the GPU; grids of at most
// three blocks per SM form the scalars themselves.  Returns the number of launches.
constexpr int kFxPerBlock = 6;

// A launch that may become resident while the kernel before it in the stream ends: K1 (288
// threads) and K2 in fixed point wait for that kernel (its memory included) before they read
// anything, and let their successor in late, when K1 has its hops and K2 its vector stored:
// blocks that wait keep others' branches out.  Solves at 4^4 with 1 source 3268 -> 2963 us, 8^4
// with 4 6570 -> 5923, 6 x 10 x 4 x 14 with 3 5700 -> 5250; let in from the start: 3033, 5908,
// 5638, and a gradient at 8^4 11690 -> 12195 instead of 11419.  With fx_begin_kernel ahead of
// K1, in large grids, it costs 3 %: ordinary launches there.
template <typename... P, typename... A>
void launch_early(void (*k)(P...), dim3 grid, int nt, cudaStream_t s, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3(nt);
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, k, P(args)...);
}

template <typename R>
int launch_k1(const SolveWs<R>& w, const SolveArgs<R>& a, int n, cudaStream_t s, bool joined = false) {
  if constexpr (std::is_same<R, FX>::value) {
    int ng = (n + kFxPerBlock - 1) / kFxPerBlock;
    while (ng < n && (size_t)w.nblk1 * ng < 4 * 4 * 152) ++ng;
    const int per = (n + ng - 1) / ng;
    const unsigned grid = (unsigned)w.nblk1 * ((n + per - 1) / per);
    if (grid <= 3 * 152) {
      // two branches meet ahead of it (`joined`): an ordinary launch
      if (joined)
        fx_lanczos_hw_kernel<kFxNT + 32><<<grid, kFxNT + 32, 0, s>>>(a, n, per);
      else
        launch_early(fx_lanczos_hw_kernel<kFxNT + 32>, grid, kFxNT + 32, s, a, n, per);
      return 1;
    }
    fx_begin_kernel<<<n, 32, 0, s>>>(a);
    fx_lanczos_hw_kernel<kFxNT><<<grid, kFxNT, 0, s>>>(a, n, per);
    return 2;
  } else {
    lanczos_hw_kernel<R><<<k1_grid(w, n), NT1, 0, s>>>(a);
    return 1;
  }
}

// K2, in FP64 and double-float with the nodes in groups
template <typename R>
void launch_k2(const SolveWs<R>& w, const SolveArgs<R>& a, int n, cudaStream_t s, bool early = false) {
  if constexpr (std::is_same<R, FX>::value) {
    if (early)
      launch_early(lanczos_update_kernel<FX>, dim3(w.nblk2u, n), NT2, s, a);
    else
      lanczos_update_kernel<R><<<dim3(w.nblk2u, n), NT2, 0, s>>>(a);
  } else
    lanczos_update_kernel<R><<<dim3(w.nblk2u, n, w.ngrp), NT2, 0, s>>>(a);
}

// Node checks and, in fixed point with per-node vectors, their updates.  Returns the number of
// launches.
template <typename R>
int launch_node_check(const SolveWs<R>& w, const SolveArgs<R>& a, int nsrc, cudaStream_t s, bool final = false) {
  if constexpr (std::is_same<R, FX>::value) {
    fx_node_check_kernel<<<dim3(1, nsrc), NT1, 0, s>>>(a, final);
    if (!a.pv) return 1;
    const dim3 grid((unsigned)((w.nvec + 255) / 256), nsrc, w.ngrp);
    if (a.xv)
      fx_node_update_kernel<true><<<grid, 256, 0, s>>>(a);
    else
      fx_node_update_kernel<false><<<grid, 256, 0, s>>>(a);
    return 2;
  } else {
    node_check_kernel<R><<<dim3(1, nsrc), NT1, 0, s>>>(a);
    return 1;
  }
}

// One Lanczos iteration (K1, K2); `it` counts iterations from 0 within the loop, and a
// scalar-only form with deferred node recurrences checks its nodes after every
// kNodeCheck-th.  Returns the number of launches.
template <typename R>
int launch_iteration(ov_ctx* ctx, const SolveWs<R>& w, int nsrc, cudaStream_t s, int it) {
  cudaEvent_t ev;
  kt_begin(ctx, KC_LANCZOS_HW, s, &ev);
  int n = launch_k1<R>(w, w.a, nsrc, s);
  kt_end(ctx, KC_LANCZOS_HW, s, ev);
  kt_begin(ctx, KC_SHIFT_UPDATE, s, &ev);
  launch_k2<R>(w, w.a, nsrc, s);
  kt_end(ctx, KC_SHIFT_UPDATE, s, ev);
  ++n;
  if (w.defer && (it + 1) % kNodeCheck == 0) {
    n += launch_node_check<R>(w, w.a, nsrc, s);
  }
  return n;
}

// Run iterations until every source is done or max_iter is reached.
template <typename R>
int run_iterations(ov_ctx* ctx, const SolveWs<R>& w, int nsrc, int nshift, int flavour, int max_iter,
                   const ov_solve_opts& o, cudaStream_t s, double* launches) {
  NvtxRange nvtx_("lanczos iterations");
  int chunk = o.check_every > 0 ? o.check_every : 32;
  // deferred node checks run after every kNodeCheck-th iteration counted from the start,
  // whatever the chunking: a replayed chunk must span whole check intervals
  if (w.defer) chunk = (chunk + kNodeCheck - 1) / kNodeCheck * kNodeCheck;
  const bool graph = o.use_graph && !ctx->timing;
  cudaGraphExec_t exec = nullptr;
  double graph_launches = 0.0;  // per replay
  if (graph) {
    const int G = source_groups<R>(ctx, nsrc, w.nblk1);
    GraphKey key{{(const void*)w.a.ring, w.a.pv ? (const void*)w.a.pv : (const void*)w.a.p,
                  w.a.pv ? (const void*)w.a.xv : (const void*)w.a.x, (const void*)w.a.sacc},
                 nsrc, nshift, flavour * 128 + G, chunk, w.nslots, w.max_iter};
    auto it = ctx->graphs.find(key);
    if (it != ctx->graphs.end()) {
      exec = it->second;
      graph_launches = ctx->graph_launches[key];
    } else {
      // the graph replays identical launches: every argument is a workspace pointer
      // and all per-iteration state lives in device memory
      const int st = capture_groups<R>(
          ctx, w, nsrc, G,
          [&](cudaStream_t cs, cudaStream_t side, cudaEvent_t fork, cudaEvent_t join, const SolveArgs<R>& a, int n) {
            // fixed point: the node checks run on a side branch beside the next interval
            constexpr bool beside = std::is_same<R, FX>::value;
            for (int k = 0; k < chunk; ++k) {
              const int n1 = launch_k1<R>(w, a, n, cs, beside && k % kNodeCheck == 0);
              launch_k2<R>(w, a, n, cs, n1 == 1);
              graph_launches += n1 + 1;
              if (!w.defer || (k + 1) % kNodeCheck != 0) continue;
              if (beside) {
                if (k >= kNodeCheck) cudaStreamWaitEvent(cs, join, 0);
                cudaEventRecord(fork, cs);
                cudaStreamWaitEvent(side, fork, 0);
                graph_launches += launch_node_check<R>(w, a, n, side);
                cudaEventRecord(join, side);
              } else {
                graph_launches += launch_node_check<R>(w, a, n, cs);
              }
            }
            if (beside && w.defer) cudaStreamWaitEvent(cs, join, 0);
          },
          &exec);
      if (st != OV_OK) return st;
      ctx->graphs[key] = exec;
      ctx->graph_launches[key] = graph_launches;
    }
  }
  int done_iters = 0;
  while (done_iters < max_iter) {
    const int n = std::min(chunk, max_iter - done_iters);
    if (graph && n == chunk) {
      cudaError_t e = cudaGraphLaunch(exec, s);
      if (e != cudaSuccess) return ctx_cuda(ctx, e, "cudaGraphLaunch");
      *launches += graph_launches;
    } else {
      for (int k = 0; k < n; ++k) *launches += launch_iteration<R>(ctx, w, nsrc, s, done_iters + k);
      OV_CHECK_LAUNCH(ctx, "lanczos kernels");
    }
    done_iters += n;
    cudaError_t e = cudaMemcpyAsync(ctx->host_flag, w.a.done_count, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return ctx_cuda(ctx, e, "cudaMemcpyAsync(done)");
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return ctx_cuda(ctx, e, "cudaStreamSynchronize");
    kt_collect(ctx);
    if (*ctx->host_flag >= nsrc) break;
  }
  if (w.defer) {  // the iterations since the last check (final node residuals and status)
    *launches += launch_node_check<R>(w, w.a, nsrc, s, true);
    OV_CHECK_LAUNCH(ctx, "node_check_kernel");
  }
  return OV_OK;
}

// The persistent form of the iteration loop (lanczos_coop_kernel) when it applies:
// scalar-only node recurrences, at most kCoopMaxSrc sources, and a grid that is
// co-resident (one block per 32-site tile and source, capped by occupancy).  Returns
// OV_ERR_INVALID_ARG (nothing launched) when it does not apply.
template <typename R>
int run_coop(ov_ctx* ctx, SolveWs<R>& w, int nsrc, cudaStream_t s, double* launches) {
  if (nsrc > kCoopMaxSrc || ctx->no_coop) return OV_ERR_INVALID_ARG;
  int dev = 0, coop = 0, nsm = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (!coop) return OV_ERR_INVALID_ARG;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, lanczos_coop_kernel<R>, NT1, 0) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    return OV_ERR_INVALID_ARG;
  }
  const int ntile = (ctx->g.V + kSplitSites - 1) / kSplitSites;
  const int G = std::min(per_sm * nsm, ntile * nsrc);
  SolveArgs<R> a = w.a;
  // block partials, indexed source * G + block
  int st = OV_OK;
  a.part1 = (double*)ws_get(ctx, "coop.part1", sizeof(double) * (size_t)G * nsrc, &st);
  a.part2 = (double*)ws_get(ctx, "coop.part2", sizeof(double) * (size_t)G * nsrc, &st);
  if (st != OV_OK) return st;
  void* args[] = {(void*)&a, (void*)&nsrc};
  cudaEvent_t ev;
  kt_begin(ctx, KC_COOP, s, &ev);
  cudaError_t e = cudaLaunchCooperativeKernel((const void*)lanczos_coop_kernel<R>, dim3(G), dim3(NT1), args, 0, s);
  kt_end(ctx, KC_COOP, s, ev);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "cudaLaunchCooperativeKernel");
  *launches += 1.0;
  return OV_OK;
}

template <typename R>
int init_solve(ov_ctx* ctx, SolveWs<R>& w, const double2* b_soa, int nsrc, int ns,
               const std::vector<double2>& zh, const std::vector<double2>& ch, double2 c0,
               double tol, int max_iter, cudaStream_t s, int vec_shifts = 1) {
  // scalar-only forms with nodes defer the per-node recurrences (they record alpha, beta)
  w.defer = (vec_shifts == 0 && ns > 0 && w.a.hist_a && w.a.hist_b);
  SolveParams prm{tol, max_iter, ns, vec_shifts, w.nslots, w.nslots > 3 ? 1 : 0, w.defer ? 1 : 0, w.slot_mask};
  cudaError_t e = cudaMemcpyAsync(w.prm_dev, &prm, sizeof(prm), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "copy params");
  if (ns > 0) {
    e = cudaMemcpyAsync((void*)w.a.z, zh.data(), sizeof(double2) * zh.size(), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return ctx_cuda(ctx, e, "copy nodes");
    e = cudaMemcpyAsync((void*)w.a.c, ch.data(), sizeof(double2) * ch.size(), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return ctx_cuda(ctx, e, "copy coefficients");
  }
  cudaMemsetAsync(w.a.cnt, 0, sizeof(unsigned) * 2 * nsrc, s);
  cudaMemsetAsync(w.a.done_count, 0, sizeof(int), s);
  if (w.a.sgrp)
    cudaMemsetAsync(w.a.sgrp, 0, sizeof(double2) * 12 * (size_t)w.a.g.V * nsrc * (w.ngrp - 1), s);
  if (w.a.bins1) cudaMemsetAsync(w.a.bins1, 0, sizeof(long long) * 4 * kFxBins * kFxWords * nsrc, s);
  if constexpr (!std::is_same<R, FX>::value) {  // fixed point keeps no per-node vectors
    const size_t n = (size_t)12 * ctx->g.V * nsrc * ns;
    if (w.a.x) zero_kernel<R><<<1024, 256, 0, s>>>(w.a.x, n);
  }
  cudaEvent_t ev;
  kt_begin(ctx, KC_MISC, s, &ev);
  lanczos_init_kernel<R><<<dim3(w.nblk2, nsrc), NT2, 0, s>>>(w.a, b_soa, c0);
  if constexpr (std::is_same<R, FX>::value)
    fx_quantize_kernel<<<dim3(std::min(w.nblk2, 1024), nsrc), NT2, 0, s>>>(w.a, b_soa);
  kt_end(ctx, KC_MISC, s, ev);
  OV_CHECK_LAUNCH(ctx, "lanczos_init_kernel");
  return OV_OK;
}

template <typename R>
int finish_solve(ov_ctx* ctx, SolveWs<R>& w, int nsrc, int ns, const std::vector<double2>& zh,
                 const std::vector<double2>& ch, SolveOut* so, cudaStream_t s) {
  std::vector<SrcState> S(nsrc);
  std::vector<ShiftState> Q((size_t)nsrc * (ns > 0 ? ns : 1));
  cudaError_t e = cudaMemcpyAsync(S.data(), w.a.src, sizeof(SrcState) * nsrc, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && ns > 0)
    e = cudaMemcpyAsync(Q.data(), w.a.sh, sizeof(ShiftState) * (size_t)nsrc * ns, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "read solver state");
  int status = OV_OK;
  so->iterations = 0;
  so->converged = 1;
  so->max_residual = 0.0;
  so->error_bound = 0.0;
  so->node_updates = 0.0;
  for (int r = 0; r < nsrc; ++r) {
    so->node_updates += S[r].node_updates;
    so->iterations = std::max(so->iterations, S[r].iter - 1);
    if (!S[r].done) S[r].status = OV_ERR_NOT_CONVERGED;
    if (S[r].status != OV_OK) {
      so->converged = 0;
      if (status == OV_OK || S[r].status == OV_ERR_BREAKDOWN) status = S[r].status;
    }
    double bound = 0.0;
    for (int j = 0; j < ns; ++j) {
      const ShiftState& q = Q[(size_t)r * ns + j];
      const double res = std::sqrt(q.res2);
      so->max_residual = std::max(so->max_residual, res);
      const double2 zz = zh[(size_t)r * ns + j], cc = ch[(size_t)r * ns + j];
      bound += std::hypot(cc.x, cc.y) * res / std::fabs(zz.y);
    }
    so->error_bound = std::max(so->error_bound, bound);
  }
  if (status == OV_ERR_NOT_CONVERGED)
    return ctx_fail(ctx, status, "shifted solve hit the iteration limit before every node met tol");
  if (status == OV_ERR_BREAKDOWN) return ctx_fail(ctx, status, "non-finite Lanczos scalar (NaN/Inf in input?)");
  return OV_OK;
}

}  // namespace

// out = the weighted sum, its node groups added up in order
static __global__ void sum_groups_kernel(const double2* __restrict__ sacc, const double2* __restrict__ sgrp, int ngrp,
                                         double2* __restrict__ out, size_t n12) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y;
  if (e >= n12) return;
  double2 t = sacc[r * n12 + e];
  for (int z = 0; z < ngrp - 1; ++z) {
    const double2 q = sgrp[(r * (ngrp - 1) + z) * n12 + e];
    t.x += q.x;
    t.y += q.y;
  }
  out[r * n12 + e] = t;
}

// Shifted FP64 solve with an explicit node list per source (zh, ch: nsrc x ns): the
// weighted sum c0 b + sum_j c_j y_j goes to out_soa (if not null) and, if xs_soa is
// not null, every node's solution y_j to xs_soa[src][j][12V].
// The vector-space shifted solve for explicit nodes (per source), optionally keeping every
// node's solution (xs, in the vector storage type): FP64 or double-float vectors.
template <typename R>
static int solve_nodes_t(ov_ctx* ctx, const double2* b_soa, int nsrc, int ns, const std::vector<double2>& zh,
                         const std::vector<double2>& ch, double2 c0, double2* out_soa, typename Store<R>::T* xs,
                         const ov_solve_opts& o, SolveOut* so, cudaStream_t s, const char* tag) {
  SolveWs<R> w;
  int st = setup_ws<R>(ctx, nsrc, ns, false, true, false, o.max_iter, &w, tag);
  if (st != OV_OK) return st;
  w.a.x = xs;
  st = init_solve<R>(ctx, w, b_soa, nsrc, ns, zh, ch, c0, o.tol, o.max_iter, s);
  if (st != OV_OK) return st;
  double launches = 1.0 + (xs ? 1.0 : 0.0);  // init (+ zeroing)
  st = run_iterations<R>(ctx, w, nsrc, ns, xs ? 1 : 0, o.max_iter, o, s, &launches);
  if (st != OV_OK) return st;
  st = finish_solve<R>(ctx, w, nsrc, ns, zh, ch, so, s);
  so->launches = launches + 2.0;  // pack + unpack/epilogue issued by the caller
  if (out_soa) {
    // the weighted sum, even when not converged (best iterate)
    const size_t n12 = 12 * (size_t)ctx->g.V;
    sum_groups_kernel<<<dim3((unsigned)((n12 + 255) / 256), nsrc), 256, 0, s>>>(w.a.sacc, w.a.sgrp, w.ngrp, out_soa, n12);
    OV_CHECK_LAUNCH(ctx, "sum_groups_kernel");
    so->launches += 1.0;
  }
  return st;
}

// solve_nodes_t with the Lanczos vectors in fixed point (a ring of kNodeRun of them) and the
// per-node vectors in FP64.  OV_ERR_OUT_OF_MEMORY: its workspace, larger than the FP64 form's
// by kNodeRun - 3 vectors per source, does not fit.
static int solve_nodes_fx(ov_ctx* ctx, const double2* b_soa, int nsrc, int ns, const std::vector<double2>& zh,
                          const std::vector<double2>& ch, double2 c0, double2* out_soa, double2* xs,
                          const ov_solve_opts& o, SolveOut* so, cudaStream_t s) {
  NvtxRange nvtx_("solve: vector space, fixed-point Lanczos vectors");
  const size_t n12 = 12 * (size_t)ctx->g.V, nvec = vec_elems<FX>(ctx->g.V);
  const char* const names[] = {"fxv.ring", "fxv.pv"};
  const double need = (double)sizeof(double2) * nvec * nsrc * (kNodeRun + ns);
  double held = 0.0;
  for (const char* n : names) {
    auto it = ctx->bufs.find(n);
    if (it != ctx->bufs.end()) held += (double)it->second.bytes;
  }
  size_t freeb = 0, totalb = 0;
  cudaMemGetInfo(&freeb, &totalb);
  if (need > held && need - held > (double)freeb - 0.10 * (double)totalb) return OV_ERR_OUT_OF_MEMORY;
  SolveWs<FX> w;
  int st = setup_ws<FX>(ctx, nsrc, ns, false, true, true, o.max_iter, &w, "fxv", kNodeRun, false);
  w.slot_mask = kNodeRun - 1;
  w.ngrp = k2_groups((int)std::min<size_t>((nvec + 255) / 256, INT_MAX / nsrc), nsrc, ns);
  w.a.sgrp = w.ngrp > 1 ? (double2*)ws_get(ctx, "fxv.sgrp", sizeof(double2) * n12 * (size_t)nsrc * (w.ngrp - 1), &st)
                        : nullptr;
  w.a.pv = (double2*)ws_get(ctx, "fxv.pv", sizeof(double2) * nvec * (size_t)nsrc * ns, &st);
  w.a.nco = (double2*)ws_get(ctx, "fxv.nco", sizeof(double2) * 3 * kNodeRun * (size_t)nsrc * ns, &st);
  w.a.nin = (double*)ws_get(ctx, "fxv.nin", sizeof(double) * kNodeRun * (size_t)nsrc, &st);
  w.a.xv = xs;
  if (st != OV_OK) return st;
  if (xs) cudaMemsetAsync(xs, 0, sizeof(double2) * n12 * (size_t)nsrc * ns, s);
  st = init_solve<FX>(ctx, w, b_soa, nsrc, ns, zh, ch, c0, o.tol, o.max_iter, s, 0);
  if (st != OV_OK) return st;
  double launches = 2.0;
  st = run_iterations<FX>(ctx, w, nsrc, ns, xs ? 9 : 8, o.max_iter, o, s, &launches);
  if (st != OV_OK) return st;
  st = finish_solve<FX>(ctx, w, nsrc, ns, zh, ch, so, s);
  so->launches = launches + 2.0;  // pack + unpack/epilogue issued by the caller
  if (out_soa) {
    sum_groups_kernel<<<dim3((unsigned)((n12 + 255) / 256), nsrc), 256, 0, s>>>(w.a.sacc, w.a.sgrp, w.ngrp, out_soa, n12);
    OV_CHECK_LAUNCH(ctx, "sum_groups_kernel");
    so->launches += 1.0;
  }
  return st;
}

// Whether the stored-basis and vector-space forms of a solver mode run in fixed point
// (fixed.cuh): links of about unit norm (the bounds there) and |4 - m0| <= 4.  Other links and masses,
// the persistent loop and OV_MODE_FP64_REGEN (its gradients included) keep the FP64 and
// double-float kernels.
static bool fixed_point_fits(const ov_ctx* ctx, int mode) {
  return ctx->no_coop && ctx->fx_ok && mode != OV_MODE_FP64_REGEN;
}

int solve_nodes_soa(ov_ctx* ctx, const double2* b_soa, int nsrc, int ns, const std::vector<double2>& zh,
                    const std::vector<double2>& ch, double2 c0, double2* out_soa, double2* xs_soa,
                    const ov_solve_opts& o, SolveOut* so, cudaStream_t s) {
  if (fixed_point_fits(ctx, o.mode) && ns > 0) {
    const int st = solve_nodes_fx(ctx, b_soa, nsrc, ns, zh, ch, c0, out_soa, xs_soa, o, so, s);
    if (st != OV_ERR_OUT_OF_MEMORY) return st;
    ws_release(ctx, "fxv.");
  }
  return solve_nodes_t<double>(ctx, b_soa, nsrc, ns, zh, ch, c0, out_soa, xs_soa, o, so, s, "fp64");
}

namespace {
__global__ void df_to_double_kernel(const float4* __restrict__ in, double2* __restrict__ out, size_t n) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
    const float4 v = in[t];
    out[t] = make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
  }
}
}  // namespace

int solve_nodes_soa_df(ov_ctx* ctx, const double2* b_soa, int nsrc, int ns, const std::vector<double2>& zh,
                       const std::vector<double2>& ch, double2 c0, double2* out_soa, double2* xs_soa,
                       const ov_solve_opts& o, SolveOut* so, cudaStream_t s) {
  int st = ensure_links_df(ctx, s);
  if (st != OV_OK) return st;
  const size_t nx = (size_t)12 * ctx->g.V * nsrc * ns;
  float4* xd = xs_soa ? (float4*)ws_get(ctx, "dfn.xs", sizeof(float4) * nx, &st) : nullptr;
  if (st != OV_OK) return st;
  st = solve_nodes_t<DF>(ctx, b_soa, nsrc, ns, zh, ch, c0, out_soa, xd, o, so, s, "dfn");
  if (xs_soa && (st == OV_OK || st == OV_ERR_NOT_CONVERGED)) {
    df_to_double_kernel<<<152 * 8, 256, 0, s>>>(xd, xs_soa, nx);
    OV_CHECK_LAUNCH(ctx, "df_to_double_kernel");
  }
  return st;
}

int solve_sign_soa(ov_ctx* ctx, const double2* b_soa, double2* out_soa, int nsrc, const ov_solve_opts& o,
                   SolveOut* so, cudaStream_t s, double2* xs_soa) {
  NvtxRange nvtx_("solve: vector-space form");
  const int ns = (int)ctx->z.size();
  std::vector<double2> zh((size_t)nsrc * ns), ch((size_t)nsrc * ns);
  for (int r = 0; r < nsrc; ++r)
    for (int j = 0; j < ns; ++j) {
      zh[(size_t)r * ns + j] = ctx->z[j];
      ch[(size_t)r * ns + j] = ctx->c[j];
    }
  return solve_nodes_soa(ctx, b_soa, nsrc, ns, zh, ch, ctx->c0, out_soa, xs_soa, o, so, s);
}

// FOM coefficients y = (z - T_k)^-1 e_1 ||b|| of one node from the recorded Lanczos
// scalars al[0..k), be[0..k): forward LDL^T sweep (d_i, l_i = -beta_i / d_i, zeta_i =
// omega_i / d_i) and back substitution y_i = zeta_i - l_i y_{i+1}.
struct FomScratch {
  std::vector<std::complex<double>> dd, ll, zt;
};
static void fom_coefficients(const double* al, const double* be, int k, double bnorm, std::complex<double> z,
                             FomScratch& sc, std::vector<std::complex<double>>& yy) {
  sc.dd.assign(k, 0.0);
  sc.ll.assign(k, 0.0);
  sc.zt.assign(k, 0.0);
  yy.assign(k, 0.0);
  if (k < 1) return;
  std::complex<double> om = bnorm;
  for (int i = 0; i < k; ++i) {
    if (i == 0) {
      sc.dd[0] = z - al[0];
    } else {
      sc.dd[i] = z - al[i] - be[i - 1] * be[i - 1] / sc.dd[i - 1];
      om = -sc.ll[i - 1] * om;
    }
    sc.ll[i] = -be[i] / sc.dd[i];
    sc.zt[i] = om / sc.dd[i];
  }
  yy[k - 1] = sc.zt[k - 1];
  for (int i = k - 2; i >= 0; --i) yy[i] = sc.zt[i] - sc.ll[i] * yy[i + 1];
}

// g = sum_j c_j (z_j - T_k)^-1 e_1 ||b|| per source, from the recorded alpha (ha) and beta
// (hb), leading dimension ld.
static void lanczos_sum_coefficients(const ov_ctx* ctx, int nsrc, const std::vector<int>& kr,
                                     const std::vector<double>& bnorm, const std::vector<double>& ha,
                                     const std::vector<double>& hb, int ld, std::vector<double2>& g) {
  const int ns = (int)ctx->z.size();
  g.assign((size_t)nsrc * ld, make_double2(0.0, 0.0));
  FomScratch sc;
  std::vector<std::complex<double>> yy;
  for (int r = 0; r < nsrc; ++r) {
    const int k = kr[r];
    if (k < 1) continue;
    for (int j = 0; j < ns; ++j) {
      const std::complex<double> zj(ctx->z[j].x, ctx->z[j].y), cj(ctx->c[j].x, ctx->c[j].y);
      fom_coefficients(ha.data() + (size_t)r * ld, hb.data() + (size_t)r * ld, k, bnorm[r], zj, sc, yy);
      for (int i = 0; i < k; ++i) {
        const std::complex<double> t = cj * yy[i];
        g[(size_t)r * ld + i].x += t.real();
        g[(size_t)r * ld + i].y += t.imag();
      }
    }
  }
}

// Stored-basis form of OV_MODE_FP64_2PASS: pass 1 keeps U_1 .. U_k (slot i), then
// s = c0 b + sum_i (g_i / ||U_i||) U_i in one read of the basis.
template <typename R>
int solve_sign_stored(ov_ctx* ctx, const double2* b_soa, double2* out_soa, int nsrc,
                             const ov_solve_opts& o, SolveOut* so, cudaStream_t s, int cap) {
  NvtxRange nvtx_("solve: stored basis");
  const int ns = (int)ctx->z.size();
  const size_t n12 = (size_t)12 * ctx->g.V;
  SolveWs<R> w;
  const std::string tag = std::string(coef_tag<R>()) + "s";
  int st = setup_ws<R>(ctx, nsrc, ns, false, true, true, cap, &w, tag.c_str(), cap + 3, false);
  if (st != OV_OK) return st;
  std::vector<double2> zh((size_t)nsrc * ns), ch((size_t)nsrc * ns);
  for (int r = 0; r < nsrc; ++r)
    for (int j = 0; j < ns; ++j) {
      zh[(size_t)r * ns + j] = ctx->z[j];
      ch[(size_t)r * ns + j] = ctx->c[j];
    }
  st = init_solve<R>(ctx, w, b_soa, nsrc, ns, zh, ch, ctx->c0, o.tol, cap, s, 0);
  if (st != OV_OK) return st;
  double launches = 1.0;
  st = run_coop<R>(ctx, w, nsrc, s, &launches);
  if (st == OV_ERR_INVALID_ARG) st = run_iterations<R>(ctx, w, nsrc, ns, 6, cap, o, s, &launches);
  if (st != OV_OK) return st;
  const int fst = finish_solve<R>(ctx, w, nsrc, ns, zh, ch, so, s);
  // not converged within the store: the caller regenerates, unless the store already
  // spans max_iter (then the best iterate is returned with OV_ERR_NOT_CONVERGED)
  if (fst != OV_OK && !(fst == OV_ERR_NOT_CONVERGED && cap >= o.max_iter)) return fst;
  std::vector<SrcState> S(nsrc);
  std::vector<double> ha((size_t)nsrc * cap), hb((size_t)nsrc * cap);
  cudaError_t e = cudaMemcpyAsync(S.data(), w.a.src, sizeof(SrcState) * nsrc, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(ha.data(), w.a.hist_a, sizeof(double) * ha.size(), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hb.data(), w.a.hist_b, sizeof(double) * hb.size(), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "read Lanczos history");
  std::vector<int> kr(nsrc);
  std::vector<double> bn(nsrc);
  for (int r = 0; r < nsrc; ++r) {
    kr[r] = std::max(0, S[r].iter - 1);
    bn[r] = S[r].bnorm;
  }
  std::vector<double2> g;
  lanczos_sum_coefficients(ctx, nsrc, kr, bn, ha, hb, cap, g);
  for (int r = 0; r < nsrc; ++r)
    for (int i = 0; i < kr[r]; ++i) {  // fold in 1 / ||U_i||
      const double ni = (i == 0) ? bn[r] : hb[(size_t)r * cap + i - 1];
      g[(size_t)r * cap + i].x /= ni;
      g[(size_t)r * cap + i].y /= ni;
    }
  // a node list closed under conjugation gives real coefficients (up to rounding):
  // then the sum takes half the multiplications
  bool real = true;
  for (int r = 0; r < nsrc && real; ++r) {
    double gmax = 0.0, imax = 0.0;
    for (int i = 0; i < kr[r]; ++i) {
      const double2 v = g[(size_t)r * cap + i];
      gmax = std::max(gmax, std::hypot(v.x, v.y));
      imax = std::max(imax, std::fabs(v.y));
    }
    real = std::isfinite(gmax) && imax <= 1e-14 * gmax;
  }
  using T = typename Store<R>::T;
  std::vector<T> gs(g.size());
  for (size_t t = 0; t < g.size(); ++t) gs[t] = host_store(g[t], (T*)nullptr);
  T* gd = (T*)ws_get(ctx, (tag + ".g").c_str(), sizeof(T) * gs.size(), &st);
  int* krd = (int*)ws_get(ctx, (tag + ".kr").c_str(), sizeof(int) * nsrc, &st);
  if (st != OV_OK) return st;
  e = cudaMemcpyAsync(gd, gs.data(), sizeof(T) * gs.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(krd, kr.data(), sizeof(int) * nsrc, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "copy coefficients");
  cudaEvent_t ev;
  kt_begin(ctx, KC_BASIS_SUM, s, &ev);
  const dim3 gsum((unsigned)((n12 + 255) / 256), nsrc);
  if (real)
    basis_sum_kernel<R, true><<<gsum, 256, 0, s>>>(w.a.ring, cap + 3, gd, cap, krd, w.a.sacc, n12);
  else
    basis_sum_kernel<R, false><<<gsum, 256, 0, s>>>(w.a.ring, cap + 3, gd, cap, krd, w.a.sacc, n12);
  kt_end(ctx, KC_BASIS_SUM, s, ev);
  OV_CHECK_LAUNCH(ctx, "basis_sum_kernel");
  so->launches = launches + 3.0;
  e = cudaMemcpyAsync(out_soa, w.a.sacc, sizeof(double2) * n12 * nsrc, cudaMemcpyDeviceToDevice, s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "copy sum");
  return fst;
}

// Device workspace of the fixed-point coefficients.
struct FxCoef {
  double2 *Y = nullptr, *g = nullptr;
  int4* G = nullptr;
  double* scale = nullptr;  // [src][ng] of G's groups
  int ng = 0;
  FxSumInfo* info = nullptr;
};

// The Lanczos pass of the fixed-point forms, then (enqueued, no host read between) every node's
// coefficients and the integer coefficients of the weighted sum.
static int fx_lanczos(ov_ctx* ctx, SolveWs<FX>& w, FxCoef& f, const double2* b_soa, int nsrc, int ns,
                      const std::vector<double2>& zh, const std::vector<double2>& ch, double2 c0, double2* sums,
                      const ov_solve_opts& o, cudaStream_t s, int cap, int flavour, double* launches) {
  int st = setup_ws<FX>(ctx, nsrc, ns, false, false, true, cap, &w, "fxs", cap + 3, false);
  if (st != OV_OK) return st;
  f.Y = (double2*)ws_get(ctx, "fxs.Y", sizeof(double2) * (size_t)nsrc * cap * ns, &st);
  f.g = (double2*)ws_get(ctx, "fxs.gd", sizeof(double2) * (size_t)nsrc * cap, &st);
  f.G = (int4*)ws_get(ctx, "fxs.g", sizeof(int4) * (size_t)nsrc * cap, &st);
  f.ng = fx_groups(cap);
  f.scale = (double*)ws_get(ctx, "fxs.gs", sizeof(double) * (size_t)nsrc * f.ng, &st);
  f.info = (FxSumInfo*)ws_get(ctx, "fxs.info", sizeof(FxSumInfo) * nsrc, &st);
  w.a.fd = (double2*)ws_get(ctx, "fxs.D", sizeof(double2) * (size_t)nsrc * cap * ns, &st);
  w.a.fz = f.Y;
  if (st != OV_OK) return st;
  w.a.sacc = sums;  // c0 b, written by the init kernel only
  st = init_solve<FX>(ctx, w, b_soa, nsrc, ns, zh, ch, c0, o.tol, cap, s, 0);
  w.a.sacc = nullptr;
  if (st != OV_OK) return st;
  *launches = 2.0;
  st = run_iterations<FX>(ctx, w, nsrc, ns, flavour, cap, o, s, launches);
  if (st != OV_OK) return st;
  cudaEvent_t ev;
  kt_begin(ctx, KC_MISC, s, &ev);
  fx_node_coef_kernel<<<dim3((ns + 31) / 32, nsrc), 32, 0, s>>>(w.a, ns);
  fx_sum_nodes_kernel<<<dim3(std::min((cap + 7) / 8, 64), nsrc), 256, 0, s>>>(w.a, ns, f.Y, f.g);
  fx_sum_quant_kernel<<<nsrc, kCoefNT, 0, s>>>(w.a, f.g, f.G, f.scale, f.ng, f.info);
  kt_end(ctx, KC_MISC, s, ev);
  OV_CHECK_LAUNCH(ctx, "fx_node_coef_kernel");
  *launches += 3.0;
  return OV_OK;
}

static int launch_fx_basis_sum(ov_ctx* ctx, const SolveWs<FX>& w, const FxCoef& f, int nsrc, int cap, double2* sums,
                               cudaStream_t s) {
  cudaEvent_t ev;
  kt_begin(ctx, KC_BASIS_SUM, s, &ev);
  fx_basis_sum_kernel<<<dim3((unsigned)((w.nvec + 255) / 256), nsrc), 256, 0, s>>>(w.a.ring, cap + 3, f.G, cap, f.scale,
                                                                                f.ng, f.info, sums, ctx->g.V);
  kt_end(ctx, KC_BASIS_SUM, s, ev);
  OV_CHECK_LAUNCH(ctx, "fx_basis_sum_kernel");
  return OV_OK;
}

// solve_sign_stored in fixed point: the sum goes straight to out_soa, and the host waits for
// the device once, at the end.
template <>
int solve_sign_stored<FX>(ov_ctx* ctx, const double2* b_soa, double2* out_soa, int nsrc, const ov_solve_opts& o,
                          SolveOut* so, cudaStream_t s, int cap) {
  NvtxRange nvtx_("solve: stored basis, fixed point");
  const int ns = (int)ctx->z.size();
  std::vector<double2> zh, ch;
  for (int r = 0; r < nsrc; ++r) {
    zh.insert(zh.end(), ctx->z.begin(), ctx->z.end());
    ch.insert(ch.end(), ctx->c.begin(), ctx->c.end());
  }
  SolveWs<FX> w;
  FxCoef f;
  double launches = 0.0;
  int st = fx_lanczos(ctx, w, f, b_soa, nsrc, ns, zh, ch, ctx->c0, out_soa, o, s, cap, 6, &launches);
  if (st == OV_OK) st = launch_fx_basis_sum(ctx, w, f, nsrc, cap, out_soa, s);
  if (st != OV_OK) return st;
  st = finish_solve<FX>(ctx, w, nsrc, ns, zh, ch, so, s);
  so->launches = launches + 3.0;
  return st;
}

// OV_MODE_FP64_2PASS.  Pass 1: the Lanczos process with every node's LDL^T scalar
// recurrence (for the stopping test) but no per-node vectors; alpha_i and beta_i
// are recorded.  Host: for every node the FOM coefficients y^j = (z_j - T_k)^-1 e_1 ||b||
// (forward LDL^T sweep, back substitution), summed as g = sum_j c_j y^j.  Pass 2:
// regenerate v_1 .. v_k with bit-identical arithmetic and accumulate
// s = c0 b + sum_i g_i v_i.  Same result as OV_MODE_FP64 up to rounding; the vector
// work no longer grows with the number of nodes.
template <typename R>
static int solve_sign_regen(ov_ctx* ctx, const double2* b_soa, double2* out_soa, int nsrc,
                            const ov_solve_opts& o, SolveOut* so, cudaStream_t s);

// Fold the statistics of one batch of sources into the call's.
void merge_stats(SolveOut* tot, const SolveOut& b, bool first) {
  if (first) {
    *tot = b;
    return;
  }
  tot->iterations = std::max(tot->iterations, b.iterations);
  tot->converged = tot->converged && b.converged;
  tot->max_residual = std::max(tot->max_residual, b.max_residual);
  tot->error_bound = std::max(tot->error_bound, b.error_bound);
  tot->refine_rounds += b.refine_rounds;
  tot->inner_iterations += b.inner_iterations;
  tot->node_updates += b.node_updates;
  tot->launches += b.launches;
}

// Coefficient-space solve.  Preferred: keep the Lanczos basis in HBM (pass 2 is one read
// of it instead of a second Lanczos pass), for as many sources at a time as fit the store
// budget -- 40% of device memory, and no more than what is free beyond a 10% reserve (a
// store this context already holds counts as free).  The store depth is min(max_iter,
// 1024) vectors, or 1.25x the iterations of the previous batch or call (plus 32) once
// those are known; a batch that outgrows its store, or that cannot be allocated, is
// solved by regenerating the basis instead.  OV_MODE_FP64_REGEN always regenerates.
template <typename R>
static int solve_sign_coef(ov_ctx* ctx, const double2* b_soa, double2* out_soa, int nsrc, const ov_solve_opts& o,
                           SolveOut* so, cudaStream_t s) {
  NvtxRange nvtx_("solve: coefficient space");
  auto regen = [&](int r0, int nb, SolveOut* sb) {
    const size_t off = (size_t)r0 * 12 * ctx->g.V;
    if (o.mode != OV_MODE_F32X2) return solve_sign_regen<double>(ctx, b_soa + off, out_soa + off, nb, o, sb, s);
    const int st = ensure_links_df(ctx, s);
    return st != OV_OK ? st : solve_sign_regen<DF>(ctx, b_soa + off, out_soa + off, nb, o, sb, s);
  };
  if (o.mode == OV_MODE_FP64_REGEN) return regen(0, nsrc, so);
  size_t freeb = 0, totalb = 0;
  cudaMemGetInfo(&freeb, &totalb);
  const std::string ring = std::string(coef_tag<R>()) + "s.ring";
  auto it = ctx->bufs.find(ring);
  const double held = it != ctx->bufs.end() ? (double)it->second.bytes : 0.0;
  const double budget = std::min(0.40 * (double)totalb, (double)freeb + held - 0.10 * (double)totalb);
  const size_t n12 = (size_t)12 * ctx->g.V;
  const double per_vec = (double)vec_elems<R>(ctx->g.V) * sizeof(double2);
  int cap = std::min(o.max_iter, ctx->coef_iter_hint > 0 ? std::max(64, ctx->coef_iter_hint * 5 / 4 + 32) : 1024);
  int r0 = 0, worst = OV_OK;
  bool first = true;
  while (r0 < nsrc) {
    const int rem = nsrc - r0;
    const int nb_max = (int)std::min<double>(rem, std::floor(budget / ((cap + 3) * per_vec)));
    const int nbat = nb_max >= 1 ? (rem + nb_max - 1) / nb_max : 1;
    const int nb = nb_max >= 1 ? (rem + nbat - 1) / nbat : rem;  // even batches
    SolveOut sb;
    int st = OV_ERR_OUT_OF_MEMORY;
    if (nb_max >= 1) st = solve_sign_stored<R>(ctx, b_soa + r0 * n12, out_soa + r0 * n12, nb, o, &sb, s, cap);
    if (st == OV_ERR_OUT_OF_MEMORY || (st == OV_ERR_NOT_CONVERGED && cap < o.max_iter)) {
      cudaGetLastError();
      sb = SolveOut();
      st = regen(r0, nb, &sb);
    }
    if (st != OV_OK && st != OV_ERR_NOT_CONVERGED) return st;
    if (st == OV_ERR_NOT_CONVERGED) worst = st;
    merge_stats(so, sb, first);
    first = false;
    if (sb.converged) {
      ctx->coef_iter_hint = sb.iterations;
      cap = std::min(o.max_iter, std::max(64, sb.iterations * 5 / 4 + 32));
    }
    r0 += nb;
  }
  return worst;
}

// OV_MODE_FP64_REGEN and the fallback of the stored form: pass 1 records alpha_i, beta_i,
// pass 2 regenerates v_1 .. v_k with bit-identical arithmetic and sums g_i v_i.
template <typename R>
static int solve_sign_regen(ov_ctx* ctx, const double2* b_soa, double2* out_soa, int nsrc,
                            const ov_solve_opts& o, SolveOut* so, cudaStream_t s) {
  const int ns = (int)ctx->z.size();
  SolveWs<R> w;
  const std::string tag = coef_tag<R>();
  int st = setup_ws<R>(ctx, nsrc, ns, false, true, true, o.max_iter, &w, tag.c_str(), 3, false);
  if (st != OV_OK) return st;
  double2* gco = (double2*)ws_get(ctx, (tag + ".gco").c_str(), sizeof(double2) * (size_t)nsrc * o.max_iter, &st);
  if (st != OV_OK) return st;
  const size_t n12 = (size_t)12 * ctx->g.V;
  float4* ssum = nullptr;
  if (std::is_same<R, DF>::value) {
    ssum = (float4*)ws_get(ctx, "df.ssum", sizeof(float4) * n12 * nsrc, &st);
    if (st != OV_OK) return st;
  }
  w.a.p = nullptr;
  std::vector<double2> zh((size_t)nsrc * ns), ch((size_t)nsrc * ns);
  for (int r = 0; r < nsrc; ++r)
    for (int j = 0; j < ns; ++j) {
      zh[(size_t)r * ns + j] = ctx->z[j];
      ch[(size_t)r * ns + j] = ctx->c[j];
    }
  st = init_solve<R>(ctx, w, b_soa, nsrc, ns, zh, ch, ctx->c0, o.tol, o.max_iter, s, 0);
  if (st != OV_OK) return st;
  double launches = 1.0;
  st = run_iterations<R>(ctx, w, nsrc, ns, 2, o.max_iter, o, s, &launches);
  if (st != OV_OK) return st;
  const int fst = finish_solve<R>(ctx, w, nsrc, ns, zh, ch, so, s);
  if (fst != OV_OK && fst != OV_ERR_NOT_CONVERGED) return fst;
  // coefficients of the sum in the Lanczos basis
  std::vector<SrcState> S(nsrc);
  cudaError_t e = cudaMemcpyAsync(S.data(), w.a.src, sizeof(SrcState) * nsrc, cudaMemcpyDeviceToHost, s);
  std::vector<double> ha((size_t)nsrc * o.max_iter), hb((size_t)nsrc * o.max_iter);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(ha.data(), w.a.hist_a, sizeof(double) * ha.size(), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(hb.data(), w.a.hist_b, sizeof(double) * hb.size(), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "read Lanczos history");
  int kmax = 0;
  std::vector<int> kr(nsrc);
  std::vector<double> bn(nsrc);
  for (int r = 0; r < nsrc; ++r) {
    kr[r] = std::max(0, S[r].iter - 1);
    bn[r] = S[r].bnorm;
    S[r].k_final = kr[r];
    kmax = std::max(kmax, kr[r]);
    if (kr[r] >= 1) {
      S[r].iter = 1;
      S[r].done = 0;
    }
  }
  std::vector<double2> g;
  lanczos_sum_coefficients(ctx, nsrc, kr, bn, ha, hb, o.max_iter, g);
  e = cudaMemcpyAsync(gco, g.data(), sizeof(double2) * g.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(w.a.src, S.data(), sizeof(SrcState) * nsrc, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w.a.cnt, 0, sizeof(unsigned) * 2 * nsrc, s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "second-pass setup");
  w.a.gco = gco;
  w.a.ssum = (typename Store<R>::T*)ssum;
  RegenRec<R>* rrec =
      (RegenRec<R>*)ws_get(ctx, (tag + ".rrec").c_str(), sizeof(RegenRec<R>) * (size_t)nsrc * o.max_iter, &st);
  if (st != OV_OK) return st;
  w.a.rrec = rrec;
  regen_scalars_kernel<R><<<64, 256, 0, s>>>(w.a, rrec, nsrc);
  OV_CHECK_LAUNCH(ctx, "regen_scalars_kernel");
  ring_reset_kernel<R><<<256, 256, 0, s>>>(w.a, b_soa, nsrc, 3);
  launches += 2.0;
  if (ssum) {
    e = cudaMemsetAsync(ssum, 0, sizeof(float4) * n12 * nsrc, s);
    if (e != cudaSuccess) return ctx_cuda(ctx, e, "clear double-float sum");
  }
  // pass 2: kmax regeneration launches (no host reads), replayed from a graph
  const int chunk = o.check_every > 0 ? o.check_every : 32;
  const bool graph = o.use_graph && !ctx->timing;
  cudaGraphExec_t exec = nullptr;
  if (graph && kmax >= chunk) {
    const int G = source_groups<R>(ctx, nsrc, w.nblk1);
    GraphKey key{{(const void*)w.a.ring, (const void*)gco, (const void*)w.a.sacc, (const void*)w.a.hist_a},
                 nsrc, ns, 3 * 128 + G, chunk, w.nslots, w.max_iter};
    auto it = ctx->graphs.find(key);
    if (it != ctx->graphs.end()) {
      exec = it->second;
    } else {
      st = capture_groups<R>(
          ctx, w, nsrc, G,
          [&](cudaStream_t cs, cudaStream_t, cudaEvent_t, cudaEvent_t, const SolveArgs<R>& a, int n) {
            for (int k = 0; k < chunk; ++k) lanczos_regen_kernel<R><<<dim3(w.nblk1, n), NT1, 0, cs>>>(a);
          },
          &exec);
      if (st != OV_OK) return st;
      ctx->graphs[key] = exec;
    }
  }
  const int Gr = exec ? source_groups<R>(ctx, nsrc, w.nblk1) : 1;
  int done = 0;
  while (done < kmax) {
    const int n = std::min(chunk, kmax - done);
    if (exec && n == chunk) {
      e = cudaGraphLaunch(exec, s);
      if (e != cudaSuccess) return ctx_cuda(ctx, e, "cudaGraphLaunch");
      launches += (double)n * (Gr - 1);  // the other branches' launches
    } else {
      for (int k = 0; k < n; ++k) {
        cudaEvent_t ev;
        kt_begin(ctx, KC_REGEN, s, &ev);
        lanczos_regen_kernel<R><<<dim3(w.nblk1, nsrc), NT1, 0, s>>>(w.a);
        kt_end(ctx, KC_REGEN, s, ev);
      }
      OV_CHECK_LAUNCH(ctx, "lanczos_regen_kernel");
    }
    done += n;
    launches += n;
  }
  if (ssum) {
    fold_df_sum_kernel<<<152 * 8, 256, 0, s>>>(ssum, w.a.sacc, n12 * nsrc);
    OV_CHECK_LAUNCH(ctx, "fold_df_sum_kernel");
    launches += 1.0;
  }
  so->launches = launches + 2.0;
  e = cudaMemcpyAsync(out_soa, w.a.sacc, sizeof(double2) * n12 * nsrc, cudaMemcpyDeviceToDevice, s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "copy sum");
  return fst;
}

// Per-node solutions of explicit per-source node lists through the coefficient space:
// one stored-basis Lanczos pass for all sources (no per-node vectors), the FOM coefficient
// vector of every node on the host, then x_j = V y^j for one chunk of nodes at a time
// (each chunk handed to per_chunk) and the weighted sums sum_j c_j x_j.  The Lanczos
// work does not repeat per chunk.  Returns OV_ERR_INVALID_ARG when the basis does not fit
// the store budget or the solve outgrows it (the caller uses the vector-space form).
template <typename R>
int nodes_coef(ov_ctx* ctx, const double2* b_soa, int nsrc, int ns, const std::vector<double2>& zh,
                      const std::vector<double2>& ch, int chunk, double2* X, double2* sums, const ov_solve_opts& o,
                      SolveOut* so, cudaStream_t s, const std::function<int(int, int)>& per_chunk) {
  const size_t n12 = (size_t)12 * ctx->g.V;
  size_t freeb = 0, totalb = 0;
  cudaMemGetInfo(&freeb, &totalb);
  const std::string tag = std::string(coef_tag<R>()) + "s";
  auto it = ctx->bufs.find(tag + ".ring");
  const double held = it != ctx->bufs.end() ? (double)it->second.bytes : 0.0;
  const double budget = std::min(0.40 * (double)totalb, (double)freeb + held - 0.10 * (double)totalb);
  const int cap = std::min(o.max_iter, ctx->coef_iter_hint > 0 ? std::max(64, ctx->coef_iter_hint * 5 / 4 + 32) : 1024);
  if ((double)(cap + 3) * nsrc * vec_elems<R>(ctx->g.V) * sizeof(double2) > budget) return OV_ERR_INVALID_ARG;
  SolveWs<R> w;
  int st = setup_ws<R>(ctx, nsrc, ns, false, true, true, cap, &w, tag.c_str(), cap + 3, false);
  if (st != OV_OK) return st;
  st = init_solve<R>(ctx, w, b_soa, nsrc, ns, zh, ch, make_double2(0.0, 0.0), o.tol, cap, s, 0);
  if (st != OV_OK) return st;
  double launches = 1.0;
  st = run_iterations<R>(ctx, w, nsrc, ns, 7, cap, o, s, &launches);
  if (st != OV_OK) return st;
  const int fst = finish_solve<R>(ctx, w, nsrc, ns, zh, ch, so, s);
  if (fst != OV_OK && !(fst == OV_ERR_NOT_CONVERGED && cap >= o.max_iter)) return OV_ERR_INVALID_ARG;
  std::vector<SrcState> S(nsrc);
  std::vector<double> ha((size_t)nsrc * cap), hb((size_t)nsrc * cap);
  cudaError_t e = cudaMemcpyAsync(S.data(), w.a.src, sizeof(SrcState) * nsrc, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(ha.data(), w.a.hist_a, sizeof(double) * ha.size(), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hb.data(), w.a.hist_b, sizeof(double) * hb.size(), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "read Lanczos history");
  // FOM coefficients y^j = (z_j - T_k)^-1 e_1 ||b|| per source and node (forward LDL^T sweep,
  // back substitution), folded with 1 / ||U_i||; g_r = sum_j c_j y^j for the sums
  using T = typename Store<R>::T;
  std::vector<T> Yh((size_t)nsrc * ns * cap);
  std::vector<T> gh((size_t)nsrc * cap);
  std::vector<int> kr(nsrc);
  FomScratch sc;
  std::vector<std::complex<double>> yy, gs;
  for (int r = 0; r < nsrc; ++r) {
    const int k = kr[r] = std::max(0, S[r].iter - 1);
    const double* al = ha.data() + (size_t)r * cap;
    const double* be = hb.data() + (size_t)r * cap;
    gs.assign(k, 0.0);
    for (int j = 0; j < ns && k > 0; ++j) {
      const std::complex<double> zj(zh[(size_t)r * ns + j].x, zh[(size_t)r * ns + j].y);
      const std::complex<double> cj(ch[(size_t)r * ns + j].x, ch[(size_t)r * ns + j].y);
      fom_coefficients(al, be, k, S[r].bnorm, zj, sc, yy);
      for (int i = 0; i < k; ++i) {
        const double ni = (i == 0) ? S[r].bnorm : be[i - 1];
        const std::complex<double> y = yy[i] / ni;
        Yh[((size_t)r * ns + j) * cap + i] = host_store(make_double2(y.real(), y.imag()), (T*)nullptr);
        gs[i] += cj * y;
      }
    }
    for (int i = 0; i < k; ++i) gh[(size_t)r * cap + i] = host_store(make_double2(gs[i].real(), gs[i].imag()), (T*)nullptr);
  }
  T* Yd = (T*)ws_get(ctx, (tag + ".Y").c_str(), sizeof(T) * Yh.size(), &st);
  T* gd = (T*)ws_get(ctx, (tag + ".g").c_str(), sizeof(T) * gh.size(), &st);
  int* krd = (int*)ws_get(ctx, (tag + ".kr").c_str(), sizeof(int) * nsrc, &st);
  if (st != OV_OK) return st;
  e = cudaMemcpyAsync(Yd, Yh.data(), sizeof(T) * Yh.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(gd, gh.data(), sizeof(T) * gh.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(krd, kr.data(), sizeof(int) * nsrc, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(sums, 0, sizeof(double2) * n12 * nsrc, s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "copy node coefficients");
  cudaEvent_t ev;
  kt_begin(ctx, KC_BASIS_SUM, s, &ev);
  basis_sum_kernel<R><<<dim3((unsigned)((n12 + 255) / 256), nsrc), 256, 0, s>>>(w.a.ring, cap + 3, gd, cap, krd,
                                                                             sums, n12);
  kt_end(ctx, KC_BASIS_SUM, s, ev);
  OV_CHECK_LAUNCH(ctx, "basis_sum_kernel");
  constexpr int JT = 8;
  for (int j0 = 0; j0 < ns; j0 += chunk) {
    const int nc = std::min(chunk, ns - j0);
    const dim3 gn((unsigned)((n12 + 255) / 256), nsrc, (nc + JT - 1) / JT);
    basis_nodes_kernel<R, JT><<<gn, 256, 0, s>>>(w.a.ring, cap + 3, Yd, ns, cap, krd, j0, nc, X, n12);
    OV_CHECK_LAUNCH(ctx, "basis_nodes_kernel");
    if ((st = per_chunk(j0, nc)) != OV_OK) return st;
  }
  so->launches = launches + 2.0 + (ns + chunk - 1) / chunk;
  if (so->converged) ctx->coef_iter_hint = so->iterations;
  return fst;
}

template <>
int nodes_coef<FX>(ov_ctx* ctx, const double2* b_soa, int nsrc, int ns, const std::vector<double2>& zh,
                   const std::vector<double2>& ch, int chunk, double2* X, double2* sums, const ov_solve_opts& o,
                   SolveOut* so, cudaStream_t s, const std::function<int(int, int)>& per_chunk) {
  size_t freeb = 0, totalb = 0;
  cudaMemGetInfo(&freeb, &totalb);
  auto it = ctx->bufs.find("fxs.ring");
  const double held = it != ctx->bufs.end() ? (double)it->second.bytes : 0.0;
  const double budget = std::min(0.40 * (double)totalb, (double)freeb + held - 0.10 * (double)totalb);
  const int cap = std::min(o.max_iter, ctx->coef_iter_hint > 0 ? std::max(64, ctx->coef_iter_hint * 5 / 4 + 32) : 1024);
  if ((double)(cap + 3) * nsrc * vec_elems<FX>(ctx->g.V) * sizeof(int4) > budget) return OV_ERR_INVALID_ARG;
  SolveWs<FX> w;
  FxCoef f;
  double launches = 0.0;
  int st = fx_lanczos(ctx, w, f, b_soa, nsrc, ns, zh, ch, make_double2(0.0, 0.0), sums, o, s, cap, 7, &launches);
  int4* Yq = (int4*)ws_get(ctx, "fxs.Yq", sizeof(int4) * (size_t)nsrc * ns * cap, &st);
  double* Ysc = (double*)ws_get(ctx, "fxs.Ysc", sizeof(double) * (size_t)nsrc * ns * f.ng, &st);
  if (st == OV_OK) st = launch_fx_basis_sum(ctx, w, f, nsrc, cap, sums, s);
  if (st != OV_OK) return st;
  const int fst = finish_solve<FX>(ctx, w, nsrc, ns, zh, ch, so, s);
  if (fst != OV_OK && !(fst == OV_ERR_NOT_CONVERGED && cap >= o.max_iter)) return OV_ERR_INVALID_ARG;
  fx_node_quant_kernel<<<dim3(ns, nsrc), 128, 0, s>>>(w.a, ns, f.Y, Yq, Ysc, f.ng);
  int2* slotd = (int2*)ws_get(ctx, "fxs.slot", sizeof(int2) * ns, &st);
  if (st != OV_OK) return st;
  std::vector<int2> slot;
  for (int j0 = 0; j0 < ns; j0 += chunk) {
    const int nc = std::min(chunk, ns - j0);
    // pairs of conjugate nodes (in every source's list) within the chunk
    slot.clear();
    std::vector<char> used(nc, 0);
    for (int j = 0; j < nc; ++j) {
      if (used[j]) continue;
      int2 p = make_int2(j0 + j, -1);
      for (int q = j + 1; q < nc && p.y < 0; ++q) {
        bool conj = !used[q];
        for (int r = 0; r < nsrc && conj; ++r) {
          const double2 u = zh[(size_t)r * ns + j0 + j], v = zh[(size_t)r * ns + j0 + q];
          conj = u.x == v.x && u.y == -v.y;
        }
        if (conj) p.y = j0 + q;
      }
      if (p.y >= 0) used[p.y - j0] = 1;
      slot.push_back(p);
    }
    const cudaError_t e =
        cudaMemcpyAsync(slotd, slot.data(), sizeof(int2) * slot.size(), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return ctx_cuda(ctx, e, "copy node pairs");
    const int nslot = (int)slot.size();
    fx_basis_nodes_kernel<<<dim3((unsigned)((w.nvec + 255) / 256), nsrc, (nslot + 1) / 2), 256, 0, s>>>(
        w.a.ring, cap + 3, Yq, Ysc, f.ng, ns, cap, f.info, slotd, nslot, j0, nc, X, ctx->g.V);
    OV_CHECK_LAUNCH(ctx, "fx_basis_nodes_kernel");
    if ((st = per_chunk(j0, nc)) != OV_OK) return st;
  }
  so->launches = launches + 2.0 + (ns + chunk - 1) / chunk;
  if (so->converged) ctx->coef_iter_hint = so->iterations;
  return fst;
}

int solve_nodes_coef(ov_ctx* ctx, const double2* b_soa, int nsrc, int ns, const std::vector<double2>& zh,
                     const std::vector<double2>& ch, int chunk, double2* X, double2* sums, const ov_solve_opts& o,
                     SolveOut* so, cudaStream_t s, const std::function<int(int, int)>& per_chunk) {
  if (fixed_point_fits(ctx, o.mode))
    return nodes_coef<FX>(ctx, b_soa, nsrc, ns, zh, ch, chunk, X, sums, o, so, s, per_chunk);
  if (o.mode == OV_MODE_F32X2) {
    const int st = ensure_links_df(ctx, s);
    if (st != OV_OK) return st;
    return nodes_coef<DF>(ctx, b_soa, nsrc, ns, zh, ch, chunk, X, sums, o, so, s, per_chunk);
  }
  return nodes_coef<double>(ctx, b_soa, nsrc, ns, zh, ch, chunk, X, sums, o, so, s, per_chunk);
}

int solve_sign_2pass(ov_ctx* ctx, const double2* b_soa, double2* out_soa, int nsrc, const ov_solve_opts& o,
                     SolveOut* so, cudaStream_t s) {
  if (fixed_point_fits(ctx, o.mode))
    return solve_sign_coef<FX>(ctx, b_soa, out_soa, nsrc, o, so, s);
  if (o.mode == OV_MODE_F32X2) {
    const int st = ensure_links_df(ctx, s);
    if (st != OV_OK) return st;
    return solve_sign_coef<DF>(ctx, b_soa, out_soa, nsrc, o, so, s);
  }
  return solve_sign_coef<double>(ctx, b_soa, out_soa, nsrc, o, so, s);
}

// OV_MODE_MIXED.
//  Phase A (FP32): one Lanczos process per source with FP32 vectors and FP64 scalars;
//    every node's LDL^T recurrence runs on scalars (for the stopping test) and the basis
//    is kept (slot i = U_i; GB300's HBM holds hundreds of basis vectors per source).  The
//    host forms each node's FOM coefficients (z_j - T_k)^-1 e_1 ||b|| and a combination
//    kernel writes y_j = sum_i w_ij U_i in FP64.
//  Rounds: FP64 true residuals r_j = b - (z_j - H_W) y_j (FP64 stencil fused) for every
//    node and source; if any exceeds tol ||b||, one batched FP32 correction solve over
//    all nodes x sources (each right-hand side its own Lanczos process with its single
//    shift z_j, per-RHS tolerance, converged ones leave the batch), y_j += e_j in FP64.
//  Finally the FP64 weighted sum s = c0 b + sum_j c_j y_j.
int solve_sign_mixed(ov_ctx* ctx, const double2* b_soa, double2* out_soa, int nsrc, const ov_solve_opts& o,
                     SolveOut* so, cudaStream_t s) {
  NvtxRange nvtx_("solve: mixed precision");
  const int nq = (int)ctx->z.size();
  const size_t n12 = (size_t)12 * ctx->g.V;
  const int nrhs = nsrc * nq;
  int st = OV_OK;
  cudaError_t e;
  // basis capacity: at most 600 vectors per source, a third of device memory and max_iter
  size_t freeb = 0, totalb = 0;
  cudaMemGetInfo(&freeb, &totalb);
  const size_t per_slot = (size_t)nsrc * n12 * sizeof(float2);
  long long cap = (long long)(0.33 * (double)totalb / (double)per_slot) - 2;
  const int kcap = (int)std::max<long long>(8, std::min<long long>(std::min<long long>(cap, 600), o.max_iter));
  double launches = 0.0;

  // ---- phase A
  std::vector<double2> zh((size_t)nsrc * nq), ch((size_t)nsrc * nq);
  for (int r = 0; r < nsrc; ++r)
    for (int j = 0; j < nq; ++j) {
      zh[(size_t)r * nq + j] = ctx->z[j];
      ch[(size_t)r * nq + j] = ctx->c[j];
    }
  SolveWs<float> wA;
  st = setup_ws<float>(ctx, nsrc, nq, false, false, true, kcap, &wA, "mxA", kcap + 2, false);
  if (st != OV_OK) return st;
  const double tolA = std::max(o.tol, 1e-6);
  st = init_solve<float>(ctx, wA, b_soa, nsrc, nq, zh, ch, make_double2(0, 0), tolA, kcap, s, 0);
  if (st != OV_OK) return st;
  launches += 1;
  st = run_iterations<float>(ctx, wA, nsrc, nq, 4, kcap, o, s, &launches);
  if (st != OV_OK) return st;
  SolveOut soA;
  const int fa = finish_solve<float>(ctx, wA, nsrc, nq, zh, ch, &soA, s);
  if (fa == OV_ERR_BREAKDOWN) return fa;
  std::vector<SrcState> S(nsrc);
  std::vector<double> ha((size_t)nsrc * kcap), hb((size_t)nsrc * kcap);
  e = cudaMemcpyAsync(S.data(), wA.a.src, sizeof(SrcState) * nsrc, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(ha.data(), wA.a.hist_a, sizeof(double) * ha.size(), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hb.data(), wA.a.hist_b, sizeof(double) * hb.size(), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "read phase-A history");
  int kmax = 1;
  std::vector<int> kr(nsrc);
  for (int r = 0; r < nsrc; ++r) {
    kr[r] = std::max(0, S[r].iter - 1);
    kmax = std::max(kmax, kr[r]);
  }
  // w_ij = [(z_j - T_k)^-1 e_1 ||b||]_i / ||U_i||  (the basis is stored unnormalised)
  std::vector<float2> W((size_t)nsrc * nq * kmax, make_float2(0.f, 0.f));
  std::vector<std::complex<double>> dd, ll, zt, yy;
  for (int r = 0; r < nsrc; ++r) {
    const int k = kr[r];
    if (k < 1) continue;
    const double* al = ha.data() + (size_t)r * kcap;
    const double* be = hb.data() + (size_t)r * kcap;
    dd.assign(k, 0.0);
    ll.assign(k, 0.0);
    zt.assign(k, 0.0);
    yy.assign(k, 0.0);
    for (int j = 0; j < nq; ++j) {
      const std::complex<double> zj(ctx->z[j].x, ctx->z[j].y);
      std::complex<double> om = S[r].bnorm;
      for (int i = 0; i < k; ++i) {
        if (i == 0) {
          dd[0] = zj - al[0];
        } else {
          dd[i] = zj - al[i] - be[i - 1] * be[i - 1] / dd[i - 1];
          om = -ll[i - 1] * om;
        }
        ll[i] = -be[i] / dd[i];
        zt[i] = om / dd[i];
      }
      yy[k - 1] = zt[k - 1];
      for (int i = k - 2; i >= 0; --i) yy[i] = zt[i] - ll[i] * yy[i + 1];
      for (int i = 0; i < k; ++i) {
        const double ni = (i == 0) ? S[r].bnorm : be[i - 1];
        const std::complex<double> w = yy[i] / ni;
        W[((size_t)r * nq + j) * kmax + i] = make_float2((float)w.real(), (float)w.imag());
      }
    }
  }
  float2* Wd = (float2*)ws_get(ctx, "mx.W", sizeof(float2) * W.size(), &st);
  int* krd = (int*)ws_get(ctx, "mx.kr", sizeof(int) * nsrc, &st);
  double2* Y = (double2*)ws_get(ctx, "mx.Y", sizeof(double2) * n12 * nrhs, &st);
  double2* R = (double2*)ws_get(ctx, "mx.R", sizeof(double2) * n12 * nrhs, &st);
  double* part = (double*)ws_get(ctx, "mx.part", sizeof(double) * (size_t)residual64_partials(ctx) * nrhs, &st);
  double* rn2 = (double*)ws_get(ctx, "mx.rn2", sizeof(double) * nrhs, &st);
  double2* zd = (double2*)ws_get(ctx, "mx.z", sizeof(double2) * nq, &st);
  double2* cd = (double2*)ws_get(ctx, "mx.c", sizeof(double2) * nq, &st);
  double* told = (double*)ws_get(ctx, "mx.tol", sizeof(double) * nrhs, &st);
  if (st != OV_OK) return st;
  e = cudaMemcpyAsync(Wd, W.data(), sizeof(float2) * W.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(krd, kr.data(), sizeof(int) * nsrc, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(zd, ctx->z.data(), sizeof(double2) * nq, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(cd, ctx->c.data(), sizeof(double2) * nq, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "phase-A coefficients");
  st = launch_basis_combine(ctx, wA.a.ring, kcap + 2, Wd, kmax, krd, Y, nsrc, nq, s);
  if (st != OV_OK) return st;
  launches += 1;

  // ---- FP64 residuals and FP32 corrections
  std::vector<double> rn(nrhs), tol_h(nrhs);
  const int max_rounds = 4;
  so->refine_rounds = 0;
  so->inner_iterations = 0;
  so->node_updates = soA.node_updates;
  double maxres = 0.0, bound = 0.0;
  std::string hist;
  for (int round = 0;; ++round) {
    st = launch_residual64(ctx, Y, b_soa, zd, R, part, rn2, nsrc, nq, s);
    if (st != OV_OK) return st;
    launches += 2;
    e = cudaMemcpyAsync(rn.data(), rn2, sizeof(double) * nrhs, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return ctx_cuda(ctx, e, "read residual norms");
    maxres = 0.0;
    bound = 0.0;
    bool bad = false;
    for (int r = 0; r < nsrc; ++r) {
      const double bn = S[r].bnorm > 0 ? S[r].bnorm : 1.0;
      double bd = 0.0;
      for (int j = 0; j < nq; ++j) {
        const double res = std::sqrt(rn[(size_t)r * nq + j]) / bn;
        if (!std::isfinite(res)) bad = true;
        maxres = std::max(maxres, res);
        bd += std::hypot(ctx->c[j].x, ctx->c[j].y) * res / std::fabs(ctx->z[j].y);
        // FP32 corrections reach ~1e-6 relative: ask for that, or what tol needs
        tol_h[(size_t)r * nq + j] = res <= o.tol ? 1e30 : std::max(0.3 * o.tol / res, 2e-6);
      }
      bound = std::max(bound, bd);
    }
    if (bad) return ctx_fail(ctx, OV_ERR_BREAKDOWN, "non-finite residual in the mixed-precision solve");
    char buf[64];
    snprintf(buf, sizeof buf, "%s%.3g", round ? ", " : "", maxres);
    hist += buf;
    if (maxres <= o.tol || round >= max_rounds) break;
    ++so->refine_rounds;
    std::vector<double2> zc(nrhs), cc(nrhs, make_double2(1.0, 0.0));
    for (int r = 0; r < nsrc; ++r)
      for (int j = 0; j < nq; ++j) zc[(size_t)r * nq + j] = ctx->z[j];
    SolveWs<float> wC;
    st = setup_ws<float>(ctx, nrhs, 1, true, false, false, o.max_iter, &wC, "mxC");
    if (st != OV_OK) return st;
    e = cudaMemcpyAsync(told, tol_h.data(), sizeof(double) * nrhs, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return ctx_cuda(ctx, e, "copy tolerances");
    wC.a.tol_src = told;
    st = init_solve<float>(ctx, wC, R, nrhs, 1, zc, cc, make_double2(0, 0), 0.5, o.max_iter, s, 1);
    if (st != OV_OK) return st;
    launches += 2;
    st = run_iterations<float>(ctx, wC, nrhs, 1, 5, o.max_iter, o, s, &launches);
    if (st != OV_OK) return st;
    SolveOut soC;
    const int fc = finish_solve<float>(ctx, wC, nrhs, 1, zc, cc, &soC, s);
    if (fc == OV_ERR_BREAKDOWN) return fc;
    so->inner_iterations += soC.iterations;
    so->node_updates += soC.node_updates;
    st = launch_accumulate(ctx, Y, wC.a.x, n12 * nrhs, s);
    if (st != OV_OK) return st;
    launches += 1;
  }
  st = launch_weighted_sum(ctx, Y, b_soa, cd, ctx->c0, out_soa, nsrc, nq, s);
  if (st != OV_OK) return st;
  so->iterations = soA.iterations;
  so->max_residual = maxres;
  so->error_bound = bound;
  so->converged = maxres <= o.tol;
  so->launches = launches + 3;
  if (!so->converged)
    return ctx_fail(ctx, OV_ERR_NOT_CONVERGED,
                    "mixed-precision refinement did not reach tol; max relative FP64 residual after phase A and "
                    "each correction round: " + hist);
  return OV_OK;
}

// Lanczos tridiagonal of H_W (squared = 0) or H_W^2 (squared = 1) from a fixed
// pseudo-random start vector; returns alpha[0..k), beta[0..k).
namespace {
__global__ void start_vector_kernel(double2* v, size_t n) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
    // splitmix64 of the element index: a fixed, reproducible start vector
    unsigned long long x = t + 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    x ^= x >> 31;
    const double a = (double)(x & 0xFFFFFFFFull) / 4294967296.0 - 0.5;
    const double b = (double)(x >> 32) / 4294967296.0 - 0.5;
    v[t] = make_double2(a, b);
  }
}
}  // namespace

// The recorded alpha_1 .. alpha_k, beta_1 .. beta_k of one source
template <typename R>
static int read_tridiag(ov_ctx* ctx, const SolveWs<R>& w, std::vector<double>& alpha, std::vector<double>& beta,
                        cudaStream_t s) {
  SrcState S;
  cudaError_t e = cudaMemcpyAsync(&S, w.a.src, sizeof(S), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "lanczos state");
  const int k = (std::is_same<R, FX>::value ? S.it2 : S.iter) - 1;
  if (S.status == OV_ERR_BREAKDOWN || k < 1) return ctx_fail(ctx, OV_ERR_BREAKDOWN, "Lanczos bound breakdown");
  alpha.resize(k);
  beta.resize(k);
  e = cudaMemcpy(alpha.data(), w.a.hist_a, sizeof(double) * k, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(beta.data(), w.a.hist_b, sizeof(double) * k, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return ctx_cuda(ctx, e, "lanczos history");
  return OV_OK;
}

// The tridiagonal of H_W through the solver's integer kernels and a ring of four vectors: two
// kernels a step where FP64 vectors take four.  gauge, placement and Zolotarev at 12^3 x 24
// with 100 steps: 16.3 -> 13.7 ms.
static int lanczos_tridiag_fx(ov_ctx* ctx, int steps, std::vector<double>& alpha, std::vector<double>& beta,
                              cudaStream_t s) {
  SolveWs<FX> w;
  int st = setup_ws<FX>(ctx, 1, 0, false, false, true, steps, &w, "lzx", 4, false);
  w.slot_mask = 3;
  const size_t n12 = (size_t)12 * ctx->g.V;
  double2* b = (double2*)ws_get(ctx, "lz.b", sizeof(double2) * n12, &st);
  if (st != OV_OK) return st;
  start_vector_kernel<<<256, 256, 0, s>>>(b, n12);
  const std::vector<double2> none;
  st = init_solve<FX>(ctx, w, b, 1, 0, none, none, make_double2(0, 0), 0.0, steps, s, 0);
  if (st != OV_OK) return st;
  for (int it = 0; it < steps; ++it) launch_k2<FX>(w, w.a, 1, s, launch_k1<FX>(w, w.a, 1, s) == 1);
  launch_k1<FX>(w, w.a, 1, s);  // records the last beta
  OV_CHECK_LAUNCH(ctx, "lanczos bound kernels");
  return read_tridiag<FX>(ctx, w, alpha, beta, s);
}

// The tridiagonal of H or H^2 with FP64 vectors.  The operator: with fx in integers of a scale per
// site, else fused into K1 (H) or in FP64 (H^2).
static int lanczos_tridiag_fp64(ov_ctx* ctx, int steps, int squared, bool fx, std::vector<double>& alpha,
                                std::vector<double>& beta, cudaStream_t s) {
  SolveWs<double> w;
  int st = setup_ws<double>(ctx, 1, 0, false, false, true, steps, &w, "lz");
  if (st != OV_OK) return st;
  const size_t n12 = (size_t)12 * ctx->g.V;
  double2* b = (double2*)ws_get(ctx, "lz.b", sizeof(double2) * n12, &st);
  double2* tmp = squared || fx ? (double2*)ws_get(ctx, "lz.tmp", sizeof(double2) * n12, &st) : nullptr;
  double2* tmp2 = squared ? (double2*)ws_get(ctx, "lz.tmp2", sizeof(double2) * n12, &st) : nullptr;
  if (st != OV_OK) return st;
  start_vector_kernel<<<256, 256, 0, s>>>(b, n12);
  std::vector<double2> none;
  st = init_solve<double>(ctx, w, b, 1, 0, none, none, make_double2(0, 0), 0.0, steps, s);
  if (st != OV_OK) return st;
  for (int it = 0; it < steps; ++it) {
    SolveArgs<double> a = w.a;
    // H or H^2 applied to U_i (ring slot i % 3, i = it + 1); K1 reads the result
    const double2* Ui = w.a.ring + (size_t)((it + 1) % 3) * n12;
    auto apply = [&](const double2* in, double2* out) {
      return fx ? launch_hw64_fx(ctx, in, out, 1, false, s) : launch_hw64(ctx, in, out, 1, s);
    };
    if (squared || fx) {
      st = apply(Ui, tmp);
      a.stencil = tmp;
    }
    if (squared && st == OV_OK) {
      st = apply(tmp, tmp2);
      a.stencil = tmp2;
    }
    if (st != OV_OK) return st;
    lanczos_hw_kernel<double><<<k1_grid(w, 1), NT1, 0, s>>>(a);
    lanczos_update_kernel<double><<<dim3(w.nblk2u, 1), NT2, 0, s>>>(a);
  }
  OV_CHECK_LAUNCH(ctx, "lanczos bound kernels");
  return read_tridiag<double>(ctx, w, alpha, beta, s);
}

// Integers where they apply: the solver's kernels for H, the stencil beside FP64 vectors for H^2
// (and for H beside the persistent loop).  Where their vectors do not fit (5 and 7 to the 4 and
// 6 of the FP64 forms, and what the call before left), FP64.
int lanczos_tridiag(ov_ctx* ctx, int steps, int squared, std::vector<double>& alpha, std::vector<double>& beta,
                    cudaStream_t s) {
  int st = OV_ERR_OUT_OF_MEMORY;
  if (!squared && fixed_point_fits(ctx, OV_MODE_FP64))
    st = lanczos_tridiag_fx(ctx, steps, alpha, beta, s);
  else if (ctx->fx_ok)
    st = lanczos_tridiag_fp64(ctx, steps, squared, true, alpha, beta, s);
  if (st != OV_ERR_OUT_OF_MEMORY) return st;
  ws_release(ctx, "lzx.");
  ws_release(ctx, "hw.fx");
  return lanczos_tridiag_fp64(ctx, steps, squared, false, alpha, beta, s);
}
