// Whole Newton solve of a short sequence inside one thread-block cluster (Algorithm 1 with
// the full Jacobian): one cluster per sequence runs every iteration itself,
// linearisation, convergence test and the scan of Eq. bin_op_affine, with the iterate
// kept in registers. There is no launch and no host round trip per iteration, and a
// batch of short sequences is one launch in which every cluster stops on its own
// convergence.
//
// The cluster's threads own contiguous rows of the sequence in (block rank, warp, lane)
// order, R rows each. One iteration:
//   1. each thread evaluates F_t = f_t(s_{t-1}) and A_t on its rows (the row before its
//      first comes from the previous thread through shared memory, from the previous
//      block's shared memory for the first thread, s_0 at the start), tests the residual
//      r_t = s_t - F_t and composes its rows' affine steps Delta -> A_t Delta - r_t into
//      one element (P, v);
//   2. the elements are reduced by trees (lanes of a warp, the block's warps, then the
//      blocks' totals read across the cluster behind one barrier) and the correction Delta
//      entering each thread's rows comes back down them;
//   3. the test and the iteration count follow the library's convergence check, taken
//      identically by every block; unless it stops, each thread propagates Delta through
//      its rows with the A_t and F_t it kept, adding it to the iterate with the reset
//      heuristic. The largest scaled residual and sum r^2 are formed once, at the end: the
//      decisions need only votes.
// Two cluster barriers per iteration: the boundary rows, then votes and totals.
//
// What bounds an iteration is its chain of FP64 instructions: a warp issues one per 64 clocks,
// whatever its active lanes. So a composition is spread over lanes, one entry of (P, v) each,
// and only vectors come down (44 instructions at d = 2, 1024 rows, against 150 for an
// inclusive scan of whole elements per lane), the rows spread over all four warps of a
// block, and comparisons work on the bit patterns. Brusselator,
// float64, T = 1024: 13.0 -> 7.2 us per iteration (a call of 28 iterations 374 -> 254 us, of
// which about 50 is the host); 64 x 2048 rows 3.24 -> 1.77 ms.
#include <cooperative_groups.h>

#include <cfloat>

#include "dyn.cuh"
#include "kernels.h"

namespace deer {

template <class real>
constexpr real kRealMax = sizeof(real) == 8 ? real(DBL_MAX) : real(FLT_MAX);

// Half an ulp of a tolerance (0 where that underflows).
__device__ __forceinline__ double half_ulp(double t) {
  const int e = (__double2hiint(t) >> 20) & 0x7ff;
  return e > 53 ? __hiloint2double((e - 53) << 20, 0) : 0.0;
}
__device__ __forceinline__ float half_ulp(float t) {
  const int e = (__float_as_int(t) >> 23) & 0xff;
  return e > 24 ? __int_as_float((e - 24) << 23) : 0.f;
}

// !(|r| / max(1, |s|) <= tol) as the division rounds, for tol >= 0, without dividing: the quotient
// rounds to tol or below exactly when |r| <= |s| (tol + half an ulp) (no quotient lies on that
// midpoint).
template <class real>
__device__ __forceinline__ bool over_tol(real r, real s, real tol) {
  if (!(rabs(s) > real(1))) return rabs(r) > tol;
  return fma(-tol, rabs(s), rabs(r)) > rabs(s) * half_ulp(tol);
}

// the leading 32 bits of |x|
__device__ __forceinline__ unsigned mag_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ unsigned mag_hi(float x) { return mag_bits(x); }

template <class real, int D>
struct Aff {  // the affine map Delta -> P Delta + v
  real P[D][D];
  real v[D];
};

// later o earlier
template <class real, int D>
__device__ __forceinline__ Aff<real, D> compose(const Aff<real, D>& l, const Aff<real, D>& e) {
  Aff<real, D> o;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    real x = l.v[i];
#pragma unroll
    for (int k = 0; k < D; ++k) x += l.P[i][k] * e.v[k];
    o.v[i] = x;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      real y = real(0);
#pragma unroll
      for (int k = 0; k < D; ++k) y += l.P[i][k] * e.P[k][j];
      o.P[i][j] = y;
    }
  }
  return o;
}

template <class real, int D>
__device__ __forceinline__ Aff<real, D> aff_identity() {
  Aff<real, D> o;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    o.v[i] = real(0);
#pragma unroll
    for (int j = 0; j < D; ++j) o.P[i][j] = i == j ? real(1) : real(0);
  }
  return o;
}

// Trees of affine maps in shared memory: n leaves (a power of two), the level of m nodes at
// offset 2 n - 2 m, an element as D rows of (P[i][0..D), v[i]).
template <int D>
constexpr int kEl = D * (D + 1);

// every node = later child o earlier child; one warp, one entry per lane and step
template <class real, int D>
__device__ __forceinline__ void tree_up(real* tree, int n, int lane) {
  constexpr int E = kEl<D>;
  for (int m = n >> 1; m >= 1; m >>= 1) {
    const real* child = tree + (2 * n - 4 * m) * E;
    real* node = tree + (2 * n - 2 * m) * E;
    for (int t = lane; t < m * E; t += 32) {
      const int q = t / E, e = t % E, i = e / (D + 1), j = e % (D + 1);
      const real* early = child + 2 * q * E;
      const real* late = early + E + i * (D + 1);
      real x = j == D ? late[D] : real(0);
#pragma unroll
      for (int k = 0; k < D; ++k) x += late[k] * early[k * (D + 1) + j];
      node[t] = x;
    }
    __syncwarp();
  }
}

// Delta entering every node from the one entering the root (x: D values per node, the tree's
// numbering)
template <class real, int D>
__device__ __forceinline__ void tree_down(const real* tree, real* x, int n, int lane) {
  constexpr int E = kEl<D>;
  for (int m = 1; m < n; m <<= 1) {
    const real* xp = x + (2 * n - 2 * m) * D;
    real* xc = x + (2 * n - 4 * m) * D;
    const real* child = tree + (2 * n - 4 * m) * E;
    for (int t = lane; t < m * D; t += 32) {
      const int q = t / D, i = t % D;
      const real* early = child + 2 * q * E + i * (D + 1);
      real y = early[D];
#pragma unroll
      for (int k = 0; k < D; ++k) y += early[k] * xp[q * D + k];
      xc[2 * q * D + i] = xp[t];
      xc[(2 * q + 1) * D + i] = y;
    }
    __syncwarp();
  }
}

__device__ __forceinline__ int pow2_at_least(int n) {
  int p = 1;
  while (p < n) p <<= 1;
  return p;
}

template <class real, int D, int KIND, int NT, int RPT>
__global__ void __launch_bounds__(NT) k_block_solve(BlockSolveArgs<real> a) {
  namespace cg = cooperative_groups;
  constexpr int NW = NT / 32, E = kEl<D>, MAXB = 16;
  // each warp's tree over its threads, and the Delta entering its nodes
  extern __shared__ __align__(16) unsigned char block_smem[];
  real (*s_tree)[63 * E] = reinterpret_cast<real (*)[63 * E]>(block_smem);
  real (*s_x)[63 * D] = reinterpret_cast<real (*)[63 * D]>(block_smem + sizeof(real) * NW * 63 * E);
  __shared__ real s_wtree[(2 * NW - 1) * E];  // the block's warps (root: the block's element)
  __shared__ real s_wx[(2 * NW - 1) * D];
  __shared__ real s_btree[(2 * MAXB - 1) * E];  // the blocks before this one
  __shared__ real s_last[NT][D];  // each thread's last row of the iterate
  __shared__ int s_votes[NW];     // 1: a row fails the test, 2: a non-finite entry
  __shared__ int s_vote;          // this block's (read across the cluster)
  __shared__ int s_all;           // the cluster's
  __shared__ real s_mx[NW];
  __shared__ double s_sq[NW];
  __shared__ double s_part[2];  // this block's max scaled residual and sum r^2
  cg::cluster_group cl = cg::this_cluster();
  const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int64_t seq = blockIdx.x / CL;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t r0 = a.offsets[seq];
  const int64_t T = a.offsets[seq + 1] - r0;
  // rows spread evenly over the cluster's blocks (rpc each, in rank order), then over a
  // block's warps (rpt rows for each of a warp's first `per` lanes; the host sizes the
  // cluster so that rpt <= RPT); the threads with rows are a prefix in (block, warp, lane)
  // order
  const int64_t rpc = (T + CL - 1) / CL;
  const int rpt = (int)((rpc + NT - 1) / NT);
  const int threads = rpt > 0 ? (int)((rpc + rpt - 1) / rpt) : 0;  // with rows, full block
  const int per = (threads + NW - 1) / NW;
  const int n = pow2_at_least(per);  // leaves of a warp's tree
  const int64_t cbeg = (int64_t)rank * rpc;
  const int64_t cend = cbeg + rpc < T ? cbeg + rpc : T;
  const int q = warp * per + lane;  // thread index among those with rows
  const int64_t k0 = cbeg + (int64_t)q * rpt;
  const int nmine = lane >= per || cend - k0 <= 0 ? 0 : (cend - k0 < rpt ? (int)(cend - k0) : rpt);
  // the last thread of the previous block (full whenever this one has rows)
  const int prev_last = threads - 1;
  const real scale = a.damp == DEER_DAMP_SCALE ? real(1) - a.dparam : real(1);
  // the test in the kernel's precision: the largest value not above tol. A negative or NaN
  // tolerance is met by nothing (the comparisons below drop its sign), also with no rows
  const bool tol_met = a.tol >= 0.0;
  const real tol = sizeof(real) == 8 ? (real)a.tol : (real)__double2float_rd(a.tol);
  const auto thr_bits = mag_bits(a.reset_thr);
  real s[RPT][D];
  real s0[D];
#pragma unroll
  for (int i = 0; i < D; ++i) s0[i] = a.s0[seq * D + i];
#pragma unroll
  for (int k = 0; k < RPT; ++k)
#pragma unroll
    for (int i = 0; i < D; ++i) s[k][i] = k < nmine ? a.s[(r0 + k0 + k) * D + i] : real(0);
  real last[D];  // this thread's last row
#pragma unroll
  for (int i = 0; i < D; ++i) last[i] = real(0);
#pragma unroll
  for (int k = 0; k < RPT; ++k)
#pragma unroll
    for (int i = 0; i < D; ++i) last[i] = k < nmine ? s[k][i] : last[i];
  int passes = 0;
  bool done = false, nonfinite = false;
  int iters = 0;
  real Fk[RPT][D], Ak[RPT][D][D];
  for (int it = 0;; ++it) {
    // the row before this thread's first is the previous thread's last, in this block or
    // in the previous block of the cluster; a thread without rows is followed only by
    // threads without rows
    if (nmine > 0) {
#pragma unroll
      for (int i = 0; i < D; ++i) s_last[q][i] = last[i];
    }
    cl.sync();
    real sp[D];
    if (nmine == 0) {
#pragma unroll
      for (int i = 0; i < D; ++i) sp[i] = real(0);  // unused: no rows
    } else if (q > 0) {
#pragma unroll
      for (int i = 0; i < D; ++i) sp[i] = s_last[q - 1][i];
    } else if (rank > 0) {
      const real* pl = cl.map_shared_rank(&s_last[prev_last][0], rank - 1);
#pragma unroll
      for (int i = 0; i < D; ++i) sp[i] = pl[i];
    } else {
#pragma unroll
      for (int i = 0; i < D; ++i) sp[i] = s0[i];
    }
    // 1. linearise, test, this thread's element; F and A are kept for the apply pass
    Aff<real, D> e = aff_identity<real, D>();
    bool fail = !tol_met, bad = false, near = false;
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      if (k < nmine) {
        eval_f<real, D, KIND, 1>(a.dv, seq, r0 + k0 + k, sp, Fk[k], Ak[k], nullptr);
        Aff<real, D> st;
#pragma unroll
        for (int i = 0; i < D; ++i) {
          const real r = s[k][i] - Fk[k][i];
          st.v[i] = -r;
          const unsigned rh = mag_hi(r), sh = mag_hi(s[k][i]);
          // |r| against tol max(1, |s|) by their leading 32 bits, where those differ enough
          const unsigned lh =
              mag_hi(sh >= mag_hi(real(1)) ? tol * rabs(s[k][i]) : tol);
          fail |= rh > lh + 2u;
          near |= rh - lh + 2u <= 4u;
          bad |= rh >= mag_hi(real(INFINITY)) || sh >= mag_hi(real(INFINITY));
#pragma unroll
          for (int j = 0; j < D; ++j) {
            if (scale != real(1)) Ak[k][i][j] *= scale;
            st.P[i][j] = Ak[k][i][j];
          }
        }
        if (k == 0) e = st;
        else e = compose<real, D>(st, e);
#pragma unroll
        for (int i = 0; i < D; ++i) sp[i] = s[k][i];
      }
    }
    if (__any_sync(0xffffffffu, near)) {  // (rare)
#pragma unroll
      for (int k = 0; k < RPT; ++k)
        if (k < nmine) {
#pragma unroll
          for (int i = 0; i < D; ++i)
            fail |= over_tol(s[k][i] - Fk[k][i], s[k][i], tol);
        }
    }
    // 2. votes and elements up the trees
    const int vote = (__any_sync(0xffffffffu, fail) ? 1 : 0) | (__any_sync(0xffffffffu, bad) ? 2 : 0);
    if (lane == 0) s_votes[warp] = vote;
    real* tree = s_tree[warp];
    if (lane < n) {
#pragma unroll
      for (int i = 0; i < D; ++i) {
#pragma unroll
        for (int j = 0; j < D; ++j) tree[lane * E + i * (D + 1) + j] = e.P[i][j];
        tree[lane * E + i * (D + 1) + D] = e.v[i];
      }
    }
    __syncwarp();
    tree_up<real, D>(tree, n, lane);
    for (int t = lane; t < E; t += 32) s_wtree[warp * E + t] = tree[(2 * n - 2) * E + t];
    __syncthreads();
    if (warp == 0) {
      tree_up<real, D>(s_wtree, NW, lane);
      if (lane == 0) {
        int v = 0;
        for (int w = 0; w < NW; ++w) v |= s_votes[w];
        s_vote = v;
      }
    }
    cl.sync();
    if (warp == 0) {
      // the cluster's vote; the blocks before this one: Delta entering this block
      const int v = lane < CL ? *cl.map_shared_rank(&s_vote, lane) : 0;
      const int any = (__any_sync(0xffffffffu, v & 1) ? 1 : 0) |
                      (__any_sync(0xffffffffu, v & 2) ? 2 : 0);
      const int nb = pow2_at_least(rank);
      for (int t = lane; t < nb * E; t += 32) {
        const int b = t / E, x = t % E;
        s_btree[t] = b < rank ? *cl.map_shared_rank(&s_wtree[(2 * NW - 2) * E + x], b)
                              : (x % (D + 1) == x / (D + 1) ? real(1) : real(0));
      }
      __syncwarp();
      tree_up<real, D>(s_btree, nb, lane);
      if (lane < D)
        s_wx[(2 * NW - 2) * D + lane] =
            rank > 0 ? s_btree[(2 * nb - 2) * E + lane * (D + 1) + D] : real(0);
      if (lane == 0) s_all = any;
      __syncwarp();
      tree_down<real, D>(s_wtree, s_wx, NW, lane);
    }
    __syncthreads();
    const int all = s_all;
    nonfinite = (all & 2) != 0;
    passes = all == 0 ? passes + 1 : 0;
    if (passes >= a.confirm) {
      done = true;
      iters = it;
      break;
    }
    iters = it < a.max_iters ? it + 1 : it;
    if ((nonfinite && !a.reset) || it >= a.max_iters) break;
    // 3. Delta down to this thread, then through its rows
    real* xs = s_x[warp];
    if (lane < D) xs[(2 * n - 2) * D + lane] = s_wx[warp * D + lane];
    __syncwarp();
    tree_down<real, D>(tree, xs, n, lane);
    real din[D];
#pragma unroll
    for (int i = 0; i < D; ++i) din[i] = lane < n ? xs[lane * D + i] : real(0);
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      if (k < nmine) {
        real dn[D];
#pragma unroll
        for (int i = 0; i < D; ++i) {
          real x = Fk[k][i] - s[k][i];
#pragma unroll
          for (int j = 0; j < D; ++j) x += Ak[k][i][j] * din[j];
          dn[i] = x;
        }
#pragma unroll
        for (int i = 0; i < D; ++i) {
          const real y = s[k][i] + dn[i];
          s[k][i] = a.reset && mag_bits(y) > thr_bits ? real(0) : y;
          last[i] = s[k][i];
          din[i] = dn[i];
        }
      }
    }
    // (the next iteration's first cluster barrier orders the rewrites of the shared
    // buffers after every block's reads of them)
  }
  // The statistics of the last iterate: the largest scaled residual |r| / max(1, |s|), kept as
  // a fraction fn / fd compared by cross-multiplication (one division per warp), and sum r^2.
  {
    real fn = real(0), fd = real(1);
    bool fnan = false;
    double sq = 0.0;
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      if (k < nmine) {
#pragma unroll
        for (int i = 0; i < D; ++i) {
          const real r = s[k][i] - Fk[k][i];
          const real sabs = rabs(s[k][i]);
          const real num = rabs(r), den = sabs > real(1) ? sabs : real(1);
          if (!(num <= kRealMax<real>) || !(den <= kRealMax<real>)) {
            fnan = true;
          } else if (num * fd > fn * den) {
            fn = num;
            fd = den;
          }
          sq += (double)r * (double)r;
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const real on = __shfl_xor_sync(0xffffffffu, fn, o);
      const real od = __shfl_xor_sync(0xffffffffu, fd, o);
      fnan |= __shfl_xor_sync(0xffffffffu, (int)fnan, o) != 0;
      if (on * fd > fn * od) {
        fn = on;
        fd = od;
      }
      sq += __shfl_xor_sync(0xffffffffu, sq, o);
    }
    if (lane == 0) {
      s_mx[warp] = fnan ? real(NAN) : fn / fd;
      s_sq[warp] = sq;
    }
    __syncthreads();
    if (tid == 0) {
      double bm = 0.0, bs = 0.0;
      for (int w = 0; w < NW; ++w) {
        bm = nanmax(bm, (double)s_mx[w]);
        bs += s_sq[w];
      }
      s_part[0] = bm;
      s_part[1] = bs;
    }
  }
#pragma unroll
  for (int k = 0; k < RPT; ++k)
    if (k < nmine)
#pragma unroll
      for (int i = 0; i < D; ++i) a.s[(r0 + k0 + k) * D + i] = s[k][i];
  cl.sync();
  if (tid == 0 && rank == 0) {
    double bm = 0.0, bs = 0.0;
    for (int b = 0; b < CL; ++b) {
      const double* pp = cl.map_shared_rank(&s_part[0], b);
      bm = nanmax(bm, pp[0]);
      bs += pp[1];
    }
    SeqInfo inf = a.info[seq];
    inf.iters = iters;
    inf.done = done ? 1 : 0;
    inf.passes = passes;
    inf.merit = 0.5 * bs;
    inf.max_resid = bm;
    a.info[seq] = inf;
    if (nonfinite) atomicAdd(&a.flags->n_nonfinite, 1);
    if (done) atomicSub(&a.flags->n_active, 1);  // the active-set pass counted every sequence
  }
  cl.sync();  // no block leaves while another may still read its shared memory
}

// Threads per block and the most rows per thread by state size (each thread keeps its
// rows' iterate, F_t and A_t in registers). A sequence is spread over a cluster of up to
// 16 blocks (one row per thread where it fits), whose shared memory the blocks read from
// each other: the more SMs, the more of the GPU's float64 units (a small fraction of its
// float32 rate) a single sequence gets.
constexpr int kBlockThreads = 128;
constexpr int kMaxCluster = 8;    // portable cluster size: sets the longest sequence taken
constexpr int kWideCluster = 16;  // non-portable, used when the GPU schedules it
template <int D>
struct BlockRows { static constexpr int n = D <= 2 ? 8 : 2; };

int64_t block_solve_max_T(int kind, int d) {
  const bool kind_ok = kind == DEER_F_BRUSSELATOR_EULER || kind == DEER_F_MASSACTION_EULER ||
                       kind == DEER_F_MASSACTION_RK4 || kind == DEER_F_LINEAR ||
                       kind == DEER_F_RNN_TANH || kind == DEER_F_LANGEVIN_2WELL;
  if (!kind_ok) return 0;
  const int64_t per = (int64_t)kMaxCluster * kBlockThreads;
  switch (d) {
    case 1: return per * BlockRows<1>::n;
    case 2: return per * BlockRows<2>::n;
    case 4: return per * BlockRows<4>::n;
    default: return 0;
  }
}

template <class real, int D, int KIND>
static cudaError_t block_launch(const BlockSolveArgs<real>& a, cudaStream_t st) {
  auto kern = k_block_solve<real, D, KIND, kBlockThreads, BlockRows<D>::n>;
  // cluster size: 64 rows per block where the longest sequence allows it (the float64
  // pipe is the SM's, shared by its warps), up to 16 blocks when the GPU can schedule
  // that, else 8
  int64_t cl = (a.max_T + kBlockThreads / 2 - 1) / (kBlockThreads / 2);
  cl = cl < 1 ? 1 : (cl > kWideCluster ? kWideCluster : cl);
  if (cl > kMaxCluster) {
    static DeviceOnce wide;
    int dev = 0;
    cudaGetDevice(&dev);
    if (wide.ensure(dev, [&] {
          return cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        }) != cudaSuccess)
      cl = kMaxCluster;
    (void)cudaGetLastError();
  }
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.blockDim = dim3(kBlockThreads, 1, 1);
  cfg.dynamicSmemBytes = sizeof(real) * (kBlockThreads / 32) * 63 * (kEl<D> + D);
  static DeviceOnce smem_ok;
  const cudaError_t se = allow_smem(smem_ok, kern, cfg.dynamicSmemBytes);
  if (se != cudaSuccess) return se;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  for (;;) {
    attr[0].val.clusterDim.x = (unsigned)cl;
    cfg.gridDim = dim3((unsigned)(a.B * cl), 1, 1);
    // a cluster of 16 that cannot be placed: take 8 instead (the longest sequence taken
    // fits 8)
    if (cl > kMaxCluster) {
      // (asked once per host thread, device and cluster size: the query takes longer than the
      // launch)
      static thread_local signed char placed[16][kWideCluster + 1] = {};
      int dev = 0;
      cudaGetDevice(&dev);
      signed char unknown = 0;
      signed char& fits = dev < 16 ? placed[dev][cl] : unknown;
      if (fits == 0) {
        int nclusters = 0;
        fits = cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) == cudaSuccess &&
                       nclusters >= 1 ? 1 : -1;
        (void)cudaGetLastError();
      }
      if (fits < 0) {
        cl = kMaxCluster;
        continue;
      }
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, a);
    if (e != cudaSuccess && cl > kMaxCluster) {
      (void)cudaGetLastError();
      cl = kMaxCluster;
      continue;
    }
    if (e == cudaSuccess) note_launch();
    return e;
  }
}

template <class real, int D>
static cudaError_t block_kind(const BlockSolveArgs<real>& a, cudaStream_t st) {
  switch (a.dv.kind) {
    case DEER_F_BRUSSELATOR_EULER:
      if constexpr (D == 2) return block_launch<real, D, DEER_F_BRUSSELATOR_EULER>(a, st);
      return cudaErrorInvalidValue;
    case DEER_F_MASSACTION_EULER:
      if constexpr (D >= 2) return block_launch<real, D, DEER_F_MASSACTION_EULER>(a, st);
      return cudaErrorInvalidValue;
    case DEER_F_MASSACTION_RK4:
      if constexpr (D >= 2) return block_launch<real, D, DEER_F_MASSACTION_RK4>(a, st);
      return cudaErrorInvalidValue;
    case DEER_F_LINEAR: return block_launch<real, D, DEER_F_LINEAR>(a, st);
    case DEER_F_RNN_TANH: return block_launch<real, D, DEER_F_RNN_TANH>(a, st);
    case DEER_F_LANGEVIN_2WELL: return block_launch<real, D, DEER_F_LANGEVIN_2WELL>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

template <class real>
cudaError_t launch_block_solve(const BlockSolveArgs<real>& a, cudaStream_t st) {
  if (a.B == 0) return cudaSuccess;
  switch (a.dv.d) {
    case 1: return block_kind<real, 1>(a, st);
    case 2: return block_kind<real, 2>(a, st);
    case 4: return block_kind<real, 4>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t launch_block_solve<float>(const BlockSolveArgs<float>&, cudaStream_t);
template cudaError_t launch_block_solve<double>(const BlockSolveArgs<double>&, cudaStream_t);

}  // namespace deer
