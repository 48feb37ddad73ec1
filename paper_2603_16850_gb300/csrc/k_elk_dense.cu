// Dense (full-Jacobian) ELK (Sec. 4.2-4.3): the Kalman filter of the linearised dynamics
// s_t = A_t s_{t-1} + b_t + N(0, I) with the previous iterate as emissions, variance 1/lambda.
// In the correction form of the scan the filtered mean is a linear recurrence again:
// Delta_t = Gamma_t A_t Delta_{t-1} - Gamma_t r_t, Gamma_t = (I + lambda P^-_t)^{-1}, where
// P^-_t = A_t P_{t-1} A_t^T + I, P_t = Gamma_t P^-_t and P = 0 before the first solved row
// (s_0, or the frozen state under a sliding window, is known). This kernel runs the
// covariance recursion and rewrites A_t <- Gamma_t A_t, b_t <- Gamma_t b_t in place; the
// dense scan then solves the mean in parallel over t. The covariance recursion does not
// depend on the emissions, only on A_t; it is a dependent chain over t, run per sequence, or,
// for few, long sequences, in parallel over time (chunk elements, carry, then this recursion
// per chunk from the carried covariance; see below).
//
// What bounds these kernels is the chain of small dense products and inverses per row: in
// float64 a warp issues one FP64 instruction per 64 clocks whatever the number of active
// lanes, so a row costs its FP64 instruction count. Each chunk (or sequence) gets a group of
// min(32, d^2) lanes, or more in the carry, and every d x d product is spread over all of
// them, one or a few entries per lane (16 instructions per product at d = 8 against 64 with a
// row per lane); inverses are in place (half the entries of an augmented elimination) and
// their reciprocals take four FP64 instructions of 64 clocks instead of a division's 1490. Mass action d = 8,
// float64, 4 sequences of 4096 rows, per iteration (d lanes per chunk, a row per lane, blocks
// of 16 chunks before): chunk elements 2626 -> 300 us, carry 1696 (64 steps) -> 536 (128
// steps, 4.2 us each: pivots in order), restart 1538 -> 194 us.
#include "kernels.h"

namespace deer {
namespace {

// Lanes of the group that owns one chunk (or sequence): a warp or part of one; in the carry
// pass of d >= 8 a block of several warps (one block per sequence).
template <int D>
constexpr int elk_lanes() { return D * D < 32 ? D * D : 32; }
template <int D>
constexpr int elk_carry_lanes() { return D == 8 ? 64 : D == 16 ? 128 : elk_lanes<D>(); }

// larger magnitude = larger key, from the bit pattern (no FP64 comparison)
__device__ __forceinline__ int mag_key(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ int mag_key(float x) { return __float_as_int(x) & 0x7fffffff; }

// d x d matrices of a group: entry e = lane + m GW (row e / D, column e % D) is slot m of a
// lane; operands are read from shared memory (rows padded against bank conflicts).
template <class real, int D, int GW>
struct Grp {
  static constexpr int EPL = D * D / GW;
  static constexpr int RS = D + (D >= 4 ? 16 / (int)sizeof(real) : 1);
  static constexpr int SZ = D * RS;
  int lane;
  unsigned mask;

  __device__ __forceinline__ Grp() {
    lane = threadIdx.x % GW;
    mask = GW >= 32 ? 0xffffffffu : ((1u << (GW & 31)) - 1u) << (threadIdx.x & 31 & ~(GW - 1));
  }
  __device__ __forceinline__ void sync() const {
    if constexpr (GW > 32) __syncthreads();  // the block is the group
    else __syncwarp(mask);
  }
  __device__ __forceinline__ int row(int m) const { return (lane + m * GW) / D; }
  __device__ __forceinline__ int col(int m) const { return (lane + m * GW) % D; }
  __device__ __forceinline__ real eye(int m) const { return row(m) == col(m) ? real(1) : real(0); }
  __device__ __forceinline__ void store(real* M, const real (&v)[EPL]) const {
#pragma unroll
    for (int m = 0; m < EPL; ++m) M[row(m) * RS + col(m)] = v[m];
  }
  // row-major dense blocks in global memory
  __device__ __forceinline__ void gload(const real* g, real (&v)[EPL]) const {
#pragma unroll
    for (int m = 0; m < EPL; ++m) v[m] = g[lane + m * GW];
  }
  __device__ __forceinline__ void gstore(real* g, const real (&v)[EPL]) const {
#pragma unroll
    for (int m = 0; m < EPL; ++m) g[lane + m * GW] = v[m];
  }
  __device__ __forceinline__ void fetch(real* M, const real* g) const {
#pragma unroll
    for (int m = 0; m < EPL; ++m)
      cp_async_small<sizeof(real)>(M + row(m) * RS + col(m), g + lane + m * GW);
  }
  // entries of op(X) op(Y), op = transpose where TX / TY
  template <bool TX, bool TY>
  __device__ __forceinline__ void mul(const real* X, const real* Y, real (&v)[EPL]) const {
#pragma unroll
    for (int m = 0; m < EPL; ++m) v[m] = real(0);
#pragma unroll(D <= 8 ? D : 2)
    for (int k = 0; k < D; ++k)
#pragma unroll
      for (int m = 0; m < EPL; ++m)
        v[m] += X[TX ? k * RS + row(m) : row(m) * RS + k] *
                Y[TY ? col(m) * RS + k : k * RS + col(m)];
  }
  // Gauss-Jordan inverse of the matrix in M0, in place (M1: scratch of the same size). With
  // PIVOT, the pivot of column c is the unused row w_c of largest magnitude; rows stay where
  // they are, and at the end row w_c holds row c of the inverse, its stored column k belonging
  // to right-hand side w_k. The result is left in `out` (not M0 or M1).
  template <bool PIVOT>
  __device__ __forceinline__ void inverse(real* M0, real* M1, real* out) const {
    unsigned long long where = 0ull;  // 4 bits per column: w_c
    unsigned used = 0u;
    real v[EPL];
#pragma unroll(D <= 8 ? D : 1)
    for (int c = 0; c < D; ++c) {
      const real* src = c & 1 ? M1 : M0;
      real* dst = c & 1 ? M0 : M1;
      int w = c;
      if constexpr (PIVOT) {
        int best = -2;
#pragma unroll
        for (int i = 0; i < D; ++i) {
          const int key = (used >> i) & 1u ? -1 : mag_key(src[i * RS + c]);
          if (key > best) { best = key; w = i; }
        }
        used |= 1u << w;
        where |= (unsigned long long)w << (4 * c);
      }
      const real ip = recip(src[w * RS + c]);
#pragma unroll
      for (int m = 0; m < EPL; ++m) {
        const int i = row(m), j = col(m);
        // the pivot row is scaled (its pivot entry becomes 1 / p); the others lose their
        // pivot-column entry f times it (that entry itself becomes -f / p)
        const real q = (j == c ? real(1) : src[w * RS + j]) * ip;
        const real o = j == c ? real(0) : src[i * RS + j];
        v[m] = i == w ? q : o - src[i * RS + c] * q;
        if (c < D - 1) dst[i * RS + j] = v[m];
      }
      if (c < D - 1) sync();
    }
#pragma unroll
    for (int m = 0; m < EPL; ++m) {
      int i = row(m), j = col(m);
      if constexpr (PIVOT) {
        int c = 0;
#pragma unroll
        for (int k = 0; k < D; ++k)
          if ((int)((where >> (4 * k)) & 15ull) == i) c = k;
        i = c;
        j = (int)((where >> (4 * j)) & 15ull);
      }
      out[i * RS + j] = v[m];
    }
    sync();
  }
};

}  // namespace

// One group per sequence (CHUNKED = false: the covariance starts at zero at the sequence's
// first row) or per chunk (CHUNKED = true: it starts from the filtered covariance the carry
// pass computed for the chunk).
template <class real, int D, bool CHUNKED>
__global__ void __launch_bounds__(32) k_elk_dense(ElkDenseArgs<real> a) {
  constexpr int GW = elk_lanes<D>();
  using G = Grp<real, D, GW>;
  constexpr int EPL = G::EPL, SZ = G::SZ;
  __shared__ real sm[32 / GW][8 * SZ];
  __shared__ real sb[32 / GW][2][D];
  const G g;
  const int grp = threadIdx.x / GW;
  real* F[2] = {sm[grp], sm[grp] + SZ};
  real *P = sm[grp] + 2 * SZ, *T = sm[grp] + 3 * SZ, *Pm = sm[grp] + 4 * SZ;
  real *S0 = sm[grp] + 5 * SZ, *S1 = sm[grp] + 6 * SZ, *N = sm[grp] + 7 * SZ;
  const int64_t k = blockIdx.x * (int64_t)(32 / GW) + grp;
  int64_t r0, r1;
  real v[EPL], u[EPL];
#pragma unroll
  for (int m = 0; m < EPL; ++m) v[m] = real(0);
  if constexpr (CHUNKED) {
    if (k >= a.bt.act_chunks()) return;  // whole groups
    int64_t seq, c;
    int n;
    act_chunk(a.bt, k, seq, c, r0, n);
    r1 = r0 + n;
    g.gload(a.cov_in + c * (int64_t)(D * D), v);
  } else {
    if (k >= a.bt.n_act()) return;  // whole groups
    const int64_t seq = a.bt.act_seq[k];
    const int64_t cf = a.bt.chunk_first[seq];
    r0 = a.bt.offsets[seq] + ((win_first(a.bt, seq) - cf) << a.bt.log2L);
    r1 = a.bt.offsets[seq + 1];
  }
  g.store(P, v);
  auto fetch = [&](int64_t row) {
    if (row < r1) {
      const int s = (int)((row - r0) & 1);
      g.fetch(s ? F[1] : F[0], a.A + row * (int64_t)(D * D));
      if (g.lane < D) cp_async_small<sizeof(real)>(&sb[grp][s][g.lane], a.b + row * D + g.lane);
    }
    cp_async_commit();
  };
  fetch(r0);
  for (int64_t row = r0; row < r1; ++row) {
    const int s = (int)((row - r0) & 1);
    real* Ft = s ? F[1] : F[0];
    cp_async_wait<0>();
    g.sync();
    fetch(row + 1);
    // P^- = F P F^T + I, S = I + lambda P^-
    g.template mul<false, false>(Ft, P, v);
    g.store(T, v);
    g.sync();
    g.template mul<false, true>(T, Ft, v);
#pragma unroll
    for (int m = 0; m < EPL; ++m) {
      v[m] += g.eye(m);
      u[m] = g.eye(m) + a.lambda * v[m];
    }
    g.store(Pm, v);
    g.store(S0, u);
    g.sync();
    // Gamma = S^{-1} (symmetric positive definite: no pivoting)
    g.template inverse<false>(S0, S1, N);
    // P = Gamma P^-, A <- Gamma A, b <- Gamma b (the lanes of a row share its sum)
    g.template mul<false, false>(N, Pm, v);
    g.store(P, v);
    g.template mul<false, false>(N, Ft, u);
    g.gstore(a.A + row * (int64_t)(D * D), u);
    constexpr int PARTS = GW / D;
    const int i = g.lane / PARTS;
    real x = real(0);
#pragma unroll
    for (int q = 0; q < D / PARTS; ++q) {
      const int kk = q * PARTS + g.lane % PARTS;
      x += N[i * G::RS + kk] * sb[grp][s][kk];
    }
#pragma unroll
    for (int o = 1; o < PARTS; o <<= 1) x += __shfl_xor_sync(g.mask, x, o, GW);
    if (g.lane % PARTS == 0) a.b[row * D + i] = x;
  }
  cp_async_wait<0>();
}

// ---------------------------------------------------------------------------
// The covariance recursion in parallel over time. One filtering step maps the incoming
// covariance P to A (I + P J)^{-1} P A^T + C with the step's element
// (A, C, J) = (c F_t, c I, lambda c F_t^T F_t), c = 1 / (1 + lambda) (process noise I,
// emission variance 1/lambda); elements combine associatively, e_i then e_j giving
// (A_j N A_i, A_j N C_i A_j^T + C_j, A_i^T J_j N A_i + J_i) with N = (I + C_i J_j)^{-1}
// (Sarkka and Garcia-Fernandez's parallel Kalman filter; N^T J_j = J_j N). The chunk pass
// folds each chunk's elements in order; the carry pass walks a sequence's chunks applying
// their aggregates to the covariance (one short chain per sequence: T / L steps instead of
// T); the per-chunk recursion above then rewrites (A_t, b_t) from the carried covariance.
// Inverses with partial pivoting (I + C J is not symmetric).
// ---------------------------------------------------------------------------
template <class real, int D>
__global__ void __launch_bounds__(32) k_elk_cov_chunk(ElkDenseArgs<real> a) {
  constexpr int GW = elk_lanes<D>();
  using G = Grp<real, D, GW>;
  constexpr int EPL = G::EPL, SZ = G::SZ;
  __shared__ real sm[32 / GW][9 * SZ];
  const G g;
  const int grp = threadIdx.x / GW;
  const int64_t k = blockIdx.x * (int64_t)(32 / GW) + grp;
  if (k >= a.bt.act_chunks()) return;  // whole groups
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, k, seq, c, r0, n);
  real* F0 = sm[grp];
  real *F1 = F0 + SZ, *A = F0 + 2 * SZ, *C = F0 + 3 * SZ, *J = F0 + 4 * SZ;
  real *S0 = F0 + 5 * SZ, *S1 = F0 + 6 * SZ, *N = F0 + 7 * SZ, *X = F0 + 8 * SZ;
  const real lam = a.lambda, cc = real(1) / (real(1) + lam);
  real ca[EPL], aa[EPL], ja[EPL], v[EPL], w[EPL];
  auto fetch = [&](int t) {
    if (t < n) g.fetch(t & 1 ? F1 : F0, a.A + (r0 + t) * (int64_t)(D * D));
    cp_async_commit();
  };
  fetch(0);
  for (int t = 0; t < n; ++t) {
    real* F = t & 1 ? F1 : F0;
    cp_async_wait<0>();
    g.sync();
    fetch(t + 1);
    g.template mul<true, false>(F, F, v);
#pragma unroll
    for (int m = 0; m < EPL; ++m) v[m] *= lam * cc;
    if (t == 0) {
#pragma unroll
      for (int m = 0; m < EPL; ++m) {
        aa[m] = cc * F[g.row(m) * G::RS + g.col(m)];
        ca[m] = cc * g.eye(m);
        ja[m] = v[m];
      }
    } else {
      g.store(J, v);  // the row's J
      g.sync();
      // N = (I + C_a J)^{-1}
      g.template mul<false, false>(C, J, v);
#pragma unroll
      for (int m = 0; m < EPL; ++m) v[m] += g.eye(m);
      g.store(S0, v);
      g.sync();
      g.template inverse<true>(S0, S1, N);
      // X = N A_a, Y = N C_a, V = J A_a
      g.template mul<false, false>(N, A, v);
      g.store(X, v);
      g.template mul<false, false>(N, C, v);
      g.store(S0, v);
      g.template mul<false, false>(J, A, v);
      g.store(S1, v);
      g.sync();
      // A = c F X, Z = F Y, J = J_a + V^T X, C = c^2 Z F^T + c I
      g.template mul<false, false>(F, X, aa);
      g.template mul<false, false>(F, S0, v);
      g.store(N, v);
      g.template mul<true, false>(S1, X, w);
      g.sync();
      g.template mul<false, true>(N, F, ca);
#pragma unroll
      for (int m = 0; m < EPL; ++m) {
        aa[m] *= cc;
        ca[m] = cc * cc * ca[m] + cc * g.eye(m);
        ja[m] += w[m];
      }
    }
    g.store(A, aa);
    g.store(C, ca);
  }
  cp_async_wait<0>();
  real* out = a.cov_agg + c * (int64_t)(3 * D * D);
  g.gstore(out, aa);
  g.gstore(out + D * D, ca);
  g.gstore(out + 2 * D * D, ja);
}

template <class real, int D>
__global__ void __launch_bounds__(elk_carry_lanes<D>() < 32 ? 32 : elk_carry_lanes<D>())
    k_elk_cov_carry(ElkDenseArgs<real> a) {
  constexpr int GW = elk_carry_lanes<D>();
  constexpr int GPB = GW < 32 ? 32 / GW : 1;
  using G = Grp<real, D, GW>;
  constexpr int EPL = G::EPL, SZ = G::SZ;
  __shared__ real sm[GPB][6 * SZ];
  const G g;
  const int grp = GPB == 1 ? 0 : threadIdx.x / GW;
  const int64_t kq = blockIdx.x * (int64_t)GPB + grp;
  if (kq >= a.bt.n_act()) return;  // whole groups
  const int64_t seq = a.bt.act_seq[kq];
  const int64_t c0 = win_first(a.bt, seq), c1 = a.bt.chunk_first[seq + 1];
  real *P = sm[grp], *A = P + SZ, *J = P + 2 * SZ, *S0 = P + 3 * SZ, *S1 = P + 4 * SZ,
       *N = P + 5 * SZ;
  // the next chunk's element is loaded ahead
  real p[EPL], an[EPL], cn[EPL], jn[EPL];
  auto next = [&](int64_t c) {
    if (c < c1) {
      const real* e = a.cov_agg + c * (int64_t)(3 * D * D);
      g.gload(e, an);
      g.gload(e + D * D, cn);
      g.gload(e + 2 * D * D, jn);
    }
  };
  next(c0);
#pragma unroll
  for (int m = 0; m < EPL; ++m) p[m] = real(0);
  for (int64_t c = c0; c < c1; ++c) {
    g.gstore(a.cov_in + c * (int64_t)(D * D), p);
    g.store(P, p);
    g.store(A, an);
    g.store(J, jn);
    real ca[EPL], v[EPL];
#pragma unroll
    for (int m = 0; m < EPL; ++m) ca[m] = cn[m];
    g.sync();
    next(c + 1);
    // N = (I + P J)^{-1}; P <- A N P A^T + C
    g.template mul<false, false>(P, J, v);
#pragma unroll
    for (int m = 0; m < EPL; ++m) v[m] += g.eye(m);
    g.store(S0, v);
    g.sync();
    g.template inverse<true>(S0, S1, N);
    g.template mul<false, false>(N, P, v);
    g.store(S0, v);
    g.sync();
    g.template mul<false, false>(A, S0, v);
    g.store(S1, v);
    g.sync();
    g.template mul<false, true>(S1, A, p);
#pragma unroll
    for (int m = 0; m < EPL; ++m) p[m] += ca[m];
    g.sync();  // every read of this chunk's matrices done
  }
}

template <class real, int D>
static void elk_dense_launch(const ElkDenseArgs<real>& a, cudaStream_t st) {
  constexpr int GPB = 32 / elk_lanes<D>();
  if (a.cov_agg) {
    constexpr int CW = elk_carry_lanes<D>();
    const unsigned gc = grid_for(a.bt.act_chunks(), GPB);
    k_elk_cov_chunk<real, D><<<gc, 32, 0, st>>>(a);
    k_elk_cov_carry<real, D>
        <<<grid_for(a.bt.n_act(), CW < 32 ? 32 / CW : 1), CW < 32 ? 32 : CW, 0, st>>>(a);
    k_elk_dense<real, D, true><<<gc, 32, 0, st>>>(a);
    note_launch(3);
  } else {
    k_elk_dense<real, D, false><<<grid_for(a.bt.n_act(), GPB), 32, 0, st>>>(a);
    note_launch();
  }
}

template <class real>
cudaError_t launch_elk_dense(const ElkDenseArgs<real>& a, cudaStream_t st) {
  if (a.bt.n_act() == 0) return cudaSuccess;
  switch (a.d) {
    case 1: elk_dense_launch<real, 1>(a, st); break;
    case 2: elk_dense_launch<real, 2>(a, st); break;
    case 4: elk_dense_launch<real, 4>(a, st); break;
    case 8: elk_dense_launch<real, 8>(a, st); break;
    case 16: elk_dense_launch<real, 16>(a, st); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template cudaError_t launch_elk_dense<float>(const ElkDenseArgs<float>&, cudaStream_t);
template cudaError_t launch_elk_dense<double>(const ElkDenseArgs<double>&, cudaStream_t);

}  // namespace deer
