// Convergence check and the chunked parallel scans (dense and diagonal families).
//
// Scan structure (three phases, no host involvement): every chunk of L consecutive rows
// of one sequence is reduced to its aggregate under the affine composition of Eq.
// bin_op_affine, (A_j, b_j) o (A_i, b_i) = (A_j A_i, b_j + A_j b_i); a per-sequence pass
// composes the chunk aggregates in order (the operation does not commute) to obtain the
// state entering every chunk; a final pass re-runs each chunk from its carry.
#include <cfloat>

#include "kernels.h"
#include "tc.cuh"

namespace deer {

// ----------------------------------------------------------------------------
// Convergence / merit (one block): per sequence max |r| / max(1, |s|) vs tol, merit
// 1/2 |r|^2; then the sequences still iterating are compacted (in order) into the active
// lists that size and index every later launch. Thread t owns a contiguous range of
// sequences so that a block-wide exclusive scan gives each its output offsets.
// ----------------------------------------------------------------------------
__device__ __forceinline__ void block_excl_scan3(long long& a, long long& b, long long& c,
                                                 long long& ta, long long& tb, long long& tc) {
  __shared__ long long sa[32], sb[32], sc[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned full = 0xffffffffu;
  long long ia = a, ib = b, ic = c;  // inclusive warp scan
  for (int o = 1; o < 32; o <<= 1) {
    long long xa = __shfl_up_sync(full, ia, o), xb = __shfl_up_sync(full, ib, o),
              xc = __shfl_up_sync(full, ic, o);
    if (lane >= o) { ia += xa; ib += xb; ic += xc; }
  }
  if (lane == 31) { sa[warp] = ia; sb[warp] = ib; sc[warp] = ic; }
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    long long va = lane < nw ? sa[lane] : 0, vb = lane < nw ? sb[lane] : 0,
              vc = lane < nw ? sc[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      long long xa = __shfl_up_sync(full, va, o), xb = __shfl_up_sync(full, vb, o),
                xc = __shfl_up_sync(full, vc, o);
      if (lane >= o) { va += xa; vb += xb; vc += xc; }
    }
    if (lane < nw) { sa[lane] = va; sb[lane] = vb; sc[lane] = vc; }
  }
  __syncthreads();
  const int nw = blockDim.x >> 5;
  const long long wa = warp > 0 ? sa[warp - 1] : 0, wb = warp > 0 ? sb[warp - 1] : 0,
                  wc = warp > 0 ? sc[warp - 1] : 0;
  ta = sa[nw - 1]; tb = sb[nw - 1]; tc = sc[nw - 1];
  a = wa + ia - a; b = wb + ib - b; c = wc + ic - c;
}

// whether the Newton loop goes on after the check of iteration `it` (the host loop's
// stopping rules, evaluated on the device)
__device__ __forceinline__ bool loop_goes_on(const Flags* f, int it, int max_iters,
                                             int reset) {
  if (f->bad_input || f->timeout) return false;
  if (f->n_nonfinite > 0 && !reset) return false;
  if (f->n_active == 0) return false;
  return it < max_iters;
}

__global__ void k_loop_gate(Flags* f, int max_iters, int reset,
                            cudaGraphConditionalHandle cond) {
  if (threadIdx.x == 0 && blockIdx.x == 0)
    cudaGraphSetConditional(cond, loop_goes_on(f, f->iter - 1, max_iters, reset) ? 1u : 0u);
}

cudaError_t launch_loop_gate(Flags* flags, int max_iters, int reset,
                             cudaGraphConditionalHandle cond, cudaStream_t st) {
  k_loop_gate<<<1, 32, 0, st>>>(flags, max_iters, reset, cond);
  note_launch();
  return cudaGetLastError();
}

__global__ void __launch_bounds__(1024) k_check(CheckArgs a) {
  // iteration index: the host's, or the device loop's counter (read by every thread
  // before thread 0 advances it at the end)
  const int it_now = a.device_it ? a.flags->iter : a.it;
  a.it = it_now;
  const int64_t per = (a.B + blockDim.x - 1) / blockDim.x;
  const int64_t lo = threadIdx.x * per;
  const int64_t hi = lo + per < a.B ? lo + per : a.B;
  int nonfinite = 0;
  long long n_act = 0, rows = 0, chunks = 0;
  double h_merit = 0.0, h_max = 0.0;  // history: over the sequences tested here
  for (int64_t seq = lo; seq < hi; ++seq) {
    SeqInfo inf = a.info[seq];
    if (!inf.done && !a.compact_only) {
      SeqAcc acc = a.acc[seq];
      a.acc[seq] = SeqAcc{0ull, 0.0, 0ull};
      const double mr = __longlong_as_double((long long)acc.max_bits);
      inf.max_resid = mr;
      inf.merit = 0.5 * acc.sumsq;
      h_merit += inf.merit;
      h_max = nanmax(h_max, mr);
      if (!(mr <= DBL_MAX)) ++nonfinite;  // NaN or Inf
      inf.passes = mr <= a.tol ? inf.passes + 1 : 0;
      if (inf.passes >= a.confirm) {
        inf.done = 1;
        inf.iters = a.it;
      } else {
        inf.iters = a.it < a.max_iters ? a.it + 1 : a.it;
        if (a.window) {
          // rows that passed in one more consecutive iterate than the convergence test asks
          // for (so every frozen row has had one further Newton step after it first
          // qualified) are frozen, in whole chunks
          const int64_t len = a.offsets[seq + 1] - a.offsets[seq];
          const int64_t nch = a.chunk_first[seq + 1] - a.chunk_first[seq];
          const int64_t fb = acc.badkey ? (int64_t)(~acc.badkey) : len;
          int64_t fbw = fb < inf.fb_prev ? fb : (int64_t)inf.fb_prev;
          if (a.confirm >= 2 && inf.fb_prev2 < fbw) fbw = inf.fb_prev2;
          inf.fb_prev2 = inf.fb_prev;
          inf.fb_prev = (int32_t)fb;
          int64_t j0 = fbw >> a.log2L;
          if (j0 < inf.j0) j0 = inf.j0;
          if (j0 > nch - 1) j0 = nch - 1 > 0 ? nch - 1 : 0;
          inf.j0 = (int32_t)j0;
          a.win_chunk[seq] = a.chunk_first[seq] + j0;
        }
      }
      a.info[seq] = inf;
    }
    if (!inf.done) {
      ++n_act;
      rows += a.offsets[seq + 1] - a.offsets[seq] - ((int64_t)inf.j0 << a.log2L);
      chunks += a.chunk_first[seq + 1] - a.chunk_first[seq] - inf.j0;
    }
  }
  long long tn, tr, tc;
  long long pn = n_act, pr = rows, pc = chunks;
  block_excl_scan3(pn, pr, pc, tn, tr, tc);
  for (int64_t seq = lo; seq < hi; ++seq) {
    const SeqInfo inf = a.info[seq];
    if (inf.done) continue;
    a.act_seq[pn] = seq;
    a.act_row_off[pn] = pr;
    a.act_chunk_off[pn] = pc;
    ++pn;
    pr += a.offsets[seq + 1] - a.offsets[seq] - ((int64_t)inf.j0 << a.log2L);
    pc += a.chunk_first[seq + 1] - a.chunk_first[seq] - inf.j0;
  }
  __shared__ int s_nonfinite;
  if (threadIdx.x == 0) s_nonfinite = 0;
  __syncthreads();
  if (nonfinite) atomicAdd(&s_nonfinite, nonfinite);
  __syncthreads();
  if (threadIdx.x == 0) {
    a.act_row_off[tn] = tr;
    a.act_chunk_off[tn] = tc;
    a.flags->n_active = (int32_t)tn;
    a.flags->n_nonfinite = s_nonfinite;
    a.flags->active_rows = tr;
    a.flags->active_chunks = tc;
  }
  if (a.device_it) {
    __syncthreads();  // every thread has read the counter
    if (threadIdx.x == 0) {
      a.flags->iter = it_now + 1;
      if (a.set_cond)
        cudaGraphSetConditional(
            a.cond, loop_goes_on(a.flags, it_now, a.max_iters, a.reset) ? 1u : 0u);
    }
  }
  if (a.history && !a.compact_only && a.it < a.history_len) {
    // block reduction of the tested sequences' merit sum and largest scaled residual
    __shared__ double s_sum[32], s_max[32];
    const unsigned full = 0xffffffffu;
    for (int o = 16; o > 0; o >>= 1) {
      h_merit += __shfl_xor_sync(full, h_merit, o);
      h_max = nanmax(h_max, __shfl_xor_sync(full, h_max, o));
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { s_sum[warp] = h_merit; s_max[warp] = h_max; }
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0.0, mx = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        sum += s_sum[w];
        mx = nanmax(mx, s_max[w]);
      }
      double* h = a.history + 4 * (int64_t)a.it;
      h[0] = (double)a.it;
      h[1] = sum;
      h[2] = mx;
      h[3] = (double)tn;
    }
  }
}

__global__ void k_uniform_tables(int64_t* off, int64_t* cf, int64_t B, int64_t T,
                                 int64_t cps) {
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b <= B;
       b += (int64_t)gridDim.x * blockDim.x) {
    off[b] = b * T;
    cf[b] = b * cps;
  }
}

cudaError_t launch_uniform_tables(int64_t* offsets, int64_t* chunk_first, int64_t B,
                                  int64_t T, int64_t chunks_per_seq, cudaStream_t st) {
  const int64_t n = B + 1;
  const unsigned g = (unsigned)((n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024);
  k_uniform_tables<<<g, 256, 0, st>>>(offsets, chunk_first, B, T, chunks_per_seq);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_check(const CheckArgs& a, cudaStream_t st) {
  k_check<<<1, 1024, 0, st>>>(a);
  note_launch();
  return cudaGetLastError();
}

template <class real>
__device__ __forceinline__ real reset_val(real v, real thr, int reset) {
  // (bit patterns: no float64 comparison, NaN orders above every threshold)
  return reset && mag_bits(v) > mag_bits(thr) ? real(0) : v;
}

// 16 bytes (four floats or two doubles) from a 16-byte aligned address. Plain (coherent)
// load: used for data the same launch never writes, and for data written by earlier
// launches.
template <class real>
__device__ __forceinline__ void ld16(const real* p, real* v) {
  if constexpr (sizeof(real) == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
    const double2 q = *reinterpret_cast<const double2*>(p);
    v[0] = q.x; v[1] = q.y;
  }
}

// ----------------------------------------------------------------------------
// Diagonal family (one thread per (chunk, coordinate))
// ----------------------------------------------------------------------------
template <class real>
__device__ __forceinline__ void diag_elem(const DiagScanArgs<real>& a, int64_t row, int j,
                                          real& at, real& bt) {
  at = a.amode == 0 ? __ldg(a.a + row * a.d + j) : a.aconst;
  bt = __ldg(a.b + row * a.d + j);
}

template <class real>
__global__ void __launch_bounds__(128) k_diag_chunk(DiagScanArgs<real> a) {
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (id >= a.bt.act_chunks() * a.d) return;
  const int64_t ac = id / a.d;
  const int j = (int)(id - ac * a.d);
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, ac, seq, c, r0, n);
  real A = real(1), Bv = real(0);
  for (int t = 0; t < n; ++t) {
    real at, bt;
    diag_elem(a, r0 + t, j, at, bt);
    Bv = at * Bv + bt;
    A = at * A;
  }
  a.aggA[c * a.d + j] = A;
  a.aggB[c * a.d + j] = Bv;
}

constexpr int kCarry = 16;

template <class real>
__global__ void __launch_bounds__(128) k_diag_carry(DiagScanArgs<real> a) {
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (id >= a.bt.n_act() * a.d) return;
  const int64_t k = id / a.d;
  const int j = (int)(id - k * a.d);
  const int64_t seq = a.bt.act_seq[k];
  const int64_t cf = a.bt.chunk_first[seq], c0 = win_first(a.bt, seq);
  const int64_t c1 = a.bt.chunk_first[seq + 1];
  real x = c0 == cf ? a.s0[seq * a.d + j]
                   : a.s[(a.bt.offsets[seq] + ((c0 - cf) << a.bt.log2L) - 1) * a.d + j];
  // the aggregates of kCarry chunks are loaded at a time (they do not depend on x): one
  // memory latency per batch instead of one per chunk
  for (int64_t cb = c0; cb < c1; cb += kCarry) {
    real av[kCarry], bv[kCarry];
#pragma unroll
    for (int k = 0; k < kCarry; ++k) {
      const int64_t c = cb + k < c1 ? cb + k : c1 - 1;
      av[k] = a.aggA[c * a.d + j];
      bv[k] = a.aggB[c * a.d + j];
    }
#pragma unroll
    for (int k = 0; k < kCarry; ++k) {
      if (cb + k >= c1) break;
      a.cin[(cb + k) * a.d + j] = x;
      x = av[k] * x + bv[k];
    }
  }
}

template <class real>
__global__ void __launch_bounds__(128) k_diag_apply(DiagScanArgs<real> a) {
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (id >= a.bt.act_chunks() * a.d) return;
  const int64_t ac = id / a.d;
  const int j = (int)(id - ac * a.d);
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, ac, seq, c, r0, n);
  real x = a.cin[c * a.d + j];
  for (int t = 0; t < n; ++t) {
    real at, bt;
    diag_elem(a, r0 + t, j, at, bt);
    x = at * x + bt;
    a.s[(r0 + t) * a.d + j] = reset_val(x, a.reset_thr, a.reset);
  }
}

// --- Kalman-filter damping (quasi-ELK), per coordinate -----------------------
// The filtered variance obeys P_t = sigma2 (a_t^2 P_{t-1} + 1) / (a_t^2 P_{t-1} + 1 + sigma2),
// a linear-fractional (Moebius) map of P_{t-1} with matrix
// [[sigma2 a^2, sigma2], [a^2, 1 + sigma2]]; maps compose by matrix product, scaled by the
// power of two of their largest entry to stay finite (a Moebius map is invariant under
// scaling, and this one rounds nothing and needs no division).
// What bounds these passes is latency: a few flops per element behind a load, a chain of
// L rows per thread. They load kElkRows rows at a time ahead of the chain. GRU, d = 64,
// 16 x 16384 rows, float32, per pass: variance chunks 55 -> 39, variance carry 70 -> 16, mean
// chunks 95 -> 41, mean carry 68 -> 13, apply 114 -> 48 us.
constexpr int kElkRows = 8;

// 2^-e for m = f 2^e, f in [1, 2) (from the exponent bits; non-finite and zero m give a
// finite factor)
__device__ __forceinline__ float pow2_inverse(float m) {
  const unsigned e = (__float_as_uint(m) >> 23) & 0xffu;
  return __uint_as_float((e >= 254u ? 1u : e == 0u ? 253u : 254u - e) << 23);
}
__device__ __forceinline__ double pow2_inverse(double m) {
  const unsigned e = ((unsigned)__double2hiint(m) >> 20) & 0x7ffu;
  return __hiloint2double((int)((e >= 2046u ? 1u : e == 0u ? 2045u : 2046u - e) << 20), 0);
}

template <class real>
__device__ __forceinline__ void mob_elem(real at, real s2, real& m00, real& m01, real& m10,
                                         real& m11) {
  const real a2 = at * at;
  m00 = s2 * a2; m01 = s2; m10 = a2; m11 = real(1) + s2;
}

template <class real>
__global__ void __launch_bounds__(128) k_elk_chunk(DiagScanArgs<real> a) {
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (id >= a.bt.act_chunks() * a.d) return;
  const int64_t ac = id / a.d;
  const int j = (int)(id - ac * a.d);
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, ac, seq, c, r0, n);
  real p00 = 1, p01 = 0, p10 = 0, p11 = 1;
  for (int tb = 0; tb < n; tb += kElkRows) {
    real av[kElkRows];
#pragma unroll
    for (int k = 0; k < kElkRows; ++k) {
      const int t = tb + k < n ? tb + k : n - 1;
      av[k] = a.amode == 0 ? __ldg(a.a + (r0 + t) * a.d + j) : a.aconst;
    }
#pragma unroll
    for (int k = 0; k < kElkRows; ++k) {
      if (tb + k >= n) break;
      real m00, m01, m10, m11;
      mob_elem(av[k], a.sigma2, m00, m01, m10, m11);
      const real q00 = m00 * p00 + m01 * p10, q01 = m00 * p01 + m01 * p11;
      const real q10 = m10 * p00 + m11 * p10, q11 = m10 * p01 + m11 * p11;
      const real inv = pow2_inverse(fmax(fmax(fabs(q00), fabs(q01)), fmax(fabs(q10), fabs(q11))));
      p00 = q00 * inv; p01 = q01 * inv; p10 = q10 * inv; p11 = q11 * inv;
    }
  }
  real* o = a.mob + (c * a.d + j) * 4;
  o[0] = p00; o[1] = p01; o[2] = p10; o[3] = p11;
}

template <class real>
__global__ void __launch_bounds__(128) k_elk_carry(DiagScanArgs<real> a) {
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (id >= a.bt.n_act() * a.d) return;
  const int64_t k = id / a.d;
  const int j = (int)(id - k * a.d);
  const int64_t seq = a.bt.act_seq[k];
  real P = real(0);  // the state before the first solved row (s_0 or frozen) is known exactly
  const int64_t c0 = win_first(a.bt, seq), c1 = a.bt.chunk_first[seq + 1];
  for (int64_t cb = c0; cb < c1; cb += kCarry) {
    real m[kCarry][4];
#pragma unroll
    for (int k = 0; k < kCarry; ++k) {
      const int64_t c = cb + k < c1 ? cb + k : c1 - 1;
      ld16<real>(a.mob + (c * a.d + j) * 4, m[k]);
      if constexpr (sizeof(real) == 8) ld16<real>(a.mob + (c * a.d + j) * 4 + 2, m[k] + 2);
    }
#pragma unroll
    for (int k = 0; k < kCarry; ++k) {
      if (cb + k >= c1) break;
      a.pin[(cb + k) * a.d + j] = P;
      P = (m[k][0] * P + m[k][1]) / (m[k][2] * P + m[k][3]);
    }
  }
}

// The filtered mean's transition of a row, with the attenuation recomputed from the
// variance carried along the chunk: P^-_t = a_t^2 P_{t-1} + 1, Gamma_t = sigma2 / (P^-_t +
// sigma2), P_t = Gamma_t P^-_t; mu_t = Gamma_t a_t mu_{t-1} + Gamma_t b_t + (1 - Gamma_t) y_t.
template <class real>
__device__ __forceinline__ void elk_row(real sigma2, real a0, real b0, real y, real& P, real& at,
                                        real& bt) {
  const real Pm = a0 * a0 * P + real(1);
  const real g = sigma2 / (Pm + sigma2);
  P = g * Pm;
  at = g * a0;
  bt = g * b0 + (real(1) - g) * y;
}

// a_t, b_t and y_t = s_t of kElkRows rows from row tb of a chunk (the last row again past its end)
template <class real>
struct ElkRows {
  real a[kElkRows], b[kElkRows], y[kElkRows];
  __device__ __forceinline__ void load(const DiagScanArgs<real>& g, int64_t r0, int tb, int n, int j) {
#pragma unroll
    for (int k = 0; k < kElkRows; ++k) {
      const int64_t e = (r0 + (tb + k < n ? tb + k : n - 1)) * g.d + j;
      a[k] = g.amode == 0 ? __ldg(g.a + e) : g.aconst;
      b[k] = __ldg(g.b + e);
      y[k] = g.s[e];
    }
  }
};

// Mean aggregates of the chunks (quasi-ELK): the variance entering the chunk (pin) is known
// from the Moebius carry, so the attenuations are formed on the fly instead of being
// stored and read back.
template <class real>
__global__ void __launch_bounds__(128) k_elk_mean_chunk(DiagScanArgs<real> a) {
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (id >= a.bt.act_chunks() * a.d) return;
  const int64_t ac = id / a.d;
  const int j = (int)(id - ac * a.d);
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, ac, seq, c, r0, n);
  real P = a.pin[c * a.d + j];
  real A = real(1), Bv = real(0);
  for (int tb = 0; tb < n; tb += kElkRows) {
    ElkRows<real> r;
    r.load(a, r0, tb, n, j);
#pragma unroll
    for (int k = 0; k < kElkRows; ++k) {
      if (tb + k >= n) break;
      real at, bt;
      elk_row(a.sigma2, r.a[k], r.b[k], r.y[k], P, at, bt);
      Bv = at * Bv + bt;
      A = at * A;
    }
  }
  a.aggA[c * a.d + j] = A;
  a.aggB[c * a.d + j] = Bv;
}

template <class real>
__global__ void __launch_bounds__(128) k_elk_apply(DiagScanArgs<real> a) {
  const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (id >= a.bt.act_chunks() * a.d) return;
  const int64_t ac = id / a.d;
  const int j = (int)(id - ac * a.d);
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, ac, seq, c, r0, n);
  real P = a.pin[c * a.d + j];
  real x = a.cin[c * a.d + j];
  for (int tb = 0; tb < n; tb += kElkRows) {
    ElkRows<real> r;  // y_t = s_t is read before it is overwritten
    r.load(a, r0, tb, n, j);
#pragma unroll
    for (int k = 0; k < kElkRows; ++k) {
      if (tb + k >= n) break;
      real at, bt;
      elk_row(a.sigma2, r.a[k], r.b[k], r.y[k], P, at, bt);
      x = at * x + bt;
      a.s[(r0 + tb + k) * a.d + j] = reset_val(x, a.reset_thr, a.reset);
    }
  }
}

template <class real>
cudaError_t launch_diag_scan(const DiagScanArgs<real>& a, cudaStream_t st) {
  if (a.bt.act_rows() == 0) return cudaSuccess;
  const unsigned gc = grid_for(a.bt.act_chunks() * a.d, 128);
  const unsigned gs = grid_for(a.bt.n_act() * a.d, 128);
  if (a.elk) {
    // variance: Moebius chunk aggregates and their carry; mean: aggregates, carry and
    // apply with the attenuations recomputed from the carried variance
    k_elk_chunk<real><<<gc, 128, 0, st>>>(a);
    k_elk_carry<real><<<gs, 128, 0, st>>>(a);
    k_elk_mean_chunk<real><<<gc, 128, 0, st>>>(a);
    k_diag_carry<real><<<gs, 128, 0, st>>>(a);
    k_elk_apply<real><<<gc, 128, 0, st>>>(a);
    note_launch(5);
    return cudaGetLastError();
  }
  k_diag_chunk<real><<<gc, 128, 0, st>>>(a);
  k_diag_carry<real><<<gs, 128, 0, st>>>(a);
  k_diag_apply<real><<<gc, 128, 0, st>>>(a);
  note_launch(3);
  return cudaGetLastError();
}

template cudaError_t launch_diag_scan<float>(const DiagScanArgs<float>&, cudaStream_t);
template cudaError_t launch_diag_scan<double>(const DiagScanArgs<double>&, cudaStream_t);

}  // namespace deer

namespace deer {

// ----------------------------------------------------------------------------
// Dense scan: D lanes per chunk (per sequence in the carry pass; two or four warps per
// chunk in the d = 32 chunk pass). Lane j owns column j of the chunk product P and
// entry j of the vectors; the Jacobian rows and chunk aggregates are staged in a
// shared-memory ring ahead of use, vector entries travel by shuffles.
// For d <= 8 what bounds these passes is the dependent chain per row (and, in float64, the
// issue rate of the FP64 pipe): one thread per chunk loading its own rows was tried first
// and spent a row's time on uncoalesced loads and D^3 serial products. Two-well Langevin,
// float64, 4 sequences of 10000 rows, d = 4, per pass: chunk 236 -> 61 us, carry 179 -> 40,
// apply 200 -> 59; float32 d = 8, 512 x 16384 rows, four Newton steps: 30.8 -> 12.8 ms. d = 1
// keeps a thread per chunk (k_scalar_*: 8 % faster there, nothing to share in a group).
// ----------------------------------------------------------------------------
// lanes of a group: D rounded up to a power of two (d = 5 leaves three lanes idle; they
// take part in the group's shuffles and barriers with lane 0's data and store nothing)
template <int D>
constexpr int group_lanes() { return D <= 2 ? D : D <= 4 ? 4 : D <= 8 ? 8 : D <= 16 ? 16 : 32; }

template <int D>
__device__ __forceinline__ unsigned group_mask() {
  constexpr int W = group_lanes<D>();
  if constexpr (W == 32) return 0xffffffffu;
  return ((1u << W) - 1u) << (threadIdx.x & 31 & ~(W - 1));
}

// ----------------------------------------------------------------------------
// Asynchronous row staging for the dense scans. The lanes of a group copy a d x d block in
// 16-byte pieces, and one entry of a vector each, from global
// memory into a slot of a shared-memory ring with cp.async; the ring runs K slots
// ahead of the rows being consumed, so the DRAM latency of a row is hidden behind the
// dependent work on the rows before it. Rows are padded to D + 16 B so that 128-bit
// reads of eight lanes' rows hit distinct banks. Every stage commits one (possibly empty)
// group, and cp.async.wait_group(kRing - 1) before a slot is read guarantees that the
// slot's copies (issued kRing commits earlier) have landed: the wait ends when the copies
// do, with no spin loop of our own.
// ----------------------------------------------------------------------------
template <class real, int D = 32>
constexpr int ring_depth() { return sizeof(real) == 4 || D <= 8 ? 8 : 4; }

template <class real, int D>
struct RowRing {
  static constexpr int K = ring_depth<real, D>();
  // rows of whole 16-byte pieces (d = 1, 5 and float d = 2 go entry by entry)
  static constexpr bool VEC = D * (int)sizeof(real) % 16 == 0;
  static constexpr int RS = VEC ? D + 16 / (int)sizeof(real) : D;
  real m[K][D][RS];  // row `lane` of a d x d block per slot
  real v[K][D];      // one vector entry per lane per slot

  // copy the block at `blk` (16-byte aligned; the group's lanes take consecutive pieces:
  // lane-owned rows cost a separate memory transaction per lane, 2063 against 1335 us for the
  // adjoint's apply pass over 2.1 M rows, d = 32) and vec[lane] into `slot`
  __device__ __forceinline__ void issue(int slot, int lane, const real* blk, const real* vec) {
    if (lane >= D) return;
    if constexpr (VEC) {
      constexpr int VW = 16 / (int)sizeof(real), PR = D / VW;  // pieces per row
#pragma unroll
      for (int q = 0; q < PR; ++q) {
        const int e = q * D + lane;  // consecutive lanes copy consecutive pieces
        cp_async16(&m[slot][e / PR][e % PR * VW], blk + e * VW);
      }
    } else {
#pragma unroll
      for (int q = 0; q < D; ++q) {
        const int e = q * D + lane;
        cp_async_small<sizeof(real)>(&m[slot][e / D][e % D], blk + e);
      }
    }
    cp_async_small<sizeof(real)>(&v[slot][lane], vec + lane);
  }
  __device__ __forceinline__ void row(int slot, int r, real (&out)[D]) const {
    if constexpr (!VEC) {
#pragma unroll
      for (int k = 0; k < D; ++k) out[k] = m[slot][r][k];
      return;
    }
#pragma unroll
    for (int k = 0; VEC && k < D; k += 16 / (int)sizeof(real)) {
      if constexpr (!VEC) {
      } else if constexpr (sizeof(real) == 4) {
        const float4 q = *reinterpret_cast<const float4*>(&m[slot][r][k]);
        out[k] = q.x; out[k + 1] = q.y; out[k + 2] = q.z; out[k + 3] = q.w;
      } else {
        const double2 q = *reinterpret_cast<const double2*>(&m[slot][r][k]);
        out[k] = q.x; out[k + 1] = q.y;
      }
    }
  }
};

// What one group folds: rows r0 .. r0 + n - 1 of (A, b) into aggregate `out`. SEG = false: a
// chunk of rows into the chunk aggregates; SEG = true: a segment of consecutive chunk
// aggregates of one active sequence (blockIdx.y) into the segment aggregates.
struct Span {
  int64_t r0, out;
  int n;
  bool need_P;
};

template <bool SEG, class real>
__device__ __forceinline__ bool get_span(const DenseScanArgs<real>& a, int64_t idx, Span& p) {
  if constexpr (!SEG) {
    if (idx >= a.bt.act_chunks()) return false;
    int64_t seq;
    act_chunk(a.bt, idx, seq, p.out, p.r0, p.n);
    p.need_P = p.out != win_first(a.bt, seq);
  } else {
    if ((int64_t)blockIdx.y >= a.bt.n_act()) return false;
    const int64_t seq = __ldg(a.bt.act_seq + blockIdx.y);
    const int64_t c1 = __ldg(a.bt.chunk_first + seq + 1);
    p.r0 = win_first(a.bt, seq) + (idx << a.log2M);
    if (p.r0 >= c1) return false;
    p.n = (int)(c1 - p.r0 < (1 << a.log2M) ? c1 - p.r0 : (1 << a.log2M));
    p.need_P = idx > 0;
    // sequence b's segments start at chunk_first[b] / M + b: disjoint, since
    // floor(x + y) + 1 >= floor(x) + ceil(y)
    p.out = (__ldg(a.bt.chunk_first + seq) >> a.log2M) + seq + idx;
  }
  return true;
}

template <bool SEG, class real, int D>
__device__ __forceinline__ void span_ptrs(const DenseScanArgs<real>& a, const Span& p,
                                          const real*& A0, const real*& b0, real*& Po,
                                          real*& vo) {
  A0 = (SEG ? a.aggP : a.A) + p.r0 * (int64_t)(D * D);
  b0 = (SEG ? a.aggv : a.b) + p.r0 * D;
  Po = (SEG ? a.segP : a.aggP) + p.out * (int64_t)(D * D);
  vo = (SEG ? a.segv : a.aggv) + p.out * D;
}

// Chunk pass: one group of D lanes per chunk (one warp per block), lane j owns
// column j of the chunk product P and entry j of the vector part. Row t's Jacobian is
// staged in the ring; every lane reads all of its rows (broadcast) for P <- A_t P and
// its own row for v <- A_t v + b_t.
template <class real, int D, bool SEG>
__global__ void __launch_bounds__(32) k_dense_chunk_ring(DenseScanArgs<real> a) {
  constexpr int W = group_lanes<D>(), G = 32 / W;
  using Ring = RowRing<real, D>;
  constexpr int K = Ring::K;
  constexpr int kUnroll = D == 8 || D == 5 ? 1 : K;  // d^3 products per row: keep the code small
  __shared__ __align__(16) Ring ring[G];
  const int grp = threadIdx.x / W, lane = threadIdx.x % W;
  const int li = lane < D ? lane : 0;  // this lane's row / column
  const unsigned gm = group_mask<D>();
  Span p;
  if (!get_span<SEG>(a, blockIdx.x * (int64_t)G + grp, p))
    return;  // whole groups; groups never synchronise with each other
  const real *A0, *b0;
  real *Po, *vo;
  span_ptrs<SEG, real, D>(a, p, A0, b0, Po, vo);
  const int n = p.n;
  const bool need_P = p.need_P;
  Ring& R = ring[grp];
#pragma unroll
  for (int s = 0; s < K; ++s) {
    if (s < n) R.issue(s, lane, A0 + s * (int64_t)(D * D), b0 + s * D);
    cp_async_commit();
  }
  real Pc[D];  // column `lane` of P
  real v = real(0);
#pragma unroll
  for (int i = 0; i < D; ++i) Pc[i] = i == li ? real(1) : real(0);
  for (int t0 = 0; t0 < n; t0 += K) {
#pragma unroll(kUnroll)
    for (int s = 0; s < K; ++s) {
      const int t = t0 + s;
      cp_async_wait<K - 1>();
      __syncwarp(gm);  // the other lanes' rows of this slot have landed
      if (t < n) {
        real own[D];
        R.row(s, li, own);
        real nv = R.v[s][li];
#pragma unroll
        for (int k = 0; k < D; ++k) nv += own[k] * __shfl_sync(gm, v, k, W);
        v = nv;
        if (need_P) {
          real np[D];
#pragma unroll
          for (int i = 0; i < D; ++i) {
            real ar[D];
            R.row(s, i, ar);
            real x = real(0);
#pragma unroll
            for (int k = 0; k < D; ++k) x += ar[k] * Pc[k];
            np[i] = x;
          }
#pragma unroll
          for (int i = 0; i < D; ++i) Pc[i] = np[i];
        }
      }
      __syncwarp(gm);  // every lane is done with the slot before it is refilled
      if (t + K < n) R.issue(s, lane, A0 + (t + K) * (int64_t)(D * D), b0 + (t + K) * D);
      cp_async_commit();
    }
  }
  cp_async_wait<0>();
  if (lane >= D) return;
#pragma unroll
  for (int i = 0; i < D; ++i) Po[i * D + lane] = Pc[i];
  vo[lane] = v;
}

// Chunk pass, float64, few chunks: a warp per chunk with the entries of [P | v] spread over
// its lanes. A warp issues one FP64 instruction per 64 clocks whatever its active lanes, so
// while chunks are too few to give every SM sub-partition (608) a warp of whole groups, one
// entry per lane shortens a row from d^2 + d instructions to d (d = 4, 5) or 3 d (d = 8).
// Langevin, d = 4, 4 x 10000 rows: 62 us a pass in chunks of 64 rows, 14 us so in chunks of
// 32. The sums run in the same order.
template <int D, bool SEG>
__global__ void __launch_bounds__(32) k_dense_chunk_entry(DenseScanArgs<double> a) {
  constexpr int K = 8, E = D * (D + 1), EPL = (E + 31) / 32;
  __shared__ double sA[K][D * D], sB[K][D], sX[2][E];
  const int lane = threadIdx.x;
  Span p;
  if (!get_span<SEG>(a, blockIdx.x, p)) return;
  const double *A0, *b0;
  double *Po, *vo;
  span_ptrs<SEG, double, D>(a, p, A0, b0, Po, vo);
  auto issue = [&](int t) {
    if (t < p.n) {
      const int s = t & (K - 1);
      for (int e = lane; e < D * D; e += 32)
        cp_async_small<8>(&sA[s][e], A0 + t * (int64_t)(D * D) + e);
      if (lane < D) cp_async_small<8>(&sB[s][lane], b0 + t * D + lane);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int t = 0; t < K - 1; ++t) issue(t);
  int row[EPL], col[EPL];
  double x[EPL];
#pragma unroll
  for (int m = 0; m < EPL; ++m) {
    const int e = lane + 32 * m < E ? lane + 32 * m : E - 1;
    row[m] = e / (D + 1);
    col[m] = e % (D + 1);
    x[m] = row[m] == col[m] ? 1.0 : 0.0;
  }
  for (int t = 0; t < p.n; ++t) {
    double* X = sX[t & 1];
#pragma unroll
    for (int m = 0; m < EPL; ++m)
      if (lane + 32 * m < E) X[lane + 32 * m] = x[m];
    cp_async_wait<K - 2>();
    __syncwarp();  // row t and every entry of [P | v] in place; row t - 1's slot is free
    issue(t + K - 1);
    const double* A = sA[t & (K - 1)];
#pragma unroll
    for (int m = 0; m < EPL; ++m) {
      if (!p.need_P && col[m] != D) continue;
      double y = col[m] == D ? sB[t & (K - 1)][row[m]] : 0.0;
#pragma unroll
      for (int k = 0; k < D; ++k) y += A[row[m] * D + k] * X[k * (D + 1) + col[m]];
      x[m] = y;
    }
  }
  cp_async_wait<0>();
#pragma unroll
  for (int m = 0; m < EPL; ++m)
    if (lane + 32 * m < E) {
      if (col[m] == D) vo[row[m]] = x[m];
      else Po[row[m] * D + col[m]] = x[m];
    }
}

// Chunk pass, d = 32: one chunk per block of four warps. The staged rows of A_t are shared
// by the block (its 128 threads copy the 4 KB block together); warp w forms rows
// 8w .. 8w+7 of P <- A_t P for all 32 columns (lane j owns column j), the new rows meet
// in shared memory and every warp reloads its full column. The vector part
// v <- A_t v + b_t is formed redundantly by every warp (lane i, row i). A quarter of the
// dependent work per warp compared with one warp per chunk, and four times the warps:
// the single long sequences that leave few chunks stay busy.
template <class real, bool SEG>
__global__ void __launch_bounds__(128) k_dense_chunk_ring4(DenseScanArgs<real> a) {
  constexpr int D = 32;
  constexpr int W = 4;                       // warps per chunk
  constexpr int RW = D / W;                  // rows of P per warp
  constexpr int K = ring_depth<real>();
  constexpr int RS = D + 16 / (int)sizeof(real);
  constexpr int VW = 16 / (int)sizeof(real);
  constexpr int PIECES = D * D / VW;         // 16-byte pieces of one A_t
  __shared__ __align__(16) real sA[K][D][RS];
  __shared__ __align__(16) real sB[K][D];
  __shared__ real sP[D][D + 1];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  Span p;
  if (!get_span<SEG>(a, blockIdx.x, p)) return;  // uniform over the block
  const real *A0, *b0;
  real *Po, *vo;
  span_ptrs<SEG, real, D>(a, p, A0, b0, Po, vo);
  const int n = p.n;
  const bool need_P = p.need_P;
  auto issue = [&](int slot, int t) {
    if (t < n) {
      const real* src = A0 + t * (int64_t)(D * D);
      for (int q = tid; q < PIECES; q += 128)
        cp_async16(&sA[slot][q / (D / VW)][(q % (D / VW)) * VW], src + q * VW);
      if (tid < D / VW) cp_async16(&sB[slot][tid * VW], b0 + t * D + tid * VW);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int s = 0; s < K; ++s) issue(s, s);
  real Pc[D];  // column `lane` of P (the same in every warp)
  real v = real(0);
#pragma unroll
  for (int i = 0; i < D; ++i) Pc[i] = i == lane ? real(1) : real(0);
  for (int t0 = 0; t0 < n; t0 += K) {
#pragma unroll
    for (int s = 0; s < K; ++s) {
      const int t = t0 + s;
      cp_async_wait<K - 1>();
      __syncthreads();  // slot s complete for the block; last row's column reloads done
      if (t < n) {
        real own[D];
#pragma unroll
        for (int k = 0; k < D; k += VW) ld16<real>(&sA[s][lane][k], own + k);
        real nv = sB[s][lane];
#pragma unroll
        for (int k = 0; k < D; ++k) nv += own[k] * __shfl_sync(0xffffffffu, v, k);
        v = nv;
        if (need_P) {
#pragma unroll
          for (int ii = 0; ii < RW; ++ii) {
            const int i = warp * RW + ii;
            real x = real(0);
#pragma unroll
            for (int k = 0; k < D; k += VW) {
              real ar[VW];
              ld16<real>(&sA[s][i][k], ar);
#pragma unroll
              for (int q = 0; q < VW; ++q) x += ar[q] * Pc[k + q];
            }
            sP[i][lane] = x;
          }
        }
      }
      __syncthreads();  // new rows of P complete; every read of slot s done
      if (need_P && t < n) {
#pragma unroll
        for (int k = 0; k < D; ++k) Pc[k] = sP[k][lane];
      }
      issue(s, t + K);
    }
  }
  cp_async_wait<0>();
  if (warp == 0) {
#pragma unroll
    for (int i = 0; i < D; ++i) Po[i * D + lane] = Pc[i];
    vo[lane] = v;
  }
}

// Chunk pass, d = 32, float32, on the tensor cores. P <- A_t P acts on every column of P
// independently, so the chunk product is carried transposed, P^T <- P^T A_t^T, and split
// by rows of P^T (columns of P) over two warps: warp w owns rows 16w .. 16w + 15 of P^T and
// never exchanges data with the other warp. Each row step is a 16 x 32 x 32 product per
// warp as warp-level tf32 MMAs (m16n8k8, float32 accumulation) with the three-term split
// x = x_hi + x_lo (x_hi = x rounded to tf32): A B ~ A_hi B_hi + A_hi B_lo + A_lo B_hi, a
// relative error of about 2^-21, so the aggregates keep float32 accuracy. The A operand is
// the previous accumulator re-laid by shuffles within each quad of lanes (the accumulator
// holds columns 2t, 2t+1 of a row where the operand wants t, t + 4); the B operand
// A_t^T[k][n] = A_t[n][k] is read from the row-major staged A_t (rows padded to 36 floats:
// the 32 lanes' words fall in distinct banks). The vector part v <- A_t v + b_t is formed
// by lane i (row i) of warp 0. Rows are staged through the same cp.async ring as
// k_dense_chunk_ring4.
__global__ void __launch_bounds__(64) k_dense_chunk_mma32(DenseScanArgs<float> a) {
  constexpr int D = 32;
  constexpr int K = ring_depth<float>();
  constexpr int RS = D + 4;
  constexpr int PIECES = D * D / 4;  // 16-byte pieces of one A_t
  __shared__ __align__(16) float sA[K][D][RS];
  __shared__ __align__(16) float sB[K][D];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tq = lane & 3;
  Span p;
  if (!get_span<false>(a, blockIdx.x, p)) return;  // uniform over the block
  const float *A0, *b0;
  float *Po, *vo;
  span_ptrs<false, float, D>(a, p, A0, b0, Po, vo);
  const int n = p.n;
  const bool need_P = p.need_P;
  auto issue = [&](int slot, int t) {
    if (t < n) {
      const float* src = A0 + t * (int64_t)(D * D);
      for (int q = tid; q < PIECES; q += 64)
        cp_async16(&sA[slot][q / (D / 4)][(q % (D / 4)) * 4], src + q * 4);
      if (tid < D / 4) cp_async16(&sB[slot][tid * 4], b0 + t * D + tid * 4);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int s = 0; s < K; ++s) issue(s, s);
  // accumulator of this warp's 16 rows of P^T: n-tile j holds P^T[m][8j + 2tq (+1)] for
  // m = 16 warp + g (entries 0, 1) and m + 8 (entries 2, 3); P^T starts as I
  float acc[4][4];
  const int m0 = 16 * warp + g;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int n0 = 8 * j + 2 * tq;
    acc[j][0] = m0 == n0 ? 1.f : 0.f;
    acc[j][1] = m0 == n0 + 1 ? 1.f : 0.f;
    acc[j][2] = m0 + 8 == n0 ? 1.f : 0.f;
    acc[j][3] = m0 + 8 == n0 + 1 ? 1.f : 0.f;
  }
  float v = 0.f;
  const int qsrc = (lane & ~3) + (tq >> 1);  // quad lane holding column tq of a tile
  const bool odd = tq & 1;
  for (int t0 = 0; t0 < n; t0 += K) {
#pragma unroll
    for (int s = 0; s < K; ++s) {
      const int t = t0 + s;
      cp_async_wait<K - 1>();
      __syncthreads();  // slot s complete for the block
      if (t < n) {
        if (warp == 0) {
          float nv = sB[s][lane];
#pragma unroll
          for (int k = 0; k < D; k += 4) {
            const float4 q = *reinterpret_cast<const float4*>(&sA[s][lane][k]);
            nv += q.x * __shfl_sync(0xffffffffu, v, k) + q.y * __shfl_sync(0xffffffffu, v, k + 1) +
                  q.z * __shfl_sync(0xffffffffu, v, k + 2) + q.w * __shfl_sync(0xffffffffu, v, k + 3);
          }
          v = nv;
        }
        if (need_P) {
          // A operand (P^T rows, K = columns of P^T) from the accumulator, split
          uint32_t ah[4][4], al[4][4];
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const float x0 = __shfl_sync(0xffffffffu, acc[kk][0], qsrc);
            const float x1 = __shfl_sync(0xffffffffu, acc[kk][1], qsrc);
            const float x2 = __shfl_sync(0xffffffffu, acc[kk][2], qsrc);
            const float x3 = __shfl_sync(0xffffffffu, acc[kk][3], qsrc);
            const float y0 = __shfl_sync(0xffffffffu, acc[kk][0], qsrc + 2);
            const float y1 = __shfl_sync(0xffffffffu, acc[kk][1], qsrc + 2);
            const float y2 = __shfl_sync(0xffffffffu, acc[kk][2], qsrc + 2);
            const float y3 = __shfl_sync(0xffffffffu, acc[kk][3], qsrc + 2);
            const float av[4] = {odd ? x1 : x0, odd ? x3 : x2, odd ? y1 : y0, odd ? y3 : y2};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              ah[kk][e] = tc::tf32_rna(av[e]);
              al[kk][e] = tc::tf32_rna(av[e] - __uint_as_float(ah[kk][e]));
            }
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float dn[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              // B[k][n] = A_t[n][k]: n = 8j + g, k = 8kk + tq (+ 4)
              const float bx0 = sA[s][8 * j + g][8 * kk + tq];
              const float bx1 = sA[s][8 * j + g][8 * kk + tq + 4];
              const uint32_t bh0 = tc::tf32_rna(bx0), bh1 = tc::tf32_rna(bx1);
              const uint32_t bl0 = tc::tf32_rna(bx0 - __uint_as_float(bh0));
              const uint32_t bl1 = tc::tf32_rna(bx1 - __uint_as_float(bh1));
              tc::mma_1688_tf32(dn, al[kk], bh0, bh1);
              tc::mma_1688_tf32(dn, ah[kk], bl0, bl1);
              tc::mma_1688_tf32(dn, ah[kk], bh0, bh1);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[j][e] = dn[e];
          }
        }
      }
      __syncthreads();  // every read of slot s done before it is refilled
      issue(s, t + K);
    }
  }
  cp_async_wait<0>();
  // P[i][j] = P^T[j][i]
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int n0 = 8 * j + 2 * tq;
    Po[n0 * D + m0] = acc[j][0];
    Po[(n0 + 1) * D + m0] = acc[j][1];
    Po[n0 * D + m0 + 8] = acc[j][2];
    Po[(n0 + 1) * D + m0 + 8] = acc[j][3];
  }
  if (warp == 0) vo[lane] = v;
}

// x <- P_c x + v_c over the aggregates c0 .. c1 - 1, streamed through the ring; the x entering
// each goes to `in` (if any). `first`: c0 starts from Delta = 0 and its P is not formed. With
// CHECK, returns the first aggregate that would leave x non-finite, x being the value that
// enters it; otherwise c1.
template <bool CHECK, class real, int D>
__device__ __forceinline__ int64_t carry_walk(RowRing<real, D>& R, const real* P, const real* v,
                                              real* in, int64_t c0, int64_t c1, bool first,
                                              real& x) {
  constexpr int W = group_lanes<D>(), K = RowRing<real, D>::K;
  const int lane = threadIdx.x % W, li = lane < D ? lane : 0;  // this lane's row
  const unsigned gm = group_mask<D>();
#pragma unroll
  for (int s = 0; s < K; ++s) {
    if (c0 + s < c1) R.issue(s, lane, P + (c0 + s) * (int64_t)(D * D), v + (c0 + s) * D);
    cp_async_commit();
  }
  int64_t stop = c1;
  for (int64_t cb = c0; cb < c1 && stop == c1; cb += K) {
#pragma unroll
    for (int s = 0; s < K; ++s) {
      const int64_t c = cb + s;
      cp_async_wait<K - 1>();
      __syncwarp(gm);  // the other lanes' pieces of this slot have landed
      if (c < stop) {
        if (in && lane < D) in[c * D + lane] = x;
        real y = R.v[s][li];
        if (!first || c > c0) {
          real pr[D];
          R.row(s, li, pr);
#pragma unroll
          for (int k = 0; k < D; ++k) y += pr[k] * __shfl_sync(gm, x, k, W);
        }
        if (CHECK && __any_sync(gm, mag_bits(y) >= mag_bits(real(INFINITY)))) stop = c;
        else x = y;
      }
      __syncwarp(gm);  // every lane is done with the slot before it is refilled
      if (c + K < stop)
        R.issue(s, lane, P + (c + K) * (int64_t)(D * D), v + (c + K) * D);
      cp_async_commit();
    }
  }
  cp_async_wait<0>();
  __syncwarp(gm);  // the ring may be refilled
  return stop;
}

// Carry pass: x_c = P_c x_{c-1} + v_c along each active sequence's chunks. MODE 0: one group
// per sequence, over its
// chunks. Few sequences of many chunks make that the longest chain of the iteration (3125
// chunks of the mean-field RNN, d = 32, T = 100000: 580 us); the chunks are then folded into
// segments of M (the chunk pass again, over the aggregates), MODE 1 walks a sequence's
// segments, MODE 2 the chunks of each segment from the value entering it: 39 + 20 + 10 us
// there. The folds are float32 multiply-adds, as the walk over the chunks is, also where the
// chunk pass uses the tensor cores. (Mixed-precision ragged batch, d = 16, up to 3125 chunks a sequence: 134 -> 27 ms of
// scans per solve, against a carry that loaded each aggregate when it needed it.)
// A product over a segment (up to 64 chunks) can overflow where those over its chunks do not,
// and inf times a Delta of zero would then spread NaN over rows that are solved already: MODE
// 1 walks such a segment's chunks one by one.
template <class real, int D, int MODE>
__global__ void __launch_bounds__(32) k_dense_carry_ring(DenseScanArgs<real> a) {
  constexpr int W = group_lanes<D>(), G = 32 / W;
  __shared__ __align__(16) RowRing<real, D> ring[G];
  const int grp = threadIdx.x / W, lane = threadIdx.x % W;
  const int64_t kq = blockIdx.x * (int64_t)G + grp;
  RowRing<real, D>& R = ring[grp];
  real x = real(0);
  if constexpr (MODE == 2) {
    Span p;
    if (!get_span<true>(a, kq, p)) return;
    x = a.segin[p.out * D + (lane < D ? lane : 0)];
    carry_walk<false, real, D>(R, a.aggP, a.aggv, a.cin, p.r0, p.r0 + p.n, !p.need_P, x);
  } else {
    if (kq >= a.bt.n_act()) return;
    const int64_t seq = a.bt.act_seq[kq];
    const int64_t c0 = win_first(a.bt, seq), c1 = a.bt.chunk_first[seq + 1];
    if constexpr (MODE == 0) {
      carry_walk<false, real, D>(R, a.aggP, a.aggv, a.cin, c0, c1, true, x);
    } else {
      const int64_t M = (int64_t)1 << a.log2M;
      const int64_t s0 = (a.bt.chunk_first[seq] >> a.log2M) + seq;
      const int64_t s1 = s0 + ((c1 - c0 + M - 1) >> a.log2M);
      carry_walk<false, real, D>(R, a.segP, a.segv, a.segin, s0, s1, true, x);
      const unsigned gm = group_mask<D>();
      auto nonfinite = [&](real y) {
        return __any_sync(gm, mag_bits(y) >= mag_bits(real(INFINITY))) != 0;
      };
      // a non-finite entry makes every value after it non-finite: only the end is looked at
      if (!nonfinite(x)) return;
      // the first segment that leaves x non-finite, by bisection over the values stored
      const int li = lane < D ? lane : 0;
      int64_t k = s0, end = s1;
      while (end - k > 1) {
        const int64_t mid = k + (end - k) / 2;
        if (nonfinite(a.segin[mid * D + li])) end = mid;
        else k = mid;
      }
      x = a.segin[k * D + li];
      for (;;) {
        const int64_t q0 = c0 + (k - s0) * M;
        carry_walk<false, real, D>(R, a.aggP, a.aggv, nullptr, q0, q0 + M < c1 ? q0 + M : c1,
                                   k == s0, x);
        // (non-finite chunk by chunk too: the values stored stand)
        if (++k >= s1 || nonfinite(x)) return;
        k = carry_walk<true, real, D>(R, a.segP, a.segv, a.segin, k, s1, false, x);
        if (k == s1) return;
      }
    }
  }
}

// Apply pass: Delta_t = A_t Delta_{t-1} + b_t from the chunk's carry, s_t += Delta_t; lane
// i reads its own row of each staged A_t.
template <class real, int D>
__global__ void __launch_bounds__(32) k_dense_apply_ring(DenseScanArgs<real> a) {
  constexpr int W = group_lanes<D>(), G = 32 / W;
  using Ring = RowRing<real, D>;
  constexpr int K = Ring::K;
  __shared__ __align__(16) Ring ring[G];
  __shared__ real st[G][K][2][W];  // the rows' states (and compensation), staged with them
  const int grp = threadIdx.x / W, lane = threadIdx.x % W;
  const int li = lane < D ? lane : 0;  // this lane's row
  const unsigned gm = group_mask<D>();
  const int64_t ac = blockIdx.x * (int64_t)G + grp;
  if (ac >= a.bt.act_chunks()) return;
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, ac, seq, c, r0, n);
  const real* A0 = a.A + r0 * (int64_t)(D * D);
  const real* b0 = a.b + r0 * D;
  Ring& R = ring[grp];
  real* s0 = a.s + r0 * D + li;
  real* l0 = a.slo ? a.slo + r0 * D + li : nullptr;
  auto issue = [&](int s, int t) {
    if (t < n) {
      R.issue(s, lane, A0 + t * (int64_t)(D * D), b0 + t * D);
      cp_async_small<sizeof(real)>(&st[grp][s][0][lane], s0 + t * D);
      if (l0) cp_async_small<sizeof(real)>(&st[grp][s][1][lane], l0 + t * D);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int s = 0; s < K; ++s) issue(s, s);
  real x = a.cin[c * D + li];
  for (int t0 = 0; t0 < n; t0 += K) {
#pragma unroll
    for (int s = 0; s < K; ++s) {
      const int t = t0 + s;
      cp_async_wait<K - 1>();
      __syncwarp(gm);
      if (t < n) {
        real ar[D];
        R.row(s, li, ar);
        real y = R.v[s][li];
#pragma unroll
        for (int k = 0; k < D; ++k) y += ar[k] * __shfl_sync(gm, x, k, W);
        x = y;
        const real so = st[grp][s][0][lane];
        if (lane >= D) {
          // idle lane (d = 5)
        } else if (l0) {
          // compensated state: (s, slo) += Delta with error-free transformations
          real hi = so, lo = st[grp][s][1][lane];
          cs_add(hi, lo, y);
          if (a.reset && !(hi <= a.reset_thr && hi >= -a.reset_thr)) {
            hi = real(0);
            lo = real(0);
          }
          s0[t * D] = hi;
          l0[t * D] = lo;
        } else {
          s0[t * D] = reset_val(so + y, a.reset_thr, a.reset);
        }
      }
      __syncwarp(gm);
      issue(s, t + K);
    }
  }
  cp_async_wait<0>();
}

// d = 1: one thread per chunk (per sequence in the carry pass).
template <class real>
__global__ void __launch_bounds__(128) k_scalar_chunk(DenseScanArgs<real> a) {
  const int64_t ac = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (ac >= a.bt.act_chunks()) return;
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, ac, seq, c, r0, n);
  real P = real(1), v = real(0);
  for (int t = 0; t < n; ++t) {
    const real at = __ldg(a.A + r0 + t);
    v = at * v + __ldg(a.b + r0 + t);
    P = at * P;
  }
  a.aggP[c] = P;
  a.aggv[c] = v;
}

template <class real>
__global__ void __launch_bounds__(128) k_scalar_carry(DenseScanArgs<real> a) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= a.bt.n_act()) return;
  const int64_t seq = a.bt.act_seq[k];
  const int64_t c0 = win_first(a.bt, seq), c1 = a.bt.chunk_first[seq + 1];
  real x = real(0);
#pragma unroll 4
  for (int64_t c = c0; c < c1; ++c) {
    a.cin[c] = x;
    x = c > c0 ? a.aggP[c] * x + a.aggv[c] : a.aggv[c];
  }
}

template <class real>
__global__ void __launch_bounds__(128) k_scalar_apply(DenseScanArgs<real> a) {
  const int64_t ac = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (ac >= a.bt.act_chunks()) return;
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, ac, seq, c, r0, n);
  real x = a.cin[c];
  for (int t = 0; t < n; ++t) {
    x = __ldg(a.A + r0 + t) * x + __ldg(a.b + r0 + t);
    a.s[r0 + t] = reset_val(a.s[r0 + t] + x, a.reset_thr, a.reset);
  }
}

// Segments shorten the carry when few sequences have many chunks: a chain of n steps becomes
// M + n / M + M with M about sqrt(n), at the price of folding the aggregates once more. At
// 157 chunks (Langevin, d = 4, float64) 28 us against 40 in one level; below 128 the two
// extra launches cost what is saved. The folds are d^3 work per chunk of every sequence, the chain
// that they save is one sequence's, so they pay up to a number of sequences that hardly depends
// on their length. Per iteration with segments less without, us, 160 / 1024 chunks a sequence:
//   float32 d = 8, 256 sequences -8 / -130, 512 +5 / -79; d = 16, 128: -10 / -85, 256: +8 / -15,
//   512: +34 / +137; d = 32, 16: -1 / -80, 32: +9 / -10, 64: +30 / +119, 256: +152
//   float64 d = 8, 128: -21 / -263, 256: +4 / -74, 512: +58 / +189; d = 16, 32: -13 / -380, 64: +1 /
//   -199, 128: +80 / +522; d = 32, 4: -132 / -946, 16: +19 / -129, 32: +263
// and at d = 4 they pay up to the 512 sequences measured (beyond as many as there are schedulers
// times groups in a warp the sequences hide the chain by themselves). The batch size decides, not
// the active set: the two forms round differently, and a call keeps one of them, whatever else is
// still active and whichever loop runs.
template <class real, int D>
constexpr int64_t segment_batch() {
  constexpr bool f64 = sizeof(real) == 8;
  if (D <= 4) return kSchedulers * (32 / group_lanes<D>());
  if (D <= 8) return f64 ? 256 : 512;
  if (D <= 16) return f64 ? 64 : 224;
  return f64 ? 12 : 24;
}

template <class real, int D>
static void set_segments(DenseScanArgs<real>& a) {
  a.log2M = 0;
  const int64_t n = a.max_chunks;
  if (!a.segP || n < 128 || a.bt.B > segment_batch<real, D>()) return;
  a.log2M = 3;
  while (a.log2M < 6 && ((int64_t)1 << (2 * a.log2M + 2)) <= n) ++a.log2M;
}

template <class real, int D, bool SEG>
static void dense_chunk_launch(const DenseScanArgs<real>& a, int64_t spans, unsigned ny,
                               cudaStream_t st) {
  constexpr int G = D == 32 ? 1 : 32 / group_lanes<D>();
  const dim3 g(grid_for(spans, G), ny);
  if constexpr (D == 32) {
    if constexpr (sizeof(real) == 4 && !SEG) {
      if (a.tensor_cores) {
        k_dense_chunk_mma32<<<g, 64, 0, st>>>(a);
        return;
      }
    }
    k_dense_chunk_ring4<real, SEG><<<g, 128, 0, st>>>(a);
  } else {
    if constexpr (sizeof(real) == 8 && D >= 4 && D <= 8) {
      // warps per sub-partition x instructions per row: entries against whole groups
      const int64_t warps = (spans * ny + kSchedulers - 1) / kSchedulers;
      if (warps * (D == 8 ? 3 : 1) < D + 1) {
        k_dense_chunk_entry<D, SEG><<<dim3((unsigned)spans, ny), 32, 0, st>>>(a);
        return;
      }
    }
    k_dense_chunk_ring<real, D, SEG><<<g, 32, 0, st>>>(a);
  }
}

template <class real, int D>
static void dense_carry(DenseScanArgs<real> a, cudaStream_t st) {
  constexpr int G = 32 / group_lanes<D>();
  set_segments<real, D>(a);
  if (a.log2M == 0) {
    k_dense_carry_ring<real, D, 0><<<grid_for(a.bt.n_act(), G), 32, 0, st>>>(a);
    note_launch();
    return;
  }
  const int64_t segs = (a.max_chunks + (1 << a.log2M) - 1) >> a.log2M;
  const unsigned ny = (unsigned)a.bt.n_act();
  dense_chunk_launch<real, D, true>(a, segs, ny, st);
  k_dense_carry_ring<real, D, 1><<<grid_for(a.bt.n_act(), G), 32, 0, st>>>(a);
  k_dense_carry_ring<real, D, 2><<<dim3(grid_for(segs, G), ny), 32, 0, st>>>(a);
  note_launch(3);
}

cudaError_t launch_dense_carry(const DenseScanArgs<float>& a, cudaStream_t st) {
  if (a.bt.n_act() == 0) return cudaSuccess;
  if (a.d == 16) dense_carry<float, 16>(a, st);
  else if (a.d == 32) dense_carry<float, 32>(a, st);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

template <class real, int D>
static void dense_launch(const DenseScanArgs<real>& a, cudaStream_t st) {
  if constexpr (D == 1) {
    const unsigned gc = grid_for(a.bt.act_chunks(), 128);
    k_scalar_chunk<real><<<gc, 128, 0, st>>>(a);
    k_scalar_carry<real><<<grid_for(a.bt.n_act(), 128), 128, 0, st>>>(a);
    k_scalar_apply<real><<<gc, 128, 0, st>>>(a);
    note_launch(3);
  } else {
    dense_chunk_launch<real, D, false>(a, a.bt.act_chunks(), 1, st);
    dense_carry<real, D>(a, st);
    k_dense_apply_ring<real, D>
        <<<grid_for(a.bt.act_chunks(), 32 / group_lanes<D>()), 32, 0, st>>>(a);
    note_launch(2);
  }
}

template <class real>
cudaError_t launch_dense_scan(const DenseScanArgs<real>& a, cudaStream_t st) {
  if (a.bt.act_rows() == 0) return cudaSuccess;
  switch (a.d) {
    case 1: dense_launch<real, 1>(a, st); break;
    case 2: dense_launch<real, 2>(a, st); break;
    case 4: dense_launch<real, 4>(a, st); break;
    case 5: dense_launch<real, 5>(a, st); break;
    case 8: dense_launch<real, 8>(a, st); break;
    case 16: dense_launch<real, 16>(a, st); break;
    case 32: dense_launch<real, 32>(a, st); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template cudaError_t launch_dense_scan<float>(const DenseScanArgs<float>&, cudaStream_t);
template cudaError_t launch_dense_scan<double>(const DenseScanArgs<double>&, cudaStream_t);

}  // namespace deer

namespace deer {

// ----------------------------------------------------------------------------
// Reverse (adjoint) dense scan, rows visited from the end of the sequence:
// lambda_t = M_t lambda_{t+1} + g_t with M_t = A_{t+1}^T and lambda_{T+1} = 0; chunk
// aggregates compose in reverse row order. Groups, rings and staging as in the forward scan
// (lane i owns entry i of the vectors and column i of the chunk product; A_{t+1} and g_t
// share a slot); every sum runs over k in ascending order, so the results do not depend on
// which kernel forms them. Thread-per-chunk kernels (d <= 8) and direct global reads (d = 16,
// 32) took, per pass: d = 8, 512 x 2047 rows: chunk 446, carry 182, apply 359 us (now 116, 9,
// 75); d = 32, 128 x 16384 rows: chunk 7990, carry 1090, apply 1390 us (now 2835, 88, 1335: A
// is 8.6 GB).
// ----------------------------------------------------------------------------
template <class real, int D>
__device__ __forceinline__ void adj_issue(RowRing<real, D>& R, int slot, int lane,
                                          const AdjScanArgs<real>& a, int64_t row, int64_t rend) {
  if (row + 1 < rend)
    R.issue(slot, lane, a.A + (row + 1) * (int64_t)(D * D), a.g + row * D);
  else if (lane < D)
    cp_async_small<sizeof(real)>(&R.v[slot][lane], a.g + row * D + lane);
}

template <class real, int D>
__global__ void __launch_bounds__(32) k_adj_chunk_ring(AdjScanArgs<real> a) {
  constexpr int W = group_lanes<D>(), G = 32 / W;
  using Ring = RowRing<real, D>;
  constexpr int K = Ring::K;
  __shared__ __align__(16) Ring ring[G];
  const int grp = threadIdx.x / W, lane = threadIdx.x % W;
  const int li = lane < D ? lane : 0;
  const unsigned gm = group_mask<D>();
  const int64_t c = blockIdx.x * (int64_t)G + grp;
  if (c >= a.bt.n_chunks) return;  // whole groups
  int64_t seq, r0;
  int n;
  chunk_rows(a.bt, c, seq, r0, n);
  const int64_t rend = __ldg(a.bt.offsets + seq + 1);              // one past the last row
  const bool need_P = c != __ldg(a.bt.chunk_first + seq + 1) - 1;  // last chunk: carry 0
  Ring& R = ring[grp];
#pragma unroll
  for (int s = 0; s < K; ++s) {
    if (s < n) adj_issue<real, D>(R, s, lane, a, r0 + n - 1 - s, rend);
    cp_async_commit();
  }
  real Pc[D];  // column `lane` of P
  real v = real(0);
#pragma unroll
  for (int i = 0; i < D; ++i) Pc[i] = i == li ? real(1) : real(0);
  for (int j = 0; j < n; ++j) {
    const int s = j & (K - 1);
    const int64_t row = r0 + n - 1 - j;
    cp_async_wait<K - 1>();
    __syncwarp(gm);  // the other lanes' rows of this slot have landed
    real nv = R.v[s][li];
    if (row + 1 < rend) {
#pragma unroll
      for (int k = 0; k < D; ++k) nv += R.m[s][k][li] * __shfl_sync(gm, v, k, W);
      if (need_P) {
        real np[D];
#pragma unroll
        for (int i = 0; i < D; ++i) np[i] = real(0);
#pragma unroll
        for (int k = 0; k < D; ++k) {
          real ar[D];
          R.row(s, k, ar);
          axpy_row<D>(Pc[k], ar, np);
        }
#pragma unroll
        for (int i = 0; i < D; ++i) Pc[i] = np[i];
      }
    } else {
      // last row of the sequence: lambda_T = g_T, the carry (lambda_{T+1} = 0) is dropped
#pragma unroll
      for (int i = 0; i < D; ++i) Pc[i] = real(0);
    }
    v = nv;
    __syncwarp(gm);  // every lane is done with the slot before it is refilled
    if (j + K < n) adj_issue<real, D>(R, s, lane, a, row - K, rend);
    cp_async_commit();
  }
  cp_async_wait<0>();
  if (lane >= D) return;
  real* Po = a.aggP + c * (int64_t)(D * D);
#pragma unroll
  for (int i = 0; i < D; ++i) Po[i * D + lane] = Pc[i];
  a.aggv[c * D + lane] = v;
}

// Chunk pass, d = 32, float32: one warp per chunk, each lane an 8 x 4 tile of the chunk
// product (lane / 8 picks the rows, lane % 8 the columns), so that one 16-byte read of P and
// two of A_{t+1} feed 32 multiply-adds instead of eight reads; P alternates between two
// shared buffers. Bound by the FP32 pipe (32768 multiply-adds per row: 1.8 of its 2.8 ms
// for 2.1 M rows).
__global__ void __launch_bounds__(32) k_adj_chunk_tile32(AdjScanArgs<float> a) {
  constexpr int D = 32, K = 4;
  __shared__ __align__(16) float sA[K][D][D];
  __shared__ __align__(16) float sG[K][D];
  __shared__ __align__(16) float sP[2][D][D];
  __shared__ __align__(16) float sV[2][D];
  const int lane = threadIdx.x, i0 = 8 * (lane >> 3), j0 = 4 * (lane & 7);
  const int64_t c = blockIdx.x;
  int64_t seq, r0;
  int n;
  chunk_rows(a.bt, c, seq, r0, n);
  const int64_t rend = __ldg(a.bt.offsets + seq + 1);
  const bool need_P = c != __ldg(a.bt.chunk_first + seq + 1) - 1;
  auto issue = [&](int slot, int64_t row) {
    if (row + 1 < rend) {
      const float* src = a.A + (row + 1) * (int64_t)(D * D);
#pragma unroll
      for (int p = 0; p < 8; ++p)
        cp_async16(&sA[slot][0][0] + (p * 32 + lane) * 4, src + (p * 32 + lane) * 4);
    }
    cp_async_small<4>(&sG[slot][lane], a.g + row * D + lane);
  };
#pragma unroll
  for (int s = 0; s < K; ++s) {
    if (s < n) issue(s, r0 + n - 1 - s);
    cp_async_commit();
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) sP[0][i0 + i][j0 + j] = i0 + i == j0 + j ? 1.f : 0.f;
  float v = 0.f;
  int cur = 0;
  for (int t = 0; t < n; ++t) {
    const int s = t & (K - 1);
    const int64_t row = r0 + n - 1 - t;
    cp_async_wait<K - 1>();
    sV[t & 1][lane] = v;
    __syncwarp();
    float nv = sG[s][lane];
    if (row + 1 < rend) {
#pragma unroll
      for (int k = 0; k < D; k += 4) {
        const float4 x = *reinterpret_cast<const float4*>(&sV[t & 1][k]);
        nv += sA[s][k][lane] * x.x;
        nv += sA[s][k + 1][lane] * x.y;
        nv += sA[s][k + 2][lane] * x.z;
        nv += sA[s][k + 3][lane] * x.w;
      }
      if (need_P) {
        float2 acc[4][4];  // rows i0 + 2 q, + 1; column j0 + j
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[q][j] = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int k = 0; k < D; ++k) {
          const float4 x = *reinterpret_cast<const float4*>(&sA[s][k][i0]);
          const float4 y = *reinterpret_cast<const float4*>(&sA[s][k][i0 + 4]);
          const float4 p = *reinterpret_cast<const float4*>(&sP[cur][k][j0]);
          const float2 m[4] = {make_float2(x.x, x.y), make_float2(x.z, x.w),
                               make_float2(y.x, y.y), make_float2(y.z, y.w)};
          const float pj[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float2 pp = make_float2(pj[j], pj[j]);
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q][j] = __ffma2_rn(m[q], pp, acc[q][j]);
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          *reinterpret_cast<float4*>(&sP[cur ^ 1][i0 + 2 * q][j0]) =
              make_float4(acc[q][0].x, acc[q][1].x, acc[q][2].x, acc[q][3].x);
          *reinterpret_cast<float4*>(&sP[cur ^ 1][i0 + 2 * q + 1][j0]) =
              make_float4(acc[q][0].y, acc[q][1].y, acc[q][2].y, acc[q][3].y);
        }
        cur ^= 1;
      }
    } else {
      // last row of the sequence: the carry (lambda_{T+1} = 0) is dropped
#pragma unroll
      for (int i = 0; i < 8; ++i)
        *reinterpret_cast<float4*>(&sP[cur][i0 + i][j0]) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    v = nv;
    __syncwarp();  // every lane is done with the slot before it is refilled
    if (t + K < n) issue(s, row - K);
    cp_async_commit();
  }
  cp_async_wait<0>();
  __syncwarp();
  float* Po = a.aggP + c * (int64_t)(D * D);
#pragma unroll
  for (int p = 0; p < 8; ++p)
    reinterpret_cast<float4*>(Po)[p * 32 + lane] =
        reinterpret_cast<const float4*>(&sP[cur][0][0])[p * 32 + lane];
  a.aggv[c * D + lane] = v;
}

template <class real, int D>
__global__ void __launch_bounds__(32) k_adj_carry_ring(AdjScanArgs<real> a) {
  constexpr int W = group_lanes<D>(), G = 32 / W;
  using Ring = RowRing<real, D>;
  constexpr int K = Ring::K;
  __shared__ __align__(16) Ring ring[G];
  const int grp = threadIdx.x / W, lane = threadIdx.x % W;
  const int li = lane < D ? lane : 0;
  const unsigned gm = group_mask<D>();
  const int64_t seq = blockIdx.x * (int64_t)G + grp;
  if (seq >= a.bt.B) return;
  const int64_t c0 = a.bt.chunk_first[seq], c1 = a.bt.chunk_first[seq + 1];
  Ring& R = ring[grp];
#pragma unroll
  for (int s = 0; s < K; ++s) {
    if (c1 - 1 - s >= c0)
      R.issue(s, lane, a.aggP + (c1 - 1 - s) * (int64_t)(D * D), a.aggv + (c1 - 1 - s) * D);
    cp_async_commit();
  }
  real x = real(0);
  int s = 0;
  for (int64_t c = c1 - 1; c >= c0; --c) {
    cp_async_wait<K - 1>();
    __syncwarp(gm);
    if (lane < D) a.cin[c * D + lane] = x;
    real y = R.v[s][li];
    real pr[D];
    R.row(s, li, pr);
#pragma unroll
    for (int k = 0; k < D; ++k) y += pr[k] * __shfl_sync(gm, x, k, W);
    x = y;
    __syncwarp(gm);
    if (c - K >= c0)
      R.issue(s, lane, a.aggP + (c - K) * (int64_t)(D * D), a.aggv + (c - K) * D);
    cp_async_commit();
    s = (s + 1) & (K - 1);
  }
  cp_async_wait<0>();
}

template <class real, int D>
__global__ void __launch_bounds__(32) k_adj_apply_ring(AdjScanArgs<real> a) {
  constexpr int W = group_lanes<D>(), G = 32 / W;
  using Ring = RowRing<real, D>;
  constexpr int K = Ring::K;
  __shared__ __align__(16) Ring ring[G];
  const int grp = threadIdx.x / W, lane = threadIdx.x % W;
  const int li = lane < D ? lane : 0;
  const unsigned gm = group_mask<D>();
  const int64_t c = blockIdx.x * (int64_t)G + grp;
  if (c >= a.bt.n_chunks) return;
  int64_t seq, r0;
  int n;
  chunk_rows(a.bt, c, seq, r0, n);
  const int64_t rend = __ldg(a.bt.offsets + seq + 1);
  Ring& R = ring[grp];
#pragma unroll
  for (int s = 0; s < K; ++s) {
    if (s < n) adj_issue<real, D>(R, s, lane, a, r0 + n - 1 - s, rend);
    cp_async_commit();
  }
  real x = a.cin[c * D + li];
  for (int j = 0; j < n; ++j) {
    const int s = j & (K - 1);
    const int64_t row = r0 + n - 1 - j;
    cp_async_wait<K - 1>();
    __syncwarp(gm);
    real y = R.v[s][li];
    if (row + 1 < rend) {
#pragma unroll
      for (int k = 0; k < D; ++k) y += R.m[s][k][li] * __shfl_sync(gm, x, k, W);
    }
    x = y;
    if (lane < D) a.lam[row * D + lane] = y;
    __syncwarp(gm);
    if (j + K < n) adj_issue<real, D>(R, s, lane, a, row - K, rend);
    cp_async_commit();
  }
  cp_async_wait<0>();
}

// d = 1: one thread per chunk (per sequence in the carry pass), as in the forward scan: groups of
// one lane staged through rings took 1.1 to 1.4 times as long (1 x 5000 rows, float32: a gradient
// call 0.205 ms against 0.147).
template <class real>
__global__ void __launch_bounds__(128) k_scalar_adj_chunk(AdjScanArgs<real> a) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= a.bt.n_chunks) return;
  int64_t seq, r0;
  int n;
  chunk_rows(a.bt, c, seq, r0, n);
  const int64_t rend = __ldg(a.bt.offsets + seq + 1);  // one past the last row
  real P = real(1), v = real(0);
  for (int64_t row = r0 + n - 1; row >= r0; --row) {
    // (the last row of the sequence drops the carry, lambda_{T+1} = 0)
    const real An = row + 1 < rend ? __ldg(a.A + row + 1) : real(0);
    v = row + 1 < rend ? An * v + __ldg(a.g + row) : __ldg(a.g + row);
    P = An * P;
  }
  a.aggP[c] = P;
  a.aggv[c] = v;
}

template <class real>
__global__ void __launch_bounds__(128) k_scalar_adj_carry(AdjScanArgs<real> a) {
  const int64_t seq = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (seq >= a.bt.B) return;
  const int64_t c0 = a.bt.chunk_first[seq];
  real x = real(0);
  // (loads of kCarry aggregates at a time: they do not depend on x)
  for (int64_t cb = a.bt.chunk_first[seq + 1] - 1; cb >= c0; cb -= kCarry) {
    real P[kCarry], v[kCarry];
#pragma unroll
    for (int k = 0; k < kCarry; ++k) {
      const int64_t c = cb - k >= c0 ? cb - k : c0;
      P[k] = a.aggP[c];
      v[k] = a.aggv[c];
    }
#pragma unroll
    for (int k = 0; k < kCarry; ++k) {
      if (cb - k < c0) break;
      a.cin[cb - k] = x;
      x = P[k] * x + v[k];
    }
  }
}

template <class real>
__global__ void __launch_bounds__(128) k_scalar_adj_apply(AdjScanArgs<real> a) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= a.bt.n_chunks) return;
  int64_t seq, r0;
  int n;
  chunk_rows(a.bt, c, seq, r0, n);
  const int64_t rend = __ldg(a.bt.offsets + seq + 1);
  real x = a.cin[c];
  for (int64_t row = r0 + n - 1; row >= r0; --row) {
    x = row + 1 < rend ? __ldg(a.A + row + 1) * x + __ldg(a.g + row) : __ldg(a.g + row);
    a.lam[row] = x;
  }
}

template <class real, int D>
static void adj_launch(const AdjScanArgs<real>& a, cudaStream_t st) {
  if constexpr (D == 1) {
    const unsigned gc = grid_for(a.bt.n_chunks, 128);
    k_scalar_adj_chunk<real><<<gc, 128, 0, st>>>(a);
    k_scalar_adj_carry<real><<<grid_for(a.bt.B, 128), 128, 0, st>>>(a);
    k_scalar_adj_apply<real><<<gc, 128, 0, st>>>(a);
    note_launch(3);
  } else {
    constexpr int G = 32 / group_lanes<D>();
    const unsigned gc = grid_for(a.bt.n_chunks, G);
    if constexpr (D == 32 && sizeof(real) == 4) k_adj_chunk_tile32<<<gc, 32, 0, st>>>(a);
    else k_adj_chunk_ring<real, D><<<gc, 32, 0, st>>>(a);
    k_adj_carry_ring<real, D><<<grid_for(a.bt.B, G), 32, 0, st>>>(a);
    k_adj_apply_ring<real, D><<<gc, 32, 0, st>>>(a);
    note_launch(3);
  }
}

template <class real>
cudaError_t launch_adjoint_scan(const AdjScanArgs<real>& a, cudaStream_t st) {
  if (a.bt.N == 0) return cudaSuccess;
  switch (a.d) {
    case 1: adj_launch<real, 1>(a, st); break;
    case 2: adj_launch<real, 2>(a, st); break;
    case 4: adj_launch<real, 4>(a, st); break;
    case 5: adj_launch<real, 5>(a, st); break;
    case 8: adj_launch<real, 8>(a, st); break;
    case 16: adj_launch<real, 16>(a, st); break;
    case 32: adj_launch<real, 32>(a, st); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template cudaError_t launch_adjoint_scan<float>(const AdjScanArgs<float>&, cudaStream_t);
template cudaError_t launch_adjoint_scan<double>(const AdjScanArgs<double>&, cudaStream_t);

}  // namespace deer
