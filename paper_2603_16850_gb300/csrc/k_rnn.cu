// Mean-field RNN, d = 32, float32, full Jacobian: the dense scan without stored Jacobians.
//
// A_t = W diag(e_t), e_t = 1 - tanh(s_{t-1})^2 (times the scale damping): 32 values per row
// instead of 1024. The linearisation stores e_t where the Jacobians would go, and the chunk and
// apply passes hold W in registers for a whole chunk:
//   chunk   P^T <- (P^T diag(e_t)) W^T  as warp-level tf32 MMAs with the three-term split, W's
//           fragments split once, and v <- W (e_t o v) + b_t
//   apply   Delta_t = W (e_t o Delta_{t-1}) + b_t, s_t += Delta_t
// Dense passes read 4 KB per row twice after writing it once; these are bound by the MMAs
// (chunk) and the chain of a row (apply). 100000 rows, g = 0.5, per iteration: linearisation
// 178 -> 64 us, chunk 204 -> 135, apply 74 -> 20.
#include "kernels.h"
#include "tc.cuh"

namespace deer {
namespace {

constexpr int kD = 32;
constexpr int kRing = 8;  // rows copied ahead

// 32 values of a row-major 32 x 32 matrix's row
__device__ __forceinline__ void load_row32(const float* p, float (&w)[kD]) {
#pragma unroll
  for (int k = 0; k < kD; k += 4) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(p + k));
    w[k] = q.x; w[k + 1] = q.y; w[k + 2] = q.z; w[k + 3] = q.w;
  }
}

// W x for this lane's row w, x from shared memory (four partial sums)
__device__ __forceinline__ float row_dot(const float (&w)[kD], const float* x) {
  float y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < kD; k += 4) {
    const float4 q = *reinterpret_cast<const float4*>(x + k);
    y[0] += w[k] * q.x;
    y[1] += w[k + 1] * q.y;
    y[2] += w[k + 2] * q.z;
    y[3] += w[k + 3] * q.w;
  }
  return (y[0] + y[1]) + (y[2] + y[3]);
}

// One chunk per block of two warps; warp w carries rows 16 w .. 16 w + 15 of P^T (columns of
// P) in the accumulator layout (see k_dense_chunk_mma32), warp 0 also the vector part.
__global__ void __launch_bounds__(64) k_rnn_chunk32(DenseScanArgs<float> a, DynView<float> dv) {
  constexpr int D = kD, K = kRing;
  __shared__ __align__(16) float sE[K][D], sB[K][D], sX[D];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tq = lane & 3;
  if ((int64_t)blockIdx.x >= a.bt.act_chunks()) return;  // uniform over the block
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, blockIdx.x, seq, c, r0, n);
  const bool need_P = c != win_first(a.bt, seq);
  const float* W = dv.params + seq * dv.pstride;
  auto issue = [&](int t) {
    if (t < n) {
      const int s = t & (K - 1);
      if (warp == 0) cp_async_small<4>(&sE[s][lane], a.A + (r0 + t) * D + lane);
      else cp_async_small<4>(&sB[s][lane], a.b + (r0 + t) * D + lane);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int t = 0; t < K - 1; ++t) issue(t);
  // B operand W^T[k][m] = W[m][k]: m = 8 j + g, k = 8 kk + tq (+ 4), split
  uint32_t bh[4][4][2], bl[4][4][2];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float x = __ldg(W + (8 * j + g) * D + 8 * kk + tq + 4 * e);
        bh[j][kk][e] = tc::tf32_rna(x);
        bl[j][kk][e] = tc::tf32_rna(x - __uint_as_float(bh[j][kk][e]));
      }
  float w[D];
  load_row32(W + lane * D, w);
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
  for (int t = 0; t < n; ++t) {
    const int s = t & (K - 1);
    cp_async_wait<K - 2>();
    __syncthreads();  // row t has landed; row t - 1's slot is free
    issue(t + K - 1);
    if (warp == 0) {
      sX[lane] = sE[s][lane] * v;
      __syncwarp();
      v = row_dot(w, sX) + sB[s][lane];
      __syncwarp();
    }
    if (need_P) {
      float next[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) next[j][e] = 0.f;
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        // A operand: P^T columns 8 kk + tq (+ 4), scaled by e_t, split
        const float x0 = __shfl_sync(0xffffffffu, acc[kk][0], qsrc);
        const float x1 = __shfl_sync(0xffffffffu, acc[kk][1], qsrc);
        const float x2 = __shfl_sync(0xffffffffu, acc[kk][2], qsrc);
        const float x3 = __shfl_sync(0xffffffffu, acc[kk][3], qsrc);
        const float y0 = __shfl_sync(0xffffffffu, acc[kk][0], qsrc + 2);
        const float y1 = __shfl_sync(0xffffffffu, acc[kk][1], qsrc + 2);
        const float y2 = __shfl_sync(0xffffffffu, acc[kk][2], qsrc + 2);
        const float y3 = __shfl_sync(0xffffffffu, acc[kk][3], qsrc + 2);
        const float e0 = sE[s][8 * kk + tq], e1 = sE[s][8 * kk + tq + 4];
        const float av[4] = {e0 * (odd ? x1 : x0), e0 * (odd ? x3 : x2), e1 * (odd ? y1 : y0),
                             e1 * (odd ? y3 : y2)};
        uint32_t ah[4], al[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          ah[e] = tc::tf32_rna(av[e]);
          al[e] = tc::tf32_rna(av[e] - __uint_as_float(ah[e]));
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          tc::mma_1688_tf32(next[j], al, bh[j][kk][0], bh[j][kk][1]);
          tc::mma_1688_tf32(next[j], ah, bl[j][kk][0], bl[j][kk][1]);
          tc::mma_1688_tf32(next[j], ah, bh[j][kk][0], bh[j][kk][1]);
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = next[j][e];
    }
  }
  cp_async_wait<0>();
  // P[i][j] = P^T[j][i]
  float* Po = a.aggP + c * (int64_t)(D * D);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int n0 = 8 * j + 2 * tq;
    Po[n0 * D + m0] = acc[j][0];
    Po[(n0 + 1) * D + m0] = acc[j][1];
    Po[n0 * D + m0 + 8] = acc[j][2];
    Po[(n0 + 1) * D + m0 + 8] = acc[j][3];
  }
  if (warp == 0) a.aggv[c * D + lane] = v;
}

// One warp per chunk, lane i owns row i of W and entry i of Delta.
__global__ void __launch_bounds__(32) k_rnn_apply32(DenseScanArgs<float> a, DynView<float> dv) {
  constexpr int D = kD, K = kRing;
  __shared__ __align__(16) float sX[2][D];
  __shared__ float sE[K][D], sB[K][D], sS[K][D];
  const int lane = threadIdx.x;
  if ((int64_t)blockIdx.x >= a.bt.act_chunks()) return;
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, blockIdx.x, seq, c, r0, n);
  float* s0 = a.s + r0 * D + lane;
  auto issue = [&](int t) {
    if (t < n) {
      const int s = t & (K - 1);
      cp_async_small<4>(&sE[s][lane], a.A + (r0 + t) * D + lane);
      cp_async_small<4>(&sB[s][lane], a.b + (r0 + t) * D + lane);
      cp_async_small<4>(&sS[s][lane], s0 + t * D);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int t = 0; t < K; ++t) issue(t);
  float w[D];
  load_row32(dv.params + seq * dv.pstride + lane * D, w);
  float x = a.cin[c * D + lane];
  for (int t = 0; t < n; ++t) {
    const int s = t & (K - 1);
    cp_async_wait<K - 1>();  // each lane reads only its own entries
    float* X = sX[t & 1];
    X[lane] = sE[s][lane] * x;
    __syncwarp();
    x = row_dot(w, X) + sB[s][lane];
    const float y = sS[s][lane] + x;
    s0[t * D] = a.reset && !(y <= a.reset_thr && y >= -a.reset_thr) ? 0.f : y;
    issue(t + K);
  }
  cp_async_wait<0>();
}

}  // namespace

cudaError_t launch_rnn_scan(const DenseScanArgs<float>& a, const DynView<float>& dv,
                            cudaStream_t st) {
  if (a.bt.act_rows() == 0) return cudaSuccess;
  if (a.d != kD) return cudaErrorInvalidValue;
  const unsigned g = grid_for(a.bt.act_chunks(), 1);
  k_rnn_chunk32<<<g, 64, 0, st>>>(a, dv);
  const cudaError_t e = launch_dense_carry(a, st);
  if (e != cudaSuccess) return e;
  k_rnn_apply32<<<g, 32, 0, st>>>(a, dv);
  note_launch(2);
  return cudaGetLastError();
}

}  // namespace deer
