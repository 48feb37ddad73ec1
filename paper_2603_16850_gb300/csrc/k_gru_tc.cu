// GRU (d = d_in = 64, float32) linearisation on the 5th-generation tensor cores.
//
// Per row t with h = s_{t-1} the step needs three products with fixed 64 x 64 weights
// (GRU cell with zero biases, as in k_gru.cu):
//   G1 = h [Uz; Ur]^T (128 outputs), G2 = (r o h) Uh^T, G3 = (h o r o (1 - r)) M^T,
// M = Uh o Ur^T. For a tile of 128 rows these are 128 x N x 64 matrix products with the
// weights shared by every row, i.e. real GEMMs: they run as tcgen05.mma (kind::tf32) with
// the float32 accumulators in tensor memory. float32 accuracy comes from a three-term split
// x = x_hi + x_lo (x_hi = x truncated to tf32): A B ~ A_hi B_hi + A_hi B_lo + A_lo B_hi,
// relative error about 2^-21 per product, so the residual the Newton iteration is refined
// against keeps float32 accuracy.
//
// One persistent CTA of 16 warps per SM. Shared memory (224 KB) holds the weights, split and
// staged once in the canonical no-swizzle K-major layout, and three 32 KB row buffers; the
// activations (h, then r o h and h o r o (1 - r)) are split straight into tensor memory, where
// the MMAs read their A operand, beside the accumulators (all 512 columns). Warp w works on
// tensor-memory lanes 32 (w % 4) .. + 31 = tile rows and a quarter w / 4 of the columns.
//
// What bounds a tile of 128 rows is its 196 KB of rows (s twice, three input projections, a
// and b written: about 9100 clocks of HBM time per SM) and the gates' arithmetic (about 8000
// issue slots per scheduler), not the MMAs (3300 clocks). So a warp's part of the row buffers
// (its 32 rows x 16 columns of each) is its own: it is filled by cp.async in 64-byte row
// segments ahead of use and emptied without a barrier (pieces swizzled by row),
//   buffer 0: h, then s; the next tile's h while this tile's gates are formed
//   buffer 1: r's projection, then h~'s; the next tile's r
//   buffer 2: z's projection, then a, then b on their way out; the next tile's z
// and only the two hand-overs of operands to the tensor core are block-wide. Two threads of
// different warps issue half of the products each. Per pass over 4.19 M rows: 3.76 ms with
// every thread reading its own row (32 rows per instruction) and the three products back to
// back, 2.42 ms so (39 % of issue slots: four warps per scheduler, dependent gate arithmetic).
// Every mbarrier wait is bounded; a wait that gives up sets the timeout flag and the kernel
// winds down, freeing its tensor memory.
#include "kernels.h"
#include "tc.cuh"

namespace deer {
namespace {

using namespace tc;

constexpr int kD = 64;        // state size = input size
constexpr int kTM = 128;      // rows per tile = MMA M
constexpr int kThreads = 512;  // 16 warps: lane quadrant w % 4, column quarter w / 4
constexpr int kCols = kD / 4;   // columns of each 64-wide block per thread
// tensor memory: D1 (z, r) 128 columns, D2 64, D3 64, operands h / r o h (hi, lo) 128 and
// h o r o (1 - r) (hi, lo) 128
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColA = 256, kColA3 = 384;
constexpr uint32_t kNoRow = 0xffffffffu;
constexpr unsigned kWaitLimit = 1u << 24;

// Canonical no-swizzle K-major layout of an R x 64 float32 operand: core matrices of
// 8 rows x 16 bytes (4 elements) stored contiguously (128 B); core (r / 8, k / 4) at
// ((k / 4) (R / 8) + r / 8) 128 bytes. Leading-dimension byte offset (next core along K)
// R / 8 x 128, stride-dimension byte offset (next 8 rows) 128.
__host__ __device__ constexpr uint32_t core_off(int R, int r, int k) {
  return (uint32_t)(((k >> 2) * (R >> 3) + (r >> 3)) * 128 + (r & 7) * 16 + (k & 3) * 4);
}

struct TcSmem {
  float B1h[128 * kD], B1l[128 * kD];  // [Uz; Ur]
  float B2h[kD * kD], B2l[kD * kD];    // Uh
  float B3h[kD * kD], B3l[kD * kD];    // M
  float buf[3][16][32 * kCols];        // row buffers by warp, 16-byte pieces swizzled by row
};

__device__ __forceinline__ float tf32_hi(float x) {
  return __uint_as_float(__float_as_uint(x) & 0xffffe000u);
}

__device__ __forceinline__ void split_store4(float* hi, float* lo, uint32_t byte_off,
                                             float4 v) {
  const float4 h = make_float4(tf32_hi(v.x), tf32_hi(v.y), tf32_hi(v.z), tf32_hi(v.w));
  *reinterpret_cast<float4*>(reinterpret_cast<unsigned char*>(hi) + byte_off) = h;
  *reinterpret_cast<float4*>(reinterpret_cast<unsigned char*>(lo) + byte_off) =
      make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w);
}

__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
  return tc::bar_wait(bar, parity, kWaitLimit);
}

// D (+)= A B^T (64 outputs) over K = 64 with the three-term split: 8 K-steps of 8 (two core
// matrices of B, whose operand has R rows and whose row `r0` is the first output; eight
// tensor-memory columns of A, hi at `a`, lo 64 columns on)
__device__ __forceinline__ void gemm3(uint32_t dtmem, uint32_t a, const float* Bh,
                                      const float* Bl, int R, int r0) {
  const uint32_t idesc = idesc_tf32(kD, kTM);
  const uint32_t lboB = (uint32_t)(R / 8) * 128, sbo = 128;
  const uint32_t bh = su32(Bh) + r0 / 8 * 128, bl = su32(Bl) + r0 / 8 * 128;
#pragma unroll
  for (int s = 0; s < kD / 8; ++s) {
    const uint32_t bo = (uint32_t)s * 2 * lboB;
    mma_tf32_ts(dtmem, a + 8 * s, sdesc(bh + bo, lboB, sbo), idesc, s > 0);
    mma_tf32_ts(dtmem, a + 8 * s, sdesc(bl + bo, lboB, sbo), idesc, 1u);
    mma_tf32_ts(dtmem, a + kD + 8 * s, sdesc(bh + bo, lboB, sbo), idesc, 1u);
  }
}

// the split of 16 values into an operand's hi and lo columns of this thread's lane
__device__ __forceinline__ void split_tmem(uint32_t taddr, const float (&v)[kCols]) {
  float h[kCols], l[kCols];
#pragma unroll
  for (int j = 0; j < kCols; ++j) {
    h[j] = tf32_hi(v[j]);
    l[j] = v[j] - h[j];
  }
  tmem_st16(taddr, h);
  tmem_st16(taddr + kD, l);
}

// float offset of piece p (four columns) of row r in a warp's part of a row buffer: eight
// rows' equal pieces fall in distinct banks
__device__ __forceinline__ int piece(int r, int p) { return r * kCols + ((p ^ ((r >> 1) & 3)) << 2); }

__device__ __forceinline__ float fsig(float v) { return 1.f / (1.f + __expf(-v)); }

__device__ __forceinline__ float4 ldg4(const float* p) {
  return __ldg(reinterpret_cast<const float4*>(p));
}

}  // namespace

__global__ void __launch_bounds__(kThreads, 1) k_gru_lin_tc(GruTileArgs a) {
  extern __shared__ __align__(1024) unsigned char smraw[];
  TcSmem& S = *reinterpret_cast<TcSmem*>(smraw);
  __shared__ float2 s_diag[kD];  // diagonals of Uz and Uh
  __shared__ __align__(8) unsigned long long mbar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int s_ok1, s_ok2;  // the waits for the first / the other two products succeeded
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int qd = warp & 3, qc = warp >> 2;
  const int rl = 32 * qd + lane;  // tile row = tensor-memory lane
  const int c0 = kCols * qc;      // this thread's columns c0 .. c0 + kCols - 1 of each block
  const float* Uz = a.dv.params + 3 * kD * a.dv.d_in;
  const float* Ur = Uz + kD * kD;
  const float* Uh = Ur + kD * kD;
  // weights, split and staged once: row = output, K = input
  for (int e = tid; e < kD * (kD / 4); e += kThreads) {
    const int i = e / (kD / 4), k = 4 * (e % (kD / 4));
    split_store4(S.B1h, S.B1l, core_off(128, i, k), ldg4(Uz + i * kD + k));
    split_store4(S.B1h, S.B1l, core_off(128, kD + i, k), ldg4(Ur + i * kD + k));
    split_store4(S.B2h, S.B2l, core_off(kD, i, k), ldg4(Uh + i * kD + k));
    split_store4(S.B3h, S.B3l, core_off(kD, i, k), ldg4(a.dv.gru_M + i * kD + k));
  }
  if (tid < kD) s_diag[tid] = make_float2(Uz[tid * kD + tid], Uh[tid * kD + tid]);
  const uint32_t bar = su32(&mbar);
  if (tid == 0) {
    s_ok1 = s_ok2 = 1;
    // two issuing threads commit per phase
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 2;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(&tmem_base_sh)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const int64_t act_rows = a.bt.act_rows();
  const int64_t n_tiles = (act_rows + kTM - 1) / kTM;
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_base_sh;
  const uint32_t tl = tmem + ((uint32_t)(32 * qd) << 16);  // this warp's lanes, column 0
  uint32_t phase = 0, last = 0;
  const float kk = a.dparam;
  float* B0 = S.buf[0][warp];
  float* B1 = S.buf[1][warp];
  float* B2 = S.buf[2][warp];
  // this lane's row of a tile: 2 row + (1 if the first of its sequence), kNoRow past the end
  auto find_row = [&](int64_t tile, uint32_t& code, int64_t& seq) {
    const int64_t ar = tile * kTM + rl;
    code = kNoRow;
    seq = 0;
    if (tile < n_tiles && ar < act_rows) {
      int64_t row;
      act_row(a.bt, ar, seq, row);
      code = 2 * (uint32_t)row + (row == __ldg(a.bt.offsets + seq) ? 1u : 0u);
    }
  };
  // copy the warp's rows (16 columns each, four lanes per row) into its part of a buffer
  enum { SRC_H, SRC_S, SRC_XZ, SRC_XR, SRC_XH };
  auto copy_rows = [&](float* B, int src, uint32_t code, int64_t seq) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = 8 * q + (lane >> 2), p = lane & 3;
      const uint32_t cr = __shfl_sync(0xffffffffu, code, r);
      const int64_t row = cr >> 1;
      const float* g;
      if (src == SRC_H) {
        const int64_t sr = __shfl_sync(0xffffffffu, (long long)seq, r);
        g = (cr & 1u) ? a.s0 + sr * kD : a.s + (row - 1) * kD;
      } else if (src == SRC_S) {
        g = a.s + row * kD;
      } else {
        g = a.xproj + row * (3 * kD) + (src == SRC_XZ ? 0 : src == SRC_XR ? kD : 2 * kD);
      }
      if (cr != kNoRow) cp_async16(B + piece(r, p), g + c0 + 4 * p);
    }
  };
  auto read16 = [&](const float* B, float (&v)[kCols]) {
#pragma unroll
    for (int p = 0; p < kCols / 4; ++p) {
      const float4 x = *reinterpret_cast<const float4*>(B + piece(lane, p));
      v[4 * p] = x.x; v[4 * p + 1] = x.y; v[4 * p + 2] = x.z; v[4 * p + 3] = x.w;
    }
  };
  // the warp's part of buffer 2, filled with this lane's 16 values, to its rows of `dst`
  auto rows_out = [&](const float (&v)[kCols], float* dst, uint32_t code) {
    __syncwarp();
#pragma unroll
    for (int p = 0; p < kCols / 4; ++p)
      *reinterpret_cast<float4*>(B2 + piece(lane, p)) =
          make_float4(v[4 * p], v[4 * p + 1], v[4 * p + 2], v[4 * p + 3]);
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = 8 * q + (lane >> 2), p = lane & 3;
      const uint32_t cr = __shfl_sync(0xffffffffu, code, r);
      if (cr != kNoRow)
        *reinterpret_cast<float4*>(dst + (int64_t)(cr >> 1) * kD + c0 + 4 * p) =
            *reinterpret_cast<const float4*>(B2 + piece(r, p));
    }
  };
  // wait (bounded) for the products committed last
  auto wait_mma = [&](int& flag) {
    last = phase;
    if (!bar_wait(bar, last)) flag = 0;
    phase ^= 1u;
    fence_after();
  };
  // operands complete in tensor memory: hand over to the issuing threads
  auto hand_over = [&]() {
    tmem_wait_st();
    fence_before();
    __syncthreads();
    fence_after();
  };
  const bool issuer = tid == 0 || tid == 128;

  uint32_t code;
  int64_t seq;
  find_row(blockIdx.x, code, seq);
  copy_rows(B0, SRC_H, code, seq);
  copy_rows(B1, SRC_XR, code, seq);
  cp_async_commit();
  copy_rows(B2, SRC_XZ, code, seq);
  cp_async_commit();
  bool ok = true;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const bool v = code != kNoRow;
    // stage 1: h into tensor memory, [z; r] products
    float h[kCols], r[kCols];
    cp_async_wait<1>();
    __syncwarp();  // the warp's h and r rows have landed
    read16(B0, h);
    read16(B1, r);
    if (!v) {
#pragma unroll
      for (int j = 0; j < kCols; ++j) h[j] = 0.f;
    }
    split_tmem(tl + kColA + c0, h);
    hand_over();
    if (!(ok = s_ok2 != 0)) break;  // (of the tile before; written before the barrier)
    if (issuer) {
      if (tid == 0) gemm3(tmem + kD, tmem + kColA, S.B1h, S.B1l, 128, kD);
      else gemm3(tmem, tmem + kColA, S.B1h, S.B1l, 128, 0);
      mma_commit(bar);
    }
    __syncwarp();
    copy_rows(B0, SRC_S, code, seq);
    copy_rows(B1, SRC_XH, code, seq);
    cp_async_commit();
    uint32_t ncode;
    int64_t nseq;
    find_row(tile + gridDim.x, ncode, nseq);
    // stage 2: r = sig(Wr x + Ur h), then the operands of the two remaining products
    wait_mma(s_ok1);
    {
      float rp[kCols];
      tmem_ld16(tl + kD + c0, rp);
      tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < kCols; ++j) r[j] = fsig(rp[j] + r[j]);
#pragma unroll
      for (int j = 0; j < kCols; ++j) rp[j] = r[j] * h[j];
      split_tmem(tl + kColA + c0, rp);
#pragma unroll
      for (int j = 0; j < kCols; ++j) rp[j] = h[j] * r[j] * (1.f - r[j]);
      split_tmem(tl + kColA3 + c0, rp);
    }
    hand_over();
    if (!(ok = s_ok1 != 0)) break;
    if (issuer) {
      if (tid == 0) gemm3(tmem + 128, tmem + kColA, S.B2h, S.B2l, kD, 0);
      else gemm3(tmem + 192, tmem + kColA3, S.B3h, S.B3l, kD, 0);
      mma_commit(bar);
    }
    __syncwarp();
    float sc[kCols], xz[kCols], xh[kCols];
    cp_async_wait<0>();
    __syncwarp();  // the warp's s, z and h~ rows have landed
    read16(B0, sc);
    read16(B1, xh);
    read16(B2, xz);
    __syncwarp();
    copy_rows(B0, SRC_H, ncode, nseq);
    copy_rows(B1, SRC_XR, ncode, nseq);
    cp_async_commit();
    wait_mma(s_ok2);
    // gates, F, diagonal Jacobian, residual (two halves of 8 columns); a and b replace the z
    // and h~ projections
    float mx = 0.f, sq = 0.f;
#pragma unroll
    for (int hh = 0; hh < kCols; hh += 8) {
      float zp[8], hq[8], mc[8];
      tmem_ld8(tl + c0 + hh, zp);
      tmem_ld8(tl + 128 + c0 + hh, hq);
      tmem_ld8(tl + 192 + c0 + hh, mc);
      tmem_wait_ld();
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int j = hh + e;
        const float zi = fsig(zp[e] + xz[j]);
        const float ri = r[j];
        const float ht = tanhf(hq[e] + xh[j]);
        const float hv = h[j];
        const float F = (1.f - zi) * hv + zi * ht;
        float ai;
        if (a.jac == DEER_JAC_DIAG) {
          const float2 dg = s_diag[c0 + j];
          ai = (1.f - zi) + (ht - hv) * zi * (1.f - zi) * dg.x +
               zi * (1.f - ht * ht) * (dg.y * ri + mc[e]);
        } else {
          ai = a.jac == DEER_JAC_IDENTITY ? 1.f : 0.f;
        }
        if (a.damp == DEER_DAMP_SCALE) ai *= (1.f - kk);
        else if (a.damp == DEER_DAMP_CLIP) ai = fminf(fmaxf(ai, -kk), kk);
        xz[j] = ai;
        xh[j] = F - ai * hv;
        const float res = sc[j] - F;
        const float sa = fabsf(sc[j]);
        const float m = sa > 1.f ? fabsf(res) / sa : fabsf(res);
        mx = (m > mx || m != m) ? m : mx;
        sq += res * res;
      }
    }
    fence_before();  // (the next hand-over orders these reads before the products after it)
    if (a.jac == DEER_JAC_DIAG) rows_out(xz, a.A, code);
    rows_out(xh, a.b, code);
    acc_resid_f(a.acc, seq, v, mx, sq,
                bad_key(v && !(mx <= a.tol_f),
                        (int64_t)(code >> 1) - (v ? __ldg(a.bt.offsets + seq) : 0)));
    __syncwarp();
    code = ncode;
    seq = nseq;
    copy_rows(B2, SRC_XZ, code, seq);
    cp_async_commit();
  }
  __syncthreads();
  if (s_ok2 == 0) ok = false;
  cp_async_wait<0>();
  if (!ok) {
    if (tid == 0) atomicExch(&a.status->timeout, 1);
    // products may still be in flight: give them (bounded) time before tensor memory is
    // released
    bar_wait(bar, last);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kTmemCols)
                 : "memory");
}

cudaError_t launch_gru_lin_tc(const GruTileArgs& a, cudaStream_t st) {
  if (a.bt.act_rows() == 0) return cudaSuccess;
  const int smem = (int)sizeof(TcSmem);
  static DeviceOnce configured;
  const cudaError_t e = allow_smem(configured, k_gru_lin_tc, smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t tiles = (a.bt.act_rows() + kTM - 1) / kTM;
  const int64_t g = tiles < sms ? tiles : sms;
  k_gru_lin_tc<<<(unsigned)(g > 0 ? g : 1), kThreads, smem, st>>>(a);
  note_launch();
  return cudaGetLastError();
}

}  // namespace deer
