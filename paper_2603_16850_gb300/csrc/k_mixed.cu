// Mixed-precision full-Jacobian iteration for mass-action kinetics with d = 16 / 32 (see
// MixedLinArgs / MixedScanArgs in kernels.h). The residual the Newton iteration is refined
// against, and the state, stay in float64; the Jacobian only steers the correction, so it
// is formed in float32 and stored (minus the identity) in bfloat16, halving its traffic.
#include "kernels.h"
#include "tc.cuh"

namespace deer {

template <int D>
__device__ __forceinline__ unsigned gmask_mixed() {
  return D == 32 ? 0xffffffffu : (0xffffu << (16 * ((threadIdx.x >> 4) & 1)));
}

// Species adjacency: for sequence b and species i, the reactions r that change species i
// and the change nu_{r,i} (reactants -1 each, products +1 each).
// A warp per sequence, lane i on species i: counts, a prefix sum for the offsets, then the
// entries (one thread per sequence took 402 us for 256 networks of 32 species, 48 reactions).
__global__ void __launch_bounds__(32) k_ma_adjacency(int d, int R,
                                                     const int32_t* __restrict__ topo,
                                                     int64_t tstride,
                                                     int32_t* __restrict__ adj_off,
                                                     int32_t* __restrict__ adj_e) {
  const int64_t seq = blockIdx.x;
  const int lane = threadIdx.x;
  const int32_t* tt = topo + seq * tstride;
  int32_t* off = adj_off + seq * (d + 1);
  int32_t* e = adj_e + seq * (int64_t)(4 * R);
  auto change = [&](int r, int i) {
    const int i1 = __ldg(tt + 4 * r), i2 = __ldg(tt + 4 * r + 1);
    const int p1 = __ldg(tt + 4 * r + 2), p2 = __ldg(tt + 4 * r + 3);
    return (i == p1) + (i == p2) - (i == i1) - (i == i2);
  };
  int base = 0;
  for (int i0 = 0; i0 < d; i0 += 32) {  // uniform over the warp
    const int i = i0 + lane;
    int n = 0;
    if (i < d)
      for (int r = 0; r < R; ++r) n += change(r, i) != 0;
    int at = n;  // inclusive prefix
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += x;
    }
    const int total = __shfl_sync(0xffffffffu, at, 31);
    int pos = base + at - n;
    if (i < d) {
      off[i] = pos;
      for (int r = 0; r < R; ++r) {
        const int nu = change(r, i);
        if (nu != 0 && pos < 4 * R) e[pos++] = r | ((nu + 4) << 16);
      }
    }
    base += total;
  }
  if (lane == 0) off[d] = base;
}

cudaError_t launch_ma_adjacency(int64_t n_seq, int d, int R, const int32_t* topo,
                                int64_t tstride, int32_t* adj_off, int32_t* adj_e,
                                cudaStream_t st) {
  if (n_seq == 0) return cudaSuccess;
  k_ma_adjacency<<<(unsigned)n_seq, 32, 0, st>>>(d, R, topo, tstride, adj_off, adj_e);
  note_launch();
  return cudaGetLastError();
}

// Float32 value of a float64 by truncating its mantissa with integer operations (no FP64
// pipe, the scarce unit on this GPU). Used only where the float32 value steers the
// Jacobian, or for a float32 evaluation far from convergence, so rounding toward zero
// (relative error < 2^-23) is immaterial. Magnitudes below the float32 normal range give
// zero, above it the largest float32; NaN stays NaN.
__device__ __forceinline__ float d2f_trunc(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned sign = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7ffu);
  const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29);
  if (e == 0x7ff) return __uint_as_float(sign | 0x7f800000u | (m ? 0x400000u : 0u));
  const int fe = e - 1023 + 127;
  if (fe <= 0) return __uint_as_float(sign);
  if (fe >= 255) return __uint_as_float(sign | 0x7f7fffffu);
  return __uint_as_float(sign | ((unsigned)fe << 23) | m);
}

// Stoichiometric change nu in {-2, -1, 1, 2} as a float64 assembled from its bit pattern.
__device__ __forceinline__ double nu_f64(int nu) {
  const unsigned m = (unsigned)(nu < 0 ? -nu : nu);
  const unsigned hi = (nu < 0 ? 0x80000000u : 0u) | (m == 2u ? 0x40000000u : 0x3ff00000u);
  return __hiloint2double((int)hi, 0);
}

// Scaled residual above which a sequence's rows are evaluated in float32: the float32
// rounding error (~1e-7 relative) is then far below the residual being removed. A float32
// evaluation never reports less than kMixedFloor, so only float64 evaluations can pass the
// convergence test.
constexpr double kMixedFastAbove = 1e-4;
constexpr float kMixedFloor = 1e-6f;

// A species' reactions in shared memory, lane-contiguous (entry e of species i at e D + i):
// reaction | (nu + 4) << 6 | first reactant << 10 | (second reactant + 1) << 16. The walk over
// them gathered both from global memory once per entry, stage and row before.
constexpr int kMixList = 16;

template <int D>
__device__ __forceinline__ void mixed_list(uint32_t* lst, int lane, const int4* tt,
                                           const int32_t* ae, int e0, int e1) {
  for (int e = 0; e < kMixList && e0 + e < e1; ++e) {
    const int code = __ldg(ae + e0 + e), r = code & 0xffff;
    const int4 q = __ldg(tt + r);
    // (a reaction naming no species changes nothing here; the set-up kernel reports it)
    const bool ok = q.x >= 0 && q.x < D && q.y >= -1 && q.y < D;
    lst[e * D + lane] = ok ? (uint32_t)r | (uint32_t)(code >> 16) << 6 | (uint32_t)q.x << 10 |
                                 (uint32_t)(q.y + 1) << 16
                           : (uint32_t)r | 4u << 6;
  }
}

// A row of D floats from shared memory in 16-byte pieces (16-byte aligned).
template <int D>
__device__ __forceinline__ void ld_row4(const float* p, float (&v)[D]) {
#pragma unroll
  for (int j = 0; j < D; j += 4) {
    const float4 q = *reinterpret_cast<const float4*>(p + j);
    v[j] = q.x; v[j + 1] = q.y; v[j + 2] = q.z; v[j + 3] = q.w;
  }
}

// One row of the mixed linearisation with the dynamics' value path (stage states, reaction
// rates, slopes, F, residual) in V = float or double; the Jacobian path is float32 either
// way. Writes E and b for the row and returns its scaled residual and squared residual.
//
// A lane per species: the form of d = 32 and of the recomputing path. The row's outputs go to
// Eo (its D x D block of E) and bo (its entry of b = -r): bfloat16 in global memory, or float32
// in shared memory on the recomputing path. sc is the row's own state s_t (read by the caller).
template <class V, int D, bool RK4, int RPL, class TE>
__device__ __forceinline__ void mixed_row(const MixedLinArgs& a, bool valid, int64_t row,
                                          int lane, unsigned gm, double s_prev_d, double sc,
                                          const int4 (&q)[RPL], const double (&kd)[RPL],
                                          const float (&kf)[RPL], int R, const int4* tt,
                                          const int32_t* ae, int e0, int e1,
                                          const uint32_t* lst, float (*sG)[D + 4],
                                          float (*sK)[D + 4], V* sRate, float* sD1,
                                          float* sD2, float& mx, float& sq,
                                          int64_t seq, unsigned long long& key,
                                          float* bo, TE* Eo) {
  constexpr bool F64 = sizeof(V) == 8;
  const V s_prev = F64 ? (V)s_prev_d : (V)d2f_trunc(s_prev_d);
  const V h = F64 ? (V)a.dv.dt : (V)a.dt_f;
  const float hf = a.dt_f;
  V c = s_prev, acc = V(0);
  float Kacc[D];
#pragma unroll
  for (int j = 0; j < D; ++j) Kacc[j] = 0.f;
  const int nst = RK4 ? 4 : 1;
  for (int stage = 0; stage < nst; ++stage) {
    // RK4 tableau: stage derivative weights (1, 2, 2, 1), stage offsets (h/2, h/2, h)
    const float cK = stage == 0 ? 0.f : (stage == 3 ? hf : 0.5f * hf);
    const V w = (stage == 1 || stage == 2) ? V(2) : V(1);
    const float cf = F64 ? d2f_trunc((double)c) : (float)c;
    // every reaction's rate once (reaction r on lane r mod d) and its two partials
#pragma unroll
    for (int k = 0; k < RPL; ++k) {
      if (k * D >= R) break;  // uniform over the group
      const int r = k * D + lane;
      const int j2 = q[k].y < 0 ? 0 : q[k].y;
      const V c1 = __shfl_sync(gm, c, q[k].x, D);
      const V c2 = __shfl_sync(gm, c, j2, D);
      float c1f, c2f;
      if constexpr (F64) {
        c1f = __shfl_sync(gm, cf, q[k].x, D);
        c2f = __shfl_sync(gm, cf, j2, D);
      } else {
        c1f = (float)c1;  // the value path's own concentrations
        c2f = (float)c2;
      }
      if (r < R) {
        const bool bi = q[k].y >= 0;
        const V kr = F64 ? (V)kd[k] : (V)kf[k];
        sRate[r] = bi ? kr * c1 * c2 : kr * c1;
        sD1[r] = bi ? kf[k] * c2f : kf[k];
        sD2[r] = kf[k] * c1f;
      }
    }
#pragma unroll
    for (int j = 0; j < D; j += 4)
      *reinterpret_cast<float4*>(&sG[lane][j]) = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp(gm);
    // this species' slope and its row of the rate Jacobian, from its own reactions
    V g = V(0);
    const int n1 = e1 - e0 < kMixList ? e1 - e0 : kMixList;
    auto entry = [&](int r, int nu, int i1, int i2) {
      g += (F64 ? (V)nu_f64(nu) : (V)nu) * sRate[r];
      const float nuf = (float)nu;
      sG[lane][i1] += nuf * sD1[r];
      if (i2 >= 0) sG[lane][i2] += nuf * sD2[r];
    };
    for (int e = 0; e < n1; ++e) {
      const uint32_t w = lst[e * D + lane];
      entry((int)(w & 63u), (int)((w >> 6) & 15u) - 4, (int)((w >> 10) & 63u),
            (int)(w >> 16) - 1);
    }
    for (int e = e0 + kMixList; e < e1; ++e) {  // the rest of a long list
      const int code = __ldg(ae + e);
      const int4 qq = __ldg(tt + (code & 0xffff));
      if (qq.x >= 0 && qq.x < D && qq.y >= -1 && qq.y < D)  // (as in mixed_list)
        entry(code & 0xffff, (code >> 16) - 4, qq.x, qq.y);
    }
    __syncwarp(gm);
    float Gi[D], Kn[D];
    ld_row4<D>(&sG[lane][0], Gi);
#pragma unroll
    for (int j = 0; j < D; ++j) Kn[j] = Gi[j];
    if (stage > 0) {
#pragma unroll
      for (int m = 0; m < D; ++m) {
        float km[D];
        ld_row4<D>(&sK[m][0], km);  // the same row for every lane of the group
        axpy_row<D>(cK * Gi[m], km, Kn);
      }
    }
    __syncwarp(gm);
    const float wf = (stage == 1 || stage == 2) ? 2.f : 1.f;
#pragma unroll
    for (int j = 0; j < D; j += 4)
      *reinterpret_cast<float4*>(&sK[lane][j]) = make_float4(Kn[j], Kn[j + 1], Kn[j + 2], Kn[j + 3]);
    axpy_row<D>(wf, Kn, Kacc);
    acc += w * g;
    const V cs = stage == 2 ? h : V(0.5) * h;
    c = s_prev + cs * g;
    __syncwarp(gm);
  }
  const V hw = RK4 ? h / V(6) : h;
  const V F = s_prev + hw * acc;
  if (valid) {
    const float scf = d2f_trunc(sc);
    float rf;
    if constexpr (F64) rf = d2f_trunc(sc - (double)F);
    else rf = scf - (float)F;
    const float sabs = fabsf(scf);
    float m = fabsf(rf) / (sabs > 1.f ? sabs : 1.f);
    if (!F64 && !(m != m)) m = m > kMixedFloor ? m : kMixedFloor;
    mx = nanmaxf(mx, m);
    sq += rf * rf;
    if (!(m <= a.tol_f) && key == 0ull) key = bad_key(true, row - __ldg(a.bt.offsets + seq));
    const float scale = a.scale_f;
    const float hwf = RK4 ? hf / 6.f : hf;
    // E = A - I with A = I + hw Kacc (scaled by (1 - k) under scale-ELK: E = s A - I):
    // bfloat16, or float32 with rows padded to 20
    auto e = [&](int j) { return scale * hwf * Kacc[j] + (j == lane ? scale - 1.f : 0.f); };
    if constexpr (sizeof(TE) == 4) {
#pragma unroll
      for (int j = 0; j < D; j += 4)
        *reinterpret_cast<float4*>(Eo + lane * 20 + j) =
            make_float4(e(j), e(j + 1), e(j + 2), e(j + 3));
    } else {
#pragma unroll
      for (int j = 0; j < D; j += 8) {
        __nv_bfloat162 w[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) w[m] = __floats2bfloat162_rn(e(j + 2 * m), e(j + 2 * m + 1));
        *reinterpret_cast<uint4*>(Eo + lane * D + j) = *reinterpret_cast<const uint4*>(w);
      }
    }
    bo[lane] = -rf;
  }
}

// ---- linearisation, d = 16: two columns per lane ----------------------------------------
// D / 2 lanes share a row: each forms the rate-Jacobian rows of its two species, then takes
// its two columns of every stage Jacobian K_j = G_j (I + c_j K_{j-1}) with both factors of a
// column at hand: K_{j-1}'s columns in registers, G's rows broadcast from shared memory, so
// the products are two-wide FMAs and K is never exchanged. What bounds it is shared-memory
// wavefronts. With a lane per species (row i of K, K_{j-1} broadcast) 94 % of their rate was
// in use, the FMA pipe at 17 %: half of them the scatter of every reaction's partials into G
// (zero, add in place, read back), half the K rows. Here G's entries are sums of products
// coefficient x concentration, listed once per sequence in the order of their entries, so
// that each is summed in a register and stored once; entries that no term names stay zero.
// Sums keep the reactions' order and the products round alike (nu is a power of two up to
// sign), so the results are those of the scatter. 3.2 M rows, d = 16, 24 reactions:
// 8.8 -> 6.1 ms, evaluated in float64 9.7 -> 8.6 (then the float64 pipe counts too). Tried and
// slower: the products as tf32 MMAs with the three-term split (fewer reads of G, but the splits
// cost more instructions: 7.6 ms), and more rows per warp (128: partly filled last rounds).
//
// A warp walks kMixRows consecutive rows, 32 / (D / 2) at a time, all of one sequence, so that
// it holds one network: lists and rate constants are built once per warp and sequence, and the
// residual statistics flushed once.
constexpr int kMixRows = 32;
constexpr int kMixTerms = 2 * kMixList;  // entries of G named by a species' listed reactions
constexpr int kMixReact = 64;            // reactions per network (the host checks)
constexpr int kMixBatch = 4;             // list entries whose loads are issued together
static_assert(kMixList % kMixBatch == 0, "lists are filled up to whole batches");

template <int D>
struct MixNet {  // one per warp
  // term e of species i: coefficient, byte offset in G | last of its entry | byte offset of the
  // source concentration << 16
  uint2 term[kMixTerms][D];
  uint32_t run[kMixList][D];   // reaction e of species i: change (float bits) | reaction
  uint32_t react[kMixReact];   // first reactant | second << 8 (D, whose concentration is 1)
  double kd[kMixReact];
  float kf[kMixReact];
};

template <int D>
struct MixRow {  // one per row in flight
  float G[D * (D + 4) + 4];
  float c[D + 4];   // c[D] = 1
  double cd[D + 2];
  double rate[kMixReact + 2];  // [kMixReact] = 0; floats in float32 mode
  float pad[8];  // the rows of a warp in different banks (d = 16)
};

__device__ __forceinline__ float mix_nu(uint32_t w, float) {
  return __uint_as_float(w & 0xffffff80u);
}
__device__ __forceinline__ double mix_nu(uint32_t w, double) {  // +-1 or +-2 (or next to 0)
  return __hiloint2double(
      (int)((w & 0x80000000u) | (((w >> 3) & 0x0ff00000u) + 0x38000000u)), 0);
}

// The sequence's lists, by the whole warp, and the lengths of the longest: most_t entries of G
// and most_g reactions of a species (shorter lists are filled up with entries of no effect).
template <int D>
__device__ __forceinline__ void mix_net(const MixedLinArgs& a, int64_t seq, int R, int l32,
                                        MixNet<D>& W, int& most_t, int& most_g) {
  constexpr int RS = D + 4;
  const double* kk = a.dv.params + seq * a.dv.pstride;
  const int4* tt = reinterpret_cast<const int4*>(a.dv.topo + seq * a.dv.tstride);
  const int32_t* aoff = a.adj_off + (a.adj_stride ? seq : 0) * (D + 1);
  const int32_t* ae = a.adj_e + (a.adj_stride ? seq : 0) * a.adj_stride;
  int nt = 0, ng = 0;
  if (l32 < D) {
    const int e0 = __ldg(aoff + l32), e1 = __ldg(aoff + l32 + 1);
    auto put = [&](float k, int j, int m) {  // stable insertion by the place in G
      const uint32_t at = 4u * (uint32_t)(l32 * RS + j);
      int e = nt++;
      for (; e > 0 && (W.term[e - 1][l32].y & 0xffffu) > at; --e)
        W.term[e][l32] = W.term[e - 1][l32];
      W.term[e][l32] = make_uint2(__float_as_uint(k), at | (uint32_t)m << 18);
    };
    for (; ng < kMixList && e0 + ng < e1; ++ng) {
      const int code = __ldg(ae + e0 + ng), r = code & 0xffff;
      const int4 q = __ldg(tt + r);
      // (a reaction naming no species changes nothing here; the set-up kernel reports it)
      const bool ok = q.x >= 0 && q.x < D && q.y >= -1 && q.y < D;
      const float nu = ok ? (float)((code >> 16) - 4) : 0.f;
      W.run[ng][l32] = __float_as_uint(nu) | (uint32_t)(r < kMixReact ? r : kMixReact);
      if (ok) {
        const float k = nu * d2f_trunc(__ldg(kk + r));
        put(k, q.x, q.y < 0 ? D : q.y);      // d rate / d c_i1
        if (q.y >= 0) put(k, q.y, q.x);      // d rate / d c_i2
      }
    }
    for (int e = 0; e < nt; ++e)
      if (e + 1 == nt || (W.term[e + 1][l32].y & 0xffffu) != (W.term[e][l32].y & 0xffffu))
        W.term[e][l32].y |= 1u;
  }
  // (whole batches of kMixBatch)
  most_t = (__reduce_max_sync(0xffffffffu, nt) + kMixBatch - 1) / kMixBatch * kMixBatch;
  most_g = (__reduce_max_sync(0xffffffffu, ng) + kMixBatch - 1) / kMixBatch * kMixBatch;
  if (l32 < D) {
    for (int e = nt; e < most_t; ++e) W.term[e][l32] = make_uint2(0u, (uint32_t)D << 18);
    for (int e = ng; e < most_g; ++e) W.run[e][l32] = (uint32_t)kMixReact;
  }
  for (int r = l32; r < R; r += 32) {
    const int4 q = __ldg(tt + r);
    const double k = __ldg(kk + r);
    W.react[r] = (q.x >= 0 && q.x < D ? (uint32_t)q.x : (uint32_t)D) |
                 (q.y >= 0 && q.y < D ? (uint32_t)q.y : (uint32_t)D) << 8;
    W.kd[r] = k;
    W.kf[r] = d2f_trunc(k);
  }
}

// One row, with the dynamics' value path in V = float or double (see mixed_row). `tail`: some
// species of the network has reactions beyond its list.
template <class V, int D, bool RK4>
__device__ __forceinline__ void mixed_row_cols(const MixedLinArgs& a, bool valid, int64_t seq,
                                               int64_t row, int lane, const MixNet<D>& W,
                                               MixRow<D>& S, int R, int most_t, int most_g,
                                               bool tail, const double (&spd)[2],
                                               const double (&sc)[2], float& mx, float& sq,
                                               unsigned long long& key) {
  constexpr bool F64 = sizeof(V) == 8;
  constexpr int LPR = D / 2, RS = D + 4;  // G's rows padded by 16 bytes
  V* rate = reinterpret_cast<V*>(S.rate);
  const V h = F64 ? (V)a.dv.dt : (V)a.dt_f;
  const float hf = a.dt_f;
  V prev[2], c[2], acc[2];
  float2 K[D], Kacc[D];
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    prev[x] = F64 ? (V)spd[x] : (V)d2f_trunc(spd[x]);
    c[x] = prev[x];
    acc[x] = V(0);
  }
#pragma unroll
  for (int i = 0; i < D; ++i) Kacc[i] = make_float2(0.f, 0.f);
  constexpr int NST = RK4 ? 4 : 1;
#pragma unroll 1
  for (int stage = 0; stage < NST; ++stage) {
    // RK4 tableau: stage derivative weights (1, 2, 2, 1), stage offsets (h/2, h/2, h)
    const float cK = stage == 3 ? hf : 0.5f * hf;
    const V w = (stage == 1 || stage == 2) ? V(2) : V(1);
    const float wf = (stage == 1 || stage == 2) ? 2.f : 1.f;
    if constexpr (F64) {
      *reinterpret_cast<float2*>(&S.c[2 * lane]) =
          make_float2(d2f_trunc((double)c[0]), d2f_trunc((double)c[1]));
      *reinterpret_cast<double2*>(&S.cd[2 * lane]) = make_double2((double)c[0], (double)c[1]);
    } else {
      *reinterpret_cast<float2*>(&S.c[2 * lane]) = make_float2((float)c[0], (float)c[1]);
    }
    if (tail) {  // entries that only unlisted reactions name
      for (int j = 0; j < RS / 2; ++j)
        *reinterpret_cast<float4*>(&S.G[2 * lane * RS + 4 * j]) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncwarp();
    // (loads of a batch first: the stores between them could alias)
    for (int r0 = lane; r0 < R; r0 += 4 * LPR) {
      V v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = r0 + u * LPR < R ? r0 + u * LPR : lane;
        const uint32_t q = W.react[r];
        if constexpr (F64) v[u] = W.kd[r] * S.cd[q & 0xffu] * S.cd[q >> 8];
        else v[u] = W.kf[r] * S.c[q & 0xffu] * S.c[q >> 8];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (r0 + u * LPR < R) rate[r0 + u * LPR] = v[u];
    }
    char* Gb = reinterpret_cast<char*>(S.G);
    const char* cb = reinterpret_cast<const char*>(S.c);
    float ga = 0.f, gb = 0.f;
    for (int e = 0; e < most_t; e += kMixBatch) {
      uint4 q[kMixBatch];
      float va[kMixBatch], vb[kMixBatch];
#pragma unroll
      for (int u = 0; u < kMixBatch; ++u)
        q[u] = *reinterpret_cast<const uint4*>(&W.term[e + u][2 * lane]);
#pragma unroll
      for (int u = 0; u < kMixBatch; ++u) {
        va[u] = __fmul_rn(__uint_as_float(q[u].x),
                          *reinterpret_cast<const float*>(cb + (q[u].y >> 16)));
        vb[u] = __fmul_rn(__uint_as_float(q[u].z),
                          *reinterpret_cast<const float*>(cb + (q[u].w >> 16)));
      }
#pragma unroll
      for (int u = 0; u < kMixBatch; ++u) {
        ga = __fadd_rn(ga, va[u]);
        gb = __fadd_rn(gb, vb[u]);
        if (q[u].y & 1u) *reinterpret_cast<float*>(Gb + (q[u].y & 0xfffcu)) = ga;
        if (q[u].w & 1u) *reinterpret_cast<float*>(Gb + (q[u].w & 0xfffcu)) = gb;
        ga = q[u].y & 1u ? 0.f : ga;
        gb = q[u].w & 1u ? 0.f : gb;
      }
    }
    __syncwarp();  // the rates
    V g[2] = {V(0), V(0)};
    for (int e = 0; e < most_g; e += kMixBatch) {
      uint2 q[kMixBatch];
      V ra[kMixBatch], rb[kMixBatch];
#pragma unroll
      for (int u = 0; u < kMixBatch; ++u) {
        q[u] = *reinterpret_cast<const uint2*>(&W.run[e + u][2 * lane]);
        ra[u] = rate[q[u].x & 0x7fu];
        rb[u] = rate[q[u].y & 0x7fu];
      }
#pragma unroll
      for (int u = 0; u < kMixBatch; ++u) {
        g[0] += mix_nu(q[u].x, V(0)) * ra[u];
        g[1] += mix_nu(q[u].y, V(0)) * rb[u];
      }
    }
    if (tail) {
      const int32_t* aoff = a.adj_off + (a.adj_stride ? seq : 0) * (D + 1) + 2 * lane;
      const int32_t* ae = a.adj_e + (a.adj_stride ? seq : 0) * a.adj_stride;
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        float* Gi = &S.G[(2 * lane + x) * RS];
        V gx = g[x];
        const int e1 = __ldg(aoff + x + 1);
        for (int e = __ldg(aoff + x) + kMixList; e < e1; ++e) {
          const int code = __ldg(ae + e), r = code & 0xffff;
          if (r >= R) continue;
          const uint32_t q = W.react[r];
          const float nu = (float)((code >> 16) - 4);
          const uint32_t i1 = q & 0xffu, i2 = q >> 8;
          gx += mix_nu(__float_as_uint(nu), V(0)) * rate[r];
          if (i1 < D) Gi[i1] += nu * (W.kf[r] * S.c[i2]);
          if (i2 < D) Gi[i2] += nu * (W.kf[r] * S.c[i1]);
        }
        g[x] = gx;
      }
      __syncwarp();
    }
    if (stage == 0) {
#pragma unroll
      for (int i = 0; i < D; ++i) K[i] = *reinterpret_cast<const float2*>(&S.G[i * RS + 2 * lane]);
    } else {
      float2 Y[D];
      const float2 cK2 = make_float2(cK, cK);
      constexpr int IB = 4;  // rows in flight: independent chains for the FMA latency
#pragma unroll
      for (int i = 0; i < D; i += IB) {
#pragma unroll
        for (int x = 0; x < IB; ++x)
          Y[i + x] = *reinterpret_cast<const float2*>(&S.G[(i + x) * RS + 2 * lane]);
#pragma unroll
        for (int m = 0; m < D; m += 4) {
          float2 q0[IB], q1[IB];
#pragma unroll
          for (int x = 0; x < IB; ++x) {
            const float4 q = *reinterpret_cast<const float4*>(&S.G[(i + x) * RS + m]);
            q0[x] = __fmul2_rn(make_float2(q.x, q.y), cK2);
            q1[x] = __fmul2_rn(make_float2(q.z, q.w), cK2);
          }
#pragma unroll
          for (int x = 0; x < IB; ++x)
            Y[i + x] = __ffma2_rn(make_float2(q0[x].x, q0[x].x), K[m], Y[i + x]);
#pragma unroll
          for (int x = 0; x < IB; ++x)
            Y[i + x] = __ffma2_rn(make_float2(q0[x].y, q0[x].y), K[m + 1], Y[i + x]);
#pragma unroll
          for (int x = 0; x < IB; ++x)
            Y[i + x] = __ffma2_rn(make_float2(q1[x].x, q1[x].x), K[m + 2], Y[i + x]);
#pragma unroll
          for (int x = 0; x < IB; ++x)
            Y[i + x] = __ffma2_rn(make_float2(q1[x].y, q1[x].y), K[m + 3], Y[i + x]);
        }
      }
#pragma unroll
      for (int i = 0; i < D; ++i) K[i] = Y[i];
    }
    const V cs = stage == 2 ? h : V(0.5) * h;
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      acc[x] += w * g[x];
      c[x] = prev[x] + cs * g[x];
    }
#pragma unroll
    for (int i = 0; i < D; ++i) Kacc[i] = __ffma2_rn(make_float2(wf, wf), K[i], Kacc[i]);
    __syncwarp();  // the next stage or row overwrites G, the rates and the concentrations
  }
  if (!valid) return;
  const V hw = RK4 ? h / V(6) : h;
  float rf[2];
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const V F = prev[x] + hw * acc[x];
    const float scf = d2f_trunc(sc[x]);
    if constexpr (F64) rf[x] = d2f_trunc(sc[x] - (double)F);
    else rf[x] = scf - (float)F;
    const float sabs = fabsf(scf);
    float m = fabsf(rf[x]) / (sabs > 1.f ? sabs : 1.f);
    if (!F64 && !(m != m)) m = m > kMixedFloor ? m : kMixedFloor;
    mx = nanmaxf(mx, m);
    sq += rf[x] * rf[x];
    if (!(m <= a.tol_f) && key == 0ull) key = bad_key(true, row - __ldg(a.bt.offsets + seq));
  }
  const float scale = a.scale_f;
  const float hwf = RK4 ? hf / 6.f : hf;
  // E = A - I with A = I + hw Kacc (scaled by (1 - k) under scale-ELK: E = s A - I)
  __nv_bfloat16* Eo = a.E + row * (int64_t)(D * D) + 2 * lane;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const float x0 = scale * hwf * Kacc[i].x + (i == 2 * lane ? scale - 1.f : 0.f);
    const float x1 = scale * hwf * Kacc[i].y + (i == 2 * lane + 1 ? scale - 1.f : 0.f);
    *reinterpret_cast<__nv_bfloat162*>(Eo + i * D) = __floats2bfloat162_rn(x0, x1);
  }
  *reinterpret_cast<float2*>(a.b + row * D + 2 * lane) = make_float2(-rf[0], -rf[1]);
}

template <int D>
constexpr size_t kMixSmem = 4 * sizeof(MixNet<D>) + 256 / D * sizeof(MixRow<D>);

template <bool RK4>
__global__ void __launch_bounds__(128, 3) k_lin_ma_mixed_cols(MixedLinArgs a) {
  constexpr int D = 16, LPR = D / 2;
  extern __shared__ __align__(16) unsigned char mix_smem[];
  MixNet<D>& W = reinterpret_cast<MixNet<D>*>(mix_smem)[threadIdx.x >> 5];
  MixRow<D>& S =
      reinterpret_cast<MixRow<D>*>(mix_smem + 4 * sizeof(MixNet<D>))[threadIdx.x / LPR];
  const int l32 = threadIdx.x & 31, lane = l32 % LPR, grp = l32 / LPR;
  const int64_t rows = a.bt.act_rows();
  const int64_t lo = (blockIdx.x * 4ll + (threadIdx.x >> 5)) * kMixRows;
  const int64_t hi = lo + kMixRows < rows ? lo + kMixRows : rows;
  const int R = a.dv.R < kMixReact ? a.dv.R : kMixReact;
  int64_t cur = -1;
  int most_t = 0, most_g = 0;
  bool tail = false, fast = true;
  float mx = 0.f, sq = 0.f;
  unsigned long long key = 0ull;  // first failing row (sliding window)
  if (lane == 0) {
    S.c[D] = 1.f;
    S.cd[D] = 1.0;
  }
  for (int64_t pos = lo; pos < hi;) {  // uniform over the warp
    int64_t seq, row;
    act_row(a.bt, pos + grp < hi ? pos + grp : hi - 1, seq, row);
    // the step's rows are those of its first row's sequence
    const int64_t sq0 = __shfl_sync(0xffffffffu, seq, 0);
    const bool valid = pos + grp < hi && seq == sq0;
    pos += __popc(__ballot_sync(0xffffffffu, valid)) / LPR;
    if (sq0 != cur) {
      if (cur >= 0) acc_resid_group<32>(a.acc, cur, mx, sq, key, l32, 0xffffffffu);
      cur = sq0;
      mx = 0.f;
      sq = 0.f;
      key = 0ull;
      fast = a.it == 0 || a.info[cur].max_resid > kMixedFastAbove;
      __syncwarp();
      mix_net<D>(a, cur, R, l32, W, most_t, most_g);
      const int32_t* aoff = a.adj_off + (a.adj_stride ? cur : 0) * (D + 1);
      tail = __any_sync(0xffffffffu,
                        l32 < D && __ldg(aoff + (l32 < D ? l32 : 0) + 1) -
                                           __ldg(aoff + (l32 < D ? l32 : 0)) > kMixList);
      for (int j = lane; j < D * (D + 4); j += LPR) S.G[j] = 0.f;
      if (lane == 0) {
        if (fast) reinterpret_cast<float*>(S.rate)[kMixReact] = 0.f;
        else S.rate[kMixReact] = 0.0;
      }
      __syncwarp();
    }
    const bool row_first = row == __ldg(a.bt.offsets + seq);
    double sp[2], sc[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      sp[x] = row_first ? a.s0[seq * D + 2 * lane + x] : a.s[(row - 1) * D + 2 * lane + x];
      sc[x] = a.s[row * D + 2 * lane + x];
    }
    if (fast)
      mixed_row_cols<float, D, RK4>(a, valid, cur, row, lane, W, S, R, most_t, most_g, tail, sp,
                                    sc, mx, sq, key);
    else
      mixed_row_cols<double, D, RK4>(a, valid, cur, row, lane, W, S, R, most_t, most_g, tail,
                                     sp, sc, mx, sq, key);
  }
  if (cur >= 0) acc_resid_group<32>(a.acc, cur, mx, sq, key, l32, 0xffffffffu);
}

// ---- linearisation, d = 32 and few rows: a lane per species -------------------------------
// d = 16 takes two columns per lane from kMixColsRows rows on: its lists cost more to build and its
// warps hold 32 rows, which fewer rows do not pay for. Six iterations, 24 reactions, a lane per
// species against two columns: 300 rows 0.61 / 1.10 ms, 10000 rows 0.95 / 1.30, 80000 rows 2.30 /
// 2.47, 160000 rows 3.94 / 3.49 (64 reactions: 0.69 / 1.56, 1.20 / 1.75, 3.37 / 3.85, 5.98 / 5.27).
constexpr int64_t kMixColsRows = 1 << 17;

// Two columns of K and of their sum take 128 registers at d = 32, which spills (255 registers,
// 1124 bytes): 0.8 M rows, 48 reactions take 7.2 ms that way and 6.7 with a lane per species,
// evaluated in float64 8.1 and 7.0. A group walks up to kMixLaneRows consecutive rows: reactions,
// rate constants and lists are loaded once per group and sequence, and the residual statistics
// flushed once.
constexpr int kMixLaneRows = 8;

template <int D>
struct MixLane {  // one per group
  // rows padded to D + 4 floats: 16-byte row accesses of eight lanes fall in distinct banks
  float G[D][D + 4], K[D][D + 4];
  double rate[kMixReact];               // floats use the first half in float32 mode
  float d1[kMixReact], d2[kMixReact];   // d rate / d c_i1, d c_i2
  uint32_t list[kMixList * D];
  float pad[D == 16 ? 16 : 4];          // the two groups of a warp in different banks
};

template <int D, bool RK4>
__global__ void __launch_bounds__(128) k_lin_ma_mixed_lane(MixedLinArgs a, int per) {
  constexpr int RPL = kMixReact / D;  // reactions per lane
  extern __shared__ __align__(16) unsigned char mix_smem[];
  MixLane<D>& S = reinterpret_cast<MixLane<D>*>(mix_smem)[threadIdx.x / D];
  const int lane = threadIdx.x % D;
  const unsigned gm = gmask_mixed<D>();
  const int64_t rows = a.bt.act_rows();
  const int64_t lo = (blockIdx.x * (int64_t)(128 / D) + threadIdx.x / D) * per;
  const int R = a.dv.R < kMixReact ? a.dv.R : kMixReact;
  int64_t cur = -1;
  const int4* tt = nullptr;
  const int32_t* ae = nullptr;
  int e0 = 0, e1 = 0;
  int4 q[RPL];
  double kd[RPL];
  float kf[RPL];
  bool fast = true;
  float mx = 0.f, sq = 0.f;
  unsigned long long key = 0ull;  // first failing row (sliding window)
  for (int64_t pos = lo; pos < lo + per && pos < rows; ++pos) {  // uniform over the group
    int64_t seq, row;
    act_row(a.bt, pos, seq, row);
    if (seq != cur) {
      if (cur >= 0) acc_resid_group<D>(a.acc, cur, mx, sq, key, lane, gm);
      cur = seq;
      mx = 0.f;
      sq = 0.f;
      key = 0ull;
      const double* kk = a.dv.params + seq * a.dv.pstride;
      tt = reinterpret_cast<const int4*>(a.dv.topo + seq * a.dv.tstride);
      const int32_t* aoff = a.adj_off + (a.adj_stride ? seq : 0) * (D + 1);
      ae = a.adj_e + (a.adj_stride ? seq : 0) * a.adj_stride;
      e0 = __ldg(aoff + lane);
      e1 = __ldg(aoff + lane + 1);
      mixed_list<D>(S.list, lane, tt, ae, e0, e1);  // (each lane reads only its own column)
#pragma unroll
      for (int k = 0; k < RPL; ++k) {
        const int r = k * D + lane;
        q[k] = __ldg(tt + (r < R ? r : 0));
        kd[k] = r < R ? __ldg(kk + r) : 0.0;
        kf[k] = d2f_trunc(kd[k]);
      }
      fast = a.it == 0 || a.info[seq].max_resid > kMixedFastAbove;
    }
    const double sp = row == __ldg(a.bt.offsets + seq) ? a.s0[seq * D + lane]
                                                      : a.s[(row - 1) * D + lane];
    const double sc = a.s[row * D + lane];
    __nv_bfloat16* Eo = a.E + row * (int64_t)(D * D);
    float* bo = a.b + row * D;
    if (fast)
      mixed_row<float, D, RK4, RPL>(a, true, row, lane, gm, sp, sc, q, kd, kf, R, tt, ae, e0, e1,
                                    S.list, S.G, S.K, reinterpret_cast<float*>(S.rate), S.d1,
                                    S.d2, mx, sq, seq, key, bo, Eo);
    else
      mixed_row<double, D, RK4, RPL>(a, true, row, lane, gm, sp, sc, q, kd, kf, R, tt, ae, e0, e1,
                                     S.list, S.G, S.K, S.rate, S.d1, S.d2, mx, sq, seq, key, bo,
                                     Eo);
  }
  if (cur >= 0) acc_resid_group<D>(a.acc, cur, mx, sq, key, lane, gm);
}

// Rows per group of d lanes: kMixLaneRows, fewer while the groups are less than 16 warps per
// scheduler, where a pass waits for one group's chain. Six iterations with 1, 2, 4, 8 rows, d = 32:
// 300 rows 1.87, 1.92, 2.07, 2.36 ms; 40000 rows 6.1, 6.0, 6.1, 6.1; 320000 rows 39.6, 37.9, 37.1,
// 36.6.
static int mix_lane_rows(int64_t rows, int d) {
  int n = kMixLaneRows;
  while (n > 1 && rows / n * d < (int64_t)kSchedulers * 32 * 16) n /= 2;
  return n;
}

template <bool RK4>
static cudaError_t lin_mixed_launch(const MixedLinArgs& a, cudaStream_t st) {
  static DeviceOnce cols, lane16, lane32;
  const int64_t rows = a.bt.act_rows();
  cudaError_t e;
  if (a.dv.d == 16 && rows >= kMixColsRows) {
    constexpr size_t smem = kMixSmem<16>;
    e = allow_smem(cols, k_lin_ma_mixed_cols<RK4>, smem);
    if (e != cudaSuccess) return e;
    k_lin_ma_mixed_cols<RK4><<<grid_for(rows, 4 * kMixRows), 128, smem, st>>>(a);
  } else if (a.dv.d == 16) {
    constexpr size_t smem = 8 * sizeof(MixLane<16>);
    e = allow_smem(lane16, k_lin_ma_mixed_lane<16, RK4>, smem);
    if (e != cudaSuccess) return e;
    const int per = mix_lane_rows(rows, 16);
    k_lin_ma_mixed_lane<16, RK4><<<grid_for(rows, 8 * per), 128, smem, st>>>(a, per);
  } else if (a.dv.d == 32) {
    constexpr size_t smem = 4 * sizeof(MixLane<32>);
    e = allow_smem(lane32, k_lin_ma_mixed_lane<32, RK4>, smem);
    if (e != cudaSuccess) return e;
    const int per = mix_lane_rows(rows, 32);
    k_lin_ma_mixed_lane<32, RK4><<<grid_for(rows, 4 * per), 128, smem, st>>>(a, per);
  } else {
    return cudaErrorInvalidValue;
  }
  note_launch();
  return cudaGetLastError();
}

// ---- mixed dense scan: lane j owns column j of P and entry j of the vectors ----------
template <int D>
__global__ void __launch_bounds__(128) k_mixed_chunk(MixedScanArgs a) {
  constexpr int G = 128 / D;
  const int grp = threadIdx.x / D, lane = threadIdx.x % D;
  const unsigned gm = gmask_mixed<D>();
  const int64_t ac = blockIdx.x * (int64_t)G + grp;
  const bool valid = ac < a.bt.act_chunks();
  int64_t seq = 0, c = 0, r0 = 0;
  int n = 0;
  if (valid) act_chunk(a.bt, ac, seq, c, r0, n);
  const bool need_P = valid && c != win_first(a.bt, seq);
  float Pc[D];
  float v = 0.f;
#pragma unroll
  for (int i = 0; i < D; ++i) Pc[i] = i == lane ? 1.f : 0.f;
  for (int t = 0; t < n; ++t) {
    const __nv_bfloat16* Et = a.E + (r0 + t) * (int64_t)(D * D);
    float nv = __ldg(a.b + (r0 + t) * D + lane) + v;
#pragma unroll
    for (int k = 0; k < D; ++k)
      nv += __bfloat162float(Et[lane * D + k]) * __shfl_sync(gm, v, k, D);
    v = nv;
    if (need_P) {
      float np[D];
#pragma unroll
      for (int i = 0; i < D; ++i) {
        float x = Pc[i];
#pragma unroll
        for (int k = 0; k < D; ++k) x += __bfloat162float(Et[i * D + k]) * Pc[k];
        np[i] = x;
      }
#pragma unroll
      for (int i = 0; i < D; ++i) Pc[i] = np[i];
    }
  }
  if (valid) {
    float* Po = a.aggP + c * (int64_t)(D * D);
#pragma unroll
    for (int i = 0; i < D; ++i) Po[i * D + lane] = Pc[i];
    a.aggv[c * D + lane] = v;
  }
}

// The aggregates are float32: the carry is the dense scans' (one or two levels).
static cudaError_t mixed_carry(const MixedScanArgs& m, cudaStream_t st) {
  DenseScanArgs<float> a{};
  a.bt = m.bt;
  a.d = m.d;
  a.aggP = m.aggP;
  a.aggv = m.aggv;
  a.cin = m.cin;
  a.segP = m.segP;
  a.segv = m.segv;
  a.segin = m.segin;
  a.max_chunks = m.max_chunks;
  return launch_dense_carry(a, st);
}

template <int D>
__global__ void __launch_bounds__(128) k_mixed_apply(MixedScanArgs a) {
  constexpr int G = 128 / D;
  const int grp = threadIdx.x / D, lane = threadIdx.x % D;
  const unsigned gm = gmask_mixed<D>();
  const int64_t ac = blockIdx.x * (int64_t)G + grp;
  const bool valid = ac < a.bt.act_chunks();
  int64_t seq = 0, c = 0, r0 = 0;
  int n = 0;
  if (valid) act_chunk(a.bt, ac, seq, c, r0, n);
  float x = valid ? a.cin[c * D + lane] : 0.f;
  for (int t = 0; t < n; ++t) {
    const int64_t row = r0 + t;
    const __nv_bfloat16* Et = a.E + row * (int64_t)(D * D) + lane * D;
    float y = __ldg(a.b + row * D + lane) + x;
#pragma unroll
    for (int k = 0; k < D; ++k) y += __bfloat162float(Et[k]) * __shfl_sync(gm, x, k, D);
    x = y;
    double* sp = a.s + row * D + lane;
    double nsv = *sp + (double)y;
    if (a.reset && !(nsv <= a.reset_thr && nsv >= -a.reset_thr)) nsv = 0.0;
    *sp = nsv;
  }
}

// ---- d = 16 on the tensor cores: one warp per chunk --------------------------------
// The chunk aggregate P <- (I + E_t) P is carried transposed, P^T <- P^T + P^T E_t^T, as
// one warp-level bf16 MMA pair (m16n8k16, float32 accumulate) per row: the float32
// accumulator fragment of P^T is exactly the A-operand fragment of the next product once
// rounded to bf16, and the B operand E_t^T is read straight from the row-major bf16 E_t
// (lane (g, t) of the warp, g = lane / 4, t = lane % 4, holds E[g][2t..2t+1],
// E[g][2t+8..2t+9] for columns 0-7 and the same entries of row g + 8 for columns 8-15).
// The vector part v <- v + E_t v + b_t stays in float32 on the same fragments: lane (g, t)
// forms the partial dot products of rows g and g + 8 over its four columns, a two-step
// shuffle sums the four lanes of row g, and each lane then fetches the four entries
// (2t, 2t+1, 2t+8, 2t+9) it needs for the next row.
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4],
                                               uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One row of the vector recurrence x <- x + E x + b on the fragments described above.
// lo / hi: x[g], x[g + 8] (same in the four lanes of row g); q[0..3]: x[2t], x[2t+1],
// x[2t+8], x[2t+9]. e0..e3: the lane's four words of E (rows g and g + 8).
__device__ __forceinline__ void frag_matvec16(uint32_t e0, uint32_t e1, uint32_t e2,
                                              uint32_t e3, float b_lo, float b_hi, float& lo,
                                              float& hi, float (&q)[4], int t) {
  float pl = bf_lo(e0) * q[0] + bf_hi(e0) * q[1] + bf_lo(e1) * q[2] + bf_hi(e1) * q[3];
  float ph = bf_lo(e2) * q[0] + bf_hi(e2) * q[1] + bf_lo(e3) * q[2] + bf_hi(e3) * q[3];
  pl += __shfl_xor_sync(0xffffffffu, pl, 1);
  ph += __shfl_xor_sync(0xffffffffu, ph, 1);
  pl += __shfl_xor_sync(0xffffffffu, pl, 2);
  ph += __shfl_xor_sync(0xffffffffu, ph, 2);
  lo = lo + pl + b_lo;
  hi = hi + ph + b_hi;
  q[0] = __shfl_sync(0xffffffffu, lo, 8 * t);
  q[1] = __shfl_sync(0xffffffffu, lo, 8 * t + 4);
  q[2] = __shfl_sync(0xffffffffu, hi, 8 * t);
  q[3] = __shfl_sync(0xffffffffu, hi, 8 * t + 4);
}

__global__ void __launch_bounds__(128) k_mixed_chunk_tc16(MixedScanArgs a) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int64_t ac = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
  if (ac >= a.bt.act_chunks()) return;  // whole warps
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, ac, seq, c, r0, n);
  const bool need_P = c != win_first(a.bt, seq);
  // P^T = I: fragment entries (g, 2t), (g, 2t+1), (g+8, 2t), (g+8, 2t+1) of the two tiles
  float p0[4] = {g == 2 * t ? 1.f : 0.f, g == 2 * t + 1 ? 1.f : 0.f, 0.f, 0.f};
  float p1[4] = {0.f, 0.f, g == 2 * t ? 1.f : 0.f, g == 2 * t + 1 ? 1.f : 0.f};
  float lo = 0.f, hi = 0.f, q[4] = {0.f, 0.f, 0.f, 0.f};
  for (int k = 0; k < n; ++k) {
    const int64_t row = r0 + k;
    const uint32_t* Ew = reinterpret_cast<const uint32_t*>(a.E + row * 256);
    const uint32_t e0 = __ldg(Ew + g * 8 + t), e1 = __ldg(Ew + g * 8 + t + 4);
    const uint32_t e2 = __ldg(Ew + (g + 8) * 8 + t), e3 = __ldg(Ew + (g + 8) * 8 + t + 4);
    const float b_lo = __ldg(a.b + row * 16 + g), b_hi = __ldg(a.b + row * 16 + g + 8);
    if (need_P) {
      const uint32_t A[4] = {pack_bf16x2(p0[0], p0[1]), pack_bf16x2(p0[2], p0[3]),
                             pack_bf16x2(p1[0], p1[1]), pack_bf16x2(p1[2], p1[3])};
      mma_bf16_16816(p0, A, e0, e1);
      mma_bf16_16816(p1, A, e2, e3);
    }
    frag_matvec16(e0, e1, e2, e3, b_lo, b_hi, lo, hi, q, t);
  }
  // P[i][j] = P^T[j][i]: tile 0 holds P^T[g][2t], P^T[g][2t+1], P^T[g+8][2t], P^T[g+8][2t+1]
  float* Po = a.aggP + c * 256;
  Po[(2 * t) * 16 + g] = p0[0];
  Po[(2 * t + 1) * 16 + g] = p0[1];
  Po[(2 * t) * 16 + g + 8] = p0[2];
  Po[(2 * t + 1) * 16 + g + 8] = p0[3];
  Po[(2 * t + 8) * 16 + g] = p1[0];
  Po[(2 * t + 9) * 16 + g] = p1[1];
  Po[(2 * t + 8) * 16 + g + 8] = p1[2];
  Po[(2 * t + 9) * 16 + g + 8] = p1[3];
  if (t == 0) {
    a.aggv[c * 16 + g] = lo;
    a.aggv[c * 16 + g + 8] = hi;
  }
}

// |x| >= 2^60 (about 1.15e18), Inf or NaN, from the exponent bits (no FP64 pipe)
__device__ __forceinline__ bool overflowed(double x) {
  return ((((unsigned)__double2hiint(x)) >> 20) & 0x7ffu) >= 1023u + 60u;
}

__global__ void __launch_bounds__(128) k_mixed_apply_tc16(MixedScanArgs a) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int64_t ac = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
  if (ac >= a.bt.act_chunks()) return;  // whole warps
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, ac, seq, c, r0, n);
  const float* ci = a.cin + c * 16;
  float lo = ci[g], hi = ci[g + 8];
  float q[4] = {ci[2 * t], ci[2 * t + 1], ci[2 * t + 8], ci[2 * t + 9]};
  for (int k = 0; k < n; ++k) {
    const int64_t row = r0 + k;
    const uint32_t* Ew = reinterpret_cast<const uint32_t*>(a.E + row * 256);
    const uint32_t e0 = __ldg(Ew + g * 8 + t), e1 = __ldg(Ew + g * 8 + t + 4);
    const uint32_t e2 = __ldg(Ew + (g + 8) * 8 + t), e3 = __ldg(Ew + (g + 8) * 8 + t + 4);
    const float b_lo = __ldg(a.b + row * 16 + g), b_hi = __ldg(a.b + row * 16 + g + 8);
    frag_matvec16(e0, e1, e2, e3, b_lo, b_hi, lo, hi, q, t);
    // s += Delta in float64; lanes t = 0 (row g) and t = 1 (row g + 8) write
    if (t < 2) {
      double* sp = a.s + row * 16 + g + 8 * t;
      double v = *sp + (double)(t == 0 ? lo : hi);
      if (a.reset && overflowed(v)) v = 0.0;
      *sp = v;
    }
  }
}

// ---- d = 16 without stored Jacobians: one warp per chunk ----------------------------
// The two half-warps linearise rows t and t + 1 of the chunk (16 lanes per row, as in
// k_lin_ma_mixed) into shared memory; the whole warp then folds them into the chunk
// aggregate (pass 1) or applies the correction to them (pass 2). The Jacobians never go to
// HBM here, so they are kept in float32 and the chunk product is formed to float32
// accuracy: P^T <- P^T + P^T E_t^T as warp-level tf32 MMAs (m16n8k8) with the three-term
// split x = x_hi + x_lo, the accumulator of P^T re-laid into the next A operand by quad
// shuffles (as in k_dense_chunk_mma32). Over horizons of 1e5 steps the rounding of E_t
// to bf16 compounds in the chunk products and slows Newton's convergence to linear on
// the stiffer networks; float32 Jacobians keep it fast. The vector part
// v <- v + E_t v + b_t: lane l forms half a row (row l mod 16, columns 8 (l / 16) ..) and
// the two halves meet by a shuffle.
constexpr int kRcWarps = 4;
constexpr int kRcRmax = 64;
constexpr int kRcES = 20;  // float32 E rows padded: the fragment reads hit distinct banks

struct RcSmem {
  float G[2][16][20];
  float K[2][17][20];
  double rate[2][kRcRmax];
  float d1[2][kRcRmax], d2[2][kRcRmax];
  float E[2][16 * kRcES];
  float b[2][16];
  uint32_t list[kMixList * 16];
  double old[16];  // pass 2: old state of the previous pair's second row
};

// per-lane network data of the sequence (reactions r = k * 16 + lane)
struct RcNet {
  int4 q[kRcRmax / 16];
  double kd[kRcRmax / 16];
  float kf[kRcRmax / 16];
  const int4* tt;
  const int32_t* ae;
  int e0, e1, R;
};

__device__ __forceinline__ void rc_net(const MixedLinArgs& a, int64_t seq, int lane,
                                       RcNet& n) {
  const double* kk = a.dv.params + seq * a.dv.pstride;
  n.tt = reinterpret_cast<const int4*>(a.dv.topo + seq * a.dv.tstride);
  const int32_t* aoff = a.adj_off + (a.adj_stride ? seq : 0) * 17;
  n.ae = a.adj_e + (a.adj_stride ? seq : 0) * a.adj_stride;
  n.e0 = __ldg(aoff + lane);
  n.e1 = __ldg(aoff + lane + 1);
  n.R = a.dv.R < kRcRmax ? a.dv.R : kRcRmax;
#pragma unroll
  for (int k = 0; k < kRcRmax / 16; ++k) {
    const int r = k * 16 + lane;
    n.q[k] = __ldg(n.tt + (r < n.R ? r : 0));
    n.kd[k] = r < n.R ? __ldg(kk + r) : 0.0;
    n.kf[k] = d2f_trunc(n.kd[k]);
  }
}

// linearise one row into the half-warp's shared buffers (float32 E, b): value path per
// `fast`
template <bool RK4>
__device__ __forceinline__ void rc_row(const MixedLinArgs& a, bool fast, bool valid,
                                       int64_t row, int half, int lane, unsigned gm,
                                       double sp, double sc, const RcNet& n, RcSmem& S,
                                       float& mx, float& sq, int64_t seq,
                                       unsigned long long& key) {
  if (fast)
    mixed_row<float, 16, RK4, kRcRmax / 16>(
        a, valid, row, lane, gm, sp, sc, n.q, n.kd, n.kf, n.R, n.tt, n.ae, n.e0, n.e1,
        S.list, S.G[half], S.K[half], reinterpret_cast<float*>(S.rate[half]), S.d1[half],
        S.d2[half], mx, sq, seq, key, S.b[half], S.E[half]);
  else
    mixed_row<double, 16, RK4, kRcRmax / 16>(
        a, valid, row, lane, gm, sp, sc, n.q, n.kd, n.kf, n.R, n.tt, n.ae, n.e0, n.e1,
        S.list, S.G[half], S.K[half], S.rate[half], S.d1[half], S.d2[half], mx, sq, seq, key,
        S.b[half], S.E[half]);
}

// P^T <- P^T + P^T E^T for the warp's 16 x 16 accumulator acc[n-tile][4] (lane (g, t):
// rows g, g + 8, columns 8 j + 2 t, + 1), three-term tf32 split
__device__ __forceinline__ void rc_compose(float (&acc)[2][4], const float* E, int g, int t,
                                           int lane) {
  const int qsrc = (lane & ~3) + (t >> 1);
  const bool odd = t & 1;
  uint32_t ah[2][4], al[2][4];
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
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
  for (int j = 0; j < 2; ++j) {
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
      // B[k][n] = E^T[k][n] = E[n][k]: n = 8 j + g, k = 8 kk + t (+ 4)
      const float bx0 = E[(8 * j + g) * kRcES + 8 * kk + t];
      const float bx1 = E[(8 * j + g) * kRcES + 8 * kk + t + 4];
      const uint32_t bh0 = tc::tf32_rna(bx0), bh1 = tc::tf32_rna(bx1);
      const uint32_t bl0 = tc::tf32_rna(bx0 - __uint_as_float(bh0));
      const uint32_t bl1 = tc::tf32_rna(bx1 - __uint_as_float(bh1));
      tc::mma_1688_tf32(acc[j], al[kk], bh0, bh1);
      tc::mma_1688_tf32(acc[j], ah[kk], bl0, bl1);
      tc::mma_1688_tf32(acc[j], ah[kk], bh0, bh1);
    }
  }
}

// v <- v + E v + b with lane l holding v[l mod 16]; returns the new v[l mod 16]
__device__ __forceinline__ float rc_matvec(float v, const float* E, const float* b,
                                           int lane) {
  const int i = lane & 15, c = lane >> 4;
  float part = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k)
    part += E[i * kRcES + 8 * c + k] * __shfl_sync(0xffffffffu, v, 8 * c + k);
  part += __shfl_xor_sync(0xffffffffu, part, 16);
  return v + part + b[i];
}

template <bool RK4>
__global__ void __launch_bounds__(32 * kRcWarps) k_mixed_lin_agg16(MixedRcArgs r) {
  __shared__ __align__(16) RcSmem smem[kRcWarps];
  const MixedLinArgs& a = r.lin;
  const int warp = threadIdx.x >> 5, l32 = threadIdx.x & 31;
  const int half = l32 >> 4, lane = l32 & 15, g = l32 >> 2, tq = l32 & 3;
  const unsigned gm = gmask_mixed<16>();
  const int64_t ac = blockIdx.x * (int64_t)kRcWarps + warp;
  if (ac >= a.bt.act_chunks()) return;  // whole warps
  RcSmem& S = smem[warp];
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, ac, seq, c, r0, n);
  const int64_t base = __ldg(a.bt.offsets + seq);
  RcNet net;
  rc_net(a, seq, lane, net);
  if (half == 0) mixed_list<16>(S.list, lane, net.tt, net.ae, net.e0, net.e1);
  __syncwarp();
  const bool fast = a.it == 0 || a.info[seq].max_resid > kMixedFastAbove;
  if (l32 == 0) r.fastsel[seq] = fast ? 1 : 0;  // the same value from every chunk
  // the old state before the chunk, kept for the second pass (whose neighbouring chunk may
  // already have updated it)
  const double prev0 = r0 == base ? a.s0[seq * 16 + lane] : a.s[(r0 - 1) * 16 + lane];
  if (half == 0 && r0 > base) r.sbound[c * 16 + lane] = prev0;
  const bool need_P = c != win_first(a.bt, seq);
  // P^T = I
  float acc[2][4];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int n0 = 8 * j + 2 * tq;
    acc[j][0] = g == n0 ? 1.f : 0.f;
    acc[j][1] = g == n0 + 1 ? 1.f : 0.f;
    acc[j][2] = g + 8 == n0 ? 1.f : 0.f;
    acc[j][3] = g + 8 == n0 + 1 ? 1.f : 0.f;
  }
  float v = 0.f;
  float mx = 0.f, sq = 0.f;
  unsigned long long key = 0ull;
  for (int t = 0; t < n; t += 2) {
    const int tr = t + half;
    const bool vld = tr < n;
    const int64_t row = r0 + (vld ? tr : 0);
    const double sp = tr == 0 ? prev0 : (vld ? a.s[(row - 1) * 16 + lane] : prev0);
    const double sc = vld ? a.s[row * 16 + lane] : prev0;
    rc_row<RK4>(a, fast, vld, row, half, lane, gm, sp, sc, net, S, mx, sq, seq, key);
    __syncwarp();
    for (int h = 0; h < 2 && t + h < n; ++h) {
      if (need_P) rc_compose(acc, S.E[h], g, tq, l32);
      v = rc_matvec(v, S.E[h], S.b[h], l32);
    }
    __syncwarp();
  }
  // P[i][j] = P^T[j][i]
  float* Po = r.aggP + c * 256;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int n0 = 8 * j + 2 * tq;
    Po[n0 * 16 + g] = acc[j][0];
    Po[(n0 + 1) * 16 + g] = acc[j][1];
    Po[n0 * 16 + g + 8] = acc[j][2];
    Po[(n0 + 1) * 16 + g + 8] = acc[j][3];
  }
  if (half == 0) r.aggv[c * 16 + lane] = v;
  acc_resid_f(a.acc, seq, true, mx, sq, key);
}

template <bool RK4>
__global__ void __launch_bounds__(32 * kRcWarps) k_mixed_apply_rc16(MixedRcArgs r) {
  __shared__ __align__(16) RcSmem smem[kRcWarps];
  const MixedLinArgs& a = r.lin;
  const int warp = threadIdx.x >> 5, l32 = threadIdx.x & 31;
  const int half = l32 >> 4, lane = l32 & 15;
  const unsigned gm = gmask_mixed<16>();
  const int64_t ac = blockIdx.x * (int64_t)kRcWarps + warp;
  if (ac >= a.bt.act_chunks()) return;  // whole warps
  RcSmem& S = smem[warp];
  int64_t seq, c, r0;
  int n;
  act_chunk(a.bt, ac, seq, c, r0, n);
  const int64_t base = __ldg(a.bt.offsets + seq);
  RcNet net;
  rc_net(a, seq, lane, net);
  if (half == 0) mixed_list<16>(S.list, lane, net.tt, net.ae, net.e0, net.e1);
  __syncwarp();
  const bool fast = r.fastsel[seq] != 0;
  const double prev0 = r0 == base ? a.s0[seq * 16 + lane] : r.sbound[c * 16 + lane];
  float x = r.cin[c * 16 + lane];  // Delta entering the chunk, entry lane mod 16
  float mx = 0.f, sq = 0.f;  // recomputed statistics, not reported again
  unsigned long long key = 0ull;
  double* s = const_cast<double*>(a.s);
  for (int t = 0; t < n; t += 2) {
    const int tr = t + half;
    const bool vld = tr < n;
    const int64_t row = r0 + (vld ? tr : 0);
    // old s_{t-1}: the chunk's saved boundary, the previous pair's second row (saved
    // before it was updated), or row t of this pair (not updated yet)
    double sp = prev0;
    if (tr > 0) sp = half == 0 ? S.old[lane] : (vld ? s[(row - 1) * 16 + lane] : prev0);
    const double sc = vld ? s[row * 16 + lane] : prev0;
    rc_row<RK4>(a, fast, vld, row, half, lane, gm, sp, sc, net, S, mx, sq, seq, key);
    __syncwarp();
    if (half == 1 && vld) S.old[lane] = sc;
    __syncwarp();
    for (int h = 0; h < 2 && t + h < n; ++h) {
      x = rc_matvec(x, S.E[h], S.b[h], l32);
      if (half == 0) {
        double* sp2 = s + (r0 + t + h) * 16 + lane;
        double nv = *sp2 + (double)x;
        if (r.reset && overflowed(nv)) nv = 0.0;
        *sp2 = nv;
      }
    }
    __syncwarp();
  }
}

cudaError_t launch_mixed_lin_agg(const MixedRcArgs& a, cudaStream_t st) {
  if (a.lin.bt.act_chunks() == 0) return cudaSuccess;
  if (a.lin.dv.d != 16) return cudaErrorInvalidValue;
  const unsigned g = grid_for(a.lin.bt.act_chunks(), kRcWarps);
  if (a.lin.dv.kind == DEER_F_MASSACTION_RK4) k_mixed_lin_agg16<true><<<g, 32 * kRcWarps, 0, st>>>(a);
  else k_mixed_lin_agg16<false><<<g, 32 * kRcWarps, 0, st>>>(a);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_mixed_apply_rc(const MixedRcArgs& a, const MixedScanArgs& carry,
                                  cudaStream_t st) {
  if (a.lin.bt.act_chunks() == 0) return cudaSuccess;
  if (a.lin.dv.d != 16) return cudaErrorInvalidValue;
  const cudaError_t e = mixed_carry(carry, st);
  if (e != cudaSuccess) return e;
  const unsigned g = grid_for(a.lin.bt.act_chunks(), kRcWarps);
  if (a.lin.dv.kind == DEER_F_MASSACTION_RK4) k_mixed_apply_rc16<true><<<g, 32 * kRcWarps, 0, st>>>(a);
  else k_mixed_apply_rc16<false><<<g, 32 * kRcWarps, 0, st>>>(a);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_lin_ma_mixed(const MixedLinArgs& a, cudaStream_t st) {
  if (a.bt.act_rows() == 0) return cudaSuccess;
  return a.dv.kind == DEER_F_MASSACTION_RK4 ? lin_mixed_launch<true>(a, st)
                                            : lin_mixed_launch<false>(a, st);
}

template <int D>
static cudaError_t mixed_launch(const MixedScanArgs& a, cudaStream_t st) {
  if constexpr (D == 16) {
    const unsigned gw = grid_for(a.bt.act_chunks(), 4);  // one warp per chunk
    if (a.tc_mode == 2) {
      const cudaError_t e = launch_mixed_chunk_tcgen05(a, st);
      if (e != cudaSuccess) return e;
    } else {
      k_mixed_chunk_tc16<<<gw, 128, 0, st>>>(a);
    }
    const cudaError_t e = mixed_carry(a, st);
    if (e != cudaSuccess) return e;
    k_mixed_apply_tc16<<<gw, 128, 0, st>>>(a);
  } else {
    const unsigned gc = grid_for(a.bt.act_chunks(), 128 / D);
    k_mixed_chunk<D><<<gc, 128, 0, st>>>(a);
    const cudaError_t e = mixed_carry(a, st);
    if (e != cudaSuccess) return e;
    k_mixed_apply<D><<<gc, 128, 0, st>>>(a);
  }
  note_launch(2);
  return cudaGetLastError();
}

cudaError_t launch_dense_scan_mixed(const MixedScanArgs& a, cudaStream_t st) {
  if (a.bt.act_rows() == 0) return cudaSuccess;
  if (a.d == 16) return mixed_launch<16>(a, st);
  if (a.d == 32) return mixed_launch<32>(a, st);
  return cudaErrorInvalidValue;
}

}  // namespace deer
