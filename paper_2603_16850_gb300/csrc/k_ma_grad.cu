// Rate-constant gradient of the mass-action kinetics at the adjoint, d = 16 and 32: lane
// groups instead of one thread per row, whose stage states and cotangents (9 d values) live
// in local memory and whose every reaction ends in a warp reduction and an atomic. 2.1 M rows,
// d = 32, 48 reactions, float32: 3.70 -> 2.04 ms. (d = 8 stays with a thread per row, k_lin.cu:
// 290 us against 480 for 1.05 M rows; its arrays are short.)
#include "kernels.h"

namespace deer {
namespace {

template <int D>
__device__ __forceinline__ unsigned seq_mask() {
  if constexpr (D == 32) return 0xffffffffu;
  return ((1u << D) - 1u) << (threadIdx.x & 31 & ~(D - 1));
}

__device__ __forceinline__ bool reaction_ok(const int4& q, int d) {
  return q.x >= 0 && q.x < d && q.z >= 0 && q.z < d && q.y >= -1 && q.y < d && q.w >= -1 &&
         q.w < d;
}

// Reactions of the group's network, reaction r = k D + lane on this lane. Rows with species
// outside [0, d) are dropped (the set-up kernel reports them). RPL rounds hold up to RPL D <= 128 reactions.
template <class real, int D, int RPL>
__device__ __forceinline__ void load_reactions(const DynView<real>& dv, int64_t seq, int lane,
                                               int4 (&q)[RPL], real (&kr)[RPL]) {
  const int4* tt = reinterpret_cast<const int4*>(dv.topo + seq * dv.tstride);
  const real* kk = dv.params + seq * dv.pstride;
#pragma unroll
  for (int k = 0; k < RPL; ++k) {
    const int r = k * D + lane;
    q[k] = make_int4(0, -1, 0, -1);
    kr[k] = real(0);
    if (r < dv.R) {
      const int4 t = __ldg(tt + r);
      if (reaction_ok(t, D)) {
        q[k] = t;
        kr[k] = __ldg(kk + r);
      }
    }
  }
}

// This lane's species in a list of (reaction, mark) entries, 8 bits each (reaction < 128,
// mark in bit 7), four to a register: entries of reactants only (mark = second reactant
// slot) or of every change (mark = consumed). More than kList entries: n = -1, and the
// sums below walk every reaction instead.
constexpr int kList = 16;
struct SpeciesList {
  uint32_t w0, w1, w2, w3;
  int n, most;  // entries; the group's largest count, or -1
};

template <class real, int D, bool REACTANTS>
__device__ __forceinline__ SpeciesList species_list(const DynView<real>& dv, int64_t seq,
                                                    int lane, unsigned gm) {
  const int4* tt = reinterpret_cast<const int4*>(dv.topo + seq * dv.tstride);
  uint32_t w0 = 0u, w1 = 0u, w2 = 0u, w3 = 0u;
  int n = 0;
  auto push = [&](int r, int mark) {
    const uint32_t code = (uint32_t)(r | (mark << 7)) << (8 * (n & 3));
    w0 |= n < 4 ? code : 0u;
    w1 |= n >= 4 && n < 8 ? code : 0u;
    w2 |= n >= 8 && n < 12 ? code : 0u;
    w3 |= n >= 12 && n < 16 ? code : 0u;
    ++n;
  };
  for (int r = 0; r < dv.R; ++r) {
    const int4 t = __ldg(tt + r);
    if (!reaction_ok(t, D)) continue;
    if (t.x == lane) push(r, REACTANTS ? 0 : 1);
    if (t.y == lane) push(r, 1);
    if (!REACTANTS && t.z == lane) push(r, 0);
    if (!REACTANTS && t.w == lane) push(r, 0);
  }
  int m = n;
#pragma unroll
  for (int o = D / 2; o > 0; o >>= 1) {
    const int x = __shfl_xor_sync(gm, m, o, D);
    m = x > m ? x : m;
  }
  return SpeciesList{w0, w1, w2, w3, n, m <= kList ? m : -1};
}

// sum over the list of get(reaction, mark): four independent reads at a time
template <class real, class Get>
__device__ __forceinline__ real list_sum(const SpeciesList& L, Get get) {
  real x = real(0), y = real(0);
#pragma unroll
  for (int e = 0; e < kList; e += 4) {
    if (e >= L.most) break;  // uniform over the group
    const uint32_t w = e == 0 ? L.w0 : e == 4 ? L.w1 : e == 8 ? L.w2 : L.w3;
    real v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      v[k] = e + k < L.n ? get((w >> (8 * k)) & 127u, (w >> (8 * k + 7)) & 1u) : real(0);
    x += v[0] + v[1];
    y += v[2] + v[3];
  }
  return x + y;
}

// Rate-constant gradient dl/dk_r = sum_t lambda_t^T df_t/dk_r (s_{t-1}): reverse mode
// through the integrator's stages, a group of D lanes per `a.rows` consecutive rows of a sequence,
// lane i on species i and on reactions i, i + D, ... The group's sums stay in registers and
// reach dparams with one atomic per reaction and group.
template <class real, int D, bool RK4, int RPL>
__global__ void __launch_bounds__(128) k_ma_param_grad(MaGradArgs<real> a) {
  constexpr int G = 128 / D, NS = RK4 ? 4 : 1;
  __shared__ real sR[G][RPL * D][2];  // per reaction: its rate, or its pull on either reactant
  const int grp = threadIdx.x / D, lane = threadIdx.x % D;
  const unsigned gm = seq_mask<D>();
  const int64_t per = (a.T + a.rows - 1) / a.rows;
  const int64_t id = blockIdx.x * (int64_t)G + grp;
  if (id >= a.B * per) return;  // whole groups
  const int64_t seq = id / per, t0 = (id - seq * per) * a.rows;
  const int64_t t1 = t0 + a.rows < a.T ? t0 + a.rows : a.T;
  int4 q[RPL];
  real kr[RPL];
  load_reactions<real, D, RPL>(a.dv, seq, lane, q, kr);
  const SpeciesList Lc = species_list<real, D, false>(a.dv, seq, lane, gm);
  const SpeciesList Lr = species_list<real, D, true>(a.dv, seq, lane, gm);
  const int4* tt = reinterpret_cast<const int4*>(a.dv.topo + seq * a.dv.tstride);
  const real h = a.dv.dt;
  real (*R)[2] = sR[grp];
  real c1[NS][RPL], c2[NS][RPL], dk[RPL];
#pragma unroll
  for (int k = 0; k < RPL; ++k) dk[k] = real(0);
  // reactant concentrations of stage st from this lane's species value; with `want`, the
  // slope of this lane's species
  auto stage = [&](int st, real c, bool want) -> real {
#pragma unroll
    for (int k = 0; k < RPL; ++k) {
      c1[st][k] = __shfl_sync(gm, c, q[k].x, D);
      const real x = __shfl_sync(gm, c, q[k].y < 0 ? 0 : q[k].y, D);
      c2[st][k] = q[k].y < 0 ? real(1) : x;
      if (want) R[k * D + lane][0] = kr[k] * c1[st][k] * c2[st][k];
    }
    if (!want) return real(0);
    __syncwarp(gm);
    real g;
    if (Lc.most >= 0) {
      g = list_sum<real>(Lc, [&](unsigned r, unsigned neg) { return neg ? -R[r][0] : R[r][0]; });
    } else {
      g = real(0);
      for (int r = 0; r < a.dv.R; ++r) {
        const int4 t = __ldg(tt + r);
        if (!reaction_ok(t, D)) continue;
        const int nu = (lane == t.z) + (lane == t.w) - (lane == t.x) - (lane == t.y);
        if (nu != 0) g += real(nu) * R[r][0];
      }
    }
    __syncwarp(gm);
    return g;
  };
  // dk += phi (nu . u) for the cotangent u of stage st's slope; with `want`, G(c)^T u
  auto pull = [&](int st, real u, bool want) -> real {
#pragma unroll
    for (int k = 0; k < RPL; ++k) {
      real nu = __shfl_sync(gm, u, q[k].z, D) - __shfl_sync(gm, u, q[k].x, D);
      const real u2 = __shfl_sync(gm, u, q[k].y < 0 ? 0 : q[k].y, D);
      const real p2 = __shfl_sync(gm, u, q[k].w < 0 ? 0 : q[k].w, D);
      if (q[k].y >= 0) nu -= u2;
      if (q[k].w >= 0) nu += p2;
      dk[k] += c1[st][k] * c2[st][k] * nu;
      if (want) {
        const real w = kr[k] * nu;
        R[k * D + lane][0] = w * c2[st][k];
        R[k * D + lane][1] = w * c1[st][k];
      }
    }
    if (!want) return real(0);
    __syncwarp(gm);
    real b;
    if (Lr.most >= 0) {
      b = list_sum<real>(Lr, [&](unsigned r, unsigned slot) { return R[r][slot]; });
    } else {
      b = real(0);
      for (int r = 0; r < a.dv.R; ++r) {
        const int4 x = __ldg(tt + r);
        if (!reaction_ok(x, D)) continue;
        if (x.x == lane) b += R[r][0];
        if (x.y == lane) b += R[r][1];
      }
    }
    __syncwarp(gm);
    return b;
  };
  const real* s = a.s + (seq * a.T - 1) * D + lane;  // s[t D]: the state before row t
  const real* lam = a.lam + seq * a.T * D + lane;
  real c = t0 == 0 ? a.s0[seq * D + lane] : s[t0 * D];
  real l = lam[t0 * D];
  for (int64_t t = t0; t < t1; ++t) {
    const bool more = t + 1 < t1;
    const real cn = more ? s[(t + 1) * D] : real(0), ln = more ? lam[(t + 1) * D] : real(0);
    if constexpr (RK4) {
      const real ca = c + real(0.5) * h * stage(0, c, true);
      const real cb = c + real(0.5) * h * stage(1, ca, true);
      stage(3, c + h * stage(2, cb, true), false);
      const real b3 = pull(3, h / real(6) * l, true);
      const real b2 = pull(2, h / real(3) * l + h * b3, true);
      const real b1 = pull(1, h / real(3) * l + real(0.5) * h * b2, true);
      pull(0, h / real(6) * l + real(0.5) * h * b1, false);
    } else {
      stage(0, c, false);
      pull(0, h * l, false);
    }
    c = cn;
    l = ln;
  }
#pragma unroll
  for (int k = 0; k < RPL; ++k) {
    const int r = k * D + lane;
    if (r < a.dv.R) atomicAdd(a.dparams + seq * a.pstride + r, dk[k]);
  }
}

template <class real, int D, int RPL>
void param_grad_launch(const MaGradArgs<real>& a, cudaStream_t st) {
  const unsigned g = grid_for(a.B * ((a.T + a.rows - 1) / a.rows), 128 / D);
  if (a.dv.kind == DEER_F_MASSACTION_RK4) k_ma_param_grad<real, D, true, RPL><<<g, 128, 0, st>>>(a);
  else k_ma_param_grad<real, D, false, RPL><<<g, 128, 0, st>>>(a);
  note_launch();
}

template <class real, int D>
cudaError_t param_grad_rounds(const MaGradArgs<real>& a, cudaStream_t st) {
  if (a.dv.R <= D) param_grad_launch<real, D, 1>(a, st);
  else if (a.dv.R <= 2 * D) param_grad_launch<real, D, 2>(a, st);
  else if (a.dv.R <= 4 * D) param_grad_launch<real, D, 4>(a, st);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

}  // namespace

bool ma_param_grad_supported(int kind, int d, int R) {
  return (kind == DEER_F_MASSACTION_EULER || kind == DEER_F_MASSACTION_RK4) && R <= 4 * d &&
         (d == 16 || d == 32);
}

template <class real>
cudaError_t launch_ma_param_grad(const MaGradArgs<real>& a, cudaStream_t st) {
  if (a.B == 0 || a.T == 0) return cudaSuccess;
  MaGradArgs<real> b = a;
  // 64 rows per group (the reaction lists are built once per group), fewer while the batch
  // leaves the GPU short of eight warps per SM
  b.rows = 64;
  while (b.rows > 8 && a.B * a.T / b.rows * a.dv.d < kSMs * 8 * 32) b.rows /= 2;
  switch (a.dv.d) {
    case 16: return param_grad_rounds<real, 16>(b, st);
    case 32: return param_grad_rounds<real, 32>(b, st);
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t launch_ma_param_grad<float>(const MaGradArgs<float>&, cudaStream_t);
template cudaError_t launch_ma_param_grad<double>(const MaGradArgs<double>&, cudaStream_t);

}  // namespace deer
