// Coding of a pixel by a quad: four neighbouring lanes, lane q of the quad
// holding the mixture components k = q + 4 i (i < KI = ceil(K / 4)) in
// registers, eight pixels per warp.  The arithmetic of every component and of
// every table value is that of the whole-warp group of nlc_model.cuh (maxima
// are exact, sums are integer sums, everything else is per component), so
// both give the same tables bit for bit.
//
// Why quads: a wavefront step codes up to 128 pixels per CTA and its length
// is a chain of latencies (maximum, sum, weights, search rounds, posterior,
// three channels one after another).  Sixteen lanes per pixel need three
// passes over that chain for the 81 pixels that a CTA gets at the largest
// batches; quads take one pass, with a third of the warp-level instructions
// per pixel, because the reductions run over registers first and the search
// evaluates 4 x 3 boundaries per channel instead of 2 x 15.
#pragma once

#include "nlc_model.cuh"

namespace nlc {

// Number of pixels that one warp codes at once.
constexpr int kQuads = 8;

template <int KI>
struct QuadState {
  float lw[KI];  // running log weights of the lane's components
};

// Parameters of one channel's components.
template <int KI>
struct QuadChan {
  float m[KI];    // locations within +-2^100
  float c[KI];    // log2(e) / s
  float w[KI];    // weights 2^23, 0 below kWmin
  float inv[KI];  // 1 / s
  float ls[KI];   // log s
};

__device__ __forceinline__ float quad_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ uint32_t quad_isum(uint32_t v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// Log mixture weights: log pi_k = logit_k - LSE(logits) (see comp_init).
// P(p, i): output p (0 logit, 1..3 location, 4..6 log-scale, 7..9 coupling)
// of the lane's i-th component; components past K are skipped.
template <int KI, class Param>
__device__ __forceinline__ void quad_init(Param P, int K, int q, QuadState<KI>& s) {
  float mx = -INFINITY;
#pragma unroll
  for (int i = 0; i < KI; i++) {
    s.lw[i] = q + 4 * i < K ? no_nan(P(0, i)) : -INFINITY;
    mx = fmaxf(mx, s.lw[i]);
  }
  mx = quad_max(mx);
  uint32_t E = 0;
#pragma unroll
  for (int i = 0; i < KI; i++)
    if (q + 4 * i < K) E += fix23(exp_f(__fsub_rn(s.lw[i], mx)));
  const uint32_t S = quad_isum(E);
  const float lse = __fadd_rn(mx, __fsub_rn(log_f((float)S), kLn2x23));
#pragma unroll
  for (int i = 0; i < KI; i++) s.lw[i] = __fsub_rn(s.lw[i], lse);
}

// Channel CH (compile-time) of the pixel, given the decoded r, g (see
// channel_setup: the same weights, locations and cut-off).
template <int CH, int KI, class Param>
__device__ __forceinline__ void quad_channel(Param P, int K, int q, const QuadState<KI>& s, int r,
                                             int g, QuadChan<KI>& o) {
  float wf = kFixOne;
  if (CH == 0) {
#pragma unroll
    for (int i = 0; i < KI; i++) o.w[i] = __fmul_rn(fminf(exp_f(s.lw[i]), 1.f), kFixOne);
  } else {
    float mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < KI; i++)
      if (q + 4 * i < K) mx = fmaxf(mx, no_nan(s.lw[i]));
    mx = quad_max(mx);
    uint32_t E[KI], Es = 0;
#pragma unroll
    for (int i = 0; i < KI; i++) {
      E[i] = q + 4 * i < K ? fix23(exp_f(__fsub_rn(no_nan(s.lw[i]), mx))) : 0u;
      Es += E[i];
    }
    wf = __fmul_rn(kFixOne, rcp_approx((float)quad_isum(Es)));
#pragma unroll
    for (int i = 0; i < KI; i++) o.w[i] = fminf(__fmul_rn((float)E[i], wf), kFixOne);
  }
  const float xr = xval_f(r), xg = xval_f(g);
#pragma unroll
  for (int i = 0; i < KI; i++) {
    const bool in = q + 4 * i < K;
    float m = 0.f, ls = 0.f;
    if (in) {
      m = P(1 + CH, i);
      if (CH == 1) m = __fadd_rn(m, __fmul_rn(tanh_f(P(7, i)), xr));
      if (CH == 2)
        m = __fadd_rn(__fadd_rn(m, __fmul_rn(tanh_f(P(8, i)), xr)), __fmul_rn(tanh_f(P(9, i)), xg));
      m = fminf(fmaxf(m, -kMMax), kMMax);
      ls = fmaxf(P(4 + CH, i), -7.f);
    }
    o.m[i] = m;
    o.ls[i] = ls;
    o.inv[i] = exp_f(-ls);
    o.c[i] = __fmul_rn(o.inv[i], kLog2e);
    if (!(in && o.w[i] >= kWmin * kFixOne)) o.w[i] = 0.f;  // adds only zero terms
  }
}

// Fixed-point F at boundary value e over the lane's components.
template <int KI>
__device__ __forceinline__ uint32_t quad_fix(const QuadChan<KI>& o, float e) {
  uint32_t F = 0;
#pragma unroll
  for (int i = 0; i < KI; i++) F += cdf_term(e, make_float4(o.m[i], o.c[i], o.w[i], 0.f));
  return F;
}

// Posterior update after channel value v.
template <int KI>
__device__ __forceinline__ void quad_observe(const QuadChan<KI>& o, int K, int q, int v,
                                             QuadState<KI>& s) {
#pragma unroll
  for (int i = 0; i < KI; i++)
    if (q + 4 * i < K)
      s.lw[i] = __fadd_rn(s.lw[i],
                          log_bin_mass_f(o.m[i], o.inv[i], bin_log_width(o.ls[i], o.inv[i]), v));
}

// Symbol search: s with cum_s <= slot < cum_{s+1}, and both values.  Four
// rounds of base 4: every lane sums its components' terms at the round's
// three inner boundaries, the partial sums are exchanged so that lane j holds
// F of boundary j, and the quad counts the boundaries at or below the slot.
// (Base 4 needs the fewest terms of the splits of 256 whose rounds fit a
// quad: 36 per channel and lane at K = 10, against 51 for 8 x 8 x 4 and 90
// for 16 x 16.)
template <int KI>
__device__ __forceinline__ int quad_search(const QuadChan<KI>& o, uint32_t slot, int q,
                                           uint32_t& c0, uint32_t& c1) {
  const unsigned full = 0xffffffffu;
  const int shift = threadIdx.x & 28;
  const bool h2 = (q & 2) != 0, h1 = (q & 1) != 0;
  int a = 0;
  uint32_t lo = 0u, hi = 65536u;
#pragma unroll
  for (int len = 64; len > 0; len >>= 2) {
    uint32_t f0 = quad_fix(o, edge_f(a + len));
    uint32_t f1 = quad_fix(o, edge_f(a + 2 * len));
    uint32_t f2 = quad_fix(o, edge_f(a + 3 * len));
    // lanes 0, 1 collect f0, f1; lanes 2, 3 collect f2, (none)
    const uint32_t r0 = __shfl_xor_sync(full, h2 ? f0 : f2, 2);
    const uint32_t r1 = __shfl_xor_sync(full, f1, 2);
    const uint32_t k0 = (h2 ? f2 : f0) + r0;
    const uint32_t k1 = f1 + r1;
    const uint32_t r2 = __shfl_xor_sync(full, h1 ? k0 : k1, 1);
    const uint32_t F = (h1 ? k1 : k0) + r2;
    const int b = a + len * (q + 1);
    const uint32_t u = q < 3 ? cum_fix(F, b) : hi;
    const unsigned bal = __ballot_sync(full, u <= slot) >> shift;
    const int c = __popc(bal & 7u);
    const uint32_t nlo = __shfl_sync(full, u, c > 0 ? c - 1 : 0, 4);
    hi = __shfl_sync(full, u, c, 4);
    lo = c > 0 ? nlo : lo;
    a += c * len;
  }
  c0 = lo;
  c1 = hi;
  return a;
}

// cum_v and cum_{v+1} of the channel (the encoder's pair).
template <int KI>
__device__ __forceinline__ void quad_pair(const QuadChan<KI>& o, int v, uint32_t& c0, uint32_t& c1) {
  const uint32_t F0 = quad_isum(quad_fix(o, edge_f(v)));
  const uint32_t F1 = quad_isum(quad_fix(o, edge_f(v + 1)));
  c0 = cum_fix(F0, v);
  c1 = cum_fix(F1, v + 1);
}

// Model code length: adds log P(v[CH]) of channel CH to the components'
// running log-likelihoods l (the locations are not bounded here).
template <int CH, int KI, class Param>
__device__ __forceinline__ void quad_loglik(Param P, int K, int q, const int (&v)[3],
                                            float (&l)[KI]) {
  const float xr = xval_f(v[0]), xg = xval_f(v[1]);
#pragma unroll
  for (int i = 0; i < KI; i++) {
    if (q + 4 * i >= K) continue;
    float m = P(1 + CH, i);
    if (CH == 1) m = __fadd_rn(m, __fmul_rn(tanh_f(P(7, i)), xr));
    if (CH == 2)
      m = __fadd_rn(__fadd_rn(m, __fmul_rn(tanh_f(P(8, i)), xr)), __fmul_rn(tanh_f(P(9, i)), xg));
    const float ls = fmaxf(P(4 + CH, i), -7.f), inv = exp_f(-ls);
    l[i] = __fadd_rn(l[i], log_bin_mass_f(m, inv, bin_log_width(ls, inv), v[CH]));
  }
}

// -log2 sum_k e^{l_k}; the sum pairs components 8, then 4, 2, 1 apart (the
// butterfly of a 16-lane group with one component per lane).
template <int KI>
__device__ __forceinline__ float quad_bits(const float (&l)[KI], int K, int q) {
  float mx = -INFINITY;
#pragma unroll
  for (int i = 0; i < KI; i++)
    if (q + 4 * i < K) mx = fmaxf(mx, l[i]);
  mx = quad_max(mx);
  float e[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int i = 0; i < KI; i++)
    if (q + 4 * i < K) e[i] = expf(__fsub_rn(l[i], mx));
  float s = __fadd_rn(__fadd_rn(e[0], e[2]), __fadd_rn(e[1], e[3]));
  s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, 2));
  s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, 1));
  return -__fadd_rn(mx, logf(s)) * 1.4426950408889634f;
}

}  // namespace nlc
