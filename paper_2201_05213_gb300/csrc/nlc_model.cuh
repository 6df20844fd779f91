// Per-tile pipeline of the local autoregressive model (device code):
//   gather of the causal context (Eq. 3) -> local network (Section 2.1) ->
//   discretized logistic mixture -> CDF -> 16-bit frequency table.
// Used by the decoder (one wavefront step per tile) and by the encoder (any
// pixels per tile); the arithmetic per pixel is independent of the tile
// position, so both produce identical tables.
#pragma once

#include "nlc_common.cuh"

namespace nlc {

// ---------------------------------------------------------------------
// Context gather (Eq. 3): taps p enumerate rows dy=-h..-1 with dx=-h..h,
// then dy=0 with dx=-h..-1; feature 3p+c holds channel c.  Outside the
// unit the network input is zero.
// ---------------------------------------------------------------------
__device__ __forceinline__ void tap_offset(int p, int h, int& dy, int& dx) {
  int w = 2 * h + 1;
  dy = p / w - h;
  dx = p % w - h;
}

// A compile-time integer as a value.
template <int V>
struct IntC {
  static constexpr int value = V;
};

__device__ __forceinline__ float elu_f(float x) { return x > 0.f ? x : expm1f(x); }

// Floats of the packed FP32 weights:
// W0T[F][C] b0[C] {W1T[C][C] b1[C] W2T[C][C] b2[C]} x R WHT[C][NOp] bH[NOp].
__host__ __device__ inline size_t simt_floats(const Dims& d) {
  return (size_t)d.F * d.C + d.C + (size_t)d.R * (2 * d.C * d.C + 2 * d.C) + (size_t)d.C * d.NOp +
         d.NOp;
}

// ---------------------------------------------------------------------
// Discretized logistic mixture and the frequency table of one channel.
// Network outputs of a pixel: [0,K) logits, [K,4K) locations mu_{c,k},
// [4K,7K) log-scales (clamped below at -7), [7K,10K) raw coupling
// coefficients (tanh).  Coupled locations: m_R = mu_R,
// m_G = mu_G + alpha x_R, m_B = mu_B + beta x_R + gamma x_G.
// Boundary b (1..255) sits at e_b = (2b-256)/255; the table is
//   F(b) = sum_k w_k sigmoid((e_b - m_k)/s_k),
//   q_b = clamp(rint(65280 F(b)), 0, 65280), Q_b = max(Q_{b-1}, q_b),
//   cum_b = Q_b + b, cum_256 = 2^16,
// so every frequency is >= 1 and they sum to 2^16.  Component weights:
// R: pi_k; G: prop. to pi_k P_Rk(r); B: prop. to pi_k P_Rk(r) P_Gk(g).
// The device evaluates F so that it is non-decreasing in b (cdf_term
// below); then Q_b = q_b and any cum_b is computed on its own.
// ---------------------------------------------------------------------
constexpr float kInv255 = 1.f / 255.f;
constexpr float kLog2e = 1.4426950408889634f;

// Boundary e_b = (2b - 256)/255 and the scaled value x_v = (2v - 255)/255.
__device__ __forceinline__ float edge_f(int b) { return __fmul_rn((float)(2 * b - 256), kInv255); }
__device__ __forceinline__ float xval_f(int v) { return __fmul_rn((float)(2 * v - 255), kInv255); }

// e^x and log x through the MUFU ex2 / lg2 approximations (deterministic).
__device__ __forceinline__ float exp_f(float x) { return ex2_approx(__fmul_rn(x, kLog2e)); }
__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float log_f(float x) { return __fmul_rn(lg2_approx(x), 0.6931471805599453f); }

// softplus(x) = max(x, 0) + log(1 + e^{-|x|})
__device__ __forceinline__ float softplus_f(float x) {
  return __fadd_rn(fmaxf(x, 0.f), log_f(__fadd_rn(1.f, exp_f(-fabsf(x)))));
}
// log(1 - e^{-d}), d > 0.  For d < 1/8 the Taylor series
// 1 - e^{-d} = d (1 - d/2 + d^2/6 - d^3/24 + d^4/120) (relative error below
// 5e-8 there) avoids the cancellation of 1 - e^{-d}.
__device__ __forceinline__ float log1mexp_f(float d) {
  if (d < 0.125f) {
    float p = __fmaf_rn(d, 1.f / 120.f, -1.f / 24.f);
    p = __fmaf_rn(p, d, 1.f / 6.f);
    p = __fmaf_rn(p, d, -0.5f);
    p = __fmaf_rn(p, d, 1.f);
    return log_f(__fmul_rn(d, p));
  }
  return log_f(__fsub_rn(1.f, exp_f(-d)));
}

// log(1 - e^{-d}) of a component with log-scale ls and inv = e^{-ls}, where
// d = (2/255) inv is the bin width over the scale; for d < e^-14 it is taken
// as log d = log(2/255) - ls (error O(d)), which stays finite when inv
// underflows.
__device__ __forceinline__ float bin_log_width(float ls, float inv) {
  const float logd = __fsub_rn(-4.848116f, ls);
  return logd < -14.f ? logd : log1mexp_f(__fmul_rn(2.f * kInv255, inv));
}

// tanh x = sign(x) (1 - 2/(1 + e^{2|x|})), |x| capped at 20 (tanh = 1 in FP32).
__device__ __forceinline__ float tanh_f(float x) {
  const float ax = fminf(fabsf(x), 20.f);
  const float r = rcp_approx(__fadd_rn(1.f, exp_f(__fmul_rn(2.f, ax))));
  return copysignf(__fsub_rn(1.f, __fmul_rn(2.f, r)), x);
}

// log P(v) of one logistic component with location m, inv = e^{-ls} and
// lme = bin_log_width(ls, inv), stable in both tails:
// log P = -softplus(-a) - softplus(b) + log(1 - e^{-(a-b)}), a - b = (2/255)/s.
__device__ __forceinline__ float log_bin_mass_f(float m, float inv, float lme, int v) {
  if (v <= 0) return -softplus_f(-__fmul_rn(__fsub_rn(edge_f(1), m), inv));
  if (v >= 255) return -softplus_f(__fmul_rn(__fsub_rn(edge_f(255), m), inv));
  const float a = __fmul_rn(__fsub_rn(edge_f(v + 1), m), inv);
  const float b = __fmul_rn(__fsub_rn(edge_f(v), m), inv);
  return __fadd_rn(__fsub_rn(-softplus_f(-a), softplus_f(b)), lme);
}

// Scratch of one coding group in the CDF stage (a warp in the decoder, half a
// warp in the table entry point):
// the channel's active components (weight >= kWmin), compacted in
// increasing component order, as (m_k, c_k = log2(e)/s_k, w_k 2^23, 0),
// then zero entries (weight 0, term 0) up to 2 kMaxK, so that unrolled
// loops may read past the last active component.
struct alignas(16) WarpScratch {
  float4 cp[2 * kMaxK];
  float4 pad;  // 528-byte stride: two half-warp groups read different banks
};

// Table of one coding warp for decoding with an explicit cum[0..255]
// (lane-interleaved, see cum_pos); cum_256 = 2^16.
struct TableScratch {
  uint32_t cum[256];
};

// Components whose weight is below 2^-17 are left out of the CDF: together
// they move 65280 F(b) by at most half a count per component.
constexpr float kWmin = 7.62939453125e-06f;

// Bound of a component's location in the CDF (2^100; |m - e| c stays finite).
constexpr float kMMax = 1.2676506002282294e30f;

// Fixed point with 23 fraction bits: x in [0, 2^23] plus 2^23, rounded to
// nearest, is 2^23 + rint(x) (the spacing of floats in [2^23, 2^24] is 1);
// its bit pattern minus that of 2^23 is rint(x).
constexpr float kFixOne = 8388608.f;           // 2^23
constexpr uint32_t kFixOneBits = 0x4B000000u;  // bit pattern of 2^23
constexpr float kLn2x23 = 15.942385152878742f;  // 23 ln 2

// rint(e 2^23) for e in [0, 1].
__device__ __forceinline__ uint32_t fix23(float e) {
  return (uint32_t)__float_as_int(__fadd_rn(__fmul_rn(e, kFixOne), kFixOne)) - kFixOneBits;
}

// ---------------------------------------------------------------------
// Coding groups.  One pixel's channels are coded by a group of GW lanes
// (GW = 32: a whole warp; GW = 16: half a warp, so that a warp codes two
// pixels at once); lanes gl < K of a group hold component gl.  Group
// reductions over floats are xor butterflies, which give the same value in
// every lane of the group and, for K <= 16, the same value for GW = 16 and
// GW = 32 (the upper half adds exact zeros first).
// ---------------------------------------------------------------------
template <int GW>
__device__ __forceinline__ float grp_max(float v) {
#pragma unroll
  for (int o = GW / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o, GW));
  return v;
}
template <int GW>
__device__ __forceinline__ unsigned grp_mask(int lane) {
  return GW == 32 ? 0xffffffffu : (0xFFFFu << (lane & 16));
}
// Exact group maximum of floats and exact group sum of integers.  A whole
// warp uses redux.sync (the maximum on order-preserving integer keys:
// negative floats get their magnitude bits flipped); a 16-lane group uses
// xor butterflies, because redux.sync with a mask per half warp is slower
// than the butterfly.  Both forms give the same value for inputs that are
// not NaN (the integer keys would rank a NaN above +inf, fmaxf drops it), so
// the callers map NaN to -inf first (no_nan).
template <int GW>
__device__ __forceinline__ float grp_max_r(float v) {
  if constexpr (GW == 32) {
    int k = __float_as_int(v);
    k = k >= 0 ? k : k ^ 0x7FFFFFFF;
    k = __reduce_max_sync(0xffffffffu, k);
    return __int_as_float(k >= 0 ? k : k ^ 0x7FFFFFFF);
  } else {
    return grp_max<GW>(v);
  }
}
__device__ __forceinline__ float no_nan(float v) { return v == v ? v : -INFINITY; }
template <int GW>
__device__ __forceinline__ uint32_t grp_isum(uint32_t v) {
  if constexpr (GW == 32) {
    return __reduce_add_sync(0xffffffffu, v);
  } else {
#pragma unroll
    for (int o = GW / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, GW);
    return v;
  }
}
// The group's bits of a warp ballot, group lane 0 in bit 0.
template <int GW>
__device__ __forceinline__ unsigned grp_ballot(bool p) {
  const unsigned b = __ballot_sync(0xffffffffu, p);
  return GW == 32 ? b : ((b >> (threadIdx.x & 16)) & 0xFFFFu);
}

// Position of cum_b (b < 256) in TableScratch::cum for groups of GW lanes:
// lane gl's boundaries b = BPL gl + q sit at q GW + gl, so the group's
// stores and loads of one q hit consecutive banks.
template <int GW>
__device__ __forceinline__ int cum_pos(int b) {
  constexpr int BPL = 256 / GW;
  return (b % BPL) * GW + b / BPL;
}
template <int GW>
__device__ __forceinline__ uint32_t cum_at(const TableScratch& ws, int b) {
  return b >= 256 ? 65536u : ws.cum[cum_pos<GW>(b)];
}

// Per-pixel mixture state held by lane k (< K) for component k.
struct CompState {
  float logpi, lw;      // log pi_k, running log weight
  float mu[3], co[3];   // locations, coupling coefficients (tanh)
  float inv[3];         // 1/s = e^{-ls} (log-scale ls clamped at -7)
  float c[3];           // log2(e) / s
  float lme[3];         // bin_log_width(ls, 1/s)
};

template <int GW = 32>
__device__ __forceinline__ void comp_init(const float* P, int K, int gl, CompState& cs) {
  // log-sum-exp of the logits: exact max, then the sum of e^{logit - max}
  // in fixed point (an exact integer sum, S >= 2^23 from the max itself)
  const float logit = gl < K ? no_nan(P[gl]) : -INFINITY;  // a NaN logit: weight 0
  const float mx = grp_max_r<GW>(logit);
  const uint32_t E = fix23(gl < K ? exp_f(__fsub_rn(logit, mx)) : 0.f);
  const uint32_t S = grp_isum<GW>(E);
  const float lse = __fadd_rn(mx, __fsub_rn(log_f((float)S), kLn2x23));
  cs.logpi = __fsub_rn(logit, lse);
  cs.lw = cs.logpi;
  if (gl < K) {
#pragma unroll
    for (int c = 0; c < 3; c++) {
      cs.mu[c] = P[K + c * K + gl];
      const float ls = fmaxf(P[4 * K + c * K + gl], -7.f);
      cs.co[c] = tanh_f(P[7 * K + c * K + gl]);
      cs.inv[c] = exp_f(-ls);
      cs.c[c] = __fmul_rn(cs.inv[c], kLog2e);
      cs.lme[c] = bin_log_width(ls, cs.inv[c]);
    }
  }
}

// a[ch] by selects (ch need not be a compile-time constant, so the arrays
// stay in registers when the channel loop is not unrolled).
template <class T>
__device__ __forceinline__ T pick3(const T (&a)[3], int ch) {
  return ch == 0 ? a[0] : (ch == 1 ? a[1] : a[2]);
}

// Location of channel ch of component (lane) given decoded r, g.
__device__ __forceinline__ float comp_mean(const CompState& cs, int ch, int r, int g) {
  const float xr = xval_f(r), xg = xval_f(g);
  if (ch == 0) return cs.mu[0];
  if (ch == 1) return __fadd_rn(cs.mu[1], __fmul_rn(cs.co[0], xr));
  return __fadd_rn(__fadd_rn(cs.mu[2], __fmul_rn(cs.co[1], xr)), __fmul_rn(cs.co[2], xg));
}

// ---------------------------------------------------------------------
// Pointwise quantised CDF.  F(b) is a fixed-point number in units of 2^-23:
// the sum over the active components of rint(w_k 2^23 sigmoid((e_b-m_k)/s_k)).
// Every operation from b to a term is non-decreasing in b: correctly
// rounded arithmetic with fixed operands, rint, and the MUFU approximations
// ex2.approx (over all floats, saturating to +0 and +inf) and rcp.approx (on
// [1, +inf]), which are monotone on sm_103 (checked exhaustively over those
// ranges by the library before a context is created, see
// mono_check_kernel).  So F is non-decreasing in b as computed, the running
// max of the quantiser leaves q unchanged, and each cum_b follows from b
// alone.  Integer sums do not depend on the order of their terms: every
// split of the components over lanes, in the encoder, the decoder or the
// table entry point, gives the same cum_b.
// ---------------------------------------------------------------------

// One component's term of F at boundary value e: the logistic is
// 1/(1 + 2^z) with z = (m - e) log2(e)/s (a z beyond the float range of 2^z
// gives 2^z = +inf or +0, hence the term's limits 0 and w), and the fused
// w sigmoid + 2^23, rounded once to nearest, is 2^23 + rint(w 2^23 sigmoid)
// (w 2^23 sigmoid lies in [0, 2^23], float spacing 1 in [2^23, 2^24]), read
// back from its bits.  kClamp clamps z to [-126, 126] first, which changes no
// term: past 126 the term is 0 and below -126 it is rint(w) either way
// (1 + 2^z rounds to 1).  The whole-warp search, one pixel per warp and bound
// by latency, measured faster with the clamp; the quads, bound by instruction
// issue, go without it.
template <bool kClamp = false>
__device__ __forceinline__ uint32_t cdf_term(float e, const float4& p) {
  float z = __fmul_rn(__fsub_rn(p.x, e), p.y);
  if (kClamp) z = fminf(fmaxf(z, -126.f), 126.f);
  const float y = __fmaf_rn(p.z, rcp_approx(__fadd_rn(1.f, ex2_approx(z))), kFixOne);
  return (uint32_t)__float_as_int(y) - kFixOneBits;
}

// Partial fixed-point F at boundary value e over components i0, i0 + di, ...
// (di <= 4), five independent terms at a time (the K = 10 mixture in two
// rounds); entries past the active ones are zero, so the reads stay below
// nact - 1 + 4 di + 1 <= 32 entries.  (Handling the remainder exactly
// instead of padding it measured slower: the larger code costs more than
// the skipped terms.)
template <bool kClamp = false>
__device__ __forceinline__ uint32_t cdf_fix(const WarpScratch& ws, int nact, float e, int i0,
                                            int di) {
  uint32_t F = 0;
  for (int i = i0; i < nact; i += 5 * di) {
    const uint32_t t0 = cdf_term<kClamp>(e, ws.cp[i]);
    const uint32_t t1 = cdf_term<kClamp>(e, ws.cp[i + di]);
    const uint32_t t2 = cdf_term<kClamp>(e, ws.cp[i + 2 * di]);
    const uint32_t t3 = cdf_term<kClamp>(e, ws.cp[i + 3 * di]);
    const uint32_t t4 = cdf_term<kClamp>(e, ws.cp[i + 4 * di]);
    F += ((t0 + t1) + (t2 + t3)) + t4;
  }
  return F;
}

// cum_b = q_b + b with q_b = clamp(rint(65280 F), 0, 65280), F = Fi 2^-23
// (ties to even); cum_0 = 0 and cum_256 = 2^16.
__device__ __forceinline__ uint32_t cum_fix(uint32_t Fi, int b) {
  if (b <= 0) return 0u;
  if (b >= 256) return 65536u;
  const unsigned long long P = (unsigned long long)Fi * (unsigned long long)kMq;
  uint32_t q = (uint32_t)(P >> 23);
  const uint32_t r = (uint32_t)(P & 0x7FFFFFull);
  q += (r > 0x400000u || (r == 0x400000u && (q & 1u))) ? 1u : 0u;
  return (q < (uint32_t)kMq ? q : (uint32_t)kMq) + (uint32_t)b;
}

// Channel ch of the pixel: component weights (softmax of the running log
// weights) and locations, compacted into ws.cp.  Returns the location of the
// lane's component (for the posterior update); nact = active components.
template <int GW>
__device__ __forceinline__ float channel_setup(const CompState& cs, int K, int ch, int r, int g,
                                               int gl, WarpScratch& ws, int& nact) {
  // w_k 2^23: for R the mixture weights pi_k = e^{log pi_k} (normalised by
  // comp_init); for G and B the posterior e^{lw_k - max} / sum, the sum taken
  // exactly in fixed point
  float wS = 0.f;
  if (ch == 0) {
    if (gl < K) wS = __fmul_rn(fminf(exp_f(cs.logpi), 1.f), kFixOne);
  } else {
    const float lw = gl < K ? no_nan(cs.lw) : -INFINITY;
    const float mx = grp_max_r<GW>(lw);
    const uint32_t E = fix23(gl < K ? exp_f(__fsub_rn(lw, mx)) : 0.f);
    const uint32_t S = grp_isum<GW>(E);
    wS = fminf(__fmul_rn((float)E, __fmul_rn(kFixOne, rcp_approx((float)S))), kFixOne);
  }
  // the location within +-2^100 (a NaN network output becomes -2^100), so
  // that every term is a number: past |m| = 2^100 the CDF is a step either way
  const float m = gl < K ? fminf(fmaxf(comp_mean(cs, ch, r, g), -kMMax), kMMax) : 0.f;
  // the weights sum to one, so at least one component is active
  const bool on = gl < K && wS >= kWmin * kFixOne;
  const unsigned bits = grp_ballot<GW>(on);
  nact = __popc(bits);
  for (int p = gl; p < 2 * kMaxK; p += GW)
    if (p >= nact) ws.cp[p] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (on) ws.cp[__popc(bits & ((1u << gl) - 1u))] = make_float4(m, pick3(cs.c, ch), wS, 0.f);
  __syncwarp();
  return m;
}

// Whole-warp symbol search for slot in [0, 2^16): s with cum_s <= slot <
// cum_{s+1}, and those two values.  Two rounds of base 16; the lanes l and l +
// 16 share boundary l's components (even and odd ones), so that a round of a
// K = 10 mixture is one chunk of five terms per lane.  (31 boundaries with all
// components each in the first round and 7 in the second took 14 % longer:
// three chunks instead of two on the chain of every channel.)
__device__ __forceinline__ int cdf_search(const WarpScratch& ws, int nact, uint32_t slot, int lane,
                                          uint32_t& c0, uint32_t& c1) {
  const unsigned full = 0xffffffffu;
  const int j = lane & 15, half = lane >> 4;
  uint32_t F = cdf_fix<true>(ws, nact, edge_f(16 * (j + 1)), half, 2);
  F += __shfl_xor_sync(full, F, 16);
  const uint32_t u1 = j < 15 ? cum_fix(F, 16 * (j + 1)) : 65536u;
  const int c = __popc(__ballot_sync(full, u1 <= slot) & 0xFFFFu);
  const int b2 = 16 * c + j + 1;
  F = cdf_fix<true>(ws, nact, edge_f(b2), half, 2);
  F += __shfl_xor_sync(full, F, 16);
  const uint32_t top = __shfl_sync(full, u1, c);  // cum_{16 (c+1)}
  const uint32_t u2 = j < 15 ? cum_fix(F, b2) : top;
  const int c2 = __popc(__ballot_sync(full, u2 <= slot) & 0xFFFFu);
  c1 = __shfl_sync(full, u2, c2);
  const uint32_t lo2 = __shfl_sync(full, u2, c2 > 0 ? c2 - 1 : 0);
  const uint32_t lo1 = __shfl_sync(full, u1, c > 0 ? c - 1 : 0);
  c0 = c2 > 0 ? lo2 : (c > 0 ? lo1 : 0u);
  return 16 * c + c2;
}

// Symbol s with cum_s <= slot < cum_{s+1} in an explicit table.
template <int GW>
__device__ __forceinline__ int table_search(const TableScratch& ws, uint32_t slot, int lane) {
  constexpr int BPL = 256 / GW;
  const int gl = lane & (GW - 1);
  int cnt = 0;
#pragma unroll
  for (int q = 0; q < BPL; q++) {
    const int b = gl * BPL + q;
    cnt += (b >= 1 && ws.cum[q * GW + gl] <= slot) ? 1 : 0;
  }
  return __reduce_add_sync(grp_mask<GW>(lane), cnt);
}

// Posterior update after channel ch took value v (lanes < K).
__device__ __forceinline__ void comp_observe(CompState& cs, int K, int ch, float m, int v, int gl) {
  if (gl < K) cs.lw = __fadd_rn(cs.lw, log_bin_mass_f(m, pick3(cs.inv, ch), pick3(cs.lme, ch), v));
}

}  // namespace nlc
