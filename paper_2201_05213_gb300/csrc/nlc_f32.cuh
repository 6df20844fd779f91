// FP32 local network of a tile of up to 64 pixels on a 256-thread CTA.
//
// A wavefront step gives a CTA few pixels (often one to eight), so the tile's
// shape follows their number: a thread computes PX pixels x NB outputs, and a
// layer uses as many threads as there are such blocks.  Every output is the
// same chain of fused multiply-adds over ascending inputs whatever the shape,
// so its bits do not depend on it.  Activations are feature-major with PX
// pixels of a feature read as one vector (the same for all outputs of a warp),
// the weights of one input read across the warp; a block of the residual
// stream stays in the registers of its thread, and each layer writes the next
// one's input (ELU applied) into the other of two buffers: one CTA barrier per
// layer.  Bound: the FMA pipe from 16 pixels up (64 x 64 x 64 at 128 FMA per
// clock and SM: 2048 cycles), below that the chain of 4-cycle FMAs and the
// shared-memory reads of the weights (64 inputs: ~500 cycles at 8 pixels).
#pragma once

#include "nlc_model.cuh"

namespace nlc {

constexpr int kF32Rows = 64;

// Offsets in floats: the packed weights, two activation buffers and one region
// for the context tile, then the head outputs P[rows][ldP].
struct F32Plan {
  int w, h0, h1, u, end;
};
__host__ __device__ inline F32Plan f32_plan(const Dims& d) {
  F32Plan p;
  p.w = 0;
  p.h0 = ((int)simt_floats(d) + 3) & ~3;
  p.h1 = p.h0 + d.C * (kF32Rows + 4);
  p.u = p.h1 + d.C * (kF32Rows + 4);
  int u = d.F * (kF32Rows + 4);
  if (kF32Rows * d.ldP > u) u = kF32Rows * d.ldP;
  p.end = p.u + ((u + 3) & ~3);
  return p;
}

// Row stride (floats) of the feature-major tiles of n pixels: whole vectors,
// and 4 more so that the writes of neighbouring outputs fall on other banks.
__device__ __forceinline__ int f32_ldm(int n) {
  return (n <= 4 ? 4 : n <= 8 ? 8 : n <= 16 ? 16 : n <= 32 ? 32 : kF32Rows) + 4;
}

template <int N>
__device__ __forceinline__ void f32_load(const float* p, float (&v)[N]) {
  if constexpr (N == 4) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
  } else if constexpr (N == 2) {
    const float2 x = *reinterpret_cast<const float2*>(p);
    v[0] = x.x, v[1] = x.y;
  } else {
#pragma unroll
    for (int i = 0; i < N; i++) v[i] = p[i];
  }
}

// The operands of U inputs, and their multiply-adds.
template <int U, int PX, int NB>
struct F32Step {
  float x[U][PX], v[U][NB];
  __device__ __forceinline__ void load(const float* in, int ldm, const float* w, int N) {
#pragma unroll
    for (int k = 0; k < U; k++) {
      f32_load<PX>(in + k * ldm, x[k]);
      f32_load<NB>(w + k * N, v[k]);
    }
  }
  __device__ __forceinline__ void fma(float (&acc)[NB][PX]) const {
#pragma unroll
    for (int k = 0; k < U; k++)
#pragma unroll
      for (int b = 0; b < NB; b++)
#pragma unroll
        for (int a = 0; a < PX; a++) acc[b][a] = __fmaf_rn(x[k][a], v[k][b], acc[b][a]);
  }
};

// acc[b][a] = sum over k < Kd (a multiple of 4, at least 12), ascending, of
// w[k][b] in[k][a].  The next U inputs are read while the present ones are
// multiplied; blocks of few outputs read further ahead, to cover the reads'
// latency with as many multiply-adds.
template <int PX, int NB>
__device__ __forceinline__ void f32_dot(const float* in, int ldm, int Kd, const float* w, int N,
                                        float (&acc)[NB][PX]) {
  constexpr int U = PX * NB <= 4 ? 8 : 4;
#pragma unroll
  for (int b = 0; b < NB; b++)
#pragma unroll
    for (int a = 0; a < PX; a++) acc[b][a] = 0.f;
  F32Step<U, PX, NB> s0, s1;
  const int n = Kd / U * U;
  s0.load(in, ldm, w, N);
  int k = U;
#pragma unroll 1
  for (; k + U < n; k += 2 * U) {
    s1.load(in + k * ldm, ldm, w + k * N, N);
    s0.fma(acc);
    s0.load(in + (k + U) * ldm, ldm, w + (k + U) * N, N);
    s1.fma(acc);
  }
  if (k < n) {
    s1.load(in + k * ldm, ldm, w + k * N, N);
    s0.fma(acc);
    s1.fma(acc);
  } else {
    s0.fma(acc);
  }
  if (U > 4 && n < Kd) {
    F32Step<4, PX, NB> s;
    s.load(in + n * ldm, ldm, w + n * N, N);
    s.fma(acc);
  }
}

// X (features of n pixels, stride f32_ldm(n)) -> P[m][ldP]; the caller's
// writes of X must be visible (a CTA barrier); so is P on return.  MG: number
// of pixel groups (a power of two).
template <int PX, int NB>
__device__ __noinline__ void f32_layers(Dims d, float* sm, int n, int MG) {
  __builtin_assume(__isShared(sm));  // else every operand is a generic load
  const F32Plan pl = f32_plan(d);
  const int C = d.C, NOp = d.NOp, ldm = f32_ldm(n);
  const int mg = threadIdx.x & (MG - 1), ng = threadIdx.x / MG;
  const bool on = NB * ng < C;
  const float* w = sm + pl.w;
  float res[NB][PX];
  float* h0 = sm + pl.h0;
  float* h1 = sm + pl.h1;
  auto store = [&](float* h, const float (&v)[NB][PX]) {  // ELU of the block
#pragma unroll
    for (int b = 0; b < NB; b++)
#pragma unroll
      for (int a = 0; a < PX; a++) h[(NB * ng + b) * ldm + PX * mg + a] = elu_f(v[b][a]);
  };
  if (on) {
    f32_dot<PX, NB>(sm + pl.u + PX * mg, ldm, d.F, w + NB * ng, C, res);
    const float* bias = w + d.F * C + NB * ng;
#pragma unroll
    for (int b = 0; b < NB; b++)
#pragma unroll
      for (int a = 0; a < PX; a++) res[b][a] = __fadd_rn(res[b][a], bias[b]);
    store(h0, res);
  }
  w += d.F * C + C;
  __syncthreads();
  for (int r = 0; r < d.R; r++) {
    float acc[NB][PX];
    if (on) {
      f32_dot<PX, NB>(h0 + PX * mg, ldm, C, w + NB * ng, C, acc);
#pragma unroll
      for (int b = 0; b < NB; b++)
#pragma unroll
        for (int a = 0; a < PX; a++) acc[b][a] = __fadd_rn(acc[b][a], w[C * C + NB * ng + b]);
      store(h1, acc);
    }
    w += C * C + C;
    __syncthreads();
    if (on) {
      f32_dot<PX, NB>(h1 + PX * mg, ldm, C, w + NB * ng, C, acc);
#pragma unroll
      for (int b = 0; b < NB; b++)
#pragma unroll
        for (int a = 0; a < PX; a++)
          res[b][a] = __fadd_rn(res[b][a], __fadd_rn(acc[b][a], w[C * C + NB * ng + b]));
      store(h0, res);
    }
    w += C * C + C;
    __syncthreads();
  }
  const float* bh = w + C * NOp;
  for (int it = threadIdx.x; it < MG * (NOp / NB); it += blockDim.x) {
    const int c = NB * (it / MG);
    float acc[NB][PX];
    f32_dot<PX, NB>(h0 + PX * (it & (MG - 1)), ldm, C, w + c, NOp, acc);
    float* o = sm + pl.u + (size_t)(PX * (it & (MG - 1))) * d.ldP + c;
#pragma unroll
    for (int b = 0; b < NB; b++)
#pragma unroll
      for (int a = 0; a < PX; a++) o[a * d.ldP + b] = __fadd_rn(acc[b][a], bh[c + b]);
  }
  __syncthreads();
}

// The shape for n <= 64 pixels (256 threads): few pixels take small blocks so
// that the layer's chain, not the number of threads, sets its time.
__device__ __forceinline__ void f32_run(const Dims& d, float* sm, int n) {
  if (n == 1) f32_layers<1, 1>(d, sm, n, 1);
  else if (n == 2) f32_layers<2, 1>(d, sm, n, 1);
  else if (n <= 8) f32_layers<4, 1>(d, sm, n, n <= 4 ? 1 : 2);
  else if (n <= 32) f32_layers<4, 2>(d, sm, n, n <= 16 ? 4 : 8);
  else f32_layers<4, 4>(d, sm, n, 16);
}

// Context tile of the slots (Slot: px, i, j, Wu, row_bytes as in DecSlot),
// feature-major.  kCoherent: the image is being decoded (loads through L2).
template <bool kCoherent, class Slot>
__device__ __forceinline__ void f32_gather(const Slot* slots, int n, const Dims d, float* sm) {
  float* X = sm + f32_plan(d).u;
  const int h = d.h, ldm = f32_ldm(n), ntap = 2 * h * (h + 1), np = ldm - 4;
  const int lg = 31 - __clz(np);
  for (int it = threadIdx.x; it < ntap << lg; it += blockDim.x) {
    const int m = it & (np - 1), p = it >> lg;
    float v0 = 0.f, v1 = 0.f, v2 = 0.f;
    if (m < n) {
      const Slot s = slots[m];
      // tap_offset; p < 24, so the quotients by 3, 5 and 7 fit in a multiply
      const int row = h == 1 ? (p * 43) >> 7 : h == 2 ? (p * 52) >> 8 : (p * 37) >> 8;
      const int dy = row - h, dx = p - row * (2 * h + 1) - h;
      if (s.i + dy >= 0 && s.j + dx >= 0 && s.j + dx < s.Wu) {
        const uint8_t* px = s.px + (long long)dy * s.row_bytes + 3 * dx;
        const int a = kCoherent ? ld_cg_u8(px) : px[0], b = kCoherent ? ld_cg_u8(px + 1) : px[1],
                  c = kCoherent ? ld_cg_u8(px + 2) : px[2];
        v0 = __fdiv_rn((float)(2 * a - 255), 255.f);
        v1 = __fdiv_rn((float)(2 * b - 255), 255.f);
        v2 = __fdiv_rn((float)(2 * c - 255), 255.f);
      }
    }
    X[(3 * p + 0) * ldm + m] = v0;
    X[(3 * p + 1) * ldm + m] = v1;
    X[(3 * p + 2) * ldm + m] = v2;
  }
}

}  // namespace nlc
