// Maximum-likelihood training of the local model (Eq. 2): one fused kernel
// runs, per 32-pixel tile, the forward pass, the mixture NLL with its
// analytic gradient, and the adjoint of the 1x1 residual blocks and of the
// masked first layer; weight gradients accumulate in a per-CTA slot that a
// second kernel reduces in a fixed order (deterministic).
#include <cuda_runtime.h>
#include <stdint.h>

#include "nlc_common.cuh"
#include "nlc_f32.cuh"
#include "nlc_kernels.cuh"
#include "nlc_model.cuh"
#include "nlc_train.cuh"

namespace nlc {

// A tile is 16 PX pixels (PX = 2, or 1 for models whose weights leave no room
// for more); its feature-major tiles have rows of 16 PX + 4 floats.  A thread
// is (mg, g): pixels PX mg .. of output group g.
constexpr int kTG = 16;
template <int PX>
__host__ __device__ constexpr int tile_px() { return kTG * PX; }
template <int PX>
__host__ __device__ constexpr int tile_ld() { return kTG * PX + 4; }
constexpr int kLanes = 8;       // lanes per pixel of the likelihood
static_assert(kTG * kTG == kThreads, "one block of every layer per thread");

// Shared memory (float offsets): the weights WT[k][n] of every layer (rows of
// ld(N) floats), the context X, the activations u_0, v_0, u_1, .. (2R + 1
// tiles), dP, and one region for the head outputs P, then the two gradient
// tiles.  All tiles are [feature][16 px + 4].
struct TrainPlan {
  int w0, w1, wstride, wh, bias, X, U, DP, P, ldp, G, G2, red, slots, end;
};
// Weight row stride: 4 modulo 8, so that neighbouring rows start on other
// banks (the adjoint reads one column of 8 rows at once) and stay aligned.
__host__ __device__ inline int train_ld(int N) { return ((N + 7) & ~7) + 4; }

__host__ __device__ inline TrainPlan train_plan(const Dims& d, int px) {
  const int tm = kTG * px, ld = tm + 4;
  TrainPlan p;
  int o = 0;
  p.w0 = o; o += d.F * train_ld(d.C);
  p.w1 = o; p.wstride = d.C * train_ld(d.C); o += 2 * d.R * p.wstride;
  p.wh = o; o += d.C * train_ld(d.NOp);
  p.bias = o; o += d.C + 2 * d.R * d.C + d.NOp;
  p.X = o; o += d.F * ld;
  p.U = o; o += (2 * d.R + 1) * d.C * ld;
  p.DP = o; o += d.NO * ld;
  p.ldp = d.NOp + 4;
  p.P = o; p.G = o; p.G2 = o + d.C * ld;
  o += 2 * d.C * ld > tm * p.ldp ? 2 * d.C * ld : tm * p.ldp;
  p.red = o; o += 32;
  p.slots = o; o += tm * 4;
  p.end = o;
  return p;
}

inline size_t train_smem_bytes(const Dims& d, int px) { return (size_t)train_plan(d, px).end * 4; }
// PX of the model's tiles, 0 if even the small ones do not fit.
static int train_px(const Dims& d) {
  return train_smem_bytes(d, 2) <= 227 * 1024 ? 2 : train_smem_bytes(d, 1) <= 227 * 1024 ? 1 : 0;
}

// Blocks of the backward products: a warp is 8 x 4 of the 16 x 16 threads, so
// that its 16-byte reads of eight neighbouring rows fill one wavefront.
__device__ __forceinline__ int fast16() { return (threadIdx.x & 7) + 8 * ((threadIdx.x >> 5) & 1); }
__device__ __forceinline__ int slow16() {
  return ((threadIdx.x >> 3) & 3) + 4 * (threadIdx.x >> 6);
}

// ELU'(x) = e^min(x, 0) from the pre-activation x: ELU(x) + 1 would lose the bits
// of e^x that the subtraction of 1 rounded away (all of them below -17).  The
// exponential of a selected argument, because a branch around it took 15 us of
// a 64 x 32^2 step.
__device__ __forceinline__ float elu_d(float x) {
  const float y = x > 0.f ? 0.f : x;
  return expf(y);
}

template <int N>
__device__ __forceinline__ void f32_store(float* p, const float (&v)[N]) {
  if constexpr (N == 2) {
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  } else {
#pragma unroll
    for (int i = 0; i < N; i++) p[i] = v[i];
  }
}

// weight_grad of a thread that has had tiny sums (from then on: a zero would
// flush them): the same sums, one after another.  Asking for it takes a call
// without tiny sums from 543 to 551 us (64 x 32^2), because no reduction starts
// before the last sum is known; the choice at each of the unrolled sums takes
// it to 554-580.
template <int PX>
__device__ __noinline__ void weight_grad_tiny(const float* G, int Nn, const float* X, int Kk,
                                              float* __restrict__ gW, float* __restrict__ gb,
                                              int n0, int NB, int KB) {
  constexpr int kTM = tile_px<PX>(), kTLd = tile_ld<PX>();
  const int kg = fast16();
  for (int n = n0; n < Nn && n < n0 + 16 * NB; n += 16) {
    for (int k = kg; k < Kk && k < kg + 16 * KB; k += 16) {
      float acc = 0.f;
      for (int m = 0; m < kTM; m++) acc = __fmaf_rn(G[n * kTLd + m], X[k * kTLd + m], acc);
      slot_add(gW + (size_t)n * Kk + k, acc);
    }
    if (kg == 0) {
      float bs = 0.f;
      for (int m = 0; m < kTM; m++) bs = __fadd_rn(bs, G[n * kTLd + m]);
      slot_add(gb + n, bs);
    }
  }
}

// Weight gradient of one layer: gW[n][k] += sum_m G[n][m] X[k][m] for n < Nn,
// k < Kk, and gb[n] += sum_m G[n][m], in the CTA's slot.  A thread owns the
// NB x KB block n = first + ng + 16 b, k = kg + 16 j: neighbouring lanes read
// neighbouring rows (conflict-free 16-byte reads along the pixels) and write
// neighbouring elements.  The sums go to the slot as reductions: an element is
// always added to by the same thread, tile after tile, so their order is
// fixed, and no thread waits for the old value (reading it back cost 119 of
// 626 us per 64 x 32^2 step).
template <int PX, int NB, int KB>
__device__ __forceinline__ void weight_grad(bool& tiny, const float* G, int Nn, const float* X, int Kk,
                                            float* __restrict__ gW, float* __restrict__ gb,
                                            int first = 0) {
  constexpr int kTM = tile_px<PX>(), kTLd = tile_ld<PX>();
  const int kg = fast16(), n0 = first + slow16();
  if (n0 >= Nn) return;
  float acc[NB][KB], bs[NB];
#pragma unroll
  for (int b = 0; b < NB; b++) {
    bs[b] = 0.f;
#pragma unroll
    for (int j = 0; j < KB; j++) acc[b][j] = 0.f;
  }
  // rows past the end repeat a row inside (their sums are not stored)
  const float* gp[NB];
  const float* xp[KB];
#pragma unroll
  for (int b = 0; b < NB; b++) gp[b] = G + (n0 + 16 * b < Nn ? n0 + 16 * b : n0) * kTLd;
#pragma unroll
  for (int j = 0; j < KB; j++) xp[j] = X + (kg + 16 * j < Kk ? kg + 16 * j : 0) * kTLd;
  float4 g[2][NB], x[2][KB];  // the next four pixels are read behind the present ones' products
  auto load = [&](int i, int m) {
#pragma unroll
    for (int b = 0; b < NB; b++) g[i][b] = *reinterpret_cast<const float4*>(gp[b] + m);
#pragma unroll
    for (int j = 0; j < KB; j++) x[i][j] = *reinterpret_cast<const float4*>(xp[j] + m);
  };
  auto fma = [&](int i) {
#pragma unroll
    for (int b = 0; b < NB; b++) {
      const float4 y = g[i][b];
      bs[b] = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(bs[b], y.x), y.y), y.z), y.w);
#pragma unroll
      for (int j = 0; j < KB; j++) {
        acc[b][j] = __fmaf_rn(y.x, x[i][j].x, acc[b][j]);
        acc[b][j] = __fmaf_rn(y.y, x[i][j].y, acc[b][j]);
        acc[b][j] = __fmaf_rn(y.z, x[i][j].z, acc[b][j]);
        acc[b][j] = __fmaf_rn(y.w, x[i][j].w, acc[b][j]);
      }
    }
  };
  load(0, 0);
#pragma unroll 1
  for (int m = 0; m < kTM; m += 8) {
    load(1, m + 4);
    fma(0);
    if (m + 8 < kTM) load(0, m + 8);
    fma(1);
  }
  // smallest magnitude but 0, as twice the bits less 1 (a chain per output)
  unsigned lo[NB];
#pragma unroll
  for (int b = 0; b < NB; b++) {
    lo[b] = 2u * __float_as_uint(bs[b]) - 1u;
#pragma unroll
    for (int j = 0; j < KB; j++) lo[b] = min(lo[b], 2u * __float_as_uint(acc[b][j]) - 1u);
  }
#pragma unroll
  for (int b = 1; b < NB; b++) lo[0] = min(lo[0], lo[b]);
  tiny |= lo[0] < 2u * __float_as_uint(kSlotTiny) - 1u;
  if (tiny) {
    weight_grad_tiny<PX>(G, Nn, X, Kk, gW, gb, n0, NB, KB);
    return;
  }
#pragma unroll
  for (int b = 0; b < NB; b++) {
    const int n = n0 + 16 * b;
    if (n >= Nn) continue;
#pragma unroll
    for (int j = 0; j < KB; j++) {
      const int k = kg + 16 * j;
      if (k < Kk) slot_red(gW + (size_t)n * Kk + k, acc[b][j]);
    }
    if (kg == 0) slot_red(gb + n, bs[b]);
  }
}

// Adjoint of a layer: acc[j][a] = sum_n WT[k][n] G[n][PX mg + a] for the
// thread's k = g + 16 j.
template <int PX, int NB>
__device__ __forceinline__ void input_grad(const float* WT, int ld, const float* G, int Nn,
                                           float (&acc)[NB][PX]) {
  constexpr int kTLd = tile_ld<PX>();
  const int g = fast16(), mg = slow16();
#pragma unroll
  for (int j = 0; j < NB; j++)
#pragma unroll
    for (int a = 0; a < PX; a++) acc[j][a] = 0.f;
  const float* w = WT + g * ld;
  const float* y = G + PX * mg;
  float4 v[2][NB];
  float x[2][4][PX];
  auto load = [&](int s, int n) {
#pragma unroll
    for (int i = 0; i < 4; i++) f32_load<PX>(y + (n + i) * kTLd, x[s][i]);
#pragma unroll
    for (int j = 0; j < NB; j++) v[s][j] = *reinterpret_cast<const float4*>(w + 16 * j * ld + n);
  };
  auto fma = [&](int s) {
#pragma unroll
    for (int j = 0; j < NB; j++)
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const float vi = i == 0 ? v[s][j].x : i == 1 ? v[s][j].y : i == 2 ? v[s][j].z : v[s][j].w;
#pragma unroll
        for (int a = 0; a < PX; a++) acc[j][a] = __fmaf_rn(vi, x[s][i][a], acc[j][a]);
      }
  };
  // groups of four outputs, the next one read behind the present one's products
  const int n4 = Nn & ~3;
  load(0, 0);
  int n = 4;
#pragma unroll 1
  for (; n + 4 < n4; n += 8) {
    load(1, n);
    fma(0);
    load(0, n + 4);
    fma(1);
  }
  if (n < n4) {
    load(1, n);
    fma(0);
    fma(1);
  } else {
    fma(0);
  }
  n = n4;
  for (; n < Nn; n++) {  // 10 K may be 2 modulo 4
    float x[PX];
    f32_load<PX>(y + n * kTLd, x);
#pragma unroll
    for (int j = 0; j < NB; j++) {
      const float v = w[16 * j * ld + n];
#pragma unroll
      for (int a = 0; a < PX; a++) acc[j][a] = __fmaf_rn(v, x[a], acc[j][a]);
    }
  }
}

__device__ __forceinline__ float oct_sum(float v) {
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float oct_max(float v) {
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Per-pixel NLL (nats) of the discretized logistic mixture with coupled
// means and its gradient with respect to the 10K network outputs, by eight
// lanes (lane l holds the components k = l, l + 8); writes scale * dL/dP into
// DP[n][m].
__device__ float pixel_nll_grad(const float* P, int K, const int (&v)[3], float scale, float* DP,
                                int kTLd, int l) {
  constexpr int KI = kMaxK / kLanes;
  const float xr = __fdiv_rn((float)(2 * v[0] - 255), 255.f);
  const float xg = __fdiv_rn((float)(2 * v[1] - 255), 255.f);
  // log pi_k = logit_k - LSE(logits)
  float mx = -INFINITY, se = 0.f;
#pragma unroll
  for (int i = 0; i < KI; i++)
    if (l + kLanes * i < K) mx = fmaxf(mx, P[l + kLanes * i]);
  mx = oct_max(mx);
#pragma unroll
  for (int i = 0; i < KI; i++)
    if (l + kLanes * i < K) se = __fadd_rn(se, expf(__fsub_rn(P[l + kLanes * i], mx)));
  const float lse_pi = __fadd_rn(mx, logf(oct_sum(se)));
  float lp[KI], dlm[KI][3], dll[KI][3], co[KI][3];
#pragma unroll
  for (int i = 0; i < KI; i++) {
    const int k = l + kLanes * i;
    lp[i] = -INFINITY;
    if (k >= K) continue;
    lp[i] = __fsub_rn(P[k], lse_pi);
#pragma unroll
    for (int c = 0; c < 3; c++) co[i][c] = tanh_f(P[(7 + c) * K + k]);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      float mc = P[(1 + c) * K + k];
      if (c == 1) mc = __fadd_rn(mc, __fmul_rn(co[i][0], xr));
      if (c == 2) mc = __fadd_rn(__fadd_rn(mc, __fmul_rn(co[i][1], xr)), __fmul_rn(co[i][2], xg));
      const float ls = fmaxf(P[(4 + c) * K + k], -7.f), inv = exp_f(-ls);
      lp[i] = __fadd_rn(lp[i], log_bin_mass_f(mc, inv, bin_log_width(ls, inv), v[c]));
      if (v[c] == 0) {
        const float a = __fmul_rn(__fsub_rn(edge_f(1), mc), inv);
        const float sa = 1.f / (1.f + expf(a));  // sigmoid(-a)
        dlm[i][c] = -inv * sa;
        dll[i][c] = -a * sa;
      } else if (v[c] == 255) {
        const float bb = __fmul_rn(__fsub_rn(edge_f(255), mc), inv);
        const float sb = 1.f / (1.f + expf(-bb));  // sigmoid(b)
        dlm[i][c] = inv * sb;
        dll[i][c] = bb * sb;
      } else {
        const float a = __fmul_rn(__fsub_rn(edge_f(v[c] + 1), mc), inv);
        const float bb = __fmul_rn(__fsub_rn(edge_f(v[c]), mc), inv);
        const float dd = __fmul_rn(__fdiv_rn(2.f, 255.f), inv);
        const float gk = 1.f / expm1f(dd);
        const float sa = 1.f / (1.f + expf(a)), sb = 1.f / (1.f + expf(-bb));
        dlm[i][c] = -inv * (sa - sb);
        dll[i][c] = -a * sa + bb * sb - gk * dd;
      }
    }
  }
  mx = -INFINITY;
#pragma unroll
  for (int i = 0; i < KI; i++) mx = fmaxf(mx, lp[i]);
  mx = oct_max(mx);
  float e[KI];
  se = 0.f;
#pragma unroll
  for (int i = 0; i < KI; i++) {
    e[i] = l + kLanes * i < K ? expf(__fsub_rn(lp[i], mx)) : 0.f;
    se = __fadd_rn(se, e[i]);
  }
  se = oct_sum(se);
#pragma unroll
  for (int i = 0; i < KI; i++) {
    const int k = l + kLanes * i;
    if (k >= K) continue;
    const float rho = e[i] / se, pi = expf(__fsub_rn(P[k], lse_pi));
    const float dmR = -rho * dlm[i][0], dmG = -rho * dlm[i][1], dmB = -rho * dlm[i][2];
    DP[(0 * K + k) * kTLd] = scale * (pi - rho);
    DP[(1 * K + k) * kTLd] = scale * dmR;
    DP[(2 * K + k) * kTLd] = scale * dmG;
    DP[(3 * K + k) * kTLd] = scale * dmB;
#pragma unroll
    for (int c = 0; c < 3; c++)
      DP[((4 + c) * K + k) * kTLd] =
          P[(4 + c) * K + k] > -7.f ? scale * (-rho * dll[i][c]) : 0.f;
    DP[(7 * K + k) * kTLd] = scale * dmG * xr * (1.f - co[i][0] * co[i][0]);
    DP[(8 * K + k) * kTLd] = scale * dmB * xr * (1.f - co[i][1] * co[i][1]);
    DP[(9 * K + k) * kTLd] = scale * dmB * xg * (1.f - co[i][2] * co[i][2]);
  }
  return -__fadd_rn(mx, logf(se));
}

// Loss and gradient of a batch, C = 16 NB channels, per tile of 32 pixels:
// forward, mixture NLL with its analytic gradient, adjoint and weight
// gradients.  dparams == nullptr: dP = gradient of the batch's mean code
// length (bits per dimension); else dP = dparams [n_px][10K] (an upstream
// gradient of the network outputs, raster order of the batch) and no loss is
// computed.
//
// Bound: the FMA pipe (3 x 27,400 multiply-adds per pixel: 19 k cycles per
// tile at 128 per clock).  Why this shape: 32 pixels leave room for all
// weights (one transposed copy serves both directions: the forward reads a
// row across the outputs, the adjoint a column of neighbouring rows, apart by
// 4 banks), so no layer waits for L2; a thread holds its block of the residual
// stream and of its gradient in registers; a layer costs one barrier.
// Measured, 64 x 32^2 (h = 3, C = 64, R = 2, K = 10): 1424 us with 64-pixel tiles and
// weights read through L2, 505 us so (FMA pipe about a third busy; the rest is
// latency at two warps per scheduler).  The pre-activations, which the adjoint
// needs for ELU', do not fit in shared memory beside the activations (46 KB):
// they pass through the workspace (40 KB per CTA, in L2), and their reads and
// exponentials take the call (kernel and reduction) from 521 to 543 us; the
// small sums of weight_grad take it to 551.
template <int NB, int PX>
__global__ void __launch_bounds__(kThreads, 1)
    loss_grad_kernel(Dims d, const float* __restrict__ wt, const uint8_t* __restrict__ batch,
                     int N, int H, int W, const float* __restrict__ dparams,
                     float* __restrict__ part_g, float* __restrict__ part_l, int n_w,
                     float* pre_act) {
  extern __shared__ __align__(16) float sm[];
  constexpr int kTM = tile_px<PX>(), kTLd = tile_ld<PX>();
  const TrainPlan pl = train_plan(d, PX);
  const int C = d.C, F = d.F, R = d.R, K = d.K, NO = d.NO, h = d.h;
  const int ldc = train_ld(C), ldh = train_ld(d.NOp);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* gW = part_g + (size_t)blockIdx.x * n_w;
  for (int i = threadIdx.x; i < n_w; i += blockDim.x) gW[i] = 0.f;
  if (threadIdx.x < 32) sm[pl.red + threadIdx.x] = 0.f;
  // canonical offsets of the gradient
  const size_t oW0 = 0, ob0 = (size_t)C * F, oblk = ob0 + C;
  const size_t blk = 2 * (size_t)C * C + 2 * C;
  const size_t oWH = oblk + (size_t)R * blk, obH = oWH + (size_t)NO * C;
  // packed transposed weights W0T[F][C] b0 {W1T[C][C] b1 W2T b2}xR WHT[C][NOp] bH
  {
    const float* src = wt;
    float* bias = sm + pl.bias;
    // 16 bytes a thread (every row and matrix is a multiple of 16 floats)
    auto rows = [&](float* dst, int ld, int nr, int nc) {
      const float4* v = reinterpret_cast<const float4*>(src);
      const unsigned c4 = (unsigned)nc / 4u, n = (unsigned)nr * c4;
#pragma unroll 8
      for (unsigned e = threadIdx.x; e < n; e += kThreads) {
        const unsigned r = e / c4;
        *reinterpret_cast<float4*>(dst + r * ld + 4u * (e - r * c4)) = v[e];
      }
      src += nr * nc;
      for (int e = threadIdx.x; e < nc; e += kThreads) bias[e] = src[e];
      src += nc;
      bias += nc;
    };
    rows(sm + pl.w0, ldc, F, C);
    for (int l = 0; l < 2 * R; l++) rows(sm + pl.w1 + l * pl.wstride, ldc, C, C);
    rows(sm + pl.wh, ldh, C, d.NOp);
  }
  int4* slots = reinterpret_cast<int4*>(sm + pl.slots);
  const long long HW = (long long)H * W, n_px = (long long)N * HW;
  const float scale = 1.f / (0.6931471805599453f * 3.f * (float)n_px);
  const long long ntiles = (n_px + kTM - 1) / kTM;
  // the CTA's pre-activations [2R + 1][C][kTM], written and read by this CTA only
  float* Z = pre_act + (size_t)blockIdx.x * (2 * R + 1) * C * kTM;
  // forward: pixels PX fm .. (neighbouring lanes) of outputs NB fg ..;
  // adjoint: the same pixels of mg, outputs g + 16 j (neighbouring lanes)
  const int fm = threadIdx.x & 15, fg = threadIdx.x >> 4;
  const int g = fast16(), mg = slow16();
  float loss = 0.f;
  bool tiny = false;  // a sum below kSlotTiny is in the thread's part of the slot
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    if (threadIdx.x < kTM) {
      const long long q = tile * kTM + threadIdx.x;
      int4 s = make_int4(-1, 0, 0, 0);
      if (q < n_px) {
        const int im = (int)(q / HW), r = (int)(q - im * HW);
        s = make_int4(im, r / W, r % W, 0);
      }
      slots[threadIdx.x] = s;
    }
    __syncthreads();
    // context (each image is one unit; zero outside it)
    const int ntap = 2 * h * (h + 1);
    for (int it = threadIdx.x; it < kTM * ntap; it += blockDim.x) {
      const int m = it % kTM, p = it / kTM;
      const int4 s = slots[m];
      float v0 = 0.f, v1 = 0.f, v2 = 0.f;
      int dy, dx;
      tap_offset(p, h, dy, dx);
      const int ii = s.y + dy, jj = s.z + dx;
      if (s.x >= 0 && ii >= 0 && jj >= 0 && jj < W) {
        const uint8_t* px = batch + ((long long)s.x * HW + (long long)ii * W + jj) * 3;
        v0 = __fdiv_rn((float)(2 * px[0] - 255), 255.f);
        v1 = __fdiv_rn((float)(2 * px[1] - 255), 255.f);
        v2 = __fdiv_rn((float)(2 * px[2] - 255), 255.f);
      }
      float* X = sm + pl.X + 3 * p * kTLd + m;
      X[0] = v0;
      X[kTLd] = v1;
      X[2 * kTLd] = v2;
    }
    __syncthreads();
    // ---- forward ----
    {
      float res[NB][PX];
      const float* bias = sm + pl.bias + NB * fg;
      float* U = sm + pl.U + NB * fg * kTLd + PX * fm;  // the thread's block of the next tile
      float* z = Z + NB * fg * kTM + PX * fm;
      auto store = [&](const float (&v)[NB][PX]) {
#pragma unroll
        for (int b = 0; b < NB; b++) {
          f32_store<PX>(z + b * kTM, v[b]);
#pragma unroll
          for (int a = 0; a < PX; a++) U[b * kTLd + a] = elu_f(v[b][a]);
        }
        U += C * kTLd;
        z += C * kTM;
        bias += C;
      };
      f32_dot<PX, NB>(sm + pl.X + PX * fm, kTLd, F, sm + pl.w0 + NB * fg, ldc, res);
#pragma unroll
      for (int b = 0; b < NB; b++)
#pragma unroll
        for (int a = 0; a < PX; a++) res[b][a] = __fadd_rn(res[b][a], bias[b]);
      store(res);
      __syncthreads();
      for (int l = 0; l < 2 * R; l++) {
        float acc[NB][PX];
        f32_dot<PX, NB>(sm + pl.U + l * C * kTLd + PX * fm, kTLd, C,
                       sm + pl.w1 + l * pl.wstride + NB * fg, ldc, acc);
#pragma unroll
        for (int b = 0; b < NB; b++)
#pragma unroll
          for (int a = 0; a < PX; a++) {
            acc[b][a] = __fadd_rn(acc[b][a], bias[b]);
            if (l & 1) acc[b][a] = res[b][a] = __fadd_rn(res[b][a], acc[b][a]);
          }
        store(acc);
        __syncthreads();
      }
      // head: blocks of four outputs
      const float* in = sm + pl.U + 2 * R * C * kTLd + PX * fm;
      for (int c = 4 * fg; c < d.NOp; c += 4 * kTG) {
        float acc[4][PX];
        f32_dot<PX, 4>(in, kTLd, C, sm + pl.wh + c, ldh, acc);
        const float* bh = sm + pl.bias + (1 + 2 * R) * C + c;
#pragma unroll
        for (int a = 0; a < PX; a++)
          *reinterpret_cast<float4*>(sm + pl.P + (PX * fm + a) * pl.ldp + c) =
              make_float4(__fadd_rn(acc[0][a], bh[0]), __fadd_rn(acc[1][a], bh[1]),
                          __fadd_rn(acc[2][a], bh[2]), __fadd_rn(acc[3][a], bh[3]));
      }
    }
    __syncthreads();
    // ---- likelihood and its gradient (zero for pixels past the batch) ----
    if (dparams) {
      for (int e = threadIdx.x; e < kTM * NO; e += blockDim.x) {
        const int m = e / NO, k = e - m * NO;
        const long long q = tile * kTM + m;
        sm[pl.DP + k * kTLd + m] = q < n_px ? dparams[q * NO + k] : 0.f;
      }
    } else if (threadIdx.x < kLanes * kTM) {
      const int m = threadIdx.x / kLanes, l = threadIdx.x % kLanes;
      const int4 s = slots[m];
      int v[3] = {0, 0, 0};
      if (s.x >= 0) {
        const uint8_t* px = batch + ((long long)s.x * HW + (long long)s.y * W + s.z) * 3;
        v[0] = px[0], v[1] = px[1], v[2] = px[2];
      }
      const float nll = pixel_nll_grad(sm + pl.P + m * pl.ldp, K, v, scale, sm + pl.DP + m, kTLd, l);
      if (s.x < 0) {  // its terms may be infinite: not multiplied by 0 but left out
        __syncwarp(0xffu << (threadIdx.x & 24));
        for (int k = l; k < NO; k += kLanes) sm[pl.DP + k * kTLd + m] = 0.f;
      } else if (l == 0) {
        loss = __fadd_rn(loss, nll);
      }
    }
    __syncthreads();
    // ---- adjoint ----
    const float* Ul = sm + pl.U + 2 * R * C * kTLd;  // the layer's input activations
    float da[NB][PX], acc[NB][PX];
    float* G = sm + pl.G;
    float* G2 = sm + pl.G2;
    // gradient through ELU of the thread's block of layer l
    auto through = [&](int l, float (&v)[NB][PX]) {
      const float* z = Z + (l * C + g) * kTM + PX * mg;
#pragma unroll
      for (int j = 0; j < NB; j++) {
        float x[PX];
        f32_load<PX>(z + 16 * j * kTM, x);
#pragma unroll
        for (int a = 0; a < PX; a++) v[j][a] = __fmul_rn(v[j][a], elu_d(x[a]));
      }
    };
    auto put = [&](float* o, const float (&v)[NB][PX]) {
#pragma unroll
      for (int j = 0; j < NB; j++)
#pragma unroll
        for (int a = 0; a < PX; a++) o[(g + 16 * j) * kTLd + PX * mg + a] = v[j][a];
    };
    input_grad<PX, NB>(sm + pl.wh, ldh, sm + pl.DP, NO, da);  // WH^T dP
    through(2 * R, da);
    put(G, da);  // P is dead: the likelihood has read it
    for (int n = 0; n < NO; n += 16 * 4) {  // 16 x 4 outputs a round, the last as many as needed
      if (NO - n > 48) weight_grad<PX, 4, NB>(tiny, sm + pl.DP, NO, Ul, C, gW + oWH, gW + obH, n);
      else if (NO - n > 16) weight_grad<PX, 3, NB>(tiny, sm + pl.DP, NO, Ul, C, gW + oWH, gW + obH, n);
      else weight_grad<PX, 1, NB>(tiny, sm + pl.DP, NO, Ul, C, gW + oWH, gW + obH, n);
    }
    __syncthreads();
    for (int r = R - 1; r >= 0; r--) {
      const size_t oW1 = oblk + r * blk, ob1 = oW1 + (size_t)C * C;
      const size_t oW2 = ob1 + C, ob2 = oW2 + (size_t)C * C;
      const float* V = sm + pl.U + (2 * r + 1) * C * kTLd;
      input_grad<PX, NB>(sm + pl.w1 + (2 * r + 1) * pl.wstride, ldc, G, C, acc);  // dv = W2^T da
      through(2 * r + 1, acc);
      put(G2, acc);
      weight_grad<PX, NB, NB>(tiny, G, C, V, C, gW + oW2, gW + ob2);
      __syncthreads();
      const float* Ur = V - C * kTLd;
      input_grad<PX, NB>(sm + pl.w1 + 2 * r * pl.wstride, ldc, G2, C, acc);  // du = W1^T dz
      through(2 * r, acc);
#pragma unroll
      for (int j = 0; j < NB; j++)
#pragma unroll
        for (int a = 0; a < PX; a++) da[j][a] = __fadd_rn(da[j][a], acc[j][a]);
      put(G, da);
      weight_grad<PX, NB, NB>(tiny, G2, C, Ur, C, gW + oW1, gW + ob1);
      __syncthreads();
    }
    switch ((F + 15) / 16) {
      case 1: weight_grad<PX, NB, 1>(tiny, G, C, sm + pl.X, F, gW + oW0, gW + ob0); break;
      case 3: weight_grad<PX, NB, 3>(tiny, G, C, sm + pl.X, F, gW + oW0, gW + ob0); break;
      default: weight_grad<PX, NB, 5>(tiny, G, C, sm + pl.X, F, gW + oW0, gW + ob0); break;
    }
    __syncthreads();
  }
  // loss: the pixels' lanes of every warp, then the warps, in a fixed order
#pragma unroll
  for (int o = kLanes; o < 32; o <<= 1)
    loss = __fadd_rn(loss, __shfl_xor_sync(0xffffffffu, loss, o));
  if (lane == 0) sm[pl.red + warp] = loss;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int i = 0; i < kWarps; i++) t = __fadd_rn(t, sm[pl.red + i]);
    part_l[blockIdx.x] = t;
  }
}

// grad[i] = sum over the slots b of part_g[b][i], in a fixed order: 8 threads
// of a block take every eighth slot of one element, then their sums are added
// in turn.  (One thread per element was a chain of 152 additions and left two
// thirds of the SMs idle: 14 us for 152 slots of 25 k weights, now 7.7 us.)
constexpr int kRedSplit = 8;
__global__ void reduce_grad_kernel(const float* __restrict__ part_g, const float* __restrict__ part_l,
                                   int nblk, int n_w, int ldw, float inv_dims,
                                   float* __restrict__ grad, float* __restrict__ loss) {
  __shared__ float sh[kRedSplit][32];
  const int c = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + c;
  float s = 0.f;
  if (i < n_w) {
#pragma unroll 4
    for (int b = g; b < nblk; b += kRedSplit) s = __fadd_rn(s, part_g[(size_t)b * ldw + i]);
  }
  sh[g][c] = s;
  __syncthreads();
  if (g == 0 && i < n_w) {
#pragma unroll
    for (int k = 1; k < kRedSplit; k++) s = __fadd_rn(s, sh[k][c]);
    grad[i] = s;
  }
  if (blockIdx.x == 0 && g == 1 && part_l && loss) {
    float t = 0.f;
    for (int b = c; b < nblk; b += 32) t = __fadd_rn(t, part_l[b]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t = __fadd_rn(t, __shfl_xor_sync(0xffffffffu, t, o));
    if (c == 0) *loss = t * inv_dims;
  }
}

cudaError_t launch_reduce_grad(const float* part_g, const float* part_l, int nblk, int n_w, int ldw,
                               long long n_px, float* grad, float* loss, cudaStream_t s) {
  const float inv_dims = 1.f / (0.6931471805599453f * 3.f * (float)n_px);
  reduce_grad_kernel<<<(n_w + 31) / 32, 32 * kRedSplit, 0, s>>>(part_g, part_l, nblk, n_w, ldw,
                                                               inv_dims, grad, loss);
  return cudaGetLastError();
}

// The documented limit of the FP32 trainer (n_res = 2 at C = 64, K = 10, and
// what takes no more of the following measure); every such model's tiles fit.
bool simt_train_fits(const Dims& d) {
  const int wide = d.Fp > d.C ? d.Fp : d.C, out = d.NOp > d.C ? d.NOp : d.C;
  const int rows = d.Fp + (2 * d.R + 3) * d.C + d.ldP + d.NOp + wide + 4;
  return (size_t)(64 * rows + out + 32) * 4 + 1024 <= 227 * 1024;
}

static int train_grid(const Dims& d, long long n_px, int sm_count) {
  const int tm = kTG * train_px(d);
  long long t = (n_px + tm - 1) / tm;
  return (int)(t < sm_count ? (t < 1 ? 1 : t) : sm_count);
}

size_t train_ws_bytes(const Dims& d, long long n_px, int sm_count) {
  const size_t nw = (size_t)d.C * d.F + d.C + (size_t)d.R * (2 * d.C * d.C + 2 * d.C) +
                    (size_t)d.NO * d.C + d.NO;
  const int g = train_grid(d, n_px, sm_count);
  const size_t pre = (size_t)(2 * d.R + 1) * d.C * kTG * train_px(d);  // pre-activations
  return ((size_t)g * (nw + 1 + pre) + 64) * 4;
}

template <int PX>
static const void* loss_grad_fn(int C) {
  switch (C) {
    case 16: return (const void*)loss_grad_kernel<1, PX>;
    case 32: return (const void*)loss_grad_kernel<2, PX>;
    case 48: return (const void*)loss_grad_kernel<3, PX>;
    default: return (const void*)loss_grad_kernel<4, PX>;
  }
}

cudaError_t launch_loss_grad(const Dims& d, const float* wt, const uint8_t* batch, int N, int H,
                             int W, const float* dparams, float* loss, float* grad, void* ws,
                             int sm_count, cudaStream_t s) {
  const int n_w = (int)((size_t)d.C * d.F + d.C + (size_t)d.R * (2 * d.C * d.C + 2 * d.C) +
                        (size_t)d.NO * d.C + d.NO);
  const long long n_px = (long long)N * H * W;
  const int g = train_grid(d, n_px, sm_count);
  const int px = train_px(d);
  if (px == 0) return cudaErrorInvalidConfiguration;
  const size_t smem = train_smem_bytes(d, px);
  const void* fn = px == 2 ? loss_grad_fn<2>(d.C) : loss_grad_fn<1>(d.C);
  cudaError_t e = allow_smem(fn);
  if (e != cudaSuccess) return e;
  float* part_g = reinterpret_cast<float*>(ws);
  float* part_l = part_g + (size_t)g * n_w;
  // behind the slots and losses, on 256 bytes
  float* pre_act = part_g + (((size_t)g * (n_w + 1) + 63) & ~(size_t)63);
  Dims dd = d;
  int nw = n_w;
  void* args[] = {&dd, &wt, &batch, &N, &H, &W, &dparams, &part_g, &part_l, &nw, &pre_act};
  if ((e = cudaLaunchKernel(fn, dim3(g), dim3(kThreads), args, smem, s)) != cudaSuccess) return e;
  return launch_reduce_grad(part_g, dparams ? nullptr : part_l, g, n_w, n_w, n_px, grad, loss, s);
}

__global__ void adam_kernel(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int n, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

cudaError_t launch_adam(float* w, const float* g, float* m, float* v, int n, float lr, float b1,
                        float b2, float eps, long long t, cudaStream_t s) {
  const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
  adam_kernel<<<(n + 255) / 256, 256, 0, s>>>(w, g, m, v, n, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

}  // namespace nlc
