// The local network over all pixels at once (encoder and forward entry
// points), BF16: one warp per 16 pixels from the context to the last table.
//
// The decoder's arithmetic (mma.sync over ascending K steps, the same
// epilogues, the quads of nlc_quad.cuh), laid out for throughput: nothing here
// waits for another warp.  The accumulators of one layer are, lane by lane,
// the A operand of the next, so activations never leave the registers, and the
// head's weight rows are read in an order that leaves every lane with whole
// mixture components of its two pixels, so the coding starts from registers
// too.  Only the context tile (16 pixels) passes through shared memory, where
// the weights stay for the CTA's lifetime.  Bound: instruction issue (57 % of
// the slots, 310 warp instructions per pixel; MUFU 25 %, tensor pipe 21 %).
// Measured, the tables of 12.6 M pixels (h = 3, C = 64, R = 2, K = 10): 18.6 ms
// with one 128-pixel tcgen05 tile at a time per SM and 16 lanes per pixel, 5.6
// ms so.
#pragma once

#include "nlc_mma.cuh"
#include "nlc_quad.cuh"
#include "nlc_tile.cuh"

namespace nlc {

constexpr int kPxRows = 16;  // pixels per warp and pass

// One pixel of a warp's pass.
struct alignas(16) PxSlot {
  const uint8_t* px;  // its address in the image
  int i, j;           // position inside its unit
  int Wu;             // width of the unit
  int row_bytes;      // row stride of the image
  long long out;      // forward: index of its outputs (images in order, raster)
};

// Byte offsets: the weights and biases, then per warp a context tile and slots.
struct PxPlan {
  int w0, w1, wh, w0s, bias, warp0, x_bytes, per_warp;
};
__host__ __device__ inline PxPlan px_plan(const Dims& d) {
  const TcPlan tp = tc_plan(d);
  PxPlan p;
  p.w0 = tp.w0;
  p.w1 = tp.w1[0];
  p.wh = tp.wh;
  p.w0s = tp.w0s;
  p.bias = tp.bias;
  p.warp0 = align_up(tp.bias + (int)(d.C + 2 * d.R * d.C + d.NOp) * 4, 128);
  p.x_bytes = kPxRows * 2 * (d.shear ? (d.h + 1) * d.Fsp : d.Fp);
  p.per_warp = align_up(p.x_bytes + kPxRows * (int)sizeof(PxSlot), 128);
  return p;
}

// Slots of pixels q0 .. q0 + 15 of the batch, by the warp's first 16 lanes
// (past the end: the batch's last pixel again).  Returns the lane's unit as
// the hint for its next call.
__device__ __forceinline__ int px_slots(const Unit* __restrict__ units, int n_units, long long n_px,
                                        long long q0, int hint, PxSlot* slots) {
  const int lane = threadIdx.x & 31;
  if (lane < kPxRows) {
    const long long q = min(q0 + lane, n_px - 1);
    int u = hint;
    const bool hit = q >= units[u].px_base && (u + 1 == n_units || q < units[u + 1].px_base);
    if (!hit) u = find_unit_px(units, n_units, q);
    const Unit U = units[u];
    const int r = (int)(q - U.px_base);
    PxSlot s;
    s.i = r / U.Wu;
    s.j = r - s.i * U.Wu;
    const long long row = U.y0 + s.i;
    s.px = U.img + (row * U.img_W + (U.x0 + s.j)) * 3;
    s.Wu = U.Wu;
    s.row_bytes = 3 * U.img_W;
    s.out = U.img_px_base + row * U.img_W + (U.x0 + s.j);
    slots[lane] = s;
    hint = u;
  }
  __syncwarp();
  return hint;
}

// Network up to the head's input: fragments a[s] of ELU(a_R) for the warp's 16
// pixels, from the context tile at x (chunks of 256 bytes).
template <int NT8>
__device__ __forceinline__ void px_hidden(const Dims& d, const PxPlan& pl, uint32_t sb, uint32_t x,
                                          const float* bias, uint32_t (&a)[NT8 / 2][4]) {
  constexpr int KS = NT8 / 2;
  constexpr uint32_t kWBytes = 128u * NT8 * NT8;
  const uint32_t lane = threadIdx.x & 31, q = lane & 3;
  const uint32_t brow = sb + (lane & 7) * 16u;
  float acc[NT8][4], res[NT8][4];
#pragma unroll
  for (int j = 0; j < NT8; j++)
#pragma unroll
    for (int e = 0; e < 4; e++) acc[j][e] = 0.f;
  // first layer: ks K steps; a ldmatrix covers one step of two tiles
  auto first = [&](uint32_t al, uint32_t b0, int ks) {
    const uint32_t bt = (uint32_t)ks * 256u;
    const uint32_t bl = b0 + (lane >> 4) * bt + ((lane >> 3) & 1u) * 128u;
#pragma unroll 1
    for (int s = 0; s < ks; s++) {
      uint32_t f[4];
      ldsm4(al + (uint32_t)s * 512u, f[0], f[1], f[2], f[3]);
#pragma unroll
      for (int j = 0; j < NT8; j += 2) {
        uint32_t w0, w1, w2, w3;
        ldsm4(bl + (uint32_t)j * bt + (uint32_t)s * 256u, w0, w1, w2, w3);
        mma_16816(acc[j], f, w0, w1);
        mma_16816(acc[j + 1], f, w2, w3);
      }
    }
  };
  const uint32_t al = x + (lane & 15u) * 16u + (lane >> 4) * 256u;
  if (d.shear) {
    uint32_t b = brow + (uint32_t)pl.w0s;
    for (int dd = 0; dd <= d.h; dd++) {
      int c_lo, ks;
      shear_krange(d.h, d.Ws, dd, c_lo, ks);
      first(al + (uint32_t)(dd * (d.Fsp / 8) + c_lo) * 256u, b, ks);
      b += (uint32_t)(NT8 * ks) * 256u;
    }
  } else {
    first(al, brow + (uint32_t)pl.w0, d.Fp / 16);
  }
  // tile j's two accumulator rows are half of A fragment j / 2
  auto to_a = [&](int j, const float (&v)[4]) {
    a[j >> 1][(j & 1) * 2] = elu_pair(v[0], v[1]);
    a[j >> 1][(j & 1) * 2 + 1] = elu_pair(v[2], v[3]);
  };
  const float2* b2 = reinterpret_cast<const float2*>(bias) + q;
#pragma unroll
  for (int j = 0; j < NT8; j++) {
    const float2 b = b2[4 * j];
#pragma unroll
    for (int e = 0; e < 4; e++) res[j][e] = acc[j][e];
    add2(res[j][0], res[j][1], b.x, b.y);
    add2(res[j][2], res[j][3], b.x, b.y);
    to_a(j, res[j]);
  }
  uint32_t wl = brow + (uint32_t)pl.w1;
  auto layer = [&]() {
#pragma unroll
    for (int j = 0; j < NT8; j += 2) {
      uint32_t w[2][2 * KS];
#pragma unroll
      for (int i = 0; i < 2; i++) load_b<KS>(wl + (uint32_t)(j + i) * (128u * NT8), w[i]);
#pragma unroll
      for (int i = 0; i < 2; i++)
#pragma unroll
        for (int e = 0; e < 4; e++) acc[j + i][e] = 0.f;
#pragma unroll
      for (int s = 0; s < KS; s++) {
        mma_16816(acc[j], a[s], w[0][2 * s], w[0][2 * s + 1]);
        mma_16816(acc[j + 1], a[s], w[1][2 * s], w[1][2 * s + 1]);
      }
    }
    wl += kWBytes;
  };
  const float2* bn = b2 + 4 * NT8;
#pragma unroll 1
  for (int r = 0; r < d.R; r++) {
    layer();
#pragma unroll
    for (int j = 0; j < NT8; j++) {
      const float2 b = bn[4 * j];
      add2(acc[j][0], acc[j][1], b.x, b.y);
      add2(acc[j][2], acc[j][3], b.x, b.y);
      to_a(j, acc[j]);
    }
    bn += 4 * NT8;
    layer();
#pragma unroll
    for (int j = 0; j < NT8; j++) {
      const float2 b = bn[4 * j];
      add2(acc[j][0], acc[j][1], b.x, b.y);
      add2(acc[j][2], acc[j][3], b.x, b.y);
      add2(res[j][0], res[j][1], acc[j][0], acc[j][1]);
      add2(res[j][2], res[j][3], acc[j][2], acc[j][3]);
      to_a(j, res[j]);
    }
    bn += 4 * NT8;
  }
}

// The head outputs of NP parameter groups (ps[0 .. NP): 0 logits, 1..3
// locations, 4..6 log-scales, 7..9 couplings) as whole components per lane:
// v[r][p * KI + i] = output ps[p] of component q + 4 i of the lane's pixel r
// (rows g, g + 8).  Column 2 q + e of the t-th tile is value 2 t + e of lane
// q, so the tile's weight rows are gathered accordingly (ldmatrix takes a row
// address per lane); components past K read a zero row, which exists because
// 10 K is then no multiple of 16.
template <int NT8, int KI, int NP>
__device__ __forceinline__ void px_head(const Dims& d, const PxPlan& pl, uint32_t sb,
                                        const float* bh, const uint32_t (&a)[NT8 / 2][4],
                                        const int (&ps)[NP], float (&v)[2][NP * KI]) {
  constexpr int KS = NT8 / 2, S = NP * KI;
  const int lane = threadIdx.x & 31, q = lane & 3, K = d.K;
  auto row_of = [&](int slot, int qq) {  // weight row of value `slot` of quad lane qq
    const int k = qq + 4 * (slot % KI);
    return slot < S && k < K ? ps[slot / KI < NP ? slot / KI : 0] * K + k : d.NO;
  };
#pragma unroll
  for (int t = 0; t < (S + 1) / 2; t++) {
    const int qr = (lane & 7) >> 1;
    const int r0 = row_of(2 * t, qr), r1 = row_of(2 * t + 1, qr);
    const int n = (lane & 1) ? r1 : r0;
    // rows that no lane uses may lie past the matrix: any row of it will do
    const int nr = n < d.NOp ? n : 0;
    const uint32_t w0 = sb + (uint32_t)pl.wh + (uint32_t)((nr >> 3) * NT8) * 128u +
                        (uint32_t)(nr & 7) * 16u;
    uint32_t w[2 * KS];
    load_b<KS>(w0, w);
    float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int s = 0; s < KS; s++) mma_16816(c, a[s], w[2 * s], w[2 * s + 1]);
#pragma unroll
    for (int e = 0; e < 2; e++) {
      const int slot = 2 * t + e;
      if (slot < S) {
        const int nb = row_of(slot, q);
        const float b = bh[nb < d.NOp ? nb : 0];
        v[0][slot] = __fadd_rn(c[e], b);
        v[1][slot] = __fadd_rn(c[2 + e], b);
      }
    }
  }
}

}  // namespace nlc
