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
// the weights stay for the CTA's lifetime.  Bound: instruction issue (1024^2
// pixels: 63 % of the slots at sixteen warps, 284 warp instructions per pixel;
// MUFU 22 %, tensor pipe 26 %).  Measured, the tables of 12.6 M pixels (h = 3, C
// = 64, R = 2, K = 10): 18.6 ms with one 128-pixel tcgen05 tile at a time per SM
// and 16 lanes per pixel, 4.9 ms so.
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
  uint32_t row_bytes;  // row stride of the image (two rows of 2^30 pixels fit)
  long long out;      // forward: index of its outputs (images in order, raster)
};

// Byte offsets: the weights and biases, the head's tables, then per warp a
// context tile and slots.
struct PxPlan {
  int w0, w1, wh, w0s, bias, row, hbias, warp0, x_bytes, per_warp;
};
constexpr int kPxTables = 20 * 64;  // bytes of the head's tables (kTiles <= 20)
__host__ __device__ inline PxPlan px_plan(const Dims& d) {
  const TcPlan tp = tc_plan(d);
  PxPlan p;
  p.w0 = tp.w0;
  p.w1 = tp.w1[0];
  p.wh = tp.wh;
  p.w0s = tp.w0s;
  p.bias = tp.bias;
  p.row = align_up(tp.bias + (int)(d.C + 2 * d.R * d.C + d.NOp) * 4, 16);
  p.hbias = p.row + kPxTables / 2;
  p.warp0 = align_up(p.row + kPxTables, 128);
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
    s.row_bytes = 3u * U.img_W;
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
      for (int s = 0; s < KS; s++) {
        mma_step(s, acc[j], a[s], w[0][2 * s], w[0][2 * s + 1]);
        mma_step(s, acc[j + 1], a[s], w[1][2 * s], w[1][2 * s + 1]);
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

// The head as the quads want it.  Its outputs are taken in three groups (one
// per channel: logits, location, log-scale; location, log-scale, coupling;
// location, log-scale, two couplings), each as whole components per lane:
// value p * KI + i of lane q is the group's p-th output of component q + 4 i.
// Column 2 q + e of a group's t-th tile is value 2 t + e of lane q, so the
// tile's weight rows are gathered accordingly (ldmatrix takes a row address
// per lane); components past K read a zero row, which exists because 10 K is
// then no multiple of 16.  Which rows and biases these are depends on the model
// alone: they are tables in shared memory, filled once per CTA.
template <int KI>
struct PxHead {
  static constexpr int kTiles = 2 * ((3 * KI + 1) / 2) + 2 * KI;  // 8-column tiles of the groups
  static constexpr int kBytes = kTiles * (8 * 4 + 8 * 4);
  // first tile of channel ch's group
  __host__ __device__ static constexpr int first(int ch) { return ch * ((3 * KI + 1) / 2); }
};
// Output (0 logits, 1..3 locations, 4..6 log-scales, 7..9 couplings) p of
// channel ch's group.
__device__ __forceinline__ int px_output(int ch, int p) {
  return ch == 0 ? (p == 0 ? 0 : p == 1 ? 1 : 4)
                 : ch == 1 ? (p == 0 ? 2 : p == 1 ? 5 : 7)
                           : (p == 0 ? 3 : p == 1 ? 6 : 6 + p);
}
// row[t][r]: byte offset (from the head's weights) of row r of tile t; bias[t][2 q + e].
template <int NT8, int KI>
__device__ __forceinline__ void px_head_tables(const Dims& d, const float* bh, uint32_t* row,
                                               float* bias) {
  using H = PxHead<KI>;
  for (int i = threadIdx.x; i < 8 * H::kTiles; i += blockDim.x) {
    const int t = i >> 3, q = (i & 7) >> 1, e = i & 1;
    const int ch = t >= H::first(2) ? 2 : t >= H::first(1) ? 1 : 0;
    const int slot = 2 * (t - H::first(ch)) + e, np = ch == 2 ? 4 : 3;
    const int k = q + 4 * (slot % KI);
    int n = slot < np * KI && k < d.K ? px_output(ch, slot / KI) * d.K + k : d.NO;
    if (n >= d.NOp) n = 0;  // a value that no lane uses: any row will do
    row[i] = (uint32_t)((n >> 3) * NT8) * 128u + (uint32_t)(n & 7) * 16u;
    bias[i] = bh[n];
  }
}

// Channel CH's group: v[r][value] of the lane's pixel r (rows g, g + 8).
template <int NT8, int KI, int CH>
__device__ __forceinline__ void px_head(uint32_t wh, const uint32_t* row, const float* bias,
                                        const uint32_t (&a)[NT8 / 2][4],
                                        float (&v)[2][(CH == 2 ? 4 : 3) * KI]) {
  constexpr int KS = NT8 / 2, S = (CH == 2 ? 4 : 3) * KI, T0 = PxHead<KI>::first(CH);
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int t = 0; t < (S + 1) / 2; t++) {
    uint32_t w[2 * KS];
    load_b<KS>(wh + row[8 * (T0 + t) + (lane & 7)], w);
    float c[4];
#pragma unroll
    for (int s = 0; s < KS; s++) mma_step(s, c, a[s], w[2 * s], w[2 * s + 1]);
    const float2 b = *reinterpret_cast<const float2*>(bias + 8 * (T0 + t) + 2 * (lane & 3));
    add2(c[0], c[1], b.x, b.y);
    add2(c[2], c[3], b.x, b.y);
    v[0][2 * t] = c[0];
    v[1][2 * t] = c[2];
    if (2 * t + 1 < S) {
      v[0][2 * t + 1] = c[1];
      v[1][2 * t + 1] = c[3];
    }
  }
}

}  // namespace nlc
