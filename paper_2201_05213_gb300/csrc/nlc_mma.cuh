// BF16 local network of a tile of up to 128 pixels with warp-level MMAs
// (mma.sync m16n8k16, FP32 accumulation), for the wavefront decoder.
//
// What bounds it, and why not tcgen05 here: a wavefront step gives a CTA 1 to
// about 100 pixels, and the network is a chain of 2 R + 2 dependent layers of
// 64 x 64, so the step pays the latency of every layer and none of its
// throughput.  A tcgen05 layer costs an issue-to-completion round trip
// (~480 cycles alone, ~1000 in the decoder) plus tensor-memory loads, stores
// and their waits; a chained mma.sync takes 23 cycles per K step and leaves
// its result in registers.  Both instructions give the same bits (BF16
// products, FP32 accumulation over ascending K steps of 16; compared over 45 M
// dot products on GB300 with random, sparse and widely scaled operands and
// with overflow), so the containers do not depend on which one computes them.
//
// Layout.  m-tiles of 16 pixels; the CTA's 16 warps are split evenly over the
// tile's m-tiles (8, 4 or 2 warps each), and the warps of an m-tile share the
// output columns in 8-column tiles.  The operand tiles are in shared memory in
// 8-feature chunks, feature k of pixel m at (k / 8) * 8 rows + 8 m + k % 8
// (BF16 elements): the 8 x 8 matrices that ldmatrix reads are 128 contiguous
// bytes, and so are the writes of the epilogues.  The weights keep the
// canonical 8 x 8 core matrices (nlc_tc.cuh), which are ldmatrix' B operand as
// they are.  Two activation buffers alternate, so a layer needs one exchange
// among its m-tile's warps.  The residual stream stays in FP32 registers.
#pragma once

#include "nlc_model.cuh"
#include "nlc_tc.cuh"

namespace nlc {

constexpr int kNetWarps = 16;   // warps of the decoder's CTA
constexpr int kNetBars = 2 + 4 + 8;  // mbarriers: m-tiles of 8, 4 and 2 warps
// Row stride (floats) of the head outputs: 4 modulo 8, so that the quads of
// eight consecutive pixels read one output from different banks.
__host__ __device__ inline int net_ldp(const Dims& d) { return d.NOp + 4; }

struct NetPlan {
  int w0, w1, wh, w0s, bias, h0, x, h1, mbar, end;  // byte offsets; w1: the blocks' layers in order
};

// rows: pixels per tile (64 or 128).  Behind the weights: H0 (the head's input
// and every second layer's), then one region for the context tile X, H1 and
// the head outputs P[rows][net_ldp], which follow each other: H1 aliases X
// where both keep a pixel in the same rows of their chunks (then only the
// pixel's own m-tile touches them; the sheared window tile is shared by
// m-tiles, so there H1 follows it), and P is written after a CTA barrier.
__host__ __device__ inline NetPlan net_plan(const Dims& d, int rows, bool win) {
  const TcPlan tp = tc_plan(d);
  NetPlan p;
  p.w0 = tp.w0;
  p.w1 = tp.w1[0];
  p.wh = tp.wh;
  p.w0s = tp.w0s;
  p.bias = tp.bias;
  const int hb = rows * d.C * 2;
  p.h0 = align_up(tp.bias + (int)(d.C + 2 * d.R * d.C + d.NOp) * 4, 128);
  p.x = p.h0 + hb;
  p.h1 = win ? p.x + align_up((rows + 8) * d.Fsp * 2, 128) : p.x;
  int e = p.h1 + hb;
  const int xe = p.x + (d.shear ? (d.h + 1) * d.Fsp : d.Fp) * rows * 2;
  if (!win && xe > e) e = xe;
  const int pe = p.x + rows * net_ldp(d) * 4;
  if (pe > e) e = pe;
  // the whole-warp groups' scratch behind 16 head-output rows
  const int we = p.x + kNetWarps * (net_ldp(d) * 4 + (int)sizeof(WarpScratch));
  if (!win && we > e) e = we;
  p.mbar = align_up(e, 16);
  p.end = align_up(p.mbar + 8 * kNetBars, 128);
  return p;
}

// The decoder's dynamic shared memory: first a record of kSharedHead bytes (its
// beginning is the NetSmem), then the regions of the plans.  Its functions
// address it through this symbol and offsets, never through pointers kept in
// memory: those would be generic addresses, and their loads slower.
extern __shared__ __align__(128) unsigned char dec_smem[];
constexpr int kSharedHead = 640;
template <class T>
__device__ __forceinline__ T* dec_at(int off) {
  return reinterpret_cast<T*>(dec_smem + kSharedHead + off);
}

struct NetSmem {
  Dims d;
  NetPlan pl;
  int rows;
  unsigned limit;  // polls of an exchange before a timeout is recorded
};
__device__ __forceinline__ const NetSmem& net_smem() {
  return *reinterpret_cast<const NetSmem*>(dec_smem);
}

// One thread; a CTA barrier must follow.
__device__ __forceinline__ void net_setup(const NetPlan& pl) {
  for (int i = 0; i < kNetBars; i++) {
    const uint32_t count = i < 2 ? 8u : i < 6 ? 4u : 2u;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(
                     smem_u32(dec_at<uint64_t>(pl.mbar) + i)),
                 "r"(count)
                 : "memory");
  }
}

__device__ __forceinline__ void net_load_weights(const Dims& d, const WeightView& w, int bias) {
  const int nh = w.umma_halves;  // multiple of 64 (core matrices)
  const uint4* src = reinterpret_cast<const uint4*>(w.umma);
  uint4* dst = dec_at<uint4>(0);
  for (int i = threadIdx.x; i < nh / 8; i += blockDim.x) dst[i] = src[i];
  const int nb = (int)bias_floats(d);
  for (int i = threadIdx.x; i < nb; i += blockDim.x) dec_at<float>(bias)[i] = w.bias[i];
}

// ldmatrix / mma.sync.  Volatile without a memory clobber: they keep their
// order among the exchanges and barriers (which do clobber memory), while the
// compiler need not reload what it holds in registers around each of them.
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2,
                                      uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void ldsm2(uint32_t addr, uint32_t& r0, uint32_t& r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
               : "=r"(r0), "=r"(r1)
               : "r"(addr));
}
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                          uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The first K step: C = 0 (no registers to clear).
__device__ __forceinline__ void mma_16816_first(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                                uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%10,%10,%10,%10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
// K step s of a chain.
__device__ __forceinline__ void mma_step(int s, float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  if (s == 0) mma_16816_first(c, a, b0, b1);
  else mma_16816(c, a, b0, b1);
}

// Two FP32 operations in one instruction, each rounded as its scalar form.
__device__ __forceinline__ void add2(float& a, float& b, float x, float y) {
  asm("{\n.reg .b64 p, q;\nmov.b64 p, {%0, %1};\nmov.b64 q, {%2, %3};\n"
      "add.rn.f32x2 p, p, q;\nmov.b64 {%0, %1}, p;\n}\n"
      : "+f"(a), "+f"(b)
      : "f"(x), "f"(y));
}
__device__ __forceinline__ void mul2(float& a, float& b, float x) {
  asm("{\n.reg .b64 p, q;\nmov.b64 p, {%0, %1};\nmov.b64 q, {%2, %2};\n"
      "mul.rn.f32x2 p, p, q;\nmov.b64 {%0, %1}, p;\n}\n"
      : "+f"(a), "+f"(b)
      : "f"(x));
}
// ELU of two values as a BF16 pair: e^x - 1 below zero, by 2^x of the product
// with log2(e), each step rounded.
__device__ __forceinline__ uint32_t elu_pair(float x, float y) {
  float a = x, b = y;
  mul2(a, b, 1.4426950408889634f);
  a = ex2_approx(a);
  b = ex2_approx(b);
  add2(a, b, -1.f, -1.f);
  return pack_bf16(x > 0.f ? x : a, y > 0.f ? y : b);
}

// B fragments of KS K steps of one 8-column tile (addr: the lane's row in the
// tile's first core matrix), two registers per step.
template <int KS>
__device__ __forceinline__ void load_b(uint32_t addr, uint32_t (&w)[2 * KS]) {
  const uint32_t lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 0; s + 1 < KS; s += 2)
    ldsm4(addr + (2u * s + (lane >> 3)) * 128u, w[2 * s], w[2 * s + 1], w[2 * s + 2],
          w[2 * s + 3]);
  if (KS & 1)
    ldsm2(addr + (2u * (KS - 1) + ((lane >> 3) & 1u)) * 128u, w[2 * KS - 2], w[2 * KS - 1]);
}

// The m-tile's warps meet (their writes of a layer's activations become
// visible to each other).  A reduced poll limit runs the meeting through the
// m-tile's mbarrier, `limit` non-blocking tests of it before it counts as
// timed out (it then waits with the default limit, so that no warp runs ahead
// of another); otherwise it is a hardware barrier, ~170 cycles shorter.
__device__ __forceinline__ bool net_exchange(uint64_t* mb, int mt, int threads, unsigned limit,
                                             uint32_t& parity) {
  if (limit >= kMbarSpin) {
    asm volatile("bar.sync %0, %1;" ::"r"(3 + mt), "r"(threads) : "memory");
    return true;
  }
  __syncwarp();
  if ((threadIdx.x & 31) == 0)
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(mb)) : "memory");
  const bool ok = mbar_test(mb, parity, limit);
  if (!ok) mbar_wait(mb, parity);
  parity ^= 1u;
  return ok;
}

// The network of a model with C = 8 NT8 channels on a tile whose m-tiles have
// NS = 8 >> LEVEL warps each (see net_run).  Everything but the first layer's
// depth, the number of blocks and the head's width is a compile-time shape, so
// that a layer is straight-line code: its B fragments are loaded before the
// exchange that precedes it, its A fragments right after.
template <int NT8, int LEVEL, bool PROF>
__device__ __noinline__ uint32_t net_layers(int n, bool win, uint32_t phase, long long* pc) {
  constexpr int NS = 8 >> LEVEL, KS = NT8 / 2, TP = (NT8 + NS - 1) / NS;
  constexpr int HG = LEVEL == 0 ? 1 : LEVEL == 1 ? 2 : 4;  // head tiles computed together
  constexpr uint32_t kWBytes = 128u * NT8 * NT8;  // bytes of a hidden layer's weights
  const NetSmem& t = net_smem();
  const Dims& d = t.d;
  const NetPlan& pl = t.pl;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int mt = warp / NS, ns = warp % NS;
  const bool live = 16 * mt < n;
  const int g = lane >> 2, q = lane & 3;
  const uint32_t sb = smem_u32(dec_smem) + (uint32_t)kSharedHead;
  const uint32_t cs = (uint32_t)t.rows * 16u;  // bytes of a chunk
  // ldmatrix rows: lanes 0-7 rows 0-7, 8-15 rows 8-15 of the even chunk, then the odd chunk
  const uint32_t arow = sb + (uint32_t)(16 * mt + (lane & 15)) * 16u + (uint32_t)(lane >> 4) * cs;
  const uint32_t brow = sb + (uint32_t)(lane & 7) * 16u;
  uint64_t* mb = dec_at<uint64_t>(pl.mbar) + (LEVEL == 0 ? 0 : LEVEL == 1 ? 2 : 6) + mt;
  const bool pr = PROF && pc != nullptr && threadIdx.x == 0;
  long long ck = pr ? clock64() : 0;
  uint32_t parity = (phase >> LEVEL) & 1u;
  const unsigned limit = t.limit;
  const int n_hidden = 1 + 2 * d.R, nht = (d.NO + 7) / 8;
  const uint32_t x = arow + (uint32_t)pl.x, h0 = arow + (uint32_t)pl.h0, h1 = arow + (uint32_t)pl.h1;
  const float* bias = dec_at<float>(pl.bias) + 2 * q;
  // the lane's columns 2q, 2q + 1 of rows g, g + 8 of the m-tile
  unsigned char* o0 = dec_at<unsigned char>(pl.h0) + (16 * mt + g) * 16 + q * 4;
  unsigned char* o1 = dec_at<unsigned char>(pl.h1) + (16 * mt + g) * 16 + q * 4;
  bool ok = true;
  if (live) {
    auto on = [&](int i) { return NT8 % NS == 0 || ns + NS * i < NT8; };
    auto tile = [&](int i) { return on(i) ? ns + NS * i : 0; };  // a tile past the end repeats tile 0
    float acc[TP][4], res[TP][4];
#pragma unroll
    for (int i = 0; i < TP; i++)
#pragma unroll
      for (int e = 0; e < 4; e++) acc[i][e] = 0.f;
    // first layer: ks K steps of A at `al` (acs bytes between chunks) and B at `b0`
    auto first = [&](uint32_t al, uint32_t acs, uint32_t b0, int ks) {
      const uint32_t bt = (uint32_t)ks * 256u;  // bytes of a tile of 8 weight rows
#pragma unroll 1
      for (int s = 0; s < ks; s += 2) {
        uint32_t a0[4], a1[4];
        ldsm4(al + (uint32_t)(2 * s) * acs, a0[0], a0[1], a0[2], a0[3]);
        if (s + 1 < ks) {
          uint32_t w[TP][4];
          ldsm4(al + (uint32_t)(2 * s + 2) * acs, a1[0], a1[1], a1[2], a1[3]);
#pragma unroll
          for (int i = 0; i < TP; i++)
            ldsm4(b0 + (uint32_t)tile(i) * bt + (uint32_t)(2 * s + (lane >> 3)) * 128u, w[i][0],
                  w[i][1], w[i][2], w[i][3]);
#pragma unroll
          for (int i = 0; i < TP; i++) mma_16816(acc[i], a0, w[i][0], w[i][1]);
#pragma unroll
          for (int i = 0; i < TP; i++) mma_16816(acc[i], a1, w[i][2], w[i][3]);
        } else {
          uint32_t w[TP][2];
#pragma unroll
          for (int i = 0; i < TP; i++)
            ldsm2(b0 + (uint32_t)tile(i) * bt + (uint32_t)(2 * s + ((lane >> 3) & 1)) * 128u,
                  w[i][0], w[i][1]);
#pragma unroll
          for (int i = 0; i < TP; i++) mma_16816(acc[i], a0, w[i][0], w[i][1]);
        }
      }
    };
    if (d.shear) {
      // Section 3.1's sheared kernels, one per window row dd, over its tap range
      const uint32_t wcs = win ? (uint32_t)(t.rows + 8) * 16u : cs;
      const uint32_t xw = x + (uint32_t)(lane >> 4) * (wcs - cs);
      uint32_t b = brow + (uint32_t)pl.w0s;
      for (int dd = 0; dd <= d.h; dd++) {
        int c_lo, ks;
        shear_krange(d.h, d.Ws, dd, c_lo, ks);
        first(xw + (win ? 16u * dd : (uint32_t)(dd * (d.Fsp / 8)) * cs) + (uint32_t)c_lo * wcs, wcs,
              b, ks);
        b += (uint32_t)(NT8 * ks) * 256u;
      }
    } else {
      first(x, cs, brow + (uint32_t)pl.w0, d.Fp / 16);
    }
    // v = acc + bias (+ residual); the next layer's operand is ELU(v) in BF16
    auto epilogue = [&](const float* b, auto mode, unsigned char* o) {
      constexpr int M = decltype(mode)::value;  // 0: a = v, 1: a += v, 2: v alone
#pragma unroll
      for (int i = 0; i < TP; i++) {
        const int j = tile(i);
        const float2 bb = *reinterpret_cast<const float2*>(b + 8 * j);
        add2(acc[i][0], acc[i][1], bb.x, bb.y);
        add2(acc[i][2], acc[i][3], bb.x, bb.y);
        if (M == 1) {
          add2(acc[i][0], acc[i][1], res[i][0], res[i][1]);
          add2(acc[i][2], acc[i][3], res[i][2], res[i][3]);
        }
        if (M != 2)
#pragma unroll
          for (int e = 0; e < 4; e++) res[i][e] = acc[i][e];
        if (on(i)) {
          *reinterpret_cast<uint32_t*>(o + j * cs) = elu_pair(acc[i][0], acc[i][1]);
          *reinterpret_cast<uint32_t*>(o + j * cs + 128) = elu_pair(acc[i][2], acc[i][3]);
        }
      }
    };
    uint32_t w[TP][2 * KS], a[KS][4];
    auto prefetch = [&](uint32_t wl) {
#pragma unroll
      for (int i = 0; i < TP; i++) load_b<KS>(wl + (uint32_t)tile(i) * (128u * NT8), w[i]);
    };
    auto load_a = [&](uint32_t h) {
#pragma unroll
      for (int s = 0; s < KS; s++)
        ldsm4(h + (uint32_t)(2 * s) * cs, a[s][0], a[s][1], a[s][2], a[s][3]);
    };
    auto hidden = [&](uint32_t h) {
      load_a(h);
#pragma unroll
      for (int s = 0; s < KS; s++)
#pragma unroll
        for (int i = 0; i < TP; i++) mma_step(s, acc[i], a[s], w[i][2 * s], w[i][2 * s + 1]);
    };
    uint32_t wl = brow + (uint32_t)pl.w1;
    epilogue(bias, IntC<0>{}, o0);
    bias += 8 * NT8;
#pragma unroll 1
    for (int l = 1; l < n_hidden; l += 2) {
      prefetch(wl);
      ok &= net_exchange(mb, mt, 32 * NS, limit, parity);
      hidden(h0);
      epilogue(bias, IntC<2>{}, o1);
      prefetch(wl + kWBytes);
      ok &= net_exchange(mb, mt, 32 * NS, limit, parity);
      hidden(h1);
      epilogue(bias + 8 * NT8, IntC<1>{}, o0);
      wl += 2 * kWBytes;
      bias += 16 * NT8;
    }
    phase = (phase & ~(1u << LEVEL)) | (parity << LEVEL);
  }
  // The head: the m-tile's warps again (all 16 for a single m-tile).  The CTA
  // barrier is the last exchange and keeps P off the tiles it aliases.
  const int all_ok = __syncthreads_and(ok ? 1 : 0);
  if (pr) {
    const long long c = clock64();
    pc[14] += c - ck;
    ck = c;
  }
  const int mts = (n + 15) >> 4;
  const int hlg = mts == 1 ? 4 : 3 - LEVEL;  // log2 of the warps per m-tile
  const int wpm = 1 << hlg, hm = warp >> hlg, hs = warp & (wpm - 1);
  if (hm < mts) {
    const uint32_t wh = brow + (uint32_t)pl.wh;
    const uint32_t h = sb + (uint32_t)pl.h0 + (uint32_t)(16 * hm + (lane & 15)) * 16u +
                       (uint32_t)(lane >> 4) * cs;
    const int ldp = net_ldp(d);
    const float* bh = dec_at<float>(pl.bias) + 8 * NT8 * n_hidden + 2 * q;
    float* o = dec_at<float>(pl.x) + (16 * hm + g) * ldp + 2 * q;
    uint32_t a[KS][4];
#pragma unroll
    for (int s = 0; s < KS; s++)
      ldsm4(h + (uint32_t)(2 * s) * cs, a[s][0], a[s][1], a[s][2], a[s][3]);
#pragma unroll 1
    for (int j0 = hs; j0 < nht; j0 += HG * wpm) {
      uint32_t w[HG][2 * KS];
      float acc[HG][4];
#pragma unroll
      for (int i = 0; i < HG; i++) {
        const int j = j0 + i * wpm;
        load_b<KS>(wh + (uint32_t)(j < nht ? j : j0) * (128u * NT8), w[i]);
      }
#pragma unroll
      for (int s = 0; s < KS; s++)
#pragma unroll
        for (int i = 0; i < HG; i++) mma_step(s, acc[i], a[s], w[i][2 * s], w[i][2 * s + 1]);
#pragma unroll
      for (int i = 0; i < HG; i++) {
        const int j = j0 + i * wpm;
        if (j < nht) {
          const float2 b = *reinterpret_cast<const float2*>(bh + 8 * j);
          *reinterpret_cast<float2*>(o + 8 * j) =
              make_float2(__fadd_rn(acc[i][0], b.x), __fadd_rn(acc[i][1], b.y));
          *reinterpret_cast<float2*>(o + 8 * ldp + 8 * j) =
              make_float2(__fadd_rn(acc[i][2], b.x), __fadd_rn(acc[i][3], b.y));
        }
      }
    }
  }
  __syncthreads();
  if (pr) pc[15] += clock64() - ck;
  return phase | (all_ok ? 0x80000000u : 0u);
}

// The whole network on the n pixels (n >= 1) of the context tile: P[m][ldp]
// = head outputs, visible to the CTA on return.  win: X is the sheared
// decoder's window tile (rows 16 bytes apart, (rows + 8) per chunk).  Returns
// false (in every thread) if an exchange timed out.  phase: the caller's record
// of the warp's mbarrier parities (bit l: m-tiles of 8 >> l warps), 0 at
// first.  PROF: thread 0 adds its cycles of the hidden layers to pc[14] and
// those of the head to pc[15].
template <int NT8, bool PROF>
__device__ __forceinline__ uint32_t net_levels(int n, bool win, uint32_t phase, long long* pc) {
  if (n <= 32) return net_layers<NT8, 0, PROF>(n, win, phase, pc);
  if (n <= 64) return net_layers<NT8, 1, PROF>(n, win, phase, pc);
  return net_layers<NT8, 2, PROF>(n, win, phase, pc);
}
template <bool PROF>
__device__ __forceinline__ bool net_run(int C, int n, bool win, uint32_t& phase, long long* pc) {
  uint32_t r;
  switch (C / 8) {
    case 2: r = net_levels<2, PROF>(n, win, phase, pc); break;
    case 4: r = net_levels<4, PROF>(n, win, phase, pc); break;
    case 6: r = net_levels<6, PROF>(n, win, phase, pc); break;
    default: r = net_levels<8, PROF>(n, win, phase, pc); break;
  }
  phase = r & 0x7FFFFFFFu;
  return (r >> 31) != 0;
}

// --- context tiles ------------------------------------------------------------

// Decoder: what one pixel of the tile needs, filled with the step's schedule.
struct alignas(16) DecSlot {
  uint8_t* px;    // its address in the image
  int i, j;       // position inside its unit
  int Wu;         // width of the unit
  uint32_t row_bytes;  // row stride of the image
  int stream;     // its rANS stream
  int unit;       // unit index; bit 31: the stream's last pixel
};

// 2 v - 255 for byte k of the words w, exactly (2^23 + v is built from the
// byte; both steps are exact), which avoids the slow integer conversion.
__device__ __forceinline__ float byte_input(uint32_t w, int k) {
  const float f = __uint_as_float(__byte_perm(w, kFixOneBits, 0x7540 + k));
  return __fmaf_rn(__fsub_rn(f, kFixOne), 2.f, -255.f);
}

template <bool kCoherent>
__device__ __forceinline__ uint32_t ld_px_word(uintptr_t a) {
  const uint32_t* p = reinterpret_cast<const uint32_t*>(a);
  return kCoherent ? ld_cg_u32(p) : __ldg(p);
}

// Masked tile: X(m, k) = 2v - 255 for feature k = 3p + c of tap p, 0 outside
// the unit and for F <= k < Fp.  One lane per (pixel, context row r): row r <
// h is image row i - h + r over columns j-h .. j+h, row h is row i over
// columns j-h .. j-1; its bytes are contiguous in the image and are read as
// the aligned 32-bit words that hold at least one byte of the row inside the
// unit, realigned with funnel shifts.  X: the pixel's row of the first chunk,
// cs: elements from one chunk to the next.
template <bool kCoherent, class Slot>
__device__ __forceinline__ void gather_row(const Slot& s, int r, int h, int F, int Fp, uint16_t* X,
                                           int cs) {
  const int w2 = 2 * h + 1;
  const int ncol = r < h ? w2 : h;  // pixels of this row's window
  const int k0 = 3 * r * w2;
  // window columns x = j - h + c, c in [0, ncol); inside the unit: [ca, cb)
  const int x0 = s.j - h;
  const int ca = x0 < 0 ? -x0 : 0;
  const int cb = min(ncol, s.Wu - x0);
  const bool row_ok = s.i - h + r >= 0 && ca < cb;
  uint32_t wv[7] = {0u, 0u, 0u, 0u, 0u, 0u, 0u};
  uint32_t sh = 0;
  if (row_ok) {
    const uintptr_t lo = (uintptr_t)(s.px + (long long)(r - h) * s.row_bytes - 3 * h);
    const uintptr_t a = lo + 3 * ca, b = lo + 3 * cb;  // bytes inside the unit
    const uintptr_t w0 = lo & ~(uintptr_t)3;
    sh = 8u * (uint32_t)(lo & 3);
#pragma unroll
    for (int q = 0; q < 6; q++) {
      const uintptr_t wa = w0 + 4 * q;
      if (wa + 4 > a && wa < b) wv[q] = ld_px_word<kCoherent>(wa);
    }
  }
  uint32_t al[6];
#pragma unroll
  for (int q = 0; q < 6; q++) al[q] = __funnelshift_r(wv[q], wv[q + 1], sh);
#pragma unroll
  for (int q = 0; q < 3 * (2 * kMaxH + 1); q++) {
    const int c = q / 3;
    if (c < ncol) {
      const float x = (row_ok && c >= ca && c < cb) ? byte_input(al[q >> 2], q & 3) : 0.f;
      const int k = k0 + q;
      X[(k >> 3) * cs + (k & 7)] = __bfloat16_as_ushort(__float2bfloat16_rn(x));
    }
  }
  if (r == h)
    for (int k = F; k < Fp; k++) X[(k >> 3) * cs + (k & 7)] = 0;
}

// Sheared model, per-pixel window row dd: its Fsp features from chunk
// dd * Fsp/8 onwards (X: the pixel's row of that chunk).
template <bool kCoherent, class Slot>
__device__ __forceinline__ void gather_row_shear(const Slot& s, int dd, int h, int Ws, int Fsp,
                                                 uint16_t* X, int cs) {
  const int dx = (h + 1) * (h - dd) - Ws;  // window column 0 from the pixel's column
  const int x0 = s.j + dx;
  const int ca = x0 < 0 ? -x0 : 0;
  const int cb = min(Ws, s.Wu - x0);
  const bool row_ok = s.i - h + dd >= 0 && ca < cb;
  uint32_t wv[13];
#pragma unroll
  for (int q = 0; q < 13; q++) wv[q] = 0u;
  uint32_t sh = 0;
  if (row_ok) {
    const uintptr_t lo = (uintptr_t)(s.px + (long long)(dd - h) * s.row_bytes + 3 * dx);
    const uintptr_t a = lo + 3 * ca, b = lo + 3 * cb;
    const uintptr_t w0 = lo & ~(uintptr_t)3;
    sh = 8u * (uint32_t)(lo & 3);
#pragma unroll
    for (int q = 0; q < 13; q++) {
      const uintptr_t wa = w0 + 4 * q;
      if (wa + 4 > a && wa < b) wv[q] = ld_px_word<kCoherent>(wa);
    }
  }
  uint32_t al[12];
#pragma unroll
  for (int q = 0; q < 12; q++) al[q] = __funnelshift_r(wv[q], wv[q + 1], sh);
  shear_row_features(al, Ws, Fsp, ca, cb, row_ok,
                     [&](int kc) { return reinterpret_cast<uint4*>(X + kc * cs); });
}

// Columns 2 part, 2 part + 1 of one context row (masked tile): the same
// features from the two or three words around their six bytes, for tiles of so
// few pixels that a lane per row would leave most warps idle (8 pixels: one
// warp with 250 instructions, 1.08 us; so 0.79).  A whole step: 7.30 against
// 7.61 us at 8 pixels, 8.09 / 8.28 at 16, 10.28 / 10.42 at 24, 10.37 / 10.41 at
// 32, where the two meet and the CTA's warps are all in use.
template <class Slot>
__device__ __forceinline__ void gather_part(const Slot& s, int r, int part, int h, int F, int Fp,
                                            uint16_t* X, int cs) {
  const int w2 = 2 * h + 1, ncol = r < h ? w2 : h;
  const int c0 = 2 * part;
  if (r == h && part == 3)
    for (int k = F; k < Fp; k++) X[(k >> 3) * cs + (k & 7)] = 0;
  if (c0 >= ncol) return;
  const int x0 = s.j - h + c0;  // image column (in the unit) of the first one
  const bool row = s.i - h + r >= 0;
  const bool in0 = row && x0 >= 0 && x0 < s.Wu;
  const bool in1 = row && c0 + 1 < ncol && x0 + 1 >= 0 && x0 + 1 < s.Wu;
  uint32_t w[3] = {0u, 0u, 0u};
  uint32_t sh = 0;
  if (in0 || in1) {
    const uintptr_t lo = (uintptr_t)(s.px + (long long)(r - h) * s.row_bytes + 3 * (c0 - h));
    const uintptr_t a = in0 ? lo : lo + 3, b = in1 ? lo + 6 : lo + 3;  // bytes inside the unit
    const uintptr_t w0 = lo & ~(uintptr_t)3;
    sh = 8u * (uint32_t)(lo & 3);
#pragma unroll
    for (int q = 0; q < 3; q++)
      if (w0 + 4 * q + 4 > a && w0 + 4 * q < b) w[q] = ld_px_word<true>(w0 + 4 * q);
  }
  const uint32_t al[2] = {__funnelshift_r(w[0], w[1], sh), __funnelshift_r(w[1], w[2], sh)};
  const int k0 = 3 * (r * w2 + c0);
#pragma unroll
  for (int q = 0; q < 6; q++) {
    if (q >= 3 && c0 + 1 >= ncol) break;
    const float x = (q < 3 ? in0 : in1) ? byte_input(al[q >> 2], q & 3) : 0.f;
    const int k = k0 + q;
    X[(k >> 3) * cs + (k & 7)] = __bfloat16_as_ushort(__float2bfloat16_rn(x));
  }
}

// The decoder's tile, from its slots: a warp covers 8 pixels x 4 rows; up to
// kFewPixels pixels (masked tile), 8 pixels x 4 column pairs of a row.
constexpr int kFewPixels = 32;
template <bool SHEAR>
__device__ __noinline__ void net_gather(int slots, int n) {
  const NetSmem& t = net_smem();
  const Dims d = t.d;
  uint16_t* X = dec_at<uint16_t>(t.pl.x);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int cs = 8 * t.rows;
  if (!SHEAR && n <= kFewPixels) {  // warp: row warp % 4 of the pixels 8 (warp / 4) ..
    const int m = 8 * (warp >> 2) + (lane & 7), r = warp & 3;
    if (m < n && r <= d.h)
      gather_part(dec_at<DecSlot>(slots)[m], r, lane >> 3, d.h, d.F, d.Fp, X + 8 * m, cs);
    return;
  }
  const int r = lane >> 3;
  for (int mb = 8 * warp; mb < n; mb += 8 * (int)(blockDim.x >> 5)) {
    const int m = mb + (lane & 7);
    if (r > d.h || m >= n) continue;
    const DecSlot s = dec_at<DecSlot>(slots)[m];
    if (SHEAR)
      gather_row_shear<true>(s, r, d.h, d.Ws, d.Fsp, X + r * (d.Fsp / 8) * cs + 8 * m, cs);
    else
      gather_row<true>(s, r, d.h, d.F, d.Fp, X + 8 * m, cs);
  }
}

// Sheared model, window tile of a wavefront step: feature k of window row rho
// at (k / 8) * 8 (rows + 8) + 8 rho + k % 8, so that consecutive rows are 16
// bytes apart and the A operand of window row dd of output row m is the tile
// started dd rows further.  wrow[rho] = (unit, unit row) of window row rho
// (unit -1: a zero row); the decoded pixels come from the units' sheared
// rings (unit u's row r at ring + 96 (u.ring_row + r)).
static __device__ __noinline__ void net_gather_win(const Unit* units, const uint8_t* ring,
                                                   int wrow_off, int step, int n_rows) {
  const NetSmem& t = net_smem();
  const int2* wrow = dec_at<int2>(wrow_off);
  const int h = t.d.h, Ws = t.d.Ws, nch = t.d.Fsp / 8, wr8 = 8 * (t.rows + 8);
  // window columns step - Ws .. step - 1: ring bytes from 3 ((step - Ws) mod 16);
  // feature k of a window row is byte k of that range
  const int c0 = step - Ws;
  const int b0 = 3 * (c0 & 15);
  uint16_t* X = dec_at<uint16_t>(t.pl.x);
  // one item per (window row, 8-feature chunk); rows past n_rows feed only
  // output rows that hold no pixel and are left as they are
  for (int it = threadIdx.x; it < n_rows * nch; it += blockDim.x) {
    const int rho = it / nch, kc = it - rho * nch;
    const int2 wr = wrow[rho];
    uint32_t w0 = 0u, w1 = 0u, w2 = 0u;
    int ca = 0, cb = 0;
    const int bs = b0 + 8 * kc;  // first ring byte of the chunk (<= 85)
    if (wr.x >= 0 && wr.y >= 0 && 8 * kc < 3 * Ws) {
      const Unit u = units[wr.x];
      const int j0 = c0 - (h + 1) * wr.y;  // image column of window column 0
      ca = j0 < 0 ? -j0 : 0;
      cb = min(Ws, u.Wu - j0);
      if (ca < cb) {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(
            ring + (long long)kRingRowBytes * (u.ring_row + wr.y) + (bs & ~3));
        w0 = ld_cg_u32(src);
        w1 = ld_cg_u32(src + 1);
        if ((bs & ~3) + 8 < kRingRowBytes) w2 = ld_cg_u32(src + 2);
      }
    }
    const uint32_t sh = 8u * (uint32_t)(bs & 3);
    const uint32_t lo = __funnelshift_r(w0, w1, sh), hi = __funnelshift_r(w1, w2, sh);
    uint32_t pk[4];
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
      float xv[2];
#pragma unroll
      for (int f = 0; f < 2; f++) {
        const int k = 8 * kc + e + f, q = k / 3;
        const float x = byte_input((e + f) < 4 ? lo : hi, (e + f) & 3);
        xv[f] = (k < 3 * Ws && q >= ca && q < cb) ? x : 0.f;
      }
      pk[e / 2] = pack_bf16(xv[0], xv[1]);
    }
    *reinterpret_cast<uint4*>(X + (size_t)kc * wr8 + (size_t)rho * 8) =
        make_uint4(pk[0], pk[1], pk[2], pk[3]);
  }
}

}  // namespace nlc
