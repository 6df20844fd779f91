// BF16 tensor-core building blocks: the layout of a model's BF16 weight tiles
// (shared by the codec's warp-level network and the trainer), PTX wrappers of
// tcgen05 / mbarrier / tensor memory, and the sheared first layer's features.
//
// Weight tiles are in the canonical no-swizzle K-major layout:
//   element (r, k) of an R x Kd matrix at
//   ((r/8) * (Kd/8) + k/8) * 64 + (r%8) * 8 + (k%8)   (BF16 elements)
// i.e. 8x8 core matrices of 128 contiguous bytes; the leading-dimension byte
// offset (next core matrix along K) is 128 and the stride-dimension byte
// offset (next 8-row group) is Kd/8 * 128.
//
// Network input: the integer 2v-255 (exact in BF16); the 1/255 of the scaled
// pixel value (2v-255)/255 is folded into the first-layer weights.
#pragma once

#include <cuda_bf16.h>

#include "nlc_common.cuh"
#include "nlc_model.cuh"

namespace nlc {

constexpr int kTileMax = 128;  // most pixels of a decoder tile
constexpr unsigned kMbarSpin = 1u << 22;

__host__ __device__ inline int align_up(int x, int a) { return (x + a - 1) / a * a; }

// Byte offsets of the BF16 weight tiles and of the FP32 biases behind them.
struct TcPlan {
  int w0, w1[kMaxR], w2[kMaxR], wh, w0s, bias;
};

__host__ __device__ inline TcPlan tc_plan(const Dims& d) {
  TcPlan p;
  int o = 0;
  p.w0 = o;
  o += d.C * d.Fp * 2;
  for (int r = 0; r < kMaxR; r++) {
    p.w1[r] = o;
    if (r < d.R) o += d.C * d.C * 2;
    p.w2[r] = o;
    if (r < d.R) o += d.C * d.C * 2;
  }
  p.wh = o;
  o += d.NOp * d.C * 2;
  // sheared first layer: h+1 tiles [C][16 ks(dd)], one per window row (top
  // first), each only over the window row's tap range
  p.w0s = o;
  if (d.shear) o += shear_tile_off(d, d.h + 1) * 2;
  p.bias = o;
  return p;
}

// BF16 weight tiles: the tap-ordered first layer, the residual blocks and the
// head (umma_plain_halves), then, for a sheared model, the sheared first layer.
__host__ __device__ inline size_t umma_plain_halves(const Dims& d) {
  return (size_t)d.C * d.Fp + 2 * (size_t)d.R * d.C * d.C + (size_t)d.NOp * d.C;
}
__host__ __device__ inline size_t umma_halves(const Dims& d) {
  return umma_plain_halves(d) + (d.shear ? (size_t)shear_tile_off(d, d.h + 1) : 0);
}
__host__ __device__ inline size_t bias_floats(const Dims& d) { return (size_t)d.C + 2 * (size_t)d.R * d.C + d.NOp; }

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__host__ __device__ __forceinline__ int umma_off(int r, int k, int Kd) {
  return ((r >> 3) * (Kd >> 3) + (k >> 3)) * 64 + (r & 7) * 8 + (k & 7);
}

// --- PTX wrappers --------------------------------------------------------
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version for tcgen05
  return d;                // base offset 0, relative LBO, no swizzle
}

// kind::f16 instruction descriptor: D FP32, A and B BF16, both K-major.
__device__ __forceinline__ uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t dtm, uint64_t ad, uint64_t bd, uint32_t idesc,
                                         uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtm),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* mbar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(mbar))
      : "memory");
}

__device__ __forceinline__ bool mbar_wait(uint64_t* mbar, uint32_t phase,
                                          unsigned limit = kMbarSpin) {
  for (unsigned it = 0; it < limit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(mbar)), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Non-blocking test of an mbarrier phase, at most `limit` times.
__device__ __forceinline__ bool mbar_test(uint64_t* mbar, uint32_t phase, unsigned limit) {
  for (unsigned it = 0; it < limit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(mbar)), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void fence_before_sync() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after_sync() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Two floats as a BF16 pair (a in the low half), each rounded to nearest even.
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
  return r;
}

// --- sheared first layer (Section 3.1, Fig. 5) ---------------------------------
// Window row dd (0 = top, h = the pixel's own row) of pixel (i, j) at
// wavefront step t = j + (h+1) i: unit row i - h + dd, the Ws = h(h+2)
// sheared columns t - Ws .. t - 1, i.e. image columns j0 .. j0 + Ws - 1 with
// j0 = j + (h+1)(h - dd) - Ws; feature 3q + c is channel c of window column
// q (2v - 255, 0 outside the unit), features 3 Ws .. Fsp - 1 are 0.  The
// sheared kernels give the taps of Eq. 3 their weights and every other
// window position 0, so the layer equals the masked one.

// Writes the Fsp features of one window row (3 Ws bytes at the realigned
// words al[], zero outside columns [ca, cb) of the window) as BF16 8-feature
// chunks: chunk kc to dst(kc).
template <class Dst>
__device__ __forceinline__ void shear_row_features(const uint32_t (&al)[12], int Ws, int Fsp,
                                                   int ca, int cb, bool ok, Dst dst) {
#pragma unroll
  for (int kc = 0; kc < 7; kc++) {  // Fsp <= 56
    if (kc >= Fsp / 8) break;
    uint32_t pk[4];
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
      float xv[2];
#pragma unroll
      for (int f = 0; f < 2; f++) {
        const int k = 8 * kc + e + f, q = k / 3;
        const int v = (int)((al[(k >> 2) < 12 ? (k >> 2) : 11] >> (8 * (k & 3))) & 0xFFu);
        xv[f] = (k < 3 * Ws && ok && q >= ca && q < cb) ? (float)(2 * v - 255) : 0.f;
      }
      pk[e / 2] = pack_bf16(xv[0], xv[1]);
    }
    *dst(kc) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
  }
}

// Bytes of a unit row in the sheared ring: the pixel of sheared column c is
// stored twice, at slots c mod 16 and c mod 16 + 16 (3 bytes each), so that
// the Ws <= 15 columns before any column are one contiguous byte range.
constexpr int kRingRowBytes = 96;

__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// 8 consecutive FP32 columns of this thread's TMEM lane, without waiting:
// the registers hold the values only after tmem_wait_ld() and tmem_touch().
__device__ __forceinline__ void tmem_ld8_nw(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// Orders every use of r after the preceding tmem_wait_ld (the registers pass
// through an asm that the compiler cannot move above the wait).
__device__ __forceinline__ void tmem_touch(uint32_t (&r)[8]) {
  asm volatile(""
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                 "+r"(r[6]), "+r"(r[7]));
}

cudaError_t launch_repack_umma(const Dims& d, const float* w, uint16_t* umma, float* bias,
                               cudaStream_t s);

}  // namespace nlc
