// Training launchers (maximum likelihood, Eq. 2): loss and gradient of the
// mean code length in bits per dimension, and the Adam update.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "nlc_common.cuh"

namespace nlc {

#ifdef __CUDACC__
// Sums into a CTA's gradient slot, every element always by the same thread.
// They are reductions, so that no thread waits for the old value, except for
// sums so small that the memory's adder would lose them: it takes subnormal
// operands and results as zero.  A sum of at least 2^-102 has a rounding unit
// of at least 2^-125, so such a loss stays below its rounding (and a difference
// of two such sums is a multiple of 2^-126); smaller ones are added by the
// thread, and zeros, which would flush a subnormal old value, not at all.
// (Flushed, the gradient of outputs scaled by 1e-39 was wrong by 27 %.)
constexpr float kSlotTiny = 0x1p-102f;
__device__ __forceinline__ void slot_red(float* p, float v) {
  asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
__device__ __forceinline__ void slot_red2(float* p, float a, float b) {  // p: 8-byte aligned
  asm volatile("red.relaxed.gpu.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a), "f"(b)
               : "memory");
}
// Any sum (the callers take slot_red where all of theirs are large enough).
__device__ __forceinline__ void slot_add(float* p, float v) {
  if (!(fabsf(v) < kSlotTiny)) {
    slot_red(p, v);
  } else if (v != 0.f) {
    asm volatile(
        "{\n.reg .f32 t;\nld.relaxed.gpu.global.f32 t, [%0];\nadd.rn.f32 t, t, %1;\n"
        "st.relaxed.gpu.global.f32 [%0], t;\n}\n" ::"l"(p), "f"(v) : "memory");
  }
}
#endif

size_t train_ws_bytes(const Dims& d, long long n_px, int sm_count);
// FP32 SIMT path.  dparams == nullptr: loss (bits per dimension) and its
// gradient; else the gradient of sum(dparams * network outputs) (loss
// untouched).
cudaError_t launch_loss_grad(const Dims& d, const float* wt, const uint8_t* batch, int N, int H,
                             int W, const float* dparams, float* loss, float* grad, void* ws,
                             int sm_count, cudaStream_t s);
// Sums per-CTA gradient slots (and loss partials, if part_l and loss are
// non-null) in a fixed order.
cudaError_t launch_reduce_grad(const float* part_g, const float* part_l, int nblk, int n_w, int ldw,
                               long long n_px, float* grad, float* loss, cudaStream_t s);
// Whether the FP32 SIMT training kernel's tiles fit in one CTA.
bool simt_train_fits(const Dims& d);
// BF16 tensor-core path (tcgen05), same contract; fits: whether the model's
// tiles fit in one CTA's shared memory.
bool tc_train_fits(const Dims& d);
size_t tc_train_ws_bytes(const Dims& d, long long n_px, int sm_count);
cudaError_t launch_tc_train(const Dims& d, const uint16_t* umma, const float* bias,
                            const uint8_t* batch, int N, int H, int W, const float* dparams,
                            float* loss, float* grad, void* ws, int sm_count, int* status,
                            cudaStream_t s);
cudaError_t launch_adam(float* w, const float* g, float* m, float* v, int n, float lr, float b1,
                        float b2, float eps, long long t, cudaStream_t s);

}  // namespace nlc
