// The local network over all pixels at once: the encoder's first stage (the
// frequencies of every symbol, with the decoder's own device code) and the
// forward entry point (network outputs, model code length).
#include "nlc_f32.cuh"
#include "nlc_px.cuh"

namespace nlc {

// Warps per CTA of the BF16 kernel.  Four per scheduler at 128 registers (up to
// 32 bytes spilled) hide the chains better than three at 168: 4.9 against 5.3 ms
// for the tables of 12.6 M pixels; 14 leave the schedulers uneven (5.6 ms).
constexpr int kPxWarps = 16;

struct PxArgs {
  DeviceModel m;
  const Unit* units;
  int n_units;
  long long n_px;
  uint32_t* stage;  // encoder: start | freq << 16 per symbol
  float* params;    // forward: network outputs and / or code lengths
  float* bits;
};

// Symbols' (start, freq) of one pixel, channel by channel, given its
// parameters P(p, i); the lanes of a quad return the same values.
template <int CH, int KI, class Param>
__device__ __forceinline__ uint32_t enc_channel(Param P, int K, int q, const int (&v)[3],
                                                QuadState<KI>& st) {
  QuadChan<KI> o;
  quad_channel<CH, KI>(P, K, q, st, v[0], v[1], o);
  uint32_t c0, c1;
  quad_pair<KI>(o, v[CH], c0, c1);
  if (CH < 2) quad_observe<KI>(o, K, q, v[CH], st);
  return c0 | ((c1 - c0) << 16);
}

template <int NT8, int KI, bool ENC>
__global__ void __launch_bounds__(32 * kPxWarps, 1) px_bf16_kernel(PxArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  const Dims& d = a.m.d;
  const PxPlan pl = px_plan(d);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int g = lane >> 2, q = lane & 3, K = d.K;
  float* bias = reinterpret_cast<float*>(smem + pl.bias);
  {
    const uint4* src = reinterpret_cast<const uint4*>(a.m.w.umma);
    uint4* dst = reinterpret_cast<uint4*>(smem);
    for (int i = threadIdx.x; i < a.m.w.umma_halves / 8; i += blockDim.x) dst[i] = src[i];
    const int nb = (int)bias_floats(d);
    for (int i = threadIdx.x; i < nb; i += blockDim.x) bias[i] = a.m.w.bias[i];
  }
  unsigned char* own = smem + pl.warp0 + warp * pl.per_warp;
  uint16_t* X = reinterpret_cast<uint16_t*>(own);
  PxSlot* slots = reinterpret_cast<PxSlot*>(own + pl.x_bytes);
  const uint32_t sb = smem_u32(smem), xa = smem_u32(own);
  const float* bh = bias + 8 * NT8 * (1 + 2 * d.R);
  uint32_t* row = reinterpret_cast<uint32_t*>(smem + pl.row);
  float* hbias = reinterpret_cast<float*>(smem + pl.hbias);
  static_assert(PxHead<KI>::kBytes <= kPxTables, "the tables' place");
  __syncthreads();
  px_head_tables<NT8, KI>(d, bh, row, hbias);
  __syncthreads();
  const uint32_t wh = sb + (uint32_t)pl.wh;
  const long long groups = (a.n_px + kPxRows - 1) / kPxRows;
  int hint = 0;
  for (long long grp = (long long)blockIdx.x * nw + warp; grp < groups;
       grp += (long long)gridDim.x * nw) {
    const long long q0 = grp * kPxRows;
    hint = px_slots(a.units, a.n_units, a.n_px, q0, hint, slots);
    {
      const int r = lane >> 3;
      constexpr int cs = 8 * kPxRows;
      if (r <= d.h)
        for (int m = lane & 7; m < kPxRows; m += 8) {
          const PxSlot s = slots[m];
          if (d.shear)
            gather_row_shear<false>(s, r, d.h, d.Ws, d.Fsp, X + r * (d.Fsp / 8) * cs + 8 * m, cs);
          else
            gather_row<false>(s, r, d.h, d.F, d.Fp, X + 8 * m, cs);
        }
    }
    __syncwarp();
    uint32_t f[NT8 / 2][4];
    px_hidden<NT8>(d, pl, sb, xa, bias, f);
    // the lane's pixels: rows g and g + 8
    int v[2][3] = {};
    if (ENC || a.bits) {
#pragma unroll
      for (int r = 0; r < 2; r++) {
        const uint8_t* px = slots[g + 8 * r].px;
#pragma unroll
        for (int c = 0; c < 3; c++) v[r][c] = __ldg(px + c);
      }
    }
    if constexpr (ENC) {
      QuadState<KI> st[2];
      uint32_t e[2][3];
      {
        float w[2][3 * KI];
        px_head<NT8, KI, 0>(wh, row, hbias, f, w);
#pragma unroll
        for (int r = 0; r < 2; r++) {
          auto P = [&](int p, int i) { return w[r][(p == 0 ? 0 : p == 1 ? 1 : 2) * KI + i]; };
          quad_init<KI>(P, K, q, st[r]);
          e[r][0] = enc_channel<0, KI>(P, K, q, v[r], st[r]);
        }
        px_head<NT8, KI, 1>(wh, row, hbias, f, w);
#pragma unroll
        for (int r = 0; r < 2; r++)
          e[r][1] = enc_channel<1, KI>(
              [&](int p, int i) { return w[r][(p == 2 ? 0 : p == 5 ? 1 : 2) * KI + i]; }, K, q,
              v[r], st[r]);
      }
      float w[2][4 * KI];
      px_head<NT8, KI, 2>(wh, row, hbias, f, w);
#pragma unroll
      for (int r = 0; r < 2; r++)
        e[r][2] = enc_channel<2, KI>(
            [&](int p, int i) {
              return w[r][(p == 3 ? 0 : p == 6 ? 1 : p == 8 ? 2 : 3) * KI + i];
            },
            K, q, v[r], st[r]);
      // lane q < 3 writes channel q: 24 lanes, 96 consecutive bytes
#pragma unroll
      for (int r = 0; r < 2; r++)
        if (q < 3 && q0 + g + 8 * r < a.n_px)
          a.stage[3 * (q0 + g + 8 * r) + q] = q == 0 ? e[r][0] : q == 1 ? e[r][1] : e[r][2];
    } else {
      const long long out[2] = {slots[g].out, slots[g + 8].out};
      const bool in[2] = {q0 + g < a.n_px, q0 + g + 8 < a.n_px};
      if (a.params) {
        const int NO = d.NO;
        const uint32_t wr = wh + (lane & 7) * 16u;
        // the caller's buffer is an array of floats: pairs of them only where it
        // starts on 8 bytes (NO and col are even)
        const bool pairs = (reinterpret_cast<uintptr_t>(a.params) & 7) == 0;
#pragma unroll 1
        for (int j = 0; 8 * j < NO; j++) {
          uint32_t w[NT8];
          load_b<NT8 / 2>(wr + (uint32_t)j * (128u * NT8), w);
          float c[4];
#pragma unroll
          for (int s = 0; s < NT8 / 2; s++) mma_step(s, c, f[s], w[2 * s], w[2 * s + 1]);
          const int col = 8 * j + 2 * q;
          if (col < NO) {
            const float2 b = *reinterpret_cast<const float2*>(bh + col);
#pragma unroll
            for (int r = 0; r < 2; r++) {
              if (!in[r]) continue;
              float* o = a.params + out[r] * NO + col;
              const float v0 = __fadd_rn(c[2 * r], b.x), v1 = __fadd_rn(c[2 * r + 1], b.y);
              if (pairs) {
                *reinterpret_cast<float2*>(o) = make_float2(v0, v1);
              } else {
                o[0] = v0;
                o[1] = v1;
              }
            }
          }
        }
      }
      if (a.bits) {
        QuadState<KI> st[2];
        {
          float w[2][3 * KI];
          px_head<NT8, KI, 0>(wh, row, hbias, f, w);
#pragma unroll
          for (int r = 0; r < 2; r++) {
            auto P = [&](int p, int i) { return w[r][(p == 0 ? 0 : p == 1 ? 1 : 2) * KI + i]; };
            quad_init<KI>(P, K, q, st[r]);
            quad_loglik<0, KI>(P, K, q, v[r], st[r].lw);
          }
          px_head<NT8, KI, 1>(wh, row, hbias, f, w);
#pragma unroll
          for (int r = 0; r < 2; r++)
            quad_loglik<1, KI>(
                [&](int p, int i) { return w[r][(p == 2 ? 0 : p == 5 ? 1 : 2) * KI + i]; }, K, q,
                v[r], st[r].lw);
        }
        float w[2][4 * KI];
        px_head<NT8, KI, 2>(wh, row, hbias, f, w);
#pragma unroll
        for (int r = 0; r < 2; r++) {
          quad_loglik<2, KI>(
              [&](int p, int i) {
                return w[r][(p == 3 ? 0 : p == 6 ? 1 : p == 8 ? 2 : 3) * KI + i];
              },
              K, q, v[r], st[r].lw);
          const float b = quad_bits<KI>(st[r].lw, K, q);
          if (q == 0 && in[r]) a.bits[out[r]] = b;
        }
      }
    }
    __syncwarp();  // the slots are read before the next pass writes them
  }
}

// FP32 models: a CTA per 64 pixels (nlc_f32.cuh), then a quad per pixel.
template <bool ENC>
__global__ void __launch_bounds__(kThreads, 1) px_f32_kernel(PxArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  const Dims& d = a.m.d;
  float* sm = reinterpret_cast<float*>(smem);
  const F32Plan pl = f32_plan(d);
  PxSlot* slots = reinterpret_cast<PxSlot*>(sm + pl.end);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int K = d.K, NO = d.NO;
  for (int i = threadIdx.x; i < a.m.w.simt_floats; i += blockDim.x) sm[i] = a.m.w.simt[i];
  const long long ntiles = (a.n_px + kF32Rows - 1) / kF32Rows;
  int hint = 0;
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const long long q0 = tile * kF32Rows;
    const int n = (int)min((long long)kF32Rows, a.n_px - q0);
    if (warp < kF32Rows / kPxRows)
      hint = px_slots(a.units, a.n_units, a.n_px, q0 + kPxRows * warp, hint,
                      slots + kPxRows * warp);
    __syncthreads();
    f32_gather<false>(slots, n, d, sm);
    __syncthreads();
    f32_run(d, sm, n);
    const float* P0 = sm + pl.u;
    if (!ENC && a.params) {
      for (int s = warp; s < n; s += kWarps)
        for (int k = lane; k < NO; k += 32)
          a.params[slots[s].out * NO + k] = P0[(size_t)s * d.ldP + k];
    }
    if (ENC || a.bits) {
      const int q = lane & 3;
      const bool valid = kQuads * warp + (lane >> 2) < n;
      const int s = valid ? kQuads * warp + (lane >> 2) : n - 1;
      const uint8_t* px = slots[s].px;
      const int v[3] = {px[0], px[1], px[2]};
      const float* row = P0 + (size_t)s * d.ldP + q;
      auto P = [&](int p, int i) { return row[p * K + 4 * i]; };
      auto code = [&](auto ki) {
        constexpr int KI = decltype(ki)::value;
        QuadState<KI> st;
        quad_init<KI>(P, K, q, st);
        if (ENC) {
          const uint32_t e0 = enc_channel<0, KI>(P, K, q, v, st);
          const uint32_t e1 = enc_channel<1, KI>(P, K, q, v, st);
          const uint32_t e2 = enc_channel<2, KI>(P, K, q, v, st);
          if (valid && q < 3) a.stage[3 * (q0 + s) + q] = q == 0 ? e0 : q == 1 ? e1 : e2;
        } else {
          quad_loglik<0, KI>(P, K, q, v, st.lw);
          quad_loglik<1, KI>(P, K, q, v, st.lw);
          quad_loglik<2, KI>(P, K, q, v, st.lw);
          const float b = quad_bits<KI>(st.lw, K, q);
          if (valid && q == 0) a.bits[slots[s].out] = b;
        }
      };
      switch ((K + 3) / 4) {
        case 1: code(IntC<1>{}); break;
        case 2: code(IntC<2>{}); break;
        case 3: code(IntC<3>{}); break;
        default: code(IntC<4>{}); break;
      }
    }
    __syncthreads();
  }
}

template <int NT8, bool ENC>
static const void* px_fn_k(int K) {
  switch ((K + 3) / 4) {
    case 1: return (const void*)px_bf16_kernel<NT8, 1, ENC>;
    case 2: return (const void*)px_bf16_kernel<NT8, 2, ENC>;
    case 3: return (const void*)px_bf16_kernel<NT8, 3, ENC>;
    default: return (const void*)px_bf16_kernel<NT8, 4, ENC>;
  }
}
template <bool ENC>
static const void* px_fn(const Dims& d) {
  switch (d.C / 8) {
    case 2: return px_fn_k<2, ENC>(d.K);
    case 4: return px_fn_k<4, ENC>(d.K);
    case 6: return px_fn_k<6, ENC>(d.K);
    default: return px_fn_k<8, ENC>(d.K);
  }
}

template <bool ENC>
static cudaError_t launch_px(const PxArgs& a, int sm_count, cudaStream_t s) {
  const Dims& d = a.m.d;
  const void* fn;
  int threads, grid;
  size_t smem;
  if (d.prec == PREC_BF16) {
    fn = px_fn<ENC>(d);
    const PxPlan pl = px_plan(d);
    // every SM first, then up to kPxWarps warps each (fewer where a large
    // model's weights leave no room for their tiles)
    const long long groups = (a.n_px + kPxRows - 1) / kPxRows;
    grid = grid_for(groups, 1, sm_count);
    const int fit = (227 * 1024 - pl.warp0) / pl.per_warp;
    const int cap = fit < kPxWarps ? fit : kPxWarps;
    if (cap < 1) return cudaErrorInvalidConfiguration;
    const int nw = grid_for(groups, grid, cap);
    threads = 32 * nw;
    smem = (size_t)(pl.warp0 + nw * pl.per_warp);
  } else {
    fn = (const void*)px_f32_kernel<ENC>;
    grid = grid_for((a.n_px + kF32Rows - 1) / kF32Rows, 1, sm_count);
    threads = kThreads;
    smem = (size_t)f32_plan(d).end * 4 + sizeof(PxSlot) * kF32Rows;
  }
  if (smem > kMaxSmem) return cudaErrorInvalidValue;
  cudaError_t e = allow_smem(fn);
  if (e != cudaSuccess) return e;
  PxArgs b = a;
  void* args[] = {&b};
  return cudaLaunchKernel(fn, dim3(grid), dim3(threads), args, smem, s);
}

cudaError_t launch_enc_tables(const DeviceModel& m, const CodecBufs& b, int sm_count,
                              cudaStream_t s) {
  return launch_px<true>(PxArgs{m, b.units, b.n_units, b.n_px, b.stage, nullptr, nullptr}, sm_count,
                         s);
}

cudaError_t launch_forward(const DeviceModel& m, const CodecBufs& b, float* params, float* bits,
                           int sm_count, cudaStream_t s) {
  if (b.n_px == 0) return cudaSuccess;
  return launch_px<false>(PxArgs{m, b.units, b.n_units, b.n_px, nullptr, params, bits}, sm_count,
                          s);
}

}  // namespace nlc
