// Device helpers shared by the codec kernels: unit lookup, block scans, the
// rANS decoder of a coding group and the per-stream rANS encoder.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "nlc_common.cuh"
#include "nlc_kernels.cuh"
#include "nlc_model.cuh"

namespace nlc {

// ---------------------------------------------------------------------
// Shared helpers
// ---------------------------------------------------------------------
__device__ __forceinline__ int find_unit_px(const Unit* units, int n, long long q) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (units[mid].px_base <= q) lo = mid; else hi = mid - 1;
  }
  return lo;
}
__device__ __forceinline__ int find_unit_stream(const Unit* units, int n, int s) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (units[mid].stream_base <= s) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Barrier of the first nt threads of the CTA (nt a multiple of 32): the whole
// CTA's __syncthreads when nt is its size, else named barrier 1.
__device__ __forceinline__ void part_sync(int nt) {
  if (nt == (int)blockDim.x) __syncthreads();
  else asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory");
}

// Exclusive scan of one int per thread over the first nt threads of the CTA
// (nt a multiple of 32, only they call it); returns the exclusive prefix,
// writes the total to *total.
__device__ __forceinline__ long long block_excl_scan(long long v, long long* sh, long long* total,
                                                     int nt) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = nt >> 5;
  long long x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    long long t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  if (lane == 31) sh[warp] = x;
  part_sync(nt);
  if (warp == 0) {
    long long y = lane < nw ? sh[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      long long t = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += t;
    }
    if (lane < nw) sh[lane] = y;
  }
  part_sync(nt);
  long long excl = x - v + (warp > 0 ? sh[warp - 1] : 0);
  *total = sh[nw - 1];
  part_sync(nt);
  return excl;
}
__device__ __forceinline__ long long block_excl_scan(long long v, long long* sh, long long* total) {
  return block_excl_scan(v, sh, total, (int)blockDim.x);
}

// ---------------------------------------------------------------------
// rANS: warp-level decoder of one stream position and the per-stream
// encoder (byte-wise renormalisation, state in [2^23, 2^31)).
// ---------------------------------------------------------------------
// Coding groups of the table entry point: 16 lanes (half a warp) per pixel.
constexpr int kGW = 16;
constexpr int kGroups = kThreads / kGW;

// Decoder of one rANS stream position, held uniformly by a coding group.
// The next 8 stream bytes (a pixel consumes at most 6) are held in two
// registers; w2, w3 hold the 8 after them, from which the state written back
// for the stream's next pixel takes its 8 bytes.
struct GroupRansDec {
  uint32_t x;
  uint32_t lo, hi;  // bytes pos .. pos+7, little-endian packed
  uint32_t w2, w3;  // bytes pos+8 .. pos+15
  int used;
  int avail;        // bytes of the stream left from pos, at most 8
  bool bad;

  // w2, w3 from the three aligned words at (pos + 8) & ~3 (a word is read
  // only if it starts before the stream's end, so none outside its container).
  __device__ __forceinline__ void set_window(const uint32_t* v, unsigned long long pos) {
    const uint32_t sh = 8u * (uint32_t)((pos + 8ull) & 3ull);
    w2 = __funnelshift_r(v[0], v[1], sh);
    w3 = __funnelshift_r(v[1], v[2], sh);
  }
  // The 8 bytes at pos + used (used <= 6 for a valid pixel).
  __device__ __forceinline__ void next_bytes(uint32_t& n0, uint32_t& n1) const {
    if (used < 4) {
      const uint32_t s = 8u * (uint32_t)used;
      n0 = __funnelshift_r(lo, hi, s);
      n1 = __funnelshift_r(hi, w2, s);
    } else {
      const uint32_t s = 8u * (uint32_t)(used - 4);
      n0 = __funnelshift_r(hi, w2, s);
      n1 = __funnelshift_r(w2, w3, s);
    }
  }
  __device__ __forceinline__ void set_avail(unsigned long long pos, unsigned long long end) {
    avail = pos < end ? (int)min(end - pos, 8ull) : 0;
  }

  __device__ __forceinline__ void load_bytes(const uint8_t* base, unsigned long long pos,
                                             unsigned long long end) {
    lo = hi = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const unsigned long long p = pos + (unsigned long long)k;
      const uint32_t v = p < end ? (uint32_t)base[p] : 0u;
      if (k < 4) lo |= v << (8 * k);
      else hi |= v << (8 * (k - 4));
    }
    set_avail(pos, end);
    used = 0;
  }
  // With slot = x mod 2^16 and the decoded symbol's cum_s <= slot < cum_{s+1}:
  // x = freq (x >> 16) + slot - cum_s, then shift bytes in while x < 2^23.
  __device__ __forceinline__ void advance(uint32_t slot, uint32_t c0, uint32_t c1) {
    x = (c1 - c0) * (x >> 16) + slot - c0;
    for (int it = 0; it < 3 && x < kRansL; it++) {
      const uint32_t bt = used < 4 ? (lo >> (8 * used)) & 0xFFu
                                   : used < 8 ? (hi >> (8 * (used - 4))) & 0xFFu : 0u;
      if (used >= avail) bad = true;
      x = (x << 8) | bt;
      used++;
    }
    if (x < kRansL) bad = true;
  }
  // One symbol from an explicit table.
  template <int GW>
  __device__ __forceinline__ int decode_table(const TableScratch& ws, int lane) {
    const uint32_t slot = x & 0xFFFFu;
    const int s = table_search<GW>(ws, slot, lane);
    advance(slot, cum_at<GW>(ws, s), cum_at<GW>(ws, s + 1));
    return s;
  }
};

// Reciprocal of a symbol's frequency (packed start | freq << 16) for rans_put.
__device__ __forceinline__ uint32_t rans_recip(uint32_t e) { return 0xFFFFFFFFu / (e >> 16); }

// One rANS step: the bytes that leave the state go downwards from w.  The
// quotient x / f is umulhi(x, m) with m = floor((2^32 - 1) / f), or one more:
// m > 2^32 / f - 1 - 1/f, so the product is short by less than x / 2^31 <= 1
// (x < 2^31), and one comparison corrects it.  m does not depend on the state,
// so the states' chain holds no division.
__device__ __forceinline__ void rans_put(uint32_t e, uint32_t m, uint32_t& x, uint8_t*& w,
                                         bool store = true) {
  const uint32_t start = e & 0xFFFFu, f = e >> 16;
  const uint32_t xmax = ((kRansL >> 16) << 8) * f;
  while (x >= xmax) {
    --w;
    if (store) *w = (uint8_t)(x & 0xFFu);
    x >>= 8;
  }
  uint32_t q = __umulhi(x, m);
  uint32_t r = x - q * f;
  if (r >= f) {
    q++;
    r -= f;
  }
  x = (q << 16) + r + start;
}

// The final state, 4 bytes big-endian, in front of the emitted bytes.
__device__ __forceinline__ void rans_flush(uint32_t x, uint8_t*& w) {
  *--w = (uint8_t)x;
  *--w = (uint8_t)(x >> 8);
  *--w = (uint8_t)(x >> 16);
  *--w = (uint8_t)(x >> 24);
}

// Encodes symbols k = nsym-1 .. 0 (packed start | freq << 16) ending at
// slot_end by one thread; returns the stream length.  Layout: 4-byte
// big-endian final state, then the emitted bytes in reverse emission order.
// The next four symbols are read, and the present ones' reciprocals taken,
// ahead of the chain.
template <class Get>
__device__ __forceinline__ int rans_encode_stream(Get get, long long nsym, uint8_t* slot_end) {
  uint8_t* w = slot_end;
  uint32_t x = kRansL;
  constexpr int U = 4;
  long long k = nsym;
  uint32_t n[U] = {};
#pragma unroll
  for (int i = 0; i < U; i++)
    if (k > i) n[i] = get(k - 1 - i);
  for (; k >= U; k -= U) {
    uint32_t e[U], m[U];
#pragma unroll
    for (int i = 0; i < U; i++) {
      e[i] = n[i];
      if (k - U > i) n[i] = get(k - U - 1 - i);
    }
#pragma unroll
    for (int i = 0; i < U; i++) m[i] = rans_recip(e[i]);
#pragma unroll
    for (int i = 0; i < U; i++) rans_put(e[i], m[i], x, w);
  }
#pragma unroll
  for (int i = 0; i < U; i++)
    if (k > i) rans_put(n[i], rans_recip(n[i]), x, w);
  rans_flush(x, w);
  return (int)(slot_end - w);
}

// The same by a warp: the lanes read 32 symbols and take their reciprocals at
// once, then all follow the chain (lane 0 stores).
template <class Get>
__device__ __forceinline__ int rans_encode_warp(Get get, long long nsym, uint8_t* slot_end) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  uint8_t* w = slot_end;
  uint32_t x = kRansL;
  uint32_t n = lane < nsym ? get(nsym - 1 - lane) : 0x10000u;
  for (long long k = nsym; k > 0; k -= 32) {
    const uint32_t e = n, m = rans_recip(e);
    n = k - 32 > lane ? get(k - 33 - lane) : 0x10000u;
    const int c = k < 32 ? (int)k : 32;
    if (c == 32) {
#pragma unroll 8
      for (int i = 0; i < 32; i++)
        rans_put(__shfl_sync(full, e, i), __shfl_sync(full, m, i), x, w, lane == 0);
    } else {
      for (int i = 0; i < c; i++)
        rans_put(__shfl_sync(full, e, i), __shfl_sync(full, m, i), x, w, lane == 0);
    }
  }
  if (lane == 0) rans_flush(x, w);
  else w -= 4;
  return (int)(slot_end - w);
}

__device__ __forceinline__ int unit_streams(const Unit& U, int layout) {
  return layout == 1 ? U.Hu : 1;
}

inline int grid_for(long long work, int per, int cap) {
  long long g = (work + per - 1) / per;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}

}  // namespace nlc
