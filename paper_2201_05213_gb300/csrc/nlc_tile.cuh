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

// Encodes symbols k = nsym-1 .. 0 (packed start | freq << 16) ending at
// slot_end; returns the stream length.  Layout: 4-byte big-endian final
// state, then the emitted bytes in reverse emission order.
template <class Get>
__device__ __forceinline__ int rans_encode_stream(Get get, long long nsym, uint8_t* slot_end) {
  uint8_t* w = slot_end;
  uint32_t x = kRansL;
  for (long long k = nsym - 1; k >= 0; k--) {
    const uint32_t e = get(k);
    const uint32_t start = e & 0xFFFFu, f = e >> 16;
    const uint32_t xmax = ((kRansL >> 16) << 8) * f;
    while (x >= xmax) {
      *--w = (uint8_t)(x & 0xFFu);
      x >>= 8;
    }
    x = ((x / f) << 16) + (x % f) + start;
  }
  *--w = (uint8_t)x;
  *--w = (uint8_t)(x >> 8);
  *--w = (uint8_t)(x >> 16);
  *--w = (uint8_t)(x >> 24);
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
