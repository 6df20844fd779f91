// The wavefront decoder's device code (Algorithm 1, Section 3): the
// persistent cooperative kernel and its coding functions.  Included by
// nlc_decode.cu (the launchers and the plain build) and nlc_decode_prof.cu
// (the instrumented build behind nlc_decode_profile), so that each
// compilation unit holds one build: in one unit together, ptxas gave the
// plain build's coding function and step loop more spills.
#pragma once
#include "nlc_f32.cuh"
#include "nlc_mma.cuh"
#include "nlc_quad.cuh"
#include "nlc_tile.cuh"

namespace nlc {

// ---------------------------------------------------------------------
// Decoder: persistent cooperative kernel.  Step t decodes, for every unit,
// the pixels of its front (wavefront: j = tau - (h+1) i, Section 3; raster:
// one pixel).  The step's pixels are split evenly across the CTAs; each CTA
// runs gather -> network -> per-pixel CDF + rANS for its share, then all
// CTAs meet at a grid barrier before step t+1.
// ---------------------------------------------------------------------
struct DecodeArgs {
  DeviceModel m;
  const Unit* units;
  int n_units;
  int layout, sched, T;
  const uint8_t* in;
  StreamRec* st;
  unsigned* bar;
  int* status;
  unsigned long long* prof;  // optional per-phase cycle counters
  unsigned long long* times;  // optional: [0] start, [t + 1] end of step t (ns)
  long long n_times;
  unsigned long long seed;    // sampler only
  uint8_t* ring;              // sheared wavefront decoder: the units' sheared rings
  unsigned spin_limit;        // polls of the grid barrier before a timeout
  unsigned mma_limit;         // polls of a network layer's exchange before a timeout
  int rows;                   // pixels per tile
};

// Threads of the decoder's CTA: the BF16 network runs on 16 warps, the FP32
// network on 8.
template <int PREC>
__host__ __device__ constexpr int decode_threads() { return PREC == PREC_BF16 ? 512 : kThreads; }

// Shared memory of a decoder CTA.
struct DecSmem {
  NetSmem net;            // BF16 network
  float* f32;             // FP32 network
  const float* P;         // head outputs of the tile's pixels
  int ldp;                // and their row stride
  WarpScratch* ws;        // one per warp (whole-warp coding)
  DecSlot* slots;         // the tile's pixels
  StreamRec* rec;         // their stream records
  uint32_t* win;          // per pixel, the 12 stream bytes from pos + 8, word-aligned
  int* prow;              // sheared wavefront decoder: output row of the tile's pixel s
  int* rofs;              // sheared wavefront decoder: ring byte offset of the tile's pixel s
  int2* wrow;             // sheared wavefront decoder: (unit, unit row) of window row rho
  long long* sh;
  long long* pc;          // 16 profiling accumulators (thread 0 only)
  int* pre;               // front prefix of the units
  int* flag;
};

// Carves the shared memory of a tile of `rows` pixels; returns its bytes.
// win: the sheared model's wavefront decoder.  The whole-warp groups' scratch
// lies behind the first 16 head-output rows of the BF16 tile region, which a
// tile of at most 16 pixels leaves free (not in the window tile, whose output
// rows are spread out).
__host__ __device__ inline size_t dec_carve(const Dims& d, unsigned char* smem, int n_pre, int rows,
                                            bool win, DecSmem* t) {
  size_t off;
  unsigned char* ws;
  DecSmem z{};
  if (d.prec == PREC_BF16) {
    const NetPlan p = net_plan(d, rows, win);
    off = (size_t)p.end;
    ws = win ? smem + off : smem + p.x + kNetWarps * net_ldp(d) * 4;
    if (win) off += sizeof(WarpScratch) * kNetWarps;
    z.P = reinterpret_cast<const float*>(smem + p.x);
    z.ldp = net_ldp(d);
  } else {
    const F32Plan p = f32_plan(d);
    z.f32 = reinterpret_cast<float*>(smem);
    z.P = z.f32 + p.u;
    z.ldp = d.ldP;
    off = ((size_t)p.end * 4 + 15) & ~(size_t)15;
    ws = smem + off;
    off += sizeof(WarpScratch) * (decode_threads<PREC_FP32>() / 32);
  }
  off = (off + 15) & ~(size_t)15;
  auto take = [&](size_t bytes) {
    unsigned char* q = smem + off;
    off += (bytes + 15) & ~(size_t)15;
    return q;
  };
  z.ws = reinterpret_cast<WarpScratch*>(ws);
  z.slots = reinterpret_cast<DecSlot*>(take(sizeof(DecSlot) * rows));
  z.rec = reinterpret_cast<StreamRec*>(take(sizeof(StreamRec) * rows));
  z.win = reinterpret_cast<uint32_t*>(take(4 * sizeof(uint32_t) * rows));
  if (win) {
    z.wrow = reinterpret_cast<int2*>(take(sizeof(int2) * (rows + 8)));
    z.prow = reinterpret_cast<int*>(take(sizeof(int) * rows));
    z.rofs = reinterpret_cast<int*>(take(sizeof(int) * rows));
  }
  z.sh = reinterpret_cast<long long*>(take(sizeof(long long) * 33));
  z.pc = reinterpret_cast<long long*>(take(sizeof(long long) * 16));
  z.pre = reinterpret_cast<int*>(take(sizeof(int) * (n_pre + 1 + 4)));
  z.flag = z.pre + n_pre + 1;
  if (t) *t = z;
  return off;
}

// Stores a decoded pixel in its unit's ring row at the byte offset rofs
// that the tile's schedule computed (slots tau mod 16 and tau mod 16 + 16 of
// its sheared column tau).
__device__ __forceinline__ void ring_put(const DecodeArgs& a, int rofs, const int (&v)[3]) {
  uint8_t* r = a.ring + rofs;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    r[c] = (uint8_t)v[c];
    r[48 + c] = (uint8_t)v[c];
  }
}

// A pixel's stream state from its record; the positions are read again when
// the pixel is done.
__device__ __forceinline__ GroupRansDec load_rec(const StreamRec* r) {
  GroupRansDec dec;
  const uint4 q = *reinterpret_cast<const uint4*>(r);
  const ulonglong2 pe = *reinterpret_cast<const ulonglong2*>(&r->pos);
  dec.x = q.x;
  dec.lo = q.y;
  dec.hi = q.z;
  dec.set_avail(pe.x, pe.y);
  dec.w2 = dec.w3 = 0;
  dec.used = 0;
  dec.bad = false;
  return dec;
}

// Writes the tile's pixel s back (one lane of its group): the pixel, and for
// the decoder its stream's record and the end-of-stream check.
template <bool SAMPLE, bool SHEAR>
__device__ __forceinline__ void put_pixel(const DecodeArgs& a, const DecSmem& t, int s,
                                          const int (&v)[3], GroupRansDec& dec) {
  const DecSlot ps = t.slots[s];
  ps.px[0] = (uint8_t)v[0];
  ps.px[1] = (uint8_t)v[1];
  ps.px[2] = (uint8_t)v[2];
  if (SHEAR) ring_put(a, t.rofs[s], v);
  if (SAMPLE) return;
  const ulonglong2 pe = *reinterpret_cast<const ulonglong2*>(&t.rec[s].pos);
  dec.set_window(t.win + 4 * s, pe.x);
  const unsigned long long np = pe.x + (unsigned long long)dec.used;
  uint32_t n0, n1;
  dec.next_bytes(n0, n1);
  StreamRec* r = a.st + ps.stream;
  *reinterpret_cast<uint4*>(r) = make_uint4(dec.x, n0, n1, 0u);
  r->pos = np;
  if (dec.bad || (ps.unit < 0 && (dec.x != kRansL || np != pe.y)))
    set_status(a.status, ST_CORRUPT);
}

// Counter of the sampler's uniforms for the tile's pixel s: 3 times its index.
__device__ __forceinline__ unsigned long long sample_key(const DecodeArgs& a, const DecSlot& ps) {
  const Unit& U = a.units[ps.unit & 0x7FFFFFFF];
  return 3ull * (((((unsigned long long)U.image << 21) + (unsigned long long)(U.y0 + ps.i)) << 21) +
                 (unsigned long long)(U.x0 + ps.j));
}

// Cycle counters of thread 0 (see nlc_decode_profile).
template <bool PROF>
struct Ticker {
  long long* pc;
  long long ck;
  __device__ __forceinline__ explicit Ticker(long long* p)
      : pc(PROF && p != nullptr && threadIdx.x == 0 ? p : nullptr), ck(0) {
    if (PROF && pc) ck = clock64();
  }
  __device__ __forceinline__ void operator()(int slot) {
    if (PROF && pc) {
      const long long n = clock64();
      pc[slot] += n - ck;
      ck = n;
    }
  }
};

// Codes the tile's pixels with whole warps, pixel s by warp s mod NW (the
// lowest latency per pixel; for tiles of at most NW pixels): per pixel, the
// R, G|r, B|r,g symbols from its stream (SAMPLE: from the counter-based
// uniforms by inverse CDF, Section 5).  The pixels' stream records are in
// t.rec (visible to the warp), their windows are being copied to t.win by the
// warp's lanes.
template <int NW, bool SAMPLE, bool SHEAR, bool PROF>
__device__ __noinline__ void code_wide(const DecodeArgs& a, const DecSmem& t, int n,
                                       long long* pc) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int K = a.m.d.K;
  WarpScratch& ws = t.ws[warp];
  Ticker<PROF> tick(pc);
  for (int s = warp; s < n; s += NW) {
    GroupRansDec dec;
    unsigned long long key = 0;
    if (SAMPLE) key = sample_key(a, t.slots[s]);
    else dec = load_rec(t.rec + s);
    if (PROF && tick.pc) tick.pc[12] += 1;
    CompState cs;
    comp_init<32>(t.P + (size_t)(SHEAR ? t.prow[s] : s) * t.ldp, K, lane, cs);
    int v[3] = {0, 0, 0};
    for (int ch = 0; ch < 3; ch++) {
      int nact;
      const float mloc = channel_setup<32>(cs, K, ch, v[0], v[1], lane, ws, nact);
      tick(8);
      const uint32_t slot =
          SAMPLE ? (uint32_t)(splitmix64_at(a.seed, key + ch) >> 48) : (dec.x & 0xFFFFu);
      uint32_t lo, hi;
      v[ch] = cdf_search<32>(ws, nact, slot, lane, lo, hi);
      tick(9);
      if (!SAMPLE) dec.advance(slot, lo, hi);
      tick(10);
      if (ch < 2) comp_observe(cs, K, ch, mloc, v[ch], lane);
      __syncwarp();
      tick(11);
    }
    if (!SAMPLE) {
      cp_async_wait_all();  // the window copies of the warp's lanes
      __syncwarp();
    }
    if (lane == 0) put_pixel<SAMPLE, SHEAR>(a, t, s, v, dec);
  }
}

// The same by quads, eight pixels per warp: warp w codes the tile's pixels
// 8 (w + NW j) .. + 7 (see nlc_quad.cuh).
template <int KI, int NW, bool SAMPLE, bool SHEAR, bool PROF>
__device__ __noinline__ void code_quads(const DecodeArgs& a, const DecSmem& t, int n,
                                        long long* pc) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int q = lane & 3;
  const int K = a.m.d.K;
  Ticker<PROF> tick(pc);
  for (int s0 = kQuads * warp; s0 < n; s0 += kQuads * NW) {
    const bool valid = s0 + (lane >> 2) < n;
    const int s = valid ? s0 + (lane >> 2) : n - 1;  // an idle quad shadows the last pixel
    GroupRansDec dec;
    unsigned long long key = 0;
    if (SAMPLE) key = sample_key(a, t.slots[s]);
    else dec = load_rec(t.rec + s);
    if (PROF && tick.pc) tick.pc[12] += 1;
    const float* row = t.P + (size_t)(SHEAR ? t.prow[s] : s) * t.ldp + q;
    auto P = [&](int p, int i) { return row[p * K + 4 * i]; };
    QuadState<KI> st;
    quad_init<KI>(P, K, q, st);
    int v[3] = {0, 0, 0};
    auto channel = [&](auto chc) {
      constexpr int CH = decltype(chc)::value;
      QuadChan<KI> o;
      quad_channel<CH, KI>(P, K, q, st, v[0], v[1], o);
      tick(8);
      const uint32_t slot =
          SAMPLE ? (uint32_t)(splitmix64_at(a.seed, key + CH) >> 48) : (dec.x & 0xFFFFu);
      uint32_t lo, hi;
      v[CH] = quad_search<KI>(o, slot, q, lo, hi);
      tick(9);
      if (!SAMPLE) dec.advance(slot, lo, hi);
      tick(10);
      if (CH < 2) quad_observe<KI>(o, K, q, v[CH], st);
      tick(11);
    };
    channel(IntC<0>{});
    channel(IntC<1>{});
    channel(IntC<2>{});
    if (!SAMPLE) {
      cp_async_wait_all();  // the window copies of the warp's lanes
      __syncwarp();
    }
    if (q == 0 && valid) put_pixel<SAMPLE, SHEAR>(a, t, s, v, dec);
  }
}

// SHEAR: the sheared model's wavefront decoder (Section 3.1): decoded pixels
// also go to per-unit sheared rings, and each tile's context is one window
// tile of (unit, row) rows read from the rings, every unit's piece of the
// front preceded by h halo rows, with the first layer's MMAs reading the
// window rows of output row m at rows m .. m + h.
// PROF: the instrumented build behind nlc_decode_profile.  The cycle
// counters' state, live through the whole step loop even while profiling is
// off, cost the uninstrumented decoder 7 % (register spills), so only
// launches with a counter buffer run this instantiation.
template <int PREC, bool SAMPLE, bool SHEAR, bool PROF>
__global__ void __launch_bounds__(decode_threads<PREC>(), 1) decode_kernel(DecodeArgs a) {
  constexpr int NT = decode_threads<PREC>(), NW = NT / 32;
  extern __shared__ __align__(128) unsigned char smem[];
  const Dims& d = a.m.d;
  const int rows = a.rows;
  DecSmem t;
  dec_carve(d, smem, a.n_units, rows, SHEAR, &t);
  if constexpr (PREC == PREC_BF16) {
    t.net = net_carve(d, smem, rows, SHEAR);
    t.net.limit = a.mma_limit;
    if (threadIdx.x == 0) net_setup(t.net);
    net_load_weights(d, a.m.w, t.net);
  } else {
    for (int i = threadIdx.x; i < a.m.w.simt_floats; i += blockDim.x) t.f32[i] = a.m.w.simt[i];
  }
  if (threadIdx.x == 0) t.flag[0] = 0;
  if (threadIdx.x < 16) t.pc[threadIdx.x] = 0;
  __syncthreads();
  // step end times: CTA 0 stamps each step when the grid barrier after it
  // releases (every CTA has finished it); every CTA stamps the last step's end
  const bool stamp = a.times != nullptr && threadIdx.x == 0;
  if (stamp && blockIdx.x == 0 && a.n_times > 0) a.times[0] = global_ns();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int h = d.h;
  const unsigned G = gridDim.x;
  // phase cycles of thread 0 (shared-memory accumulators): [0] front scan,
  // [1] slot fill, [2] gather + network, [3] per-pixel coding, [4] grid
  // barrier, [5] tiles
  long long* pc = PROF && a.prof != nullptr ? t.pc : nullptr;
  Ticker<PROF> tick(pc);
  // slots of the tile of n pixels starting at front position base of step
  // (by the first nt threads)
  auto fill_slots = [&](int step, long long base, int n, int nt) {
    for (int s = threadIdx.x; s < n; s += nt) {
      const int q = (int)(base + s);
      int lo2 = 0, hi2 = a.n_units - 1;  // last u with pre[u] <= q
      while (lo2 < hi2) {
        int mid = (lo2 + hi2 + 1) >> 1;
        if (t.pre[mid] <= q) lo2 = mid; else hi2 = mid - 1;
      }
      const Unit U = a.units[lo2];
      const Front fr = unit_front(U, step, h, a.sched);
      DecSlot ps;
      ps.i = fr.i_lo + (q - t.pre[lo2]);
      ps.j = front_col(U, step, ps.i, h, a.sched);
      ps.px = U.img + ((long long)(U.y0 + ps.i) * U.img_W + (U.x0 + ps.j)) * 3;
      ps.Wu = U.Wu;
      ps.row_bytes = 3 * U.img_W;
      ps.stream = U.stream_base + (a.layout == 1 ? ps.i : 0);
      const bool last = ps.j == U.Wu - 1 && (a.layout == 1 || ps.i == U.Hu - 1);
      ps.unit = lo2 | (last ? (int)0x80000000 : 0);
      if constexpr (SHEAR)  // ring bytes of the pixel's sheared column j + (h+1) i
        t.rofs[s] = kRingRowBytes * (U.ring_row + ps.i) + 3 * ((ps.j + (h + 1) * ps.i) & 15);
      t.slots[s] = ps;
    }
  };
  // Sheared tile of at most nmax pixels from front position base: the
  // pixels' slots, their output rows prow (pixel s of the tile's k-th unit
  // piece at s + h k: each piece is preceded by h halo window rows), the
  // window rows' (unit, unit row), and t.flag[1..3] = the tile's pixels,
  // output rows and window rows (the output rows stay below `rows`).
  auto fill_slots_shear = [&](int step, long long base, int nmax, int nt) {
    fill_slots(step, base, nmax, nt);
    part_sync(nt);
    if ((int)threadIdx.x < rows) {  // warps 0 .. rows/32 - 1
      const int s = threadIdx.x, w = s >> 5, l = s & 31;
      const bool valid = s < nmax;
      const int u = valid ? t.slots[s].unit & 0x7FFFFFFF : -1;
      const bool start = valid && (s == 0 || u != (t.slots[s - 1].unit & 0x7FFFFFFF));
      const unsigned bal = __ballot_sync(0xffffffffu, start);
      if (l == 0) t.sh[w] = __popc(bal);
      asm volatile("bar.sync 2, %0;" ::"r"(rows) : "memory");
      int before = 0;
      for (int k = 0; k < w; k++) before += (int)t.sh[k];
      const int seg = before + __popc(bal & (0xffffffffu >> (31 - l))) - 1;
      const int pr = s + h * seg;
      const bool fits = valid && pr < rows;
      // the tile's last pixel: the next one is missing or would not fit
      const bool valid1 = s + 1 < nmax;
      const int pr1 =
          s + 1 + h * (seg + ((valid1 && (t.slots[s + 1].unit & 0x7FFFFFFF) != u) ? 1 : 0));
      t.prow[s] = pr;
      if (fits) {
        const int i = t.slots[s].i;
        t.wrow[pr + h] = make_int2(u, i);
        if (start)
          for (int k = 1; k <= h; k++)
            t.wrow[pr + h - k] = make_int2(i - k >= 0 ? u : -1, i - k);
        if (!valid1 || pr1 >= rows) {
          t.flag[1] = s + 1;
          t.flag[2] = pr + 1;
          t.flag[3] = pr + 1 + h;
        }
      }
    }
  };
  // The schedule of step t + 1 (front sizes, this CTA's share, its first
  // tile's slots) needs no decoded data, so it is computed between arriving
  // at the grid barrier after step t and waiting for the others: the last
  // warp arrives (its release waits for the CTA's writes of step t to
  // reach GPU scope) while the other warps compute the schedule.
  const int NS = (int)blockDim.x - 32;
  int F = front_scan(a.units, a.n_units, 0, h, a.sched, t.pre, t.sh, (int)blockDim.x);
  tick(0);
  long long lo = (long long)F * blockIdx.x / G, hi = (long long)F * (blockIdx.x + 1) / G;
  if (lo < hi) {
    const int n = (int)min((long long)rows, hi - lo);
    if constexpr (SHEAR) fill_slots_shear(0, lo, n, (int)blockDim.x);
    else fill_slots(0, lo, n, (int)blockDim.x);
  }
  __syncthreads();
  tick(1);
  for (int step = 0; step < a.T; step++) {
    for (long long base = lo; base < hi;) {
      int n = (int)min((long long)rows, hi - base);
      if (base != lo) {  // further tiles of a large share
        if constexpr (SHEAR) fill_slots_shear(step, base, n, (int)blockDim.x);
        else fill_slots(step, base, n, (int)blockDim.x);
        __syncthreads();
      }
      if constexpr (SHEAR) n = t.flag[1];
      // A tile with at most one pixel per warp is coded by whole warps (lower
      // latency per pixel); otherwise by quads.  Lane l of warp w copies the
      // stream record of the warp's l-th pixel into shared memory ahead of
      // the network, asynchronously (no register waits for it, so its round
      // trip overlaps the gather's); after the network, the 12 stream bytes
      // from the record's pos + 8, read only when the pixel is done.
      const bool wide = n <= NW;
      const int sl = wide ? (lane == 0 ? warp : rows) : (lane < kQuads ? kQuads * warp + lane : rows);
      if (!SAMPLE && sl < n) {
        const StreamRec* r = a.st + t.slots[sl].stream;
        cp_async16(t.rec + sl, r);
        cp_async16(&t.rec[sl].pos, &r->pos);
      }
      if (PROF && tick.pc) tick.pc[5] += 1;
      tick(1);
      bool net_ok = true;
      if constexpr (PREC == PREC_BF16) {
        const long long c0 = PROF && tick.pc ? clock64() : 0;
        if constexpr (SHEAR)
          net_gather_win(a.units, t.wrow, a.ring, d, t.net, step, t.flag[3]);
        else if (d.shear) net_gather<true>(t.slots, d, t.net, n);
        else net_gather<false>(t.slots, d, t.net, n);
        __syncthreads();
        if (PROF && tick.pc) tick.pc[13] += clock64() - c0;
        net_ok = net_run<PROF>(d, t.net, SHEAR ? t.flag[2] : n, SHEAR, pc);
      } else {
        f32_gather<true>(t.slots, n, d, t.f32);
        __syncthreads();
        f32_run(d, t.f32, n);
      }
      // an exchange that timed out: record it and release every CTA from
      // the grid barrier (this one leaves its loop at its next wait)
      if (!net_ok && threadIdx.x == 0) {
        set_status(a.status, ST_TIMEOUT);
        atomicOr(a.bar, kBarPoison);
      }
      if (!SAMPLE) {
        cp_async_wait_all();
        if (sl < n) {
          const unsigned long long w0 = (t.rec[sl].pos + 8ull) & ~3ull, end = t.rec[sl].end;
#pragma unroll
          for (int q = 0; q < 3; q++) {
            const unsigned long long wa = w0 + 4ull * q;
            cp_async4(t.win + 4 * sl + q, a.in + (wa < end ? wa : 0ull), wa < end);
          }
        }
        __syncwarp();  // the warp's records are visible to all its lanes
      }
      tick(2);
      if (wide) {
        code_wide<NW, SAMPLE, SHEAR, PROF>(a, t, n, pc);
      } else {
        switch ((d.K + 3) / 4) {
          case 1: code_quads<1, NW, SAMPLE, SHEAR, PROF>(a, t, n, pc); break;
          case 2: code_quads<2, NW, SAMPLE, SHEAR, PROF>(a, t, n, pc); break;
          case 3: code_quads<3, NW, SAMPLE, SHEAR, PROF>(a, t, n, pc); break;
          default: code_quads<4, NW, SAMPLE, SHEAR, PROF>(a, t, n, pc); break;
        }
      }
      __syncthreads();
      tick(3);
      base += n;
    }
    if (step + 1 == a.T) break;
    const unsigned target = (unsigned)step + 1u;
    if ((int)threadIdx.x >= NS) {
      if (G > 1 && (int)threadIdx.x == NS) grid_arrive(a.bar);
    } else {
      F = front_scan(a.units, a.n_units, step + 1, h, a.sched, t.pre, t.sh, NS);
      tick(0);
      lo = (long long)F * blockIdx.x / G;
      hi = (long long)F * (blockIdx.x + 1) / G;
      if (lo < hi) {
        const int n = (int)min((long long)rows, hi - lo);
        if constexpr (SHEAR) fill_slots_shear(step + 1, lo, n, NS);
        else fill_slots(step + 1, lo, n, NS);
      }
      tick(1);
    }
    if (G > 1) {
      if (!grid_wait(a.bar, G, target, a.status, t.flag, a.spin_limit)) break;
    } else {
      __syncthreads();
    }
    if ((int)threadIdx.x >= NS) {
      F = t.pre[a.n_units];
      lo = (long long)F * blockIdx.x / G;
      hi = (long long)F * (blockIdx.x + 1) / G;
    }
    tick(4);
    if (stamp && blockIdx.x == 0 && step + 1 < a.n_times) a.times[step + 1] = global_ns();
  }
  if (stamp && a.T < a.n_times) atomicMax(a.times + a.T, global_ns());
  if (PROF && tick.pc) {
    for (int i = 0; i < 16; i++)
      if (i != 6 && i != 7) atomicAdd(a.prof + i, (unsigned long long)tick.pc[i]);
    atomicAdd(a.prof + 6, 1ull);
    if (blockIdx.x == 0) atomicAdd(a.prof + 7, (unsigned long long)a.T);
  }
}

}  // namespace nlc
