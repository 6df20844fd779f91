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

// What the schedule needs of a unit.  All of them are kept in shared memory
// when they fit: the schedule of a step is on its critical path, and each
// dependent read of the unit table through L2 added 0.3 us to it.
struct alignas(16) DecUnit {
  uint8_t* px;      // first pixel
  int Hu, Wu;       // size
  uint32_t row_bytes;  // row stride of the image (two rows of 2^30 pixels fit)
  int stream_base;  // first rANS stream
  int start_step;   // step of its first pixel
  int ring_row;     // first row in the sheared rings
};
__device__ __forceinline__ DecUnit dec_unit(const Unit& u) {
  return DecUnit{u.img + ((long long)u.y0 * u.img_W + u.x0) * 3, u.Hu, u.Wu, 3u * u.img_W,
                 u.stream_base, u.start_step, u.ring_row};
}

// x / (h + 1) for h <= 3 and x >= 0.  By 3: the high half of x times 2^33 / 3
// rounded up, exact for x < 2^32 since x times that rounding's 1/3 stays below
// 2^33 / 3 (division by a constant as in Granlund and Montgomery, 1994).
__device__ __forceinline__ int div_o(int x, int h) {
  return h == 1 ? x >> 1 : h == 3 ? x >> 2 : (int)(__umulhi((unsigned)x, 0xAAAAAAABu) >> 1);
}

// Front of a unit at global step t, tau = t - start_step its local step:
//   wavefront (Section 3): rows i with j = tau - (h+1) i in [0, Wu)
//   raster: the single pixel tau of the unit in raster order.
__device__ __forceinline__ Front dec_front(const DecUnit& u, int t, int h, int sched) {
  const int tau = t - u.start_step;
  Front f{0, 0};
  if (tau < 0) return f;
  if (sched == SCHED_WAVEFRONT) {
    const int hi = min(div_o(tau, h), u.Hu - 1);
    const int num = tau - u.Wu + 1;  // i >= ceil(num / (h + 1))
    f.i_lo = num <= 0 ? 0 : div_o(num + h, h);
    f.n = max(hi - f.i_lo + 1, 0);
  } else if (tau < u.Hu * u.Wu) {
    f.i_lo = tau / u.Wu;
    f.n = 1;
  }
  return f;
}

// Shared memory of a decoder CTA: byte offsets of its regions (dec_at).
struct DecSmem {
  int P;      // head outputs of the tile's pixels
  int ldp;    // and their row stride
  int ws;     // WarpScratch, one per warp (whole-warp coding)
  int slots;  // DecSlot: the tile's pixels
  int rec;    // StreamRec: their stream records
  int win;    // per pixel, the 12 stream bytes from pos + 8, word-aligned (4 words)
  int prow;   // sheared wavefront decoder: output row of the tile's pixel s
  int rofs;   // sheared wavefront decoder: ring byte offset of the tile's pixel s
  int wrow;   // sheared wavefront decoder: (unit, unit row) of window row rho
  int sh;     // 64 ints: the schedule's warp sums
  int pc;     // 16 profiling accumulators (thread 0 only)
  int units;  // DecUnit: the batch's units, where they fit (else 0: read from global memory)
  int pre;    // front prefix of the units
  int flag;   // [0] stop, [1..3] sheared tile, [4], [5] units of the share, [6..9] shares (share_at)
};

// Copies of the CTA's share, by the step's parity.  Every warp reads its copy
// after the barrier that ends the step before; where the share is empty (fewer
// pixels than CTAs) the next barrier is the one that ends the step itself, so a
// warp may write the share of the step after it while another has not yet read
// its own: never further ahead, so two copies keep them apart.
constexpr int kShares = 2;

// The arguments and the shared-memory map as the kernel's functions see them.
// They are kept in shared memory: as kernel parameters and locals passed by
// reference they were in local memory, whose lines every acquire of the grid
// barrier drops from L1, so the first use of each field in a step went to L2.
struct DecShared {
  NetSmem net;
  DecodeArgs a;
  DecSmem t;
};
static_assert(sizeof(DecShared) <= kSharedHead, "the record's place");
__device__ __forceinline__ DecShared& dec_shared() {
  return *reinterpret_cast<DecShared*>(dec_smem);
}

// Carves the shared memory of a tile of `rows` pixels; returns its bytes.
// win: the sheared model's wavefront decoder.  The whole-warp groups' scratch
// lies behind the first 16 head-output rows of the BF16 tile region, which a
// tile of at most 16 pixels leaves free (not in the window tile, whose output
// rows are spread out).
__host__ __device__ inline size_t dec_carve(const Dims& d, int n_pre, int rows, bool win,
                                            DecSmem* t) {
  int off;
  DecSmem z{};
  if (d.prec == PREC_BF16) {
    const NetPlan p = net_plan(d, rows, win);
    off = p.end;
    z.ws = win ? off : p.x + kNetWarps * net_ldp(d) * 4;
    if (win) off += (int)sizeof(WarpScratch) * kNetWarps;
    z.P = p.x;
    z.ldp = net_ldp(d);
  } else {
    const F32Plan p = f32_plan(d);
    z.P = 4 * p.u;
    z.ldp = d.ldP;
    off = align_up(p.end * 4, 16);
    z.ws = off;
    off += (int)sizeof(WarpScratch) * (decode_threads<PREC_FP32>() / 32);
  }
  off = align_up(off, 16);
  auto take = [&](size_t bytes) {
    const int o = off;
    off += (int)((bytes + 15) & ~(size_t)15);
    return o;
  };
  z.slots = take(sizeof(DecSlot) * rows);
  z.rec = take(sizeof(StreamRec) * rows);
  z.win = take(4 * sizeof(uint32_t) * rows);
  if (win) {
    z.wrow = take(sizeof(int2) * (rows + 8));
    z.prow = take(sizeof(int) * rows);
    z.rofs = take(sizeof(int) * rows);
  }
  z.sh = take(sizeof(int) * 64);
  z.pc = take(sizeof(long long) * 16);
  z.flag = take(sizeof(int) * (6 + 2 * kShares));
  z.pre = take(sizeof(int) * ((size_t)n_pre + 1));
  if (kSharedHead + off + sizeof(DecUnit) * (size_t)n_pre <= kMaxSmem)
    z.units = take(sizeof(DecUnit) * (size_t)n_pre);
  if (t) *t = z;
  return (size_t)kSharedHead + off;
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
  const DecSlot ps = dec_at<DecSlot>(t.slots)[s];
  ps.px[0] = (uint8_t)v[0];
  ps.px[1] = (uint8_t)v[1];
  ps.px[2] = (uint8_t)v[2];
  if (SHEAR) ring_put(a, dec_at<int>(t.rofs)[s], v);
  if (SAMPLE) return;
  const ulonglong2 pe = *reinterpret_cast<const ulonglong2*>(&dec_at<StreamRec>(t.rec)[s].pos);
  dec.set_window(dec_at<uint32_t>(t.win) + 4 * s, pe.x);
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
__device__ __noinline__ void code_wide(int n, long long* pc) {
  const DecodeArgs& a = dec_shared().a;
  const DecSmem& t = dec_shared().t;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int K = a.m.d.K;
  WarpScratch& ws = dec_at<WarpScratch>(t.ws)[warp];
  Ticker<PROF> tick(pc);
  for (int s = warp; s < n; s += NW) {
    GroupRansDec dec;
    unsigned long long key = 0;
    if (SAMPLE) key = sample_key(a, dec_at<DecSlot>(t.slots)[s]);
    else dec = load_rec(dec_at<StreamRec>(t.rec) + s);
    if (PROF && tick.pc) tick.pc[12] += 1;
    CompState cs;
    comp_init<32>(dec_at<float>(t.P) + (SHEAR ? dec_at<int>(t.prow)[s] : s) * t.ldp, K, lane, cs);
    int v[3] = {0, 0, 0};
    for (int ch = 0; ch < 3; ch++) {
      int nact;
      const float mloc = channel_setup<32>(cs, K, ch, v[0], v[1], lane, ws, nact);
      tick(8);
      const uint32_t slot =
          SAMPLE ? (uint32_t)(splitmix64_at(a.seed, key + ch) >> 48) : (dec.x & 0xFFFFu);
      uint32_t lo, hi;
      v[ch] = cdf_search(ws, nact, slot, lane, lo, hi);
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
__device__ __noinline__ void code_quads(int n, long long* pc) {
  const DecodeArgs& a = dec_shared().a;
  const DecSmem& t = dec_shared().t;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int q = lane & 3;
  const int K = a.m.d.K;
  Ticker<PROF> tick(pc);
  for (int s0 = kQuads * warp; s0 < n; s0 += kQuads * NW) {
    const bool valid = s0 + (lane >> 2) < n;
    const int s = valid ? s0 + (lane >> 2) : n - 1;  // an idle quad shadows the last pixel
    GroupRansDec dec;
    unsigned long long key = 0;
    if (SAMPLE) key = sample_key(a, dec_at<DecSlot>(t.slots)[s]);
    else dec = load_rec(dec_at<StreamRec>(t.rec) + s);
    if (PROF && tick.pc) tick.pc[12] += 1;
    const float* row = dec_at<float>(t.P) + (SHEAR ? dec_at<int>(t.prow)[s] : s) * t.ldp + q;
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

// ---------------------------------------------------------------------
// Schedule of a step, computed by the first nt threads of the CTA (functions
// of their own, with their results in shared memory: inlined, their state and
// the step loop's spilled to local memory, which the loop re-reads from L2).
// ---------------------------------------------------------------------
__device__ __forceinline__ DecUnit unit_of(int u) {
  const int in = dec_shared().t.units;
  return in ? dec_at<DecUnit>(in)[u] : dec_unit(dec_shared().a.units[u]);
}

// This CTA's share [x, y) of a step's F pixels: F / grid of them, or one more.
__device__ __forceinline__ int2 sched_share(int F) {
  const unsigned G = gridDim.x, each = (unsigned)F / G, more = (unsigned)F - each * G;
  const int lo = (int)(each * blockIdx.x + min(blockIdx.x, more));
  return make_int2(lo, lo + (int)each + (blockIdx.x < more ? 1 : 0));
}

// The CTA's share [x, y) of a step's pixels, beside the flags.
__device__ __forceinline__ int2& share_at(int* flag, int step) {
  return reinterpret_cast<int2*>(flag + 6)[(unsigned)step % kShares];
}

// Fronts of all units: pre[u] = exclusive prefix of the front sizes,
// pre[n_units] = their total F; flag[4], flag[5] = the units that hold the
// first and the last pixel of this CTA's share.
//
// Up to kWarpUnits units, every warp computes all of it (and stores the same
// values): one or two warp scans cost less than the two barriers that a scan
// over the CTA needs (a step of n units of 32 x 64 pixels: 7.23 against 7.62 us
// at n = 1, 7.37 / 7.77 at 16, 7.43 / 7.80 at 32, 7.58 / 7.80 at 33, 7.78 / 8.01
// at 64; a lane holds two units, so the line lies where a third would begin).
// With more units a thread takes one or more of them, and every warp adds up the
// warps' sums itself.
constexpr int kWarpUnits = 64;
static __device__ __forceinline__ void sched_front_warp(int step) {
  const DecodeArgs& a = dec_shared().a;
  const DecSmem& t = dec_shared().t;
  const int n_units = a.n_units, h = a.m.d.h, sched = a.sched;
  const int lane = threadIdx.x & 31;
  int* pre = dec_at<int>(t.pre);
  int* flag = dec_at<int>(t.flag);
  int c0 = lane < n_units ? dec_front(unit_of(lane), step, h, sched).n : 0;
  int c1 = lane + 32 < n_units ? dec_front(unit_of(lane + 32), step, h, sched).n : 0;
  int x0 = c0, x1 = c1;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y0 = __shfl_up_sync(0xffffffffu, x0, o), y1 = __shfl_up_sync(0xffffffffu, x1, o);
    if (lane >= o) x0 += y0, x1 += y1;
  }
  const int F0 = __shfl_sync(0xffffffffu, x0, 31), F = F0 + __shfl_sync(0xffffffffu, x1, 31);
  const int2 sh = sched_share(F);
  auto put = [&](int u, int run, int c) {
    if (u >= n_units) return;
    pre[u] = run;
    if (run <= sh.x && sh.x < run + c) flag[4] = u;
    if (run < sh.y && sh.y <= run + c) flag[5] = u;
  };
  put(lane, x0 - c0, c0);
  put(lane + 32, F0 + x1 - c1, c1);
  if (lane == 0) {
    pre[n_units] = F;
    share_at(flag, step) = sh;
  }
  __syncwarp();
}

static __device__ __forceinline__ void sched_front(int step, int nt) {
  const DecodeArgs& a = dec_shared().a;
  const DecSmem& t = dec_shared().t;
  const int n_units = a.n_units, h = a.m.d.h, sched = a.sched;
  if (n_units <= kWarpUnits) return sched_front_warp(step);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (n_units + nt - 1) / nt, nw = nt >> 5;
  const int u0 = min((int)threadIdx.x * per, n_units), u1 = min(u0 + per, n_units);
  int* pre = dec_at<int>(t.pre);
  int* flag = dec_at<int>(t.flag);
  int* sums = dec_at<int>(t.sh);
  int sum = 0, c = 0;
  for (int u = u0; u < u1; u++) {
    c = dec_front(unit_of(u), step, h, sched).n;
    if (per > 1) pre[u] = c;
    sum += c;
  }
  int x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sums[warp] = x;
  part_sync(nt);
  int y = lane < nw ? sums[lane] : 0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int z = __shfl_up_sync(0xffffffffu, y, o);
    if (lane >= o) y += z;
  }
  const int before = __shfl_sync(0xffffffffu, y, warp > 0 ? warp - 1 : 0);
  const int F = __shfl_sync(0xffffffffu, y, 31);
  const int2 share = sched_share(F);
  const int lo = share.x, hi = share.y;
  int run = x - sum + (warp > 0 ? before : 0);
  for (int u = u0; u < u1; u++) {
    if (per > 1) c = pre[u];
    pre[u] = run;
    if (run <= lo && lo < run + c) flag[4] = u;
    if (run < hi && hi <= run + c) flag[5] = u;
    run += c;
  }
  if (threadIdx.x == 0) {
    pre[n_units] = F;
    share_at(flag, step) = share;
  }
  part_sync(nt);
}

// Slots of the tile of n pixels starting at front position base.  SHEAR: a
// tile of at most n pixels: also their output rows prow (pixel s of the tile's
// k-th unit piece at s + h k: each piece is preceded by h halo window rows),
// the window rows' (unit, unit row), and flag[1..3] = the tile's pixels,
// output rows and window rows (the output rows stay below `rows`).
template <bool SHEAR>
__device__ __forceinline__ void sched_slots(int step, int base, int n, int nt) {
  const DecodeArgs& a = dec_shared().a;
  const DecSmem& t = dec_shared().t;
  const int h = a.m.d.h, sched = a.sched, layout = a.layout;
  const int* pre = dec_at<int>(t.pre);
  int* flag = dec_at<int>(t.flag);
  DecSlot* slots = dec_at<DecSlot>(t.slots);
  const int first = flag[4], last_u = flag[5];
  for (int s = threadIdx.x; s < n; s += nt) {
    const int q = base + s;
    int lo = first, hi = last_u;  // last unit of the share with pre[u] <= q
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (pre[mid] <= q) lo = mid; else hi = mid - 1;
    }
    const DecUnit U = unit_of(lo);
    const int tau = step - U.start_step;
    DecSlot ps;
    if (sched == SCHED_WAVEFRONT) {
      ps.i = dec_front(U, step, h, sched).i_lo + (q - pre[lo]);
      ps.j = tau - (h + 1) * ps.i;
    } else {
      ps.i = tau / U.Wu;
      ps.j = tau - ps.i * U.Wu;
    }
    ps.px = U.px + (long long)ps.i * U.row_bytes + 3LL * ps.j;
    ps.Wu = U.Wu;
    ps.row_bytes = U.row_bytes;
    ps.stream = U.stream_base + (layout == 1 ? ps.i : 0);
    const bool last = ps.j == U.Wu - 1 && (layout == 1 || ps.i == U.Hu - 1);
    ps.unit = lo | (last ? (int)0x80000000 : 0);
    if (SHEAR)  // ring bytes of the pixel's sheared column j + (h+1) i
      dec_at<int>(t.rofs)[s] = kRingRowBytes * (U.ring_row + ps.i) + 3 * ((ps.j + (h + 1) * ps.i) & 15);
    slots[s] = ps;
  }
  if (!SHEAR) return;
  const int rows = a.rows;
  int* sums = dec_at<int>(t.sh);
  int2* wrow = dec_at<int2>(t.wrow);
  part_sync(nt);
  if ((int)threadIdx.x < rows) {  // warps 0 .. rows/32 - 1
    const int s = threadIdx.x, w = s >> 5, l = s & 31;
    const bool valid = s < n;
    const int u = valid ? slots[s].unit & 0x7FFFFFFF : -1;
    const bool start = valid && (s == 0 || u != (slots[s - 1].unit & 0x7FFFFFFF));
    const unsigned bal = __ballot_sync(0xffffffffu, start);
    if (l == 0) sums[w] = __popc(bal);
    asm volatile("bar.sync 2, %0;" ::"r"(rows) : "memory");
    int before = 0;
    for (int k = 0; k < w; k++) before += sums[k];
    const int seg = before + __popc(bal & (0xffffffffu >> (31 - l))) - 1;
    const int pr = s + h * seg;
    const bool fits = valid && pr < rows;
    // the tile's last pixel: the next one is missing or would not fit
    const bool valid1 = s + 1 < n;
    const int pr1 =
        s + 1 + h * (seg + ((valid1 && (slots[s + 1].unit & 0x7FFFFFFF) != u) ? 1 : 0));
    dec_at<int>(t.prow)[s] = pr;
    if (fits) {
      const int i = slots[s].i;
      wrow[pr + h] = make_int2(u, i);
      if (start)
        for (int k = 1; k <= h; k++) wrow[pr + h - k] = make_int2(i - k >= 0 ? u : -1, i - k);
      if (!valid1 || pr1 >= rows) {
        flag[1] = s + 1;
        flag[2] = pr + 1;
        flag[3] = pr + 1 + h;
      }
    }
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
  const int rows = a.rows;
  const DecSmem& t = dec_shared().t;
  uint32_t phase = 0;  // of the warp's exchanges
  if (threadIdx.x == 0) {
    DecShared z;
    dec_carve(a.m.d, a.n_units, rows, SHEAR, &z.t);
    z.a = a;
    z.net.d = a.m.d;
    z.net.rows = rows;
    z.net.limit = a.mma_limit;
    if constexpr (PREC == PREC_BF16) {
      z.net.pl = net_plan(a.m.d, rows, SHEAR);
      net_setup(z.net.pl);
    }
    dec_shared() = z;
    dec_at<int>(z.t.flag)[0] = 0;
  }
  __syncthreads();
  if constexpr (PREC == PREC_BF16) {
    net_load_weights(a.m.d, a.m.w, net_smem().pl.bias);
  } else {
    for (int i = threadIdx.x; i < a.m.w.simt_floats; i += blockDim.x)
      dec_at<float>(0)[i] = a.m.w.simt[i];
  }
  if (threadIdx.x < 16) dec_at<long long>(t.pc)[threadIdx.x] = 0;
  if (t.units)
    for (int u = threadIdx.x; u < a.n_units; u += blockDim.x)
      dec_at<DecUnit>(t.units)[u] = dec_unit(a.units[u]);
  __syncthreads();
  int* flag = dec_at<int>(t.flag);
  // step end times: CTA 0 stamps each step when the grid barrier after it
  // releases (every CTA has finished it); every CTA stamps the last step's end
  const bool stamp = a.times != nullptr && threadIdx.x == 0;
  if (stamp && blockIdx.x == 0 && a.n_times > 0) a.times[0] = global_ns();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned G = gridDim.x;
  // phase cycles of thread 0 (shared-memory accumulators): [0] front scan,
  // [1] slot fill, [2] gather + network, [3] per-pixel coding, [4] grid
  // barrier, [5] tiles
  long long* pc = PROF && a.prof != nullptr ? dec_at<long long>(t.pc) : nullptr;
  Ticker<PROF> tick(pc);
  // The schedule of step t + 1 (front sizes, this CTA's share, its first
  // tile's slots) needs no decoded data, so it is computed between arriving
  // at the grid barrier after step t and waiting for the others: the last
  // warp arrives (its release waits for the CTA's writes of step t to
  // reach GPU scope) while the other warps compute the schedule.
  constexpr int NS = NT - 32;
  sched_front(0, NT);
  tick(0);
  int lo = share_at(flag, 0).x, hi = share_at(flag, 0).y;  // the CTA's share of the step's pixels
  if (lo < hi) sched_slots<SHEAR>(0, lo, min(rows, hi - lo), NT);
  __syncthreads();
  tick(1);
  for (int step = 0; step < a.T; step++) {
    for (int base = lo; base < hi;) {
      int n = min(rows, hi - base);
      if (base != lo) {  // further tiles of a large share
        sched_slots<SHEAR>(step, base, n, NT);
        __syncthreads();
      }
      if constexpr (SHEAR) n = flag[1];
      // A tile with at most one pixel per warp is coded by whole warps (lower
      // latency per pixel); otherwise by quads.  Lane l of warp w copies the
      // stream record of the warp's l-th pixel into shared memory ahead of
      // the network, asynchronously (no register waits for it, so its round
      // trip overlaps the gather's); after the network, the 12 stream bytes
      // from the record's pos + 8, read only when the pixel is done.
      const bool wide = n <= NW;
      const int sl = wide ? (lane == 0 ? warp : rows) : (lane < kQuads ? kQuads * warp + lane : rows);
      if (!SAMPLE && sl < n) {
        const StreamRec* r = a.st + dec_at<DecSlot>(t.slots)[sl].stream;
        StreamRec* rec = dec_at<StreamRec>(t.rec) + sl;
        cp_async16(rec, r);
        cp_async16(&rec->pos, &r->pos);
      }
      if (PROF && tick.pc) tick.pc[5] += 1;
      tick(1);
      bool net_ok = true;
      if constexpr (PREC == PREC_BF16) {
        const long long c0 = PROF && tick.pc ? clock64() : 0;
        if constexpr (SHEAR)
          net_gather_win(a.units, a.ring, t.wrow, step, flag[3]);
        else if (a.m.d.shear) net_gather<true>(t.slots, n);
        else net_gather<false>(t.slots, n);
        __syncthreads();
        if (PROF && tick.pc) tick.pc[13] += clock64() - c0;
        net_ok = net_run<PROF>(a.m.d.C, SHEAR ? flag[2] : n, SHEAR, phase, pc);
      } else {
        f32_gather<true>(dec_at<DecSlot>(t.slots), n, a.m.d, dec_at<float>(0));
        __syncthreads();
        f32_run(a.m.d, dec_at<float>(0), n);
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
          const unsigned long long w0 = (dec_at<StreamRec>(t.rec)[sl].pos + 8ull) & ~3ull,
                                   end = dec_at<StreamRec>(t.rec)[sl].end;
#pragma unroll
          for (int q = 0; q < 3; q++) {
            const unsigned long long wa = w0 + 4ull * q;
            cp_async4(dec_at<uint32_t>(t.win) + 4 * sl + q, a.in + (wa < end ? wa : 0ull), wa < end);
          }
        }
        __syncwarp();  // the warp's records are visible to all its lanes
      }
      tick(2);
      if (wide) {
        code_wide<NW, SAMPLE, SHEAR, PROF>(n, pc);
      } else {
        switch ((a.m.d.K + 3) / 4) {
          case 1: code_quads<1, NW, SAMPLE, SHEAR, PROF>(n, pc); break;
          case 2: code_quads<2, NW, SAMPLE, SHEAR, PROF>(n, pc); break;
          case 3: code_quads<3, NW, SAMPLE, SHEAR, PROF>(n, pc); break;
          default: code_quads<4, NW, SAMPLE, SHEAR, PROF>(n, pc); break;
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
      sched_front(step + 1, NS);
      tick(0);
      lo = share_at(flag, step + 1).x;
      hi = share_at(flag, step + 1).y;
      if (lo < hi) sched_slots<SHEAR>(step + 1, lo, min(rows, hi - lo), NS);
      tick(1);
    }
    if (G > 1) {
      if (!grid_wait(a.bar, G, target, a.status, flag, a.spin_limit)) break;
    } else {
      __syncthreads();
    }
    lo = share_at(flag, step + 1).x;
    hi = share_at(flag, step + 1).y;
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
