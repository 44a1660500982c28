// Event ingest kernels (Sec. II linear-index EER; Table 1 bin, crop, centre of
// mass and sum of all frames; Eq. 4).
//
// Every kernel re-derives each frame's event range defensively:
//   lo = min(off[f], n_idx), hi = min(max(off[f+1], lo), n_idx)
// so corrupt offsets never cause an out-of-bounds read; they set
// EER4D_ST_OFFSETS instead.  Indices >= det_w*det_h are dropped and counted.
#include <type_traits>

#include "common.cuh"

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ void frame_range(const uint64_t* off, uint64_t f, uint64_t n_idx,
                                            uint64_t& lo, uint64_t& hi, bool& bad) {
  const uint64_t a = off[f], b = off[f + 1];
  lo = a < n_idx ? a : n_idx;
  uint64_t t = b > lo ? b : lo;
  hi = t < n_idx ? t : n_idx;
  bad = (b < a) || (b > n_idx) || (a > n_idx);
}

// ---------------------------------------------------------------- a1 -------
// Offsets check, index range check, integer totals and optional PACBED.  The
// coordinates of a thread's 16 events in flight are added in 32 bits, and a
// block's totals before they go to the three global ones (a warp's own atomics
// on them, 64-bit sums and a PACBED test per event: 52e6 events 55 us, now 43;
// 32 for the bytes).
template <bool PACBED>
__global__ void __launch_bounds__(kThreads) k_validate(const uint32_t* __restrict__ idx,
                                                       uint64_t n_idx,
                                                       const uint64_t* __restrict__ off,
                                                       uint64_t n_frames, uint32_t WH, DivMod dw,
                                                       unsigned long long* pacbed,
                                                       unsigned long long* totals, uint32_t* st) {
  pdl_begin();
  const uint64_t gtid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t gsz = (uint64_t)gridDim.x * blockDim.x;
  bool bad = false;
  for (uint64_t f = gtid; f < n_frames; f += gsz) {
    uint64_t lo, hi;
    bool b;
    frame_range(off, f, n_idx, lo, hi, b);
    bad |= b;
  }
  if (bad) st_or(st, EER4D_ST_OFFSETS);
  // events referenced by the frames: [min lo, max hi) == [off[0], off[n]) for valid data
  uint64_t e0 = off[0] < n_idx ? off[0] : n_idx;
  uint64_t e1 = off[n_frames] < n_idx ? off[n_frames] : n_idx;
  if (e1 < e0) e1 = e0;
  unsigned long long sx = 0, sy = 0, sn = 0;
  uint32_t drop = 0, px = 0, py = 0, pn = 0;
  auto one = [&](uint32_t v) {
    if (v >= WH) { ++drop; return; }
    uint32_t y, x;
    dw.divmod(v, y, x);
    px += x; py += y; ++pn;
    if (PACBED) atomicAdd(pacbed + v, 1ull);
  };
  auto flush = [&] {  // x, y < 32768
    sx += px; sy += py; sn += pn;
    px = py = pn = 0;
  };
  // scalar head up to a 16-byte boundary, then 4 x uint4 per thread in flight
  uint64_t head = e0;
  const uintptr_t a = reinterpret_cast<uintptr_t>(idx + e0);
  if ((a & 3) == 0) head = e0 + (((16 - (a & 15)) & 15) >> 2);
  else head = e1;
  if (head > e1) head = e1;
  for (uint64_t i = e0 + gtid; i < head; i += gsz) { one(__ldg(idx + i)); flush(); }
  const uint64_t nv = (e1 - head) >> 2;
  const uint4* v4 = reinterpret_cast<const uint4*>(idx + head);
  uint64_t i = gtid;
  for (; i + 3 * gsz < nv; i += 4 * gsz) {
    const uint4 q0 = __ldg(v4 + i), q1 = __ldg(v4 + i + gsz), q2 = __ldg(v4 + i + 2 * gsz),
                q3 = __ldg(v4 + i + 3 * gsz);
    one(q0.x); one(q0.y); one(q0.z); one(q0.w);
    one(q1.x); one(q1.y); one(q1.z); one(q1.w);
    one(q2.x); one(q2.y); one(q2.z); one(q2.w);
    one(q3.x); one(q3.y); one(q3.z); one(q3.w);
    flush();
  }
  for (; i < nv; i += gsz) {
    const uint4 q = __ldg(v4 + i);
    one(q.x); one(q.y); one(q.z); one(q.w);
    flush();
  }
  for (uint64_t k = head + 4 * nv + gtid; k < e1; k += gsz) { one(__ldg(idx + k)); flush(); }
  if (totals) {
    __shared__ unsigned long long s_sum[kThreads / 32][3];
    sx = warp_sum_ll(sx); sy = warp_sum_ll(sy); sn = warp_sum_ll(sn);
    if ((threadIdx.x & 31) == 0) {
      unsigned long long* w = s_sum[threadIdx.x >> 5];
      w[0] = sx; w[1] = sy; w[2] = sn;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
      unsigned long long v = 0;
      for (int w = 0; w < kThreads / 32; ++w) v += s_sum[w][threadIdx.x];
      if (v) atomicAdd(totals + threadIdx.x, v);
    }
  }
  for (int o = 16; o > 0; o >>= 1) drop += __shfl_xor_sync(0xffffffffu, drop, o);
  if ((threadIdx.x & 31) == 0 && drop) {
    st_or(st, EER4D_ST_RANGE);
    st_add(st, 1, drop);
  }
}

// ---------------------------------------------------------------- a2 -------
// Per-frame integer sums (Eq. 4 on linear-index EER), one thread per frame.
// A thread reads its frame's events straight from global memory, 16-byte
// vector loads with four in flight (a frame's events are contiguous, so the
// 32 frames of a warp cover one contiguous stretch of the event array and
// every fetched sector is used); no shared staging and no block barrier
// before the sums.  Thread 0 computes the centre meanwhile.
constexpr int kComThreads = 256;
// frames of at most this many events sum x and y in 32 bits (x, y < 32768)
constexpr uint64_t kComFast = 131071;

// The COM centre as an exact integer part and a float fraction (from double):
// the PACBED centre of mass from the totals, or (cx, cy) when there are none.
struct ComCentre {
  long long ix, iy;
  float fx, fy;
};
__device__ __forceinline__ ComCentre com_centre(const long long* totals, double cx, double cy) {
  if (totals) {
    const long long n = totals[2];
    cx = n ? (double)totals[0] / (double)n : 0.0;
    cy = n ? (double)totals[1] / (double)n : 0.0;
  }
  const double rx = rint(cx), ry = rint(cy);
  ComCentre c;
  c.ix = (long long)rx;
  c.iy = (long long)ry;
  c.fx = (float)(cx - rx);
  c.fy = (float)(cy - ry);
  return c;
}
// COM of one frame relative to the centre, (Sx - N round(cx)) / N - frac(cx)
// in float32 (0 for an empty frame).
__device__ __forceinline__ void com_of_frame(long long sx, long long sy, long long sn,
                                             const ComCentre& c, float& ox, float& oy) {
  ox = oy = 0.f;
  if (sn) {
    const long long dx = sx - sn * c.ix;
    const long long dy = sy - sn * c.iy;
    ox = (float)dx / (float)sn - c.fx;
    oy = (float)dy / (float)sn - c.fy;
  }
}

__global__ void __launch_bounds__(kComThreads, 8) k_com(const uint32_t* __restrict__ idx, uint64_t n_idx,
                                                     const uint64_t* __restrict__ off, uint32_t F,
                                                     uint32_t WH, DivMod dw,
                                                     const long long* __restrict__ totals,
                                                     double cx_h, double cy_h, float zscale,
                                                     long long* sums, float* com, float2* z,
                                                     uint32_t* st) {
  pdl_begin();
  __shared__ ComCentre s_c;
  if (threadIdx.x == 0) s_c = com_centre(totals, cx_h, cy_h);
  const uint32_t f = blockIdx.x * kComThreads + threadIdx.x;
  unsigned long long sx = 0, sy = 0, sn = 0;
  uint32_t drop = 0;
  if (f < F) {
    uint64_t lo, hi;
    bool bad;
    frame_range(off, f, n_idx, lo, hi, bad);
    if (bad) st_or(st, EER4D_ST_OFFSETS);
    uint32_t px = 0, py = 0, pn = 0;
    auto one = [&](uint32_t v) {
      if (v >= WH) { ++drop; return; }
      uint32_t y, x;
      dw.divmod(v, y, x);
      px += x; py += y; ++pn;
    };
    uint64_t i = lo;
    if (hi - lo > kComFast) {
      // a frame too long for 32-bit sums (never at detector doses): 64-bit
      for (; i < hi; ++i) {
        const uint32_t v = __ldg(idx + i);
        if (v >= WH) { ++drop; continue; }
        uint32_t y, x;
        dw.divmod(v, y, x);
        sx += x; sy += y; ++sn;
      }
    } else if ((reinterpret_cast<uintptr_t>(idx) & 15) == 0) {
      for (; i < hi && (i & 3); ++i) one(__ldg(idx + i));
      for (; i + 16 <= hi; i += 16) {
        const uint4* q = reinterpret_cast<const uint4*>(idx + i);
        const uint4 a0 = __ldg(q), a1 = __ldg(q + 1), a2 = __ldg(q + 2), a3 = __ldg(q + 3);
        one(a0.x); one(a0.y); one(a0.z); one(a0.w);
        one(a1.x); one(a1.y); one(a1.z); one(a1.w);
        one(a2.x); one(a2.y); one(a2.z); one(a2.w);
        one(a3.x); one(a3.y); one(a3.z); one(a3.w);
      }
      for (; i + 4 <= hi; i += 4) {
        const uint4 a0 = __ldg(reinterpret_cast<const uint4*>(idx + i));
        one(a0.x); one(a0.y); one(a0.z); one(a0.w);
      }
    }
    for (; i < hi; ++i) one(__ldg(idx + i));
    sx += px; sy += py; sn += pn;
  }
  __syncthreads();  // the centre
  if (f < F) {
    sums[f] = (long long)sx;
    sums[F + f] = (long long)sy;
    sums[2 * (size_t)F + f] = (long long)sn;
    float ox, oy;
    com_of_frame((long long)sx, (long long)sy, (long long)sn, s_c, ox, oy);
    com[f] = ox;
    com[F + f] = oy;
    if (z) z[f] = make_float2(ox * zscale, oy * zscale);
  }
  for (int o = 16; o > 0; o >>= 1) drop += __shfl_xor_sync(0xffffffffu, drop, o);
  if ((threadIdx.x & 31) == 0 && drop) {
    st_or(st, EER4D_ST_RANGE);
    st_add(st, 1, drop);
  }
}

// COM maps from per-frame sums [3][F] already formed (by the scatter pass of
// ssb_accumulate_com): the same centre and arithmetic as k_com.
__global__ void __launch_bounds__(kComThreads) k_com_from_sums(const long long* __restrict__ sums,
                                                               uint32_t F,
                                                               const long long* __restrict__ totals,
                                                               double cx_h, double cy_h,
                                                               float zscale, float* com, float2* z) {
  pdl_begin();
  __shared__ ComCentre s_c;
  if (threadIdx.x == 0) s_c = com_centre(totals, cx_h, cy_h);
  __syncthreads();
  const uint32_t f = blockIdx.x * kComThreads + threadIdx.x;
  if (f >= F) return;
  float ox, oy;
  com_of_frame(sums[f], sums[F + f], sums[2 * (size_t)F + f], s_c, ox, oy);
  com[f] = ox;
  com[F + f] = oy;
  if (z) z[f] = make_float2(ox * zscale, oy * zscale);
}

// ---------------------------------------------------------------- a4 -------
// Bin + crop + densify.  A persistent CTA takes tasks of TF consecutive frames
// (aligned to multiples of TF in the scan) x PC pixels: it counts into a
// shared tile and writes counts[p][f] as fp16.  No global atomics; every (p, f)
// of the chunk is written exactly once, zeros included.
//
// Counters.  A tile none of whose frames has more than 255 events counts in
// bytes, four frames per word; another one counts half its frames at a time, in
// 16-bit counters in the same words, 256 events of a frame in flight (the
// chunk's pixels in two or three passes, each over all events again and 64 in
// flight, before: whole accumulation of 512 x 512 frames, 553 pixels, of 300
// events each 900 -> 653 us, of 1200 2422 -> 1221).  Rows are padded by one word
// so the pixels of a frame fall in different banks.
//
// Pixel of an event.  The kept pixels of a detector row are one interval of
// raw x (a row of a disk, or of a shard of it), so the table is one entry per
// raw row: the interval's ends and the kept pixel at its start; one divide by
// det_w, one 8-byte load, one multiplication for the binning.
//
// Pipeline.  What bounded the kernel was latency (offsets, then events, then
// barriers) at 16 warps per SM.  Offsets are loaded two tasks ahead into
// registers and published to shared memory one task ahead; the first 64 events
// of a warp's four frames are loaded while the task before is written out, and
// those of its next four frames before the current ones are counted.  The
// write-out clears the counters it reads.
//
// Now bound by instruction issue (75 %): 1024 x 1024 frames of 50 events, 553
// pixels, 487 -> 324 us (210 for the bytes at 6.8 TB/s); 256 x 256 frames of 20
// events, 1345 pixels, 112 -> 48 us (27).
constexpr int kMaxFrameEvents = 65535;
constexpr int kScatterRowsSmem = 4096;  // most raw rows whose table is copied to shared memory

template <bool SUMS>
__global__ void __launch_bounds__(kThreads, 4) k_scatter(
    const uint32_t* __restrict__ idx, uint64_t n_idx, const uint64_t* __restrict__ off,
    uint64_t first, uint64_t nfr, uint32_t WH, uint32_t H, DivMod dw, uint32_t bin_m,
    uint32_t bin_one, const uint2* __restrict__ rows, int rows_smem, int P_pad, int TF, int PC, DivMod nch,
    uint32_t ntiles, int wide, uint64_t NR, __half* counts, long long* sums,
    unsigned long long* totals, uint64_t F, uint32_t* st) {
  pdl_begin();
  // SUMS: the same pass also forms each frame's COM sums (Sx, Sy, N over its
  // in-range events; Eq. 4) into sums[3][F] and adds them to totals[3] (the
  // PACBED centre), in the tasks of pixel chunk 0; events past the first
  // 65535 of a frame (EER4D_ST_OVERFLOW) are counted in neither.
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ uint64_t s_lo[2][128];  // event range of each frame, this task's and the next one's
  __shared__ uint32_t s_n[2][128];
  __shared__ uint32_t s_mx[2][4];    // most events in one frame, per warp that publishes
  constexpr int nw = kThreads / 32;  // a multiple of 4: frames nw apart share a byte position
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint2* srow = reinterpret_cast<const uint2*>(smem);
  uint32_t* tile = smem + (rows_smem ? (2 * H + 3) / 4 * 4 : 0);
  const int words = (PC * (TF / 4 + 1) + 3) / 4 * 4;
  if (rows_smem)
    for (uint32_t i = threadIdx.x; i < H; i += kThreads)
      reinterpret_cast<uint2*>(smem)[i] = __ldg(rows + i);
  for (int i = threadIdx.x; i < words / 4; i += kThreads)
    reinterpret_cast<uint4*>(tile)[i] = make_uint4(0u, 0u, 0u, 0u);
  const uint64_t T0 = (first / TF) * TF;
  const uint64_t end = first + nfr;
  unsigned long long tsx = 0, tsy = 0, tsn = 0;  // this lane's share of the totals
  uint32_t drop = 0, over = 0;

  // task tt: frames [tf0 + j0, tf0 + j1), pixels from p0 (the chunks of one
  // frame tile are neighbours, so its events come from L2 after the first)
  auto task = [&](uint32_t tt, uint64_t& tf0, int& j0, int& j1, int& p0) {
    uint32_t ft, ch;
    nch.divmod(tt, ft, ch);
    p0 = (int)ch * PC;
    tf0 = T0 + (uint64_t)ft * TF;
    j0 = tf0 < first ? (int)(first - tf0) : 0;
    j1 = tf0 + TF > end ? (int)(end - tf0) : TF;
  };
  uint64_t na = 0, nb = 0;  // threads < TF: off[f], off[f + 1] of a frame of the task to publish
  auto load_off = [&](uint32_t tt) {
    na = nb = 0;
    if ((int)threadIdx.x < TF && tt < ntiles) {
      uint64_t tf0;
      int j0, j1, p0;
      task(tt, tf0, j0, j1, p0);
      if ((int)threadIdx.x >= j0 && (int)threadIdx.x < j1) {
        const uint64_t f = tf0 + threadIdx.x - first;
        na = off[f];
        nb = off[f + 1];
      }
    }
  };
  auto publish = [&](int b) {
    if (warp >= 4) return;
    // frame_range on the offsets loaded before (0, 0 outside the task)
    const uint64_t lo = na < n_idx ? na : n_idx;
    const uint64_t t2 = nb > lo ? nb : lo;
    uint64_t hi = t2 < n_idx ? t2 : n_idx;
    bool bad = (nb < na) || (nb > n_idx) || (na > n_idx);
    if (hi - lo > kMaxFrameEvents) {
      bad = true;
      hi = lo + kMaxFrameEvents;
      st_or(st, EER4D_ST_OVERFLOW);
    }
    if (bad) st_or(st, EER4D_ST_OFFSETS);
    s_lo[b][threadIdx.x] = lo;
    s_n[b][threadIdx.x] = (uint32_t)(hi - lo);
    const uint32_t m = __reduce_max_sync(0xffffffffu, (uint32_t)(hi - lo));
    if (lane == 0) s_mx[b][warp] = m;
  };
  // events lane and lane + 32 of frames jg, jg + nw, jg + 2 nw, jg + 3 nw
  auto fetch = [&](int b, int jg, int j1, uint32_t (&v)[8]) {
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const int j = jg + f * nw;
      const uint32_t n = j < j1 ? s_n[b][j] : 0u;
      v[2 * f] = v[2 * f + 1] = 0u;
      if (lane < n) {
        const uint32_t* q = idx + s_lo[b][j] + lane;
        v[2 * f] = __ldg(q);
        if (lane + 32 < n) v[2 * f + 1] = __ldg(q + 32);
      }
    }
  };
  // counts the events of frames jg, jg + nw, .. below j1 into the tile of bytes (or
  // 16-bit counters from frame jb on) of pixels [p0, p0 + pc): their first 64 are
  // in v, the rest are loaded here, 64 (256) at a time; once: their sums and drops too
  // (a frame is counted for every chunk of pixels)
  const int TP = TF / 4 + 1;
  auto count = [&](auto bytes, int b, int jg, int jb, int j1, const uint32_t (&v)[8], int p0, int pc,
                   uint64_t tf0, bool once) {
    constexpr bool B = decltype(bytes)::value;
    constexpr int SH = B ? 2 : 1;
    const uint32_t inc = 1u << ((32 >> SH) * (jg & ((1 << SH) - 1)));
    [[maybe_unused]] uint32_t my_x = 0u, my_y = 0u, my_n = 0u;  // lane f: sums of frame f
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const int j = jg + f * nw;
      const uint32_t n = j < j1 ? s_n[b][j] : 0u;
      // 32-bit sums: at most 65535 events of x, y < 32768; of at most 255 events
      // the number rides in the top byte of x's, of more sn counts those dropped
      [[maybe_unused]] uint32_t sx = 0u, sy = 0u, sn = 0u;
      uint32_t* col = tile + ((j - jb) >> SH);
      auto one = [&](uint32_t e, bool has) {
        if (!has) return;
        if (e >= WH) {
          drop += once;
          if (SUMS && !B) ++sn;
          return;
        }
        uint32_t x, y;
        dw.divmod(e, y, x);
        if constexpr (SUMS) {
          sx += B ? x + (1u << 24) : x;
          sy += y;
        }
        const uint2 r = rows_smem ? srow[y] : __ldg(rows + y);
        const uint32_t t = x - r.x;  // raw pixels from the row's first kept one
        const int pp = (int)((r.y >> 16) + __umulhi(t, bin_m) + t * bin_one) - p0;
        if (t < (r.y & 0xffffu) && (unsigned)pp < (unsigned)pc &&
            EER4D_IN_RANGE(pp * TP + ((j - jb) >> SH), words, st))
          atomicAdd(col + pp * TP, inc);
      };
      one(v[2 * f], lane < n);
      one(v[2 * f + 1], lane + 32 < n);
      constexpr int NL = B ? 2 : 8;  // loads of a lane in flight
      for (uint32_t k = 64; k < n; k += 32 * NL) {
        const uint32_t* q = idx + s_lo[b][j] + k + lane;
        uint32_t e[NL];
#pragma unroll
        for (int i = 0; i < NL; ++i) e[i] = k + 32 * i + lane < n ? __ldg(q + 32 * i) : 0u;
#pragma unroll
        for (int i = 0; i < NL; ++i) {
          if (!B && k + 32 * i >= n) break;  // the same on every lane
          one(e[i], k + 32 * i + lane < n);
        }
      }
      if constexpr (SUMS) {
        if (once) {
          const uint32_t rx = __reduce_add_sync(0xffffffffu, sx);
          const uint32_t ry = __reduce_add_sync(0xffffffffu, sy);
          const uint32_t rn = B ? rx >> 24 : n - __reduce_add_sync(0xffffffffu, sn);
          if (lane == f) my_x = B ? rx & 0xffffffu : rx, my_y = ry, my_n = rn;
        }
      }
    }
    if constexpr (SUMS) {
      const int j = jg + lane * nw;
      if (once && lane < 4 && j < j1 && EER4D_IN_RANGE(tf0 + j, F, st)) {
        const uint64_t g = tf0 + j;  // frame of the dataset
        sums[g] = my_x;
        sums[F + g] = my_y;
        sums[2 * F + g] = my_n;
        tsx += my_x;
        tsy += my_y;
        tsn += my_n;
      }
    }
  };
  // With every count below 1024, OR-ing 0x6400 (fp16 1024.0) into a 16-bit
  // count n gives the fp16 of 1024 + n exactly; subtracting 1024 gives n.
  const __half2 k1024 = __floats2half2_rn(1024.f, 1024.f);
  auto to_half2 = [&](uint32_t m) {
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&m), k1024);
    return *reinterpret_cast<const uint32_t*>(&h);
  };
  // frames [j, j + 4) of pixel p (fp16 pairs) -> counts, those in [j0, j1)
  auto put4 = [&](int p, uint64_t tf0, int j, int j0, int j1, uint32_t a, uint32_t b) {
    if (j + 3 < j0 || j >= j1) return;
    if (!EER4D_IN_RANGE((long long)p * (long long)NR + (long long)tf0 + (j + 4 <= j1 ? j + 3 : j1 - 1),
                        (long long)P_pad * (long long)NR, st))
      return;
    __half* dst = counts + (size_t)p * NR + tf0 + j;
    if (j0 <= j && j + 4 <= j1) {
      *reinterpret_cast<uint2*>(dst) = make_uint2(a, b);
    } else {
      const uint32_t w[2] = {a, b};
      for (int k = 0; k < 4; ++k)
        if (j + k >= j0 && j + k < j1)
          dst[k] = __ushort_as_half((unsigned short)(w[k >> 1] >> (16 * (k & 1))));
    }
  };

  uint32_t pre[8];
  load_off(blockIdx.x);
  publish(0);
  load_off(blockIdx.x + gridDim.x);
  __syncthreads();
  if (blockIdx.x < ntiles) {
    uint64_t tf0;
    int j0, j1, p0;
    task(blockIdx.x, tf0, j0, j1, p0);
    fetch(0, j0 + warp, j1, pre);
  }
  int b = 0;
  for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x, b ^= 1) {
    uint64_t tf0;
    int j0, j1, p0;
    task(t, tf0, j0, j1, p0);
    const int pc = P_pad - p0 < PC ? P_pad - p0 : PC;
    publish(b ^ 1);
    load_off(t + 2 * gridDim.x);
    uint32_t mx = s_mx[b][0];
#pragma unroll
    for (int i = 1; i < 4; ++i) mx = mx > s_mx[b][i] ? mx : s_mx[b][i];
    const bool bytes = mx <= 255u;  // uniform
    auto prefetch_next = [&] {
      if (t + gridDim.x < ntiles) {
        uint64_t ntf0;
        int nj0, nj1, np0;
        task(t + gridDim.x, ntf0, nj0, nj1, np0);
        fetch(b ^ 1, nj0 + warp, nj1, pre);
      }
    };
    if (bytes) {
      for (int jg = j0 + warp; jg < j1; jg += 4 * nw) {
        uint32_t v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = pre[i];
        if (jg + 4 * nw < j1) fetch(b, jg + 4 * nw, j1, pre);
        count(std::true_type{}, b, jg, 0, j1, v, p0, pc, tf0, p0 == 0);
      }
      __syncthreads();
      prefetch_next();
      const int TW = TF / 4;
      if (wide && j0 == 0 && j1 == TF) {
        // a thread stays at eight frames of a row and steps down the rows
        const int qs = __ffs(TW / 2) - 1, step = kThreads >> qs;
        const int w = 2 * ((int)threadIdx.x & ((1 << qs) - 1));
        int p = threadIdx.x >> qs;
        uint32_t* c = tile + p * TP + w;
        __half* dst = counts + (size_t)(p0 + p) * NR + tf0 + 4 * w;
        const int cstep = step * TP;
        const size_t dstep = (size_t)step * NR;
#pragma unroll 2
        for (; p < pc; p += step, c += cstep, dst += dstep) {
          const uint32_t w0 = c[0], w1 = c[1];
          c[0] = c[1] = 0u;
          if (!EER4D_IN_RANGE((long long)(dst - counts) + 7, (long long)P_pad * (long long)NR, st)) continue;
          *reinterpret_cast<uint4*>(dst) = make_uint4(to_half2(__byte_perm(w0, 0x64646464u, 0x4140)),
                                                      to_half2(__byte_perm(w0, 0x64646464u, 0x4342)),
                                                      to_half2(__byte_perm(w1, 0x64646464u, 0x4140)),
                                                      to_half2(__byte_perm(w1, 0x64646464u, 0x4342)));
        }
      } else {
        const int qs = __ffs(TW) - 1;
        for (int i = threadIdx.x; i < pc << qs; i += kThreads) {
          const int p = i >> qs, w = i & (TW - 1);
          const uint32_t w0 = tile[p * TP + w];
          tile[p * TP + w] = 0u;
          put4(p0 + p, tf0, 4 * w, j0, j1, to_half2(__byte_perm(w0, 0x64646464u, 0x4140)),
               to_half2(__byte_perm(w0, 0x64646464u, 0x4342)));
        }
      }
    } else {
      const int TH = TF / 2;                  // frames of a half: TF / 4 words of two
      const int step = TF >= 8 ? 2 : 1;       // words stored at a time
      const int qs = __ffs(TF / 4 / step) - 1;
      for (int jb = 0; jb < TF; jb += TH) {
        const int ja = jb > j0 ? jb : j0, je = jb + TH < j1 ? jb + TH : j1;
        if (ja >= je) continue;  // uniform
        // pre holds the first frames from ja on: of the task, or of its second half
        for (int jg = ja + warp; jg < je; jg += 4 * nw) {
          uint32_t v[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = pre[i];
          if (jg + 4 * nw < je) fetch(b, jg + 4 * nw, je, pre);
          count(std::false_type{}, b, jg, jb, je, v, p0, pc, tf0, p0 == 0);
        }
        __syncthreads();
        if (je < j1) fetch(b, je + warp, j1, pre);
        else prefetch_next();
        for (int i = threadIdx.x; i < pc << qs; i += kThreads) {
          const int p = i >> qs, w = (i & ((1 << qs) - 1)) * step;
          uint32_t* c = tile + p * TP + w;
          const uint32_t w0 = c[0], w1 = step == 2 ? c[1] : 0u;
          c[0] = 0u;
          if (step == 2) c[1] = 0u;
          uint32_t h01, h23;
          if (mx < 1024u) {
            h01 = to_half2(w0 | 0x64006400u);
            h23 = to_half2(w1 | 0x64006400u);
          } else {
            const uint32_t q0 = w0 & 0xffffu, q1 = w0 >> 16, q2 = w1 & 0xffffu, q3 = w1 >> 16;
            over += (q0 > 2048u) + (q1 > 2048u) + (q2 > 2048u) + (q3 > 2048u);
            const __half2 a = __halves2half2(__ushort2half_rn((unsigned short)q0), __ushort2half_rn((unsigned short)q1));
            const __half2 d = __halves2half2(__ushort2half_rn((unsigned short)q2), __ushort2half_rn((unsigned short)q3));
            h01 = *reinterpret_cast<const uint32_t*>(&a);
            h23 = *reinterpret_cast<const uint32_t*>(&d);
          }
          put4(p0 + p, tf0, jb + 2 * w, ja, je, h01, h23);
        }
        if (je < j1) __syncthreads();
      }
    }
    __syncthreads();
  }
  for (int o = 16; o > 0; o >>= 1) {
    drop += __shfl_xor_sync(0xffffffffu, drop, o);
    over += __shfl_xor_sync(0xffffffffu, over, o);
  }
  if (SUMS) tsx = warp_sum_ll(tsx), tsy = warp_sum_ll(tsy), tsn = warp_sum_ll(tsn);
  if (lane == 0) {
    if (drop) { st_or(st, EER4D_ST_RANGE); st_add(st, 1, drop); }
    if (over) { st_or(st, EER4D_ST_OVERFLOW); st_add(st, 2, over); }
    if (SUMS && tsn) {
      atomicAdd(totals + 0, tsx);
      atomicAdd(totals + 1, tsy);
      atomicAdd(totals + 2, tsn);
    }
  }
}

}  // namespace

// Shared memory for the counters of a task: two CTAs per SM when all of it is
// taken.  Counting 1345 pixels in one chunk of 92 KB beats two of 46 KB at four
// CTAs per SM, whose events are read and looked up twice (256 x 256 scan, whole
// path 391 against 397 us; 336 x 200, 807 against 835).
constexpr size_t kScatterTileBytes = 96 * 1024;

// Pixels of a task: all of them when their byte counters fit the tile, or
// equal chunks that do (each chunk re-reads the events of its frames, from L2).
static int scatter_pc(int P_pad, int TF) {
  int most = (int)(kScatterTileBytes / ((size_t)(TF / 4 + 1) * 4)) / 16 * 16;
  if (most < 16) most = 16;
  const int n = (P_pad + most - 1) / most;
  return ((P_pad + n - 1) / n + 15) / 16 * 16;
}

// Frames of a task unless tuned: 64 (128-byte rows of counts), fewer on scans
// too small to give every SM two tasks of that size.  (1024 x 1024: whole path
// 2058 us at 64 frames, 2125 at 32, 2325 at 128.)
int scatter_tf_for(const eer4d_plan* p) {
  if (p->tune.scatter_tf > 0) return p->tune.scatter_tf;
  int tf = 64;
  auto tasks = [&] {
    const int pc = scatter_pc(p->P_pad, tf);
    return (long long)(p->F / tf) * ((p->P_pad + pc - 1) / pc);
  };
  while (tf > 16 && tasks() < 2 * kSms)
    tf /= 2;
  return tf;
}

cudaError_t launch_validate(const eer4d_plan* p, const uint32_t* idx, uint64_t n_idx,
                            const uint64_t* off, uint64_t n_frames, int64_t* pacbed,
                            int64_t* totals, uint32_t* st, cudaStream_t s) {
  const uint64_t work = n_frames > n_idx / 16 ? n_frames : n_idx / 16;
  uint64_t blocks = (work + kThreads - 1) / kThreads;
  // one full wave of 152 SMs, no partial second one (resident CTAs of 48 registers
  // a thread, 64 with the PACBED)
  auto kv = pacbed ? k_validate<true> : k_validate<false>;
  const uint64_t wave = kSms * (pacbed ? 4 : 5);
  if (blocks > wave) blocks = wave;
  if (blocks == 0) blocks = 1;
  stage_begin(p, EER4D_STAGE_VALIDATE, s);
  launch(kv, (unsigned)blocks, kThreads, 0, s, idx, n_idx, off, n_frames,
         p->g.det_w * p->g.det_h, p->dw, reinterpret_cast<unsigned long long*>(pacbed),
         reinterpret_cast<unsigned long long*>(totals), st);
  count_launches(1);
  stage_end(p, EER4D_STAGE_VALIDATE, s);
  return cudaGetLastError();
}

cudaError_t launch_com(const eer4d_plan* p, const uint32_t* idx, uint64_t n_idx, const uint64_t* off,
                       int64_t* sums, float* com, float2* z, const int64_t* totals, double cx,
                       double cy, uint32_t* st, cudaStream_t s) {
  const uint32_t F = (uint32_t)p->F;
  const float zscale = (float)(p->g.dalpha_raw_rad / p->g.lambda_A);
  stage_begin(p, EER4D_STAGE_COM, s);
  // A thread takes a frame, so the blocks of long frames should be spread evenly
  // over the SMs.  Started ahead of the end of the kernel before they gather on the
  // SMs that it leaves first; with few events the earlier start is worth more.
  // (Validation and COM of 256 x 256 frames of 1200, 200, 50 and 30 events: 259, 74,
  // 42 and 33 us overlapped, 209, 64, 40 and 37 in order; 64 x 64 frames of 100
  // events 29 and 31.)
  const bool in_order = n_idx >= 64 * (uint64_t)F && F >= 64 * kComThreads;
  launch_as(!in_order, k_com, (F + kComThreads - 1) / kComThreads, kComThreads, 0, s, idx, n_idx, off, F,
         p->g.det_w * p->g.det_h, p->dw, reinterpret_cast<const long long*>(totals), cx, cy, zscale,
         reinterpret_cast<long long*>(sums), com, z, st);
  count_launches(1);
  stage_end(p, EER4D_STAGE_COM, s);
  return cudaGetLastError();
}

cudaError_t launch_com_from_sums(const eer4d_plan* p, const int64_t* sums, float* com, float2* z,
                                 const int64_t* totals, double cx, double cy, cudaStream_t s) {
  const uint32_t F = (uint32_t)p->F;
  const float zscale = (float)(p->g.dalpha_raw_rad / p->g.lambda_A);
  stage_begin(p, EER4D_STAGE_COM, s);
  launch(k_com_from_sums, (F + kComThreads - 1) / kComThreads, kComThreads, 0, s,
         reinterpret_cast<const long long*>(sums), F, reinterpret_cast<const long long*>(totals), cx,
         cy, zscale, com, z);
  count_launches(1);
  stage_end(p, EER4D_STAGE_COM, s);
  return cudaGetLastError();
}

cudaError_t launch_scatter(const eer4d_plan* p, const uint32_t* idx, uint64_t n_idx,
                           const uint64_t* off, uint64_t first, uint64_t n, __half* counts,
                           uint32_t* st, cudaStream_t s, int64_t* sums, int64_t* totals) {
  if (n == 0) return cudaSuccess;
  const int TF = scatter_tf_for(p);
  const int PC = scatter_pc(p->P_pad, TF);
  const int NCH = (p->P_pad + PC - 1) / PC;
  const uint32_t W = p->g.det_w, H = p->g.det_h;
  const size_t words = ((size_t)PC * (TF / 4 + 1) + 3) / 4 * 4;
  // row table in shared memory unless the detector is very tall
  const int rows_smem = H <= kScatterRowsSmem;
  const size_t sm = 4 * (words + (rows_smem ? (2 * (size_t)H + 3) / 4 * 4 : 0));
  // 16-byte stores when every row of counts starts on 16 bytes
  const int wide = TF >= 8 && p->cstride % 8 == 0 && reinterpret_cast<uintptr_t>(counts) % 16 == 0;
  const bool with_sums = sums != nullptr;
  const void* kern = with_sums ? (const void*)k_scatter<true> : (const void*)k_scatter<false>;
  cudaError_t e = ensure_smem(kern, sm);
  if (e != cudaSuccess) return e;
  const uint64_t T0 = (first / TF) * TF;
  const uint64_t tiles = (first + n - T0 + TF - 1) / TF * NCH;
  if (tiles >= (1ull << 31)) return cudaErrorInvalidValue;  // 32-bit tile indices in the kernel
  DivMod nch;
  nch.init((uint32_t)NCH);
  int dev = 0, nsm = 0, occ = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kThreads, sm);
  if (occ < 1) return cudaErrorInvalidConfiguration;  // the tile does not fit shared memory
  // tuned values from kScatterAll on mean all the CTAs that fit (kept tunings were
  // made when that was three at most): 1024 x 1024 frames of 50 events, 553 pixels,
  // 341 us with three, 325 with the four that fit
  constexpr int kScatterAll = 3;
  const int most = p->tune.scatter_ctas_per_sm;
  const int cps = most > 0 && most < kScatterAll && most < occ ? most : occ;
  uint64_t grid = (uint64_t)nsm * cps;
  if (grid > tiles) grid = tiles;
  stage_begin(p, EER4D_STAGE_SCATTER, s);
  auto kl = with_sums ? k_scatter<true> : k_scatter<false>;
  launch(kl, (unsigned)grid, kThreads, sm, s, idx, n_idx, off, first, n, W * H, H, p->dw, p->bin_m,
         p->bin_one, p->d_rowtab, rows_smem, p->P_pad, TF, PC, nch, (uint32_t)tiles, wide,
         (uint64_t)p->cstride, counts, reinterpret_cast<long long*>(sums),
         reinterpret_cast<unsigned long long*>(totals), (uint64_t)p->F, st);
  count_launches(1);
  stage_end(p, EER4D_STAGE_SCATTER, s);
  return cudaGetLastError();
}
