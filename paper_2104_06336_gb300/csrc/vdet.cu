// Virtual detectors from linear-index EER (Table 1: operations that scale with
// the number of counts): per frame, the number of events in each of n_rings
// annuli about the pattern centre, the annular bright-field, annular
// dark-field or radial-sum images of a pixelated detector, in O(C).
//
// Ring j holds the raw pixels (x, y) with r_j^2 <= (x - cx)^2 + (y - cy)^2 <
// r_{j+1}^2, every square and sum in double with round-to-nearest and no
// fused multiply-add, so an independent float64 evaluation in the same order
// decides every pixel the same way.  A first kernel writes the ring of every
// detector pixel into a table (W*H bytes of scratch); the second walks the
// frames and looks each event up in it.
#include "common.cuh"

namespace {

struct Rings {
  int n;                              // rings
  double r2[EER4D_MAX_RINGS + 1];     // squared radii, ascending
};

// the ring of raw pixel (x, y), -1: none
__device__ __noinline__ int exact_ring(uint32_t x, uint32_t y, double cx, double cy, const Rings& R) {
  const double dx = __dsub_rn((double)x, cx);
  const double dy = __dsub_rn((double)y, cy);
  const double r2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
  if (r2 >= R.r2[0])
    for (int j = 0; j < R.n; ++j)
      if (r2 < R.r2[j + 1]) return j;
  return -1;
}

// Table of the pixels' rings, a byte each (255: none), eight pixels of linear
// index a thread.  A pixel is decided in float32 unless it is within float32's
// error of an edge, and the centre and edges are formed once a block (double
// precision runs at two lanes a cycle: 576 x 576 pixels took 16 us in it, a
// thread each; now 10).  The edges are searched by halving: one after another, 64
// rings of 256 x 256 frames of 20 events took 93 us, 12 rings 29; now 56 and 21.
constexpr int kTableThreads = 256;
__global__ void __launch_bounds__(kTableThreads)
    k_ring_table(uint32_t WH, DivMod dw, const long long* __restrict__ totals, double cx_h,
                 double cy_h, const __grid_constant__ Rings R, unsigned char* lut) {
  pdl_begin();
  __shared__ float s_lo[EER4D_MAX_RINGS + 1], s_hi[EER4D_MAX_RINGS + 1];
  __shared__ double s_c[2];
  if (threadIdx.x == 0) {
    double cx = cx_h, cy = cy_h;
    if (totals) {
      const long long n = totals[2];
      cx = n ? (double)totals[0] / (double)n : 0.0;
      cy = n ? (double)totals[1] / (double)n : 0.0;
    }
    s_c[0] = cx;
    s_c[1] = cy;
  }
  // a pixel whose float32 squared radius is outside [s_lo, s_hi] is on the same
  // side of edge j as that number; an edge at radius 0 is below every pixel
  if (threadIdx.x >= 32)
    for (int j = threadIdx.x - 32; j <= R.n; j += kTableThreads - 32) {
      const double r2 = R.r2[j] < 1e30 ? R.r2[j] : 1e30;
      const double e = (r2 + 1.0) * 0x1p-19;
      s_lo[j] = r2 > 0.0 ? __double2float_rd(r2 - e) : -2.f;
      s_hi[j] = r2 > 0.0 ? __double2float_ru(r2 + e) : -1.f;
    }
  __syncthreads();
  const double cx = s_c[0], cy = s_c[1];
  // The centre as integer plus fraction: x - round(cx) is exact, and float32
  // rounds x - cx and the squared radius to within 2^-21 (r^2 + 1); pixels are
  // all decided in double about centres too far away for that (or not finite).
  const double rx = rint(cx), ry = rint(cy);
  const bool near = fabs(rx) < 1048576.0 && fabs(ry) < 1048576.0;
  const int ix = near ? (int)rx : 0, iy = near ? (int)ry : 0;
  const float gx = near ? (float)(cx - rx) : 0.f, gy = near ? (float)(cy - ry) : 0.f;
  const uint32_t n8 = (WH + 7) / 8;
  for (uint32_t i = blockIdx.x * kTableThreads + threadIdx.x; i < n8; i += gridDim.x * kTableThreads) {
    uint32_t pack[2] = {0u, 0u};
    uint32_t x, y;
    dw.divmod(i * 8, y, x);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float dx = (float)((int)x - ix) - gx, dy = (float)((int)y - iy) - gy;
      const float r2 = fmaf(dx, dx, __fmul_rn(dy, dy));
      int c = 0;  // edges below the pixel: s_hi ascends
      for (int n = R.n + 1; n > 0;) {
        const int h = n >> 1;
        const bool up = s_hi[c + h] < r2;
        c = up ? c + h + 1 : c;
        n = up ? n - h - 1 : h;
      }
      const bool sure = near && (c > R.n || r2 < s_lo[c]);
      const int ring = sure ? (c > R.n ? -1 : c - 1) : exact_ring(x, y, cx, cy, R);
      pack[k >> 2] |= (uint32_t)(ring & 255) << (8 * (k & 3));
      if (++x == dw.d) x = 0, ++y;
    }
    if (i * 8 + 7 < WH && reinterpret_cast<uintptr_t>(lut) % 8 == 0) {
      reinterpret_cast<uint2*>(lut)[i] = make_uint2(pack[0], pack[1]);
    } else {
      for (uint32_t k = 0; k < 8 && i * 8 + k < WH; ++k)
        lut[(size_t)i * 8 + k] = (unsigned char)(pack[k >> 2] >> (8 * (k & 3)));
    }
  }
}

// A warp takes `per` consecutive frames at a time (4 to 32), four at once: the
// first 64 events of each are loaded before any is looked up.  Counts go to the
// warp's shared memory [frame][ring] (an odd pitch: the lanes are in one frame,
// its rings in different banks) and leave as rows of `per` frames.
// Bound by instruction issue and the latency of the lookups, which a lane's
// eight events in flight overlap: 52e6 events of 1024 x 1024 frames 92 us, from
// 181 with one in flight and 64-bit event numbers (32 for the bytes).  The table
// in shared memory at four bits a pixel took 99; computing each event's radius
// instead of looking its ring up, 184.
constexpr int kWarps = 8;
__global__ void __launch_bounds__(kWarps * 32, 5)
    k_ring_counts(const uint32_t* __restrict__ idx, uint64_t n_idx,
                  const uint64_t* __restrict__ off, uint64_t n_frames, int per_log2, uint32_t WH,
                  const unsigned char* __restrict__ lut, int n_rings, int32_t* out, uint32_t* st) {
  pdl_begin();
  extern __shared__ int smem[];  // [kWarps][per][pitch]
  const int pitch = n_rings | 1, per = 1 << per_log2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* cnt = smem + warp * per * pitch;
  for (int i = lane; i < per * pitch; i += 32) cnt[i] = 0;
  __syncwarp();
  bool bad = false;
  uint32_t vmax = 0;  // largest index seen
  constexpr uint64_t kSpan = 1ull << 30;  // events of a frame counted with 32-bit offsets
  const uint64_t f0 = ((uint64_t)blockIdx.x * kWarps + warp) << per_log2;
  if (f0 < n_frames) {
    // lane l: the events of frame f0 + l
    const uint64_t f = f0 + lane;
    const bool mine = lane < per && f < n_frames;
    const uint64_t a = mine ? off[f] : 0, b = mine ? off[f + 1] : 0;
    uint64_t lo = a < n_idx ? a : n_idx;
    const uint64_t t = b > lo ? b : lo;
    uint64_t left = (t < n_idx ? t : n_idx) - lo;
    bad |= (b < a) || (b > n_idx) || (a > n_idx);
    do {
      const uint32_t now = left < kSpan ? (uint32_t)left : (uint32_t)kSpan;
      for (int s = 0; s < per; s += 4) {
        const uint32_t* ev[4];
        uint32_t n[4], most = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          ev[q] = idx + __shfl_sync(0xffffffffu, lo, s + q) + lane;
          n[q] = __shfl_sync(0xffffffffu, now, s + q);
          most = n[q] > most ? n[q] : most;
        }
        for (uint32_t k0 = 0; k0 < most; k0 += 64) {
          uint32_t v[8];
          bool has[8];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            has[2 * q] = k0 + lane < n[q];
            has[2 * q + 1] = k0 + lane + 32 < n[q];
            v[2 * q] = v[2 * q + 1] = 0u;
            if (has[2 * q]) v[2 * q] = __ldg(ev[q]);
            if (has[2 * q + 1]) v[2 * q + 1] = __ldg(ev[q] + 32);
            ev[q] += 64;
          }
          int ring[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            vmax = v[i] > vmax ? v[i] : vmax;
            has[i] = has[i] && v[i] < WH;
            ring[i] = (int)__ldg(lut + (has[i] ? v[i] : 0u));
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            int* c = cnt + (s + q) * pitch;
            if (has[2 * q] && ring[2 * q] != 255 && EER4D_IN_RANGE(ring[2 * q], n_rings, st))
              atomicAdd(c + ring[2 * q], 1);
            if (has[2 * q + 1] && ring[2 * q + 1] != 255 && EER4D_IN_RANGE(ring[2 * q + 1], n_rings, st))
              atomicAdd(c + ring[2 * q + 1], 1);
          }
        }
      }
      lo += now;
      left -= now;
    } while (__any_sync(0xffffffffu, left > 0));
    __syncwarp();
    for (int i = lane; i < n_rings << per_log2; i += 32) {
      const int j = i >> per_log2, fl = i & (per - 1);
      if (f0 + fl < n_frames) out[(size_t)j * n_frames + f0 + fl] = cnt[fl * pitch + j];
    }
  }
  if (bad) st_or(st, EER4D_ST_OFFSETS);
  if (vmax >= WH) st_or(st, EER4D_ST_RANGE);
}

}  // namespace

cudaError_t launch_virtual_detectors(const eer4d_plan* p, const uint32_t* idx, uint64_t n_idx,
                                     const uint64_t* off, uint64_t n_frames, const double* radii,
                                     int n_rings, const int64_t* totals, double cx, double cy,
                                     void* scratch, int32_t* out, uint32_t* st, cudaStream_t s) {
  Rings R;
  R.n = n_rings;
  for (int j = 0; j <= n_rings; ++j) R.r2[j] = radii[j] * radii[j];
  for (int j = n_rings + 1; j <= EER4D_MAX_RINGS; ++j) R.r2[j] = 0.0;
  unsigned char* lut = static_cast<unsigned char*>(scratch);
  const uint32_t WH = p->g.det_w * p->g.det_h;
  launch(k_ring_table, kSms, kTableThreads, 0, s, WH, p->dw, reinterpret_cast<const long long*>(totals), cx,
         cy, R, lut);
  count_launches(1);
  if (n_frames == 0) return cudaGetLastError();
  // Frames a warp takes at a time: as many as leave every SM 32 warps with
  // work, 32 (128-byte rows of counts) at most, the counts of a block within 28 KB.
  const size_t frame = sizeof(int) * (size_t)(n_rings | 1) * kWarps;
  int per_log2 = 2;
  while (per_log2 < 5 && (n_frames >> (per_log2 + 1)) >= kSms * 32 && frame << (per_log2 + 1) <= 28 * 1024) ++per_log2;
  const size_t sm = frame << per_log2;
  const uint64_t span = (uint64_t)kWarps << per_log2;
  const uint64_t blocks = (n_frames + span - 1) / span;
  launch(k_ring_counts, (unsigned)blocks, kWarps * 32, sm, s, idx, n_idx, off, n_frames, per_log2, WH, lut,
         n_rings, out, st);
  count_launches(1);
  return cudaGetLastError();
}
