// Run-length-encoded EER (Sec. II, Fig. 1c): within a frame the hits are in
// ascending linear index and each run is the distance from the previous hit
// (run 0: from pixel 0).  Re-coding to linear-index encoding is an O(C)
// segmented inclusive prefix sum: idx_j = run_0 + ... + run_j.
//
// A warp takes up to 32 consecutive frames and walks their events, which are
// one stretch of the array, 128 at a time (16-byte loads and stores), whatever
// the frames' lengths: sums inside a lane's four events, one warp scan of the
// lanes' sums, frame starts as bytes in shared memory.  The sums are 32 bits
// wide; a sum beyond the uint32 range shows as an event whose sum is below its
// own run, and every later event of its frame is then beyond it too.  Frames
// whose offsets are not ascending within the array take the form below, one
// frame at a time in 64 bits.  (That form alone, a 64-bit scan of 32 runs at a
// time, was bound by instruction issue, 70 %: 52e6 events of 1024 x 1024 frames
// 265 us, this 73, of 62 for the bytes at 6.8 TB/s.)
#include "common.cuh"

namespace {

constexpr int kWarpsPerBlock = 8;

__device__ __forceinline__ unsigned long long warp_incl_scan_u64(unsigned long long v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// one frame in 64 bits (whole warp); true in the lanes that saw a sum out of range
__device__ bool decode_frame(const uint32_t* runs, uint64_t lo, uint64_t hi, uint32_t* idx, int lane) {
  unsigned long long carry = 0ull;
  bool over = false;
  for (uint64_t base = lo; base < hi; base += 32) {  // uniform trip count per warp
    const uint64_t i = base + lane;
    const unsigned long long r = i < hi ? (unsigned long long)runs[i] : 0ull;
    const unsigned long long s = carry + warp_incl_scan_u64(r, lane);
    if (i < hi) {
      const bool big = s > 0xFFFFFFFFull;
      over |= big;
      idx[i] = big ? 0xFFFFFFFFu : (uint32_t)s;
    }
    carry = __shfl_sync(0xffffffffu, s, 31);
  }
  return over;
}

// VEC: runs and idx are congruent modulo 16 bytes (base_al: elements from the
// 16-byte boundary at or before them)
template <bool VEC>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
    k_rle_decode(const uint32_t* runs, uint64_t n, const uint64_t* __restrict__ off,
                 uint64_t n_frames, int per_warp, int base_al, uint32_t* idx, uint32_t* st) {
  pdl_begin();
  __shared__ uint32_t s_head[kWarpsPerBlock][2][32];  // a byte per event: 1 at a frame's first
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint64_t f0 = ((uint64_t)blockIdx.x * kWarpsPerBlock + warp) * per_warp;
  if (f0 >= n_frames) return;  // whole warp
  const int nf = n_frames - f0 < (uint64_t)per_warp ? (int)(n_frames - f0) : per_warp;
  const uint64_t a = off[f0 + (lane < nf ? lane : nf)];
  const uint64_t b = off[f0 + (lane < nf ? lane + 1 : nf)];
  const uint64_t lo = __shfl_sync(0xffffffffu, a, 0);
  const uint64_t hi = __shfl_sync(0xffffffffu, b, nf - 1);
  const bool bad = (b < a) || (b > n) || (a > n);
  const bool any_bad = __any_sync(0xffffffffu, bad);
  bool over = false;
  if (any_bad || hi - lo >= (1ull << 30)) {
    if (any_bad && lane == 0) st_or(st, EER4D_ST_OFFSETS);
    for (int j = 0; j < nf; ++j) {
      const uint64_t fa = __shfl_sync(0xffffffffu, a, j), fb = __shfl_sync(0xffffffffu, b, j);
      const uint64_t l = fa < n ? fa : n;
      const uint64_t t = fb > l ? fb : l;
      over |= decode_frame(runs, l, t < n ? t : n, idx, lane);
    }
    if (over) st_or(st, EER4D_ST_RANGE);
    return;
  }
  // chunks of 128 events from the 16-byte boundary at or before event lo
  const int pad = (int)((lo + (uint64_t)base_al) & 3);
  const int m = (int)(hi - lo) + pad;              // events [pad, m) of the chunks are the warp's
  const uint32_t* src = runs + lo - pad;
  uint32_t* dst = idx + lo - pad;
  const int start = lane < nf && b > a ? (int)(a - lo) + pad : -1;  // first event of a frame that has any
  auto load = [&](int c, uint32_t (&r)[4]) {
    const int k = c + 4 * lane;
    if (VEC && k >= pad && k + 4 <= m) {
      const uint4 q = *reinterpret_cast<const uint4*>(src + k);
      r[0] = q.x; r[1] = q.y; r[2] = q.z; r[3] = q.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) r[i] = k + i >= pad && k + i < m ? src[k + i] : 0u;
    }
  };
  uint32_t carry = 0u, r[4], nx[4];
  bool cbig = false;  // the frame at the chunk's start is already out of range
  int buf = 0;
  load(0, nx);
  for (int c = 0; c < m; c += 128, buf ^= 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i) r[i] = nx[i];
    if (c + 128 < m) load(c + 128, nx);
    uint32_t* hd = s_head[warp][buf];
    hd[lane] = 0u;
    __syncwarp();
    if (start >= c && start < c + 128) reinterpret_cast<unsigned char*>(hd)[start - c] = 1;
    __syncwarp();
    const uint32_t w = hd[lane];
    const bool h0 = w & 0x1u, h1 = w & 0x100u, h2 = w & 0x10000u, h3 = w & 0x1000000u;
    // sums since the lane's first event or its last frame start
    uint32_t v[4];
    v[0] = r[0];
    v[1] = (h1 ? 0u : v[0]) + r[1];
    v[2] = (h2 ? 0u : v[1]) + r[2];
    v[3] = (h3 ? 0u : v[2]) + r[3];
    uint32_t T = v[3];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, T, o);
      if (lane >= o) T += y;
    }
    const uint32_t ex = T - v[3];                             // lanes before this one
    const uint32_t heads = __ballot_sync(0xffffffffu, w != 0u);
    const uint32_t before = heads & ((1u << lane) - 1u);
    const int hl = before ? 31 - __clz(before) : 0;           // last lane before with a frame start
    const uint32_t exh = __shfl_sync(0xffffffffu, ex, hl);
    const uint32_t in = before ? ex - exh : ex + carry;       // sum of the open frame before this lane
    const bool o0 = !h0, o1 = o0 && !h1, o2 = o1 && !h2, o3 = o2 && !h3;
    v[0] += o0 ? in : 0u;
    v[1] += o1 ? in : 0u;
    v[2] += o2 ? in : 0u;
    v[3] += o3 ? in : 0u;
    const bool w0 = v[0] < r[0], w1 = v[1] < r[1], w2 = v[2] < r[2], w3 = v[3] < r[3];
    if (__any_sync(0xffffffffu, w0 | w1 | w2 | w3 | cbig)) {
      // out of range from the first wrapped event to the end of its frame
      const bool b0 = w0, b1 = w1 || (b0 && !h1), b2 = w2 || (b1 && !h2), b3 = w3 || (b2 && !h3);
      const uint32_t bigs = __ballot_sync(0xffffffffu, b3);
      // lanes from the last frame start to the one before this
      const uint32_t span = ((1u << lane) - 1u) & ~((1u << hl) - 1u);
      const bool bin = (bigs & span) != 0u || (!before && cbig);
      const bool q0 = b0 || (o0 && bin), q1 = b1 || (o1 && bin), q2 = b2 || (o2 && bin), q3 = b3 || (o3 && bin);
      const int k = c + 4 * lane;
      over |= (q0 && k < m) || (q1 && k + 1 < m) || (q2 && k + 2 < m) || (q3 && k + 3 < m);
      cbig = __shfl_sync(0xffffffffu, (int)q3, 31) != 0;
      carry = __shfl_sync(0xffffffffu, v[3], 31);
      if (q0) v[0] = 0xFFFFFFFFu;
      if (q1) v[1] = 0xFFFFFFFFu;
      if (q2) v[2] = 0xFFFFFFFFu;
      if (q3) v[3] = 0xFFFFFFFFu;
    } else {
      carry = __shfl_sync(0xffffffffu, v[3], 31);
    }
    const int k = c + 4 * lane;
    if (!EER4D_IN_RANGE(lo - pad + (k + 4 <= m ? k + 3 : m - 1), n, st)) continue;
    if (VEC && k >= pad && k + 4 <= m) {
      *reinterpret_cast<uint4*>(dst + k) = make_uint4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (k + i >= pad && k + i < m) dst[k + i] = v[i];
    }
  }
  if (over) st_or(st, EER4D_ST_RANGE);
}

}  // namespace

cudaError_t launch_rle_decode(const uint32_t* runs, uint64_t n, const uint64_t* off,
                              uint64_t n_frames, uint32_t* idx, uint32_t* st, cudaStream_t s) {
  if (n_frames == 0) return cudaSuccess;
  // frames of a warp: enough warps to fill the GPU first (48 per SM)
  const uint64_t want = n_frames / (kSms * 48);
  const int per_warp = want < 1 ? 1 : want > 32 ? 32 : (int)want;
  const uint64_t blocks = (n_frames + (uint64_t)kWarpsPerBlock * per_warp - 1) / ((uint64_t)kWarpsPerBlock * per_warp);
  const uintptr_t pr = reinterpret_cast<uintptr_t>(runs), pi = reinterpret_cast<uintptr_t>(idx);
  const bool vec = (pr & 15) == (pi & 15);
  launch(vec ? k_rle_decode<true> : k_rle_decode<false>, (unsigned)blocks, kWarpsPerBlock * 32, 0, s, runs,
         n, off, n_frames, per_warp, (int)((pr & 15) >> 2), idx, st);
  count_launches(1);
  return cudaGetLastError();
}
