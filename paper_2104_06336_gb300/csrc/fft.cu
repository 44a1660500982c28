// Scan-axis transforms: the G function (Sec. IV, G(k,K) = F_{R->K} I(k,R)),
// the inverse transform of the SSB spectrum to the phase image, the forward
// transform of an upstream phase gradient, and the Fourier integration of the
// COM field (Sec. V).  Power-of-two lengths up to 1024 run in registers
// (fft_reg.cuh), every other length in shared memory (fft.cuh); real data use
// the two-real-rows-in-one-complex-transform form.
#include "fft.cuh"
#include "fft_reg.cuh"
#include "fft_warp.cuh"

namespace {

constexpr int kThreads = 256;
// k_gen_rows and k_rows_c2c: few transforms in small CTAs, whose barriers wait for
// less; registers for eight CTAs per SM (seven where they hold a radix above 16),
// of which shared memory leaves eight with rows of 200 points, five with 336 and
// four with 400.  (Scan DFT of 336 x 200 positions, 1248 pixels, 328 us; budgets of
// six, eight and five CTAs 341, 373 and 396; 200 x 336 377, 402, 387, 451; without
// radices above 16, 300 x 128 with eight 207, six 211, 90 x 66 72 and 78.  Longer
// rows do not tell eight, seven and six apart: 800 x 600, 1000 x 1000.)
constexpr int kDirectThreads = 128;
constexpr int direct_blocks(bool big) { return big ? 7 : 8; }

// Column transforms of a [N][ld] complex array (element n of column c at
// n*ld + c), nb (a power of two) columns per CTA, batch = blockIdx.y.
template <int DIR>
__global__ void __launch_bounds__(kThreads) k_fft_cols(const float2* in, float2* out, const __grid_constant__ FftDesc d,
                                                       int ncols, int ld_in, int ld_out,
                                                       long long bs_in, long long bs_out, int nb,
                                                       int pitch, float scale) {
  pdl_begin();
  const int N = d.N, sh = __ffs(nb) - 1;
  float2* A = fft_sm;
  const int c0 = blockIdx.x * nb;
  in += blockIdx.y * bs_in;
  out += blockIdx.y * bs_out;
  const int tot = N * nb;
  for (int w = threadIdx.x; w < tot; w += blockDim.x) {
    const int n = w >> sh, b = w & (nb - 1), c = c0 + b;
    A[b * pitch + n] = c < ncols ? in[(size_t)n * ld_in + c] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  const float2* res = fft_sm + fft_smem<DIR>(d, nb, pitch);
  for (int w = threadIdx.x; w < tot; w += blockDim.x) {
    const int n = w >> sh, b = w & (nb - 1), c = c0 + b;
    if (c < ncols) out[(size_t)n * ld_out + c] = cscale(res[b * pitch + n], scale);
  }
}

template <typename T>
__device__ __forceinline__ float to_f(T v);
template <>
__device__ __forceinline__ float to_f<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f<__half>(__half v) { return __half2float(v); }

// the pair's half spectra at k from Z = F(row_a + i row_b)
__device__ __forceinline__ float2 split_a(float2 z, float2 zm) {
  return make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
}
__device__ __forceinline__ float2 split_b(float2 z, float2 zm) {
  return make_float2(0.5f * (z.y + zm.y), -0.5f * (z.x - zm.x));
}

// Real rows -> half spectra (k = 0..N/2).  Row (a, c) starts at a*in_sa +
// c*in_sc; its spectrum value k goes to k*out_skx + a*out_sa + c*out_sc.  A CTA
// takes TA consecutive rows a0..a0+TA-1 (TA even, a power of two) at c =
// blockIdx.y + c0 and transforms pairs z = row_2b + i row_2b+1.
// BIG: radices above 16 too; without them 64 registers a thread, four CTAs per SM.
template <typename T, bool BIG>
__global__ void __launch_bounds__(kThreads, BIG ? 1 : 4) k_rows_r2c(const T* in, float2* out, const __grid_constant__ FftDesc d, int nA,
                                                       int TA, int c0, long long in_sa,
                                                       long long in_sc, long long out_skx,
                                                       long long out_sa, long long out_sc, int a_fast,
                                                       int pitch) {
  pdl_begin();
  const int N = d.N, nb = TA / 2;
  float2* A = fft_sm;
  const int a0 = blockIdx.x * TA;
  const int c = c0 + blockIdx.y;
  float* Af = reinterpret_cast<float*>(A);
  const int tid = threadIdx.x, nw = blockDim.x >> 5;
  for (int al = tid >> 5; al < TA; al += nw) {  // a warp per row
    const int a = a0 + al;
    const T* row = in + a * in_sa + c * in_sc;
    for (int n = tid & 31; n < N; n += 32)
      Af[2 * ((al >> 1) * pitch + n) + (al & 1)] = a < nA ? to_f<T>(row[n]) : 0.f;
  }
  __syncthreads();
  const float2* res = fft_sm + fft_smem<1, FFT_SMEM, false, BIG>(d, nb, pitch);
  const int nk = N / 2 + 1, sh = __ffs(TA) - 1;
  const int tot2 = TA * nk;
  for (int w = tid; w < tot2; w += blockDim.x) {
    int al, k;
    if (a_fast) {
      al = w & (TA - 1);
      k = w >> sh;
    } else {
      al = w / nk;
      k = w - al * nk;
    }
    const int a = a0 + al;
    if (a >= nA) continue;
    const float2* z0 = res + (al >> 1) * pitch;
    const float2 z = z0[k], zm = z0[k == 0 ? 0 : N - k];
    out[k * out_skx + a * out_sa + c * out_sc] = (al & 1) ? split_b(z, zm) : split_a(z, zm);
  }
}

// Scan DFT along x of fp16 counts, written where G will stand (as in
// dft_inplace.cu): tile (blockIdx.x, pair blockIdx.y) takes nb (a power of two)
// scan rows from y0 = blockIdx.x nb of the pixels p, p + 1 and writes
// G[mx][p][y].  DIRECT: the first stage reads the counts itself.
template <bool DIRECT, bool BIG>
__global__ void __launch_bounds__(kDirectThreads, direct_blocks(BIG))
    k_gen_rows(const __half* __restrict__ counts, float2* G, const __grid_constant__ FftDesc d, int Ny,
               int P_pad, long long F, int nb, int pitch) {
  pdl_begin();
  const int N = d.N, sh = __ffs(nb) - 1;
  const int y0 = blockIdx.x * nb, p = 2 * blockIdx.y;
  const int ny = Ny - y0 < nb ? Ny - y0 : nb;
  const int tid = threadIdx.x;
  // the nb rows of a pixel are one contiguous run of the counts
  const __half* ca = counts + (size_t)p * F + (size_t)y0 * N;
  const float2* res;
  if (DIRECT) {
    res = fft_sm + fft_smem<1, FFT_COUNTS, false, BIG>(d, nb, pitch, FftRows{nullptr, ca, F, nullptr, 1.f, ny});
  } else {
    for (int b = tid >> 5; b < nb; b += kDirectThreads / 32) {  // a warp per row pair
      const __half* ra = ca + (size_t)b * N;
      float2* x = fft_sm + b * pitch;
      for (int n = tid & 31; n < N; n += 32)
        x[n] = b < ny ? make_float2(__half2float(__ldcs(ra + n)), __half2float(__ldcs(ra + F + n)))
                      : make_float2(0.f, 0.f);
    }
    __syncthreads();
    res = fft_sm + fft_smem<1, FFT_SMEM, false, BIG>(d, nb, pitch);
  }
  const int tot = (N / 2 + 1) * nb;
  float2* o = G + (size_t)p * Ny + y0;
  for (int w = tid; w < tot; w += kDirectThreads) {
    const int y = w & (nb - 1), k = w >> sh;
    if (y >= ny) continue;
    const float2* z0 = res + y * pitch;
    const float2 z = z0[k], zm = z0[k == 0 ? 0 : N - k];
    float2* q = o + (size_t)k * P_pad * Ny + y;
    q[0] = split_a(z, zm);
    q[Ny] = split_b(z, zm);
  }
}

// Half spectra -> real rows (inverse).  Row (a, c) value k (0..N/2) is read at
// c*in_sc + a*in_sa + k; the real output row at c*out_sc + a*out_sa.  The
// imaginary parts of k = 0 and k = N/2 are ignored.  Output scaled by scale.
__global__ void __launch_bounds__(kThreads) k_rows_c2r(const float2* in, float* out, const __grid_constant__ FftDesc d,
                                                       int nA, int TA, long long in_sa,
                                                       long long in_sc, long long out_sa,
                                                       long long out_sc, float scale, int pitch) {
  pdl_begin();
  const int N = d.N, nb = TA / 2, h = N / 2;
  float2* A = fft_sm;
  const int a0 = blockIdx.x * TA;
  const int c = blockIdx.y;
  in += c * in_sc;
  out += c * out_sc;
  const int tid = threadIdx.x, nw = blockDim.x >> 5;
  for (int b = tid >> 5; b < nb; b += nw) {  // a warp per row pair: k and N - k
    const int ra = a0 + 2 * b, rb = ra + 1;
    float2* z = A + b * pitch;
    for (int k = tid & 31; k <= h; k += 32) {
      float2 x = ra < nA ? in[ra * in_sa + k] : make_float2(0.f, 0.f);
      float2 y = rb < nA ? in[rb * in_sa + k] : make_float2(0.f, 0.f);
      if (k == 0 || k == h) { x.y = 0.f; y.y = 0.f; }
      z[k] = make_float2(x.x - y.y, x.y + y.x);
      if (k > 0 && k < h) z[N - k] = make_float2(x.x + y.y, y.x - x.y);
    }
  }
  __syncthreads();
  const float2* res = fft_sm + fft_smem<-1>(d, nb, pitch);
  for (int al = tid >> 5; al < TA; al += nw) {
    const int a = a0 + al;
    if (a >= nA) continue;
    const float2* z = res + (al >> 1) * pitch;
    for (int n = tid & 31; n < N; n += 32) {
      const float2 v = z[n];
      out[a * out_sa + n] = ((al & 1) ? v.y : v.x) * scale;
    }
  }
}

// The same for power-of-two N in [16, 1024]: a warp takes 1024 / N row pairs.
// (64 images of 512^2: 103 us with the shared-memory form in radix 8, 22 us
// here.)
constexpr int kC2rWarps = 4;
template <int R1, int R2>
__global__ void __launch_bounds__(32 * kC2rWarps, 4)
    k_c2r_warp(const float2* __restrict__ in, float* __restrict__ out, const float2* __restrict__ tw4,
               int rows, int ld, long long bs_in, float scale) {
  pdl_begin();
  using L = WarpFft<R1, R2>;
  constexpr int N = L::N, h = N / 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int u = blockIdx.x * kC2rWarps + warp;
  if (2 * u * L::C >= rows) return;  // whole warp
  in += blockIdx.y * bs_in;
  out += (size_t)blockIdx.y * rows * N;
  float2 v[32], w[32];
  {
    const int j2 = lane % R2, c1 = lane / R2;
#pragma unroll
    for (int s = 0; s < L::S1; ++s) {
      const int ra = 2 * (u * L::C + s * (32 / R2) + c1);  // rows is even
      const float2* xa = in + (size_t)ra * ld;
#pragma unroll
      for (int j = 0; j < R1; ++j) {
        const int n = R2 * j + j2, k = n <= h ? n : N - n;
        float2 x = make_float2(0.f, 0.f), y = x;
        if (ra < rows) {
          x = xa[k];
          y = xa[ld + k];
        }
        if (k == 0 || k == h) x.y = y.y = 0.f;
        if (n > h) {
          x.y = -x.y;
          y.y = -y.y;
        }
        v[s * R1 + j] = make_float2(x.x - y.y, x.y + y.x);
      }
    }
  }
  warp_fft<R1, R2, -1>(v, w, tw4, fft_sm + warp * L::kRegion, lane);
  const int k1 = lane % R1, c2 = lane / R1;
#pragma unroll
  for (int s = 0; s < L::S2; ++s) {
    const int ra = 2 * (u * L::C + s * (32 / R1) + c2);
    if (ra >= rows) continue;
    float* o = out + (size_t)ra * N + k1;
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
      o[R1 * k2] = w[s * R2 + k2].x * scale;
      o[N + R1 * k2] = w[s * R2 + k2].y * scale;
    }
  }
}

// Complex rows [rows][N] in place; with real_out, writes Re(x)*scale to
// real_out instead.  DIRECT: the first stage reads and the last one writes the
// rows itself.
template <int DIR, bool DIRECT, bool BIG>
__global__ void __launch_bounds__(kDirectThreads, direct_blocks(BIG)) k_rows_c2c(float2* data, float* real_out, const __grid_constant__ FftDesc d,
                                                       long long rows, int nb, int pitch, float scale) {
  pdl_begin();
  const int N = d.N;
  float2* A = fft_sm;
  const long long r0 = (long long)blockIdx.x * nb;
  if (DIRECT) {
    const int here = rows - r0 < nb ? (int)(rows - r0) : nb;
    float2* x = data + (size_t)r0 * N;
    fft_smem<DIR, FFT_C2C, true, BIG>(d, nb, pitch, FftRows{x, nullptr, 0, x, scale, here});
    return;
  }
  const int tid = threadIdx.x, nw = blockDim.x >> 5;
  for (int b = tid >> 5; b < nb; b += nw)
    for (int n = tid & 31; n < N; n += 32)
      A[b * pitch + n] = r0 + b < rows ? data[(size_t)(r0 + b) * N + n] : make_float2(0.f, 0.f);
  __syncthreads();
  const float2* res = fft_sm + fft_smem<DIR, FFT_SMEM, false, BIG>(d, nb, pitch);
  for (int b = tid >> 5; b < nb; b += nw) {
    if (r0 + b >= rows) continue;
    for (int n = tid & 31; n < N; n += 32) {
      const float2 v = res[b * pitch + n];
      if (real_out) real_out[(size_t)(r0 + b) * N + n] = v.x * scale;
      else data[(size_t)(r0 + b) * N + n] = cscale(v, scale);
    }
  }
}

// Fourier integration of the COM field (Sec. V), in place on Z = F(Cx + i Cy):
// X = F(Cx) = (Z(K) + conj Z(-K))/2, Y = F(Cy) = -i (Z(K) - conj Z(-K))/2,
// Phi(K) = -i (Kx X + Ky Y) / (lam1 + K^2 + lam2 K^4), Phi(0) = 0.
// One thread per bin pair {K, -K}.
__device__ __forceinline__ float2 idpc_one(float2 z, float2 zm, float kx, float ky, float lam1,
                                           float lam2) {
  const float2 X = make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
  const float2 Y = make_float2(0.5f * (z.y + zm.y), -0.5f * (z.x - zm.x));
  const float k2 = kx * kx + ky * ky;
  const float den = lam1 + k2 + lam2 * k2 * k2;
  if (den == 0.f) return make_float2(0.f, 0.f);
  const float2 s = make_float2(kx * X.x + ky * Y.x, kx * X.y + ky * Y.y);
  return make_float2(s.y / den, -s.x / den);  // -i s / den
}

__global__ void k_idpc_filter(float2* Z, int Ny, int Nx, float inv_lx, float inv_ly, float lam1,
                              float lam2) {
  pdl_begin();
  const int F = Ny * Nx;
  for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < F; f += gridDim.x * blockDim.x) {
    const int my = f / Nx, mx = f - my * Nx;
    const int mmy = (Ny - my) % Ny, mmx = (Nx - mx) % Nx;
    const int fm = mmy * Nx + mmx;
    if (fm < f) continue;  // the partner thread handles this pair
    const float2 z = Z[f], zm = Z[fm];
    const float kx = freq_index(mx, Nx) * inv_lx, ky = freq_index(my, Ny) * inv_ly;
    const float kxm = freq_index(mmx, Nx) * inv_lx, kym = freq_index(mmy, Ny) * inv_ly;
    float2 p = idpc_one(z, zm, kx, ky, lam1, lam2);
    float2 pm = idpc_one(zm, z, kxm, kym, lam1, lam2);
    if (f == 0) p = make_float2(0.f, 0.f);
    Z[f] = p;
    if (fm != f) Z[fm] = pm;
  }
}

// out[b][c][r] = in[b][r][c] for a batch of [rows][cols] complex matrices
__global__ void k_transpose(const float2* __restrict__ in, float2* __restrict__ out, int rows,
                            int cols) {
  pdl_begin();
  __shared__ float2 t[32][33];
  const size_t b = blockIdx.z;
  in += b * (size_t)rows * cols;
  out += b * (size_t)rows * cols;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    if (r < rows && c < cols) t[i][threadIdx.x] = in[(size_t)r * cols + c];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    if (r < rows && c < cols) out[(size_t)c * rows + r] = t[threadIdx.x][i];
  }
}

// transforms per CTA: at most `most`, both buffers within 64 KB, at least one
int fft_nb(const FftDesc& d, int most) {
  int nb = most;
  while (nb > 1 && (size_t)2 * nb * fft_pitch(d, nb) * sizeof(float2) > 64 * 1024) nb >>= 1;
  return nb;
}
size_t fft_bytes(const FftDesc& d, int nb) { return (size_t)2 * nb * fft_pitch(d, nb) * sizeof(float2); }

template <typename K>
cudaError_t set_smem(K kern, size_t bytes) {
  return ensure_smem((const void*)kern, bytes);
}

cudaError_t cols(const FftDesc& d, const float2* in, float2* out, int dir, int ncols, int ld_in,
                 int ld_out, long long bs_in, long long bs_out, int nbatch, float scale,
                 cudaStream_t s) {
  // fewer columns a CTA (down to a 32-byte sector) while there are SMs to spare:
  // a launch of a few CTAs lasts as long as one of them (16 uneven scans in one
  // call 719 -> 668 us, the 336 x 200 path 563 -> 556)
  int nb = fft_nb(d, 16);
  while (nb > 4 && (ncols + nb - 1) / nb * nbatch < kSms) nb >>= 1;
  // two columns rather than one while two CTAs fit an SM and there are CTAs enough
  // (whole accumulation, 560 pixels: 2048 x 256 3.62 -> 2.86 ms, 3000 x 100 3.69 ->
  // 2.60; at 4096, where one CTA would fit, 1.75 -> 2.20; an image of 2048 x 256,
  // 129 columns, 187 -> 192 us)
  if (nb == 1 && ncols / 2 * nbatch >= kSms && fft_bytes(d, 2) <= 110 * 1024) nb = 2;
  const int pitch = fft_pitch(d, nb);
  const size_t sm = fft_bytes(d, nb);
  auto kern = dir > 0 ? k_fft_cols<1> : k_fft_cols<-1>;
  cudaError_t e = set_smem(kern, sm);
  if (e != cudaSuccess) return e;
  dim3 grid((ncols + nb - 1) / nb, nbatch);
  launch(kern, grid, kThreads, sm, s, in, out, d, ncols, ld_in, ld_out, bs_in, bs_out, nb, pitch,
         scale);
  count_launches(1);
  return cudaGetLastError();
}

// ---- register four-step dispatch (power-of-two N in [16, 1024]) ----------
bool reg_size(int N) { return N >= 16 && N <= 1024 && (N & (N - 1)) == 0; }

template <int R1, int R2, int CB, int DIR, bool TOUT>
cudaError_t cols_reg_t(const FftDesc& d, const float2* in, float2* out, int ncols, int ld_in,
                       int ld_out, long long bs_in, long long bs_out, int nbatch, float scale,
                       cudaStream_t s) {
  constexpr int NT = (R1 > R2 ? R1 : R2) * CB;
  const size_t sm = sizeof(float2) * ((size_t)R1 * CB * (R2 + 1) + 2 * CB);
  auto kern = k_colfft_reg<R1, R2, CB, DIR, TOUT>;
  cudaError_t e = set_smem(kern, sm);
  if (e != cudaSuccess) return e;
  dim3 grid((ncols + CB - 1) / CB, nbatch);
  if (!d.tw4 || reg_r1(d.N) != R1) return cudaErrorInvalidValue;
  launch(kern, grid, NT, sm, s, in, out, d.tw4, ncols, ld_in, ld_out, bs_in, bs_out, scale);
  count_launches(1);
  return cudaGetLastError();
}

template <int DIR, bool TOUT = false>
cudaError_t cols_reg(const FftDesc& d, const float2* in, float2* out, int ncols, int ld_in,
                     int ld_out, long long bs_in, long long bs_out, int nbatch, float scale,
                     cudaStream_t s) {
#define EER4D_COLS(R1, R2, CB) \
  return cols_reg_t<R1, R2, CB, DIR, TOUT>(d, in, out, ncols, ld_in, ld_out, bs_in, bs_out, nbatch, scale, s)
  switch (d.N) {
    case 1024: EER4D_COLS(32, 32, 8);
    case 512: EER4D_COLS(32, 16, 8);
    case 256: EER4D_COLS(16, 16, 16);
    case 128: EER4D_COLS(16, 8, 16);
    case 64: EER4D_COLS(8, 8, 32);
    case 32: EER4D_COLS(8, 4, 32);
    default: EER4D_COLS(4, 4, 64);
  }
#undef EER4D_COLS
}

template <int R1, int R2, int CP>
cudaError_t r2c_reg_t(const FftDesc& d, const __half* in, float2* out, int nA, int c0, int nc,
                      long long in_sa, long long in_sc, long long out_skx, long long out_sa,
                      long long out_sc, cudaStream_t s) {
  constexpr int N = R1 * R2;
  const size_t a = (size_t)R1 * CP * (R2 + 1), b = (size_t)N * CP;
  const size_t sm = sizeof(float2) * (a > b ? a : b);
  auto kern = k_rowfft_r2c_reg<R1, R2, CP>;
  cudaError_t e = set_smem(kern, sm);
  if (e != cudaSuccess) return e;
  dim3 grid((nA + 2 * CP - 1) / (2 * CP), nc);
  if (!d.tw4 || reg_r1(d.N) != R1) return cudaErrorInvalidValue;
  launch(kern, grid, R1 * CP, sm, s, in, out, d.tw4, nA, c0, in_sa, in_sc, out_skx, out_sa, out_sc);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t r2c_reg(const FftDesc& d, const __half* in, float2* out, int nA, int c0, int nc,
                    long long in_sa, long long in_sc, long long out_skx, long long out_sa,
                    long long out_sc, cudaStream_t s) {
#define EER4D_R2C(R1, R2, CP) \
  return r2c_reg_t<R1, R2, CP>(d, in, out, nA, c0, nc, in_sa, in_sc, out_skx, out_sa, out_sc, s)
  switch (d.N) {
    case 1024: EER4D_R2C(32, 32, 8);
    case 512: EER4D_R2C(32, 16, 8);
    case 256: EER4D_R2C(16, 16, 16);
    case 128: EER4D_R2C(16, 8, 16);
    case 64: EER4D_R2C(8, 8, 32);
    case 32: EER4D_R2C(8, 4, 32);
    default: EER4D_R2C(4, 4, 64);
  }
#undef EER4D_R2C
}

}  // namespace

cudaError_t launch_transpose(const float2* in, float2* out, int rows, int cols, int batch,
                             cudaStream_t s) {
  dim3 grid((cols + 31) / 32, (rows + 31) / 32, batch);
  launch(k_transpose, grid, dim3(32, 8), 0, s, in, out, rows, cols);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_stage1(const eer4d_plan* p, const __half* counts, float2* G, int y0, int y1,
                          cudaStream_t s) {
  if (y1 <= y0) return cudaSuccess;
  const FftDesc& d = p->fx;
  const long long NRl = p->cstride;
  if (reg_size(d.N) && p->precision != EER4D_FP32_STOCKHAM) {
    stage_begin(p, EER4D_STAGE_DFT_X, s);
    cudaError_t e = r2c_reg(d, counts, G, p->P_pad, y0, y1 - y0, NRl, (long long)p->g.scan_nx,
                            (long long)p->g.scan_ny * p->P_pad, 1, (long long)p->P_pad, s);
    stage_end(p, EER4D_STAGE_DFT_X, s);
    return e;
  }
  const int nb = fft_nb(d, 8);
  const int TA = 2 * nb;
  const size_t sm = fft_bytes(d, nb);
  // short rows are little work for a CTA between its barriers: four CTAs per SM
  // where shared memory holds them (4096 x 64, 560 pixels, plain form 3.29 ->
  // 2.51 ms); otherwise the registers (64 x 4096 1.07 ms, with 64 of them 1.18)
  auto kern = fft_big(d) || sm > 56 * 1024 ? k_rows_r2c<__half, true> : k_rows_r2c<__half, false>;
  cudaError_t e = set_smem(kern, sm);
  if (e != cudaSuccess) return e;
  const long long NR = p->cstride;
  dim3 grid((p->P_pad + TA - 1) / TA, y1 - y0);
  stage_begin(p, EER4D_STAGE_DFT_X, s);
  launch(kern, grid, kThreads, sm, s, counts, G, d, p->P_pad, TA, y0, NR,
         (long long)p->g.scan_nx, (long long)p->g.scan_ny * p->P_pad, 1, (long long)p->P_pad, 1,
         fft_pitch(d, nb));
  count_launches(1);
  stage_end(p, EER4D_STAGE_DFT_X, s);
  return cudaGetLastError();
}

cudaError_t launch_stage2(const eer4d_plan* p, const float2* X1, float2* G, cudaStream_t s) {
  const int Ny = p->g.scan_ny;
  const long long bs = (long long)Ny * p->P_pad;
  stage_begin(p, EER4D_STAGE_DFT_Y, s);
  cudaError_t e;
  if (reg_size(p->fy.N) && p->precision != EER4D_FP32_STOCKHAM) {
    e = cols_reg<1, true>(p->fy, X1, G, p->P_pad, p->P_pad, Ny, bs, bs, p->nkx, 1.f, s);
  } else {
    // generic lengths: in-place column FFT, then a tiled transpose into G
    e = cols(p->fy, X1, const_cast<float2*>(X1), 1, p->P_pad, p->P_pad, p->P_pad, bs, bs, p->nkx,
             1.f, s);
    if (e == cudaSuccess) e = launch_transpose(X1, G, Ny, p->P_pad, p->nkx, s);
  }
  stage_end(p, EER4D_STAGE_DFT_Y, s);
  return e;
}

template <int R1, int R2>
static cudaError_t c2r_warp_t(const FftDesc& d, const float2* H, float* phase, int rows, int ld,
                              long long bs, int n_cand, float scale, cudaStream_t s) {
  using L = WarpFft<R1, R2>;
  auto kern = k_c2r_warp<R1, R2>;
  const size_t sm = sizeof(float2) * kC2rWarps * L::kRegion;
  cudaError_t e = set_smem(kern, sm);
  if (e != cudaSuccess) return e;
  if (!d.tw4 || reg_r1(d.N) != R1) return cudaErrorInvalidValue;
  const int units = (rows / 2 + L::C - 1) / L::C;
  launch(kern, dim3((units + kC2rWarps - 1) / kC2rWarps, n_cand), 32 * kC2rWarps, sm, s, H, phase,
         d.tw4, rows, ld, bs, scale);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_c2r_image(const eer4d_plan* p, float2* H, float* phase, int n_cand,
                             cudaStream_t s) {
  const int Ny = p->g.scan_ny, Nx = p->g.scan_nx, nkx = p->nkx;
  const long long bs = (long long)Ny * nkx;
  cudaError_t e = reg_size(p->fy.N) ? cols_reg<-1>(p->fy, H, H, nkx, nkx, nkx, bs, bs, n_cand, 1.f, s)
                                    : cols(p->fy, H, H, -1, nkx, nkx, nkx, bs, bs, n_cand, 1.f, s);
  if (e != cudaSuccess) return e;
  const FftDesc& d = p->fx;
  const float scale = 1.f / ((float)Ny * (float)Nx);
  switch (reg_size(d.N) ? d.N : 0) {
#define EER4D_C2R(R1, R2) return c2r_warp_t<R1, R2>(d, H, phase, Ny, nkx, bs, n_cand, scale, s)
    case 1024: EER4D_C2R(32, 32);
    case 512: EER4D_C2R(32, 16);
    case 256: EER4D_C2R(16, 16);
    case 128: EER4D_C2R(16, 8);
    case 64: EER4D_C2R(8, 8);
    case 32: EER4D_C2R(8, 4);
    case 16: EER4D_C2R(4, 4);
#undef EER4D_C2R
    default: break;
  }
  const int nb = fft_nb(d, 4), TA = 2 * nb;
  const size_t sm = fft_bytes(d, nb);
  e = set_smem(k_rows_c2r, sm);
  if (e != cudaSuccess) return e;
  dim3 grid((Ny + TA - 1) / TA, n_cand);
  launch(k_rows_c2r, grid, kThreads, sm, s, H, phase, d, Ny, TA, nkx, bs, Nx, (long long)Ny * Nx,
         scale, fft_pitch(d, nb));
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_r2c_image(const eer4d_plan* p, const float* g, float2* W, cudaStream_t s) {
  const int Ny = p->g.scan_ny, Nx = p->g.scan_nx, nkx = p->nkx;
  const FftDesc& d = p->fx;
  const int nb = fft_nb(d, 4), TA = 2 * nb;
  const size_t sm = fft_bytes(d, nb);
  auto kern = k_rows_r2c<float, true>;
  cudaError_t e = set_smem(kern, sm);
  if (e != cudaSuccess) return e;
  dim3 grid((Ny + TA - 1) / TA, 1);
  launch(kern, grid, kThreads, sm, s, g, W, d, Ny, TA, 0, Nx, 0, 1, nkx, 0, 0,
         fft_pitch(d, nb));
  count_launches(1);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const long long bs = (long long)Ny * nkx;
  return reg_size(p->fy.N) ? cols_reg<1>(p->fy, W, W, nkx, nkx, nkx, bs, bs, 1, 1.f, s)
                           : cols(p->fy, W, W, 1, nkx, nkx, nkx, bs, bs, 1, 1.f, s);
}

// Complex rows [rows][d.N] in place (or Re(.)*scale into real_out).
static cudaError_t rows_gen(const FftDesc& d, float2* data, float* real_out, long long rows, int dir,
                            float scale, cudaStream_t s) {
  const int nb = fft_nb(d, 4);
  const size_t sm = fft_bytes(d, nb);
  const bool direct = !real_out && fft_direct(d), big = fft_big(d);
#define EER4D_C2C(D) (direct ? (big ? k_rows_c2c<D, true, true> : k_rows_c2c<D, true, false>) \
                             : (big ? k_rows_c2c<D, false, true> : k_rows_c2c<D, false, false>))
  auto kern = dir > 0 ? EER4D_C2C(1) : EER4D_C2C(-1);
#undef EER4D_C2C
  cudaError_t e = set_smem(kern, sm);
  if (e != cudaSuccess) return e;
  launch(kern, (unsigned)((rows + nb - 1) / nb), kDirectThreads, sm, s, data, real_out, d, rows, nb,
         fft_pitch(d, nb), scale);
  count_launches(1);
  return cudaGetLastError();
}

bool dft_gen_ok(const eer4d_plan* p) {
  return p->precision == EER4D_FP32_FFT && !(reg_size(p->g.scan_nx) && reg_size(p->g.scan_ny)) &&
         p->g.scan_nx <= 1024 && p->g.scan_ny <= 1024;
}

cudaError_t launch_dft_gen(const eer4d_plan* p, const __half* counts, float2* G, cudaStream_t s) {
  const FftDesc& d = p->fx;
  const int Ny = (int)p->g.scan_ny;
  const int nb = fft_nb(d, 8);
  const size_t sm = fft_bytes(d, nb);
  auto kern = fft_big(d) ? (fft_direct(d) ? k_gen_rows<true, true> : k_gen_rows<false, true>)
                         : (fft_direct(d) ? k_gen_rows<true, false> : k_gen_rows<false, false>);
  cudaError_t e = set_smem(kern, sm);
  if (e != cudaSuccess) return e;
  stage_begin(p, EER4D_STAGE_DFT_XY, s);
  launch(kern, dim3((Ny + nb - 1) / nb, p->P_pad / 2), kDirectThreads, sm, s, counts, G, d, Ny,
         p->P_pad, p->cstride, nb, fft_pitch(d, nb));
  count_launches(1);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  e = rows_gen(p->fy, G, nullptr, (long long)p->nkx * p->P_pad, 1, 1.f, s);
  stage_end(p, EER4D_STAGE_DFT_XY, s);
  return e;
}

template <int R1, int R2, int CB, int DIR, bool REAL_OUT>
cudaError_t rows_reg_t(const FftDesc& d, float2* data, float* real_out, int rows, float scale,
                       cudaStream_t s) {
  constexpr int NT = (R1 > R2 ? R1 : R2) * CB;
  const size_t sm = sizeof(float2) * (size_t)CB * R1 * (R2 + 1);
  auto kern = k_rowfft_c2c_reg<R1, R2, CB, DIR, REAL_OUT>;
  cudaError_t e = set_smem(kern, sm);
  if (e != cudaSuccess) return e;
  if (!d.tw4 || reg_r1(d.N) != R1) return cudaErrorInvalidValue;
  launch(kern, (rows + CB - 1) / CB, NT, sm, s, data, real_out, d.tw4, rows, d.N, scale);
  count_launches(1);
  return cudaGetLastError();
}

// Register four-step transform of every row of [rows][d.N] in place (or its
// real part times scale into real_out); d.N a register length (reg_size).
template <int DIR, bool REAL_OUT = false>
cudaError_t rows_reg(const FftDesc& d, float2* data, float* real_out, int rows, float scale,
                     cudaStream_t s) {
#define EER4D_ROWS(R1, R2, CB) return rows_reg_t<R1, R2, CB, DIR, REAL_OUT>(d, data, real_out, rows, scale, s)
  switch (d.N) {
    case 1024: EER4D_ROWS(32, 32, 4);
    case 512: EER4D_ROWS(32, 16, 4);
    case 256: EER4D_ROWS(16, 16, 8);
    case 128: EER4D_ROWS(16, 8, 8);
    case 64: EER4D_ROWS(8, 8, 16);
    case 32: EER4D_ROWS(8, 4, 16);
    default: EER4D_ROWS(4, 4, 32);
  }
#undef EER4D_ROWS
}

cudaError_t launch_fft2_c2c(const FftDesc& fy, const FftDesc& fx, float2* data, int dir,
                            float scale, cudaStream_t s) {
  const int My = fy.N, Mx = fx.N;
  if (reg_size(Mx) && reg_size(My)) {
    cudaError_t e = dir > 0 ? rows_reg<1>(fx, data, nullptr, My, 1.f, s)
                            : rows_reg<-1>(fx, data, nullptr, My, 1.f, s);
    if (e != cudaSuccess) return e;
    return dir > 0 ? cols_reg<1>(fy, data, data, Mx, Mx, Mx, 0, 0, 1, scale, s)
                   : cols_reg<-1>(fy, data, data, Mx, Mx, Mx, 0, 0, 1, scale, s);
  }
  cudaError_t e = rows_gen(fx, data, nullptr, My, dir, 1.f, s);
  if (e != cudaSuccess) return e;
  return cols(fy, data, data, dir, Mx, Mx, Mx, 0, 0, 1, scale, s);
}

cudaError_t launch_idpc(const eer4d_plan* p, float2* z, float* phase, double lam1, double lam2,
                        cudaStream_t s) {
  const int Ny = p->g.scan_ny, Nx = p->g.scan_nx;
  const FftDesc& dx = p->fx;
  cudaError_t e;
  stage_begin(p, EER4D_STAGE_DPC, s);
  const float inv_lx = (float)(1.0 / ((double)Nx * p->g.step_A));
  const float inv_ly = (float)(1.0 / ((double)Ny * p->g.step_A));
  if (reg_size(Nx) && reg_size(Ny)) {
    // register four-step tiles: rows, columns (in place), filter, columns, rows
    if ((e = rows_reg<1>(dx, z, nullptr, Ny, 1.f, s)) != cudaSuccess) return e;
    if ((e = cols_reg<1>(p->fy, z, z, Nx, Nx, Nx, 0, 0, 1, 1.f, s)) != cudaSuccess) return e;
    launch(k_idpc_filter, (Ny * Nx + 255) / 256, 256, 0, s, z, Ny, Nx, inv_lx, inv_ly, (float)lam1,
           (float)lam2);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cols_reg<-1>(p->fy, z, z, Nx, Nx, Nx, 0, 0, 1, 1.f, s)) != cudaSuccess) return e;
    e = rows_reg<-1, true>(dx, z, phase, Ny, 1.f / ((float)Ny * (float)Nx), s);
    stage_end(p, EER4D_STAGE_DPC, s);
    return e;
  }
  if ((e = rows_gen(dx, z, nullptr, Ny, 1, 1.f, s)) != cudaSuccess) return e;
  if ((e = cols(p->fy, z, z, 1, Nx, Nx, Nx, 0, 0, 1, 1.f, s)) != cudaSuccess) return e;
  launch(k_idpc_filter, (Ny * Nx + 255) / 256, 256, 0, s, z, Ny, Nx, inv_lx, inv_ly, (float)lam1,
         (float)lam2);
  count_launches(1);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = cols(p->fy, z, z, -1, Nx, Nx, Nx, 0, 0, 1, 1.f, s)) != cudaSuccess) return e;
  e = rows_gen(dx, z, phase, Ny, -1, 1.f / ((float)Ny * (float)Nx), s);
  stage_end(p, EER4D_STAGE_DPC, s);
  return e;
}
