// Iterative regularised DPC (Sec. V): gradient descent on ||grad phi / 2 pi - C||
// with the Fourier preconditioner 1/(lam1 + K^2 + lam2 K^4) and step mu, the
// residual taken only over the scan.  As printed the update has no residual
// term; it is read as
//   R = M (C - grad phi^l / 2 pi),
//   phi^{l+1} = phi^l + mu IFFT[ -i (Kx R^x(K) + Ky R^y(K)) / (lam1 + K^2 + lam2 K^4) ],
// phi^0 = 0, on a periodic grid of pad x the scan (pad = 1 or 2; with pad = 2
// the scan sits in the top-left quarter, M = 1 there and 0 in the padding, so
// the solution does not wrap around).  The spectral derivative is iK and the
// update's DC and Nyquist bins (m = M/2 on either axis) are zero, so phi stays
// real.  With pad = 1 and lam1 = lam2 = 0 the iteration reaches the one-shot
// Fourier integration as (1 - (1 - mu)^L).
//
// phi is kept as its spectrum Phi; each step is one inverse transform of
// (iKx + i iKy) Phi (the two real gradients packed as one complex field), the
// residual, one forward transform (the two real residuals packed) and the
// update of Phi.
//
// On grids whose sides are powers of two up to 1024 a step is two kernels:
//   k_dpc_cols: forward DFT along y of a column and of its mirror -K_x, the
//     update of Phi, its derivative and the inverse DFT along y;
//   k_dpc_rows: inverse DFT along x of a scan row, the residual, forward DFT
//     along x.
// The fields between them are kept as [K_x][y] and for the scan's rows only:
// the residual is zero in the padding, whose rows are neither stored nor
// transformed.  (Seven kernels over the whole padded grid took 52 us a step on
// 1024 x 1024, and 39 us with overlapping launches; these take 27 us.)  They
// are bound by latency: 128 and 256 blocks, 15 MB in L2 (spectrum 8.4, fields 4.2,
// COM maps 2.1).  Other grids take the kernels over the whole grid below.
#include "common.cuh"
#include "fft_warp.cuh"

namespace {

__device__ __forceinline__ bool nyq_bin(int m, int M) { return 2 * m == M; }

__global__ void k_dpc_setup(const float* __restrict__ com, int Ny, int Nx, int My, int Mx,
                            float cscale, float2* Cpk, float2* Phi) {
  pdl_begin();
  const size_t n = (size_t)My * Mx;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const int y = (int)(i / Mx), x = (int)(i - (size_t)y * Mx);
    float2 c = make_float2(0.f, 0.f);
    if (y < Ny && x < Nx) {
      const size_t f = (size_t)y * Nx + x;
      c = make_float2(com[f] * cscale, com[(size_t)Ny * Nx + f] * cscale);
    }
    Cpk[i] = c;
    Phi[i] = make_float2(0.f, 0.f);
  }
}

// Z = (i Kx + i (i Ky)) Phi = Phi (-Ky + i Kx), zero at Nyquist bins
__global__ void k_dpc_deriv(const float2* __restrict__ Phi, int My, int Mx, float inv_lx,
                            float inv_ly, float2* Z) {
  pdl_begin();
  const size_t n = (size_t)My * Mx;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const int my = (int)(i / Mx), mx = (int)(i - (size_t)my * Mx);
    float2 z = make_float2(0.f, 0.f);
    if (!nyq_bin(mx, Mx) && !nyq_bin(my, My)) {
      const float kx = freq_index(mx, Mx) * inv_lx, ky = freq_index(my, My) * inv_ly;
      const float2 p = Phi[i];
      z = make_float2(-ky * p.x - kx * p.y, -ky * p.y + kx * p.x);
    }
    Z[i] = z;
  }
}

// Z = M (C - g) with g = Z (packed gradients), M = 1 on the scan
__global__ void k_dpc_resid(const float2* __restrict__ Cpk, int Ny, int Nx, int My, int Mx,
                            float2* Z) {
  pdl_begin();
  const size_t n = (size_t)My * Mx;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const int y = (int)(i / Mx), x = (int)(i - (size_t)y * Mx);
    const float2 c = Cpk[i], g = Z[i];
    Z[i] = (y < Ny && x < Nx) ? make_float2(c.x - g.x, c.y - g.y) : make_float2(0.f, 0.f);
  }
}

// Phi(K) += mu * (-i (Kx Rx + Ky Ry) / den), Rx = (Z(K) + conj Z(-K))/2,
// Ry = -i (Z(K) - conj Z(-K))/2; DC and Nyquist bins unchanged.  One thread
// per pair {K, -K}.
__device__ __forceinline__ float2 update_one(float2 z, float2 zm, float kx, float ky, float lam1,
                                             float lam2) {
  const float2 X = make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
  const float2 Y = make_float2(0.5f * (z.y + zm.y), -0.5f * (z.x - zm.x));
  const float k2 = kx * kx + ky * ky;
  const float den = lam1 + k2 + lam2 * k2 * k2;
  if (den == 0.f) return make_float2(0.f, 0.f);
  const float2 s = make_float2(kx * X.x + ky * Y.x, kx * X.y + ky * Y.y);
  return make_float2(s.y / den, -s.x / den);
}

__global__ void k_dpc_update(const float2* __restrict__ Z, int My, int Mx, float inv_lx,
                             float inv_ly, float lam1, float lam2, float mu, float2* Phi) {
  pdl_begin();
  const size_t n = (size_t)My * Mx;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const int my = (int)(i / Mx), mx = (int)(i - (size_t)my * Mx);
    const int mmy = (My - my) % My, mmx = (Mx - mx) % Mx;
    const size_t im = (size_t)mmy * Mx + mmx;
    if (im < i) continue;  // the partner handles the pair
    if (i == 0 || nyq_bin(mx, Mx) || nyq_bin(my, My)) continue;
    const float2 z = Z[i], zm = Z[im];
    const float kx = freq_index(mx, Mx) * inv_lx, ky = freq_index(my, My) * inv_ly;
    const float kxm = freq_index(mmx, Mx) * inv_lx, kym = freq_index(mmy, My) * inv_ly;
    const float2 u = update_one(z, zm, kx, ky, lam1, lam2);
    const float2 um = update_one(zm, z, kxm, kym, lam1, lam2);
    float2 p = Phi[i];
    Phi[i] = make_float2(p.x + mu * u.x, p.y + mu * u.y);
    if (im != i) {
      p = Phi[im];
      Phi[im] = make_float2(p.x + mu * um.x, p.y + mu * um.y);
    }
  }
}

__global__ void k_dpc_out(const float2* __restrict__ Z, int Ny, int Nx, int Mx, float* phase) {
  pdl_begin();
  const size_t n = (size_t)Ny * Nx;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const int y = (int)(i / Nx), x = (int)(i - (size_t)y * Nx);
    phase[i] = Z[(size_t)y * Mx + x].x;
  }
}

// ---- two kernels a step -------------------------------------------------------
struct DpcGrid {
  int Ny, Nx, My, Mx;
  float inv_lx, inv_ly, lam1, lam2, mu;
};
constexpr int kDpcWarps = 4;

// Warps 2 i and 2 i + 1 take C columns q C + c < Mx / 2 and their mirrors
// (Mx - column) mod Mx.  The K_x Nyquist column stays zero everywhere and is
// neither stored nor read.  LAST: the inverse transform is that of Phi.
template <int R1, int R2, bool LAST>
__global__ void __launch_bounds__(32 * kDpcWarps, 4)
    k_dpc_cols(float2* Z, float2* Phi, const float2* __restrict__ tw4, const DpcGrid g, int first) {
  pdl_begin();
  using L = WarpFft<R1, R2>;
  constexpr int N = L::N;  // My
  extern __shared__ float2 sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* rg = sm + warp * L::kRegion;
  const float2* other = sm + (warp ^ 1) * L::kRegion;
  const int q = blockIdx.x * (kDpcWarps / 2) + (warp >> 1), mirror = warp & 1;
  auto column = [&](int c, bool& on) {
    const int k = q * L::C + c;
    on = k < g.Mx / 2 && !(mirror && k == 0);  // column 0 is its own mirror: stored once
    const int kk = k < g.Mx / 2 ? k : 0;
    return mirror ? (g.Mx - kk) % g.Mx : kk;
  };
  float2 v[32], w[32];
  {
    const int j2 = lane % R2, c1 = lane / R2;
#pragma unroll
    for (int s = 0; s < L::S1; ++s) {
      bool on;
      const int c = s * (32 / R2) + c1;
      const float2* z = Z + (size_t)column(c, on) * g.Ny;
      const int n = q * L::C + c < g.Mx / 2 ? g.Ny : 0;
#pragma unroll
      for (int j = 0; j < R1; ++j) {
        const int y = R2 * j + j2;
        v[s * R1 + j] = y < n ? __ldcg(z + y) : make_float2(0.f, 0.f);
      }
    }
  }
  warp_fft<R1, R2, 1>(v, w, tw4, rg, lane);
  __syncwarp();
  const int k1 = lane % R1, c2 = lane / R1;
#pragma unroll
  for (int s = 0; s < L::S2; ++s)
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2)
      rg[(s * (32 / R1) + c2) * L::kColZ + k1 + R1 * k2] = w[s * R2 + k2];
  __syncthreads();
#pragma unroll
  for (int s = 0; s < L::S2; ++s) {
    const int c = s * (32 / R1) + c2;
    bool on;
    const int kxi = column(c, on);
    const float kx = freq_index(kxi, g.Mx) * g.inv_lx;
    float2* phi = Phi + (size_t)kxi * N;
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
      const int kyi = k1 + R1 * k2;
      const float ky = freq_index(kyi, N) * g.inv_ly;
      const bool nyq = nyq_bin(kyi, N);
      const float2 z = w[s * R2 + k2], zm = other[c * L::kColZ + ((N - kyi) & (N - 1))];
      float2 p = first ? make_float2(0.f, 0.f) : __ldcg(phi + kyi);
      if (!nyq && (kxi | kyi)) {
        const float2 u = update_one(z, zm, kx, ky, g.lam1, g.lam2);
        p = make_float2(p.x + g.mu * u.x, p.y + g.mu * u.y);
      }
      if (!LAST && on) __stcg(phi + kyi, p);
      w[s * R2 + k2] = LAST ? p
                       : nyq ? make_float2(0.f, 0.f)
                             : make_float2(-ky * p.x - kx * p.y, -ky * p.y + kx * p.x);
    }
  }
  if constexpr (R1 == R2) {  // a lane's outputs are its inputs of the next transform
    __syncthreads();         // the mirror's reads of this warp's spectrum
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = w[j];
  } else {
    __syncthreads();
#pragma unroll
    for (int s = 0; s < L::S2; ++s)
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2)
        rg[(s * (32 / R1) + c2) * L::kColZ + k1 + R1 * k2] = w[s * R2 + k2];
    __syncwarp();
#pragma unroll
    for (int s = 0; s < L::S1; ++s)
#pragma unroll
      for (int j = 0; j < R1; ++j)
        v[s * R1 + j] = rg[(s * (32 / R2) + lane / R2) * L::kColZ + R2 * j + lane % R2];
    __syncwarp();
  }
  warp_fft<R1, R2, -1>(v, w, tw4, rg, lane);
#pragma unroll
  for (int s = 0; s < L::S2; ++s) {
    bool on;
    float2* z = Z + (size_t)column(s * (32 / R1) + c2, on) * g.Ny;
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
      const int y = k1 + R1 * k2;
      if (on && y < g.Ny) __stcg(z + y, w[s * R2 + k2]);
    }
  }
}

// Scan rows [RY blockIdx.x, + RY), RY = 4 C.  STEP 0: the transform of the COM
// field itself (phi = 0); 1: inverse, residual, forward; 2: inverse, Re(phi).
template <int R1, int R2, int STEP>
__global__ void __launch_bounds__(32 * kDpcWarps, 4)
    k_dpc_rows(float2* Z, const float* __restrict__ com, const float2* __restrict__ tw4,
               const DpcGrid g, float cscale_, float inv_n, float* phase) {
  pdl_begin();
  using L = WarpFft<R1, R2>;
  constexpr int N = L::N, RY = kDpcWarps * L::C;  // N = Mx
  extern __shared__ float2 sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* rg = sm + warp * L::kRegion;
  const int y0 = blockIdx.x * RY;
  float2 v[32], w[32];
  const int j2 = lane % R2, c1 = lane / R2, k1 = lane % R1, c2 = lane / R1;
  if constexpr (STEP > 0) {
    for (int i = threadIdx.x; i < N * RY; i += 32 * kDpcWarps) {
      const int y = i % RY, k = i / RY;
      sm[(y / L::C) * L::kRegion + (y % L::C) * L::kColZ + k] =
          k != N / 2 && y0 + y < g.Ny ? __ldcg(Z + (size_t)k * g.Ny + y0 + y) : make_float2(0.f, 0.f);
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < L::S1; ++s)
#pragma unroll
      for (int j = 0; j < R1; ++j) v[s * R1 + j] = rg[(s * (32 / R2) + c1) * L::kColZ + R2 * j + j2];
    __syncwarp();
    warp_fft<R1, R2, -1>(v, w, tw4, rg, lane);
  }
#pragma unroll
  for (int s = 0; s < L::S2; ++s) {
    const int y = y0 + warp * L::C + s * (32 / R1) + c2;
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
      const int x = k1 + R1 * k2;
      const bool in = y < g.Ny && x < g.Nx;
      if (STEP == 2) {
        if (in) phase[(size_t)y * g.Nx + x] = w[s * R2 + k2].x * inv_n;
      } else {
        float2 r = make_float2(0.f, 0.f);
        if (in) {
          const size_t f = (size_t)y * g.Nx + x;
          r = make_float2(__ldg(com + f) * cscale_, __ldg(com + (size_t)g.Ny * g.Nx + f) * cscale_);
          if (STEP == 1) {
            const float2 d = w[s * R2 + k2];
            r = make_float2(r.x - d.x * inv_n, r.y - d.y * inv_n);
          }
        }
        w[s * R2 + k2] = r;
      }
    }
  }
  if constexpr (STEP == 2) return;
  __syncwarp();
  if constexpr (R1 == R2) {
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = w[j];
  } else {
#pragma unroll
    for (int s = 0; s < L::S2; ++s)
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2)
        rg[(s * (32 / R1) + c2) * L::kColZ + k1 + R1 * k2] = w[s * R2 + k2];
    __syncwarp();
#pragma unroll
    for (int s = 0; s < L::S1; ++s)
#pragma unroll
      for (int j = 0; j < R1; ++j) v[s * R1 + j] = rg[(s * (32 / R2) + c1) * L::kColZ + R2 * j + j2];
    __syncwarp();
  }
  warp_fft<R1, R2, 1>(v, w, tw4, rg, lane);
  __syncwarp();
#pragma unroll
  for (int s = 0; s < L::S2; ++s)
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2)
      rg[(s * (32 / R1) + c2) * L::kColZ + k1 + R1 * k2] = w[s * R2 + k2];
  __syncthreads();
  for (int i = threadIdx.x; i < N * RY; i += 32 * kDpcWarps) {
    const int y = i % RY, k = i / RY;
    if (k != N / 2 && y0 + y < g.Ny)
      __stcg(Z + (size_t)k * g.Ny + y0 + y, sm[(y / L::C) * L::kRegion + (y % L::C) * L::kColZ + k]);
  }
}

template <int R1, int R2>
cudaError_t dpc_cols_t(const FftDesc& fy, float2* Z, float2* Phi, const DpcGrid& g, bool first, bool last,
                       cudaStream_t s) {
  using L = WarpFft<R1, R2>;
  auto kern = last ? k_dpc_cols<R1, R2, true> : k_dpc_cols<R1, R2, false>;
  const size_t sm = sizeof(float2) * kDpcWarps * L::kRegion;
  cudaError_t e = ensure_smem((const void*)kern, sm);
  if (e != cudaSuccess) return e;
  const int units = (g.Mx / 2 + L::C - 1) / L::C, per = kDpcWarps / 2;
  launch(kern, (units + per - 1) / per, 32 * kDpcWarps, sm, s, Z, Phi, fy.tw4, g, (int)first);
  count_launches(1);
  return cudaGetLastError();
}
template <int R1, int R2>
cudaError_t dpc_rows_t(const FftDesc& fx, float2* Z, const float* com, const DpcGrid& g, float cs,
                       float inv_n, float* phase, int step, cudaStream_t s) {
  using L = WarpFft<R1, R2>;
  auto kern = step == 0 ? k_dpc_rows<R1, R2, 0> : step == 1 ? k_dpc_rows<R1, R2, 1> : k_dpc_rows<R1, R2, 2>;
  const size_t sm = sizeof(float2) * kDpcWarps * L::kRegion;
  cudaError_t e = ensure_smem((const void*)kern, sm);
  if (e != cudaSuccess) return e;
  const int RY = kDpcWarps * L::C;
  launch(kern, (g.Ny + RY - 1) / RY, 32 * kDpcWarps, sm, s, Z, com, fx.tw4, g, cs, inv_n, phase);
  count_launches(1);
  return cudaGetLastError();
}
#define EER4D_DPC_SIDE(N, CALL)                                                            \
  switch (N) {                                                                             \
    case 1024: { constexpr int R1 = 32, R2 = 32; return CALL; }                            \
    case 512: { constexpr int R1 = 32, R2 = 16; return CALL; }                             \
    case 256: { constexpr int R1 = 16, R2 = 16; return CALL; }                             \
    case 128: { constexpr int R1 = 16, R2 = 8; return CALL; }                              \
    case 64: { constexpr int R1 = 8, R2 = 8; return CALL; }                                \
    case 32: { constexpr int R1 = 8, R2 = 4; return CALL; }                                \
    default: { constexpr int R1 = 4, R2 = 4; return CALL; }                                \
  }
cudaError_t dpc_cols(const FftDesc& fy, float2* Z, float2* Phi, const DpcGrid& g, bool first, bool last,
                     cudaStream_t s) {
  EER4D_DPC_SIDE(fy.N, (dpc_cols_t<R1, R2>(fy, Z, Phi, g, first, last, s)))
}
cudaError_t dpc_rows(const FftDesc& fx, float2* Z, const float* com, const DpcGrid& g, float cs, float inv_n,
                     float* phase, int step, cudaStream_t s) {
  EER4D_DPC_SIDE(fx.N, (dpc_rows_t<R1, R2>(fx, Z, com, g, cs, inv_n, phase, step, s)))
}
#undef EER4D_DPC_SIDE

unsigned grid_for(size_t n) {
  const size_t b = (n + 255) / 256;
  return (unsigned)(b < 4096 ? b : 4096);
}

}  // namespace

size_t dpc_iterative_scratch_bytes(const eer4d_plan* p, int pad) {
  return 3 * sizeof(float2) * (size_t)pad * pad * p->F;
}

cudaError_t launch_dpc_iterative(const eer4d_plan* p, const float* com, double lam1, double lam2,
                                 double mu, int n_iter, int pad, void* scratch, float* phase,
                                 cudaStream_t s) {
  const int Ny = p->g.scan_ny, Nx = p->g.scan_nx;
  const FftDesc& fy = pad == 2 ? p->fy2 : p->fy;
  const FftDesc& fx = pad == 2 ? p->fx2 : p->fx;
  const int My = fy.N, Mx = fx.N;
  const size_t n = (size_t)My * Mx;
  float2* Phi = static_cast<float2*>(scratch);
  float2* Z = Phi + n;
  float2* Cpk = Z + n;
  const float cscale = (float)(p->g.dalpha_raw_rad / p->g.lambda_A);
  const float inv_lx = (float)(1.0 / ((double)Mx * p->g.step_A));
  const float inv_ly = (float)(1.0 / ((double)My * p->g.step_A));
  const unsigned gb = grid_for(n);
  stage_begin(p, EER4D_STAGE_DPC, s);
  const auto side = [](const FftDesc& d) { return d.tw4 != nullptr; };  // powers of two, 16 ... 1024
  if (side(fy) && side(fx) && n_iter > 0) {
    const DpcGrid g{Ny, Nx, My, Mx, inv_lx, inv_ly, (float)lam1, (float)lam2, (float)mu};
    const float inv = 1.f / ((float)My * (float)Mx);
    cudaError_t e = dpc_rows(fx, Z, com, g, cscale, inv, phase, 0, s);
    for (int l = 1; l <= n_iter && e == cudaSuccess; ++l) {
      if ((e = dpc_cols(fy, Z, Phi, g, l == 1, l == n_iter, s)) != cudaSuccess) break;
      e = dpc_rows(fx, Z, com, g, cscale, inv, phase, l == n_iter ? 2 : 1, s);
    }
    stage_end(p, EER4D_STAGE_DPC, s);
    return e;
  }
  launch(k_dpc_setup, gb, 256, 0, s, com, Ny, Nx, My, Mx, cscale, Cpk, Phi);
  count_launches(1);
  cudaError_t e = cudaGetLastError();
  const float inv_n = 1.f / ((float)My * (float)Mx);
  for (int l = 0; l < n_iter && e == cudaSuccess; ++l) {
    launch(k_dpc_deriv, gb, 256, 0, s, Phi, My, Mx, inv_lx, inv_ly, Z);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) break;
    if ((e = launch_fft2_c2c(fy, fx, Z, -1, inv_n, s)) != cudaSuccess) break;
    launch(k_dpc_resid, gb, 256, 0, s, Cpk, Ny, Nx, My, Mx, Z);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) break;
    if ((e = launch_fft2_c2c(fy, fx, Z, 1, 1.f, s)) != cudaSuccess) break;
    launch(k_dpc_update, gb, 256, 0, s, Z, My, Mx, inv_lx, inv_ly, (float)lam1, (float)lam2,
           (float)mu, Phi);
    count_launches(1);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  if ((e = cudaMemcpyAsync(Z, Phi, sizeof(float2) * n, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
    return e;
  if ((e = launch_fft2_c2c(fy, fx, Z, -1, inv_n, s)) != cudaSuccess) return e;
  launch(k_dpc_out, grid_for((size_t)Ny * Nx), 256, 0, s, Z, Ny, Nx, Mx, phase);
  count_launches(1);
  stage_end(p, EER4D_STAGE_DPC, s);
  return cudaGetLastError();
}
