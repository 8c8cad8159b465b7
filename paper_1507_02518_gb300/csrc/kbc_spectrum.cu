// kbc_spectrum.cu -- shell-summed kinetic-energy spectrum E(kappa) of a velocity field on a
// periodic N^3 grid (Sec. "Numerical Simulations": k = integral of E(kappa) d kappa,
// D(kappa) = 2 nu kappa^2 E(kappa)).
//
// Per component, a copy to an aligned real buffer and a real-to-complex 3D FFT (cuFFT,
// library step) in the caller's work buffer, then shell_kernel bins 1/2 |u_hat|^2 / P^2 by m = rint(|n|) of the integer wave
// vector n in a per-block shared-memory histogram (FP64), and shell_final_kernel adds the
// block histograms in a fixed order. The n = 0 mode (the mean flow) is left out.
#include <cuda_runtime.h>
#include <cufft.h>
#include <stdint.h>

#include "kbc_ops.h"

namespace kbc {
namespace {

constexpr int kSpecBlocks = 608;  // 4 per SM on 152 SMs
constexpr size_t kAlign = 256;

size_t align_up(size_t v) { return (v + kAlign - 1) / kAlign * kAlign; }

// FP32 to FP64 by the bits (a conversion costs the FP64 pipe as much as an FMA)
__device__ __forceinline__ double widen(float v) {
  const uint32_t b = __float_as_uint(v), a = b & 0x7fffffffu;
  if (a - 0x00800000u >= 0x7f000000u) return (double)v;  // zero, subnormal, infinite, NaN
  return __hiloint2double((int)((b & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(b << 29));
}
// |c|^2 + sum
__device__ __forceinline__ double norm2(const cufftComplex& c, double sum) {
  const double x = widen(c.x), y = widen(c.y);
  return __fma_rn(x, x, __fma_rn(y, y, sum));
}
__device__ __forceinline__ double norm2(const cufftDoubleComplex& c, double sum) {
  return __fma_rn(c.x, c.x, __fma_rn(c.y, c.y, sum));
}

// A warp takes 32 consecutive kx of the up to four rows (+-ky, +-kz), whose modes lie on the same
// shells: a lane adds its four modes by FMAs (FP64 additions bound this kernel: 3.5 FP64
// instructions a mode, 9 for one row at a time, 185 us). Along kx the shells do not decrease, so
// modes of the same shell are neighbours, and the warp adds them up before one lane of each run
// adds to the histogram (an FP64 addition in shared memory is a compare-and-swap loop, which the
// modes of a row near kx = 0 all wanted at once). The shell is exact in integers: the FP32 square
// root is corrected by 4 k^2 against (2m +- 1)^2. 256^3 FP32 spectrum 3.08 -> 2.07 ms (FP64
// 12.97 -> 7.66), the shells of a component 355 -> 110 us.
template <typename C>
__global__ void __launch_bounds__(256) shell_kernel(const C* X, uint32_t n, int nbins,
                                                    double scale, double* partials) {
  extern __shared__ double hist[];
  for (int m = threadIdx.x; m < nbins; m += blockDim.x) hist[m] = 0.0;
  __syncthreads();
  const uint32_t nh = n / 2 + 1, chunks = (nh + 31) / 32, lane = threadIdx.x & 31;
  const uint32_t units = nh * nh * chunks;
  const uint32_t warps = gridDim.x * (blockDim.x >> 5);
  for (uint32_t q = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); q < units; q += warps) {
    const uint32_t row = q / chunks, kx = (q - row * chunks) * 32 + lane;
    const uint32_t kz = row / nh, ky = row - kz * nh;
    // the rows n - ky and n - kz, where they are rows of their own
    const bool my = ky != 0 && 2 * ky != n, mz = kz != 0 && 2 * kz != n;
    double v = 0.0;
    int m = 0x7fffffff;  // lanes without a mode: a run of their own
    if (kx < nh) {
      const int k2 = (int)(kx * kx + ky * ky + kz * kz);
      m = (int)(sqrtf((float)k2) + 0.5f);
      if (4 * k2 > (2 * m + 1) * (2 * m + 1)) ++m;
      else if (m > 0 && 4 * k2 < (2 * m - 1) * (2 * m - 1)) --m;
      auto at = [&](uint32_t y, uint32_t z) { return X[((uint64_t)z * n + y) * nh + kx]; };
      v = norm2(at(ky, kz), 0.0);
      if (my) v = norm2(at(n - ky, kz), v);
      if (mz) v = norm2(at(ky, n - kz), v);
      if (my && mz) v = norm2(at(n - ky, n - kz), v);
      // the half spectrum holds one of each pair (n, -n), whose two halves |u_hat|^2 / 2 are
      // equal, except on the kx = 0 and kx = n/2 planes, which hold both members
      v = __dmul_rn(v, (kx == 0 || (n % 2 == 0 && kx == n / 2)) ? scale : 2.0 * scale);
      if (k2 == 0) m = -1;  // the mean flow is left out
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int mm = __shfl_down_sync(0xffffffffu, m, o);
      const bool same = lane + o < 32 && mm == m;
      if (!__any_sync(0xffffffffu, same)) break;
      const double add = __shfl_down_sync(0xffffffffu, v, o);
      if (same) v = __dadd_rn(v, add);
    }
    const int before = __shfl_up_sync(0xffffffffu, m, 1);
    if ((lane == 0 || before != m) && m >= 0 && m < nbins) atomicAdd(&hist[m], v);
  }
  __syncthreads();
  for (int m = threadIdx.x; m < nbins; m += blockDim.x)
    partials[(uint64_t)blockIdx.x * nbins + m] = hist[m];
}

__global__ void shell_final_kernel(const double* partials, int nblocks, int nbins,
                                   double* bins) {
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < nbins; m += gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int b = 0; b < nblocks; ++b) acc += partials[(uint64_t)b * nbins + m];
    bins[m] += acc;
  }
}

struct Plan {
  cufftHandle h = 0;
  bool ok = false;
  ~Plan() {
    if (ok) cufftDestroy(h);
  }
};

// plan without its own work area; *ws receives the work-area bytes
cufftResult make_plan(Plan* p, uint32_t n, bool fp64, size_t* ws) {
  cufftResult r = cufftCreate(&p->h);
  if (r != CUFFT_SUCCESS) return r;
  p->ok = true;
  r = cufftSetAutoAllocation(p->h, 0);
  if (r != CUFFT_SUCCESS) return r;
  return cufftMakePlan3d(p->h, (int)n, (int)n, (int)n, fp64 ? CUFFT_D2Z : CUFFT_R2C, ws);
}

struct WorkLayout {
  size_t real, spec, fft, partials, bins, total;
};
WorkLayout layout(uint32_t n, bool fp64, int nbins, size_t fft_ws) {
  WorkLayout L;
  size_t off = 0;
  // one velocity component, copied to a 256-byte aligned start (the components of the
  // velocity field start at multiples of n^3 values, which cuFFT does not accept for odd n)
  L.real = off;
  off += align_up((size_t)n * n * n * (fp64 ? 8 : 4));
  L.spec = off;
  off += align_up((size_t)n * n * (n / 2 + 1) * (fp64 ? 16 : 8));
  L.fft = off;
  off += align_up(fft_ws);
  L.partials = off;
  off += align_up(sizeof(double) * (size_t)kSpecBlocks * nbins);
  L.bins = off;
  off += align_up(sizeof(double) * (size_t)nbins);
  L.total = off;
  return L;
}

}  // namespace

size_t spectrum_work_bytes(uint32_t n, bool fp64, int nbins) {
  Plan p;
  size_t ws = 0;
  if (make_plan(&p, n, fp64, &ws) != CUFFT_SUCCESS) return 0;
  return layout(n, fp64, nbins, ws).total;
}

// ufield: [3][n^3] velocity in FP64 (fp64) or FP32; bins_host receives nbins values
int spectrum(const void* ufield, uint32_t n, bool fp64, int nbins, void* work, size_t work_bytes,
             double* bins_host, cudaStream_t st, const char** why) {
  Plan p;
  size_t ws = 0;
  if (make_plan(&p, n, fp64, &ws) != CUFFT_SUCCESS) {
    *why = "cuFFT plan creation failed";
    return 3;
  }
  const WorkLayout L = layout(n, fp64, nbins, ws);
  if (work_bytes < L.total) {
    *why = "work buffer smaller than lb_spectrum_work_bytes";
    return 2;
  }
  char* base = (char*)work;
  if (cufftSetWorkArea(p.h, base + L.fft) != CUFFT_SUCCESS ||
      cufftSetStream(p.h, st) != CUFFT_SUCCESS) {
    *why = "cuFFT work area or stream";
    return 3;
  }
  double* bins = (double*)(base + L.bins);
  double* partials = (double*)(base + L.partials);
  cudaError_t e = cudaMemsetAsync(bins, 0, sizeof(double) * nbins, st);
  const uint64_t P = (uint64_t)n * n * n;
  const double scale = 0.5 / ((double)P * (double)P);
  const size_t shm = sizeof(double) * nbins;
  const size_t esz = fp64 ? 8 : 4;
  for (int a = 0; a < 3 && e == cudaSuccess; ++a) {
    e = cudaMemcpyAsync(base + L.real, (const char*)ufield + a * P * esz, P * esz,
                        cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) break;
    cufftResult r;
    if (fp64) {
      r = cufftExecD2Z(p.h, (cufftDoubleReal*)(base + L.real),
                       (cufftDoubleComplex*)(base + L.spec));
    } else {
      r = cufftExecR2C(p.h, (cufftReal*)(base + L.real), (cufftComplex*)(base + L.spec));
    }
    if (r != CUFFT_SUCCESS) {
      *why = "cuFFT execution failed";
      return 3;
    }
    if (fp64)
      shell_kernel<cufftDoubleComplex><<<kSpecBlocks, 256, shm, st>>>(
          (const cufftDoubleComplex*)(base + L.spec), n, nbins, scale, partials);
    else
      shell_kernel<cufftComplex><<<kSpecBlocks, 256, shm, st>>>(
          (const cufftComplex*)(base + L.spec), n, nbins, scale, partials);
    shell_final_kernel<<<(nbins + 255) / 256, 256, 0, st>>>(partials, kSpecBlocks, nbins, bins);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(bins_host, bins, sizeof(double) * nbins, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    *why = cudaGetErrorString(e);
    return 3;
  }
  return 0;
}

}  // namespace kbc
