// Standalone truncated SVD of a device matrix (the factorisation of the local
// update, Sec. 2.3.4): one-sided Jacobi in FP64 and the truncation rule
// k = min(chi_max, min{k : sqrt(sum_{j>k} s_j^2) <= tau_rel ||M||_F}), k >= 1,
// dropping s_j <= 1e-13 s_1. Exposed through the C ABI in include/ttfit.h.
#include <cuda_runtime.h>
#include <algorithm>
#include <cstdint>
#include <mutex>

#include "../../include/ttfit.h"
#include "common.cuh"
#include "kernels.h"

using namespace ttfit;

namespace {

// scratch layout (in doubles) for an m x n input, r = min(m, n), q = max(m, n):
// X (q r) | Ux (q r) | Vx (r r) | Vw (r r) | Sv (r) | nrm (1) | dinfo (2) | info (4 x u32 = 2) | k (1)
size_t svd_scratch_doubles(int m, int n) {
  const size_t r = std::min(m, n), q = std::max(m, n);
  return 2 * q * r + 2 * r * r + r + 1 + 2 + 2 + 1;
}
size_t svd_info_offset(int m, int n) {
  const size_t r = std::min(m, n), q = std::max(m, n);
  return 2 * q * r + 2 * r * r + r + 3;
}

__global__ void svd_outputs_kernel(int m, int n, int tr, const double* __restrict__ Ux, const double* __restrict__ Vx,
                                   const double* __restrict__ Sv, double* __restrict__ U, double* __restrict__ S,
                                   double* __restrict__ Vt, uint32_t* errw) {
  // X = Ux diag(S) Vx^T with X = M (tr = 0, Ux m x r) or X = M^T (tr = 1, Ux n x r)
  const int r = min(m, n);
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  for (long long e = t0; e < (long long)m * r; e += stride) {  // U: m x r row-major
    const int i = (int)(e / r), j = (int)(e % r);
    U[e] = tr ? Vx[(size_t)j * r + i] : Ux[(size_t)j * m + i];
  }
  for (long long e = t0; e < (long long)r * n; e += stride) {  // Vt: r x n row-major
    const int j = (int)(e / n), c = (int)(e % n);
    Vt[e] = tr ? Ux[(size_t)j * n + c] : Vx[(size_t)j * r + c];
  }
  for (long long e = t0; e < r; e += stride) {
    S[e] = Sv[e];
    if (!isfinite(Sv[e])) atomicOr(errw, ERRW_NAN);
  }
}

// Columns of V (p x p, column-major, p <= 1024) whose value is null: where V is the left factor of R^T (svd_tall64) they
// are zero, or what rounding left. Here they become the rest of an orthonormal basis: the column itself, or, where that
// is no new direction, the unit vector that the columns before it cover least (1/p of its square is left at least), less
// its part in those columns, taken away twice. One CTA; returns at once where no value is null (256 x 256: 7.86 ms a call
// before, 7.87 so; of rank 128, 7.2 and 15.9: three passes of FP64 operations a column on one SM).
__global__ void __launch_bounds__(1024) complete_basis_kernel(int p, double* V, const double* S) {
  __shared__ double w[1024], cf[1024];
  __shared__ unsigned long long best;
  const int i = threadIdx.x, warp = i >> 5, lane = i & 31;
  const double lim = 0x1p-200 * S[0];  // below it the squares of two columns' products vanish in the Jacobi
  const int k0 = __syncthreads_count(i < p && S[min(i, p - 1)] > lim);
  double left = 1.0;  // of the square of unit vector i
  if (i < p)
    for (int k = 0; k < k0 && k0 < p; ++k) left = fma(-V[(size_t)k * p + i], V[(size_t)k * p + i], left);
  for (int j = k0; j < p; ++j) {
    double nrm = 0.0;
    for (int attempt = S[j] > 0.0 ? 0 : 1; attempt < 2 && !(nrm > 0.5); ++attempt) {
      if (attempt == 1) {
        if (i == 0) best = 0;
        __syncthreads();
        // the largest `left`, as a positive float's bits above the row
        if (i < p) atomicMax(&best, ((unsigned long long)__float_as_uint(fmaxf((float)left, 0.f)) << 32) | (unsigned)i);
        __syncthreads();
      }
      const int unit = attempt == 1 ? (int)(best & 0xFFFFFFFFu) : -1;
      w[i] = i >= p ? 0.0 : attempt == 1 ? (i == unit ? 1.0 : 0.0) : V[(size_t)j * p + i];
      for (int pass = 0; pass < 2; ++pass) {
        __syncthreads();
        if (pass == 0 && attempt == 1) {
          if (i < j) cf[i] = V[(size_t)i * p + unit];
        } else {
          for (int k = warp; k < j; k += 32) {
            double s = 0.0;
            for (int r = lane; r < p; r += 32) s = fma(V[(size_t)k * p + r], w[r], s);
            s = warp_sum(s);
            if (lane == 0) cf[k] = s;
          }
        }
        __syncthreads();
        if (i < p) {
          double x = w[i];
#pragma unroll 4
          for (int k = 0; k < j; ++k) x = fma(-cf[k], V[(size_t)k * p + i], x);
          w[i] = x;
        }
      }
      __syncthreads();
      double s = 0.0;  // every warp the same sum
      for (int r = lane; r < p; r += 32) s = fma(w[r], w[r], s);
      nrm = sqrt(warp_sum(s));
    }
    if (i < p) {
      const double x = w[i] / nrm;
      V[(size_t)j * p + i] = x;
      left = fma(-x, x, left);
    }
    __syncthreads();
  }
}

cudaError_t svd_run(const double* M, int m, int n, int chi_max, double tau_rel, double* U, double* S, double* Vt,
                    int* k_dev, double* scratch, double* extra, cudaStream_t st) {
  const int r = std::min(m, n), q = std::max(m, n);
  const bool tr = m < n;
  double* X = scratch;
  double* Ux = X + (size_t)q * r;
  double* Vx = Ux + (size_t)q * r;
  double* Vw = Vx + (size_t)r * r;
  double* Sv = Vw + (size_t)r * r;
  double* nrm = Sv + r;
  double* dinfo = nrm + 1;
  uint32_t* info = (uint32_t*)(dinfo + 2);
  int* ex = (int*)info + 2;
  cudaError_t e = cudaMemsetAsync(info, 0, 4 * sizeof(uint32_t), st);
  if (e != cudaSuccess) return e;
  // X = 2^-ex M, largest entry near 1: its squares stay in range. Tall orientation, column-major: M^T column-major is M
  // row-major (tr); else transpose
  double* M1 = tr ? X : Ux;
  if ((e = scale_norm<double, double>(M, (long long)m * n, M1, ex, nrm, info, st)) != cudaSuccess) return e;
  if (!tr && (e = copy_map<double, double>(m, n, M1, IdxMap::lin(n), IdxMap::lin(1), X, IdxMap::lin(1), IdxMap::lin(m), 1.0,
                                           st)) != cudaSuccess)
    return e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = svd_tall64(q, r, X, Ux, Vw, extra, extra ? extra + (size_t)r * r : nullptr, &Ux, Sv, Vx, 60, info, sms, st)) != cudaSuccess) return e;
  if (Ux == X) {  // by way of the QR; else V is the product of the rotations
    ++tl_launches;
    complete_basis_kernel<<<1, 1024, 0, st>>>(r, Vx, Sv);
  }
  if ((e = fix_signs<double>(tr ? r : q, tr ? q : r, r, tr ? Vx : Ux, tr ? r : q, tr ? Ux : Vx, tr ? q : r, st)) !=
      cudaSuccess)
    return e;
  if ((e = truncate_rule<double>(Sv, r, nrm, ex, tau_rel, chi_max, 1e-13, k_dev, dinfo, st)) != cudaSuccess) return e;
  const long long tot = (long long)q * r;
  const int blocks = (int)std::max<long long>(1, std::min<long long>((tot + 255) / 256, 1024));
  ++tl_launches;
  svd_outputs_kernel<<<blocks, 256, 0, st>>>(m, n, tr ? 1 : 0, Ux, Vx, Sv, U, S, Vt, info);
  return cudaGetLastError();
}

tt_status svd_check(const double* M, int m, int n, int chi_max, double tau_rel, const double* U, const double* S,
                    const double* Vt, const int* k_out) {
  if (!M || !U || !S || !Vt || !k_out) return TT_ERR_INVALID_ARGUMENT;
  if (m < 1 || n < 1 || chi_max < 1 || !(tau_rel >= 0.0)) return TT_ERR_INVALID_ARGUMENT;
  if (std::min(m, n) > 1024) return TT_ERR_INVALID_ARGUMENT;
  return TT_OK;
}

}  // namespace

extern "C" tt_status tt_svd_truncated(const double* M, int m, int n, int chi_max, double tau_rel, double* U,
                                      double* S, double* Vt, int* k_out, void* stream) {
  tt_status s = svd_check(M, m, n, chi_max, tau_rel, U, S, Vt, k_out);
  if (s != TT_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t nd = svd_scratch_doubles(m, n), r2 = (size_t)std::min(m, n) * std::min(m, n);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return TT_ERR_CUDA;
  }
  size_t got = 0;
  double* scratch = (double*)block_take(dev, (nd + 2 * r2) * sizeof(double), &got);
  if (!scratch) return TT_ERR_OUT_OF_MEMORY;
  int* k_dev = (int*)(scratch + nd - 1);
  cudaError_t e = svd_run(M, m, n, chi_max, tau_rel, U, S, Vt, k_dev, scratch, scratch + nd, st);
  int k = 0;
  uint32_t flags[2] = {0, 0};
  if (e == cudaSuccess) e = cudaMemcpyAsync(&k, k_dev, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(flags, scratch + svd_info_offset(m, n), 2 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st);
  const cudaError_t es = cudaStreamSynchronize(st);  // before the block goes back, whatever failed
  if (e == cudaSuccess) e = es;
  block_give(dev, got, scratch);
  if (e != cudaSuccess) return TT_ERR_CUDA;
  if (flags[0] & (ERRW_NAN | ERRW_NOCONV)) return TT_ERR_NUMERICAL;
  *k_out = k;
  return TT_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free variant. Its scratch is this file-scope device array: every
// GPU that loads the library holds these 4 MiB until the process exits, and
// every call on a device reuses the same array (so calls that overlap on the
// GPU race). Host code may not use the array's name as a device address; the
// address is looked up per device with cudaGetSymbolAddress and cached.
// ---------------------------------------------------------------------------
namespace {

constexpr size_t kNoAllocDoubles = size_t(1) << 19;  // 4 MiB of FP64 scratch
__device__ __align__(256) double g_svd_scratch[kNoAllocDoubles];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
double* g_scratch_ptr[kMaxDevices] = {};

// Device address of g_svd_scratch on the current device (looked up on the
// first call on that device, with that device current).
cudaError_t noalloc_scratch(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_svd_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_ptr[dev] = (double*)p;
  }
  *out = g_scratch_ptr[dev];
  return cudaSuccess;
}

}  // namespace

extern "C" tt_status tt_svd_truncated_noalloc(const double* M, int m, int n, int chi_max, double tau_rel, double* U,
                                              double* S, double* Vt, int* k_out, void* stream) {
  tt_status s = svd_check(M, m, n, chi_max, tau_rel, U, S, Vt, k_out);
  if (s != TT_OK) return s;
  const size_t nd = svd_scratch_doubles(m, n);
  if (nd > kNoAllocDoubles) return TT_ERR_INVALID_ARGUMENT;  // beyond the fixed scratch
  cudaStream_t st = (cudaStream_t)stream;
  double* scratch = nullptr;
  if (noalloc_scratch(&scratch) != cudaSuccess) {
    cudaGetLastError();
    return TT_ERR_CUDA;
  }
  int* k_dev = (int*)(scratch + nd - 1);
  // the FP32 sweeps' scratch, where the array has room for it as well
  const size_t r = std::min(m, n);
  double* extra = nd + 2 * r * r <= kNoAllocDoubles ? scratch + nd : nullptr;
  // svd_run clears the error flags it reads; every other scratch word it uses
  // is written before it is read
  cudaError_t e = svd_run(M, m, n, chi_max, tau_rel, U, S, Vt, k_dev, scratch, extra, st);
  int k = 0;
  uint32_t flags[2] = {0, 0};
  if (e == cudaSuccess) e = cudaMemcpyAsync(&k, k_dev, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(flags, scratch + svd_info_offset(m, n), 2 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return TT_ERR_CUDA;
  if (flags[0] & (ERRW_NAN | ERRW_NOCONV)) return TT_ERR_NUMERICAL;
  *k_out = k;
  return TT_OK;
}
