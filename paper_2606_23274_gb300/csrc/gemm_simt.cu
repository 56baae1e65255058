// CUDA-core GEMM over arbitrary tensor layouts:
//   C[cm(m) + cn(n)] = alpha * sum_k A[am(m) + ak(k)] * B[bn(n) + bk(k)] + beta * C[...]
// Every contraction of the fit (environment diagrams, halves, two-site tensor)
// is one call with the index maps of its operands (Sec. 2.3.3 / 2.3.4 shapes).
// It serves the FP64 path, the double-FP32 (df32) path that reaches FP64-class
// accuracy on the FP32 pipes, and the plain-FP32 baseline; the tensor-core
// path lives in gemm_tc.cu.
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace ttfit {

constexpr int BK = 16, NT = 256;

// Tile edge TB = 16 MT: a 16 x 16 thread grid, MT x MT outputs a thread. FP64 and df32 tiles are bound
// by their SM's arithmetic (an FP64 multiply-add of a warp takes 19 cycles of an SM, a df32 one 15
// FP32 instructions), so a small product is cut into small tiles, which spread over more SMs and carry
// less padding; a tile's operand traffic stays far below what an SM can load in that time.
template <typename T, int MT>
__global__ void __launch_bounds__(NT, 3) gemm_simt_kernel(GemmArgs<T> g, T* __restrict__ ws, int k_per_split) {
  constexpr int TB = 16 * MT;
  __shared__ T As[BK][TB + 1];
  __shared__ T Bs[BK][TB + 1];
  __shared__ long long arow[TB], brow[TB];
  __shared__ long long akoff[BK], bkoff[BK];  // k offsets of the current tile (one index-map evaluation each)
  const int tid = threadIdx.x;
  const int m0 = blockIdx.y * TB, n0 = blockIdx.x * TB;
  const int kb = blockIdx.z * k_per_split;
  const int ke = min(g.K, kb + k_per_split);
  if (tid < TB) arow[tid] = (m0 + tid < g.M) ? g.am(m0 + tid) : 0;
  else if (tid < 2 * TB) brow[tid - TB] = (n0 + tid - TB < g.N) ? g.bn(n0 + tid - TB) : 0;
  __syncthreads();
  const int tx = tid & 15, ty = tid >> 4;
  T acc[MT][MT];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < MT; ++j) acc[i][j] = T(0);

  for (int k0 = kb; k0 < ke; k0 += BK) {
    if (tid < BK) akoff[tid] = (k0 + tid < ke) ? g.ak(k0 + tid) : 0;
    else if (tid < 2 * BK) bkoff[tid - BK] = (k0 + tid - BK < ke) ? g.bk(k0 + tid - BK) : 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < MT; ++i) {
      int e = tid + NT * i;
      int r, kk;
      if (g.a_kfast) { r = e >> 4; kk = e & 15; } else { r = e % TB; kk = e / TB; }
      T v = T(0);
      if (m0 + r < g.M && k0 + kk < ke) v = g.A[arow[r] + akoff[kk]];
      As[kk][r] = v;
      if (g.b_kfast) { r = e >> 4; kk = e & 15; } else { r = e % TB; kk = e / TB; }
      T w = T(0);
      if (n0 + r < g.N && k0 + kk < ke) w = g.B[brow[r] + bkoff[kk]];
      Bs[kk][r] = w;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      T a[MT], b[MT];
#pragma unroll
      for (int i = 0; i < MT; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < MT; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < MT; ++j) acc[i][j] = madd(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  if (ws) {  // split-K partial: dense [split][M][N]
    T* w = ws + (size_t)blockIdx.z * g.M * g.N;
#pragma unroll
    for (int i = 0; i < MT; ++i) {
      int m = m0 + ty + 16 * i;
      if (m >= g.M) continue;
#pragma unroll
      for (int j = 0; j < MT; ++j) {
        int n = n0 + tx + 16 * j;
        if (n < g.N) w[(size_t)m * g.N + n] = acc[i][j];
      }
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    int m = m0 + ty + 16 * i;
    if (m >= g.M) continue;
    long long cr = g.cm(m);
    long long cr2 = g.C2 ? g.cm2(m) : 0;
#pragma unroll
    for (int j = 0; j < MT; ++j) {
      int n = n0 + tx + 16 * j;
      if (n >= g.N) continue;
      long long o = cr + g.cn(n);
      T v = g.alpha * acc[i][j];
      if (g.C2) g.C2[cr2 + g.cn2(n)] = v;
      if (g.beta != T(0)) v += g.beta * g.C[o];
      g.C[o] = v;
    }
  }
}

// FP32. 128 threads, each 8 x 4 outputs (rows 8 ty .. 8 ty + 7, columns tx + TX j); k-tiles of 16 in two shared
// buffers, the next one's loads in registers while the present one is multiplied, and the k offsets of 256 terms
// tabulated at a time. The kernel above waits for its loads and evaluates the k maps in every k-tile: for the
// gradient's products (3072 x 384 x 96, 6144 x 192 x 192, 9216 x 32 x 128) it was bound by that latency, at
// 5 TFLOP/s. Sums run in the same order, so the results are the same bits.
template <int BM, int BN>
__global__ void __launch_bounds__(128) gemm_f32_kernel(GemmArgs<float> g, float* __restrict__ ws, int k_per_split) {
  constexpr int TX = BN / 4, KC = 256, NA = BM * BK / 128, NB = BN * BK / 128;
  static_assert(TX * (BM / 8) == 128, "8 x 4 outputs a thread");
  __shared__ __align__(16) float As[2][BK][BM + 4];
  __shared__ float Bs[2][BK][BN + 1];
  __shared__ long long arow[BM], brow[BN];
  __shared__ long long akoff[KC], bkoff[KC];
  const int tid = threadIdx.x;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int kb = blockIdx.z * k_per_split;
  const int ke = min(g.K, kb + k_per_split);
  for (int t = tid; t < BM + BN; t += 128) {
    if (t < BM) arow[t] = (m0 + t < g.M) ? g.am(m0 + t) : 0;
    else brow[t - BM] = (n0 + t - BM < g.N) ? g.bn(n0 + t - BM) : 0;
  }
  const int tx = tid % TX, ty = tid / TX;
  float acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  float ra[NA], rb[NB];
  auto load = [&](int k0) {
    const int c0 = (k0 - kb) % KC;
    if (c0 == 0) {  // the next stretch of k offsets
      __syncthreads();
      for (int t = tid; t < KC; t += 128) {
        akoff[t] = k0 + t < ke ? g.ak(k0 + t) : 0;
        bkoff[t] = k0 + t < ke ? g.bk(k0 + t) : 0;
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int e = tid + 128 * i;
      const int r = g.a_kfast ? e / BK : e % BM, kk = g.a_kfast ? e % BK : e / BM;
      ra[i] = (m0 + r < g.M && k0 + kk < ke) ? g.A[arow[r] + akoff[c0 + kk]] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int e = tid + 128 * i;
      const int r = g.b_kfast ? e / BK : e % BN, kk = g.b_kfast ? e % BK : e / BN;
      rb[i] = (n0 + r < g.N && k0 + kk < ke) ? g.B[brow[r] + bkoff[c0 + kk]] : 0.f;
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int e = tid + 128 * i;
      const int r = g.a_kfast ? e / BK : e % BM, kk = g.a_kfast ? e % BK : e / BM;
      As[buf][kk][r] = ra[i];
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int e = tid + 128 * i;
      const int r = g.b_kfast ? e / BK : e % BN, kk = g.b_kfast ? e % BK : e / BN;
      Bs[buf][kk][r] = rb[i];
    }
  };
  if (kb < ke) {
    load(kb);
    store(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = kb; k0 < ke; k0 += BK) {
      const bool more = k0 + BK < ke;
      if (more) load(k0 + BK);
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][kk][8 * ty]);
        const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][kk][8 * ty + 4]);
        const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        float b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = Bs[buf][kk][tx + TX * j];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
      }
      if (more) store(buf ^ 1);
      buf ^= 1;
      __syncthreads();
    }
  }
  if (ws) {  // split-K partial: dense [split][M][N]
    float* w = ws + (size_t)blockIdx.z * g.M * g.N;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int m = m0 + 8 * ty + i;
      if (m >= g.M) continue;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int n = n0 + tx + TX * j;
        if (n < g.N) w[(size_t)m * g.N + n] = acc[i][j];
      }
    }
    return;
  }
  long long cn[4], cn2[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int n = min(n0 + tx + TX * j, g.N - 1);
    cn[j] = g.cn(n);
    cn2[j] = g.C2 ? g.cn2(n) : 0;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = m0 + 8 * ty + i;
    if (m >= g.M) continue;
    const long long cr = g.cm(m), cr2 = g.C2 ? g.cm2(m) : 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (n0 + tx + TX * j >= g.N) continue;
      float v = g.alpha * acc[i][j];
      if (g.C2) g.C2[cr2 + cn2[j]] = v;
      if (g.beta != 0.f) v += g.beta * g.C[cr + cn[j]];
      g.C[cr + cn[j]] = v;
    }
  }
}

// Sum of the split-K partials into the output layouts. A block takes 8 rows of 32 columns: the partials are read
// along the columns, each output is written along its own fast direction, and the index maps are evaluated once
// a row and column of the tile (four maps and a 64-bit division an element took 20 us for 512 x 512 df32).
template <typename T>
__global__ void __launch_bounds__(256) splitk_reduce_kernel(GemmArgs<T> g, const T* __restrict__ ws, int splits) {
  __shared__ T tile[8][33];
  __shared__ long long rm[8], rm2[8], cn[32], cn2[32];
  const int t = threadIdx.x;
  const long long total = (long long)g.M * g.N;
  const int nct = (g.N + 31) / 32, nrt = (g.M + 7) / 8;
  for (long long b = blockIdx.x; b < (long long)nct * nrt; b += gridDim.x) {
    const int m0 = (int)(b / nct) * 8, n0 = (int)(b % nct) * 32;
    if (t < 32) cn[t] = g.cn(min(n0 + t, g.N - 1));
    else if (t < 40) rm[t - 32] = g.cm(min(m0 + t - 32, g.M - 1));
    else if (g.C2 && t >= 64 && t < 96) cn2[t - 64] = g.cn2(min(n0 + t - 64, g.N - 1));
    else if (g.C2 && t >= 96 && t < 104) rm2[t - 96] = g.cm2(min(m0 + t - 96, g.M - 1));
    {
      const int i = t >> 5, j = t & 31;
      T s = T(0);
      if (m0 + i < g.M && n0 + j < g.N) {
        const T* w = ws + (size_t)(m0 + i) * g.N + n0 + j;
#pragma unroll 4
        for (int z = 0; z < splits; ++z) s += w[(size_t)z * total];
        s = g.alpha * s;
      }
      tile[i][j] = s;
    }
    __syncthreads();
    auto each = [&](bool along_rows, auto put) {  // along_rows: neighbouring threads take neighbouring rows
      const int i = along_rows ? t & 7 : t >> 5, j = along_rows ? t >> 3 : t & 31;
      if (m0 + i < g.M && n0 + j < g.N) put(i, j);
    };
    if (g.C2) each(g.cn2.s2 != 1, [&](int i, int j) { g.C2[rm2[i] + cn2[j]] = tile[i][j]; });
    each(g.cn.s2 != 1, [&](int i, int j) {
      const long long o = rm[i] + cn[j];
      T v = tile[i][j];
      if (g.beta != T(0)) v += g.beta * g.C[o];
      g.C[o] = v;
    });
    __syncthreads();
  }
}

template <typename T>
cudaError_t splitk_reduce(const GemmArgs<T>& g, const T* ws, int splits, int sm_count, cudaStream_t st) {
  const long long tiles = (long long)((g.N + 31) / 32) * ((g.M + 7) / 8);
  const int blocks = (int)(tiles < (1 << 16) ? tiles : (1 << 16));
  (void)sm_count;
  ++tl_launches;
  splitk_reduce_kernel<T><<<blocks < 1 ? 1 : blocks, 256, 0, st>>>(g, ws, splits);
  return cudaGetLastError();
}
template cudaError_t splitk_reduce<double>(const GemmArgs<double>&, const double*, int, int, cudaStream_t);
template cudaError_t splitk_reduce<float>(const GemmArgs<float>&, const float*, int, int, cudaStream_t);
template cudaError_t splitk_reduce<df32>(const GemmArgs<df32>&, const df32*, int, int, cudaStream_t);

template <typename T>
cudaError_t gemm_simt(const GemmArgs<T>& g, T* ws, size_t ws_elems, int sm_count, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  if (g.K <= 0) {  // empty contraction: C = beta * C
    GemmArgs<T> z = g;
    z.alpha = T(0);
    ++tl_launches;
    splitk_reduce_kernel<T><<<256, 256, 0, st>>>(z, nullptr, 0);
    return cudaGetLastError();
  }
  const bool slow = std::is_same<T, double>::value || std::is_same<T, df32>::value;
  auto tiles_of = [&](int mt) { return (long long)((g.M + 16 * mt - 1) / (16 * mt)) * ((g.N + 16 * mt - 1) / (16 * mt)); };
  // FP64 and df32: the largest of 64, 32 and 16 that gives two tiles an SM. FP64 gradient of chi = 12
  // (products of 288 x 24 x 24 and the like): 39 us a launch with tiles of 64, 10 us so; 1.58 ms
  // against 4.44 ms for the call. FP32 has tiles of its own.
  int mt = 4;
  if (slow)
    while (mt > 1 && tiles_of(mt) < 2 * sm_count) mt /= 2;
  int tbm = 16 * mt, tbn = 16 * mt;
  // FP32: 64 x 64 tiles, 128 x 32 or 32 x 128 where one side is no wider than 32
  if (!slow && g.N <= 32) tbm = 128, tbn = 32;
  else if (!slow && g.M <= 32) tbm = 32, tbn = 128;
  int gm = (g.M + tbm - 1) / tbm, gn = (g.N + tbn - 1) / tbn;
  int tiles = gm * gn;
  int splits = 1;
  // split K while the grid covers fewer than two waves of the SMs and each
  // split keeps at least kmin terms
  const int kmin = slow ? 32 : 256;
  while (tiles * splits < 2 * sm_count && g.K / (splits * 2) >= kmin &&
         (size_t)(splits * 2) * g.M * g.N <= ws_elems)
    splits *= 2;
  int kps = (g.K + splits - 1) / splits;
  kps = (kps + BK - 1) / BK * BK;
  splits = (g.K + kps - 1) / kps;
  dim3 grid(gn, gm, splits);
  T* wsp = splits > 1 ? ws : nullptr;
  ++tl_launches;
  if constexpr (std::is_same<T, double>::value || std::is_same<T, df32>::value) {
    if (mt == 1) gemm_simt_kernel<T, 1><<<grid, NT, 0, st>>>(g, wsp, kps);
    else if (mt == 2) gemm_simt_kernel<T, 2><<<grid, NT, 0, st>>>(g, wsp, kps);
    else gemm_simt_kernel<T, 4><<<grid, NT, 0, st>>>(g, wsp, kps);
  } else {
    if (tbn == 32) gemm_f32_kernel<128, 32><<<grid, 128, 0, st>>>(g, wsp, kps);
    else if (tbm == 32) gemm_f32_kernel<32, 128><<<grid, 128, 0, st>>>(g, wsp, kps);
    else gemm_f32_kernel<64, 64><<<grid, 128, 0, st>>>(g, wsp, kps);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || splits == 1) return e;
  return splitk_reduce<T>(g, ws, splits, sm_count, st);
}

template cudaError_t gemm_simt<double>(const GemmArgs<double>&, double*, size_t, int, cudaStream_t);
template cudaError_t gemm_simt<float>(const GemmArgs<float>&, float*, size_t, int, cudaStream_t);
template cudaError_t gemm_simt<df32>(const GemmArgs<df32>&, df32*, size_t, int, cudaStream_t);

}  // namespace ttfit
