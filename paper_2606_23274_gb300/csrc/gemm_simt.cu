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
// by their SM's arithmetic (an FP64 multiply-add of a warp takes 17 cycles of an SM, a df32 one 15
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
#pragma unroll(MT == 1 ? 8 : 4)
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
  // output offsets of the tile's rows and columns: one evaluation each, one copy of each map's code
  __syncthreads();
  __shared__ long long crow2[TB], ccol2[TB];
  if (tid < TB) arow[tid] = g.cm(min(m0 + tid, g.M - 1));
  else if (tid < 2 * TB) brow[tid - TB] = g.cn(min(n0 + tid - TB, g.N - 1));
  if (g.C2) {
    if (tid < TB) crow2[tid] = g.cm2(min(m0 + tid, g.M - 1));
    else if (tid < 2 * TB) ccol2[tid - TB] = g.cn2(min(n0 + tid - TB, g.N - 1));
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    const int ml = ty + 16 * i;
    if (m0 + ml >= g.M) continue;
#pragma unroll
    for (int j = 0; j < MT; ++j) {
      const int nl = tx + 16 * j;
      if (n0 + nl >= g.N) continue;
      T v = g.alpha * acc[i][j];
      if (g.C2) g.C2[crow2[ml] + ccol2[nl]] = v;
      T* o = g.C + (arow[ml] + brow[nl]);
      if (g.beta != T(0)) v += g.beta * *o;
      *o = v;
    }
  }
}

// FP32. 128 threads, each 8 x 4 outputs (rows 8 ty .. 8 ty + 7, columns tx + TX j); k-tiles of 16 in two shared
// buffers, the next one's loads in registers while the present one is multiplied, the offsets of 256 terms of K
// tabulated at a time. The code is kept short: the loads and each index map stand once, the products are unrolled by
// 4, and the outputs go through shared memory to one small loop, which also writes them along their fast direction.
// A few warps an SM cannot hide the fetch of long straight code: with the outputs unrolled (bounds, second copy, beta)
// a 64 x 64 x 16 product took 8.2 us, and the products of the gradient (3072 x 384 x 96, ...) three times their
// arithmetic.
template <int BM, int BN>
__global__ void __launch_bounds__(128) gemm_f32_kernel(GemmArgs<float> g, float* __restrict__ ws, int k_per_split) {
  constexpr int NTH = 128, TX = BN / 4, KC = 256, NA = BM * BK / NTH, NB = BN * BK / NTH;
  constexpr int LA = BM + 4, LB = BN + 1, SA = BK * LA, SB = BK * LB;
  static_assert(TX * (BM / 8) == NTH, "8 x 4 outputs a thread");
  static_assert(2 * (SA + SB) >= BM * (BN + 1), "the output tile takes the place of the operands");
  __shared__ __align__(16) float sm[2 * (SA + SB)];  // [2][BK][LA] of A, [2][BK][LB] of B; then [BM][BN + 1] of C
  __shared__ long long arow[BM], brow[BN];
  __shared__ long long akoff[KC], bkoff[KC];
  const int tid = threadIdx.x;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int kb = blockIdx.z * k_per_split;
  const int ke = min(g.K, kb + k_per_split);
#pragma unroll 1
  for (int t = tid; t < BM; t += NTH) arow[t] = (m0 + t < g.M) ? g.am(m0 + t) : 0;
#pragma unroll 1
  for (int t = tid; t < BN; t += NTH) brow[t] = (n0 + t < g.N) ? g.bn(n0 + t) : 0;
  const int tx = tid % TX, ty = tid / TX;
  float acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  float ra[NA], rb[NB];
  int buf = 0;
#pragma unroll 1
  for (int k0 = kb - BK; k0 < ke; k0 += BK) {  // the first pass only loads
    const int kn = k0 + BK;                    // the k-tile to load
    if (kn < ke) {
      const int c0 = (kn - kb) % KC;
      if (c0 == 0) {  // the next stretch of k offsets
        __syncthreads();
        const int cnt = min(KC, (ke - kn + BK - 1) / BK * BK);
#pragma unroll 1
        for (int t = tid; t < cnt; t += NTH) {
          akoff[t] = kn + t < ke ? g.ak(kn + t) : 0;
          bkoff[t] = kn + t < ke ? g.bk(kn + t) : 0;
        }
        __syncthreads();
      }
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        const int e = tid + NTH * i;
        const int r = g.a_kfast ? e / BK : e % BM, kk = g.a_kfast ? e % BK : e / BM;
        ra[i] = (m0 + r < g.M && kn + kk < ke) ? g.A[arow[r] + akoff[c0 + kk]] : 0.f;
      }
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        const int e = tid + NTH * i;
        const int r = g.b_kfast ? e / BK : e % BN, kk = g.b_kfast ? e % BK : e / BN;
        rb[i] = (n0 + r < g.N && kn + kk < ke) ? g.B[brow[r] + bkoff[c0 + kk]] : 0.f;
      }
    }
    if (k0 >= kb) {
      const float* As = sm + buf * SA + 8 * ty;
      const float* Bs = sm + 2 * SA + buf * SB + tx;
#pragma unroll 4
      for (int kk = 0; kk < BK; ++kk) {
        float a[8], b[4];
        *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(As + kk * LA);
        *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(As + kk * LA + 4);
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = Bs[kk * LB + TX * j];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
      }
    }
    buf ^= 1;
    if (kn < ke) {
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        const int e = tid + NTH * i;
        const int r = g.a_kfast ? e / BK : e % BM, kk = g.a_kfast ? e % BK : e / BM;
        sm[buf * SA + kk * LA + r] = ra[i];
      }
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        const int e = tid + NTH * i;
        const int r = g.b_kfast ? e / BK : e % BN, kk = g.b_kfast ? e % BK : e / BN;
        sm[2 * SA + buf * SB + kk * LB + r] = rb[i];
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) sm[(8 * ty + i) * (BN + 1) + tx + TX * j] = acc[i][j];
  // output offsets of the tile's rows and columns, in the tables that are free now (split-K partials: dense [M][N])
#pragma unroll 1
  for (int t = tid; t < BM; t += NTH) {
    const int m = min(m0 + t, g.M - 1);
    arow[t] = ws ? (long long)m * g.N : g.cm(m);
    if (g.C2) akoff[t] = g.cm2(m);
  }
#pragma unroll 1
  for (int t = tid; t < BN; t += NTH) {
    const int n = min(n0 + t, g.N - 1);
    brow[t] = ws ? n : g.cn(n);
    if (g.C2) bkoff[t] = g.cn2(n);
  }
  __syncthreads();
  const int mh = min(BM, g.M - m0), nh = min(BN, g.N - n0);
  float* out = ws ? ws + (size_t)blockIdx.z * g.M * g.N : g.C;
  const float alpha = ws ? 1.f : g.alpha, beta = ws ? 0.f : g.beta;
  const bool by_rows = !ws && g.cn.s2 != 1 && g.cm.s2 == 1;  // neighbouring threads take neighbouring rows
#pragma unroll 4
  for (int e = tid; e < BM * BN; e += NTH) {
    const int ml = by_rows ? e % BM : e / BN, nl = by_rows ? e / BM : e % BN;
    if (ml < mh && nl < nh) {
      float v = alpha * sm[ml * (BN + 1) + nl];
      float* o = out + (arow[ml] + brow[nl]);
      if (beta != 0.f) v += beta * *o;
      *o = v;
    }
  }
  if (g.C2 && !ws) {
    const bool rows2 = g.cn2.s2 != 1 && g.cm2.s2 == 1;
#pragma unroll 4
    for (int e = tid; e < BM * BN; e += NTH) {
      const int ml = rows2 ? e % BM : e / BN, nl = rows2 ? e / BM : e % BN;
      if (ml < mh && nl < nh) g.C2[akoff[ml] + bkoff[nl]] = alpha * sm[ml * (BN + 1) + nl];
    }
  }
}

// Sum of the split-K partials into the output layouts. A block takes R rows of 32 columns: the partials are read
// along the columns, each output is written along its own fast direction, and the index maps are evaluated once
// a row and column of the tile (four maps and a 64-bit division an element took 20 us for 512 x 512 df32).
// R = 32 keeps four loads a thread in flight where one partial is all there is (32768 x 256 df32, the digit
// products: 66 us with 8 rows, 51 so); R = 8 spreads small outputs over the SMs (512 x 512, 32 partials: 11.7 us).
template <typename T, int R>
__global__ void __launch_bounds__(256) splitk_reduce_kernel(GemmArgs<T> g, const T* __restrict__ ws, int splits) {
  __shared__ T tile[R][33];
  __shared__ long long rm[R], rm2[R], cn[32], cn2[32];
  const int t = threadIdx.x;
  const long long total = (long long)g.M * g.N;
  const int nct = (g.N + 31) / 32, nrt = (g.M + R - 1) / R;
  for (long long b = blockIdx.x; b < (long long)nct * nrt; b += gridDim.x) {
    const int m0 = (int)(b / nct) * R, n0 = (int)(b % nct) * 32;
    if (t < 32) cn[t] = g.cn(min(n0 + t, g.N - 1));
    else if (t < 32 + R) rm[t - 32] = g.cm(min(m0 + t - 32, g.M - 1));
    else if (g.C2 && t >= 64 && t < 96) cn2[t - 64] = g.cn2(min(n0 + t - 64, g.N - 1));
    else if (g.C2 && t >= 96 && t < 96 + R) rm2[t - 96] = g.cm2(min(m0 + t - 96, g.M - 1));
    {
      const int i = t >> 5, j = t & 31;
      T s[R / 8];
      const T* w[R / 8];  // rows past the end read the last one, so that no test stands between the loads
#pragma unroll
      for (int k = 0; k < R / 8; ++k) {
        s[k] = T(0);
        w[k] = ws + (size_t)min(m0 + i + 8 * k, g.M - 1) * g.N + n0 + j;
      }
      if (n0 + j < g.N) {
#pragma unroll 4
        for (int z = 0; z < splits; ++z)
#pragma unroll
          for (int k = 0; k < R / 8; ++k) s[k] += w[k][(size_t)z * total];
      }
#pragma unroll
      for (int k = 0; k < R / 8; ++k) tile[i + 8 * k][j] = g.alpha * s[k];
    }
    __syncthreads();
    auto each = [&](bool along_rows, auto put) {  // along_rows: neighbouring threads take neighbouring rows
#pragma unroll
      for (int k = 0; k < R / 8; ++k) {
        const int i = along_rows ? t % R : (t >> 5) + 8 * k, j = along_rows ? t / R + 256 / R * k : t & 31;
        if (m0 + i < g.M && n0 + j < g.N) put(i, j);
      }
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
  const long long nct = (g.N + 31) / 32, tall = nct * ((g.M + 31) / 32);
  const bool big = tall >= 8LL * sm_count;  // the 32-row blocks fill the SMs: 2048 of them 19.3 us, with 8 rows 19.8
  const long long tiles = big ? tall : nct * ((g.M + 7) / 8);
  const int blocks = (int)(tiles < 1 ? 1 : tiles < (1 << 16) ? tiles : (1 << 16));
  ++tl_launches;
  if (big) splitk_reduce_kernel<T, 32><<<blocks, 256, 0, st>>>(g, ws, splits);
  else splitk_reduce_kernel<T, 8><<<blocks, 256, 0, st>>>(g, ws, splits);
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
    splitk_reduce_kernel<T, 8><<<256, 256, 0, st>>>(z, nullptr, 0);
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
