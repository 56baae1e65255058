// Exact per-site MPO product, the contraction step of the naive algorithm
// (Sec. 2.1, Alg. 1): C_l[(i_a i_b), s, t, (j_a j_b)] =
// sum_u A_l[i_a, s, u, j_a] B_l[i_b, u, t, j_b]. Exposed through the C ABI in
// include/ttfit.h; the compression that follows it in Alg. 1 is tt_mpo_compress.
#include <cuda_runtime.h>
#include <algorithm>
#include <vector>

#include "../../include/ttfit.h"
#include "common.cuh"

using namespace ttfit;

namespace {

// Output cores, row-major (a0 b0, s, t, a1 b1); the output is the dominant traffic (chi_A chi_B times the
// inputs), so the kernel is bound by writing it. A thread keeps its VW neighbouring columns (16 bytes where
// the rows allow it) and walks down the rows: the column's split into (j_a, j_b) is done once, and the entries
// of A and B come from L1. Narrow sites put several rows side by side in a block. All sites of a call go into
// one launch, so that short sites do not each leave a last wave and a gap behind.
// L = 8, chi 48 x 40, FP32 (354 MB, a call): one thread an element with 64-bit divisions took 748 us; so, with
// scalar loads of A and B for every column 218, with vector loads of B 156, and with each row's digits stepped on
// from the last row's, where four divisions a row were most of the instructions, 120 (C at 2.9 TB/s).
constexpr int NP_SITES = 32;  // sites of one launch (the table is a kernel parameter)
constexpr int NP_ROWS = 16;   // rows a thread walks down

template <typename F>
struct NaiveSite {
  const F *A, *B;
  F* C;
  int a0, a1, b0, b1, s, u, t;
  int cx;      // threads along the columns (a power of two <= 256), 256 / cx rows side by side
  long long ncol;  // column tiles
  int vec;     // 1: 16-byte stores, 2: 16-byte loads of B as well
  long long first;  // first block of the site
};
template <typename F>
struct NaiveTable {
  NaiveSite<F> site[NP_SITES];
  int n;
};

// BLOCK: b1 is a multiple of VW, so that the VW columns share j_a and their entries of B are one aligned vector.
template <typename F, int VW, bool BLOCK>
__device__ __forceinline__ void naive_tile(const NaiveSite<F>& S, long long tile) {
  const int cx = S.cx, ry = 256 / cx;
  const long long cols = (long long)S.a1 * S.b1, ct = tile % S.ncol, rt = tile / S.ncol;
  const long long col = (ct * cx + (long long)(threadIdx.x & (cx - 1))) * VW;
  if (col >= cols) return;
  int ja[VW], jb[VW];
#pragma unroll
  for (int v = 0; v < VW; ++v) ja[v] = (int)((col + v) / S.b1), jb[v] = (int)((col + v) - (long long)ja[v] * S.b1);
  const long long rows = (long long)S.a0 * S.b0 * S.s * S.t;
  long long row = rt * (NP_ROWS * ry) + threadIdx.x / cx;
  // the row's digits (i_a, i_b, s, t) come from divisions once; then the digits of ry are added with their carries
  unsigned tt, ss, ib, ia, dt = ry, ds, db, da;
  if (rows <= 0x7FFFFFFF) {
    unsigned r = (unsigned)row;
    tt = r % (unsigned)S.t, r /= (unsigned)S.t;
    ss = r % (unsigned)S.s, r /= (unsigned)S.s;
    ib = r % (unsigned)S.b0, ia = r / (unsigned)S.b0;
  } else {
    long long r = row;
    tt = (unsigned)(r % S.t), r /= S.t;
    ss = (unsigned)(r % S.s), r /= S.s;
    ib = (unsigned)(r % S.b0), ia = (unsigned)(r / S.b0);
  }
  ds = dt / (unsigned)S.t, dt %= (unsigned)S.t;
  db = ds / (unsigned)S.s, ds %= (unsigned)S.s;
  da = db / (unsigned)S.b0, db %= (unsigned)S.b0;
  auto carry = [](unsigned& x, unsigned n) {  // x < 2n on entry (n < 2^31)
    const unsigned c = x >= n;
    x -= c ? n : 0u;
    return c;
  };
#pragma unroll 2
  for (int i = 0; i < NP_ROWS && row < rows; ++i, row += ry) {
    const F* pa = S.A + ((long long)ia * S.s + ss) * S.u * S.a1;
    const F* pb = S.B + ((long long)ib * S.u * S.t + tt) * S.b1;
    F acc[VW];
#pragma unroll
    for (int v = 0; v < VW; ++v) acc[v] = F(0);
    for (int uu = 0; uu < S.u; ++uu) {
      if constexpr (BLOCK) {
        struct __align__(16) V {
          F e[VW];
        };
        const F x = pa[ja[0]];
        const V y = *reinterpret_cast<const V*>(pb + jb[0]);
#pragma unroll
        for (int v = 0; v < VW; ++v) acc[v] += x * y.e[v];
      } else {
#pragma unroll
        for (int v = 0; v < VW; ++v) acc[v] += pa[ja[v]] * pb[jb[v]];
      }
      pa += S.a1;
      pb += (long long)S.t * S.b1;
    }
    F* out = S.C + row * cols + col;
    if constexpr (VW == 1) out[0] = acc[0];
    else if constexpr (VW == 2) *reinterpret_cast<double2*>(out) = make_double2(acc[0], acc[1]);
    else *reinterpret_cast<float4*>(out) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    tt += dt;
    ss += ds + carry(tt, (unsigned)S.t);
    ib += db + carry(ss, (unsigned)S.s);
    ia += da + carry(ib, (unsigned)S.b0);
  }
}

template <typename F>
__global__ void __launch_bounds__(256) naive_product_kernel(const __grid_constant__ NaiveTable<F> T) {
  int k = 0;
  while (k + 1 < T.n && (long long)blockIdx.x >= T.site[k + 1].first) ++k;
  const NaiveSite<F>& S = T.site[k];
  if (S.vec == 2) naive_tile<F, 16 / (int)sizeof(F), true>(S, blockIdx.x - S.first);
  else if (S.vec) naive_tile<F, 16 / (int)sizeof(F), false>(S, blockIdx.x - S.first);
  else naive_tile<F, 1, false>(S, blockIdx.x - S.first);
}

template <typename F>
cudaError_t naive_product(const tt_mpo_desc* A, const tt_mpo_desc* B, const tt_mpo_desc* C, cudaStream_t st) {
  constexpr int VW = 16 / (int)sizeof(F);
  for (int l0 = 0; l0 < A->L; l0 += NP_SITES) {
    NaiveTable<F> T;
    T.n = std::min(NP_SITES, A->L - l0);
    long long blocks = 0;
    for (int k = 0; k < T.n; ++k) {
      const int l = l0 + k;
      NaiveSite<F>& S = T.site[k];
      S.A = (const F*)A->cores[l];
      S.B = (const F*)B->cores[l];
      S.C = (F*)C->cores[l];
      S.a0 = A->bond[l], S.a1 = A->bond[l + 1], S.b0 = B->bond[l], S.b1 = B->bond[l + 1];
      S.s = A->d_out[l], S.u = A->d_in[l], S.t = B->d_in[l];
      const long long cols = (long long)S.a1 * S.b1, rows = (long long)S.a0 * S.b0 * S.s * S.t;
      S.vec = cols % VW == 0 && ((uintptr_t)S.C & 15) == 0 ? 1 : 0;
      if (S.vec && S.b1 % VW == 0 && ((uintptr_t)S.B & 15) == 0) S.vec = 2;  // a row's entries of B are aligned too
      const long long wide = S.vec ? cols / VW : cols;
      S.cx = 1;
      while (S.cx < 256 && S.cx < wide) S.cx *= 2;
      S.ncol = (wide + S.cx - 1) / S.cx;
      S.first = blocks;
      const long long per = (long long)NP_ROWS * (256 / S.cx);
      blocks += S.ncol * ((rows + per - 1) / per);
    }
    ++tl_launches;
    naive_product_kernel<F><<<(unsigned)blocks, 256, 0, st>>>(T);  // a block writes 4096 values or more: far below 2^31
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

bool desc_ok(const tt_mpo_desc* X) {
  if (!X || X->L < 1 || !X->d_out || !X->d_in || !X->bond || !X->cores) return false;
  if (X->dtype != TT_DTYPE_F64 && X->dtype != TT_DTYPE_F32) return false;
  for (int l = 0; l < X->L; ++l)
    if (!X->cores[l] || X->d_out[l] < 1 || X->d_in[l] < 1 || X->bond[l] < 1) return false;
  return X->bond[X->L] >= 1;
}

}  // namespace

extern "C" tt_status tt_mpo_naive_product(const tt_mpo_desc* A, const tt_mpo_desc* B, const tt_mpo_desc* C,
                                          void* stream) {
  if (!desc_ok(A) || !desc_ok(B) || !desc_ok(C)) return TT_ERR_INVALID_ARGUMENT;
  if (A->dtype != B->dtype || A->dtype != C->dtype) return TT_ERR_INVALID_ARGUMENT;
  const int L = A->L;
  if (B->L != L || C->L != L) return TT_ERR_SHAPE_MISMATCH;
  if (A->bond[0] != 1 || A->bond[L] != 1 || B->bond[0] != 1 || B->bond[L] != 1) return TT_ERR_SHAPE_MISMATCH;
  for (int l = 0; l <= L; ++l)
    if ((long long)C->bond[l] != (long long)A->bond[l] * B->bond[l]) return TT_ERR_SHAPE_MISMATCH;
  for (int l = 0; l < L; ++l)
    if (A->d_in[l] != B->d_out[l] || C->d_out[l] != A->d_out[l] || C->d_in[l] != B->d_in[l])
      return TT_ERR_SHAPE_MISMATCH;
  cudaStream_t st = (cudaStream_t)stream;
  const cudaError_t e = A->dtype == TT_DTYPE_F64 ? naive_product<double>(A, B, C, st) : naive_product<float>(A, B, C, st);
  return e == cudaSuccess ? TT_OK : TT_ERR_CUDA;
}
