// Householder QR with the columns in registers (FP64 and double-FP32 arithmetic): the input
// preparation, the random guess and the FP64 factorisations.
#include <cooperative_groups.h>
#include <algorithm>
#include <type_traits>
#include "common.cuh"
#include "kernels.h"
#include "scalar_ops.cuh"

namespace cg = cooperative_groups;

namespace ttfit {

// Arithmetic of the register QR in its two types. null: the squared norm of a column without a reflector; finite: one
// that is neither infinite (an entry, or its square) nor NaN; safe: one that the reflector can be formed from as it is.
// field: the exponent field of an entry; shift: the power of two by which a column is scaled whose largest field is f
// and whose squared norm is not safe; scaled: x 2^s. lift: the power of two by which a column of X is scaled on
// loading, f the largest exponent field (FP64) of its entries.
template <typename C>
struct QrArith;

template <>
struct QrArith<df32> {
  static __device__ __forceinline__ df32 fma(df32 a, df32 b, df32 c) { return madd(a, b, c); }
  static __device__ __forceinline__ df32 sqrt(df32 x) { return qsqrt(x); }
  static __device__ __forceinline__ df32 rcp(df32 x) { return qrcp(x); }
  static __device__ __forceinline__ df32 abs(df32 x) { return x.hi < 0.0f ? -x : x; }
  static __device__ __forceinline__ bool neg(df32 x) { return x.hi < 0.0f; }
  static __device__ __forceinline__ bool null(df32 ss) { return ss.hi <= 0.0f; }
  static __device__ __forceinline__ bool finite(df32 ss) { return isfinite(ss.hi); }
  static constexpr bool RESCUES = true;
  static __device__ __forceinline__ int lift(int f, int) { return f == 0 || f == 0x7FF ? 0 : 1023 - f; }
  // the products' low words are exact to 2^-149: 1024 of them leave 2^-43 of the smallest norm taken as it is at worst
  static __device__ __forceinline__ bool safe(df32 ss) { return ss.hi >= 0x1p-96f && ss.hi <= 0x1p80f; }
  static __device__ __forceinline__ int field(df32 x) { return (__float_as_int(x.hi) >> 23) & 0xFF; }
  static __device__ __forceinline__ int shift(int f) { return f == 0 || f == 0xFF ? 0 : min(max(127 - f, -100), 100); }
  static __device__ __forceinline__ df32 scaled(df32 x, int s) {
    const float w = __int_as_float((127 + s) << 23);
    return df32(x.hi * w, x.lo * w);
  }
};

// FP64: the FP64 pipe takes 64 cycles for a warp instruction on this GPU, so square root and reciprocal
// start from FP32 estimates and take one third-order step; conversions and comparisons go by the bits.
template <>
struct QrArith<double> {
  static __device__ __forceinline__ double fma(double a, double b, double c) { return ::fma(a, b, c); }
  // x > 0 normal: mantissa m in [1, 4) and even exponent e with x = m 2^e
  static __device__ __forceinline__ double split_even(double x, int& e) {
    const int hi = __double2hiint(x);
    e = (((hi >> 20) & 0x7FF) - 1023) & ~1;
    return __hiloint2double(hi - (e << 20), __double2loint(x));
  }
  static __device__ __forceinline__ double times_pow2(double x, int e) {
    return __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x));
  }
  // leading bits of a double in [1, 4) as a float, and a float in (1/4, 4) as a double
  static __device__ __forceinline__ float lead(double x) {
    return __uint_as_float((((unsigned)__double2hiint(x) - (896u << 20)) << 3) | ((unsigned)__double2loint(x) >> 29));
  }
  static __device__ __forceinline__ double wide(float f) {
    const unsigned u = __float_as_uint(f);
    return __hiloint2double((int)((((u >> 23) + 896u) << 20) | ((u >> 3) & 0xFFFFFu)), (int)(u << 29));
  }
  // x r with r = 1/sqrt(x): r0 (1 + d/2 + 3 d^2/8), d = 1 - x r0^2 (|d| < 2^-20: the error is d^3)
  static __device__ __forceinline__ double sqrt(double x) {
    int e;
    const double m = split_even(x, e);
    const double r0 = wide(rsqrtf(lead(m)));
    const double d = ::fma(-m, r0 * r0, 1.0);
    return times_pow2(m * ::fma(r0 * d, ::fma(0.375, d, 0.5), r0), e >> 1);
  }
  // r0 (1 + d + d^2), d = 1 - x r0
  static __device__ __forceinline__ double rcp(double x) {
    int e;
    const double m = split_even(x, e);
    const double r0 = wide(__fdividef(1.f, lead(m)));
    const double d = ::fma(-m, r0, 1.0);
    return times_pow2(::fma(r0, ::fma(d, d, d), r0), -e);
  }
  static __device__ __forceinline__ double abs(double x) {
    return __hiloint2double(__double2hiint(x) & 0x7FFFFFFF, __double2loint(x));
  }
  static __device__ __forceinline__ bool neg(double x) { return __double2hiint(x) < 0; }
  static __device__ __forceinline__ bool null(double ss) { return (__double2hiint(ss) & 0x7FFFFFFF) <= 0x00100000; }
  static __device__ __forceinline__ bool finite(double ss) { return (__double2hiint(ss) & 0x7FFFFFFF) < 0x7FF00000; }
  // only columns below 2^-300, whose squares lose accuracy, and those above the field `top`
  static constexpr bool RESCUES = false;
  static __device__ __forceinline__ int lift(int f, int top) {
    return f == 0 || f == 0x7FF || (f > 723 && f <= top) ? 0 : 1023 - f;
  }
  static __device__ __forceinline__ bool safe(double) { return true; }
  static __device__ __forceinline__ int field(double) { return 0; }
  static __device__ __forceinline__ int shift(int) { return 0; }
  static __device__ __forceinline__ double scaled(double x, int) { return x; }
};

template <typename C>
struct __align__(16) Vec16 {
  static constexpr int N = 16 / (int)sizeof(C);
  C e[N];
};

template <typename C, int LP>
__device__ __forceinline__ C group_sum(C v, unsigned mask) {
#pragma unroll
  for (int o = LP / 2; o > 0; o >>= 1) {
    if constexpr (std::is_same<C, df32>::value)
      v = v + df32(__shfl_xor_sync(mask, v.hi, o), __shfl_xor_sync(mask, v.lo, o));
    else v += __shfl_xor_sync(mask, v, o);
  }
  return v;
}

// Householder QR with the columns in registers, on a cluster of NC CTAs. Column c lives in LP lanes of
// CTA c mod NC, RP vectors of 16 bytes a lane (vector l + LP t). Step j: the lanes of column j have put it
// into every CTA's shared memory (zeros above the diagonal); after one cluster barrier every column takes
// its dot product with it and |x_j|^2, forms the same reflector H = I - beta v v^T (v = x_j with
// v_j = x_jj - alpha, alpha = -sign(x_jj) |x_j|, beta = 1 / (|x_j|^2 + |x_jj| |x_j|)) and applies it
// (v^T a = x_j^T a - alpha a_j, so one pass of dot products serves norm and update). The reflectors go to
// X, from where the columns of Q, held the same way, take them back in reverse order without a barrier.
// A null column gives no reflector and R_jj = 0; one whose squared norm is not finite gives NaN.
// Where the squared norm is not safe, x_j is first brought near 1 by a power of two, which H does not depend on: in
// df32 |x_j| < 5e-20 made beta infinite and every later column NaN, and ordinary operators reach that (bond weights
// 2^-k, from k = 64 on). Every thread sees the same |x_j|^2. The loop stands twice, first without the scaling, up to
// the first column that needs it: in one loop, at the limit of registers, 512 x 128 df32 took 694 us instead of 628.
// The columns of X are each brought near 1 on loading, and those of R back, so that df32, whose exponents are FP32's,
// takes the range of FP64 (a site below 1e-45 came out null, one above 3e38 was refused); in FP64 the very small ones
// (below 1.5e-154, where the square is not a normal number, they came out null) and, for decompositions, very large.
//
// What bounds it is the chain of one step: the barrier (400 cycles), the dot products, two butterflies over
// LP lanes, root and reciprocal, the update. Finished rows are skipped.
template <typename S, typename C, int LP, int RP>
__global__ void __launch_bounds__(RP == 16 ? 256 : 512)
    qr_reg_kernel(int q, int p, int top, S* __restrict__ Xg, S* __restrict__ Qg, S* __restrict__ Rg) {
  using A = QrArith<C>;
  using V = Vec16<C>;
  constexpr int N = V::N;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), NC = (int)cl.num_blocks();
  const int r = min(q, p);
  extern __shared__ __align__(16) unsigned char qrs[];
  V* pub = (V*)qrs;                                 // [2][LP RP] the column of this step
  C* diag = (C*)(pub + 2 * LP * RP);                // [r] alpha
  C* beta = diag + r;                               // [r]
  C* Hg = (C*)Xg;                                   // the reflectors, in place of X (S and C: same size)
  static_assert(sizeof(S) == sizeof(C), "the reflectors take the place of X");
  const int grp = threadIdx.x / LP, l = threadIdx.x & (LP - 1);
  const int c = grp * NC + rank;                    // my column
  const C zero = C(0.0f), one = C(1.0f);
  V a[RP];
  C mine = zero;  // the reflector's entry on the diagonal
  // per column: the powers of two by which it was scaled on loading, and its rows from the diagonal on are to be
  __shared__ int lifts[64], ups[64];
  if (l == 0) ups[grp] = 0;
  {
    S x[RP][N];
    int f = 0;
#pragma unroll
    for (int t = 0; t < RP; ++t)
#pragma unroll
      for (int h = 0; h < N; ++h) {
        const int i = N * (l + LP * t) + h;
        x[t][h] = (c < p && i < q) ? Xg[(size_t)c * q + i] : S(0);
        f = max(f, (__double2hiint(x[t][h]) >> 20) & 0x7FF);
      }
#pragma unroll
    for (int o = LP / 2; o > 0; o >>= 1) f = max(f, __shfl_xor_sync(0xffffffffu, f, o));
    const int lift = A::lift(f, top);
    if (l == 0) lifts[grp] = lift;
#pragma unroll
    for (int t = 0; t < RP; ++t)
#pragma unroll
      for (int h = 0; h < N; ++h) a[t].e[h] = C(shift_bits(x[t][h], lift));
  }
  auto publish = [&](int j) {  // my column (j) to every CTA, zeros above row j
    V* dst = pub + (j & 1) * LP * RP + l;
#pragma unroll
    for (int t = 0; t < RP; ++t) {
      V v;
#pragma unroll
      for (int h = 0; h < N; ++h) v.e[h] = N * (l + LP * t) + h >= j ? a[t].e[h] : zero;
      for (int k = 0; k < NC; ++k) cl.map_shared_rank(dst, k)[LP * t] = v;
    }
  };
  cl.sync();  // every CTA runs
  if (c == 0) publish(0);
  cl.sync();
  // one step; without `rescue` it does nothing and returns false where the column has to be scaled first
  auto step = [&](auto rescue, int j) -> bool {
    V* xj = pub + (j & 1) * LP * RP;
    const int jv = j / N, jh = j % N, t0 = jv / LP, lj = jv & (LP - 1);  // row j: element jh of vector t0, lane lj
    V v[RP];
    C ss, dot, arow = zero;
    int k = 0;  // x_j was scaled by 2^k
    for (;;) {
      C d[2], s[2];
      d[0] = d[1] = s[0] = s[1] = zero;
#pragma unroll
      for (int t = 0; t < RP; ++t) {
        if (t >= t0) {
          v[t] = xj[l + LP * t];
#pragma unroll
          for (int h = 0; h < N; ++h) {
            d[h & 1] = A::fma(v[t].e[h], a[t].e[h], d[h & 1]);
            s[h & 1] = A::fma(v[t].e[h], v[t].e[h], s[h & 1]);
          }
        }
        if (t == t0) {
#pragma unroll
          for (int h = 0; h < N; ++h)
            if (h == jh) arow = a[t].e[h];
        }
      }
      ss = group_sum<C, LP>(s[0] + s[1], 0xffffffffu);
      dot = group_sum<C, LP>(d[0] + d[1], 0xffffffffu);
      if (A::safe(ss) || k != 0) break;  // the same in every thread
      if constexpr (!decltype(rescue)::value) return false;
      C* x = (C*)xj;
      int f = 0;
      for (int i = threadIdx.x & 31; i < N * LP * RP; i += 32) f = max(f, A::field(x[i]));
      k = A::shift(__reduce_max_sync(0xffffffffu, f));
      if (k == 0) break;
      __syncthreads();  // this CTA's copy has been read
      for (int i = threadIdx.x; i < N * LP * RP; i += blockDim.x) x[i] = A::scaled(x[i], k);
      __syncthreads();
    }
    arow = qshfl(arow, (threadIdx.x & 31 & ~(LP - 1)) + lj);
    const C x0 = xj[jv].e[jh];
    const bool live = !A::null(ss);
    C alpha = zero, be = zero;
    if (live) {
      const C nrm = A::sqrt(ss);
      alpha = A::neg(x0) ? nrm : -nrm;
      be = A::rcp(A::fma(A::abs(x0), nrm, ss));
    }
    if (!A::finite(ss)) alpha = be = C(__int_as_float(0x7FC00000));  // NaN, into R and Q: the caller's checks see it
    if (threadIdx.x == 0) diag[j] = alpha, beta[j] = be;
    if (c == j) {  // my rows above j are final, those below stay as the reflector
      mine = live ? x0 - alpha : zero;
      if (l == 0) ups[grp] = k;
    } else if (live && c > j && c < p) {
      const C v0 = x0 - alpha;
      const C w = -(be * A::fma(-alpha, arow, dot));
#pragma unroll
      for (int t = 0; t < RP; ++t)
        if (t >= t0) {
#pragma unroll
          for (int h = 0; h < N; ++h) {
            const C vi = (t == t0 && N * (l + LP * t) + h == j) ? v0 : v[t].e[h];
            a[t].e[h] = A::fma(w, vi, a[t].e[h]);
          }
        }
    }
    if (j + 1 < r && c == j + 1) publish(j + 1);
    cl.sync();
    return true;
  };
  int j = 0;
#pragma unroll 1
  while (j < r && step(std::false_type{}, j)) ++j;
  if constexpr (A::RESCUES) {
#pragma unroll 1
    for (; j < r; ++j) step(std::true_type{}, j);
  }
  // R (r x p, ld r) with diag >= 0, and the reflectors in place of X (not earlier: a barrier would wait
  // for stores to global memory at every step)
  if (c < p) {
    const int up = ups[grp], lift = lifts[grp];
    const bool dead = c < r && beta[c] == zero;  // a null column
#pragma unroll
    for (int t = 0; t < RP; ++t)
#pragma unroll
      for (int h = 0; h < N; ++h) {
        const int i = N * (l + LP * t) + h;
        if (c < r && i < q) Hg[(size_t)c * q + i] = i > c ? (dead ? zero : A::scaled(a[t].e[h], up)) : (i == c ? mine : zero);
        if (i >= r) continue;
        const C x = i > c ? zero : (i == c ? A::scaled(diag[c], -up) : a[t].e[h]);
        Rg[(size_t)c * r + i] = shift_bits(S(A::neg(diag[i]) ? -x : x), -lift);
      }
  }
  if (Qg != nullptr) {  // uniform
    __threadfence();
    cl.sync();
  }
  const unsigned mask = __ballot_sync(0xffffffffu, c < r);  // whole groups: c is uniform over a group's lanes
  if (Qg == nullptr || c >= r) return;                      // no barrier follows
  // Q = H_0 ... H_{r-1} [I; 0]: column c is touched by H_j, j <= c
#pragma unroll
  for (int t = 0; t < RP; ++t)
#pragma unroll
    for (int h = 0; h < N; ++h) a[t].e[h] = N * (l + LP * t) + h == c ? one : zero;
  const int jmax = __reduce_max_sync(mask, c);
  auto fetch = [&](int j, V (&v)[RP]) {  // written by other CTAs: not from L1
#pragma unroll
    for (int t = 0; t < RP; ++t)
#pragma unroll
      for (int h = 0; h < N; ++h) {
        const int i = N * (l + LP * t) + h;
        const C* x = Hg + (size_t)max(j, 0) * q + i;
        if constexpr (std::is_same<C, df32>::value) {
          const float2 u = (j >= 0 && i < q) ? __ldcg(reinterpret_cast<const float2*>(x)) : make_float2(0.f, 0.f);
          v[t].e[h] = df32(u.x, u.y);
        } else {
          v[t].e[h] = (j >= 0 && i < q) ? __ldcg(x) : zero;
        }
      }
  };
  V vn[RP];
  fetch(jmax, vn);
  for (int j = jmax; j >= 0; --j) {
    V v[RP];
#pragma unroll
    for (int t = 0; t < RP; ++t) v[t] = vn[t];
    fetch(j - 1, vn);  // the next reflector's loads run under this one's arithmetic
    const int t0 = (j / N) / LP;
    C d[2];
    d[0] = d[1] = zero;
#pragma unroll
    for (int t = 0; t < RP; ++t)
      if (t >= t0) {
#pragma unroll
        for (int h = 0; h < N; ++h) d[h & 1] = A::fma(v[t].e[h], a[t].e[h], d[h & 1]);
      }
    const C dot = group_sum<C, LP>(d[0] + d[1], mask);
    const C w = c >= j ? -(beta[j] * dot) : zero;
#pragma unroll
    for (int t = 0; t < RP; ++t)
      if (t >= t0) {
#pragma unroll
        for (int h = 0; h < N; ++h) a[t].e[h] = A::fma(w, v[t].e[h], a[t].e[h]);
      }
  }
  const bool flip = A::neg(diag[c]);
#pragma unroll
  for (int t = 0; t < RP; ++t)
#pragma unroll
    for (int h = 0; h < N; ++h) {
      const int i = N * (l + LP * t) + h;
      if (i < q) Qg[(size_t)c * q + i] = S(flip ? -a[t].e[h] : a[t].e[h]);
    }
}

template <typename S, typename C>
cudaError_t qr_reg_launch(int nc, int lp, int q, int p, int top, S* X, S* Q, S* R, cudaStream_t st) {
  constexpr int N = Vec16<C>::N;
  const int threads = ((p + nc - 1) / nc * lp + 31) / 32 * 32;
  const int rp = q <= 4 * N * lp ? 4 : q <= 8 * N * lp ? 8 : 16;
  if (threads > (rp == 16 ? 256 : 512) || q > 16 * N * lp) return cudaErrorNotSupported;
  if (lp < 32 && rp != 4) return cudaErrorNotSupported;  // the callers take 32 lanes for such columns
  const size_t sm = (size_t)2 * lp * rp * 16 + 2 * (size_t)std::min(q, p) * sizeof(C);  // 20 KB at most
  auto launch = [&](auto kern) -> cudaError_t {
    cudaError_t e;
    if (nc > 8 &&
        (e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
      return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nc);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = nc;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (nc > 8) {  // a 16-CTA cluster must fit in one GPC: check it can be placed
      int nclu = 0;
      if (cudaOccupancyMaxActiveClusters(&nclu, kern, &cfg) != cudaSuccess || nclu < 1) {
        cudaGetLastError();
        return cudaErrorNotSupported;
      }
    }
    ++tl_launches;
    e = cudaLaunchKernelEx(&cfg, kern, q, p, top, X, Q, R);
    return e != cudaSuccess ? e : cudaGetLastError();
  };
  if constexpr (std::is_same<C, double>::value)
    if (lp == 8) return launch(qr_reg_kernel<S, C, 8, 4>);
  if (lp == 16) return launch(qr_reg_kernel<S, C, 16, 4>);
  return rp == 4 ? launch(qr_reg_kernel<S, C, 32, 4>) : rp == 8 ? launch(qr_reg_kernel<S, C, 32, 8>) : launch(qr_reg_kernel<S, C, 32, 16>);
}

// FP64. CTAs and lanes a column by the measured times (us, with Q; the blocked cluster kernel or, for the
// rows marked *, the one-CTA kernel takes): 64 x 20 *298: 4 CTAs of 8 lanes 72; 64 x 64 *1203: 8 x 8 209;
// 100 x 37 *620: 8 x 16 138; 128 x 128 1397: 8 x 16 630; 256 x 74 934: 8 x 16 444, 16 x 32 328;
// 512 x 128 2312: 8 x 16 1825, 16 x 32 1095.
cudaError_t qr_reg64(int q, int p, double* X, double* Q, double* R, cudaStream_t st, bool any_scale) {
  const int top = any_scale ? 1023 + 300 : 0x7FE;
  const int lp = q <= 64 ? 8 : q <= 128 ? 16 : 32;
  if (q > 128 && p > 32) {
    const cudaError_t e = qr_reg_launch<double, double>(16, lp, q, p, top, X, Q, R, st);
    if (e != cudaErrorNotSupported) return e;
  }
  return qr_reg_launch<double, double>(p <= 32 ? 4 : 8, lp, q, p, top, X, Q, R, st);
}

// Double-FP32 arithmetic on FP64 storage. 128 x 128: 888 us by the blocked kernel, 284 here (8 CTAs of
// 16 lanes); 256 x 64: 420, 165 (8 x 32); 512 x 128: 1199, 628 (8 x 32). Clusters of 16 take 578 for the
// last, but two chains and the random guess prepare at once, and 8 leave them room.
cudaError_t qr_reg_df32(int q, int p, double* X, double* Q, double* R, cudaStream_t st) {
  return qr_reg_launch<double, df32>(8, q <= 128 ? 16 : 32, q, p, 0, X, Q, R, st);
}

}  // namespace ttfit
