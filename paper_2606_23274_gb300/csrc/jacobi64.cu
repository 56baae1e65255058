// One-sided Jacobi SVD in FP64 for this GPU's slow FP64 pipe (Sec. 2.3.4's
// factorisation in the FP64 precision, tt_svd_truncated, the zip-up).
#include <cooperative_groups.h>
#include <algorithm>
#include <cfloat>
#include "common.cuh"
#include "kernels.h"
#include "scalar_ops.cuh"

namespace cg = cooperative_groups;

namespace ttfit {

// ---------------------------------------------------------------------------
// One-sided Jacobi in FP64 (cluster of 1, 8 or 16 CTAs), organised around the
// FP64 pipe: a warp-wide FP64 instruction occupies its SM quadrant for 64 cycles
// whatever number of lanes is active (measured; an SM issues one per 17 cycles),
// so what counts is the number of warp instructions, not of operations.
//  * A column pair is worked by LP lanes, and a warp holds 32 / LP pairs: the
//    butterfly of the dot product and the rotation angle, which every lane of a
//    pair computes, cost 1 / (32 / LP) of a warp instruction per pair.
//  * |x|^2 and |y|^2 are carried along (a - t g, b + t g) and recomputed at the
//    start of every sweep, so that a pair takes one dot product instead of three.
//  * The tangent t is formed in FP32 from the leading bits of g and b - a: a
//    slightly wrong angle leaves the pair at 1e-6 of its cosine and the next sweep
//    takes the rest. Only cos and sin have to be exact to FP64 (they keep the
//    rotation orthogonal): one third-order step from the FP32 reciprocal root.
//  * The rotations are applied in scaled form (Gentleman, J. Inst. Math. Appl. 12
//    (1973)): with x = dx x~, y = dy y~ a rotation is x~ -= (t dy / dx) y~,
//    y~ += (t dx / dy) x~, two multiply-adds a row instead of four operations; the
//    scales take the factor cos and are multiplied in once a sweep.
//  * A very large or small W is brought to exponent 0 by a power of two while it lies in shared memory, and S
//    back: squared norms and products of two of them must neither overflow nor vanish (from entries of 1e77 and
//    1e-77 on no pair rotated any more, and the norms of the columns were returned as singular values).
// ---------------------------------------------------------------------------
struct Rot64 {
  double t, cs, s;  // tangent, cosine, 1 + t^2
};

// double of a finite float, by its bits (a conversion would take the FP64 pipe)
__device__ __forceinline__ double widen_bits(float f, int shift) {
  const unsigned u = __float_as_uint(f);
  const unsigned hi = (u & 0x80000000u) | ((((u >> 23) & 0xFFu) + 896u + (unsigned)shift) << 20) | ((u >> 3) & 0xFFFFFu);
  return __hiloint2double((int)hi, (int)(u << 29));
}

// Rotation that zeroes the (x, y) entry g of [[a, g], [g, b]], d = b - a; g != 0.
__device__ __forceinline__ Rot64 rotation64(double g, double d) {
  const unsigned gh = (unsigned)__double2hiint(g), dh = (unsigned)__double2hiint(d);
  // mantissas in [1, 2) and the exponent of zeta = d / (2 g)
  const float mg = __uint_as_float(0x3F800000u | ((gh & 0xFFFFFu) << 3) | ((unsigned)__double2loint(g) >> 29));
  const float md = __uint_as_float(0x3F800000u | ((dh & 0xFFFFFu) << 3) | ((unsigned)__double2loint(d) >> 29));
  const int k = (int)((dh >> 20) & 0x7FFu) - (int)((gh >> 20) & 0x7FFu) - 1;
  const unsigned sign = (d != 0.0 ? (gh ^ dh) : 0u) & 0x80000000u;
  float tm;
  int sh = 0;
  if (k > 60) {  // |zeta| > 2^60: t = 1 / (2 zeta) = (mg / md) 2^(-k-1)
    tm = __fdividef(mg, md);
    sh = max(-k - 1, -1000);
  } else {
    const float zeta = __fdividef(md, mg) * __uint_as_float((unsigned)(max(k, -60) + 127) << 23);
    tm = __fdividef(1.f, zeta + sqrtf(fmaf(zeta, zeta, 1.f)));
  }
  Rot64 r;
  r.t = widen_bits(__uint_as_float(__float_as_uint(tm) | sign), sh);
  const double s = fma(r.t, r.t, 1.0);  // in [1, 2 + 1e-6]
  const float sf = __uint_as_float((((unsigned)__double2hiint(s) - (896u << 20)) << 3) |
                                   ((unsigned)__double2loint(s) >> 29));
  const double r0 = widen_bits(rsqrtf(sf), 0);
  const double e = fma(-s, r0 * r0, 1.0);
  r.cs = fma(r0 * e, fma(0.375, e, 0.5), r0);  // r0 (1 + e/2 + 3 e^2/8): error e^3 ~ 2^-63
  r.s = s;
  return r;
}

// sum over the LP lanes of a pair
template <int LP>
__device__ __forceinline__ double lanes_sum(double v) {
#pragma unroll
  for (int o = LP / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Trailer of a column (after its rows): |w|^2, scale, 1 / scale, unused.
constexpr int J64_TAIL = 4;

// One pair: columns xi, xj of ld doubles, nq (nr) double2 of rows in the dot product (in all). Every
// lane of the warp calls it; act is uniform over the lanes of a pair.
template <int LP, bool SCALED>
__device__ __forceinline__ bool jacobi64_pair(double* __restrict__ xi, double* __restrict__ xj, int nq, int nr, int ld,
                                              double tol2, bool act) {
  const int l = threadIdx.x & (LP - 1);
  double2* x2 = reinterpret_cast<double2*>(xi);
  double2* y2 = reinterpret_cast<double2*>(xj);
  double g = 0.0, g1 = 0.0;
  if (act) {
#pragma unroll 2
    for (int r = l; r < nq; r += LP) {
      const double2 x = x2[r], y = y2[r];
      g = fma(x.x, y.x, g);
      g1 = fma(x.y, y.y, g1);
    }
  }
  g = lanes_sum<LP>(g + g1);
  double a = 0.0, b = 0.0, di = 1.0, dj = 1.0, ii = 1.0, ij = 1.0;
  if (act) {
    a = xi[ld - 4], b = xj[ld - 4];
    if (SCALED) di = xi[ld - 3], ii = xi[ld - 2], dj = xj[ld - 3], ij = xj[ld - 2];
  }
  if (SCALED) g *= di * dj;
  const long long lhs = __double_as_longlong(g * g), rhs = __double_as_longlong(tol2 * a * b);
  // positive doubles order as their bits; the comparisons stay off the FP64 pipe
  const bool rot = act && __double2hiint(a) > 0 && __double2hiint(b) > 0 && lhs > rhs && lhs < 0x7FF0000000000000ll;
  __syncwarp();  // every lane of the pair has read the trailers
  if (rot) {
    const Rot64 R = rotation64(g, b - a);
    if (SCALED) {
      const double al = -R.t * (dj * ii), be = R.t * (di * ij);
#pragma unroll 4
      for (int r = l; r < nr; r += LP) {
        const double2 x = x2[r], y = y2[r];
        x2[r] = make_double2(fma(al, y.x, x.x), fma(al, y.y, x.y));
        y2[r] = make_double2(fma(be, x.x, y.x), fma(be, x.y, y.y));
      }
      const double sec = R.s * R.cs, ci = di * R.cs, cj = dj * R.cs;
      double si = ii * sec, sj = ij * sec;
      si = fma(si, fma(-ci, si, 1.0), si);  // keeps scale times its inverse at 1 to the last place
      sj = fma(sj, fma(-cj, sj, 1.0), sj);
      if (l == 0) xi[ld - 3] = ci, xi[ld - 2] = si, xj[ld - 3] = cj, xj[ld - 2] = sj;
    } else {
      const double sn = R.cs * R.t;
#pragma unroll 4
      for (int r = l; r < nr; r += LP) {
        const double2 x = x2[r], y = y2[r];
        x2[r] = make_double2(fma(-sn, y.x, R.cs * x.x), fma(-sn, y.y, R.cs * x.y));
        y2[r] = make_double2(fma(R.cs, y.x, sn * x.x), fma(R.cs, y.y, sn * x.y));
      }
    }
    if (l == 0) xi[ld - 4] = fma(-R.t, g, a), xj[ld - 4] = fma(R.t, g, b);
  }
  return rot;
}

__host__ __device__ inline int jacobi64_ld(int q, int p, bool want_v) {
  return (q + 1) / 2 * 2 + (want_v ? (p + 1) / 2 * 2 : 0) + J64_TAIL;
}

template <int LP, bool SCALED>
__global__ void __launch_bounds__(1024)
    jacobi64_kernel(int q, int p, int b, const double* Win, const double* Vin, int max_sweeps, double tol,
                    uint32_t* errw, double* Uo, double* __restrict__ So, double* Vo) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), NC = (int)cl.num_blocks();
  const int P = 2 * NC;
  const bool want_v = Vo != nullptr;
  const int qs = (q + 1) / 2 * 2;
  const int ld = jacobi64_ld(q, p, want_v);
  const int nq = qs / 2, nr = (ld - J64_TAIL) / 2;
  const int nbuf = NC > 1 ? 2 : 1;
  extern __shared__ __align__(16) unsigned char j64s[];
  double* buf = (double*)j64s;                                // [nbuf][2 slots][b][ld]
  int* ids = (int*)(buf + (size_t)nbuf * 2 * b * ld);         // [nbuf][2 slots][b] global column or -1
  double* nrm = (double*)(ids + 4 * b + 4);                   // [2 slots][b] final column norms
  __shared__ int flag[2], top;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  constexpr int G = 32 / LP;
  const int grp = warp * G + lane / LP, ng = nw * G, l = lane & (LP - 1);
  auto col = [&](int bi, int sl, int k) { return buf + ((size_t)(bi * 2 + sl) * b + k) * ld; };
  auto cid = [&](int bi, int sl, int k) -> int& { return ids[(bi * 2 + sl) * b + k]; };
  const double tol2 = tol * tol;

  if (threadIdx.x == 0) top = 0;
  __syncthreads();
  int field = 0;  // largest exponent field of my entries of W
  for (int sl = 0; sl < 2; ++sl) {  // CTA c holds the blocks at positions c and P-1-c
    const int blk = sl == 0 ? rank : P - 1 - rank;
    for (int k = 0; k < b; ++k) {
      const int gid = blk * b + k;
      if (threadIdx.x == 0) cid(0, sl, k) = gid < p ? gid : -1;
      double* x = col(0, sl, k);
      for (int r = threadIdx.x; r < ld; r += blockDim.x) {
        double v = 0.0;
        if (r == ld - 3 || r == ld - 2) v = 1.0;
        else if (gid < p && r < q) {
          v = Win[(size_t)gid * q + r];
          field = max(field, (__double2hiint(v) >> 20) & 0x7FF);
        } else if (gid < p && r >= qs && r - qs < p && r < ld - J64_TAIL)
          v = Vin ? Vin[(size_t)gid * p + r - qs] : (r - qs == gid ? 1.0 : 0.0);
        x[r] = v;
      }
    }
  }
  if (threadIdx.x < 2) flag[threadIdx.x] = 0;
  field = __reduce_max_sync(0xffffffffu, field);
  if (lane == 0) atomicMax(&top, field);
  cl.sync();
  field = __reduce_max_sync(0xffffffffu, lane < NC ? *cl.map_shared_rank(&top, lane) : 0);
  // not where an entry is not finite, and not within 2^-64 .. 2^64, where it changes nothing
  const int shift = field == 0 || field == 0x7FF || abs(field - 1023) <= 64 ? 0 : 1023 - field;
  if (shift != 0) {
    for (int sl = 0; sl < 2; ++sl)
      for (int k = 0; k < b; ++k) {
        double* x = col(0, sl, k);
        for (int r = threadIdx.x; r < q; r += blockDim.x) x[r] = shift_bits(x[r], shift);
      }
    __syncthreads();
  }

  int cur = 0, sweep = 0;
  // multiply the scales into the columns and recompute |w|^2
  auto refresh = [&]() {
    for (int w0 = 0; w0 < 2 * b; w0 += ng) {
      const int w = w0 + grp;
      double s = 0.0;
      double* x = col(cur, w < b ? 0 : 1, w < 2 * b ? w % b : 0);
      if (w < 2 * b) {
        const double d = x[ld - 3];
        double2* x2 = reinterpret_cast<double2*>(x);
        for (int r = l; r < nr; r += LP) {
          double2 v = x2[r];
          if (d != 1.0) x2[r] = v = make_double2(v.x * d, v.y * d);
          if (r < nq) s = fma(v.x, v.x, fma(v.y, v.y, s));
        }
      }
      s = lanes_sum<LP>(s);
      __syncwarp();  // every lane has read the scale
      if (w < 2 * b && l == 0) x[ld - 4] = s, x[ld - 3] = 1.0, x[ld - 2] = 1.0;
    }
    __syncthreads();
  };
  bool done = false;
  while (!done && sweep < max_sweeps) {
    bool rot = false;
    refresh();
    for (int sr = 0; sr < P - 1; ++sr) {
      if (sr == 0) {  // pairs inside each block (round robin over the b columns of both slots)
        const int B = b + (b & 1), half = B / 2;
        for (int mr = 0; mr < B - 1; ++mr) {
          const int sl = grp / half, k = grp % half;
          int i = b, j = b;
          if (grp < 2 * half) rr_pair(mr, k, B, i, j);
          const bool act = i < b && j < b;
          rot |= jacobi64_pair<LP, SCALED>(col(cur, act ? sl : 0, act ? i : 0), col(cur, act ? sl : 0, act ? j : 0), nq, nr, ld,
                                   tol2, act);
          __syncthreads();
        }
      }
      {  // pairs between the two blocks: group w keeps column w of slot 0 and meets column (w + mr) mod b of slot 1
        const bool act = grp < b;
        double* xi = col(cur, 0, act ? grp : 0);
        int j = act ? grp : 0;
        for (int mr = 0; mr < b; ++mr) {
          rot |= jacobi64_pair<LP, SCALED>(xi, col(cur, 1, j), nq, nr, ld, tol2, act);
          j = (j + 1 == b) ? 0 : j + 1;
          __syncthreads();
        }
      }
      if (NC == 1) break;  // two blocks: one super-round
      // rotate the positions 1..P-1 by one (position 0 stays): pull the next two blocks
      cl.sync();
      const int nb = cur ^ 1;
#pragma unroll
      for (int sl = 0; sl < 2; ++sl) {
        const int x = sl == 0 ? rank : P - 1 - rank;
        const int src = x == 0 ? 0 : (x == 1 ? P - 1 : x - 1);
        const int scta = src < NC ? src : P - 1 - src, ssl = src < NC ? 0 : 1;
        const uint4* rsrc = reinterpret_cast<const uint4*>(cl.map_shared_rank(col(cur, ssl, 0), scta));
        const int* rid = cl.map_shared_rank(&cid(cur, ssl, 0), scta);
        uint4* dst = reinterpret_cast<uint4*>(col(nb, sl, 0));
        const int n16 = b * ld / 2;
#pragma unroll 4
        for (int e = threadIdx.x; e < n16; e += blockDim.x) dst[e] = rsrc[e];
        if (threadIdx.x < b) cid(nb, sl, threadIdx.x) = rid[threadIdx.x];
      }
      cur = nb;
      __syncthreads();
    }
    // the cluster-wide "any rotation" of this sweep decides, identically in every CTA
    const int any = __syncthreads_or(rot ? 1 : 0);
    int* f0 = cl.map_shared_rank(&flag[sweep & 1], 0);
    if (any && threadIdx.x == 0) atomicOr(f0, 1);
    cl.sync();
    done = (*f0 == 0);
    if (rank == 0 && threadIdx.x == 0) flag[(sweep + 1) & 1] = 0;  // next sweep's flag (last read a sweep ago)
    ++sweep;
    cl.sync();
  }
  if (!done && rank == 0 && threadIdx.x == 0 && errw) atomicOr(errw, ERRW_NOCONV);
  if (rank == 0 && threadIdx.x == 0 && errw) atomicMax((int*)errw + 1, sweep);
  refresh();
  for (int w = threadIdx.x; w < 2 * b; w += blockDim.x) {
    const int sl = w / b, k = w % b;
    double v = cid(cur, sl, k) >= 0 ? sqrt(col(cur, sl, k)[ld - 4]) : -1.0;
    if (!(v <= DBL_MAX)) {  // reported; and NaN would have no place in the order, so that outputs stayed unwritten
      v = __longlong_as_double(0x7FF0000000000000ll);
      if (errw) atomicOr(errw, ERRW_NAN);
    }
    nrm[w] = v;
  }
  cl.sync();
  for (int w = warp; w < 2 * b; w += nw) {  // every column's rank among all p (descending, ties by column index)
    const int sl = w / b, k = w % b;
    const int me = cid(cur, sl, k);
    if (me < 0) continue;
    const double v = nrm[w];
    int rk = 0;
    for (int c = 0; c < NC; ++c) {
      const double* rn = cl.map_shared_rank(nrm, c);
      const int* ri = cl.map_shared_rank(&cid(cur, 0, 0), c);
      for (int t = lane; t < 2 * b; t += 32) {
        const int o = ri[t];  // ids of slot 0 then slot 1 are contiguous
        const double u = rn[t];
        rk += (o >= 0) && (u > v || (u == v && o < me));
      }
    }
    rk = warp_sum(rk);
    const double* x = col(cur, sl, k);
    const double inv = v > 0.0 ? 1.0 / v : 0.0;
    for (int r = lane; r < q; r += 32) Uo[(size_t)rk * q + r] = x[r] * inv;
    if (want_v)
      for (int r = lane; r < p; r += 32) Vo[(size_t)rk * p + r] = x[qs + r];
    if (lane == 0) So[rk] = scalbn(v, -shift);
  }
  cl.sync();  // no CTA leaves while another may still read its shared memory
}

inline size_t jacobi64_smem(int q, int p, bool want_v, int nc) {
  const size_t b = (p + 2 * nc - 1) / (2 * nc), nbuf = nc > 1 ? 2 : 1;
  return nbuf * 2 * b * jacobi64_ld(q, p, want_v) * sizeof(double) + (4 * b + 4) * sizeof(int) + 2 * b * sizeof(double) + 16;
}

// Singular value decomposition of the q x p column-major W (q >= p) as jacobi_svd
// gives it. cudaErrorNotSupported when the columns do not fit into the shared
// memory of a cluster (the caller then takes the one-CTA kernel on global memory).
//
// CTAs: one up to 23 columns, 8 up to 95, 16 above, where they are the fastest
// (measured, us for a decomposition of G1 D G2 with a spectrum of 1 .. 1e-4;
// one CTA / 4 / 8 / 16): 24 x 16: 297 / 311 / 388 / 813; 40 x 31: 1235 / 888 / 766 / 1026;
// 104 x 48: 4125 / 2011 / 1722 / 2405; 203 x 101: - / 14478 / 10267 / 8694;
// 128 x 128: - / 17161 / 11309 / 7950. A larger cluster is taken where the columns need its shared
// memory, a smaller one where 16 CTAs cannot be placed. Lanes per pair: 16 in one CTA (8 to 11 pairs,
// one or two warps on each quadrant), 32 in a cluster, whose CTAs hold few pairs. The scaled rotations
// pay from 300 rows on (256 x 74: 5.3 ms against 5.6 ms; 128 x 128: 8.2 against 7.9).
namespace {

using Jacobi64Kernel = void (*)(int, int, int, const double*, const double*, int, double, uint32_t*, double*, double*,
                                double*);

struct Jacobi64Plan {
  Jacobi64Kernel kern = nullptr;  // null: does not fit
  int nc = 0, b = 0;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
};

// The kernel and its launch for a q x p decomposition (plan.cfg points into plan: not to be copied).
cudaError_t jacobi64_plan(int q, int p, bool want_v, cudaStream_t st, Jacobi64Plan& plan) {
  const bool scaled = q + (want_v ? p : 0) > 300;
  const int order[3][3] = {{1, 8, 16}, {8, 16, 0}, {16, 8, 0}};
  for (const int nc : order[p < 24 ? 0 : p < 96 ? 1 : 2]) {
    if (nc == 0) continue;
    const size_t sm = jacobi64_smem(q, p, want_v, nc);
    const int b = (p + 2 * nc - 1) / (2 * nc), B = b + (b & 1);
    const int lp = nc == 1 ? 16 : 32;
    const int threads = std::max(128, 32 * ((B * lp + 31) / 32));
    if (sm > 220 * 1024 || threads > 1024) continue;
    Jacobi64Kernel kern = nc == 1 ? (scaled ? jacobi64_kernel<16, true> : jacobi64_kernel<16, false>)
                                  : (scaled ? jacobi64_kernel<32, true> : jacobi64_kernel<32, false>);
    cudaError_t e = ensure_smem((const void*)kern, sm);
    if (e != cudaSuccess) return e;
    if (nc > 8 && (e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
      return e;
    plan.cfg.gridDim = dim3(nc);
    plan.cfg.blockDim = dim3(threads);
    plan.cfg.dynamicSmemBytes = sm;
    plan.cfg.stream = st;
    plan.at[0].id = cudaLaunchAttributeClusterDimension;
    plan.at[0].val.clusterDim.x = nc;
    plan.at[0].val.clusterDim.y = 1;
    plan.at[0].val.clusterDim.z = 1;
    plan.cfg.attrs = plan.at;
    plan.cfg.numAttrs = 1;
    if (nc > 8) {  // a 16-CTA cluster must fit in one GPC: check it can be placed
      int nclu = 0;
      if (cudaOccupancyMaxActiveClusters(&nclu, kern, &plan.cfg) != cudaSuccess || nclu < 1) {
        cudaGetLastError();
        continue;
      }
    }
    plan.kern = kern;
    plan.nc = nc;
    plan.b = b;
    return cudaSuccess;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t jacobi_svd64(int q, int p, const double* W, const double* Vin, double* U, double* Sv, double* V,
                         int max_sweeps, uint32_t* errw, cudaStream_t st) {
  const double tol = 4.0 * DBL_EPSILON * sqrt((double)q);  // as in jacobi_svd
  Jacobi64Plan plan;
  cudaError_t e = jacobi64_plan(q, p, V != nullptr, st, plan);
  if (e != cudaSuccess) return e;
  if (!plan.kern) return cudaErrorNotSupported;
  ++tl_launches;
  e = cudaLaunchKernelEx(&plan.cfg, plan.kern, q, p, plan.b, W, Vin, max_sweeps, tol, errw, U, Sv, V);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// SVD of a p x p matrix with graded columns, L = U diag(S) W^T.
// The first sweeps, eight at most, run in FP32, where they cost a quarter: an FP32 Jacobi of L gives rotations W0, made
// orthonormal to FP64 rounding by two Newton-Schulz steps, and the FP64 Jacobi of L W0 needs 3 or 4 sweeps for its own
// stopping rule instead of 10 (spectra down to 1e-18 s_1: the columns are graded, so FP32 keeps each to its own
// rounding). The result is as accurate as without: every rotation that counts is taken in FP64.
// U must not be L; e0, e1: p x p scratch each, or null (no room: all sweeps in FP64).
// 128 x 128 in an FP64 fit: 3.3 ms by FP64 sweeps alone; so 0.6 ms of FP32 sweeps, 0.9 ms of FP64 ones and six
// products of 10 us. 256 x 256: 13 ms; 1.9, 4.0 and 0.3.
cudaError_t svd_graded64(int p, const double* L, double* U, double* Sv, double* W, double* e0, double* e1, int max_sweeps,
                         uint32_t* errw, int sm_count, cudaStream_t st) {
  Jacobi64Plan plan;
  cudaError_t e = jacobi64_plan(p, p, true, st, plan);
  if (e != cudaSuccess) return e;
  if (!plan.kern) return cudaErrorNotSupported;
  if (p < 32 || !e0 || !e1 || !jacobi32_rotations_fits(p))
    return jacobi_svd64(p, p, L, nullptr, U, Sv, W, max_sweeps, errw, st);
  const long long n = (long long)p * p;
  double* t = U;  // scratch until the decomposition writes it
  float *L32 = (float*)t, *V32 = L32 + n;
  int* ex = (int*)Sv;  // free until the decomposition writes it
  if ((e = absmax_exponent<double>(L, n, ex, st)) != cudaSuccess) return e;
  if ((e = copy_pow2<double, float>(n, L, L32, ex, st)) != cudaSuccess) return e;
  if ((e = jacobi32_rotations(p, L32, V32, 8, st)) != cudaSuccess) return e;
  const IdxMap one = IdxMap::lin(1), row = IdxMap::lin(p), zero = IdxMap::lin(0);
  if ((e = copy_map<float, double>(1, (int)n, V32, zero, one, W, zero, one, 1.0, st)) != cudaSuccess) return e;
  double *X = W, *Xn = e1;
  for (int it = 0; it < 2; ++it) {  // X <- X (3 I - X^T X) / 2
    GemmArgs<double> g;
    g.M = g.N = g.K = p;
    g.A = X; g.am = row; g.ak = one;
    g.B = X; g.bn = row; g.bk = one;
    g.C = e0; g.cm = one; g.cn = row;
    if ((e = gemm_simt<double>(g, nullptr, 0, sm_count, st)) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(Xn, X, sizeof(double) * n, cudaMemcpyDeviceToDevice, st)) != cudaSuccess) return e;
    GemmArgs<double> a;
    a.M = a.N = a.K = p;
    a.A = X; a.am = one; a.ak = row; a.a_kfast = false;
    a.B = e0; a.bn = row; a.bk = one;
    a.C = Xn; a.cm = one; a.cn = row;
    a.alpha = -0.5;
    a.beta = 1.5;
    if ((e = gemm_simt<double>(a, nullptr, 0, sm_count, st)) != cudaSuccess) return e;
    std::swap(X, Xn);
  }
  GemmArgs<double> g;  // t = L W0 (W0 is back in W)
  g.M = g.N = g.K = p;
  g.A = L; g.am = one; g.ak = row; g.a_kfast = false;
  g.B = W; g.bn = row; g.bk = one;
  g.C = t; g.cm = one; g.cn = row;
  if ((e = gemm_simt<double>(g, nullptr, 0, sm_count, st)) != cudaSuccess) return e;
  // outputs may take the inputs' place: the kernel reads both before its first barrier and writes after its last sweep
  return jacobi_svd64(p, p, t, W, U, Sv, W, max_sweeps, errw, st);
}

// The same decomposition by way of X = Q R: Jacobi on R^T, whose columns come graded (row i of R is of the
// size of the i-th singular value), R^T = U' S W^T, so that X = (Q W) S U'^T. On the square or tall matrix
// itself the columns are of one size and Jacobi needs two to four times the sweeps (128 x 128, spectrum
// 1 .. 1e-4: 22 against 9; 1 .. 1e-14: 36 against 10). Below 32 columns the QR costs what it saves.
cudaError_t svd_tall64(int q, int p, double* X, double* T1, double* T2, double* e0, double* e1, double** U,
                       double* Sv, double* V, int max_sweeps, uint32_t* errw, int sm_count, cudaStream_t st) {
  *U = T1;
  if (q <= 0 || p <= 0) return cudaSuccess;
  Jacobi64Plan plan;
  cudaError_t e = cudaSuccess;
  if (p >= 32 && q <= 1024 && (e = jacobi64_plan(p, p, true, st, plan)) != cudaSuccess) return e;
  if (!plan.kern) return jacobi_svd<double, double>(q, p, X, T1, Sv, V, T2, max_sweeps, errw, st);
  e = qr_reg64(q, p, X, T1, T2, st, true);  // Q: T1, R: T2
  if (e == cudaErrorNotSupported) e = qr_householder<double, double>(q, p, X, T1, T2, st);
  if (e != cudaSuccess) return e;
  const IdxMap one = IdxMap::lin(1), row = IdxMap::lin(p);
  if ((e = copy_map<double, double>(p, p, T2, one, row, X, row, one, 1.0, st)) != cudaSuccess) return e;
  if ((e = svd_graded64(p, X, V, Sv, T2, e0, e1, max_sweeps, errw, sm_count, st)) != cudaSuccess) return e;
  GemmArgs<double> g;  // U = Q W
  g.M = q; g.N = p; g.K = p;
  g.A = T1; g.am = one; g.ak = IdxMap::lin(q); g.a_kfast = false;
  g.B = T2; g.bn = row; g.bk = one;
  g.C = *U = X; g.cm = one; g.cn = IdxMap::lin(q);
  return gemm_simt<double>(g, nullptr, 0, sm_count, st);
}

}  // namespace ttfit
