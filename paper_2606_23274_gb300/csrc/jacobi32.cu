// FP32 one-sided Jacobi that returns the rotations alone: the cheap sweeps of the FP64 decomposition
// (svd_graded64).
#include <cooperative_groups.h>
#include <algorithm>
#include <cfloat>
#include "common.cuh"
#include "kernels.h"
#include "scalar_ops.cuh"

namespace cg = cooperative_groups;

namespace ttfit {

// The block tournament of the other Jacobi kernels (columns in blocks of b, two blocks a CTA, circle method over a
// cluster), with one column of a pair kept in registers while it meets its partners, and |w|^2 carried along. A pair's
// micro-round is a chain of about 500 cycles (loads, dot product, butterfly, angle, update); 138 columns take 64 us a
// sweep on 8 CTAs, 75 on 4; 74 columns 31 on 4, 35 on 8.
// One pair of FP32 columns, worked by a warp, with the rows of x in registers (kept by the caller), those of y loaded
// and stored.
template <int NV>
struct Col32 {
  float4 v[NV];
};

constexpr int J32_TAIL = 4;  // trailer of a column: |w|^2

template <int NV>
__device__ __forceinline__ bool jacobi32_pair(Col32<NV>& x, float& a, float* __restrict__ xj, int nq, int nr, int ld,
                                              float tol, bool act) {
  const int l = threadIdx.x & 31;
  float4* y4 = reinterpret_cast<float4*>(xj);
  Col32<NV> y;
  float g0 = 0.f, g1 = 0.f;
  const float b = xj[ld - J32_TAIL];
#pragma unroll
  for (int t = 0; t < NV; ++t) {
    const int r = l + 32 * t;
    if (r < nr) y.v[t] = y4[r];
    else y.v[t] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll
  for (int t = 0; t < NV; ++t)
    if (l + 32 * t < nq) {
      g0 = fmaf(x.v[t].x, y.v[t].x, g0);
      g1 = fmaf(x.v[t].y, y.v[t].y, g1);
      g0 = fmaf(x.v[t].z, y.v[t].z, g0);
      g1 = fmaf(x.v[t].w, y.v[t].w, g1);
    }
  const float g = warp_sum(g0 + g1);
  // the cosine itself: squares of small columns' products would underflow; columns below 1e-16 of the largest stay
  const bool rot = act && a > 1e-32f && b > 1e-32f && fabsf(g) * rsqrtf(a) * rsqrtf(b) > tol;
  __syncwarp();  // every lane has read the trailers, which lane 0 is about to replace (a shuffle orders no memory)
  if (rot) {
    const float zeta = __fdividef(b - a, 2.f * g);
    const float z2 = fmaf(zeta, zeta, 1.f);  // overflows for columns of very different size: t = 1 / (2 zeta) there
    const float t = fabsf(zeta) > 1e9f ? __fdividef(0.5f, zeta)
                                       : __fdividef(copysignf(1.f, zeta), fabsf(zeta) + z2 * rsqrtf(z2));
    const float cs = rot_rsqrt(fmaf(t, t, 1.f));
    const float sn = cs * t;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const float4 u = x.v[k], w = y.v[k];
      x.v[k] = make_float4(fmaf(cs, u.x, -sn * w.x), fmaf(cs, u.y, -sn * w.y), fmaf(cs, u.z, -sn * w.z), fmaf(cs, u.w, -sn * w.w));
      const float4 z = make_float4(fmaf(cs, w.x, sn * u.x), fmaf(cs, w.y, sn * u.y), fmaf(cs, w.z, sn * u.z), fmaf(cs, w.w, sn * u.w));
      if (l + 32 * k < nr) y4[l + 32 * k] = z;
    }
    a = fmaf(-t, g, a);
    if (l == 0) xj[ld - J32_TAIL] = fmaf(t, g, b);
  }
  return rot;
}

template <int NV>
__device__ __forceinline__ void load32(Col32<NV>& x, const float* p, int nr) {
  const int l = threadIdx.x & 31;
#pragma unroll
  for (int t = 0; t < NV; ++t)
    x.v[t] = l + 32 * t < nr ? reinterpret_cast<const float4*>(p)[l + 32 * t] : make_float4(0.f, 0.f, 0.f, 0.f);
}
template <int NV>
__device__ __forceinline__ void store32(const Col32<NV>& x, float* p, int nr) {
  const int l = threadIdx.x & 31;
#pragma unroll
  for (int t = 0; t < NV; ++t)
    if (l + 32 * t < nr) reinterpret_cast<float4*>(p)[l + 32 * t] = x.v[t];
}

__host__ __device__ inline int jacobi32_ld(int q, int p) {
  return (q + 3) / 4 * 4 + (p + 3) / 4 * 4 + J32_TAIL;
}

template <int NV>
__global__ void __launch_bounds__(640)
    jacobi32_kernel(int q, int p, int b, const float* __restrict__ Win, int max_sweeps, float ftol,
                    float* __restrict__ Vo) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), NC = (int)cl.num_blocks();
  const int P = 2 * NC;
  const int qs = (q + 3) / 4 * 4;
  const int ld = jacobi32_ld(q, p);
  const int nq = qs / 4, nr = (ld - J32_TAIL) / 4;
  extern __shared__ __align__(16) unsigned char j32s[];
  float* buf = (float*)j32s;                                  // [2][2 slots][b][ld]
  int* ids = (int*)(buf + (size_t)4 * b * ld);                // [2][2 slots][b] global column or -1
  float* nrm = (float*)(ids + 4 * b + 4);                     // [2 slots][b] final column norms
  __shared__ int flag[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  auto col = [&](int bi, int sl, int k) { return buf + ((size_t)(bi * 2 + sl) * b + k) * ld; };
  auto cid = [&](int bi, int sl, int k) -> int& { return ids[(bi * 2 + sl) * b + k]; };

  for (int sl = 0; sl < 2; ++sl) {  // CTA c holds the blocks at positions c and P-1-c
    const int blk = sl == 0 ? rank : P - 1 - rank;
    for (int k = 0; k < b; ++k) {
      const int gid = blk * b + k;
      if (threadIdx.x == 0) cid(0, sl, k) = gid < p ? gid : -1;
      float* x = col(0, sl, k);
      for (int r = threadIdx.x; r < ld; r += blockDim.x) {
        float v = 0.f;
        if (gid < p && r < ld - J32_TAIL) v = r < q ? Win[(size_t)gid * q + r] : (r >= qs && r - qs == gid ? 1.f : 0.f);
        x[r] = v;
      }
    }
  }
  if (threadIdx.x < 2) flag[threadIdx.x] = 0;
  cl.sync();

  int cur = 0, sweep = 0;
  auto refresh = [&]() {  // |w|^2 of every column, from its rows
    for (int w0 = 0; w0 < 2 * b; w0 += nw) {
      const int w = w0 + warp;
      float s = 0.f;
      float* x = col(cur, w < b ? 0 : 1, w < 2 * b ? w % b : 0);
      if (w < 2 * b) {
        const float4* x4 = reinterpret_cast<const float4*>(x);
        for (int r = lane; r < nq; r += 32) {
          const float4 v = x4[r];
          s = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, s))));
        }
      }
      s = warp_sum(s);
      if (w < 2 * b && lane == 0) x[ld - J32_TAIL] = s;
    }
    __syncthreads();
  };
  bool done = false;
  Col32<NV> x;
  while (!done && sweep < max_sweeps) {
    bool rot = false;
    refresh();
    for (int sr = 0; sr < P - 1; ++sr) {
      if (sr == 0) {  // pairs inside each block (round robin over the b columns of both slots)
        const int B = b + (b & 1), half = B / 2;
        for (int mr = 0; mr < B - 1; ++mr) {
          const int sl = warp / half, k = warp % half;
          int i = b, j = b;
          if (warp < 2 * half) rr_pair(mr, k, B, i, j);
          const bool act = i < b && j < b;
          float* xi = col(cur, act ? sl : 0, act ? i : 0);
          float a = xi[ld - J32_TAIL];
          load32(x, xi, act ? nr : 0);
          const bool r1 = jacobi32_pair<NV>(x, a, col(cur, act ? sl : 0, act ? j : 0), nq, nr, ld, ftol, act);
          if (r1) {
            store32(x, xi, nr);
            if (lane == 0) xi[ld - J32_TAIL] = a;
          }
          rot |= r1;
          __syncthreads();
        }
      }
      {  // pairs between the two blocks: warp w keeps column w of slot 0 in registers and meets column
         // (w + mr) mod b of slot 1
        const bool act = warp < b;
        float* xi = col(cur, 0, act ? warp : 0);
        float a = xi[ld - J32_TAIL];
        load32(x, xi, act ? nr : 0);
        bool changed = false;
        int j = act ? warp : 0;
        for (int mr = 0; mr < b; ++mr) {
          changed |= jacobi32_pair<NV>(x, a, col(cur, 1, j), nq, nr, ld, ftol, act);
          j = (j + 1 == b) ? 0 : j + 1;
          __syncthreads();
        }
        if (changed) {
          store32(x, xi, nr);
          if (lane == 0) xi[ld - J32_TAIL] = a;
        }
        rot |= changed;
      }
      // rotate the positions 1..P-1 by one (position 0 stays): pull the next two blocks
      cl.sync();
      const int nb = cur ^ 1;
      {
        const uint4* rsrc[2];
        const int* rid[2];
#pragma unroll
        for (int sl = 0; sl < 2; ++sl) {
          const int xp = sl == 0 ? rank : P - 1 - rank;
          const int src = xp == 0 ? 0 : (xp == 1 ? P - 1 : xp - 1);
          const int scta = src < NC ? src : P - 1 - src, ssl = src < NC ? 0 : 1;
          rsrc[sl] = reinterpret_cast<const uint4*>(cl.map_shared_rank(col(cur, ssl, 0), scta));
          rid[sl] = cl.map_shared_rank(&cid(cur, ssl, 0), scta);
        }
        const int n16 = b * ld / 4;
        for (int e0 = threadIdx.x; e0 < n16; e0 += 2 * blockDim.x) {  // every remote load before the first store
          uint4 v[2][2];
#pragma unroll
          for (int sl = 0; sl < 2; ++sl)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int e = e0 + u * blockDim.x;
              if (e < n16) v[sl][u] = rsrc[sl][e];
            }
#pragma unroll
          for (int sl = 0; sl < 2; ++sl)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int e = e0 + u * blockDim.x;
              if (e < n16) reinterpret_cast<uint4*>(col(nb, sl, 0))[e] = v[sl][u];
            }
        }
        for (int t = threadIdx.x; t < b; t += blockDim.x) {
          cid(nb, 0, t) = rid[0][t];
          cid(nb, 1, t) = rid[1][t];
        }
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
  refresh();
  for (int w = threadIdx.x; w < 2 * b; w += blockDim.x) {
    const int sl = w / b, k = w % b;
    nrm[w] = cid(cur, sl, k) >= 0 ? sqrtf(col(cur, sl, k)[ld - J32_TAIL]) : -1.f;
  }
  cl.sync();
  for (int w = warp; w < 2 * b; w += nw) {  // every column's rank among all p (descending, ties by column index)
    const int sl = w / b, k = w % b;
    const int me = cid(cur, sl, k);
    if (me < 0) continue;
    const float v = nrm[w];
    int rk = 0;
    for (int c = 0; c < NC; ++c) {
      const float* rn = cl.map_shared_rank(nrm, c);
      const int* ri = cl.map_shared_rank(&cid(cur, 0, 0), c);
      for (int t = lane; t < 2 * b; t += 32) {
        const int o = ri[t];  // ids of slot 0 then slot 1 are contiguous
        const float u = rn[t];
        rk += (o >= 0) && (u > v || (u == v && o < me));
      }
    }
    rk = warp_sum(rk);
    const float* xc = col(cur, sl, k);
    for (int r = lane; r < p; r += 32) Vo[(size_t)rk * p + r] = xc[qs + r];
  }
  cl.sync();  // no CTA leaves while another may still read its shared memory
}

inline size_t jacobi32_smem(int q, int p, int nc) {
  const size_t b = (p + 2 * nc - 1) / (2 * nc);
  return 4 * b * jacobi32_ld(q, p) * sizeof(float) + (4 * b + 4) * sizeof(int) + 2 * b * sizeof(float) + 16;
}

namespace {

struct Jacobi32Shape {
  int nc, nv, b, threads;
  size_t smem;
  bool ok;
};
Jacobi32Shape jacobi32_shape(int p) {
  Jacobi32Shape s{};
  s.nc = p < 96 ? 4 : 8;
  s.b = (p + 2 * s.nc - 1) / (2 * s.nc);
  const int B = s.b + (s.b & 1);
  s.threads = std::max(128, 32 * B);
  s.smem = jacobi32_smem(p, p, s.nc);
  s.nv = ((jacobi32_ld(p, p) - J32_TAIL) / 4 + 31) / 32;
  s.ok = s.threads <= 640 && s.smem <= 220 * 1024 && s.nv <= 5;
  return s;
}

}  // namespace

bool jacobi32_rotations_fits(int p) { return jacobi32_shape(p).ok; }

cudaError_t jacobi32_rotations(int p, const float* W, float* V, int sweeps, cudaStream_t st) {
  const Jacobi32Shape s = jacobi32_shape(p);
  if (!s.ok) return cudaErrorNotSupported;
  auto launch = [&](auto kern) -> cudaError_t {
    cudaError_t e = ensure_smem((const void*)kern, s.smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(s.nc);
    cfg.blockDim = dim3(s.threads);
    cfg.dynamicSmemBytes = s.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = s.nc;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    ++tl_launches;
    e = cudaLaunchKernelEx(&cfg, kern, p, p, s.b, W, sweeps, 4.f * FLT_EPSILON * sqrtf((float)p), V);
    return e != cudaSuccess ? e : cudaGetLastError();
  };
  switch (s.nv) {
    case 1: return launch(jacobi32_kernel<1>);
    case 2: return launch(jacobi32_kernel<2>);
    case 3: return launch(jacobi32_kernel<3>);
    case 4: return launch(jacobi32_kernel<4>);
    default: return launch(jacobi32_kernel<5>);
  }
}

}  // namespace ttfit
