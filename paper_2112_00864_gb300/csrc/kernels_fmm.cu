// Evaluation kernels of the boundary-concentrated FMM (Sec. 3.3, Algorithms
// 1-3): source weights, moments (P2M), upward pass (M2M), interaction phase
// on CUDA cores (M2L), downward pass (L2L), evaluation (L2P) and near field
// (P2P over the extended neighbour list N*), fused in FP64, and the Galerkin
// element sums plus near-rule corrections.
//
// Expansions are box-scaled: moments m^b = sum_j W_j ((y_j - c)/s)^b, locals
// phi(x) = sum_a l^a ((x - c)/s)^a, so one M2L table per integer offset
// serves every level (the 1/s factor is applied here).
#include <cstdio>

#include "kernels.cuh"

namespace bcfmm {

constexpr double kInv4Pi = 0.079577471545947667884441881686257;

// ------------------------------------------------------------ weights
// W[d][j] = w_j * dens[d][elem(j)] (d < ndens), zero for ndens <= d < ndp.
template <typename T>
__global__ void k_weights(const double4_32a* __restrict__ pt, const int* __restrict__ elem, int64_t n,
                          const double* __restrict__ dens, int64_t nel, int ndens, int ndp, T* __restrict__ W) {
  int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= n) return;
  double w = pt[j].w;
  int e = elem[j];
  for (int d = 0; d < ndp; ++d) W[(int64_t)d * n + j] = (T)(d < ndens ? w * dens[(int64_t)d * nel + e] : 0.0);
}

template <typename T>
cudaError_t launch_weights(const DevGeom& G, int cls, int64_t n, const double* dens, int64_t nel, int ndens,
                           int ndp, T* W, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_weights<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(G.pt64[cls], G.pt_elem[cls], n, dens, nel, ndens, ndp, W);
  return cudaGetLastError();
}

// degree-major position of the multi-index (i, j, k): degree d, then i
// descending, then j descending
__device__ __forceinline__ int midx3(int i, int j, int k) {
  const int d = i + j + k;
  return d * (d + 1) * (d + 2) / 6 + (j + k) * (j + k + 1) / 2 + k;
}

// ---------------------------------------------------------------- P2M
// One CTA per leaf (and four densities).  The moments are an outer-product sum
// over the leaf's points: powers of x against products y^b z^c.  A thread
// takes one (b, c) and a share of the points: one load of its product and the
// point's powers of x (two or three 16-byte loads, the same for all lanes)
// serve PX coefficients per density.  (A thread per coefficient needed four
// loads for each and formed the monomial anew for every density.)  The shares
// are added through shared memory.  Rows of kPwS = 65: threads of one warp
// read rows of different exponents at the same point, an odd stride puts them
// in different banks.  Shared-memory loads and latency bound it: 767,360
// points at p = 7 take 63 us with one density (as before); with sixteen
// densities (25,040 points) the upward pass went from 1.01 ms to 0.05 ms.
constexpr int kPwS = 65;
constexpr int kP2mDens = 4;

// offset of point j from the leaf's centre in units of the box side
template <typename T>
__device__ __forceinline__ void point_xhat(const DevGeom& G, int cls, int64_t j, const double4_32a& cs, double inv_s, T& x,
                                           T& y, T& z) {
  if constexpr (sizeof(T) == 4) {
    const float4 v = G.xhat[cls][j];
    x = v.x; y = v.y; z = v.z;
  } else {
    const double4_32a q = G.pt64[cls][j];
    x = (q.x - cs.x) * inv_s; y = (q.y - cs.y) * inv_s; z = (q.z - cs.z) * inv_s;
  }
}

template <typename T, int PX, int NDC>
__global__ void __launch_bounds__(128) k_p2m(DevGeom G, const int* __restrict__ leaves, int cls, const T* __restrict__ W,
                                            int64_t nsp, int ndp, T* __restrict__ mom) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int P = G.p, np = G.np, npair = (P + 1) * (P + 2) / 2, NS = 128 / npair;
  T* xp = reinterpret_cast<T*>(smraw);               // [64][PX] powers of x
  T* ws = xp + 64 * PX;                              // [NDC][64]
  T* py = ws + NDC * 64;                             // [P+1][kPwS]
  T* pz = py + (P + 1) * kPwS;                       // [P+1][kPwS]
  T* yz = pz + (P + 1) * kPwS;                       // [npair][kPwS]
  T* red = yz + npair * kPwS;                        // [NDC][np]
  const int leaf = leaves[blockIdx.x], d0 = blockIdx.y * NDC;
  const double4_32a cs = G.box_cs[leaf];
  const int2 r = G.box_rng[cls][leaf];
  const double inv_s = sizeof(T) == 8 ? 1.0 / cs.w : 0.0;
  const int split = threadIdx.x / npair, pair = threadIdx.x - split * npair;
  // (b, c) of this thread: pair = c + (b + c)(b + c + 1) / 2
  int deg = 0, c = pair;
  while (c > deg) { c -= deg + 1; ++deg; }
  const int b = deg - c, na = P - deg;
  T acc[NDC][PX];
#pragma unroll
  for (int d = 0; d < NDC; ++d)
#pragma unroll
    for (int k = 0; k < PX; ++k) acc[d][k] = (T)0;
  for (int j0 = r.x; j0 < r.y; j0 += 64) {
    const int m = min(64, r.y - j0);
    __syncthreads();
    if (threadIdx.x < m) {
      const int j = threadIdx.x;
      T x, y, z;
      point_xhat<T>(G, cls, j0 + j, cs, inv_s, x, y, z);
      T vx = (T)1, vy = (T)1, vz = (T)1;
#pragma unroll
      for (int k = 0; k < PX; ++k) { xp[j * PX + k] = vx; vx *= x; }
      for (int k = 0; k <= P; ++k) { py[k * kPwS + j] = vy; pz[k * kPwS + j] = vz; vy *= y; vz *= z; }
    } else if (threadIdx.x >= 64) {
      const int j = threadIdx.x - 64;
      if (j < m)
        for (int d = 0; d < NDC; ++d) ws[d * 64 + j] = d0 + d < ndp ? W[(int64_t)(d0 + d) * nsp + j0 + j] : (T)0;
    }
    __syncthreads();
    if (split < NS)
      for (int j = split; j < m; j += NS) {
        T t = py[b * kPwS + j] * pz[c * kPwS + j];
        if constexpr (NDC == 1) t *= ws[j];
        yz[pair * kPwS + j] = t;
      }
    // (a thread reads the products it wrote itself)
    if (split < NS)
      for (int j = split; j < m; j += NS) {
        const T t = yz[pair * kPwS + j];
        T x[PX];
#pragma unroll
        for (int k = 0; k < PX; k += 16 / sizeof(T))
          *reinterpret_cast<float4*>(x + k) = *reinterpret_cast<const float4*>(xp + j * PX + k);
#pragma unroll
        for (int d = 0; d < NDC; ++d) {
          const T v = NDC == 1 ? t : t * ws[d * 64 + j];
#pragma unroll
          for (int k = 0; k < PX; ++k) acc[d][k] += v * x[k];
        }
      }
  }
  for (int sp = 0; sp < NS; ++sp) {
    __syncthreads();
    if (split == sp) {
#pragma unroll
      for (int k = 0; k < PX; ++k) {
        if (k > na) break;
        const int q = midx3(k, b, c);
#pragma unroll
        for (int d = 0; d < NDC; ++d) red[d * np + q] = sp == 0 ? acc[d][k] : red[d * np + q] + acc[d][k];
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < NDC * np; i += 128) {
    const int d = i / np;
    if (d0 + d < ndp) mom[((int64_t)leaf * ndp + d0 + d) * G.ms + i - d * np] = red[i];
  }
}

template <typename T, int PX, int NDC>
cudaError_t launch_p2m_t(const DevGeom& G, const DevTaskLists& L, const T* W, int64_t nsp, int ndp, T* mom, cudaStream_t st) {
  const int npair = (G.p + 1) * (G.p + 2) / 2;
  const size_t sm = sizeof(T) * (64 * PX + NDC * (64 + G.np) + (2 * (G.p + 1) + npair) * kPwS);
  if (sm > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k_p2m<T, PX, NDC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  k_p2m<T, PX, NDC><<<dim3(L.n_p2m, (ndp + NDC - 1) / NDC), 128, sm, st>>>(G, L.p2m_leaf, L.src_cls, W, nsp, ndp, mom);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_p2m(const DevGeom& G, const DevTaskLists& L, const T* W, int64_t nsrc_pts, int ndp,
                       T* mom, cudaStream_t st) {
  if (L.n_p2m == 0) return cudaSuccess;
  if (ndp == 1) {
    if (G.p < 8) return launch_p2m_t<T, 8, 1>(G, L, W, nsrc_pts, ndp, mom, st);
    if (G.p < 12) return launch_p2m_t<T, 12, 1>(G, L, W, nsrc_pts, ndp, mom, st);
    return launch_p2m_t<T, 16, 1>(G, L, W, nsrc_pts, ndp, mom, st);
  }
  if (G.p < 8) return launch_p2m_t<T, 8, kP2mDens>(G, L, W, nsrc_pts, ndp, mom, st);
  if (G.p < 12) return launch_p2m_t<T, 12, kP2mDens>(G, L, W, nsrc_pts, ndp, mom, st);
  return launch_p2m_t<T, 16, kP2mDens>(G, L, W, nsrc_pts, ndp, mom, st);
}

// ------------------------------------------------------- M2M and L2L shifts
// Shifts between a box and its child in octant o (centre offset sigma s_p/4,
// sigma_i = +-1 by the octant's bits; child side s_p/2), box-scaled:
//   M2M  mhat_p[b] = sum_{g <= b} prod_i C(b_i, g_i) (sigma_i/4)^(b_i - g_i) 2^-|g| mhat_c[g]
//   L2L  lhat_c[a] = 2^-|a| sum_{b >= a} prod_i C(b_i, a_i) (sigma_i/4)^(b_i - a_i) lhat_p[b]
// Both factor into three 1-D binomial shifts, one per axis (the Taylor
// shift of (u + d)^n along each coordinate); every intermediate index stays
// within the total-degree bound (its components lie between those of the
// input and the output), so the passes are exact on the truncated arrays.
// One pass costs about n (p+1)/2 products instead of the dense table's
// n^2 / 2 (n = nterms(p)), and no table is read from memory.

// tab[s][n][k] = C(n, k) (+-1/4)^(n - k), s = 0: -1/4, s = 1: +1/4 (the
// table is built on the host, G.shift64 / G.shift32)
template <typename T>
__device__ __forceinline__ const T* shift_src(const DevGeom& G);
template <>
__device__ __forceinline__ const float* shift_src<float>(const DevGeom& G) { return G.shift32; }
template <>
__device__ __forceinline__ const double* shift_src<double>(const DevGeom& G) { return G.shift64; }
template <typename T>
__device__ void shift_table(const DevGeom& G, T* tab) {
  const T* src = shift_src<T>(G);
  for (int e = threadIdx.x; e < 2 * (G.p + 1) * (G.p + 1); e += blockDim.x) tab[e] = src[e];
}

// ---------------------------------------------------------------- M2M
// One CTA per parent box and density.  The children's moments are merged axis
// by axis: the x shift adds the two children of each (y, z), the y shift the
// two sums of each z, the z shift the last two: 7 np outputs of two 1-D
// shifts each and three barriers, where shifting child by child took 24 np
// outputs and forty barriers.  Latency-bound: a level of 64 to 360 parents 10 us
// (20 - 22 before), the finest of the level-4 ball, 1,908 parents, 23 us (46).
// Children without sources count as zero (their moments are never written).
template <typename T>
__global__ void __launch_bounds__(256) k_m2m(DevGeom G, const int* __restrict__ parents, int cls, int ndp, T* __restrict__ mom) {
  extern __shared__ unsigned char smraw[];
  const int np = G.np, P1 = G.p + 1;
  T* tab = reinterpret_cast<T*>(smraw);              // [2][P+1][P+1]
  T* v8 = tab + 2 * P1 * P1;                         // [8 octants][np]
  T* v4 = v8 + 8 * np;                               // [4 (y, z)][np]
  T* v2 = v4 + 4 * np;                               // [2 (z)][np]
  __shared__ int child[8];
  shift_table(G, tab);
  const int P = parents[blockIdx.x], d = blockIdx.y;
  const int c0 = G.box_child0[P], nc = G.box_nchild[P];
  if (threadIdx.x < 8) child[threadIdx.x] = -1;
  __syncthreads();
  if (threadIdx.x < nc) {
    const int2 r = G.box_rng[cls][c0 + threadIdx.x];
    if (r.y > r.x) child[G.box_octant[c0 + threadIdx.x]] = c0 + threadIdx.x;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 8 * np; i += blockDim.x) {
    const int o = i / np, q = i - o * np, c = child[o];
    T v = 0;
    if (c >= 0) {
      const int mi = G.mi[q];
      v = mom[((int64_t)c * ndp + d) * G.ms + q] * ((T)1 / (T)(1 << ((mi & 255) + ((mi >> 8) & 255) + ((mi >> 16) & 255))));
    }
    v8[i] = v;
  }
  const T* lo = tab;
  const T* hi = tab + P1 * P1;
  // x: input position of (k, j, l) moves on by the degree's count
  __syncthreads();
  for (int i = threadIdx.x; i < 4 * np; i += blockDim.x) {
    const int o = i / np, q = i - o * np, mi = G.mi[q];
    const int n = mi & 255, j = (mi >> 8) & 255, l = (mi >> 16) & 255;
    const T* in0 = v8 + 2 * o * np;
    const T* in1 = in0 + np;
    T acc = 0;
    int pos = midx3(0, j, l), deg = j + l;
    for (int k = 0; k <= n; ++k) {
      acc += lo[n * P1 + k] * in0[pos] + hi[n * P1 + k] * in1[pos];
      pos += (deg + 1) * (deg + 2) / 2;
      ++deg;
    }
    v4[i] = acc;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * np; i += blockDim.x) {
    const int o = i / np, q = i - o * np, mi = G.mi[q];
    const int a = mi & 255, n = (mi >> 8) & 255, l = (mi >> 16) & 255;
    const T* in0 = v4 + 2 * o * np;
    const T* in1 = in0 + np;
    T acc = 0;
    for (int k = 0; k <= n; ++k) {
      const int pos = midx3(a, k, l);
      acc += lo[n * P1 + k] * in0[pos] + hi[n * P1 + k] * in1[pos];
    }
    v2[i] = acc;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < np; q += blockDim.x) {
    const int mi = G.mi[q];
    const int a = mi & 255, b = (mi >> 8) & 255, n = (mi >> 16) & 255;
    T acc = 0;
    for (int k = 0; k <= n; ++k) {
      const int pos = midx3(a, b, k);
      acc += lo[n * P1 + k] * v2[pos] + hi[n * P1 + k] * v2[np + pos];
    }
    mom[((int64_t)P * ndp + d) * G.ms + q] = acc;
  }
}

template <typename T>
cudaError_t launch_m2m(const DevGeom& G, const int* parents, int n, int cls, int ndp, T* mom, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const size_t sm = sizeof(T) * (2 * (G.p + 1) * (G.p + 1) + 14 * G.np);
  if (sm > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k_m2m<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  k_m2m<T><<<dim3(n, ndp), 256, sm, st>>>(G, parents, cls, ndp, mom);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- M2L
// One CTA per target box, thread per row alpha of the local expansion.
// Tt[code][b][a] is the transposed table (coalesced over alpha).  The level
// of the target box has order q <= p (Sec. 4.3): rows |alpha| <= q, and row
// alpha needs only b < nterms(q - |alpha|) (|alpha| + |beta| <= q).
template <typename T, int ND>
__global__ void k_m2l_simt(DevGeom G, DevTaskLists L, const int* __restrict__ sel, const T* __restrict__ Tt, int ndp,
                           const T* __restrict__ mom, T* __restrict__ loc) {
  extern __shared__ unsigned char smraw[];
  T* ms = reinterpret_cast<T*>(smraw);               // [ND][nq]
  const int np = G.np;
  const int ki = sel ? sel[blockIdx.x] : (int)blockIdx.x;   // index into the task's M2L targets
  const int tb = L.m2l_tgt[ki];
  const int q = G.box_q[tb], nq = nterms_q(q);
  const int a = threadIdx.x;
  int K = 0;
  if (a < nq) {
    const int mi = G.mi[a];
    K = nterms_q(q - ((mi & 255) + ((mi >> 8) & 255) + ((mi >> 16) & 255)));
  }
  // products of one translation in T, the sum over the interaction list
  // (~10^3 entries for eta0 = 0.5) in FP64
  double acc[ND];
#pragma unroll
  for (int d = 0; d < ND; ++d) acc[d] = 0.0;
  const int e0 = L.vl_off[ki], e1 = L.vl_off[ki + 1];
  for (int e = e0; e < e1; ++e) {
    const int sb = L.vl_src[e];
    const T* Tc = Tt + (int64_t)L.vl_code[e] * np * np;
    __syncthreads();
    for (int i = threadIdx.x; i < ND * nq; i += blockDim.x) ms[i] = mom[((int64_t)sb * ndp + i / nq) * G.ms + i % nq];
    __syncthreads();
    if (a < nq) {
      T part[ND];
#pragma unroll
      for (int d = 0; d < ND; ++d) part[d] = 0;
      for (int b = 0; b < K; ++b) {
        const T t = Tc[(int64_t)b * np + a];
#pragma unroll
        for (int d = 0; d < ND; ++d) part[d] += t * ms[d * nq + b];
      }
#pragma unroll
      for (int d = 0; d < ND; ++d) acc[d] += (double)part[d];
    }
  }
  if (a < nq) {
    const double inv_s = 1.0 / G.box_cs[tb].w;
#pragma unroll
    for (int d = 0; d < ND; ++d) loc[((int64_t)tb * ndp + d) * G.ms + a] = (T)(acc[d] * inv_s);
  }
}

template <typename T>
cudaError_t launch_m2l_simt(const DevGeom& G, const DevTaskLists& L, const T* Tt, int ndp, const T* mom, T* loc,
                            cudaStream_t st, const int* sel, int nsel) {
  const int n = sel ? nsel : L.n_m2l;
  if (n == 0) return cudaSuccess;
  int threads = ((G.np + 31) / 32) * 32;
  size_t sm = sizeof(T) * ndp * G.np;
  switch (ndp) {
    case 1: k_m2l_simt<T, 1><<<n, threads, sm, st>>>(G, L, sel, Tt, ndp, mom, loc); break;
    case 2: k_m2l_simt<T, 2><<<n, threads, sm, st>>>(G, L, sel, Tt, ndp, mom, loc); break;
    case 4: k_m2l_simt<T, 4><<<n, threads, sm, st>>>(G, L, sel, Tt, ndp, mom, loc); break;
    case 8: k_m2l_simt<T, 8><<<n, threads, sm, st>>>(G, L, sel, Tt, ndp, mom, loc); break;
    case 16: k_m2l_simt<T, 16><<<n, threads, sm, st>>>(G, L, sel, Tt, ndp, mom, loc); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------- L2L
// One CTA per parent box and density, the mirror image of M2M: the z shift
// gives the two z halves, the y shift their four (y, z) parts, the x shift the
// children, which add it to their own.  The parent's expansion has its level's
// order qp, the child's is cut to its own (Sec. 4.3): the passes run over
// |b| <= qp, the child receives |a| <= min(q_child, qp).  parents: (box, mask of
// the child slots that take part).  The level-4 ball's finest level (14,976
// children) takes 28 us, 37 with one CTA per child.
template <typename T>
__global__ void __launch_bounds__(256) k_l2l(DevGeom G, const int2* __restrict__ parents, int ndp, T* __restrict__ loc) {
  extern __shared__ unsigned char smraw[];
  const int P1 = G.p + 1;
  const int2 pm = parents[blockIdx.x];
  const int P = pm.x, d = blockIdx.y, qp = G.box_q[P], nqp = nterms_q(qp);
  T* tab = reinterpret_cast<T*>(smraw);              // [2][P+1][P+1]
  T* v1 = tab + 2 * P1 * P1;                         // [np]
  T* v2 = v1 + G.np;                                 // [2 (z)][np]
  T* v4 = v2 + 2 * G.np;                             // [4 (y, z)][np]
  shift_table(G, tab);
  for (int q = threadIdx.x; q < nqp; q += blockDim.x) v1[q] = loc[((int64_t)P * ndp + d) * G.ms + q];
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * nqp; i += blockDim.x) {
    const int o = i / nqp, q = i - o * nqp, mi = G.mi[q];
    const int a = mi & 255, b = (mi >> 8) & 255, c = (mi >> 16) & 255;
    const T* tb = tab + o * P1 * P1;
    T acc = 0;
    for (int k = c; a + b + k <= qp; ++k) acc += tb[k * P1 + c] * v1[midx3(a, b, k)];
    v2[o * nqp + q] = acc;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 4 * nqp; i += blockDim.x) {
    const int o = i / nqp, q = i - o * nqp, mi = G.mi[q];          // o = y + 2 z
    const int a = mi & 255, b = (mi >> 8) & 255, c = (mi >> 16) & 255;
    const T* tb = tab + (o & 1) * P1 * P1;
    const T* in = v2 + (o >> 1) * nqp;
    T acc = 0;
    for (int k = b; a + k + c <= qp; ++k) acc += tb[k * P1 + b] * in[midx3(a, k, c)];
    v4[o * nqp + q] = acc;
  }
  __syncthreads();
  const int c0 = G.box_child0[P], nc = G.box_nchild[P];
  for (int i = threadIdx.x; i < nc * nqp; i += blockDim.x) {
    const int s = i / nqp, q = i - s * nqp, C = c0 + s;
    // a child of a higher order than its parent gets nothing above |a| = qp
    if (!(pm.y >> s & 1) || q >= nterms_q(G.box_q[C])) continue;
    const int oc = G.box_octant[C], mi = G.mi[q];
    const int a = mi & 255, b = (mi >> 8) & 255, c = (mi >> 16) & 255;
    const T* tb = tab + (oc & 1) * P1 * P1;
    const T* in = v4 + (oc >> 1) * nqp;
    T* out = loc + ((int64_t)C * ndp + d) * G.ms + q;
    const T own = *out;
    T acc = 0;
    for (int k = a; k + b + c <= qp; ++k) acc += tb[k * P1 + a] * in[midx3(k, b, c)];
    *out = own + acc * ((T)1 / (T)(1 << (a + b + c)));
  }
}

template <typename T>
cudaError_t launch_l2l(const DevGeom& G, const int2* parents, int n, int ndp, T* loc, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const size_t sm = sizeof(T) * (2 * (G.p + 1) * (G.p + 1) + 7 * G.np);
  k_l2l<T><<<dim3(n, ndp), 256, sm, st>>>(G, parents, ndp, loc);
  return cudaGetLastError();
}

// ------------------------------------------------ evaluation + near field
// One CTA (128 threads) per target leaf or chunk block; thread groups split
// each source tile and are reduced at the end.  The sources of N* arrive as
// merged runs of the sorted point array and are streamed through shared memory
// in tiles that span run boundaries.  FP32 coordinates are translated to the
// target leaf's frame with double-float (hi + lo) arithmetic, so differences
// keep full relative accuracy.  Only the leaf's own run (first, VtV) can hold
// the target point itself; tiles overlapping it skip r == 0.  FP32 partial
// sums are folded into compensated (hi + lo) sums tile by tile.
constexpr int kTile = 256;
constexpr int kRunBatch = 256;

__device__ __forceinline__ void split_df(double v, float& hi, float& lo) {
  hi = (float)v;
  lo = (float)(v - (double)hi);
}

// largest r in [0, n) with pre[r] <= v  (pre[0] = 0 <= v < pre[n])
__device__ __forceinline__ int find_run(const int* pre, int n, int v) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (pre[mid] <= v) lo = mid; else hi = mid;
  }
  return lo;
}

// prefix sums of the run lengths of one batch (warp 0), starts into rst
__device__ __forceinline__ void scan_runs(const int2* __restrict__ runs, int nr, int* pre, int* rst) {
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    int carry = 0;
    if (lane == 0) pre[0] = 0;
    for (int c = 0; c < nr; c += 32) {
      const int r = c + lane;
      int len = 0;
      if (r < nr) { const int2 rr = runs[r]; len = rr.y - rr.x; rst[r] = rr.x; }
      int x = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += y; }
      if (r < nr) pre[r + 1] = carry + x;
      carry += __shfl_sync(0xffffffffu, x, 31);
    }
  }
}

template <typename T, int ND>
__device__ __forceinline__ void l2p_and_store(const DevGeom& G, int leaf, int ndp, const T* __restrict__ loc,
                                              double xs, double ys, double zs, const double* near, int64_t pos,
                                              int64_t ntp, double* __restrict__ phi) {
  T far[ND];
#pragma unroll
  for (int d = 0; d < ND; ++d) far[d] = (T)0;
  // L2P: phi_far(x) = sum_a l^a xhat^a, xhat = (x - c)/s (locals of boxes
  // without an interaction list are zero)
  if (loc != nullptr) {
    T px[16], py[16], pz[16];
    px[0] = py[0] = pz[0] = (T)1;
    for (int k = 1; k <= G.p; ++k) { px[k] = px[k - 1] * (T)xs; py[k] = py[k - 1] * (T)ys; pz[k] = pz[k - 1] * (T)zs; }
    const T* lb = loc + (int64_t)leaf * ndp * G.ms;
    const int nq = nterms_q(G.box_q[leaf]);          // the leaf level's order
    for (int q = 0; q < nq; ++q) {
      const int mi = G.mi[q];
      const T mono = px[mi & 255] * py[(mi >> 8) & 255] * pz[(mi >> 16) & 255];
#pragma unroll
      for (int d = 0; d < ND; ++d) far[d] += lb[d * G.ms + q] * mono;
    }
  }
#pragma unroll
  for (int d = 0; d < ND; ++d) phi[(int64_t)d * ntp + pos] = near[d] * kInv4Pi + (double)far[d];
}

// ------------------------------------------------ L2P (FP32 tasks)
// sum_{|a| <= Q} l^a x^a: Horner in x for every (j, k), then the products
// y^j z^k (about 1.5 FMA a term and no table of multi-indices)
template <int Q>
__device__ __forceinline__ float l2p_eval(const float* __restrict__ sl, float x, float y, float z) {
  float far = 0.f, yp = 1.f;
#pragma unroll
  for (int j = 0; j <= Q; ++j) {
    float yz = yp;
    asm volatile("" ::: "memory");       // this j's coefficients only (registers)
#pragma unroll
    for (int k = 0; k <= Q - j; ++k) {
      float h = sl[midx3(Q - j - k, j, k)];
#pragma unroll
      for (int i = Q - j - k - 1; i >= 0; --i) h = fmaf(h, x, sl[midx3(i, j, k)]);
      far = fmaf(h, yz, far);
      yz *= z;
    }
    yp *= y;
  }
  return far;
}
__device__ float l2p_loop(const float* sl, int q, float x, float y, float z) {
  float far = 0.f, yp = 1.f;
  for (int j = 0; j <= q; ++j) {
    float yz = yp;
    for (int k = 0; k <= q - j; ++k) {
      float h = sl[midx3(q - j - k, j, k)];
      for (int i = q - j - k - 1; i >= 0; --i) h = fmaf(h, x, sl[midx3(i, j, k)]);
      far = fmaf(h, yz, far);
      yz *= z;
    }
    yp *= y;
  }
  return far;
}

// phi += far field of the leaf's local expansion, one CTA per target leaf, one
// target point per thread and round; the coefficients are staged in shared
// memory (locals of boxes without an interaction list are zero).  Latency: two
// dependent loads and some 400 instructions a CTA, so small CTAs, twelve on an
// SM; 767,360 points at orders 6 and 7 take 35 us (as the tail of the near-
// field CTAs, with FP64 scaling and indexed powers, it cost them about 0.1 ms).
// Unrolled for the leaf orders 4 to 8 that the level schedules give; the loop
// costs a whole VtV evaluation of the h = 1/16 cube 194 against 180 us at order 4,
// 786 against 769 us at order 8.
constexpr int kL2pThreads = 64;
__global__ void __launch_bounds__(kL2pThreads, 12) k_l2p(DevGeom G, const int* __restrict__ leaves, int tc, int64_t ntp,
                                                         int ndp, const float* __restrict__ loc,
                                                         double* __restrict__ phi) {
  __shared__ float sl[456];
  const int leaf = leaves[blockIdx.x];
  const int2 tr = G.box_rng[tc][leaf];
  const int q = G.box_q[leaf], nq = nterms_q(q);
  for (int d = 0; d < ndp; ++d) {
    if (d > 0) __syncthreads();
    for (int a = threadIdx.x; a < nq; a += kL2pThreads) sl[a] = loc[((int64_t)leaf * ndp + d) * G.ms + a];
    __syncthreads();
    for (int j = tr.x + threadIdx.x; j < tr.y; j += kL2pThreads) {
      const float4 v = G.xhat[tc][j];
      const float x = v.x, y = v.y, z = v.z;
      float far;
      switch (q) {
        case 4: far = l2p_eval<4>(sl, x, y, z); break;
        case 5: far = l2p_eval<5>(sl, x, y, z); break;
        case 6: far = l2p_eval<6>(sl, x, y, z); break;
        case 7: far = l2p_eval<7>(sl, x, y, z); break;
        case 8: far = l2p_eval<8>(sl, x, y, z); break;
        default: far = l2p_loop(sl, q, x, y, z); break;
      }
      phi[(int64_t)d * ntp + j] += (double)far;
    }
  }
}

cudaError_t launch_l2p_f32(const DevGeom& G, const DevTaskLists& L, int64_t ntgt_pts, int ndp, const float* loc,
                           double* phi, cudaStream_t st) {
  if (L.n_p2p == 0) return cudaSuccess;
  k_l2p<<<L.n_p2p, kL2pThreads, 0, st>>>(G, L.p2p_leaf, L.tgt_cls, ntgt_pts, ndp, loc, phi);
  return cudaGetLastError();
}

// The hardware reciprocal square root (PTX rsqrt.approx.ftz.f32: maximum
// relative error about 2^-22.9, subnormal inputs and results flushed to
// zero).  Squared distances of distinct quadrature points lie far above the
// subnormal range; r^2 = 0 is selected out where it can occur, and the
// padding point's r^2 = inf gives 0.  Without the flush the compiler wraps
// the same instruction in a subnormal rescaling that costs several extra
// instructions per pair.
__device__ __forceinline__ float rsqrt_ftz(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void two_sum_f(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bb = s - hi;
  lo += (hi - (s - bb)) + (x - bb);
  hi = s;
}

// The packed pair loop over pairs [k0, k1) of a staged tile: per pair and
// target, three packed subtractions (the sources are stored negated), the
// packed r^2 (one multiply, two FMAs), two rsqrt and one packed FMA per
// density.  CHECK: the tile holds the target points themselves (r^2 = 0).
// w2: the weights of densities 1.. of pair k at w2[d - 1][k].
template <int ND, int TPT, int PAIRS, bool CHECK>
__device__ __forceinline__ void p2p_pairs_x2(const float4* __restrict__ xy, const float4* __restrict__ zw,
                                             const float2* __restrict__ w2, int k0, int k1, const float2 (&X)[TPT],
                                             const float2 (&Y)[TPT], const float2 (&Z)[TPT], float2 (&acc)[TPT][ND]) {
#pragma unroll(ND <= 4 ? 4 : 2)
  for (int k = k0; k < k1; ++k) {
    const float4 a = xy[k], c = zw[k];
    const float2 nx = make_float2(a.x, a.y), ny = make_float2(a.z, a.w), nz = make_float2(c.x, c.y);
    float2 ri[TPT];
#pragma unroll
    for (int u = 0; u < TPT; ++u) {
      const float2 dx = __fadd2_rn(X[u], nx), dy = __fadd2_rn(Y[u], ny), dz = __fadd2_rn(Z[u], nz);
      const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
      if constexpr (CHECK) ri[u] = make_float2(r2.x > 0.f ? rsqrt_ftz(r2.x) : 0.f, r2.y > 0.f ? rsqrt_ftz(r2.y) : 0.f);
      else ri[u] = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
      acc[u][0] = __ffma2_rn(make_float2(c.z, c.w), ri[u], acc[u][0]);
    }
#pragma unroll
    for (int d = 1; d < ND; ++d) {
      const float2 w = w2[(d - 1) * PAIRS + k];
#pragma unroll
      for (int u = 0; u < TPT; ++u) acc[u][d] = __ffma2_rn(w, ri[u], acc[u][d]);
    }
  }
}

// Packed form: TPT targets per thread (4 for one density, 1 for sixteen) and
// source points taken two at a time, every arithmetic instruction on a float2
// (the two sources of a pair: __fadd2_rn / __fmul2_rn / __ffma2_rn), so a
// target keeps two independent partial sums and the instructions issued per
// point pair nearly halve.  A tile of source points is staged pair-interleaved
// in shared memory, negated and relative to the target leaf's centre: xy[k] =
// (x0, x1, y0, y1), zw[k] = (z0, z1, w0, w1) for the pair k = (2k, 2k + 1), so
// one pair costs two 16-byte shared loads and 8 bytes per further density.
// Each of the NG thread groups takes a contiguous range of pairs (odd length,
// so two groups' loads in one quarter-warp fall in different banks) walked
// with unit stride.  An odd tile is padded with a weightless point at -1e30,
// whose distance overflows to inf (rsqrt 0).  Only the pairs that hold the
// leaf's own points (the first run of a VtV list) select r^2 = 0 out.  After
// the source loop all threads reduce the group sums, one target each.
// The weights of the densities after the first go straight to shared memory
// (4-byte cp.async), and from four densities on the compensated sums live there
// and are folded every other tile (130 products at most; the scalar form before
// had 256): the registers then hold enough targets that
// the shared-memory loads of the weights do not bound the loop.
template <int ND>
struct P2pShape {
  static constexpr int TPT = ND == 1 || ND == 4 ? 4 : 2;
  static constexpr int kTile = ND <= 4 ? 512 : 256;      // source points per tile
  static constexpr int kPairs = kTile / 2;
  static constexpr bool kSumsShared = ND >= 4;
  static constexpr int kFold = kSumsShared ? 2 : 1;      // tiles between folds (a tile: at most 65 products a sum, 129 for ND = 2)
  static constexpr int kW2 = ND > 1 ? 2 * (ND - 1) * kPairs : 0;     // float2
  static constexpr int kRed = ND * 128 * TPT;                        // float2
  // (the sums of fewer densities are laid over the weights at the end)
  static constexpr size_t smem = 2 * 2 * kPairs * sizeof(float4) +
                                 (kSumsShared ? kW2 + kRed : (kW2 > kRed ? kW2 : kRed)) * sizeof(float2);
};

// 4-byte asynchronous copy to shared memory
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

template <int ND>
__global__ void __launch_bounds__(128) k_p2p_f32x2(DevGeom G, DevTaskLists L, const float* __restrict__ W, int64_t nsp,
                                                   int64_t ntp, double* __restrict__ phi) {
  constexpr int TPT = P2pShape<ND>::TPT, kTile = P2pShape<ND>::kTile, kPairs = P2pShape<ND>::kPairs;
  constexpr bool SM = P2pShape<ND>::kSumsShared;
  constexpr int PPT = kPairs / 128;                // pairs loaded per thread per tile
  extern __shared__ __align__(16) unsigned char smraw[];
  float4(*sxy)[kPairs] = reinterpret_cast<float4(*)[kPairs]>(smraw);
  float4(*szw)[kPairs] = sxy + 2;
  float2* sw2 = reinterpret_cast<float2*>(szw + 2);            // weights of the further densities
  float2* red = SM ? sw2 + P2pShape<ND>::kW2 : sw2;            // group sums [ND][128 TPT]
  __shared__ int pre[kRunBatch + 1], rst[kRunBatch];
  const int b = blockIdx.x;
  const int leaf = L.sp_leaf[b];
  const int sc = L.src_cls, tc = L.tgt_cls;
  const float4 ch = G.box_hi[leaf], cl = G.box_lo[leaf];
  const float chx = ch.x, chy = ch.y, chz = ch.z, clx = cl.x, cly = cl.y, clz = cl.z;
  const int2 tr = G.box_rng[tc][leaf];
  const int nt = tr.y - tr.x;
  const int TS = (nt + TPT - 1) / TPT;
  const int NG = 128 / TS;
  const int ts = threadIdx.x % TS, gi_raw = threadIdx.x / TS;
  float2 X[TPT], Y[TPT], Z[TPT];
#pragma unroll
  for (int u = 0; u < TPT; ++u) {
    const int t = ts + u * TS;
    float xt = 1e30f, yt = 1e30f, zt = 1e30f;      // padding targets: far away, discarded
    if (t < nt) {
      const float4 h = G.pthi[tc][tr.x + t], l = G.ptlo[tc][tr.x + t];
      xt = (h.x - chx) + (l.x - clx);
      yt = (h.y - chy) + (l.y - cly);
      zt = (h.z - chz) + (l.z - clz);
    }
    X[u] = make_float2(xt, xt);
    Y[u] = make_float2(yt, yt);
    Z[u] = make_float2(zt, zt);
  }
  float shi[SM ? 1 : TPT][ND], slo[SM ? 1 : TPT][ND];
  float2 acc[TPT][ND];
#pragma unroll
  for (int u = 0; u < TPT; ++u)
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      acc[u][d] = make_float2(0.f, 0.f);
      if constexpr (SM) red[(d * TPT + u) * 128 + threadIdx.x] = make_float2(0.f, 0.f);
      else shi[u][d] = slo[u][d] = 0.f;
    }
  auto fold = [&]() {
#pragma unroll
    for (int u = 0; u < TPT; ++u)
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        if constexpr (SM) {
          float2 v = red[(d * TPT + u) * 128 + threadIdx.x];
          two_sum_f(v.x, v.y, acc[u][d].x);
          two_sum_f(v.x, v.y, acc[u][d].y);
          red[(d * TPT + u) * 128 + threadIdx.x] = v;
        } else {
          two_sum_f(shi[u][d], slo[u][d], acc[u][d].x);
          two_sum_f(shi[u][d], slo[u][d], acc[u][d].y);
        }
        acc[u][d] = make_float2(0.f, 0.f);
      }
  };
  int nfold = 0;
  const int r0 = L.sp_run_off[b], r1 = L.sp_run_off[b + 1];
  const int self_len = L.sp_self[b];
  float4 rxy[PPT], rzw[PPT];
  for (int rb = r0; rb < r1; rb += kRunBatch) {
    const int nr = min(kRunBatch, r1 - rb);
    __syncthreads();
    scan_runs(L.sp_runs + rb, nr, pre, rst);
    __syncthreads();
    const int total = pre[nr];
    const int ntiles = (total + kTile - 1) / kTile;
    // source point v of this batch (r: its run), negated, relative to the centre
    auto fetch = [&](int v, int r, float& x, float& y, float& z, float& w) {
      const int src = rst[r] + (v - pre[r]);
      const float4 h = G.pthi[sc][src], l = G.ptlo[sc][src];
      x = -((h.x - chx) + (l.x - clx));
      y = -((h.y - chy) + (l.y - cly));
      z = -((h.z - chz) + (l.z - clz));
      w = W[src];
      return src;
    };
    auto load_tile = [&](int t, int buf) {
#pragma unroll
      for (int q = 0; q < PPT; ++q) {
        const int k = threadIdx.x + q * 128, v0 = t * kTile + 2 * k;
        float x0 = 1e30f, y0 = 1e30f, z0 = 1e30f, w0 = 0.f;   // negated padding points
        float x1 = 1e30f, y1 = 1e30f, z1 = 1e30f, w1 = 0.f;
        int s0 = -1, s1 = -1;
        if (v0 < total) {
          int r = find_run(pre, nr, v0);
          s0 = fetch(v0, r, x0, y0, z0, w0);
          if (v0 + 1 < total) {
            while (r + 1 < nr && pre[r + 1] <= v0 + 1) ++r;
            s1 = fetch(v0 + 1, r, x1, y1, z1, w1);
          }
        }
        rxy[q] = make_float4(x0, x1, y0, y1);
        rzw[q] = make_float4(z0, z1, w0, w1);
        if constexpr (ND > 1) {
          float2* w = sw2 + buf * (ND - 1) * kPairs + k;
#pragma unroll
          for (int d = 1; d < ND; ++d, w += kPairs) {
            if (s0 >= 0) cp_async4(&w->x, W + d * nsp + s0); else w->x = 0.f;
            if (s1 >= 0) cp_async4(&w->y, W + d * nsp + s1); else w->y = 0.f;
          }
        }
      }
    };
    auto store_tile = [&](int buf) {
#pragma unroll
      for (int q = 0; q < PPT; ++q) {
        const int k = threadIdx.x + q * 128;
        sxy[buf][k] = rxy[q];
        szw[buf][k] = rzw[q];
      }
      if constexpr (ND > 1) asm volatile("cp.async.wait_all;" ::: "memory");
    };
    if (ntiles > 0) {
      load_tile(0, 0);
      store_tile(0);
    }
    __syncthreads();
    for (int t = 0; t < ntiles; ++t) {
      const int cur = t & 1;
      if (t + 1 < ntiles) load_tile(t + 1, cur ^ 1);
      const int m = min(kTile, total - t * kTile);
      const int mp = (m + 1) >> 1;
      // group gi_raw's contiguous pair range, odd length
      const int len = ((mp + NG - 1) / NG) | 1;
      const int k0 = gi_raw < NG ? min(gi_raw * len, mp) : mp;
      const int k1 = min(k0 + len, mp);
      // pairs that hold one of the leaf's own points (first run of a VtV list)
      const int ks = rb == r0 ? max(0, min(mp, (self_len - t * kTile + 1) >> 1)) : 0;
      const float2* w2 = sw2 + cur * (ND - 1) * kPairs;
      if (k0 < ks) p2p_pairs_x2<ND, TPT, kPairs, true>(sxy[cur], szw[cur], w2, k0, min(k1, ks), X, Y, Z, acc);
      p2p_pairs_x2<ND, TPT, kPairs, false>(sxy[cur], szw[cur], w2, max(k0, ks), k1, X, Y, Z, acc);
      if (++nfold == P2pShape<ND>::kFold) { fold(); nfold = 0; }
      if (t + 1 < ntiles) store_tile(cur ^ 1);
      __syncthreads();
    }
  }
  if constexpr (SM) {
    if (nfold) fold();
  } else {
#pragma unroll
    for (int u = 0; u < TPT; ++u)
#pragma unroll
      for (int d = 0; d < ND; ++d) red[(d * TPT + u) * 128 + threadIdx.x] = make_float2(shi[u][d], slo[u][d]);
  }
  __syncthreads();
  // every thread: one target, the group sums in group order; a chunk of a
  // split leaf stores them in its scratch row, and the leaf's last chunk
  // to finish adds the rows in chunk order
  const int2 grp = L.sp_grp[b];
  __shared__ int last_chunk;
  if (grp.x >= 0) {
    const int2 gi = L.grp_info[grp.x];
    float2* row = L.sp_scratch + (int64_t)(gi.x + grp.y) * ND * 128;
    for (int tt = threadIdx.x; tt < nt; tt += 128) {
      const int u = tt / TS, tsl = tt - u * TS;
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        float hi = 0.f, lo = 0.f;
        for (int g = 0; g < NG; ++g) {
          const float2 v = red[(d * TPT + u) * 128 + g * TS + tsl];
          two_sum_f(hi, lo, v.x);
          lo += v.y;
        }
        __stcg(row + d * 128 + tt, make_float2(hi, lo));
      }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      const unsigned ticket = atomicAdd(L.grp_cnt + grp.x, 1u);
      last_chunk = ticket + 1 == (unsigned)gi.y;
      if (last_chunk) L.grp_cnt[grp.x] = 0u;      // ready for the next launch
    }
    __syncthreads();
    if (!last_chunk) return;
    __threadfence();
  }
  for (int tt = threadIdx.x; tt < nt; tt += 128) {
    const int u = tt / TS, tsl = tt - u * TS;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      float hi = 0.f, lo = 0.f;
      if (grp.x < 0) {
        for (int g = 0; g < NG; ++g) {
          const float2 v = red[(d * TPT + u) * 128 + g * TS + tsl];
          two_sum_f(hi, lo, v.x);
          lo += v.y;
        }
      } else {
        const int2 gi = L.grp_info[grp.x];
        for (int c = 0; c < gi.y; ++c) {
          const float2 v = __ldcg(L.sp_scratch + (int64_t)(gi.x + c) * ND * 128 + d * 128 + tt);
          two_sum_f(hi, lo, v.x);
          lo += v.y;
        }
      }
      phi[(int64_t)d * ntp + tr.x + tt] = ((double)hi + (double)lo) * kInv4Pi;
    }
  }
}

// FP64 near field with L2P: a thread per target point, 128 / nt groups share the
// sources.  FP64 instructions bound it (some 14 a pair, two lanes a cycle and SM;
// the square root and a division took some twenty).  3,072-tet cube, 18.2 M pairs:
// 1.23 -> 0.56 ms (the target slots were padded to powers of two before); level-3
// ball, 816 M pairs, the whole evaluation 59.1 -> 29.7 ms.
template <int ND>
__global__ void __launch_bounds__(128) k_p2p_l2p_f64(DevGeom G, DevTaskLists L, const double* __restrict__ W,
                                                     int64_t nsp, int64_t ntp, int ndp,
                                                     const double* __restrict__ loc, double* __restrict__ phi) {
  constexpr int TL = kTile / 2;
  __shared__ double4_32a tile[TL];
  __shared__ double tw[ND > 1 ? ND - 1 : 1][TL];
  __shared__ int pre[kRunBatch + 1], rst[kRunBatch];
  __shared__ double red[ND][128];
  const int b = blockIdx.x;
  const int leaf = L.p2p_leaf[b];
  const int sc = L.src_cls, tc = L.tgt_cls;
  const double4_32a cs = G.box_cs[leaf];
  const int2 tr = G.box_rng[tc][leaf];
  const int nt = tr.y - tr.x;
  const int NG = 128 / nt;
  const int ti = threadIdx.x % nt, gi = threadIdx.x / nt;
  const bool active = gi < NG;
  double xt = 0, yt = 0, zt = 0;
  if (active) {
    const double4_32a x = G.pt64[tc][tr.x + ti];
    xt = x.x; yt = x.y; zt = x.z;
  }
  double acc[ND];
#pragma unroll
  for (int d = 0; d < ND; ++d) acc[d] = 0.0;
  const int r0 = L.run_off[b], r1 = L.run_off[b + 1];
  for (int rb = r0; rb < r1; rb += kRunBatch) {
    const int nr = min(kRunBatch, r1 - rb);
    __syncthreads();
    scan_runs(L.runs + rb, nr, pre, rst);
    __syncthreads();
    const int total = pre[nr];
    for (int j0 = 0; j0 < total; j0 += TL) {
      const int m = min(TL, total - j0);
      __syncthreads();
      for (int j = threadIdx.x; j < m; j += 128) {
        const int v = j0 + j;
        const int r = find_run(pre, nr, v);
        const int src = rst[r] + (v - pre[r]);
        const double4_32a y = G.pt64[sc][src];
        tile[j] = make_double4_32a(y.x, y.y, y.z, W[src]);
#pragma unroll
        for (int d = 1; d < ND; ++d) tw[d - 1][j] = W[(int64_t)d * nsp + src];
      }
      __syncthreads();
      if (active) {
        for (int j = gi; j < m; j += NG) {
          const double4_32a s = tile[j];
          const double dx = xt - s.x, dy = yt - s.y, dz = zt - s.z;
          const double r2 = dx * dx + dy * dy + dz * dz;
          // (an integer test: a comparison would go through the FP64 pipe)
          const double ri = (__double2hiint(r2) | __double2loint(r2)) ? rsqrt(r2) : 0.0;
          acc[0] += s.w * ri;
#pragma unroll
          for (int d = 1; d < ND; ++d) acc[d] += tw[d - 1][j] * ri;
        }
      }
    }
  }
#pragma unroll
  for (int d = 0; d < ND; ++d) red[d][threadIdx.x] = acc[d];
  __syncthreads();
  if (gi == 0 && active) {
    double near[ND];
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      double s = 0.0;
      for (int g = 0; g < NG; ++g) s += red[d][g * nt + ti];
      near[d] = s;
    }
    const double inv_s = 1.0 / cs.w;
    l2p_and_store<double, ND>(G, leaf, ndp, loc, (xt - cs.x) * inv_s, (yt - cs.y) * inv_s, (zt - cs.z) * inv_s, near,
                              tr.x + ti, ntp, phi);
  }
}

#define P2P_DISPATCH(KER, ...)                                               \
  switch (ndp) {                                                             \
    case 1: KER<1><<<L.n_p2p, 128, 0, st>>>(__VA_ARGS__); break;             \
    case 2: KER<2><<<L.n_p2p, 128, 0, st>>>(__VA_ARGS__); break;             \
    case 4: KER<4><<<L.n_p2p, 128, 0, st>>>(__VA_ARGS__); break;             \
    case 8: KER<8><<<L.n_p2p, 128, 0, st>>>(__VA_ARGS__); break;             \
    case 16: KER<16><<<L.n_p2p, 128, 0, st>>>(__VA_ARGS__); break;           \
    default: return cudaErrorInvalidValue;                                   \
  }

template <int ND>
cudaError_t launch_p2p_nd(const DevGeom& G, const DevTaskLists& L, const float* W, int64_t nsp, int64_t ntp, double* phi,
                          cudaStream_t st) {
  constexpr size_t sm = P2pShape<ND>::smem;
  if (sm > 44 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k_p2p_f32x2<ND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  k_p2p_f32x2<ND><<<L.sp_n, 128, sm, st>>>(G, L, W, nsp, ntp, phi);
  return cudaGetLastError();
}

cudaError_t launch_p2p_f32(const DevGeom& G, const DevTaskLists& L, const float* W, int64_t nsrc_pts, int64_t ntgt_pts,
                           int ndp, double* phi, cudaStream_t st) {
  if (L.n_p2p == 0) return cudaSuccess;
  switch (ndp) {
    case 1: return launch_p2p_nd<1>(G, L, W, nsrc_pts, ntgt_pts, phi, st);
    case 2: return launch_p2p_nd<2>(G, L, W, nsrc_pts, ntgt_pts, phi, st);
    case 4: return launch_p2p_nd<4>(G, L, W, nsrc_pts, ntgt_pts, phi, st);
    case 8: return launch_p2p_nd<8>(G, L, W, nsrc_pts, ntgt_pts, phi, st);
    case 16: return launch_p2p_nd<16>(G, L, W, nsrc_pts, ntgt_pts, phi, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_p2p_l2p_f64(const DevGeom& G, const DevTaskLists& L, const double* W, int64_t nsrc_pts,
                               int64_t ntgt_pts, int ndp, const double* loc, double* phi, cudaStream_t st) {
  if (L.n_p2p == 0) return cudaSuccess;
  P2P_DISPATCH(k_p2p_l2p_f64, G, L, W, nsrc_pts, ntgt_pts, ndp, loc, phi);
  return cudaGetLastError();
}


// ------------------------------------------- near corrections, Galerkin sums
// The near corrections read the densities only, so they run beside the
// expansions and the near field, and the Galerkin sums of the potentials are
// added at the end.
// LANES lanes per target element and density: out[d][e] = sum_k C[k] dens[d][col[k]].
// On large meshes the FP64 pipe bounds it (two lanes a cycle and SM, so
// sixteen cycles for any FP64 instruction of a warp): with a warp per element
// the five reduction steps cost nearly as much as the seven products of an
// average row (214 near pairs); with eight lanes four elements share three
// steps (level-4 ball, with the Galerkin sums: 190 -> 137 us).  On small ones it
// is latency, and a warp per element has the loads in flight sooner.
template <int LANES>
__global__ void __launch_bounds__(256) k_near_cor(DevTaskLists L, const double* __restrict__ dens,
                                                  const double* __restrict__ dens_dl, double* __restrict__ out) {
  const int64_t e = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / LANES;
  const int lane = threadIdx.x % LANES;
  const bool live = e < L.ntgt_el;
  const int64_t k0 = live ? L.cor_off[e] : 0, k1 = live ? L.cor_off[e + 1] : 0;
  const int64_t d = blockIdx.y;
  double s = 0.0;
#pragma unroll 8
  for (int64_t k = k0 + lane; k < k1; k += LANES) s += L.cor_val[k] * dens[d * L.nsrc_el + L.cor_col[k]];
  // BtV double layer: - (N - Q) of dG/dn_y times g
  if (dens_dl)
    for (int64_t k = k0 + lane; k < k1; k += LANES) s -= L.cor_val_dl[k] * dens_dl[d * L.nsrc_el + L.cor_col[k]];
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (live && lane == 0) out[d * L.ntgt_el + e] = s;
}

// out[d][e] += sum_q w_q phi[d][pos_q] (the points of an element have one weight)
__global__ void k_elem_add(DevTaskLists L, const double* __restrict__ phi, int64_t ntp, int ndens, double* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= L.ntgt_el * ndens) return;
  const int64_t d = i / L.ntgt_el, e = i - d * L.ntgt_el;
  const int4 pos = reinterpret_cast<const int4*>(L.elem_pts)[e];
  const double* ph = phi + d * ntp;
  double s = ph[pos.x] + ph[pos.y] + ph[pos.z];
  if (pos.w >= 0) s += ph[pos.w];
  out[i] += L.elem_w[e] * s;
}

cudaError_t launch_near_cor(const DevTaskLists& L, const double* dens_src, int ndens, double* out, cudaStream_t st,
                            const double* dens_dl) {
  if (L.ntgt_el == 0) return cudaSuccess;
  if (dens_dl && !L.cor_val_dl) return cudaErrorInvalidValue;
  // 65,536 elements at eight lanes fill the SMs' warps twice
  if (L.ntgt_el * ndens >= 65536)
    k_near_cor<8><<<dim3((unsigned)((L.ntgt_el * 8 + 255) / 256), ndens), 256, 0, st>>>(L, dens_src, dens_dl, out);
  else
    k_near_cor<32><<<dim3((unsigned)((L.ntgt_el * 32 + 255) / 256), ndens), 256, 0, st>>>(L, dens_src, dens_dl, out);
  return cudaGetLastError();
}

cudaError_t launch_elem_add(const DevTaskLists& L, const double* phi, int64_t ntgt_pts, int ndens, double* out, cudaStream_t st) {
  const int64_t n = L.ntgt_el * ndens;
  if (n == 0) return cudaSuccess;
  k_elem_add<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(L, phi, ntgt_pts, ndens, out);
  return cudaGetLastError();
}

// ------------------------------------------------- double layer (BtV)
// Moments of the double-layer density g (Algorithm 3: m^b includes
// - <gamma_1 (y - c)^b, g>; this pass adds that term).  Box-scaled, with
// u = (y - c)/s: n . grad_y (u^b) = (1/s) sum_i n_i b_i u^(b - e_i), so
// mhat^b -= (Wg_j / s) sum_i n_i b_i u_j^(b - e_i), Wg_j = w_j g(elem j),
// n the unit normal of point j's triangle.
template <typename T>
__global__ void k_p2m_dl(DevGeom G, const int* __restrict__ leaves, const T* __restrict__ W, int64_t nsp, int ndp,
                         T* __restrict__ mom) {
  extern __shared__ unsigned char smraw[];
  const int P = G.p, np = G.np;
  T* pw = reinterpret_cast<T*>(smraw);               // [3][P+1][64]
  T* wn = pw + 3 * (P + 1) * kPwS;                   // [ndp][3][64]: Wg n_i / s
  const int leaf = leaves[blockIdx.x];
  const double4_32a cs = G.box_cs[leaf];
  const int2 r = G.box_rng[1][leaf];
  const double inv_s = 1.0 / cs.w;
  for (int j0 = r.x; j0 < r.y; j0 += 64) {
    const int m = min(64, r.y - j0);
    __syncthreads();
    for (int j = threadIdx.x; j < m; j += blockDim.x) {
      const double4_32a y = G.pt64[1][j0 + j];
      const T d[3] = {(T)((y.x - cs.x) * inv_s), (T)((y.y - cs.y) * inv_s), (T)((y.z - cs.z) * inv_s)};
      for (int ax = 0; ax < 3; ++ax) {
        T v = (T)1;
        for (int k = 0; k <= P; ++k) { pw[(ax * (P + 1) + k) * kPwS + j] = v; v *= d[ax]; }
      }
      const double4_32a nr = G.tri_nrm[G.pt_elem[1][j0 + j]];
      for (int dd = 0; dd < ndp; ++dd) {
        const double wg = (double)W[(int64_t)dd * nsp + j0 + j] * inv_s;
        wn[(dd * 3 + 0) * 64 + j] = (T)(wg * nr.x);
        wn[(dd * 3 + 1) * 64 + j] = (T)(wg * nr.y);
        wn[(dd * 3 + 2) * 64 + j] = (T)(wg * nr.z);
      }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < np; q += blockDim.x) {
      const int mi = G.mi[q];
      const int a = mi & 255, b = (mi >> 8) & 255, c = (mi >> 16) & 255;
      const T* px = pw + (0 * (P + 1)) * kPwS;
      const T* py = pw + (1 * (P + 1)) * kPwS;
      const T* pz = pw + (2 * (P + 1)) * kPwS;
      for (int dd = 0; dd < ndp; ++dd) {
        const T* wx = wn + (dd * 3 + 0) * 64;
        const T* wy = wn + (dd * 3 + 1) * 64;
        const T* wz = wn + (dd * 3 + 2) * 64;
        T acc = 0;
        for (int j = 0; j < m; ++j) {
          T g = 0;
          if (a) g += (T)a * wx[j] * px[(a - 1) * kPwS + j] * py[b * kPwS + j] * pz[c * kPwS + j];
          if (b) g += (T)b * wy[j] * px[a * kPwS + j] * py[(b - 1) * kPwS + j] * pz[c * kPwS + j];
          if (c) g += (T)c * wz[j] * px[a * kPwS + j] * py[b * kPwS + j] * pz[(c - 1) * kPwS + j];
          acc += g;
        }
        mom[((int64_t)leaf * ndp + dd) * G.ms + q] -= acc;
      }
    }
  }
}

template <typename T>
cudaError_t launch_p2m_dl(const DevGeom& G, const DevTaskLists& L, const T* W, int64_t nsrc_pts, int ndp, T* mom,
                          cudaStream_t st) {
  if (L.n_p2m == 0) return cudaSuccess;
  const size_t sm = sizeof(T) * (3 * (G.p + 1) * kPwS + 3 * ndp * 64);
  k_p2m_dl<T><<<L.n_p2m, 128, sm, st>>>(G, L.p2m_leaf, W, nsrc_pts, ndp, mom);
  return cudaGetLastError();
}

// Near field of the double layer over the extended neighbour list:
// phi(x) -= (1/4pi) sum_j Wg_j n_j.(x - y_j) / |x - y_j|^3 for the leaf's
// target points, one CTA per target leaf, one target point per thread
// (chunks of 128 target points); sources stream through shared memory.
// FP32: leaf-frame double-float coordinates as in the single-layer pass,
// tile sums folded into FP64; FP64: plain.
template <typename T>
__global__ void __launch_bounds__(128) k_p2p_dl(DevGeom G, DevTaskLists L, const T* __restrict__ W, int64_t nsp,
                                                int64_t ntp, int ndp, double* __restrict__ phi) {
  constexpr int kT = 128;
  __shared__ T sx[kT], sy[kT], sz[kT], snx[kT], sny[kT], snz[kT];
  __shared__ int pre[kRunBatch + 1], rst[kRunBatch];
  const int b = blockIdx.x;
  const int leaf = L.p2p_leaf[b];
  const int tc = L.tgt_cls;
  const double4_32a cs = G.box_cs[leaf];
  float chx, clx, chy, cly, chz, clz;
  split_df(cs.x, chx, clx); split_df(cs.y, chy, cly); split_df(cs.z, chz, clz);
  const int2 tr = G.box_rng[tc][leaf];
  const int nt = tr.y - tr.x;
  const int r0 = L.run_off[b], r1 = L.run_off[b + 1];
  for (int t0 = 0; t0 < nt; t0 += kT) {
  const int t = t0 + threadIdx.x;
  const bool act = t < nt;
  T xt = 0, yt = 0, zt = 0;
  if (act) {
    if (sizeof(T) == 4) {
      const float4 h = G.pthi[tc][tr.x + t], l = G.ptlo[tc][tr.x + t];
      xt = (T)((h.x - chx) + (l.x - clx));
      yt = (T)((h.y - chy) + (l.y - cly));
      zt = (T)((h.z - chz) + (l.z - clz));
    } else {
      const double4_32a x = G.pt64[tc][tr.x + t];
      xt = (T)(x.x - cs.x); yt = (T)(x.y - cs.y); zt = (T)(x.z - cs.z);
    }
  }
  for (int d = 0; d < ndp; ++d) {
    double total = 0.0;
    for (int rb = r0; rb < r1; rb += kRunBatch) {
      const int nr = min(kRunBatch, r1 - rb);
      __syncthreads();
      scan_runs(L.runs + rb, nr, pre, rst);
      __syncthreads();
      const int cnt = pre[nr];
      for (int v0 = 0; v0 < cnt; v0 += kT) {
        const int m = min(kT, cnt - v0);
        __syncthreads();
        if (threadIdx.x < m) {
          const int v = v0 + threadIdx.x;
          const int rr = find_run(pre, nr, v);
          const int src = rst[rr] + (v - pre[rr]);
          T px, py, pz;
          if (sizeof(T) == 4) {
            const float4 h = G.pthi[1][src], l = G.ptlo[1][src];
            px = (T)((h.x - chx) + (l.x - clx));
            py = (T)((h.y - chy) + (l.y - cly));
            pz = (T)((h.z - chz) + (l.z - clz));
          } else {
            const double4_32a y = G.pt64[1][src];
            px = (T)(y.x - cs.x); py = (T)(y.y - cs.y); pz = (T)(y.z - cs.z);
          }
          const double4_32a nr3 = G.tri_nrm[G.pt_elem[1][src]];
          const T wg = W[(int64_t)d * nsp + src];
          sx[threadIdx.x] = px; sy[threadIdx.x] = py; sz[threadIdx.x] = pz;
          snx[threadIdx.x] = wg * (T)nr3.x; sny[threadIdx.x] = wg * (T)nr3.y; snz[threadIdx.x] = wg * (T)nr3.z;
        }
        __syncthreads();
        if (act) {
          T acc = 0;
          for (int j = 0; j < m; ++j) {
            const T dx = xt - sx[j], dy = yt - sy[j], dz = zt - sz[j];
            const T r2 = dx * dx + dy * dy + dz * dz;
            if (r2 > (T)0) {
              const T ri = (sizeof(T) == 4) ? (T)rsqrt_ftz((float)r2) : (T)rsqrt((double)r2);
              acc += (snx[j] * dx + sny[j] * dy + snz[j] * dz) * ri * ri * ri;
            }
          }
          total += (double)acc;
        }
      }
    }
    if (act) phi[(int64_t)d * ntp + tr.x + t] -= total * kInv4Pi;
  }
  }
}

template <typename T>
cudaError_t launch_p2p_dl(const DevGeom& G, const DevTaskLists& L, const T* W, int64_t nsrc_pts, int64_t ntgt_pts,
                          int ndp, double* phi, cudaStream_t st) {
  if (L.n_p2p == 0) return cudaSuccess;
  k_p2p_dl<T><<<L.n_p2p, 128, 0, st>>>(G, L, W, nsrc_pts, ntgt_pts, ndp, phi);
  return cudaGetLastError();
}

template cudaError_t launch_p2m_dl<float>(const DevGeom&, const DevTaskLists&, const float*, int64_t, int, float*, cudaStream_t);
template cudaError_t launch_p2m_dl<double>(const DevGeom&, const DevTaskLists&, const double*, int64_t, int, double*, cudaStream_t);
template cudaError_t launch_p2p_dl<float>(const DevGeom&, const DevTaskLists&, const float*, int64_t, int64_t, int, double*, cudaStream_t);
template cudaError_t launch_p2p_dl<double>(const DevGeom&, const DevTaskLists&, const double*, int64_t, int64_t, int, double*, cudaStream_t);

template cudaError_t launch_weights<float>(const DevGeom&, int, int64_t, const double*, int64_t, int, int, float*, cudaStream_t);
template cudaError_t launch_weights<double>(const DevGeom&, int, int64_t, const double*, int64_t, int, int, double*, cudaStream_t);
template cudaError_t launch_p2m<float>(const DevGeom&, const DevTaskLists&, const float*, int64_t, int, float*, cudaStream_t);
template cudaError_t launch_p2m<double>(const DevGeom&, const DevTaskLists&, const double*, int64_t, int, double*, cudaStream_t);
template cudaError_t launch_m2m<float>(const DevGeom&, const int*, int, int, int, float*, cudaStream_t);
template cudaError_t launch_m2m<double>(const DevGeom&, const int*, int, int, int, double*, cudaStream_t);
template cudaError_t launch_m2l_simt<float>(const DevGeom&, const DevTaskLists&, const float*, int, const float*, float*, cudaStream_t, const int*, int);
template cudaError_t launch_m2l_simt<double>(const DevGeom&, const DevTaskLists&, const double*, int, const double*, double*, cudaStream_t, const int*, int);
template cudaError_t launch_l2l<float>(const DevGeom&, const int2*, int, int, float*, cudaStream_t);
template cudaError_t launch_l2l<double>(const DevGeom&, const int2*, int, int, double*, cudaStream_t);

}  // namespace bcfmm
