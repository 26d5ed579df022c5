// Learned correction of near-singular element pairs (near pairs whose
// closures are apart).  The near field of Sec. 3.3 treats every near pair
// with an accurate rule; here a small network predicts, from the pair's
// relative geometry, corrections dw_ij of the product rule's 4 x 4 (or
// 4 x 3) weights:  C_ts ~ sum_ij dw_ij q_ij,  q_ij = W_i W_j / (4 pi r_ij).
//
//   features  the source vertices in the affine frame of the target,
//             centred at the target centroid (12 numbers; both vertex
//             orders canonical: by distance to the other element's centroid)
//   network   12 -> 64 -> 64 -> 16, exact GELU, BF16 weights, FP32 math
//   loss      (sum_ij dw_ij qhat_ij - chat)^2, qhat = q / Q, chat = C / Q,
//             Q = sum_ij q_ij (the pair's product-rule value)
//
// Parameter vector (FP32, 6032): W1[64][12] b1[64] W2[64][64] b2[64]
// W3[16][64] b3[16].  Training keeps FP32 master weights and runs the
// forward and backward passes on their BF16 roundings.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "kernels.cuh"
#include "mlp.cuh"

namespace bcfmm {

constexpr double kInv4PiM = 0.079577471545947667884441881686257;
constexpr int kMlpThreads = 128, kMlpSms = 152;        // (the chip's SMs)

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_d(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// ------------------------------------------------------------ geometry
struct D3 { double x, y, z; };
__device__ __forceinline__ D3 dsub(D3 a, D3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ double ddot(D3 a, D3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ D3 dcross(D3 a, D3 b) { return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x}; }

__device__ void load_elem(const double* V, int64_t e, int nv, D3* v) {
  for (int i = 0; i < nv; ++i) v[i] = {V[(e * nv + i) * 3], V[(e * nv + i) * 3 + 1], V[(e * nv + i) * 3 + 2]};
}

__device__ D3 centroid(const D3* v, int nv) {
  D3 c = {0, 0, 0};
  for (int i = 0; i < nv; ++i) { c.x += v[i].x; c.y += v[i].y; c.z += v[i].z; }
  return {c.x / nv, c.y / nv, c.z / nv};
}

__device__ double radius(const D3* v, int nv, D3 c) {
  double r = 0;
  for (int i = 0; i < nv; ++i) { D3 d = dsub(v[i], c); r = fmax(r, sqrt(ddot(d, d))); }
  return r;
}

// Lower bound of the distance between two convex elements (separating
// axes: face normals of both and cross products of edge pairs).  The true
// distance is at least the largest projected gap over any axis.
__device__ double sat_gap(const D3* a, int na, const D3* b, int nb) {
  const int tet_e[6][2] = {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}};
  const int tri_e[3][2] = {{0, 1}, {1, 2}, {0, 2}};
  const int tet_f[4][3] = {{1, 2, 3}, {0, 2, 3}, {0, 1, 3}, {0, 1, 2}};
  double best = -1e300;
  auto test = [&](D3 u) {
    const double l2 = ddot(u, u);
    if (!(l2 > 0)) return;
    const double s = 1.0 / sqrt(l2);
    double amin = 1e300, amax = -1e300, bmin = 1e300, bmax = -1e300;
    for (int i = 0; i < na; ++i) { const double p = ddot(a[i], u) * s; amin = fmin(amin, p); amax = fmax(amax, p); }
    for (int i = 0; i < nb; ++i) { const double p = ddot(b[i], u) * s; bmin = fmin(bmin, p); bmax = fmax(bmax, p); }
    best = fmax(best, fmax(bmin - amax, amin - bmax));
  };
  const int nfa = na == 4 ? 4 : 1, nfb = nb == 4 ? 4 : 1;
  for (int f = 0; f < nfa; ++f) {
    const int* F = na == 4 ? tet_f[f] : tet_f[3];
    test(dcross(dsub(a[F[1]], a[F[0]]), dsub(a[F[2]], a[F[0]])));
  }
  for (int f = 0; f < nfb; ++f) {
    const int* F = nb == 4 ? tet_f[f] : tet_f[3];
    test(dcross(dsub(b[F[1]], b[F[0]]), dsub(b[F[2]], b[F[0]])));
  }
  const int nea = na == 4 ? 6 : 3, neb = nb == 4 ? 6 : 3;
  for (int i = 0; i < nea; ++i) {
    const int* E = na == 4 ? tet_e[i] : tri_e[i];
    const D3 ea = dsub(a[E[1]], a[E[0]]);
    for (int j = 0; j < neb; ++j) {
      const int* G = nb == 4 ? tet_e[j] : tri_e[j];
      const D3 u = dcross(ea, dsub(b[G[1]], b[G[0]]));
      if (ddot(u, u) > 1e-24 * ddot(ea, ea) * ddot(ea, ea)) test(u);
    }
  }
  return best;
}

// calibration bin of a near-singular pair: centroid distance over the
// radius sum (8 bins on [0,1)) x gap lower bound over the radius sum
// (4 bins: [0,.05) [.05,.15) [.15,.3) [.3,inf))
__device__ int pair_bin(double dist_ratio, double gap_ratio) {
  const int a = min(kMlpBinsEta - 1, max(0, (int)(dist_ratio * kMlpBinsEta)));
  const int b = gap_ratio < 0.05 ? 0 : (gap_ratio < 0.15 ? 1 : (gap_ratio < 0.3 ? 2 : 3));
  return a * kMlpBinsGap + b;
}

// Features, normalised product-rule terms and Q of one pair.
//   tgt (nvt vertices), src (nvs vertices); quadrature point k of an
//   element carries the largest barycentric weight at vertex k.
__device__ void pair_features(const D3* tv_in, int nvt, double tvol, const D3* sv_in, int nvs, double svol,
                              float* feat, float* qhat, double* Q) {
  const D3 ct = centroid(tv_in, nvt), cs = centroid(sv_in, nvs);
  // canonical vertex orders: by distance to the other element's centroid
  int pt[4] = {0, 1, 2, 3}, ps[4] = {0, 1, 2, 3};
  double dt[4], ds[4];
  // (squared distances rounded as written, no fused multiply-add: equal
  // distances of symmetric configurations stay exactly equal, so ties keep
  // the input order on every machine)
  auto d2 = [](D3 d) { return __dadd_rn(__dadd_rn(__dmul_rn(d.x, d.x), __dmul_rn(d.y, d.y)), __dmul_rn(d.z, d.z)); };
  for (int i = 0; i < nvt; ++i) dt[i] = d2(dsub(tv_in[i], cs));
  for (int i = 0; i < nvs; ++i) ds[i] = d2(dsub(sv_in[i], ct));
  for (int i = 1; i < nvt; ++i)
    for (int j = i; j > 0 && dt[pt[j]] < dt[pt[j - 1]]; --j) { int t = pt[j]; pt[j] = pt[j - 1]; pt[j - 1] = t; }
  for (int i = 1; i < nvs; ++i)
    for (int j = i; j > 0 && ds[ps[j]] < ds[ps[j - 1]]; --j) { int t = ps[j]; ps[j] = ps[j - 1]; ps[j - 1] = t; }
  D3 tv[4], sv[4];
  for (int i = 0; i < nvt; ++i) tv[i] = tv_in[pt[i]];
  for (int i = 0; i < nvs; ++i) sv[i] = sv_in[ps[i]];
  // target frame columns a0, a1, a2
  D3 a0 = dsub(tv[1], tv[0]), a1 = dsub(tv[2], tv[0]), a2;
  if (nvt == 4) {
    a2 = dsub(tv[3], tv[0]);
  } else {
    D3 n = dcross(a0, a1);
    const double nn = sqrt(ddot(n, n));
    const double s = sqrt(nn) / nn;                // unit normal times sqrt(2 area)
    n = {n.x * s, n.y * s, n.z * s};
    if (ddot(n, dsub(cs, ct)) < 0) n = {-n.x, -n.y, -n.z};
    a2 = n;
  }
  // inverse of [a0 a1 a2] by cofactors
  const D3 c0 = dcross(a1, a2), c1 = dcross(a2, a0), c2 = dcross(a0, a1);
  const double det = ddot(a0, c0);
  const double id = 1.0 / det;
  for (int k = 0; k < 4; ++k) {
    if (k < nvs) {
      const D3 r = dsub(sv[k], ct);
      feat[3 * k] = (float)(ddot(c0, r) * id);
      feat[3 * k + 1] = (float)(ddot(c1, r) * id);
      feat[3 * k + 2] = (float)(ddot(c2, r) * id);
    } else {
      feat[3 * k] = feat[3 * k + 1] = feat[3 * k + 2] = 0.f;
    }
  }
  // quadrature points in the canonical orders and the product-rule terms
  const double ta = (5.0 + 3.0 * sqrt(5.0)) / 20.0, tb = (5.0 - sqrt(5.0)) / 20.0;
  D3 xq[4], yq[4];
  for (int q = 0; q < nvt; ++q) {
    D3 s = {0, 0, 0};
    for (int i = 0; i < nvt; ++i) {
      const double w = nvt == 4 ? (i == q ? ta : tb) : (i == q ? 2.0 / 3.0 : 1.0 / 6.0);
      s.x += w * tv[i].x; s.y += w * tv[i].y; s.z += w * tv[i].z;
    }
    xq[q] = s;
  }
  for (int q = 0; q < nvs; ++q) {
    D3 s = {0, 0, 0};
    for (int i = 0; i < nvs; ++i) {
      const double w = nvs == 4 ? (i == q ? ta : tb) : (i == q ? 2.0 / 3.0 : 1.0 / 6.0);
      s.x += w * sv[i].x; s.y += w * sv[i].y; s.z += w * sv[i].z;
    }
    yq[q] = s;
  }
  const double wt = tvol / nvt, ws = svol / nvs;
  double q[16], sum = 0.0;
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) {
      double v = 0.0;
      if (i < nvt && j < nvs) {
        const D3 d = dsub(xq[i], yq[j]);
        const double r = sqrt(ddot(d, d));
        v = r > 0 ? wt * ws * kInv4PiM / r : 0.0;
      }
      q[4 * i + j] = v;
      sum += v;
    }
  *Q = sum;
  for (int k = 0; k < 16; ++k) qhat[k] = (float)(q[k] / sum);
}

__device__ double elem_size(const D3* v, int nv) {
  const D3 n = dcross(dsub(v[1], v[0]), dsub(v[2], v[0]));
  if (nv == 3) return 0.5 * sqrt(ddot(n, n));
  return fabs(ddot(n, dsub(v[3], v[0]))) / 6.0;
}

// ------------------------------------------------------------ network
// forward on BF16-rounded weights held in shared memory (FP32 storage)
__device__ float mlp_forward(const float* __restrict__ P, const float* x, const float* qhat) {
  float h1[kMlpH];
  for (int j = 0; j < kMlpH; ++j) {
    float s = P[kOffB1 + j];
#pragma unroll
    for (int k = 0; k < kMlpIn; ++k) s = fmaf(P[kOffW1 + j * kMlpIn + k], x[k], s);
    h1[j] = gelu(s);
  }
  float pred = 0.f;
  float h2[kMlpH];
  for (int j = 0; j < kMlpH; ++j) {
    float s = P[kOffB2 + j];
    for (int k = 0; k < kMlpH; ++k) s = fmaf(P[kOffW2 + j * kMlpH + k], h1[k], s);
    h2[j] = gelu(s);
  }
  for (int o = 0; o < kMlpOut; ++o) {
    float s = P[kOffB3 + o];
    for (int k = 0; k < kMlpH; ++k) s = fmaf(P[kOffW3 + o * kMlpH + k], h2[k], s);
    pred = fmaf(s, qhat[o], pred);
  }
  return pred;
}

__device__ void load_params_bf16(const float* __restrict__ src, float* dst) {
  for (int i = threadIdx.x; i < kMlpParams; i += blockDim.x) dst[i] = bf16r(src[i]);
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Mean loss and its gradient over n pairs (added with atomics to grad and
// loss, which k_mlp_zero cleared).  A minibatch is small (about a thousand
// pairs), so latency is the bound: a CTA takes P pairs and shares every layer
// among its NT threads, activations and weights in shared memory: 8 pairs with 256
// threads, 32 with 512, or, where they outnumber the SMs, 32 with 256.  With v =
// W3^T qhat the output layer is two dot products (pred = v.h2 + b3.qhat) and its
// backward pass is v itself: dz2 = dpred v gelu'(z2).
// The sums of a cluster's CTAs are added in FP64 through distributed shared
// memory, each CTA a share of the parameters, so that one atomic per parameter
// serves a whole cluster: every FP32 addition to a running gradient rounds it, and
// with an atomic per CTA 1,024 pairs were off by 1.9e-7 of the norm (against FP64
// autograd), twice as much as with one pair per thread in eight CTAs.  Sixteen CTAs
// of 32 pairs make two clusters of 1,024 pairs, the minibatch of a training; two
// additions to zero give the same sum in either order, so that a training repeats
// bit for bit.
// On the device: 1,024 pairs 111 us with one pair per thread (eight CTAs,
// activations in local memory), 19.3 us with an atomic per CTA, 18.2 us now; the
// gradient and the Adam step with the copies of a caller that keeps its state: 131
// us with one pair per thread, 56 us now, most of it the host's calls.
constexpr int kGradCluster = 16;                       // CTAs (opt-in; eight where the device refuses it)
constexpr int kLdW2 = kMlpH + 1;                       // padded rows: W2 is read along both indexes

template <int P>
struct GradShared {
  float W1[kMlpIn][kMlpH];                             // transposed: [k][j]
  float W2[kMlpH][kLdW2];                              // [j][k]
  float W3[kMlpOut][kMlpH];
  float b1[kMlpH], b2[kMlpH], b3[kMlpOut];
  float x[P][kMlpIn], qh[P][kMlpOut];
  float h1[P][kMlpH], d1[P][kMlpH];                    // gelu, gelu' of layer 1 (d1: then dz1)
  float h2[P][kMlpH], d2[P][kMlpH];                    // of layer 2 (d2: then dz2)
  float v[P][kMlpH];
  float part[2][P], dpred[P];
};

template <int P, int NT>
__global__ void __launch_bounds__(NT) k_mlp_grad(const float* __restrict__ params, const float* __restrict__ feat,
                                                           const float* __restrict__ qhat, const float* __restrict__ chat,
                                                           int64_t n, float inv_n, float* __restrict__ grad,
                                                           float* __restrict__ loss) {
  extern __shared__ __align__(16) unsigned char smraw[];
  GradShared<P>& S = *reinterpret_cast<GradShared<P>*>(smraw);
  // the CTA's gradient and loss, in the place of the weights once they are used up
  float* Gs = reinterpret_cast<float*>(smraw);
  static_assert(offsetof(GradShared<P>, x) >= (kMlpParams + 1) * sizeof(float), "gradient over the weights");
  const int tid = threadIdx.x, j = tid & 63, g = tid >> 6;      // unit, group: a share of the pairs
  const int64_t i0 = (int64_t)blockIdx.x * P;
  constexpr int NG = NT / 64, PQ = P / NG;
  constexpr int R2 = kMlpH / NG, R3 = kMlpOut / NG;             // rows of dW2, dW3 per group
  for (int i = tid; i < kMlpH * kMlpIn; i += NT) S.W1[i % kMlpIn][i / kMlpIn] = bf16r(params[kOffW1 + i]);
  for (int i = tid; i < kMlpH * kMlpH; i += NT) S.W2[i / kMlpH][i % kMlpH] = bf16r(params[kOffW2 + i]);
  for (int i = tid; i < kMlpOut * kMlpH; i += NT) S.W3[i / kMlpH][i % kMlpH] = bf16r(params[kOffW3 + i]);
  if (tid < kMlpH) { S.b1[tid] = bf16r(params[kOffB1 + tid]); S.b2[tid] = bf16r(params[kOffB2 + tid]); }
  if (tid < kMlpOut) S.b3[tid] = bf16r(params[kOffB3 + tid]);
  for (int i = tid; i < P * kMlpIn; i += NT) S.x[i / kMlpIn][i % kMlpIn] = i0 + i / kMlpIn < n ? feat[i0 * kMlpIn + i] : 0.f;
  for (int i = tid; i < P * kMlpOut; i += NT) S.qh[i / kMlpOut][i % kMlpOut] = i0 + i / kMlpOut < n ? qhat[i0 * kMlpOut + i] : 0.f;
  __syncthreads();
  // layer 1 and v
#pragma unroll 2
  for (int q = 0; q < PQ; ++q) {
    const int p = g * PQ + q;
    float z = S.b1[j], v = 0.f;
#pragma unroll
    for (int k = 0; k < kMlpIn; ++k) z = fmaf(S.W1[k][j], S.x[p][k], z);
#pragma unroll
    for (int o = 0; o < kMlpOut; ++o) v = fmaf(S.W3[o][j], S.qh[p][o], v);
    S.h1[p][j] = gelu(z);
    S.d1[p][j] = gelu_d(z);
    S.v[p][j] = v;
  }
  __syncthreads();
  // layer 2 and pred
  {
    float z[PQ];
#pragma unroll
    for (int q = 0; q < PQ; ++q) z[q] = S.b2[j];
    for (int k = 0; k < kMlpH; k += 4) {
      float w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) w[i] = S.W2[j][k + i];
#pragma unroll
      for (int q = 0; q < PQ; ++q) {
        const float4 h = *reinterpret_cast<const float4*>(&S.h1[g * PQ + q][k]);
        z[q] = fmaf(w[0], h.x, z[q]);
        z[q] = fmaf(w[1], h.y, z[q]);
        z[q] = fmaf(w[2], h.z, z[q]);
        z[q] = fmaf(w[3], h.w, z[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < PQ; ++q) {
      const int p = g * PQ + q;
      const float h = gelu(z[q]);
      S.h2[p][j] = h;
      S.d2[p][j] = gelu_d(z[q]);
      const float t = warp_sum(h * S.v[p][j]);
      if ((tid & 31) == 0) S.part[(tid >> 5) & 1][p] = t;
    }
  }
  __syncthreads();
  float cta_loss = 0.f;
  if (tid < 32) {
    float l = 0.f;
    for (int p = tid; p < P; p += 32) {
      float pred = S.part[0][p] + S.part[1][p];
#pragma unroll
      for (int o = 0; o < kMlpOut; ++o) pred = fmaf(S.b3[o], S.qh[p][o], pred);
      const float e = i0 + p < n ? pred - chat[i0 + p] : 0.f;
      S.dpred[p] = 2.f * e * inv_n;
      l = fmaf(e * e, inv_n, l);
    }
    cta_loss = warp_sum(l);
  }
  __syncthreads();
  // dz2 = dpred v gelu'(z2)
#pragma unroll
  for (int q = 0; q < PQ; ++q) {
    const int p = g * PQ + q;
    S.d2[p][j] *= S.dpred[p] * S.v[p][j];
  }
  __syncthreads();
  // dz1 = (W2^T dz2) gelu'(z1); dW3, db3, dW2, db2
  {
    float t[PQ];
#pragma unroll
    for (int q = 0; q < PQ; ++q) t[q] = 0.f;
    for (int k = 0; k < kMlpH; k += 4) {
      float w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) w[i] = S.W2[k + i][j];
#pragma unroll
      for (int q = 0; q < PQ; ++q) {
        const float4 d = *reinterpret_cast<const float4*>(&S.d2[g * PQ + q][k]);
        t[q] = fmaf(w[0], d.x, t[q]);
        t[q] = fmaf(w[1], d.y, t[q]);
        t[q] = fmaf(w[2], d.z, t[q]);
        t[q] = fmaf(w[3], d.w, t[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < PQ; ++q) S.d1[g * PQ + q][j] *= t[q];
  }
  __syncthreads();
  {
    float a[R2], c[R3];                         // dW2[R2 g + i][j], dW3[R3 g + i][j]
#pragma unroll
    for (int i = 0; i < R2; ++i) a[i] = 0.f;
#pragma unroll
    for (int i = 0; i < R3; ++i) c[i] = 0.f;
    for (int p = 0; p < P; ++p) {
      const float h = S.h1[p][j], u = S.h2[p][j] * S.dpred[p];
#pragma unroll
      for (int i = 0; i < R2; i += 4) {
        const float4 d = *reinterpret_cast<const float4*>(&S.d2[p][R2 * g + i]);
        a[i] = fmaf(d.x, h, a[i]);
        a[i + 1] = fmaf(d.y, h, a[i + 1]);
        a[i + 2] = fmaf(d.z, h, a[i + 2]);
        a[i + 3] = fmaf(d.w, h, a[i + 3]);
      }
#pragma unroll
      for (int i = 0; i < R3; ++i) c[i] = fmaf(S.qh[p][R3 * g + i], u, c[i]);
    }
#pragma unroll
    for (int i = 0; i < R2; ++i) Gs[kOffW2 + (R2 * g + i) * kMlpH + j] = a[i];
#pragma unroll
    for (int i = 0; i < R3; ++i) Gs[kOffW3 + (R3 * g + i) * kMlpH + j] = c[i];
    if (g == 0) {
      float t = 0.f;
      for (int p = 0; p < P; ++p) t += S.d2[p][j];
      Gs[kOffB2 + j] = t;
    } else if (g == 1 && j < kMlpOut) {
      float t = 0.f;
      for (int p = 0; p < P; ++p) t = fmaf(S.dpred[p], S.qh[p][j], t);
      Gs[kOffB3 + j] = t;
    }
  }
  // dW1[j][3 g + i] (four groups), db1
  if (g < 4) {
    float a[3] = {0.f, 0.f, 0.f}, t = 0.f;
    for (int p = 0; p < P; ++p) {
      const float d = S.d1[p][j];
      t += d;
#pragma unroll
      for (int i = 0; i < 3; ++i) a[i] = fmaf(d, S.x[p][3 * g + i], a[i]);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) Gs[kOffW1 + j * kMlpIn + 3 * g + i] = a[i];
    if (g == 0) Gs[kOffB1 + j] = t;
  }
  if (tid == 0) Gs[kMlpParams] = cta_loss;
  // the cluster's sums
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  const int nc = (int)cl.num_blocks(), slice = kMlpParams / nc + 1;
  const int r0 = (int)cl.block_rank() * slice, r1 = min(r0 + slice, kMlpParams + 1);
  for (int i = r0 + tid; i < r1; i += NT) {
    double t = 0.0;
#pragma unroll 8
    for (int c = 0; c < nc; ++c) t += (double)cl.map_shared_rank(Gs, c)[i];
    atomicAdd(i < kMlpParams ? &grad[i] : loss, (float)t);
  }
  cl.sync();                                     // (the others read this CTA's shared memory)
}

__global__ void k_mlp_zero(float* __restrict__ grad, float* __restrict__ loss) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < kMlpParams) grad[i] = 0.f;
  if (i == kMlpParams) *loss = 0.f;
}

__global__ void k_mlp_adam(float* __restrict__ params, const float* __restrict__ grad, float* __restrict__ m1,
                           float* __restrict__ m2, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kMlpParams) return;
  const float g = grad[i];
  const float a = b1 * m1[i] + (1.f - b1) * g;
  const float b = b2 * m2[i] + (1.f - b2) * g * g;
  m1[i] = a;
  m2[i] = b;
  params[i] -= lr * (a * c1) / (sqrtf(b * c2) + eps);
}

// Predictions of n pairs: a CTA takes P pairs, every layer as a register-tiled
// product out[64][P] (a thread: four units by P / 16 pairs; per input index one
// 16-byte load of weights and PT / 4 of activations for 4 PT FMAs), activations
// transposed in shared memory.  As in the gradient, v = W3^T qhat replaces the
// output layer.  Bound by the FMA pipe and the 128 error functions a pair:
// 200,000 pairs 151 us with one pair per thread, 90 us now.
// A thread's units are jg + 16 i (the weights are stored in that order), and
// activation rows are padded by four floats: the sixteen threads that share
// pairs then store to different banks.
constexpr int kPredThreads = 256;
template <int P>
struct PredShared {
  float W1[kMlpIn][kMlpH], W2[kMlpH][kMlpH], W3[kMlpOut][kMlpH];   // [input][pred_unit(unit)]
  float b1[kMlpH], b2[kMlpH], b3[kMlpOut];
  float x[kMlpIn][P + 4], qh[kMlpOut][P + 4], h1[kMlpH][P + 4];
};
__device__ __forceinline__ int pred_unit(int j) { return (j & 15) * 4 + (j >> 4); }

// acc[i][p] += sum_k W[k][4 jg + i] A[k][p0 + p]
template <int K, int LDA, int PT>
__device__ __forceinline__ void tile_product(const float (*W)[kMlpH], const float (*A)[LDA], int jg, int p0, float (&acc)[4][PT]) {
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    const float4 w = *reinterpret_cast<const float4*>(&W[k][4 * jg]);
    float a[PT];
#pragma unroll
    for (int p = 0; p < PT; p += (PT >= 4 ? 4 : 2)) {
      if constexpr (PT >= 4) *reinterpret_cast<float4*>(a + p) = *reinterpret_cast<const float4*>(&A[k][p0 + p]);
      else *reinterpret_cast<float2*>(a + p) = *reinterpret_cast<const float2*>(&A[k][p0 + p]);
    }
#pragma unroll
    for (int p = 0; p < PT; ++p) {
      acc[0][p] = fmaf(w.x, a[p], acc[0][p]);
      acc[1][p] = fmaf(w.y, a[p], acc[1][p]);
      acc[2][p] = fmaf(w.z, a[p], acc[2][p]);
      acc[3][p] = fmaf(w.w, a[p], acc[3][p]);
    }
  }
}

template <int P>
__global__ void __launch_bounds__(kPredThreads) k_mlp_predict(const float* __restrict__ params, const float* __restrict__ feat,
                                                              const float* __restrict__ qhat, int64_t n,
                                                              float* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smraw[];
  PredShared<P>& S = *reinterpret_cast<PredShared<P>*>(smraw);
  constexpr int PT = P / 16;
  const int tid = threadIdx.x, jg = tid & 15, p0 = (tid >> 4) * PT;
  for (int i = tid; i < kMlpH * kMlpIn; i += kPredThreads) S.W1[i % kMlpIn][pred_unit(i / kMlpIn)] = bf16r(params[kOffW1 + i]);
  for (int i = tid; i < kMlpH * kMlpH; i += kPredThreads) S.W2[i % kMlpH][pred_unit(i / kMlpH)] = bf16r(params[kOffW2 + i]);
  for (int i = tid; i < kMlpOut * kMlpH; i += kPredThreads) S.W3[i / kMlpH][pred_unit(i % kMlpH)] = bf16r(params[kOffW3 + i]);
  if (tid < kMlpH) { S.b1[pred_unit(tid)] = bf16r(params[kOffB1 + tid]); S.b2[pred_unit(tid)] = bf16r(params[kOffB2 + tid]); }
  if (tid < kMlpOut) S.b3[tid] = bf16r(params[kOffB3 + tid]);
  for (int64_t i0 = (int64_t)blockIdx.x * P; i0 < n; i0 += (int64_t)gridDim.x * P) {
    __syncthreads();
    for (int i = tid; i < P * kMlpIn; i += kPredThreads) S.x[i % kMlpIn][i / kMlpIn] = i0 + i / kMlpIn < n ? feat[i0 * kMlpIn + i] : 0.f;
    for (int i = tid; i < P * kMlpOut; i += kPredThreads) S.qh[i % kMlpOut][i / kMlpOut] = i0 + i / kMlpOut < n ? qhat[i0 * kMlpOut + i] : 0.f;
    __syncthreads();
    float z[4][PT], v[4][PT];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int p = 0; p < PT; ++p) z[i][p] = S.b1[4 * jg + i];
    tile_product<kMlpIn>(S.W1, S.x, jg, p0, z);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int p = 0; p < PT; ++p) {
        z[i][p] = gelu(z[i][p]);
        v[i][p] = 0.f;
      }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int p = 0; p < PT; p += 2) {
        *reinterpret_cast<float2*>(&S.h1[jg + 16 * i][p0 + p]) = make_float2(z[i][p], z[i][p + 1]);
        z[i][p] = z[i][p + 1] = S.b2[4 * jg + i];
      }
    tile_product<kMlpOut>(S.W3, S.qh, jg, p0, v);
    __syncthreads();
    tile_product<kMlpH>(S.W2, S.h1, jg, p0, z);
#pragma unroll
    for (int p = 0; p < PT; ++p) {
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) s = fmaf(gelu(z[i][p]), v[i][p], s);
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (jg == 0 && i0 + p0 + p < n) {
#pragma unroll
        for (int o = 0; o < kMlpOut; ++o) s = fmaf(S.b3[o], S.qh[o][p0 + p], s);
        out[i0 + p0 + p] = s;
      }
    }
  }
}

// ------------------------------------------------------- setup passes
// Classify every near pair k (CSR position): touching (gap bound <= 1e-9
// of the radius sum) -> FP64 near rule; near-singular -> its bit set in
// `singular` (bit k % 32 of word k / 32) and, by mode, appended to the learned
// list (its bin's calibrated error <= tol), the FP64 list (bin rejected), or
// nowhere (mode 2: product rule only).
__global__ void k_near_classify(int task, int64_t nnz, const int* __restrict__ row, const int* __restrict__ col,
                                const double* __restrict__ tgt_v, const double* __restrict__ src_v, int mode,
                                const float* __restrict__ eps_tab, float tol, int64_t* __restrict__ lists,
                                unsigned long long* __restrict__ counts, int64_t cap, unsigned* __restrict__ singular) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const unsigned in = __ballot_sync(0xffffffffu, k < nnz);
  if (k >= nnz) return;
  const int nvt = task == 1 ? 3 : 4, nvs = task == 2 ? 3 : 4;
  D3 tv[4], sv[4];
  load_elem(tgt_v, row[k], nvt, tv);
  load_elem(src_v, col[k], nvs, sv);
  const D3 ct = centroid(tv, nvt), cs = centroid(sv, nvs);
  const double rs = radius(tv, nvt, ct) + radius(sv, nvs, cs);
  const double gap = sat_gap(tv, nvt, sv, nvs);
  int cls;                                   // 0 FP64 list, 1 learned list, 2 none
  const bool touching = gap <= 1e-9 * rs;
  const unsigned bits = __ballot_sync(in, !touching);
  if ((threadIdx.x & 31) == 0) singular[k >> 5] = bits;
  if (touching) {
    cls = 0;
  } else {
    if (mode == 2) {
      cls = 2;
    } else {
      const D3 d = dsub(ct, cs);
      const int b = pair_bin(sqrt(ddot(d, d)) / rs, gap / rs);
      cls = (eps_tab != nullptr && eps_tab[b] <= tol) ? 1 : 0;
    }
  }
  if (cls < 2) {
    const unsigned long long s = atomicAdd(&counts[cls], 1ull);
    if ((int64_t)s < cap) lists[cls * cap + s] = k;
  }
}

// Fused learned correction of the pairs in sel[0..n): geometry, features,
// network (BF16 weights in shared memory, FP32 accumulation) and the
// contraction with the product-rule terms; writes C_ts = Q sum dw qhat.
__global__ void __launch_bounds__(kMlpThreads) k_near_mlp(int task, const int64_t* __restrict__ sel, int64_t n,
                                                          const int* __restrict__ row, const int* __restrict__ col,
                                                          const double* __restrict__ tgt_v,
                                                          const double* __restrict__ src_v,
                                                          const float* __restrict__ params,
                                                          double* __restrict__ cor_val) {
  __shared__ float P[kMlpParams];
  load_params_bf16(params, P);
  __syncthreads();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t k = sel[i];
  const int nvt = task == 1 ? 3 : 4, nvs = task == 2 ? 3 : 4;
  D3 tv[4], sv[4];
  load_elem(tgt_v, row[k], nvt, tv);
  load_elem(src_v, col[k], nvs, sv);
  float x[kMlpIn], qh[kMlpOut];
  double Q;
  pair_features(tv, nvt, elem_size(tv, nvt), sv, nvs, elem_size(sv, nvs), x, qh, &Q);
  cor_val[k] = Q * (double)mlp_forward(P, x, qh);
}

// Training / validation data of the pairs sel[0..n): features, qhat, Q,
// calibration bin (labels come from the FP64 near rule separately).
__global__ void k_pair_data(int task, const int64_t* __restrict__ sel, int64_t n, const int* __restrict__ row,
                            const int* __restrict__ col, const double* __restrict__ tgt_v,
                            const double* __restrict__ src_v, float* __restrict__ feat, float* __restrict__ qhat,
                            double* __restrict__ Q, int* __restrict__ bin, int* __restrict__ pairs) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t k = sel[i];
  if (pairs) { pairs[2 * i] = row[k]; pairs[2 * i + 1] = col[k]; }
  const int nvt = task == 1 ? 3 : 4, nvs = task == 2 ? 3 : 4;
  D3 tv[4], sv[4];
  load_elem(tgt_v, row[k], nvt, tv);
  load_elem(src_v, col[k], nvs, sv);
  pair_features(tv, nvt, elem_size(tv, nvt), sv, nvs, elem_size(sv, nvs), feat + i * kMlpIn, qhat + i * kMlpOut, &Q[i]);
  const D3 ct = centroid(tv, nvt), cs = centroid(sv, nvs);
  const double rs = radius(tv, nvt, ct) + radius(sv, nvs, cs);
  const D3 d = dsub(ct, cs);
  bin[i] = pair_bin(sqrt(ddot(d, d)) / rs, sat_gap(tv, nvt, sv, nvs) / rs);
}

__global__ void k_select_strided(const int64_t* __restrict__ list, int64_t n_list, int64_t m, int64_t* __restrict__ sel) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < m) sel[i] = list[(int64_t)((double)i * (double)n_list / (double)m)];
}

__global__ void k_label_ratio(const double* __restrict__ C, const double* __restrict__ Q, int64_t n,
                              float* __restrict__ chat) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) chat[i] = (float)(C[i] / Q[i]);
}

// ------------------------------------------------------------ launchers
template <int P, int NT>
static cudaError_t launch_grad_p(const float* params, const float* feat, const float* qhat, const float* chat, int64_t n,
                                 float* grad, float* loss, int cluster, cudaStream_t st) {
  auto kernel = k_mlp_grad<P, NT>;
  constexpr size_t sm = sizeof(GradShared<P>);
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess && sm > 48 * 1024) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  for (int nc = cluster; nc >= 8; nc /= 2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((n + P * nc - 1) / (P * nc) * nc));
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)nc;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel, params, feat, qhat, chat, n, 1.0f / (float)n, grad, loss);
    if (e == cudaSuccess) return cudaGetLastError();
    (void)cudaGetLastError();
  }
  return e;
}

cudaError_t launch_mlp_grad(const float* params, const float* feat, const float* qhat, const float* chat, int64_t n,
                            float* grad, float* loss, cudaStream_t st) {
  k_mlp_zero<<<(kMlpParams + 256) / 256, 256, 0, st>>>(grad, loss);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || n == 0) return e;
  // fewer pairs a CTA shorten its chain, but every cluster rounds the running
  // gradient once: 8 pairs up to two clusters (200 pairs: 15 us, 18 with 32 pairs),
  // 32 above.  Beyond one CTA an SM the work counts, and small CTAs and clusters
  // fill the SMs better (call and wait of 20,000 pairs: 79 against 86 us, of
  // 200,000: 442 against 576)
  if (n <= 2 * 8 * kGradCluster) return launch_grad_p<8, 256>(params, feat, qhat, chat, n, grad, loss, kGradCluster, st);
  if (n <= 32 * kMlpSms) return launch_grad_p<32, 512>(params, feat, qhat, chat, n, grad, loss, kGradCluster, st);
  return launch_grad_p<32, 256>(params, feat, qhat, chat, n, grad, loss, 8, st);
}

cudaError_t launch_mlp_adam(float* params, const float* grad, float* m1, float* m2, int step, float lr, float b1,
                            float b2, float eps, cudaStream_t st) {
  const float c1 = 1.0f / (1.0f - powf(b1, (float)step)), c2 = 1.0f / (1.0f - powf(b2, (float)step));
  k_mlp_adam<<<(kMlpParams + 255) / 256, 256, 0, st>>>(params, grad, m1, m2, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

template <int P>
static cudaError_t launch_predict_p(const float* params, const float* feat, const float* qhat, int64_t n, float* out,
                                    cudaStream_t st) {
  constexpr size_t sm = sizeof(PredShared<P>);
  if (sm > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k_mlp_predict<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  const int64_t tiles = (n + P - 1) / P;
  k_mlp_predict<P><<<(unsigned)std::min<int64_t>(tiles, 2 * kMlpSms), kPredThreads, sm, st>>>(params, feat, qhat, n, out);
  return cudaGetLastError();
}

cudaError_t launch_mlp_predict(const float* params, const float* feat, const float* qhat, int64_t n, float* out,
                               cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  // 128 pairs a CTA once that fills the SMs, 32 below
  return n >= 128 * kMlpSms ? launch_predict_p<128>(params, feat, qhat, n, out, st) : launch_predict_p<32>(params, feat, qhat, n, out, st);
}

cudaError_t launch_near_classify(int task, int64_t nnz, const int* row, const int* col, const double* tgt_v,
                                 const double* src_v, int mode, const float* eps_tab, float tol, int64_t* lists,
                                 unsigned long long* counts, int64_t cap, unsigned* singular, cudaStream_t st) {
  if (nnz == 0) return cudaSuccess;
  k_near_classify<<<(unsigned)((nnz + 127) / 128), 128, 0, st>>>(task, nnz, row, col, tgt_v, src_v, mode, eps_tab, tol,
                                                                 lists, counts, cap, singular);
  return cudaGetLastError();
}

cudaError_t launch_near_mlp(int task, const int64_t* sel, int64_t n, const int* row, const int* col,
                            const double* tgt_v, const double* src_v, const float* params, double* cor_val,
                            cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_near_mlp<<<(unsigned)((n + kMlpThreads - 1) / kMlpThreads), kMlpThreads, 0, st>>>(task, sel, n, row, col, tgt_v,
                                                                                    src_v, params, cor_val);
  return cudaGetLastError();
}

cudaError_t launch_select_strided(const int64_t* list, int64_t n_list, int64_t m, int64_t* sel, cudaStream_t st) {
  if (m == 0) return cudaSuccess;
  k_select_strided<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(list, n_list, m, sel);
  return cudaGetLastError();
}

cudaError_t launch_label_ratio(const double* C, const double* Q, int64_t n, float* chat, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_label_ratio<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(C, Q, n, chat);
  return cudaGetLastError();
}

cudaError_t launch_pair_data(int task, const int64_t* sel, int64_t n, const int* row, const int* col,
                             const double* tgt_v, const double* src_v, float* feat, float* qhat, double* Q, int* bin,
                             int* pairs, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_pair_data<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(task, sel, n, row, col, tgt_v, src_v, feat, qhat, Q, bin,
                                                           pairs);
  return cudaGetLastError();
}

}  // namespace bcfmm
