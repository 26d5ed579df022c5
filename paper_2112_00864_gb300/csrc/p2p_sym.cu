// Symmetric FP32 near field of VtV (see p2p_sym.cuh).
//
// Bound by the FMA pipe and the rsqrt unit alike: 8 operations (of 128 lanes a
// cycle and SM) and one rsqrt (of 16) serve both directions of a pair of
// points, where the directed kernel spends 7 and one on each; a register-only
// loop of this body reaches 80 - 84 % of the FMA rate.  The price is a slot per
// owner block and source point (45 M floats on the level-4 ball) and the pass
// that adds them.  Unit ball, level 4 (191,840 tets, 4.8e9 directed pairs, one
// density): near field 1.64 -> 1.00 ms (owners over 32 points 0.78, the others
// 0.14, gather 0.083; FMA pipe 66 % active); level-3 ball 0.32 -> 0.23 ms; a
// batch of six meshes with four densities 2.71 -> 1.57 ms (scalar kernel
// before).
#include <algorithm>
#include <climits>
#include <cmath>
#include <map>

#include "internal.h"
#include "p2p_sym.cuh"

namespace bcfmm {
namespace {

constexpr double kInv4PiS = 0.079577471545947667884441881686257;
constexpr int kSymRuns = 256;       // source runs per batch

__device__ __forceinline__ void two_sum(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float b = s - hi;
  lo += (hi - (s - b)) + (x - b);
  hi = s;
}

__device__ __forceinline__ float rsqrt_ftz(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The sources of the next round arrive by cp.async while this one is computed
// (each thread copies and converts its own, so no barrier is needed between).
// LARGE (one density): a source is two float4 whose components stand in pairs,
// ready for the packed instructions; owners that spend fewer instructions on a
// source would be bound by those loads and read one float4, and so do the forms
// for two and four densities, with the further weights beside it.
template <int ND, bool LARGE>
struct SymShared {
  static constexpr bool kLarge = LARGE;
  static constexpr int kDens = ND, kTile = ND == 4 ? 256 : 512;     // sources staged per round
  float4 xy[kTile];                 // LARGE: source k: (-x, -x, -y, -y); else (-x, -y, -z, w)
  float4 zw[LARGE ? kTile : 1];     // (-z, -z, w, w)
  float wx[ND > 1 ? ND * kTile : 1];  // [source][ND] weights (the first one again)
  float4 rh[kTile], rl[kTile];      // copies in flight: hi and lo coordinates
  float rw[ND][kTile];              // and weights
  float2 red[LARGE ? 16 : 8][ND][128];  // (hi, lo) of target slot u, density, thread
  int pre[kSymRuns + 1], rst[kSymRuns];
};

__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One staged round: source blocks of GS, one per group of GS lanes and step.  A
// lane holds 2 T2 of the owner's points as T2 packed pairs, the same in every
// group; in step s lane l takes source l ^ s of its group's block, so that
// after GS steps every pair of the block was met once, and the sum for a
// source has travelled with it through the GS lanes (one shuffle a step).
// SELF: the owner's own points, one direction only, r = 0 selected out.
template <int T2, int GS, bool SELF, class SH, int ND>
__device__ __forceinline__ void sym_round(const SH& S, int m, const float2 (&X)[T2], const float2 (&Y)[T2],
                                          const float2 (&Z)[T2], const float2 (&Wt)[T2][ND], float2 (&acc)[T2][ND],
                                          float* __restrict__ out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l = lane & (GS - 1);
  for (int k0 = warp * 32; k0 < m; k0 += 128) {
    const int kg = k0 + lane - l;
    float trav[ND];
#pragma unroll
    for (int d = 0; d < ND; ++d) trav[d] = 0.f;
#pragma unroll
    for (int s = 0; s < GS; ++s) {
      const int k = kg + (l ^ s);
      float2 nx, ny, nz, w[ND], as[ND];
      const float4 a = S.xy[k];
      if constexpr (SH::kLarge) {
        const float4 c = S.zw[k];
        nx = make_float2(a.x, a.y); ny = make_float2(a.z, a.w); nz = make_float2(c.x, c.y);
        w[0] = make_float2(c.z, c.w);
      } else {
        nx = make_float2(a.x, a.x); ny = make_float2(a.y, a.y); nz = make_float2(a.z, a.z);
        w[0] = make_float2(a.w, a.w);
      }
      if constexpr (ND == 2) {
        const float v = S.wx[2 * k + 1];
        w[ND - 1] = make_float2(v, v);
      } else if constexpr (ND == 4) {
        const float4 v = *reinterpret_cast<const float4*>(S.wx + 4 * k);
        w[1 % ND] = make_float2(v.y, v.y);
        w[2 % ND] = make_float2(v.z, v.z);
        w[3 % ND] = make_float2(v.w, v.w);
      }
#pragma unroll
      for (int u = 0; u < T2; ++u) {
        const float2 dx = __fadd2_rn(X[u], nx), dy = __fadd2_rn(Y[u], ny), dz = __fadd2_rn(Z[u], nz);
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        float2 ri;
        if constexpr (SELF) ri = make_float2(r2.x > 0.f ? rsqrt_ftz(r2.x) : 0.f, r2.y > 0.f ? rsqrt_ftz(r2.y) : 0.f);
        else ri = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
#pragma unroll
        for (int d = 0; d < ND; ++d) {
          acc[u][d] = __ffma2_rn(w[d], ri, acc[u][d]);
          if constexpr (!SELF) as[d] = u == 0 ? __fmul2_rn(Wt[u][d], ri) : __ffma2_rn(Wt[u][d], ri, as[d]);
        }
      }
      if constexpr (!SELF) {
#pragma unroll
        for (int d = 0; d < ND; ++d) {
          trav[d] += as[d].x + as[d].y;
          trav[d] = __shfl_xor_sync(0xffffffffu, trav[d], s < GS - 1 ? (s ^ (s + 1)) : GS - 1);
        }
      }
    }
    if constexpr (!SELF) {
      if (kg + l < m) {
        if constexpr (ND == 1) out[kg + l] = trav[0];
        else if constexpr (ND == 2) reinterpret_cast<float2*>(out)[kg + l] = make_float2(trav[0], trav[1]);
        else reinterpret_cast<float4*>(out)[kg + l] = make_float4(trav[0], trav[1], trav[2], trav[3]);
      }
    }
  }
}

template <int T2, class SH, int ND>
__device__ __forceinline__ void sym_fold(SH& S, float2 (&acc)[T2][ND]) {
#pragma unroll
  for (int u = 0; u < T2; ++u)
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      float2 a = S.red[2 * u][d][threadIdx.x], b = S.red[2 * u + 1][d][threadIdx.x];
      two_sum(a.x, a.y, acc[u][d].x);
      two_sum(b.x, b.y, acc[u][d].y);
      S.red[2 * u][d][threadIdx.x] = a;
      S.red[2 * u + 1][d][threadIdx.x] = b;
      acc[u][d] = make_float2(0.f, 0.f);
    }
}

template <int T2, int GS, class SH>
__device__ __forceinline__ void sym_block(const DevGeom& G, const DevSym& L, const float* __restrict__ W, int64_t nsp, SH& S,
                                          int b, int nt, int2 tr, float4 ch, float4 cl) {
  constexpr int ND = SH::kDens, kTile = SH::kTile;
  auto put = [&](int k, float x, float y, float z, float w) {
    if constexpr (SH::kLarge) {
      S.xy[k] = make_float4(x, x, y, y);
      S.zw[k] = make_float4(z, z, w, w);
    } else {
      S.xy[k] = make_float4(x, y, z, w);
    }
  };
  auto put_df = [&](int k, const float4& h, const float4& q, float w) {
    put(k, -((h.x - ch.x) + (q.x - cl.x)), -((h.y - ch.y) + (q.y - cl.y)), -((h.z - ch.z) + (q.z - cl.z)), w);
  };
  // padding: sources at -1e30 (stored negated), owner points at +1e30; the
  // distance overflows to inf, whose rsqrt is 0
  auto pad = [&](int k) {
    put(k, 1e30f, 1e30f, 1e30f, 0.f);
    if constexpr (ND > 1)
      for (int d = 0; d < ND; ++d) S.wx[ND * k + d] = 0.f;
  };
  // the owner's points, staged as the first round's sources
  if (threadIdx.x < nt) {
    const int j = tr.x + threadIdx.x;
    put_df(threadIdx.x, G.pthi[0][j], G.ptlo[0][j], W[j]);
    if constexpr (ND > 1)
      for (int d = 0; d < ND; ++d) S.wx[ND * threadIdx.x + d] = W[d * nsp + j];
  } else {
    pad(threadIdx.x);
  }
#pragma unroll
  for (int u = 0; u < 2 * T2; ++u)
#pragma unroll
    for (int d = 0; d < ND; ++d) S.red[u][d][threadIdx.x] = make_float2(0.f, 0.f);
  __syncthreads();
  float2 X[T2], Y[T2], Z[T2], Wt[T2][ND], acc[T2][ND];
  const int l = threadIdx.x & (GS - 1);
#pragma unroll
  for (int u = 0; u < T2; ++u) {
    const int t0 = 2 * GS * u + l, t1 = t0 + GS;
    const bool v0 = t0 < nt, v1 = t1 < nt;
    float4 p0 = S.xy[t0], p1 = S.xy[t1];         // (-x, -y, -z, w)
    if constexpr (SH::kLarge) {
      p0 = make_float4(p0.x, p0.z, S.zw[t0].x, S.zw[t0].z);
      p1 = make_float4(p1.x, p1.z, S.zw[t1].x, S.zw[t1].z);
    }
    X[u] = make_float2(v0 ? -p0.x : 1e30f, v1 ? -p1.x : 1e30f);
    Y[u] = make_float2(v0 ? -p0.y : 1e30f, v1 ? -p1.y : 1e30f);
    Z[u] = make_float2(v0 ? -p0.z : 1e30f, v1 ? -p1.z : 1e30f);
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      if constexpr (ND > 1) { p0.w = S.wx[ND * t0 + d]; p1.w = S.wx[ND * t1 + d]; }
      Wt[u][d] = make_float2(v0 ? p0.w : 0.f, v1 ? p1.w : 0.f);
      acc[u][d] = make_float2(0.f, 0.f);
    }
  }
  if (L.self[b]) sym_round<T2, GS, true>(S, nt, X, Y, Z, Wt, acc, nullptr);
  const int r0 = L.run_off[b], r1 = L.run_off[b + 1];
  const int2 base = L.base[b];
  float* out = L.src + (int64_t)ND * base.x;
  // a lane's FP32 sum holds at most 64 products between folds, and GS more in the
  // first interval (the owner's own points; a fold of their own costs 3 % of the
  // level-3 ball's step)
  int fold = 0;
  for (int rb = r0; rb < r1; rb += kSymRuns) {
    const int nr = min(kSymRuns, r1 - rb);
    __syncthreads();
    if (threadIdx.x < 32) {
      int carry = 0;
      if (threadIdx.x == 0) S.pre[0] = 0;
      for (int c = 0; c < nr; c += 32) {
        const int r = c + threadIdx.x;
        int x = 0;
        if (r < nr) { const int2 rr = L.runs[rb + r]; x = rr.y - rr.x; S.rst[r] = rr.x; }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, x, o); if ((int)threadIdx.x >= o) x += y; }
        if (r < nr) S.pre[r + 1] = carry + x;
        carry += __shfl_sync(0xffffffffu, x, 31);
      }
    }
    __syncthreads();
    const int total = S.pre[nr];
    int r = 0;                                   // this thread's run: its sources ascend
    auto fetch = [&](int v0) {                   // copies of this thread's sources of the round at v0
#pragma unroll
      for (int q = 0; q < kTile / 128; ++q) {
        const int k = threadIdx.x + q * 128, v = v0 + k;
        if (v < total) {
          while (S.pre[r + 1] <= v) ++r;
          const int src = S.rst[r] + (v - S.pre[r]);
          copy16(&S.rh[k], &G.pthi[0][src]);
          copy16(&S.rl[k], &G.ptlo[0][src]);
#pragma unroll
          for (int d = 0; d < ND; ++d) copy4(&S.rw[d][k], &W[d * nsp + src]);
        }
      }
    };
    if (total > 0) fetch(0);
    for (int v0 = 0; v0 < total; v0 += kTile) {
      const int m = min(kTile, total - v0), mp = (m + 31) & ~31;
      copy_wait();
#pragma unroll
      for (int q = 0; q < kTile / 128; ++q) {
        const int k = threadIdx.x + q * 128;
        if (k < m) {
          put_df(k, S.rh[k], S.rl[k], S.rw[0][k]);
          if constexpr (ND > 1) {
#pragma unroll
            for (int d = 0; d < ND; ++d) S.wx[ND * k + d] = S.rw[d][k];
          }
        } else if (k < mp) {
          pad(k);
        }
      }
      __syncthreads();
      if (v0 + kTile < total) fetch(v0 + kTile);
      sym_round<T2, GS, false>(S, m, X, Y, Z, Wt, acc, out + ND * v0);
      if (++fold >= 64 * 128 / (GS * kTile)) { sym_fold<T2>(S, acc); fold = 0; }
      __syncthreads();
    }
    out += ND * total;
  }
  sym_fold<T2>(S, acc);
  __syncthreads();
  if (threadIdx.x < nt) {
    // the groups' sums of this point, in group order
    const int t = threadIdx.x, u = t / GS;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      float hi = 0.f, lo = 0.f;
#pragma unroll 16
      for (int g = 0; g < 128 / GS; ++g) {
        const float2 v = S.red[u][d][g * GS + (t & (GS - 1))];
        two_sum(hi, lo, v.x);
        lo += v.y;
      }
      L.tgt[(int64_t)ND * (base.y + t) + d] = make_float2(hi, lo);
    }
  }
}

// Groups of four lanes for small owners, of eight and sixteen for larger ones
// (a lane holds at most eight pairs, four with several densities): the padding
// is to eight, sixteen or 32 points, and the shared loads, the shuffles and the
// sum for a source are paid once per lane of a group.  LARGE (one density):
// owners of more than 32 points (five to eight pairs, 128 registers, four CTAs
// on an SM); the others need fewer registers and run six.
template <int ND, bool LARGE>
__global__ void __launch_bounds__(128, ND == 1 && !LARGE ? 6 : 4) k_p2p_sym(DevGeom G, DevSym L, int b0,
                                                                            const float* __restrict__ W, int64_t nsp) {
  extern __shared__ __align__(16) unsigned char smraw[];
  SymShared<ND, LARGE>& S = *reinterpret_cast<SymShared<ND, LARGE>*>(smraw);
  const int b = b0 + blockIdx.x;
  const int leaf = L.leaf[b];
  const float4 ch = G.box_hi[leaf], cl = G.box_lo[leaf];
  const int2 tr = G.box_rng[0][leaf];
  const int nt = tr.y - tr.x;
  if constexpr (LARGE) {
    if (nt <= 64) {
      switch ((nt + 7) >> 3) {
        case 5: sym_block<5, 4>(G, L, W, nsp, S, b, nt, tr, ch, cl); break;
        case 6: sym_block<6, 4>(G, L, W, nsp, S, b, nt, tr, ch, cl); break;
        case 7: sym_block<7, 4>(G, L, W, nsp, S, b, nt, tr, ch, cl); break;
        default: sym_block<8, 4>(G, L, W, nsp, S, b, nt, tr, ch, cl); break;
      }
    } else {
      switch ((nt + 15) >> 4) {
        case 5: sym_block<5, 8>(G, L, W, nsp, S, b, nt, tr, ch, cl); break;
        case 6: sym_block<6, 8>(G, L, W, nsp, S, b, nt, tr, ch, cl); break;
        case 7: sym_block<7, 8>(G, L, W, nsp, S, b, nt, tr, ch, cl); break;
        default: sym_block<8, 8>(G, L, W, nsp, S, b, nt, tr, ch, cl); break;
      }
    }
  } else {
    if (nt <= 32) {
      switch ((nt + 7) >> 3) {
        case 1: sym_block<1, 4>(G, L, W, nsp, S, b, nt, tr, ch, cl); break;
        case 2: sym_block<2, 4>(G, L, W, nsp, S, b, nt, tr, ch, cl); break;
        case 3: sym_block<3, 4>(G, L, W, nsp, S, b, nt, tr, ch, cl); break;
        default: sym_block<4, 4>(G, L, W, nsp, S, b, nt, tr, ch, cl); break;
      }
    } else if constexpr (ND > 1) {
      if (nt <= 48) sym_block<3, 8>(G, L, W, nsp, S, b, nt, tr, ch, cl);
      else if (nt <= 64) sym_block<4, 8>(G, L, W, nsp, S, b, nt, tr, ch, cl);
      else if (nt <= 96) sym_block<3, 16>(G, L, W, nsp, S, b, nt, tr, ch, cl);
      else sym_block<4, 16>(G, L, W, nsp, S, b, nt, tr, ch, cl);
    }
  }
}

// ------------------------------------------------------------ gather
// One CTA per target leaf: thread groups share the leaf's slots (each takes a
// contiguous part in order, compensated sums), their sums are added in group
// order.  The slot offsets are staged first, so that a group's loads do not
// wait for them one by one.
constexpr int kGatherThreads = 256, kGatherIdx = 1024;

template <int ND>
__global__ void __launch_bounds__(kGatherThreads) k_sym_gather(DevGeom G, DevSym L, int64_t ntp, double* __restrict__ phi) {
  __shared__ float2 red[ND][kGatherThreads];
  __shared__ int idx[kGatherIdx];
  const int f = blockIdx.x, leaf = L.fin_leaf[f];
  const int2 tr = G.box_rng[0][leaf];
  const int nt = tr.y - tr.x;
  const int NG = kGatherThreads / nt, g = threadIdx.x / nt, i = threadIdx.x - g * nt;
  const int s0 = L.fin_src_off[f], s1 = L.fin_src_off[f + 1];
  float hi[ND], lo[ND];
#pragma unroll
  for (int d = 0; d < ND; ++d) hi[d] = lo[d] = 0.f;
  for (int c = s0; c < s1; c += kGatherIdx) {
    const int n = min(kGatherIdx, s1 - c);
    if (c > s0) __syncthreads();
    for (int e = threadIdx.x; e < n; e += kGatherThreads) idx[e] = L.fin_src[c + e];
    __syncthreads();
    if (g < NG) {
      const int e1 = n * (g + 1) / NG;
#pragma unroll 8
      for (int e = n * g / NG; e < e1; ++e) {
        const float* p = L.src + (int64_t)ND * (idx[e] + i);
        float v[4];
        if constexpr (ND == 1) v[0] = __ldcg(p);
        else if constexpr (ND == 2) { const float2 q = __ldcg(reinterpret_cast<const float2*>(p)); v[0] = q.x; v[1] = q.y; }
        else { const float4 q = __ldcg(reinterpret_cast<const float4*>(p)); v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w; }
#pragma unroll
        for (int d = 0; d < ND; ++d) two_sum(hi[d], lo[d], v[d]);
      }
    }
  }
  if (g == 0)
    for (int e = L.fin_tgt_off[f]; e < L.fin_tgt_off[f + 1]; ++e)
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        const float2 v = __ldcg(L.tgt + (int64_t)ND * (L.fin_tgt[e] + i) + d);
        two_sum(hi[d], lo[d], v.x);
        lo[d] += v.y;
      }
#pragma unroll
  for (int d = 0; d < ND; ++d) red[d][threadIdx.x] = make_float2(hi[d], lo[d]);
  __syncthreads();
  if ((int)threadIdx.x >= nt) return;
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    for (int h = 1; h < NG; ++h) {
      const float2 v = red[d][h * nt + i];
      two_sum(hi[d], lo[d], v.x);
      lo[d] += v.y;
    }
    phi[d * ntp + tr.x + i] = ((double)hi[d] + (double)lo[d]) * kInv4PiS;
  }
}

}  // namespace

template <int ND, bool LARGE>
cudaError_t launch_blocks(const DevGeom& G, const DevSym& S, int b0, int n, const float* W, int64_t nsp, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  constexpr size_t sm = sizeof(SymShared<ND, LARGE>);
  if (sm > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k_p2p_sym<ND, LARGE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  k_p2p_sym<ND, LARGE><<<n, 128, sm, st>>>(G, S, b0, W, nsp);
  return cudaGetLastError();
}

cudaError_t launch_p2p_sym(const DevGeom& G, const DevSym& S, const float* W, int64_t npts, int ndp, double* phi, cudaStream_t st) {
  if (!p2p_sym_takes(S, ndp)) return cudaErrorInvalidValue;
  cudaError_t e;
  switch (ndp) {
    case 1:
      e = launch_blocks<1, true>(G, S, 0, S.nlarge, W, npts, st);
      if (e == cudaSuccess) e = launch_blocks<1, false>(G, S, S.nlarge, S.nblk - S.nlarge, W, npts, st);
      break;
    case 2: e = launch_blocks<2, false>(G, S, 0, S.nblk, W, npts, st); break;
    case 4: e = launch_blocks<4, false>(G, S, 0, S.nblk, W, npts, st); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  if (ndp == 1) k_sym_gather<1><<<S.nfin, kGatherThreads, 0, st>>>(G, S, npts, phi);
  else if (ndp == 2) k_sym_gather<2><<<S.nfin, kGatherThreads, 0, st>>>(G, S, npts, phi);
  else k_sym_gather<4><<<S.nfin, kGatherThreads, 0, st>>>(G, S, npts, phi);
  return cudaGetLastError();
}

// owner of the pair of near leaves (a, b): the deeper level, then the lower index
static inline bool sym_owns(const HostSetup& H, int a, int b) {
  return H.box[a].level != H.box[b].level ? H.box[a].level > H.box[b].level : a < b;
}

// owner points a block computes: padded to its lanes' pairs
static inline int sym_pad(int nt) { return nt <= 64 ? (nt + 7) / 8 * 8 : (nt + 15) / 16 * 16; }

// Lane work of both forms over the mesh: the symmetric one pads an owner to a
// multiple of 8 or 16 points and spends 8 FP32 operations on a pair of points,
// the directed one pads to 4 and spends 7 on each direction.  Tiny leaves
// (under about 5 points) are better off with the latter.
bool p2p_sym_pays(const HostSetup& H) {
  const HostTask& T = H.task[0];
  double sym = 0, dir = 0;
  for (size_t i = 0; i < T.p2p_leaf.size(); ++i) {
    const int a = T.p2p_leaf[i];
    const double nt = H.box[a].pt1[0] - H.box[a].pt0[0];
    double ns = 0, nd = 0;
    for (int k = T.near_off[i]; k < T.near_off[i + 1]; ++k) {
      const HostBox& C = H.box[T.near_box[k]];
      nd += C.pt1[0] - C.pt0[0];
      if (!C.nchild && T.near_box[k] != a && sym_owns(H, a, T.near_box[k])) ns += C.pt1[0] - C.pt0[0];
    }
    sym += sym_pad((int)nt) * (ns + nt) * 8.0;
    dir += 4 * std::ceil(nt / 4) * nd * 7;
  }
  return sym < dir;
}

int64_t p2p_sym_chunk(const HostSetup& H, int nsm) {
  const HostTask& T = H.task[0];
  int64_t total = 0;
  for (size_t i = 0; i < T.p2p_leaf.size(); ++i)
    for (int k = T.near_off[i]; k < T.near_off[i + 1]; ++k) {
      const HostBox& C = H.box[T.near_box[k]];
      if (!C.nchild && T.near_box[k] != T.p2p_leaf[i] && sym_owns(H, T.p2p_leaf[i], T.near_box[k])) total += C.pt1[0] - C.pt0[0];
    }
  return std::min(kSymChunkMax, std::max(kSymChunkMin, total / (8 * (int64_t)nsm)));
}

bool build_p2p_sym(const HostSetup& H, int64_t chunk, HostSym& out) {
  const HostTask& T = H.task[0];
  out = HostSym();
  struct Blk { int leaf, nt, self; int64_t ns; std::vector<int> runs, src; };   // src: the source leaves in run order
  std::vector<Blk> blk;
  std::vector<int> src;
  for (size_t i = 0; i < T.p2p_leaf.size(); ++i) {
    const int a = T.p2p_leaf[i];
    src.clear();
    int64_t ns = 0;
    for (int k = T.near_off[i]; k < T.near_off[i + 1]; ++k) {
      const int c = T.near_box[k];
      if (H.box[c].nchild || c == a || !sym_owns(H, a, c)) continue;
      src.push_back(c);
      ns += H.box[c].pt1[0] - H.box[c].pt0[0];
    }
    std::sort(src.begin(), src.end(), [&](int x, int y) { return H.box[x].pt0[0] < H.box[y].pt0[0]; });
    const int nch = (int)std::max<int64_t>(1, (ns + chunk - 1) / chunk);
    const int64_t per = (ns + nch - 1) / nch;
    const int nt = H.box[a].pt1[0] - H.box[a].pt0[0];
    Blk cur{a, nt, 1, 0, {}, {}};
    for (int c : src) {
      const int s0 = H.box[c].pt0[0], s1 = H.box[c].pt1[0];
      if (cur.ns >= per) {
        blk.push_back(std::move(cur));
        cur = Blk{a, nt, 0, 0, {}, {}};
      }
      if (!cur.runs.empty() && cur.runs.back() == s0) cur.runs.back() = s1;
      else { cur.runs.push_back(s0); cur.runs.push_back(s1); }
      cur.src.push_back(c);
      cur.ns += s1 - s0;
    }
    blk.push_back(std::move(cur));
  }
  // owners of one padded size in a row, the largest first, so that the blocks on
  // an SM run the same code (mixed sizes missed the instruction cache: 1.04 ms
  // for the level-4 ball's two kernels); then longest first
  std::stable_sort(blk.begin(), blk.end(), [](const Blk& x, const Blk& y) {
    const int px = sym_pad(x.nt), py = sym_pad(y.nt);
    return px != py ? px > py : x.ns > y.ns;
  });
  std::vector<int> cnt(H.box.size() + 1, 0), tcnt(H.box.size() + 1, 0);
  int64_t ns = 0, ntg = 0;
  for (const Blk& b : blk) {
    ns += b.ns;
    ntg += b.nt;
    tcnt[b.leaf]++;
    for (int c : b.src) cnt[c]++;
  }
  if (ns >= INT_MAX || ntg >= INT_MAX) return false;
  // target leaves, most slots first
  out.fin_leaf = T.p2p_leaf;
  std::stable_sort(out.fin_leaf.begin(), out.fin_leaf.end(), [&](int x, int y) { return cnt[x] > cnt[y]; });
  std::vector<int> cur_s(H.box.size(), 0), cur_t(H.box.size(), 0);
  out.fin_src_off.push_back(0);
  out.fin_tgt_off.push_back(0);
  for (int lf : out.fin_leaf) {
    cur_s[lf] = out.fin_src_off.back();
    cur_t[lf] = out.fin_tgt_off.back();
    out.fin_src_off.push_back(cur_s[lf] + cnt[lf]);
    out.fin_tgt_off.push_back(cur_t[lf] + tcnt[lf]);
  }
  out.fin_src.resize(out.fin_src_off.back());
  out.fin_tgt.resize(out.fin_tgt_off.back());
  out.run_off.push_back(0);
  for (const Blk& b : blk) {
    out.leaf.push_back(b.leaf);
    out.nlarge += b.nt > 32;
    out.self.push_back(b.self);
    out.base.push_back((int)out.nsrc);
    out.base.push_back((int)out.ntgt);
    out.runs.insert(out.runs.end(), b.runs.begin(), b.runs.end());
    out.run_off.push_back((int)out.runs.size() / 2);
    out.fin_tgt[cur_t[b.leaf]++] = (int)out.ntgt;
    out.ntgt += b.nt;
    for (int c : b.src) {
      out.fin_src[cur_s[c]++] = (int)out.nsrc;
      out.nsrc += H.box[c].pt1[0] - H.box[c].pt0[0];
    }
  }
  return true;
}

SymFaults check_p2p_sym(const HostSetup& H, int64_t chunk, const HostSym& S) {
  const HostTask& T = H.task[0];
  SymFaults F;
  auto npt = [&](int b) { return H.box[b].pt1[0] - H.box[b].pt0[0]; };
  // near pairs of leaves as (lower box, higher box): how often they are due (1),
  // minus how often they occur
  std::map<std::pair<int, int>, int> due;
  auto key = [](int a, int b) { return std::make_pair(std::min(a, b), std::max(a, b)); };
  for (size_t i = 0; i < T.p2p_leaf.size(); ++i)
    for (int k = T.near_off[i]; k < T.near_off[i + 1]; ++k) {
      std::vector<int> todo(1, T.near_box[k]);     // the leaves of the near subtree
      while (!todo.empty()) {
        const int b = todo.back();
        todo.pop_back();
        const HostBox& B = H.box[b];
        if (B.nchild == 0 && npt(b) > 0) due[key(T.p2p_leaf[i], b)] = 1;
        for (int c = 0; c < B.nchild; ++c) todo.push_back(B.child0 + c);
      }
    }
  const int nblk = (int)S.leaf.size();
  std::vector<int> src_pt(S.nsrc, -1), tgt_pt(S.ntgt, -1);      // the point a slot was written for
  int last = INT_MAX;
  for (int b = 0; b < nblk; ++b) {
    const int a = S.leaf[b], nt = npt(a);
    if (S.self[b]) due[key(a, a)]--;
    if ((b < S.nlarge) != (nt > 32) || nt < 1 || nt > 128 || sym_pad(nt) > last) F.blocks++;
    last = sym_pad(nt);
    int64_t slot = S.base[2 * b], n = 0;
    for (int r = S.run_off[b]; r < S.run_off[b + 1]; ++r)
      for (int q = S.runs[2 * r]; q < S.runs[2 * r + 1];) {
        const int c = H.leaf_of[0][q];
        if (q != H.box[c].pt0[0] || H.box[c].pt1[0] > S.runs[2 * r + 1]) { F.pairs++; break; }   // (a part of a leaf)
        due[key(a, c)]--;
        for (; q < H.box[c].pt1[0]; ++q, ++slot, ++n) {
          if (slot < 0 || slot >= S.nsrc || src_pt[slot] >= 0) F.slots++;
          else src_pt[slot] = q;
        }
      }
    if (n > chunk + 128) F.blocks++;
    for (int i = 0; i < nt; ++i) {
      const int64_t t = (int64_t)S.base[2 * b + 1] + i;
      if (t < 0 || t >= S.ntgt || tgt_pt[t] >= 0) F.slots++;
      else tgt_pt[t] = H.box[a].pt0[0] + i;
    }
  }
  for (const auto& d : due) F.pairs += d.second != 0;
  // the gather: point i of a leaf takes slot f + i of every f in the leaf's lists
  std::vector<int> leaves = S.fin_leaf, want = T.p2p_leaf;
  std::sort(leaves.begin(), leaves.end());
  std::sort(want.begin(), want.end());
  if (leaves != want) F.slots++;
  auto gather = [&](const std::vector<int>& off, const std::vector<int>& list, std::vector<int>& pt) {
    for (size_t f = 0; f < S.fin_leaf.size(); ++f) {
      const int lf = S.fin_leaf[f];
      for (int e = off[f]; e < off[f + 1]; ++e)
        for (int i = 0; i < npt(lf); ++i) {
          const int64_t k = (int64_t)list[e] + i;
          if (k < 0 || k >= (int64_t)pt.size() || pt[k] != H.box[lf].pt0[0] + i) F.slots++;
          else pt[k] = -1;
        }
    }
    for (int v : pt) F.slots += v >= 0;
  };
  gather(S.fin_src_off, S.fin_src, src_pt);
  gather(S.fin_tgt_off, S.fin_tgt, tgt_pt);
  return F;
}

}  // namespace bcfmm
