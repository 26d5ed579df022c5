// Symmetric FP32 near field of VtV (see p2p_sym.cuh).
//
// Bound by the FMA pipe: 8 operations and one rsqrt serve both directions of a
// pair of points, where the directed kernel spends 7 and one on each.  The
// price is a slot per owner block and source point (45 M floats on the level-4
// ball) and the pass that adds them.  Unit ball, level 4 (191,840 tets, 4.8e9
// directed pairs, one density): near field 1.64 -> 1.04 ms (owners over 64
// points 0.51, the others 0.45, gather 0.085; FMA pipe 66 and 61 % active,
// what is missing goes to the staging rounds); level-3 ball 0.32 -> 0.25 ms.
#include <algorithm>
#include <climits>
#include <cmath>

#include "internal.h"
#include "p2p_sym.cuh"

namespace bcfmm {
namespace {

constexpr double kInv4PiS = 0.079577471545947667884441881686257;
constexpr int kSymTile = 512;       // sources staged per round
constexpr int kSymRuns = 256;       // source runs per batch
constexpr int kSymFold = 2;         // rounds between folds: at most 64 products per FP32 sum

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

template <bool LARGE>
struct SymShared {
  float4 xy[kSymTile];              // source k: (-x, -x, -y, -y)
  float4 zw[kSymTile];              // (-z, -z, w, w)
  float2 red[LARGE ? 16 : 8][128];  // (hi, lo) of target slot u, thread
  int pre[kSymRuns + 1], rst[kSymRuns];
};

// One staged round: source blocks of eight, four to a warp and step (one per
// group of eight lanes).  A lane holds 2 T2 of the owner's points as T2 packed
// pairs, the same in every group; in step s lane l takes source l ^ s of its
// group's block, so that after eight steps every pair of the block was met
// once, and the sum for a source has travelled with it through the eight lanes
// (one shuffle a step).  SELF: the owner's own points, one direction only,
// r = 0 selected out.
template <int T2, bool SELF, class SH>
__device__ __forceinline__ void sym_round(const SH& S, int m, const float2 (&X)[T2], const float2 (&Y)[T2],
                                          const float2 (&Z)[T2], const float2 (&Wt)[T2], float2 (&acc)[T2],
                                          float* __restrict__ out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l = lane & 7;
  const int nb = (m + 7) >> 3;
  for (int bb = warp * 4; bb < nb; bb += 16) {
    const int b8 = (bb + (lane >> 3)) * 8;
    float trav = 0.f;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const int k = b8 + (l ^ s);
      const float4 a = S.xy[k], c = S.zw[k];
      const float2 nx = make_float2(a.x, a.y), ny = make_float2(a.z, a.w), nz = make_float2(c.x, c.y);
      const float2 w = make_float2(c.z, c.w);
      float2 as = make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < T2; ++u) {
        const float2 dx = __fadd2_rn(X[u], nx), dy = __fadd2_rn(Y[u], ny), dz = __fadd2_rn(Z[u], nz);
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        float2 ri;
        if constexpr (SELF) ri = make_float2(r2.x > 0.f ? rsqrt_ftz(r2.x) : 0.f, r2.y > 0.f ? rsqrt_ftz(r2.y) : 0.f);
        else ri = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
        acc[u] = __ffma2_rn(w, ri, acc[u]);
        if constexpr (!SELF) as = u == 0 ? __fmul2_rn(Wt[u], ri) : __ffma2_rn(Wt[u], ri, as);
      }
      if constexpr (!SELF) {
        trav += as.x + as.y;
        trav = __shfl_xor_sync(0xffffffffu, trav, s < 7 ? (s ^ (s + 1)) : 7);
      }
    }
    if constexpr (!SELF)
      if (b8 + l < m) out[b8 + l] = trav;
  }
}

template <int T2, class SH>
__device__ __forceinline__ void sym_fold(SH& S, float2 (&acc)[T2]) {
#pragma unroll
  for (int u = 0; u < T2; ++u) {
    float2 a = S.red[2 * u][threadIdx.x], b = S.red[2 * u + 1][threadIdx.x];
    two_sum(a.x, a.y, acc[u].x);
    two_sum(b.x, b.y, acc[u].y);
    S.red[2 * u][threadIdx.x] = a;
    S.red[2 * u + 1][threadIdx.x] = b;
    acc[u] = make_float2(0.f, 0.f);
  }
}

template <int T2, class SH>
__device__ __forceinline__ void sym_block(const DevGeom& G, const DevSym& L, const float* __restrict__ W, SH& S,
                                          int b, int nt, int2 tr, float4 ch, float4 cl) {
  auto stage = [&](int k, int src) {
    const float4 h = G.pthi[0][src], q = G.ptlo[0][src];
    const float x = -((h.x - ch.x) + (q.x - cl.x)), y = -((h.y - ch.y) + (q.y - cl.y)), z = -((h.z - ch.z) + (q.z - cl.z));
    const float w = W[src];
    S.xy[k] = make_float4(x, x, y, y);
    S.zw[k] = make_float4(z, z, w, w);
  };
  // padding: sources at -1e30 (stored negated), owner points at +1e30; the
  // distance overflows to inf, whose rsqrt is 0
  auto pad = [&](int k) {
    S.xy[k] = make_float4(1e30f, 1e30f, 1e30f, 1e30f);
    S.zw[k] = make_float4(1e30f, 1e30f, 0.f, 0.f);
  };
  // the owner's points, staged as the first round's sources
  if (threadIdx.x < nt) stage(threadIdx.x, tr.x + threadIdx.x);
  else pad(threadIdx.x);
#pragma unroll
  for (int u = 0; u < 2 * T2; ++u) S.red[u][threadIdx.x] = make_float2(0.f, 0.f);
  __syncthreads();
  float2 X[T2], Y[T2], Z[T2], Wt[T2], acc[T2];
  const int l = threadIdx.x & 7;
#pragma unroll
  for (int u = 0; u < T2; ++u) {
    const int t0 = 16 * u + l, t1 = t0 + 8;
    const bool v0 = t0 < nt, v1 = t1 < nt;
    const float4 a0 = S.xy[t0], c0 = S.zw[t0], a1 = S.xy[t1], c1 = S.zw[t1];
    X[u] = make_float2(v0 ? -a0.x : 1e30f, v1 ? -a1.x : 1e30f);
    Y[u] = make_float2(v0 ? -a0.z : 1e30f, v1 ? -a1.z : 1e30f);
    Z[u] = make_float2(v0 ? -c0.x : 1e30f, v1 ? -c1.x : 1e30f);
    Wt[u] = make_float2(v0 ? c0.z : 0.f, v1 ? c1.z : 0.f);
    acc[u] = make_float2(0.f, 0.f);
  }
  if (L.self[b]) sym_round<T2, true>(S, nt, X, Y, Z, Wt, acc, nullptr);
  const int r0 = L.run_off[b], r1 = L.run_off[b + 1];
  const int2 base = L.base[b];
  float* out = L.src + base.x;
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
    for (int v0 = 0; v0 < total; v0 += kSymTile) {
      const int m = min(kSymTile, total - v0), mp = (m + 31) & ~31;
#pragma unroll
      for (int q = 0; q < kSymTile / 128; ++q) {
        const int k = threadIdx.x + q * 128, v = v0 + k;
        if (k < m) {
          while (S.pre[r + 1] <= v) ++r;
          stage(k, S.rst[r] + (v - S.pre[r]));
        } else if (k < mp) {
          pad(k);
        }
      }
      __syncthreads();
      sym_round<T2, false>(S, m, X, Y, Z, Wt, acc, out + v0);
      if (++fold == kSymFold) { sym_fold<T2>(S, acc); fold = 0; }
      __syncthreads();
    }
    out += total;
  }
  sym_fold<T2>(S, acc);
  __syncthreads();
  if (threadIdx.x < nt) {
    // the sixteen groups' sums of this point, in group order
    const int t = threadIdx.x, u = t >> 3;
    float hi = 0.f, lo = 0.f;
#pragma unroll
    for (int g = 0; g < 16; ++g) {
      const float2 v = S.red[u][g * 8 + (t & 7)];
      two_sum(hi, lo, v.x);
      lo += v.y;
    }
    L.tgt[base.y + t] = make_float2(hi, lo);
  }
}

// LARGE: owners of more than 64 points (up to eight pairs a lane, 128
// registers, four CTAs on an SM); the others need fewer registers and run six.
template <bool LARGE>
__global__ void __launch_bounds__(128, LARGE ? 4 : 6) k_p2p_sym(DevGeom G, DevSym L, int b0, const float* __restrict__ W) {
  __shared__ SymShared<LARGE> S;
  const int b = b0 + blockIdx.x;
  const int leaf = L.leaf[b];
  const float4 ch = G.box_hi[leaf], cl = G.box_lo[leaf];
  const int2 tr = G.box_rng[0][leaf];
  const int nt = tr.y - tr.x;
  if constexpr (LARGE) {
    switch ((nt + 15) >> 4) {
      case 5: sym_block<5>(G, L, W, S, b, nt, tr, ch, cl); break;
      case 6: sym_block<6>(G, L, W, S, b, nt, tr, ch, cl); break;
      case 7: sym_block<7>(G, L, W, S, b, nt, tr, ch, cl); break;
      default: sym_block<8>(G, L, W, S, b, nt, tr, ch, cl); break;
    }
  } else {
    switch ((nt + 15) >> 4) {
      case 1: sym_block<1>(G, L, W, S, b, nt, tr, ch, cl); break;
      case 2: sym_block<2>(G, L, W, S, b, nt, tr, ch, cl); break;
      case 3: sym_block<3>(G, L, W, S, b, nt, tr, ch, cl); break;
      default: sym_block<4>(G, L, W, S, b, nt, tr, ch, cl); break;
    }
  }
}

// ------------------------------------------------------------ gather
// One CTA per target leaf: thread groups share the leaf's slots (each takes a
// contiguous part in order, compensated sums), their sums are added in group
// order.  The slot offsets are staged first, so that a group's loads do not
// wait for them one by one.
constexpr int kGatherThreads = 256, kGatherIdx = 1024;

__global__ void __launch_bounds__(kGatherThreads) k_sym_gather(DevGeom G, DevSym L, double* __restrict__ phi) {
  __shared__ float2 red[kGatherThreads];
  __shared__ int idx[kGatherIdx];
  const int f = blockIdx.x, leaf = L.fin_leaf[f];
  const int2 tr = G.box_rng[0][leaf];
  const int nt = tr.y - tr.x;
  const int NG = kGatherThreads / nt, g = threadIdx.x / nt, i = threadIdx.x - g * nt;
  const int s0 = L.fin_src_off[f], s1 = L.fin_src_off[f + 1];
  float hi = 0.f, lo = 0.f;
  for (int c = s0; c < s1; c += kGatherIdx) {
    const int n = min(kGatherIdx, s1 - c);
    if (c > s0) __syncthreads();
    for (int e = threadIdx.x; e < n; e += kGatherThreads) idx[e] = L.fin_src[c + e];
    __syncthreads();
    if (g < NG) {
      const int e1 = n * (g + 1) / NG;
#pragma unroll 8
      for (int e = n * g / NG; e < e1; ++e) two_sum(hi, lo, __ldcg(L.src + idx[e] + i));
    }
  }
  if (g == 0)
    for (int e = L.fin_tgt_off[f]; e < L.fin_tgt_off[f + 1]; ++e) {
      const float2 v = __ldcg(L.tgt + L.fin_tgt[e] + i);
      two_sum(hi, lo, v.x);
      lo += v.y;
    }
  red[threadIdx.x] = make_float2(hi, lo);
  __syncthreads();
  if ((int)threadIdx.x >= nt) return;
  for (int h = 1; h < NG; ++h) {
    const float2 v = red[h * nt + i];
    two_sum(hi, lo, v.x);
    lo += v.y;
  }
  phi[tr.x + i] = ((double)hi + (double)lo) * kInv4PiS;
}

}  // namespace

cudaError_t launch_p2p_sym(const DevGeom& G, const DevSym& S, const float* W, double* phi, cudaStream_t st) {
  if (S.nblk == 0) return cudaSuccess;
  if (S.nlarge > 0) k_p2p_sym<true><<<S.nlarge, 128, 0, st>>>(G, S, 0, W);
  if (S.nblk > S.nlarge) k_p2p_sym<false><<<S.nblk - S.nlarge, 128, 0, st>>>(G, S, S.nlarge, W);
  k_sym_gather<<<S.nfin, kGatherThreads, 0, st>>>(G, S, phi);
  return cudaGetLastError();
}

// owner of the pair of near leaves (a, b): the deeper level, then the lower index
static inline bool sym_owns(const HostSetup& H, int a, int b) {
  return H.box[a].level != H.box[b].level ? H.box[a].level > H.box[b].level : a < b;
}

// Lane work of both forms over the mesh: the symmetric one pads an owner to a
// multiple of 16 points and spends 8 FP32 operations on a pair of points, the
// directed one pads to 4 and spends 7 on each direction.  Tiny leaves (under
// about 10 points) are better off with the latter.
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
    sym += 16 * std::ceil(nt / 16) * (ns + nt) * 8;
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
  // owners of more than 64 points (a kernel of their own) first, then longest
  // first: sources x target pairs a lane holds
  std::stable_sort(blk.begin(), blk.end(), [](const Blk& x, const Blk& y) {
    if ((x.nt > 64) != (y.nt > 64)) return x.nt > 64;
    return (x.ns + 128) * ((x.nt + 15) / 16 + 1) > (y.ns + 128) * ((y.nt + 15) / 16 + 1);
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
    out.nlarge += b.nt > 64;
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

}  // namespace bcfmm
