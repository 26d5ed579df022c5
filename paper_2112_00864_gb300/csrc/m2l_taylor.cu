// CUDA-core M2L in the Taylor-coefficient form (Sec. 3.3): prescaled
// moments, per-offset derivative coefficients, register-blocked contraction
// over gamma = a + b, chunk sums reduced per target (compensated FP32).
#include <algorithm>
#include <utility>

#include "internal.h"
#include "m2l_taylor.cuh"

namespace bcfmm {
namespace {

// degree-major multi-index position: degree d = i + j + k, then i
// descending, then j descending (the order of the expansion arrays)
__host__ __device__ constexpr int mi_idx(int i, int j, int k) {
  return (i + j + k) * (i + j + k + 1) * (i + j + k + 2) / 6 + (j + k) * (j + k + 1) / 2 + k;
}

// The (a, b, gamma = a + b) triples of order Q in contraction order: gamma in
// the order of the expansion arrays (degree-major), then a by components;
// built at compile time, so that the unrolled kernel indexes its register
// arrays with constants.  Degree-major: a piece of the g row is used up before
// the next one, and the first terms need only the first moments.
__host__ __device__ constexpr int taylor_nterms(int q) {
  int n = 0;
  for (int gi = 0; gi <= q; ++gi)
    for (int gj = 0; gj <= q - gi; ++gj)
      for (int gk = 0; gk <= q - gi - gj; ++gk) n += (gi + 1) * (gj + 1) * (gk + 1);
  return n;
}
template <int Q>
struct TaylorTerms {
  static constexpr int N = taylor_nterms(Q);
  int a[N], b[N], g[N];
  __host__ __device__ constexpr TaylorTerms() : a{}, b{}, g{} {
    int n = 0;
    for (int d = 0; d <= Q; ++d)
      for (int gi = d; gi >= 0; --gi)
        for (int gj = d - gi; gj >= 0; --gj)
          for (int gk = d - gi - gj, ai = 0; ai <= gi; ++ai)
            for (int aj = 0; aj <= gj; ++aj)
              for (int ak = 0; ak <= gk; ++ak) {
                a[n] = mi_idx(ai, aj, ak);
                b[n] = mi_idx(gi - ai, gj - aj, gk - ak);
                g[n] = mi_idx(gi, gj, gk);
                ++n;
              }
  }
};
template <int Q>
struct TaylorTab {
  static constexpr TaylorTerms<Q> v{};
};
template <int Q, int I>
struct TaylorTerm {
  static constexpr int a = TaylorTab<Q>::v.a[I], b = TaylorTab<Q>::v.b[I], g = TaylorTab<Q>::v.g[I];
};
// outputs of part `part` of `nparts`: a multi-index position a belongs to part
// a % nparts (neighbouring positions have the same degree, so the parts'
// terms balance)
template <typename T, int Q, int PART, int NPARTS, int... I>
__device__ __forceinline__ void taylor_contract(T* acc, const T* m, const T* g, std::integer_sequence<int, I...>) {
  ((TaylorTerm<Q, I>::a % NPARTS == PART
        ? (void)(acc[TaylorTerm<Q, I>::a / NPARTS] =
                     fma(g[TaylorTerm<Q, I>::g], m[TaylorTerm<Q, I>::b], acc[TaylorTerm<Q, I>::a / NPARTS]))
        : (void)0),
   ...);
}

__device__ __forceinline__ void two_sum(float& hi, float& lo, float x) {
  const float t = hi + x;
  const float b = t - hi;
  lo += (hi - (t - b)) + (x - b);
  hi = t;
}

// m'[d][box][b] = m[box][d][b] * fac[b], fac[b] = (-1)^{|b|} / b!  (b < nq; zero up to the pitch)
template <typename T>
__global__ void k_taylor_prescale(const T* __restrict__ mom, int nbox, int ndp, int ms, int nq, int pitch,
                                  const T* __restrict__ fac, T* __restrict__ momp) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= (int64_t)nbox * ndp * pitch) return;
  const int64_t row = i / pitch;
  const int b = (int)(i % pitch), d = (int)(row / nbox);
  momp[i] = b < nq ? mom[((row - (int64_t)d * nbox) * ndp + d) * ms + b] * fac[b] : (T)0;
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename T>
struct TaylorArgs {
  const int4* wb;
  const int* wslot;
  const int4* ent;
  int nwarp, ndp, pitch, nbox;
  const T* momp;       // [ndp][nbox][pitch]
  const T* g;          // [27 nD][taylor_row<T>(Q)]
  T* partial;          // [nchunk][ndp][taylor_partial<T>(Q)]
};

// Sums of the higher orders (FP64 from 6, FP32 from 8) do not fit the
// registers: the outputs are dealt to two to four passes (grid z), each
// staging the rows again
template <typename T>
__host__ __device__ constexpr int taylor_parts(int q) { return sizeof(T) == 4 ? (q <= kTaylorRegQ ? 1 : 4) : (q < 6 ? 1 : q - 4); }
constexpr int kTaylorWarps = 4;       // warps per CTA
constexpr int kTaylorStageRows = 22;  // 18 g rows + 4 moment rows
// (one stage where two leave an SM a single CTA: FP32 order 8, every level of the
// level-2 ball, VtV 209 us against 230)
template <typename T>
constexpr int taylor_stages(int q) { return q >= 8 || (sizeof(T) == 8 && q >= 7) ? 1 : 2; }
template <typename T>
size_t taylor_smem(int q) {
  return sizeof(T) * (size_t)kTaylorWarps * taylor_stages<T>(q) * kTaylorStageRows * taylor_row<T>(q);
}

// One warp = one chunk of a sibling group's entries, double-buffered: while
// the lanes contract one entry, the next one's 18 g rows (one contiguous
// block) and up to four moment rows arrive by cp.async in the warp's own stage
// (no barrier between warps).  lane = target slot + 8 * source slot.
// Bound by issue and latency at eight warps an SM (order 6: issue 68 %, FMA pipe
// 57 % of its cycles, lanes 78 % filled).  With one (target, source) pair per lane and rows read by each lane from global memory
// the L1 was the bound, one distinct line per cycle: 64 a pair of row pieces,
// where an entry has 22 and fetches them coalesced.  Unit ball, level 4 (191,840
// tets, orders 6 and 7, 7.7 M pairs): VtV's whole M2L stage 0.86 -> 0.49 ms, the
// order-6 launch 0.57 -> 0.33 ms; FP64, cube of 3,072 tets against the dense
// tables, one CTA per target: 3.37 -> 0.39 ms.
// FP32 above kTaylorRegQ: every entry's products go into a compensated sum (hi,
// lo), as in the one-CTA-per-target kernel; 42 outputs a pass leave registers
// for the three arrays.  Potentials of sources far away (level-3 ball, order 8)
// against the FP64 form: 1.85e-7 with plain sums over a chunk, 1.38e-7 with one CTA
// per target, 1.20e-7 now; VtV of the level-2 ball with order 8 on every level takes
// 209 us (194 with plain sums, 3.1 ms with one CTA per target); three, five or six
// passes take 223, 213 and 225.
template <typename T, int Q, int NP>
__global__ void __launch_bounds__(kTaylorWarps * 32) k_m2l_taylor(TaylorArgs<T> A) {
  constexpr int NQ = (Q + 1) * (Q + 2) * (Q + 3) / 6;
  constexpr int ROW = taylor_row<T>(Q), SLOT = taylor_slot<T>(Q), NS = taylor_stages<T>(Q);
  constexpr int EPC = 16 / sizeof(T);            // elements per 16-byte piece
  constexpr int GP = 18 * ROW / EPC, MP = SLOT / EPC;
  constexpr int NA = (NQ + NP - 1) / NP;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int wi = threadIdx.x >> 5, w = blockIdx.x * kTaylorWarps + wi, lane = threadIdx.x & 31, d = blockIdx.y;
  if (w >= A.nwarp) return;
  T* stage = reinterpret_cast<T*>(smraw) + (size_t)wi * NS * kTaylorStageRows * ROW;
  const int4 wb = A.wb[w];
  const int t = lane & 7, s = lane >> 3;
  const int to = (wb.z >> (3 * t)) & 7;
  const bool tlive = t < wb.w;
  const T* momd = A.momp + (int64_t)d * A.nbox * A.pitch;
  auto load = [&](const int4 e, T* sp) {
    const char* gs = reinterpret_cast<const char*>(A.g + (int64_t)e.y * ROW);
    char* gd = reinterpret_cast<char*>(sp);
#pragma unroll
    for (int i = 0; i < (GP + 31) / 32; ++i) {
      const int k = i * 32 + lane;
      if ((i + 1) * 32 <= GP || k < GP) cp_async16(gd + 16 * k, gs + 16 * k);
    }
    const unsigned sb = ((unsigned)e.z >> (8 * s)) & 255u;
    if (sb) {
      const char* ms = reinterpret_cast<const char*>(momd + (int64_t)(e.x + (int)(sb & 7u)) * A.pitch);
      char* md = reinterpret_cast<char*>(sp + (18 + s) * ROW);
#pragma unroll
      for (int i = 0; i < (MP + 7) / 8; ++i) {
        const int k = i * 8 + t;
        if (k < MP) cp_async16(md + 16 * k, ms + 16 * k);
      }
    }
  };
  constexpr bool COMP = taylor_comp<T>(Q);
  T acc[NA], lo[COMP ? NA : 1], sum[COMP ? NA : 1];
#pragma unroll
  for (int a = 0; a < NA; ++a) acc[a] = (T)0;
  if constexpr (COMP) {
#pragma unroll
    for (int a = 0; a < NA; ++a) sum[a] = lo[a] = (T)0;
  }
  int4 cur = A.ent[wb.x], nxt = cur;
  load(cur, stage);
  cp_async_commit();
  if (wb.y > 1) nxt = A.ent[wb.x + 1];
  for (int j = 0; j < wb.y; ++j) {
    int4 nn = nxt;
    if (NS == 2) {
      if (j + 1 < wb.y) load(nxt, stage + ((j + 1) & 1) * kTaylorStageRows * ROW);
      cp_async_commit();
      if (j + 2 < wb.y) nn = A.ent[wb.x + j + 2];
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
      if (j + 2 < wb.y) nn = A.ent[wb.x + j + 2];
    }
    __syncwarp();
    const unsigned sb = ((unsigned)cur.z >> (8 * s)) & 255u;
    const int so = (int)(sb >> 3);
    const int row = (to >> 2) * 9 + (((to >> 1) & 1) - ((so >> 1) & 1) + 1) * 3 + ((to & 1) - (so & 1) + 1);
    if (tlive && sb && (cur.w >> row & 1)) {
      const T* sp = stage + (NS == 2 ? (j & 1) : 0) * kTaylorStageRows * ROW;
      const T* gr = sp + row * ROW;
      const T* mr = sp + (18 + s) * ROW;
      // every (a, b) with |a + b| <= Q
      constexpr auto terms = std::make_integer_sequence<int, taylor_nterms(Q)>{};
      if constexpr (NP == 1 && sizeof(T) == 4) {
        T m[MP * EPC], g[MP * EPC];
#pragma unroll
        for (int v = 0; v < MP; ++v) {
          *reinterpret_cast<float4*>(m + v * EPC) = *reinterpret_cast<const float4*>(mr + v * EPC);
          *reinterpret_cast<float4*>(g + v * EPC) = *reinterpret_cast<const float4*>(gr + v * EPC);
        }
        taylor_contract<T, Q, 0, NP>(acc, m, g, terms);
      } else if (NP == 1 || blockIdx.z == 0) {
        // (operands straight from shared memory: the FP64 pipe is slow enough,
        // and the FP32 orders above 7 have few targets)
        taylor_contract<T, Q, 0, NP>(acc, mr, gr, terms);
      } else if (NP == 2 || blockIdx.z == 1) {
        taylor_contract<T, Q, 1 % NP, NP>(acc, mr, gr, terms);
      } else if (NP == 3 || blockIdx.z == 2) {
        taylor_contract<T, Q, 2 % NP, NP>(acc, mr, gr, terms);
      } else {
        taylor_contract<T, Q, 3 % NP, NP>(acc, mr, gr, terms);
      }
      if constexpr (COMP) {
#pragma unroll
        for (int a = 0; a < NA; ++a) {
          two_sum(sum[a], lo[a], acc[a]);
          acc[a] = (T)0;
        }
      }
    }
    __syncwarp();
    if (NS == 1 && j + 1 < wb.y) {
      load(nxt, stage);
      cp_async_commit();
    }
    cur = nxt;
    nxt = nn;
  }
  // the four lanes of a target
  if constexpr (COMP) {
#pragma unroll
    for (int a = 0; a < NA; ++a) {
#pragma unroll
      for (int m = 8; m <= 16; m <<= 1) {
        const T h = __shfl_xor_sync(0xffffffffu, sum[a], m), l = __shfl_xor_sync(0xffffffffu, lo[a], m);
        two_sum(sum[a], lo[a], h);
        lo[a] += l;
      }
    }
  } else {
#pragma unroll
    for (int a = 0; a < NA; ++a) {
      acc[a] += __shfl_xor_sync(0xffffffffu, acc[a], 8);
      acc[a] += __shfl_xor_sync(0xffffffffu, acc[a], 16);
    }
  }
  if (!tlive || s != 0) return;
  const int c = A.wslot[w * 8 + t];
  T* o = A.partial + ((int64_t)c * A.ndp + d) * taylor_partial<T>(Q);
  if constexpr (COMP) {
#pragma unroll
    for (int a = 0; a < NA; ++a)
      if (a * NP + (int)blockIdx.z < NQ) {
        o[a * NP + blockIdx.z] = sum[a];
        o[SLOT + a * NP + blockIdx.z] = lo[a];
      }
  } else if constexpr (NP == 1) {
#pragma unroll
    for (int v = 0; v < SLOT / EPC; ++v) {
      T x[EPC];
#pragma unroll
      for (int i = 0; i < EPC; ++i) x[i] = v * EPC + i < NQ ? acc[v * EPC + i < NQ ? v * EPC + i : 0] : (T)0;
      *reinterpret_cast<float4*>(o + v * EPC) = *reinterpret_cast<float4*>(x);
    }
  } else {
#pragma unroll
    for (int a = 0; a < NA; ++a)
      if (a * NP + (int)blockIdx.z < NQ) o[a * NP + blockIdx.z] = acc[a];
  }
}

// loc[t][d][a] = post[a] / s_t * (sum over the target's chunks, in chunk
// order, FP32: compensated), post[a] = 1 / a!; one thread per (target, d, a).
// slot: values of a chunk's sums; OFF: its lo parts' offset there (0: none)
template <typename T, int OFF>
__global__ void __launch_bounds__(128) k_m2l_taylor_reduce(int ntgt, const int* __restrict__ tgt,
                                                          const int* __restrict__ tchunk,
                                                          const T* __restrict__ partial, int nq, int slot,
                                                          int ndp, int ms, const T* __restrict__ post,
                                                          const double4_32a* __restrict__ box_cs,
                                                          T* __restrict__ loc) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int per = ndp * nq;
  if (i >= (int64_t)ntgt * per) return;
  const int t = (int)(i / per), r = (int)(i % per), d = r / nq, a = r % nq;
  const int tb = tgt[t], c0 = tchunk[t], c1 = tchunk[t + 1];
  T hi = 0, lo = 0;
  const T* pp = partial + (int64_t)d * slot + a;
#pragma unroll 4
  for (int c = c0; c < c1; ++c) {
    const T x = __ldg(pp + (int64_t)c * ndp * slot);
    if constexpr (sizeof(T) == 4) two_sum(hi, lo, x);
    else hi += x;
    if constexpr (OFF > 0) lo += __ldg(pp + (int64_t)c * ndp * slot + OFF);
  }
  loc[((int64_t)tb * ndp + d) * ms + a] = (hi + lo) * post[a] / (T)box_cs[tb].w;
}

// Orders above the register-blocked range (any q <= p): one CTA per target,
// the entry's g row and prescaled moment row staged in shared memory, one
// thread per output a (strided), the multi-index of a + b computed from the
// components; FP32 products per entry, compensated FP32 sum over the list.
template <int ND>
__global__ void __launch_bounds__(128) k_m2l_taylor_wide(DevGeom G, DevTaskLists L, const int* __restrict__ sel,
                                                        const float* __restrict__ g, int pitch,
                                                        const float* __restrict__ momp, const float* __restrict__ post,
                                                        float* __restrict__ loc) {
  constexpr int ndp = ND;
  extern __shared__ float wsm[];
  const int ki = sel[blockIdx.x];
  const int tb = L.m2l_tgt[ki];
  const int q = G.box_q[tb], nq = nterms_q(q);
  float* sg = wsm;                       // [nq] the entry's g row
  float* smv = sg + pitch;               // [ndp][nq] its prescaled moment rows
  int* smi = reinterpret_cast<int*>(smv + (size_t)ndp * pitch);   // [nq] packed multi-indices
  for (int i = threadIdx.x; i < nq; i += blockDim.x) smi[i] = G.mi[i];
  constexpr int kMaxPer = 4;             // outputs per thread: nq <= 4 * 128 (q <= 12)
  constexpr int kMaxD = ND;
  float hi[kMaxPer][kMaxD], lo[kMaxPer][kMaxD];
#pragma unroll
  for (int u = 0; u < kMaxPer; ++u)
#pragma unroll
    for (int d = 0; d < kMaxD; ++d) hi[u][d] = lo[u][d] = 0.f;
  const int e0 = L.vl_off[ki], e1 = L.vl_off[ki + 1];
  for (int e = e0; e < e1; ++e) {
    const int sb = L.vl_src[e];
    const float* gr = g + (int64_t)L.vl_code[e] * pitch;
    __syncthreads();
    for (int i = threadIdx.x; i < nq; i += blockDim.x) sg[i] = gr[i];
    for (int i = threadIdx.x; i < ndp * nq; i += blockDim.x)
      smv[(i / nq) * pitch + i % nq] = momp[((int64_t)(i / nq) * G.nbox + sb) * pitch + i % nq];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kMaxPer; ++u) {
      const int a = threadIdx.x + u * 128;
      if (a >= nq) break;
      const int ma = smi[a];
      const int ai = ma & 255, aj = (ma >> 8) & 255, ak = (ma >> 16) & 255;
      const int kb = nterms_q(q - ai - aj - ak);
      float part[kMaxD];
#pragma unroll
      for (int d = 0; d < kMaxD; ++d) part[d] = 0.f;
      for (int b = 0; b < kb; ++b) {
        const int mb = smi[b];
        const int gi = ai + (mb & 255), gj = aj + ((mb >> 8) & 255), gk = ak + ((mb >> 16) & 255);
        const int dg = gi + gj + gk;
        const float gv = sg[dg * (dg + 1) * (dg + 2) / 6 + (gj + gk) * (gj + gk + 1) / 2 + gk];
#pragma unroll
        for (int d = 0; d < kMaxD; ++d) part[d] = fmaf(gv, smv[d * pitch + b], part[d]);
      }
#pragma unroll
      for (int d = 0; d < kMaxD; ++d) two_sum(hi[u][d], lo[u][d], part[d]);
    }
  }
  const float inv_s = 1.0f / (float)G.box_cs[tb].w;
#pragma unroll
  for (int u = 0; u < kMaxPer; ++u) {
    const int a = threadIdx.x + u * 128;
    if (a >= nq) break;
    for (int d = 0; d < ndp; ++d) loc[((int64_t)tb * ndp + d) * G.ms + a] = (hi[u][d] + lo[u][d]) * post[a] * inv_s;
  }
}

template <typename T, int Q>
cudaError_t launch_order(const TaylorOrderSched& O, const TaylorTables& tab, const DevGeom& G, int ndp, const T* momp,
                         T* loc, T* partial, cudaStream_t st) {
  constexpr int NQ = (Q + 1) * (Q + 2) * (Q + 3) / 6, NP = taylor_parts<T>(Q);
  TaylorArgs<T> A;
  A.wb = O.wb;
  A.wslot = O.wslot;
  A.ent = O.ent;
  A.nwarp = O.nwarp;
  A.ndp = ndp;
  A.pitch = tab.gpitch;
  A.nbox = G.nbox;
  A.momp = momp;
  A.g = static_cast<const T*>(O.g);
  A.partial = partial;
  const size_t sm = taylor_smem<T>(Q);
  cudaError_t e = cudaFuncSetAttribute(k_m2l_taylor<T, Q, NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  k_m2l_taylor<T, Q, NP><<<dim3((unsigned)((O.nwarp + kTaylorWarps - 1) / kTaylorWarps), (unsigned)ndp, NP),
                           kTaylorWarps * 32, sm, st>>>(A);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int64_t n = (int64_t)O.ntgt * ndp * NQ;
  constexpr int OFF = taylor_comp<T>(Q) ? taylor_slot<T>(Q) : 0;
  k_m2l_taylor_reduce<T, OFF><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(
      O.ntgt, O.tgt, O.tchunk, partial, NQ, taylor_partial<T>(Q), ndp, G.ms,
      static_cast<const T*>(tab.fac) + tab.gpitch, G.box_cs, loc);
  return cudaGetLastError();
}

}  // namespace

int m2l_taylor_pitch(int q) { return (nterms_q(q) + 7) / 8 * 8; }

void m2l_taylor_schedule(const HostSetup& H, int task, const std::vector<int>& target_q, int nsm, TaylorOffsets& offs,
                         std::vector<TaylorOrderHost>& out, std::vector<int>& sel) {
  const HostTask& T = H.task[task];
  const int sc = T.src_cls;
  out.clear();
  sel.clear();
  const int nt = (int)T.m2l_tgt.size();
  for (int k = 0; k < nt; ++k)
    if (target_q[k] < 1 || target_q[k] > kTaylorMaxQ) sel.push_back(k);
  // index of a parent offset; components lie within +-63 (see build_lists)
  std::vector<int> dmap((size_t)1 << 21, -1);
  auto dkey = [](int x, int y, int z) { return (size_t)((z + 64) << 14 | (y + 64) << 7 | (x + 64)); };
  for (size_t i = 0; i < offs.d.size() / 3; ++i) dmap[dkey(offs.d[3 * i], offs.d[3 * i + 1], offs.d[3 * i + 2])] = (int)i;
  std::vector<int> mark(H.box.size(), -1);
  for (int q = 1; q <= kTaylorMaxQ; ++q) {
    TaylorOrderHost O;
    O.q = q;
    // sibling groups: boxes are stored level by level, children of one parent
    // in a row, and the target list is in box order
    std::vector<std::vector<int>> groups;
    int last = -1;
    for (int k = 0; k < nt; ++k) {
      if (target_q[k] != q || T.vl_off[k + 1] == T.vl_off[k]) continue;
      const int par = H.box[T.m2l_tgt[k]].parent;
      if (groups.empty() || par != last || groups.back().size() == 8) groups.emplace_back();
      last = par;
      groups.back().push_back(k);
      O.pairs += T.vl_off[k + 1] - T.vl_off[k];
    }
    if (groups.empty()) continue;
    std::vector<int4> all;                        // the groups' entries
    std::vector<size_t> goff(1, 0);
    std::vector<std::pair<int, int>> qs;          // (offset key, Q)
    for (size_t g = 0; g < groups.size(); ++g) {
      const int pb = H.box[T.m2l_tgt[groups[g][0]]].parent;
      const HostBox& P = H.box[pb];
      qs.clear();
      for (int k : groups[g])
        for (int e = T.vl_off[k]; e < T.vl_off[k + 1]; ++e) {
          const int qb = H.box[T.vl_src[e]].parent;
          if (mark[qb] == (int)g) continue;
          mark[qb] = (int)g;
          const HostBox& Q = H.box[qb];
          qs.push_back({(int)dkey((int)(P.ijk[0] - Q.ijk[0]), (int)(P.ijk[1] - Q.ijk[1]), (int)(P.ijk[2] - Q.ijk[2])), qb});
        }
      std::sort(qs.begin(), qs.end());
      for (const auto& x : qs) {
        const HostBox& Q = H.box[x.second];
        const int D[3] = {(int)(P.ijk[0] - Q.ijk[0]), (int)(P.ijk[1] - Q.ijk[1]), (int)(P.ijk[2] - Q.ijk[2])};
        int& di = dmap[x.first];
        if (di < 0) {
          di = (int)(offs.d.size() / 3);
          offs.d.insert(offs.d.end(), D, D + 3);
        }
        for (int z = 0; z < 2; ++z) {
          // rows oz * 9 + (dy + 1) * 3 + dx + 1: offset 2 D + (dx, dy, oz - z)
          unsigned far = 0, src = 0, used = 0;
          for (int r = 0; r < 18; ++r) {
            const int o[3] = {2 * D[0] + r % 3 - 1, 2 * D[1] + r / 3 % 3 - 1, 2 * D[2] + r / 9 - z};
            if (!((double)(o[0] * o[0] + o[1] * o[1] + o[2] * o[2]) * H.eta0 * H.eta0 < 3.0)) far |= 1u << r;
          }
          int n = 0;
          for (int c = 0; c < Q.nchild; ++c) {
            const HostBox& C = H.box[Q.child0 + c];
            if ((C.octant >> 2) != z || C.pt1[sc] == C.pt0[sc]) continue;
            src |= (unsigned)(c | C.octant << 3 | 0x40) << (8 * n++);
            for (int k : groups[g]) {
              const int to = H.box[T.m2l_tgt[k]].octant;
              used |= 1u << ((to >> 2) * 9 + ((to >> 1 & 1) - (C.octant >> 1 & 1) + 1) * 3 + (to & 1) - (C.octant & 1) + 1);
            }
          }
          if (!n || !(far & used)) continue;
          all.push_back(make_int4(Q.child0, 27 * di + 9 * (1 - z), (int)src, (int)far));
        }
      }
      goff.push_back(all.size());
    }
    for (size_t g = 0; g < groups.size(); ++g)      // (marks of this order must not meet the next one's)
      for (int k : groups[g])
        for (int e = T.vl_off[k]; e < T.vl_off[k + 1]; ++e) mark[H.box[T.vl_src[e]].parent] = -1;
    // entries per chunk: about four rounds of the eight warps that an SM
    // holds, at most 32 (the FP32 sum of a chunk stays short), at least 4
    // (partial-sum traffic)
    O.chunk = (int)std::min<int64_t>(32, std::max<int64_t>(4, ((int64_t)all.size() + 32LL * nsm - 1) / (32LL * nsm)));
    struct Unit { int group, first, n, piece; };
    std::vector<Unit> units;
    O.tchunk.assign(1, 0);
    std::vector<int> slot0(groups.size()), nchunk(groups.size());
    for (size_t g = 0; g < groups.size(); ++g) {
      const int n = (int)(goff[g + 1] - goff[g]), nc = (n + O.chunk - 1) / O.chunk;
      nchunk[g] = nc;
      slot0[g] = O.tchunk.back();
      for (int k : groups[g]) {
        O.tgt.push_back(T.m2l_tgt[k]);
        O.tchunk.push_back(O.tchunk.back() + nc);
      }
      for (int i = 0; i < nc; ++i) {
        const int b0 = (int)((int64_t)n * i / nc), b1 = (int)((int64_t)n * (i + 1) / nc);
        units.push_back({(int)g, b0, b1 - b0, i});
      }
    }
    O.nchunk = O.tchunk.back();
    // longest chunks first; equal ones stay in group order (neighbouring
    // groups share sources)
    std::stable_sort(units.begin(), units.end(), [](const Unit& a, const Unit& b) { return a.n > b.n; });
    for (const Unit& u : units) {
      const std::vector<int>& G = groups[u.group];
      int oct = 0;
      for (size_t t = 0; t < G.size(); ++t) oct |= H.box[T.m2l_tgt[G[t]]].octant << (3 * t);
      O.wb.push_back(make_int4((int)goff[u.group] + u.first, u.n, oct, (int)G.size()));
      for (int t = 0; t < 8; ++t)
        O.wslot.push_back(t < (int)G.size() ? slot0[u.group] + t * nchunk[u.group] + u.piece : -1);
    }
    O.ent = std::move(all);
    out.push_back(std::move(O));
  }
}

template <typename T>
void m2l_taylor_rows(const TaylorOffsets& offs, int q, std::vector<T>& rows) {
  const int nd = (int)(offs.d.size() / 3), row = taylor_row<T>(q), n = nterms_q(q);
  rows.assign((size_t)nd * 27 * row, (T)0);
#pragma omp parallel for schedule(static)
  for (int i = 0; i < nd * 27; ++i) {
    const int* D = &offs.d[3 * (i / 27)];
    const int r = i % 27;
    const double o[3] = {2.0 * D[0] + r % 3 - 1, 2.0 * D[1] + r / 3 % 3 - 1, 2.0 * D[2] + r / 9 - 1};
    if (o[0] == 0 && o[1] == 0 && o[2] == 0) continue;      // the box itself: never far
    std::vector<double> g(n);
    m2l_taylor_coeffs(q, o, g.data());
    for (int k = 0; k < n; ++k) rows[(size_t)i * row + k] = (T)g[k];
  }
}
template void m2l_taylor_rows<float>(const TaylorOffsets&, int, std::vector<float>&);
template void m2l_taylor_rows<double>(const TaylorOffsets&, int, std::vector<double>&);

template <typename T>
cudaError_t launch_m2l_taylor(const DevGeom& G, const DevTaskLists& L, const TaylorTaskSched& S,
                              const TaylorTables& tab, int ndp, const T* mom, T* loc, T* momp, T* partial,
                              cudaStream_t main, const TaylorFork* side) {
  cudaStream_t st = main;
  int qtop = 0;
  for (int q = 1; q <= kTaylorMaxQ; ++q)
    if (S.ord[q].nwarp > 0) qtop = q;
  const bool wide = sizeof(T) == 4 && S.nsimt > 0;
  if (qtop == 0 && !wide) return cudaSuccess;
  if (qtop > tab.q || tab.gpitch != m2l_taylor_pitch(tab.q) || ndp > 16 || tab.q > 12) return cudaErrorInvalidValue;
  {
    const int64_t n = (int64_t)G.nbox * ndp * tab.gpitch;
    k_taylor_prescale<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(mom, G.nbox, ndp, G.ms, nterms_q(tab.q), tab.gpitch,
                                                                      static_cast<const T*>(tab.fac), momp);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if constexpr (sizeof(T) == 4) {
    if (wide) {
      const size_t sm = sizeof(float) * (size_t)(1 + ndp) * tab.gpitch + sizeof(int) * tab.gpitch;
      const float* post = static_cast<const float*>(tab.fac) + tab.gpitch;
      switch (ndp) {
        case 1: k_m2l_taylor_wide<1><<<S.nsimt, 128, sm, st>>>(G, L, S.simt_sel, tab.g, tab.gpitch, momp, post, loc); break;
        case 2: k_m2l_taylor_wide<2><<<S.nsimt, 128, sm, st>>>(G, L, S.simt_sel, tab.g, tab.gpitch, momp, post, loc); break;
        case 4: k_m2l_taylor_wide<4><<<S.nsimt, 128, sm, st>>>(G, L, S.simt_sel, tab.g, tab.gpitch, momp, post, loc); break;
        case 8: k_m2l_taylor_wide<8><<<S.nsimt, 128, sm, st>>>(G, L, S.simt_sel, tab.g, tab.gpitch, momp, post, loc); break;
        case 16: k_m2l_taylor_wide<16><<<S.nsimt, 128, sm, st>>>(G, L, S.simt_sel, tab.g, tab.gpitch, momp, post, loc); break;
        default: return cudaErrorInvalidValue;
      }
      const cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
  }
  int norder = 0;
  for (int q = 1; q <= kTaylorMaxQ; ++q) norder += S.ord[q].nwarp > 0;
  const bool fork = side && side->side && norder > 1;
  if (fork) {
    cudaError_t e = cudaEventRecord(side->fork, main);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(side->side, side->fork, 0);
    if (e != cudaSuccess) return e;
  }
  int k = 0;
  for (int q = 1; q <= kTaylorMaxQ; ++q) {
    const TaylorOrderSched& O = S.ord[q];
    if (O.nwarp == 0) continue;
    st = fork && (k++ & 1) ? side->side : main;
    cudaError_t e = cudaSuccess;
    switch (q) {
      case 1: e = launch_order<T, 1>(O, tab, G, ndp, momp, loc, partial, st); break;
      case 2: e = launch_order<T, 2>(O, tab, G, ndp, momp, loc, partial, st); break;
      case 3: e = launch_order<T, 3>(O, tab, G, ndp, momp, loc, partial, st); break;
      case 4: e = launch_order<T, 4>(O, tab, G, ndp, momp, loc, partial, st); break;
      case 5: e = launch_order<T, 5>(O, tab, G, ndp, momp, loc, partial, st); break;
      case 6: e = launch_order<T, 6>(O, tab, G, ndp, momp, loc, partial, st); break;
      case 7: e = launch_order<T, 7>(O, tab, G, ndp, momp, loc, partial, st); break;
      case 8: e = launch_order<T, 8>(O, tab, G, ndp, momp, loc, partial, st); break;
      default: e = cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    partial += (size_t)O.nchunk * ndp * taylor_partial<T>(q);
  }
  if (fork) {
    cudaError_t e = cudaEventRecord(side->join, side->side);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(main, side->join, 0);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
template cudaError_t launch_m2l_taylor<float>(const DevGeom&, const DevTaskLists&, const TaylorTaskSched&, const TaylorTables&,
                                              int, const float*, float*, float*, float*, cudaStream_t, const TaylorFork*);
template cudaError_t launch_m2l_taylor<double>(const DevGeom&, const DevTaskLists&, const TaylorTaskSched&, const TaylorTables&,
                                               int, const double*, double*, double*, double*, cudaStream_t, const TaylorFork*);

}  // namespace bcfmm
