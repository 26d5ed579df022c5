// CUDA-core M2L of the boundary-concentrated FMM in the Taylor-coefficient
// form (FP32 products with compensated sums over work chunks, or FP64).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "kernels.cuh"

namespace bcfmm {

struct HostSetup;

// Largest order handled by the sibling-group kernel (higher orders, up to
// 12, go to a one-CTA-per-target kernel: in the same Taylor form in FP32, with
// the dense table in FP64), and the largest whose FP32 sums stay in
// registers, which the statistics list order by order.
constexpr int kTaylorMaxQ = 8, kTaylorRegQ = 7;

// The expansion coefficients of Sec. 3.3,
//   lambda^a = sum_{|b| <= q - |a|} D^{a+b} G(o) / (a! b!) (-1)^{|b|} m^b,
// depend on the offset o only through the derivatives D^gamma G(o),
// |gamma| <= q: with prescaled moments m'_b = (-1)^{|b|} m^b / b! and
// g_o[gamma] = D^gamma G(o) = D^gamma (1/r)(o) / (4 pi),
//   lambda^a = (1/a!) sum_b g_o[a + b] m'_b,
// so one offset needs nterms(q) numbers instead of an nterms(q)^2 matrix,
// and the product costs one FMA per (a, b) with |a| + |b| <= q.  (Box-
// scaled expansions: o is the integer offset in units of the box side s,
// and the stored local is lambda / s.)
//
// Work of one order: the targets with a common parent P (up to eight
// siblings) have their sources among the children of P's neighbours Q, and
// for one Q the 64 (target, source) pairs have 27 offsets, 2 D + {-1, 0, 1}^3
// with D the offset of the parents.  An entry is one Q and one z-plane of its
// children: up to four sources, whose offsets to the eight targets are 18
// consecutive rows of D's 27 (the table holds the rows of a D together).  A
// warp walks a chunk of P's entries, lane = target slot + 8 * source slot; it
// adds the four lanes of a target at the end and writes the sum to the
// target's slot of that chunk (FP32 order 8: a compensated sum, hi and lo).  A
// second kernel adds a target's slots in chunk order (FP32: compensated;
// deterministic) and stores the local expansion.
struct TaylorOrderSched {
  int q = 0, nwarp = 0, nchunk = 0, ntgt = 0, chunk = 0;
  int64_t pairs = 0;
  const int4* wb = nullptr;          // [nwarp] (first entry, entries, target octants (3 bits each), targets)
  const int* wslot = nullptr;        // [nwarp * 8] partial slot of each target (-1: none)
  const int4* ent = nullptr;         // (Q's first child, first g row, source bytes, far mask): see taylor_entry
  const int* tgt = nullptr;          // [ntgt] target boxes
  const int* tchunk = nullptr;       // [ntgt + 1] slot range of each target
  const void* g = nullptr;           // [27 nD][taylor_row<T>(q)] offset coefficients
};
// One source of an entry, byte i of its third word: child slot of Q | octant
// << 3 | 0x40; zero: none.  The far mask's bit oz * 9 + (dy + 1) * 3 + dx + 1
// (oz: the target's z bit; dx, dy: target minus source bits) says whether
// that offset is in the interaction list; it is also the offset's row among
// the entry's 18.
struct TaylorTaskSched {
  TaylorOrderSched ord[kTaylorMaxQ + 1];   // index = order q (nwarp 0: none)
  size_t partial_per_dens = 0;             // values of chunk partial sums per density (all orders)
  const int* simt_sel = nullptr;           // targets (indices into the task's list) of
  int nsimt = 0;                           // higher orders: one CTA per target
};

// Host side of one order's schedule (built at setup, uploaded by the caller).
struct TaylorOrderHost {
  int q = 0, nchunk = 0, chunk = 0;
  int64_t pairs = 0;
  std::vector<int4> wb, ent;         // ent[].y: first row of the entry's 18 (27 D + 9 (1 - z))
  std::vector<int> wslot, tgt, tchunk;
};
// The parent offsets D that occur, in the order of their first use: the g
// tables hold 27 rows for each.
struct TaylorOffsets {
  std::vector<int> d;                // (x, y, z) per D
};
// target_q[k]: order of the task's k-th M2L target.  Orders 1..kTaylorMaxQ
// are scheduled; `sel` receives the targets of every other order.  offs is
// shared by the tasks and grows.
void m2l_taylor_schedule(const HostSetup& H, int task, const std::vector<int>& target_q, int nsm, TaylorOffsets& offs,
                         std::vector<TaylorOrderHost>& out, std::vector<int>& sel);

// Elements of a g row and of a staged moment row: a row is an odd number of
// 16-byte pieces, so that the rows that the lanes of a warp read at one column
// fall in different shared-memory banks.
template <typename T>
__host__ __device__ constexpr int taylor_row(int q) {
  return (int)((((q + 1) * (q + 2) * (q + 3) / 6 * sizeof(T) + 15) / 16 | 1) * 16 / sizeof(T));
}
// elements of a partial slot: a whole number of 16-byte pieces
template <typename T>
__host__ __device__ constexpr int taylor_slot(int q) {
  return (int)(((q + 1) * (q + 2) * (q + 3) / 6 * sizeof(T) + 15) / 16 * 16 / sizeof(T));
}
// whether a chunk's sums are compensated entry by entry, (hi, lo) in its slot, and
// the slot's elements then
template <typename T>
__host__ __device__ constexpr bool taylor_comp(int q) { return sizeof(T) == 4 && q > kTaylorRegQ; }
template <typename T>
__host__ __device__ constexpr int taylor_partial(int q) { return taylor_slot<T>(q) * (taylor_comp<T>(q) ? 2 : 1); }
// g rows of one order for the parent offsets offs (host, FP64 -> T)
template <typename T>
void m2l_taylor_rows(const TaylorOffsets& offs, int q, std::vector<T>& rows);

// Offset coefficients of the one-CTA-per-target kernel (FP32, per interaction
// offset code, [ncode][gpitch], |gamma| <= q; null when no target needs it) and the
// multi-index factors fac[0..gpitch) = (-1)^{|b|} / b! (moments),
// fac[gpitch..2 gpitch) = 1 / a! (locals), in FP32 and FP64.
struct TaylorTables {
  const float* g = nullptr;
  const void* fac = nullptr;         // element type of the context's expansions
  int gpitch = 0, q = 0;
};
// row pitch (elements, a multiple of 8) of the prescaled moments for order q
int m2l_taylor_pitch(int q);

// Scratch (device memory owned by the caller):
//   momp:    ndp * nbox * m2l_taylor_pitch(tab.q) values (prescaled moments, density-major)
//   partial: ndp * S.partial_per_dens values (chunk sums)
// tab.q must be the largest order of any target (the wide kernel reads the
// g rows and moments up to it); targets in S.simt_sel use the wide kernel
// (FP32; an FP64 caller runs the dense kernel for them).
// side: a second stream for every other order (their targets differ, and
// each order has its own part of `partial`), joined before the call returns;
// null: all on st.
struct TaylorFork {
  cudaStream_t side = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
};
template <typename T>
cudaError_t launch_m2l_taylor(const DevGeom& G, const DevTaskLists& L, const TaylorTaskSched& S,
                              const TaylorTables& tab, int ndp, const T* mom, T* loc, T* momp, T* partial,
                              cudaStream_t st, const TaylorFork* side = nullptr);

}  // namespace bcfmm
