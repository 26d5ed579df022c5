// Symmetric FP32 near field of VtV (one, two or four densities): every pair of
// points is evaluated once and serves both of its directions.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "kernels.cuh"

namespace bcfmm {

struct HostSetup;

// Near-field pairs are symmetric in VtV (sources and targets are the tet
// points, and B is in A's extended neighbour list exactly when A is in B's).
// Of two leaves in each other's list the one on the deeper level owns the
// pair (the lower box index on one level): its frame is the finer one, so
// translated FP32 coordinates lose nothing against either leaf's own.  An
// owner's sources are cut into blocks at leaf boundaries.  A block writes, per
// source point, the sum over the owner's points to its own slots src[], and
// per owner point the sum over the block's sources to tgt[]; the gather kernel
// adds, per point, the slots that belong to it in a fixed order, so the result
// does not depend on the order in which blocks run.
struct DevSym {
  int nblk = 0, nlarge = 0;         // the first nlarge blocks: owners of more than 32 points
  const int* leaf = nullptr;        // [nblk] owner
  const int* run_off = nullptr;     // [nblk + 1] into runs
  const int2* runs = nullptr;       // source runs (start, end), without the owner's own points
  const int2* base = nullptr;       // [nblk] (first src slot, first tgt slot)
  const int* self = nullptr;        // [nblk] 1: the block also holds the owner's own points
  int64_t nsrc = 0, ntgt = 0;       // slots
  int cap = 0;                      // densities that the slots hold (0: no slots)
  float* src = nullptr;             // [nsrc][ndp] source-side sums
  float2* tgt = nullptr;            // [ntgt][ndp] owner-side sums (hi, lo)
  // gather kernel, per target leaf (most slots first)
  int nfin = 0;
  const int* fin_leaf = nullptr;
  const int* fin_tgt_off = nullptr;  // [nfin + 1] into fin_tgt: tgt slots of the leaf's own blocks
  const int* fin_tgt = nullptr;
  const int* fin_src_off = nullptr;  // [nfin + 1] into fin_src: src slots where the leaf is a source
  const int* fin_src = nullptr;
};

struct HostSym {
  std::vector<int> leaf, run_off, runs, base, self;   // runs, base as pairs
  std::vector<int> fin_leaf, fin_tgt_off, fin_tgt, fin_src_off, fin_src;
  int nlarge = 0;
  int64_t nsrc = 0, ntgt = 0;                          // slots
};
// Blocks of at most about `chunk` sources.  Returns false (nothing built)
// when the slots do not fit 32-bit offsets.
bool build_p2p_sym(const HostSetup& H, int64_t chunk, HostSym& out);
// sources per block: enough blocks for every SM, at most kSymChunkMax
constexpr int64_t kSymChunkMin = 512, kSymChunkMax = 4096;
int64_t p2p_sym_chunk(const HostSetup& H, int nsm);
// Faults of a schedule of build_p2p_sym (host check): pairs, a pair of near leaves
// (or of a leaf with itself) not in exactly one block; slots, a slot that is not
// written once and gathered once, for the same point; blocks, one whose sources
// exceed the chunk by more than a leaf, or out of the order the launches rely on.
struct SymFaults { int64_t pairs = 0, slots = 0, blocks = 0; };
SymFaults check_p2p_sym(const HostSetup& H, int64_t chunk, const HostSym& S);
bool p2p_sym_pays(const HostSetup& H);

// densities (padded) that the symmetric form takes; more need too many registers
constexpr int kSymDens = 4;
inline bool p2p_sym_takes(const DevSym& S, int ndp) { return ndp <= kSymDens && ndp <= S.cap; }
// phi = near field of VtV / 4 pi (every target point; npts points per density in W and phi)
cudaError_t launch_p2p_sym(const DevGeom& G, const DevSym& S, const float* W, int64_t npts, int ndp, double* phi, cudaStream_t st);

}  // namespace bcfmm
