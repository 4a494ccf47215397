// complex64 engines of the batched form (batch_dense.cu): both registers in dense blocks and gate units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "kernels.hpp"
#include "program.hpp"

namespace qec {

constexpr int kUMaxFusion = 6;       // widest pass of the unreduced engine (slab bits)

// One pass of the unreduced engine over the slab: kind 0 applies the units punits[u0, u1) (disjoint
// slab bits, together `nbits` bits listed in bits[]); kind 1 measures the ancilla of items[item].
struct UPass {
  int32_t kind;
  int32_t item;
  int32_t u0, u1;
  int32_t nbits;
  int32_t bits[kUMaxFusion];
};

// A unit inside a pass: items[item] on slab bits qa (, qb), and the pass's other bits.  A two-qubit
// unit also carries the one-qubit units folded into its matrix: entries abs0 .. abs0 + nabs - 1 of
// the program's UAbs list.
struct UPassUnit {
  int32_t item;
  int32_t nq, qa, qb;
  int32_t nother;
  int32_t other[kUMaxFusion];
  int32_t abs0, nabs;
};

// A one-qubit unit folded into a two-qubit unit's matrix: item1's matrix on the unit's local bit
// (mode bit 1: 1 = qa, 0 = qb), multiplied from the left (mode bit 0 = 1: it follows the unit) or
// from the right (it precedes).  A unit's entries list the right factors latest first, then the
// left factors in program order.
struct UAbs {
  int32_t item1;
  int32_t mode;
};

// Time-ordered plan of one round of the unreduced register for fusion width k: consecutive units whose slab
// bits are disjoint from those already in the pass (they commute with them) join it while the pass has at
// most k bits; a unit on a bit already in the pass, or a measurement, closes it.
void build_passes(const UProgram& U, int k, std::vector<UPass>& passes, std::vector<UPassUnit>& punits,
                  std::vector<UAbs>& uabs);

// What a launch of one engine works on.
struct Batch64Args {
  // the reduced register's program (every noise and coherent slot present, or the init round's)
  const ProgOp* ops;
  const BlockInfo* blocks;
  int n_ops;
  // the unreduced register's, one round, in passes
  const ProgOp* uops;
  const UItem* uitems;
  const UPass* upasses;
  const UPassUnit* upunits;
  const UAbs* uabs;
  int n_uitems, n_upasses, n_upunits;
  const double* mats;         // [M_COUNT][16][2], the coherent ones overwritten per trajectory
  const qec_noise* noise;     // [items of the run]; null: the init round (into `out`)
  const uint64_t* traj;
  const uint32_t* idx;        // [n] items of this launch
  uint32_t n;
  unsigned int* counter;      // work queue head (zeroed before every run)
  uint64_t seed;
  uint32_t snap_item;         // item whose final data-register state goes to snap (~0u = none)
  int rounds;
  const void* psi0;           // init state: [2^9], unreduced: the slab, [2^13]
  uint8_t* syn;               // [items][rounds + 1][8]
  uint8_t* bits;              // [items][9]
  uint8_t* logical;           // [items]
  double2* snap;              // [512]
  float2* out;
};

constexpr int kSlabAmps = 1 << 13;   // 9 data qubits and the active part's 4 ancillas
constexpr int kBatchOps = 512;       // ops of a round of the reduced register, every slot present, at most
constexpr int kUMaxItems = 192;      // units and measurements of a round of the unreduced one, at most

// Reduced register: `warps` trajectories per CTA, a warp each.  occ: resident CTAs per SM (0: it doesn't fit).
cudaError_t setup_batch64(int warps, int* occ);
cudaError_t launch_batch64(const Batch64Args& a, int warps, int ctas, cudaStream_t s);
// Unreduced register: a trajectory per CTA of 128, 256 or 512 threads.
cudaError_t setup_batch64_u(int threads, int items, int* occ);
cudaError_t launch_batch64_u(const Batch64Args& a, int threads, int items, int ctas, cudaStream_t s);

}  // namespace qec
