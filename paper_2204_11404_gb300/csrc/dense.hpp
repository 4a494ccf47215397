// Launch interface of the complex64 trajectories in dense blocks (dense.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.hpp"

namespace qec {

constexpr int kDenseOps = 64;   // ops of one block, at most

struct DenseArgs {
  const ProgOp* ops;
  const BlockInfo* blocks;
  const double* mats;       // [M_COUNT][16][2]
  double prob[PR_COUNT];
  int nstab, nd, rounds, nl;   // nl: data qubits 0..nl-1 make the raw logical parity
  int entries;              // of one stored Kraus matrix (dense_entries)
  unsigned long long seed, first;
  uint32_t n;               // trajectories of this launch
  const void* psi0;         // [2^nd] complex64
  float2* kraus;            // [n][rounds nstab][2][entries]: K_0, K_1
  double* u;                // [n][rounds nstab] measurement uniforms
  void* psi_out;            // the last trajectory's final state (null: none)
  uint8_t* syn;             // [n][rounds + 1][nstab] (null: none), bits [n][nd], logical [n]
  uint8_t* bits;
  uint8_t* logical;
  Ctl* ctl;                 // events' counter and capacity, spec_misses, final_norm (null: none of them)
  int32_t* events;          // [ev_cap][5], null = not recorded
};

// Entries of a register's largest Kraus matrix: 16x16 where it has weight-4 blocks, else 4x4.
inline int dense_entries(const Program& P) {
  for (const BlockInfo& b : P.blocks)
    if (b.w == 4) return 256;
  return 16;
}
// Whether the program's blocks fit the kernels' tables (build_program's all do).
inline bool dense_fits(const Program& P) {
  for (const BlockInfo& b : P.blocks)
    if (b.op_end - b.op_begin > kDenseOps) return false;
  return true;
}

// complex64 registers of 9, 11 and 13 data qubits.
bool dense_applies(int precision, int nd);
cudaError_t setup_dense(int nd);
// Two launches: every block's Kraus pair, then the trajectories, one CTA each.
cudaError_t launch_dense_runs(const DenseArgs& a, int num_sms, cudaStream_t s);

}  // namespace qec
