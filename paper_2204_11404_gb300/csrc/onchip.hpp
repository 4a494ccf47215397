// Launch interface of the on-chip trajectories (onchip.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "factor.hpp"
#include "kernels.hpp"

namespace qec {

struct OnchipArgs {
  FactorView F;
  uint64_t thr[PR_COUNT];   // draw_threshold of each probability
  double fm[FM_COUNT][4][2];
  unsigned long long seed, first;
  uint32_t n;             // trajectories
  int rounds, nl;         // nl: data qubits 0..nl-1 make the raw logical parity
  const void* psi0;       // [2^D]
  void* psi_out;          // the last trajectory's final state (null: none)
  uint8_t* syn;           // [n][rounds + 1][nstab] (null: none), bits [n][nd], logical [n]
  uint8_t* bits;
  uint8_t* logical;
  Ctl* ctl;               // events' counter and capacity, spec_misses, final_norm (null: none of them)
  int32_t* events;        // [ev_cap][5], null = not recorded
};

// complex128 registers of 9 and 11 data qubits run on chip (complex64 ones of 9 to 13: dense.hpp).
bool onchip_applies(int nd);
cudaError_t setup_onchip();
cudaError_t launch_onchip(const OnchipArgs& a, int num_sms, cudaStream_t s);

}  // namespace qec
