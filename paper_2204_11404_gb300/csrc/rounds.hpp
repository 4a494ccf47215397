// Launch interface of the factored passes over registers in HBM (rounds.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "factor.hpp"
#include "kernels.hpp"

namespace qec {

constexpr int kMaxChain = 4;    // blocks of one pass

// One pass over the register: consecutive blocks b0 .. b0 + nb - 1, whose data qubits and the lowest
// register bits make the tile.  Tile index bits: [0, lb) = register bits [0, lb), the rest hbits; obits:
// the register bits outside the tile.  bits[i]: the four tile bits of block i's groups of 16 amplitudes,
// ascending (a weight-2 block's two qubits and two spectators); qubit[i][j]: which of the block's
// qubits bits[i][j] is, 4 for a spectator.  swz: the shared-memory slot of tile index e is e with three
// of its low bits XORed by the parities of e & swz[.] (chosen per pass so that the groups of its blocks
// spread over the banks).
struct ChainDesc {
  int32_t b0, nb, lb, nh, nout;
  uint16_t swz[4];
  uint8_t hbits[16], obits[24];
  uint8_t w[kMaxChain];
  uint8_t bits[kMaxChain][4], qubit[kMaxChain][4];
};

constexpr int kChainTileBits = 11;   // 2048 amplitudes, 16 on each of 128 threads; runs of at least 8

// Splits a round's blocks into passes: as many consecutive blocks as one tile holds, at most `most`.
std::vector<ChainDesc> plan_chains(const FactorProgram& F, int precision, int most);

// What the passes of one simulator work on.  T trajectories run side by side (groups of G CTAs each).
struct RoundArgs {
  FactorView F;
  uint64_t thr[PR_COUNT];
  double fm[FM_COUNT][4][2];
  unsigned long long seed, first;   // trajectory of group 0
  int groups, G, D, rounds;
  const ChainDesc* chains;
  int nc;
  const void* psi0;                 // [2^D]
  void* buf[2];                     // [groups][2^D]; chain c of round r reads buf[p ^ 1], writes buf[p], p = parity of (r - 1) nc + c
  void* blocks;                     // [groups][rounds][nstab] compiled blocks
  unsigned char* scratch;           // [groups][rounds] compile scratch, compile_scratch_bytes each
  uint32_t* masks;                  // [groups][rounds]
  double* norm;                     // [groups]: |psi|^2 of the state in the buffer
  double* partials;                 // [2][groups G][kMaxChain]
  unsigned int* bar;                // [groups][2]: arrivals, departures (both 0 between launches)
  uint8_t* syn;                     // [groups][(rounds + 1) nstab]
  Ctl* ctl;
  int32_t* events;
};

size_t compile_scratch_bytes(const FactorProgram& F);   // for a program with every noise site
size_t compiled_block_bytes(int precision);
cudaError_t setup_rounds(int precision);
// CTAs that a pass over 2^D amplitudes uses, and that are resident at once on the GPU.
int round_ctas(int D);
int round_wave(int precision, int num_sms);
// Compiles every round's blocks (two launches), then runs rounds [r0, r1] (1-based) of every group in
// one cooperative launch.
cudaError_t launch_compile(int precision, const RoundArgs& a, cudaStream_t s);
cudaError_t launch_rounds(int precision, const RoundArgs& a, int r0, int r1, cudaStream_t s);

}  // namespace qec
