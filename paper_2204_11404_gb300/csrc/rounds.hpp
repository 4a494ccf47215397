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

// Tile bits of a rotating pass: 11 (2048 amplitudes, 16 on each of 128 threads), or, on small complex128
// registers of weight-2 blocks, 9 (512, 4 on each); runs of at least 8 amplitudes either way.
constexpr int kTileBits = 11, kSmallTileBits = 9;

// Splits blocks [b0, b1) of a round into passes: as many consecutive blocks as one tile holds, at most `most`.
std::vector<ChainDesc> plan_chains(const FactorProgram& F, int precision, int tile_bits, int most, int b0, int b1);

// A pass of blocks that rotate no qubit: diagonals only.  Tile as above, but of 2^12 complex128 or 2^13
// complex64 amplitudes (8 or 16 on each of 512 threads; runs of 128 bytes).  The blocks' data qubits are nu
// tile bits ubits (ascending; rbits: the other tile bits); at[i][j]: which of them block i's qubit j is.
constexpr int kMaxDiag = 8;
constexpr int kDiagUnion = 10;      // at most this many data qubits in a pass
struct DiagDesc {
  int32_t b0, nb, lb, nh, nout, nu;
  uint8_t hbits[16], obits[24], ubits[12], rbits[12];
  uint8_t w[kMaxDiag], at[kMaxDiag][4];
};
std::vector<DiagDesc> plan_diagonals(const FactorProgram& F, int precision, int b0, int b1);

// What the passes of one simulator work on.  T trajectories run side by side (groups of G CTAs each).
struct RoundArgs {
  FactorView F;
  uint64_t thr[PR_COUNT];
  double fm[FM_COUNT][4][2];
  unsigned long long seed, first;   // trajectory of group 0
  int groups, G, D, rounds, tb;     // tb: tile bits
  const ChainDesc* chains;          // nc rotating passes, then nd diagonal ones (of a round's last blocks)
  int nc;
  const DiagDesc* diags;
  int nd;
  int steps, step0;                 // passes of a round; those before the diagonal ones
  const void* psi0;                 // [2^D]
  void* buf[2];                     // [groups][2^D]; pass p of all reads buf[p & 1 ^ 1], writes buf[p & 1], the first reads psi0
  void* blocks;                     // [groups][rounds][nstab] compiled blocks
  unsigned char* scratch;           // [groups][rounds] compile scratch, compile_scratch_bytes each
  uint32_t* masks;                  // [groups][rounds]
  double* norm;                     // [groups]: |psi|^2 of the state in the buffer
  const double* diag_in;            // the diagonal passes' own (default: norm), in and out; [rounds] strides
  double* diag_out;
  int diag_stride;
  double* partials;                 // [2][groups G][kMaxChain]; diagonal passes: [2][CTAs][kMaxDiag + 1]
  unsigned int* bar;                // [groups][2]: arrivals, departures (both 0 between launches)
  uint8_t* syn;                     // [groups][(rounds + 1) nstab]
  Ctl* ctl;
  int32_t* events;
};

size_t compile_scratch_bytes(const FactorProgram& F);   // for a program with every noise site
size_t compiled_block_bytes(int precision);
cudaError_t setup_rounds(int precision);
// CTAs of a rotating pass that are resident at once on the GPU.
int round_wave(int precision, int tile_bits, bool early, int num_sms);
// Compiles every round's blocks (two launches), then runs rounds [r0, r1] (1-based) of every group in
// one cooperative launch.
cudaError_t launch_compile(int precision, const RoundArgs& a, cudaStream_t s);
cudaError_t launch_rounds(int precision, const RoundArgs& a, int r0, int r1, cudaStream_t s);
// The diagonal passes of round r (one group), in one cooperative launch.
cudaError_t launch_diagonals(int precision, const RoundArgs& a, int r, int num_sms, cudaStream_t s);
// The dense Kraus pairs of the blocks [0, nb) of every round, rotations included, as the tensor-core
// passes read them ([rounds nstab][KRAUS_STRIDE]), and every block's uniform u.
cudaError_t launch_dense(const RoundArgs& a, int nb, void* kraus, double* u, cudaStream_t s);

}  // namespace qec
