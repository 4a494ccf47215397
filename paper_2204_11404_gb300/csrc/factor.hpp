// Factored form of the circuit program's stabilizer blocks (host-built, read by every engine that
// compiles blocks on the device).
//
// A stabilizer circuit (Sec. II.A, Fig. 1b/c) couples its ancilla to each data qubit once, by a gate
// that is block-diagonal in its control: the ancilla's Z value in an X stabilizer, the data qubit's
// Z value in a Z stabilizer.  Everything else in a block acts on one qubit.  So the block's Kraus
// pair K_m = <m|U|0> is, exactly, K_m = (x)_j A_j . D_m . (x)_j B_j: one-qubit matrices B_j before and A_j
// after a diagonal D_m over the block's data qubits, the outcome m in D_m alone.
//   Z stabilizer: B_j / A_j are qubit j's ops before / after its gate, and D_m(z) = <m| ancilla ops and
//     the gates' blocks W_{z_j} in time order |0>.
//   X stabilizer: the ancilla's Z value selects one of two branches (Paulis on it only swap them), so
//     K_m = sum_a Q_ma (x)_j V_j^(a), V_j^(a) = L_j G_a P_j with the qubit's ops before and after its gate; with
//     G_0+ G_1 = S Lambda S+ (the same for every gate), B_j = S+ P_j, A_j = L_j G_0 S, D_m(z) = Q_m0 + Q_m1 prod_j
//     lambda(z_j); a flip of the ancilla before the gate exchanges G_0 and G_1, so lambda is conjugate.
// Consecutive blocks' A and B on a qubit merge into one 2x2 unitary, itself a diagonal times a real
// rotation times a diagonal; the diagonals go into the neighbouring D's (factor.cuh).  A dense 16x16
// block costs 64 real multiply-adds per amplitude; its factored form 2 per qubit (a real rotation)
// and 4 for the diagonal.
#pragma once
#include <cstdint>
#include <string>
#include <vector>

#include "program.hpp"

namespace qec {

// One draw of a round: op kind, probability, step and site as in ProgOp (its result is a byte:
// noise_code for OP_N1 / OP_N2, 1 for a twirled term that fires).
struct FSite {
  uint8_t kind, pidx;
  uint16_t step;
  uint32_t site;
};

// Items of a data qubit's list in its block, or of the block's ancilla list, in time order.
enum FKind : uint8_t {
  FI_MAT = 0,    // one-qubit matrix arg (FMatId)
  FI_N1 = 1,     // the Pauli that site drew (OP_N1)
  FI_T = 2,      // Pauli arg if site fired (OP_T1, or one qubit's factor of OP_T2)
  FI_N2 = 3,     // this qubit's Pauli of site's pair (OP_N2): ancilla code >> 2, data code & 3
  FI_GATE = 4    // the two-qubit gate with its coherent terms; in the ancilla list arg = data qubit j
};
struct FItem {
  uint8_t kind, arg;
  uint16_t site;
};

// Matrices of the factored program (2x2, row-major): the round-start terms, the data corrections
// with their over-rotations, the ancilla's preparation and final rotation, the two blocks G_0, G_1 of the
// gate with its coherent terms (control 0, control 1), and what an X stabilizer makes of them: with
// G_0+ G_1 = S Lambda S+, S+ (FM_SH), G_0 S and G_1 S (FM_A0, FM_A1) and Lambda (FM_LAM).
enum FMatId : uint8_t {
  FM_ROUND = 0, FM_RX1, FM_RX2, FM_RZ1, FM_RZ2, FM_PREP, FM_POST, FM_G0, FM_G1, FM_SH, FM_A0, FM_A1, FM_LAM, FM_COUNT
};

// A touch: data qubit j of block b, index 4 b + j.
struct FTouch {
  uint16_t begin, end;        // items
  int16_t prev, next;         // the same qubit's neighbouring touches in the round, -1 at its ends
};

struct FBlock {
  uint8_t w, z_type, offset, pad;
  uint8_t q[4];               // data bits, ascending
  uint16_t anc_begin, anc_end;
};

struct FactorProgram {
  int nd = 0, nstab = 0;
  std::vector<uint16_t> order;   // the used touches, those of X stabilizers first
  int n_x = 0;                   // how many those are
  std::vector<FSite> sites;
  std::vector<FItem> items;
  std::vector<FTouch> touches;   // 4 nstab, unused ones empty
  std::vector<FBlock> blocks;
};

// The same program as plain arrays (device or host pointers).
struct FactorView {
  const FSite* sites;
  const FItem* items;
  const FTouch* touches;
  const FBlock* blocks;
  const uint16_t* order;
  int nsites, nstab, nd, n_touch, n_x;
  int early = 0;   // see factor.cuh
};

inline FactorView view_of(const FactorProgram& F) {
  return {F.sites.data(), F.items.data(), F.touches.data(), F.blocks.data(), F.order.data(),
          (int)F.sites.size(), F.nstab, F.nd, (int)F.order.size(), F.n_x};
}

// Builds the factored program of P (any gate set, code and noise options, all_slots included).  False,
// with a message, if a block has ops outside the form above (none of build_program's does).
bool build_factor(const Program& P, FactorProgram& F, std::string& err);

// The FM_COUNT matrices from the program's matrix table: mats[id][16][2] as in Program, out [id][4][2].
// twirl: the coherent terms are drawn as Paulis, so their unitaries are left out.
void factor_mats(const double (*mats)[16][2], bool cr, bool twirl, double (*out)[4][2]);

}  // namespace qec
