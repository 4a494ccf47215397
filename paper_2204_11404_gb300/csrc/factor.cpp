// Builds the factored program (see factor.hpp) from the block program.
#include "factor.hpp"

#include "gate_eigen.hpp"


namespace qec {

bool build_factor(const Program& P, FactorProgram& F, std::string& err) {
  F = FactorProgram();
  F.nd = P.nd;
  F.nstab = P.nstab;
  F.touches.assign(4 * (size_t)P.nstab, FTouch{0, 0, -1, -1});
  std::vector<int> last(P.nd, -1);   // latest touch of each data qubit
  for (int b = 0; b < P.nstab; ++b) {
    const BlockInfo& bi = P.blocks[b];
    FBlock fb{};
    fb.w = (uint8_t)bi.w;
    fb.offset = (uint8_t)bi.offset;
    for (int j = 0; j < 4; ++j) fb.q[j] = (uint8_t)(j < bi.w ? bi.q[j] : 0);
    std::vector<FItem> data[4], anc;
    int gates[4] = {0, 0, 0, 0}, z_type = -1;
    // an op run of one correction or gate: its unitaries merge into one matrix, its Pauli sites follow
    // (a run's unitaries are identities wherever its twirled sites can fire, or commute with them)
    struct { int qubit = -1, count = 0, base = -1; } run;
    auto list = [&](int lq) -> std::vector<FItem>& { return lq == bi.w ? anc : data[lq]; };
    auto flush = [&]() { run.qubit = -1; run.count = 0; run.base = -1; };
    for (int oi = bi.op_begin; oi < bi.op_end; ++oi) {
      const ProgOp& op = P.ops[oi];
      const bool draws = op.kind != OP_U1 && op.kind != OP_U2;
      uint16_t site = 0;
      if (draws) {
        site = (uint16_t)F.sites.size();
        F.sites.push_back({op.kind, op.pidx, op.step, op.site});
      }
      const uint8_t pauli = op.mat == M_X ? 1 : op.mat == M_Z ? 3 : 0;
      if (op.kind == OP_U1) {
        std::vector<FItem>& L = list(op.q0);
        // over-rotations and the second round term belong to the matrix of the op before them
        if (op.mat == M_ROT_RX || op.mat == M_ROT_RXP || op.mat == M_ROT_RZ) continue;
        if (op.q0 == bi.w) {
          if (op.mat != M_H && op.mat != M_RX90 && op.mat != M_RX90DG) { err = "unexpected ancilla op"; return false; }
          flush();
          bool before = true;
          for (const FItem& i : anc) before = before && i.kind != FI_GATE;
          L.push_back({FI_MAT, (uint8_t)(before ? FM_PREP : FM_POST), 0});
        } else if (op.mat == M_ROUND_RZ || op.mat == M_ROUND_RX) {
          if (run.qubit == op.q0 && run.base == FM_ROUND) continue;
          run.qubit = op.q0;
          run.base = FM_ROUND;
          L.push_back({FI_MAT, FM_ROUND, 0});
        } else if (op.mat == M_RX90 || op.mat == M_RZ90) {
          const int base = op.mat == M_RX90 ? FM_RX1 : FM_RZ1;
          if (run.qubit == op.q0 && run.base == base) {   // the second factor of one correction
            if (++run.count > 2) { err = "correction of more than two factors"; return false; }
            for (size_t i = L.size(); i-- > 0;)
              if (L[i].kind == FI_MAT) { L[i].arg = (uint8_t)(base + 1); break; }
          } else {
            run.qubit = op.q0;
            run.base = base;
            run.count = 1;
            L.push_back({FI_MAT, (uint8_t)base, 0});
          }
        } else {
          err = "unexpected data op";
          return false;
        }
        continue;
      }
      if (op.kind == OP_U2) {
        const bool gate = op.mat == M_CNOT || op.mat == M_RZX90;
        if (!gate) continue;   // ROT_RZX, ZZ: part of the gate's matrix
        flush();
        const int first_data = op.q0 != bi.w;
        if (z_type >= 0 && z_type != first_data) { err = "mixed control sides"; return false; }
        z_type = first_data;
        const int lq = first_data ? op.q0 : op.q1;
        if (gates[lq]++) { err = "two gates on one data qubit in a block"; return false; }
        data[lq].push_back({FI_GATE, 0, 0});
        anc.push_back({FI_GATE, (uint8_t)lq, 0});
        continue;
      }
      if (op.kind == OP_N1) {
        flush();
        list(op.q0).push_back({FI_N1, 0, site});
      } else if (op.kind == OP_T1) {
        if (!pauli) { err = "unexpected twirl Pauli"; return false; }
        if (op.q0 == bi.w) flush();
        list(op.q0).push_back({FI_T, pauli, site});   // a correction's run goes on
      } else if (op.kind == OP_N2) {
        flush();
        anc.push_back({FI_N2, 0, site});
        list(op.q1).push_back({FI_N2, 0, site});
      } else {   // OP_T2: Z on the first-listed qubit, X or Z on the second
        flush();
        list(op.q0).push_back({FI_T, 3, site});
        list(op.q1).push_back({FI_T, (uint8_t)(op.mat == M_PZX ? 1 : 3), site});
      }
    }
    if (z_type < 0) { err = "block without a gate"; return false; }
    fb.z_type = (uint8_t)z_type;
    for (int j = 0; j < bi.w; ++j) {
      if (gates[j] != 1) { err = "data qubit without a gate"; return false; }
      FTouch& t = F.touches[4 * b + j];
      t.begin = (uint16_t)F.items.size();
      F.items.insert(F.items.end(), data[j].begin(), data[j].end());
      t.end = (uint16_t)F.items.size();
      t.prev = (int16_t)last[bi.q[j]];
      if (t.prev >= 0) F.touches[t.prev].next = (int16_t)(4 * b + j);
      last[bi.q[j]] = 4 * b + j;
    }
    fb.anc_begin = (uint16_t)F.items.size();
    F.items.insert(F.items.end(), anc.begin(), anc.end());
    fb.anc_end = (uint16_t)F.items.size();
    F.blocks.push_back(fb);
  }
  // the last touch of a round leaves diagonal matrices and Paulis only, so that the round's end needs
  // no rotation (a bit flip of the register's index and phases instead)
  for (int q = 0; q < P.nd; ++q) {
    if (last[q] < 0) { err = "data qubit without a stabilizer"; return false; }
    const FTouch& t = F.touches[last[q]];
    bool after = false;
    for (int i = t.begin; i < t.end; ++i) {
      if (F.items[i].kind == FI_GATE) after = true;
      else if (after && F.items[i].kind == FI_MAT && F.items[i].arg != FM_RZ1 && F.items[i].arg != FM_RZ2) {
        err = "a rotation after the round's last gate";
        return false;
      }
    }
    if (!F.blocks[last[q] / 4].z_type) { err = "a data qubit's last gate belongs to an X stabilizer"; return false; }
  }
  for (int x = 1; x >= 0; --x)
    for (int b = 0; b < P.nstab; ++b)
      for (int j = 0; j < F.blocks[b].w; ++j)
        if (F.blocks[b].z_type == 1 - x) F.order.push_back((uint16_t)(4 * b + j));
  for (uint16_t t : F.order) F.n_x += !F.blocks[t / 4].z_type;
  if (F.items.size() > 65535 || F.sites.size() > 65535) { err = "program too large"; return false; }
  return true;
}

namespace {

// Products in extended precision, rounded once: a gate's matrix is in every block, so its rounding error
// adds up along a trajectory (state error after 48 blocks 5.3e-15 with FP64 products, 2.0e-15 so).
struct M2h { long double m[4][2]; };

M2h top2(const double m[16][2]) {
  M2h r;
  const int at[4] = {0, 1, 4, 5};
  for (int i = 0; i < 4; ++i) for (int c = 0; c < 2; ++c) r.m[i][c] = m[at[i]][c];
  return r;
}

M2h block_of(const double m[16][2], int c) {   // rows and columns 2c, 2c + 1 of a 4x4
  M2h r;
  for (int i = 0; i < 4; ++i)
    for (int k = 0; k < 2; ++k) r.m[i][k] = m[(2 * c + (i >> 1)) * 4 + 2 * c + (i & 1)][k];
  return r;
}

M2h mul(const M2h& a, const M2h& b) {
  M2h r;
  for (int i = 0; i < 2; ++i)
    for (int j = 0; j < 2; ++j) {
      long double re = 0, im = 0;
      for (int k = 0; k < 2; ++k) {
        const long double* x = a.m[2 * i + k];
        const long double* y = b.m[2 * k + j];
        re += x[0] * y[0] - x[1] * y[1];
        im += x[0] * y[1] + x[1] * y[0];
      }
      r.m[2 * i + j][0] = re;
      r.m[2 * i + j][1] = im;
    }
  return r;
}

}  // namespace

void factor_mats(const double (*mats)[16][2], bool cr, bool twirl, double (*out)[4][2]) {
  M2h f[FM_COUNT];
  double one[16][2] = {};
  for (int i = 0; i < 4; ++i) one[5 * i][0] = 1.0;
  double one1[16][2] = {};   // the 2x2 identity in the top-left corner
  one1[0][0] = one1[5][0] = 1.0;
  // twirled terms are Paulis: their unitaries are not part of the program
  auto c1 = [&](int id) { return top2(twirl ? one1 : mats[id]); };
  auto c2 = [&](int id, int c) { return block_of(twirl ? one : mats[id], c); };
  f[FM_ROUND] = mul(c1(M_ROUND_RX), c1(M_ROUND_RZ));
  f[FM_RX1] = mul(c1(M_ROT_RX), top2(mats[M_RX90]));
  f[FM_RX2] = mul(f[FM_RX1], f[FM_RX1]);
  f[FM_RZ1] = mul(c1(M_ROT_RZ), top2(mats[M_RZ90]));
  f[FM_RZ2] = mul(f[FM_RZ1], f[FM_RZ1]);
  f[FM_PREP] = cr ? mul(c1(M_ROT_RXP), top2(mats[M_RX90DG])) : top2(mats[M_H]);
  f[FM_POST] = cr ? f[FM_RX1] : top2(mats[M_H]);
  for (int c = 0; c < 2; ++c) {
    const M2h zz = c2(M_ZZ, c);
    f[FM_G0 + c] = cr ? mul(zz, mul(c2(M_ROT_RZX, c), block_of(mats[M_RZX90], c)))
                      : mul(zz, block_of(mats[M_CNOT], c));
  }
  struct C { long double x, y; };
  C g[2][4], r[4][4];
  for (int i = 0; i < 4; ++i)
    for (int c = 0; c < 2; ++c) g[c][i] = {f[FM_G0 + c].m[i][0], f[FM_G0 + c].m[i][1]};
  gate_eigen<C, long double>(g[0], g[1], r[0], r[1], r[2], r[3]);
  for (int j = 0; j < 4; ++j)   // FM_SH, FM_A0, FM_A1, FM_LAM
    for (int i = 0; i < 4; ++i) {
      f[FM_SH + j].m[i][0] = r[j][i].x;
      f[FM_SH + j].m[i][1] = r[j][i].y;
    }
  for (int i = 0; i < FM_COUNT; ++i)
    for (int k = 0; k < 4; ++k)
      for (int c = 0; c < 2; ++c) out[i][k][c] = (double)f[i].m[k][c];
}

}  // namespace qec
