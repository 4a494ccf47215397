// Compile of a round's stabilizer blocks into factored form (see factor.hpp), for one trajectory:
// draws, one-qubit matrices, diagonals and their merging into rotations and diagonals.  Host and
// device run the same stage functions; a group of threads runs each stage over its index range with
// a barrier between stages.
//
// Register state.  Between blocks the stored register phi and the data state psi differ by bit flips
// only: psi(x) = phi(x ^ F).  A touch's merged unitary (A of the qubit's previous touch, then this
// block's B) is written G = X^f M X^f' with f' the qubit's flip before and f after, f chosen so that
// |M_00| >= |M_10|.  Then M = diag(u_0, u_1) [[1, -t*], [t, 1]] (the cosine inside u): the pass
// applies o_0 = x - t* y, o_1 = y + t x (|t| <= 1), and u goes into this block's diagonal, whose index
// is read flipped.  A qubit's later touches in a round use a real t: M = diag(u) [[1, -t], [t, 1]]
// diag(1, w), with w in the diagonal of the previous touch's block.  After its last touch in the
// round what remains on a qubit is a phase per value and a flip: both go into that block's diagonal
// and F.  So the diagonal of block b for outcome m, as the passes use it, is
//   D_m(z ^ f) prod_j lu_j(z_j) rw_j(z_j),  lu from the block's own touches, rw from the next ones.
// FactorView::early: the rotations between a qubit's last X and first Z stabilizer of a round run in the
// X stabilizer's pass, after its diagonal (their cosines then belong to that diagonal).  No later touch
// of a Z stabilizer rotates (between them a qubit meets diagonal matrices and Paulis only), so the Z
// part of a round is diagonal.
#pragma once
#include <math.h>
#include <string.h>

#include "common.cuh"
#include "factor.hpp"

namespace qec {
namespace fac {

struct M2 { double2 a[4]; };   // 2x2 complex, row-major

QEC_HD double2 c2(double x, double y) { double2 r; r.x = x; r.y = y; return r; }
QEC_HD double2 cmul(double2 a, double2 b) { return c2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
QEC_HD double2 cmulc(double2 a, double2 b) { return c2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y); }   // a b*
// a b + c d
QEC_HD double2 cmul2(double2 a, double2 b, double2 c, double2 d) {
  return c2(fma(-c.y, d.y, fma(c.x, d.x, fma(-a.y, b.y, a.x * b.x))), fma(c.y, d.x, fma(c.x, d.y, fma(a.y, b.x, a.x * b.y))));
}
// a b* + c d*
QEC_HD double2 cmulc2(double2 a, double2 b, double2 c, double2 d) { return cmul2(a, c2(b.x, -b.y), c, c2(d.x, -d.y)); }
QEC_HD double cnorm(double2 a) { return a.x * a.x + a.y * a.y; }
QEC_HD double rsqrt_d(double x) {
#if defined(__CUDA_ARCH__)
  return rsqrt(x);
#else
  return 1.0 / sqrt(x);
#endif
}

QEC_HD M2 mul(const M2& p, const M2& q) {
  M2 r;
  r.a[0] = cmul2(p.a[0], q.a[0], p.a[1], q.a[2]);
  r.a[1] = cmul2(p.a[0], q.a[1], p.a[1], q.a[3]);
  r.a[2] = cmul2(p.a[2], q.a[0], p.a[3], q.a[2]);
  r.a[3] = cmul2(p.a[2], q.a[1], p.a[3], q.a[3]);
  return r;
}

QEC_HD double2 times_i(double2 v, bool minus) { return minus ? c2(v.y, -v.x) : c2(-v.y, v.x); }
QEC_HD double2 neg(double2 v) { return c2(-v.x, -v.y); }

// (x, y) <- Pauli (1 X, 2 Y, 3 Z) times the column (x, y).
QEC_HD void pauli_rows(int code, double2& x, double2& y) {
  if (code == 1) {
    const double2 t = x;
    x = y;
    y = t;
  } else if (code == 2) {
    const double2 t = x;
    x = times_i(y, true);
    y = times_i(t, false);
  } else if (code == 3) {
    y = neg(y);
  }
}
QEC_HD void pauli_left(int code, M2& m) {
  pauli_rows(code, m.a[0], m.a[2]);
  pauli_rows(code, m.a[1], m.a[3]);
}

// Comparison of doubles >= 0 on their bits: FP64 comparisons go through the FP64 pipe (64 cycles per
// warp and scheduler on this chip), integer ones do not.
QEC_HD uint64_t bits_of(double x) {
#if defined(__CUDA_ARCH__)
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  memcpy(&u, &x, 8);
  return u;
#endif
}
QEC_HD double signed_by(double x, int minus) {   // minus ? -x : x
  const uint64_t u = bits_of(x) ^ ((uint64_t)minus << 63);
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)u);
#else
  double r;
  memcpy(&r, &u, 8);
  return r;
#endif
}
QEC_HD bool below(double a, double b) { return bits_of(a) < bits_of(b); }
QEC_HD bool is_zero(double x) { return (bits_of(x) << 1) == 0; }

// The draw of a site (noise_code, or 1 for a twirled term that fires).  thr[pidx] = draw_threshold of
// its probability: uniform53(w) < p exactly where w >> 11 < thr, without FP64 work.
QEC_HD int draw_site(const FSite& s, const uint64_t* thr, uint64_t seed, uint64_t traj, uint64_t rnd) {
  const bool twirl = s.kind == OP_T1 || s.kind == OP_T2;
  const uint64_t t = thr[s.pidx];
  if (t == 0) return 0;
  const U64x4 w = draw(seed, traj, rnd, s.step, s.site, twirl ? TAG_TWIRL : TAG_NOISE);
  if ((w.v[0] >> 11) >= t) return 0;
  if (twirl) return 1;
  return (int)(((w.v[1] >> 32) * (s.kind == OP_N1 ? 3ull : 15ull)) >> 32) + 1;
}
// ceil(p 2^53): (double)k 2^-53 < p exactly where the integer k is below it (p in [0, 1]).
QEC_HD uint64_t draw_threshold(double p) { return p <= 0.0 ? 0ull : (uint64_t)ceil(p * 9007199254740992.0); }

// The Pauli an item puts on its qubit (0 none); anc: the item is on the ancilla's list.
QEC_HD int item_pauli(const FItem& it, const uint8_t* code, bool anc) {
  if (it.kind == FI_N1) return code[it.site];
  if (it.kind == FI_T) return code[it.site] ? it.arg : 0;
  if (it.kind == FI_N2) return anc ? code[it.site] >> 2 : code[it.site] & 3;
  return 0;
}

// What the merge of a round's touches works on, one entry per touch (index 4 b + j).
struct Touch {
  M2 g;          // stage 1: B; stage 2: G
  M2 post;       // A
  int flip;         // X stabilizer: the ancilla is flipped before the gate (G_1 meets its |0>)
  double2 ph[2];    // stage 3: lu, then lu rw
  double2 rw[2];
};

// Stage 1: B and A of touch t (and its flip for an X stabilizer).
QEC_HD void touch_factors(const FactorView& F, int t, const uint8_t* code, const double2 (*fm)[4], Touch& out) {
  const FBlock& b = F.blocks[t >> 2];
  const FTouch& tc = F.touches[t];
  out.rw[0] = out.rw[1] = c2(1.0, 0.0);
  M2 P;
  P.a[0] = P.a[3] = c2(1.0, 0.0);
  P.a[1] = P.a[2] = c2(0.0, 0.0);
  int i = tc.begin;
  for (; i < tc.end; ++i) {
    const FItem it = F.items[i];
    if (it.kind == FI_GATE) break;
    if (it.kind == FI_MAT) {
      M2 g;
      for (int k = 0; k < 4; ++k) g.a[k] = fm[it.arg][k];
      P = mul(g, P);
    } else {
      pauli_left(item_pauli(it, code, false), P);
    }
  }
  if (b.z_type) {
    out.g = P;
    M2 L;
    L.a[0] = L.a[3] = c2(1.0, 0.0);
    L.a[1] = L.a[2] = c2(0.0, 0.0);
    for (++i; i < tc.end; ++i) {
      const FItem it = F.items[i];
      if (it.kind == FI_MAT) {
        M2 g;
        for (int k = 0; k < 4; ++k) g.a[k] = fm[it.arg][k];
        L = mul(g, L);
      } else {
        pauli_left(item_pauli(it, code, false), L);
      }
    }
    out.post = L;
    return;
  }
  // X stabilizer: the ancilla's flips before this gate select which block each branch meets
  int flip = 0;
  for (int k = b.anc_begin; k < b.anc_end; ++k) {
    const FItem it = F.items[k];
    if (it.kind == FI_GATE && it.arg == (t & 3)) break;
    const int p = item_pauli(it, code, true);
    flip ^= (p == 1 || p == 2);
  }
  out.flip = flip;
  M2 S, A;
  for (int k = 0; k < 4; ++k) {
    S.a[k] = fm[FM_SH][k];
    A.a[k] = fm[flip ? FM_A1 : FM_A0][k];
  }
  out.g = mul(S, P);
  for (++i; i < tc.end; ++i) pauli_left(item_pauli(F.items[i], code, false), A);   // after an X gate: Paulis only
  out.post = A;
}

// Stage 2: G of touch t = B A_prev, and whether it swaps (its larger column-0 entry is G_10).  Reads
// the touches' post, writes g of touch t only.
QEC_HD int touch_merge(const FactorView& F, int t, Touch* T) {
  const int pv = F.touches[t].prev;
  if (pv >= 0) T[t].g = mul(T[t].g, T[pv].post);
  return below(cnorm(T[t].g.a[0]), cnorm(T[t].g.a[2])) ? 1 : 0;
}

// The flip left on touch t's qubit at the round's end (its last touch): whether A swaps (it is a Pauli
// times diagonal matrices: its zeros are exact).
QEC_HD int touch_end_swap(const Touch& T) { return is_zero(T.post.a[0].x) && is_zero(T.post.a[0].y) ? 1 : 0; }

// Whether touch t's rotation runs in the block of the qubit's previous touch.
QEC_HD bool runs_early(const FactorView& F, int t) {
  const int pv = F.touches[t].prev;
  return F.early && pv >= 0 && F.blocks[t >> 2].z_type && !F.blocks[pv >> 2].z_type;
}

// Stage 3: rotation of touch t from G, the flips f' before and f after it; lu and the previous
// touch's rw (or, at a round's last touch, its own rw from what remains on the qubit).
QEC_HD double2 touch_rotation(const FactorView& F, int t, Touch* T, int f_before, int f_after) {
  double2 (&lu)[2] = T[t].ph;
  M2 m = T[t].g;
  if (f_before) {   // columns
    double2 x = m.a[0]; m.a[0] = m.a[1]; m.a[1] = x;
    x = m.a[2]; m.a[2] = m.a[3]; m.a[3] = x;
  }
  if (f_after) {    // rows
    double2 x = m.a[0]; m.a[0] = m.a[2]; m.a[2] = x;
    x = m.a[1]; m.a[1] = m.a[3]; m.a[3] = x;
  }
  const int pv = F.touches[t].prev;
  if (F.touches[t].next < 0) {
    const int r = touch_end_swap(T[t]);
    for (int z = 0; z < 2; ++z) {
      const int c = z ^ f_after;
      T[t].rw[z] = T[t].post.a[2 * (c ^ r) + c];
    }
  }
  const double n00 = cnorm(m.a[0]), n10 = cnorm(m.a[2]);
  lu[0] = m.a[0];
  double2 tt = c2(0.0, 0.0);
  if (below(n10, 1e-33)) {              // |t| below the last place: no rotation
    lu[1] = pv < 0 ? m.a[3] : c2(1.0, 0.0);
    if (pv >= 0) T[pv].rw[1] = m.a[3];
    return tt;
  }
  if (pv < 0) {                   // the round's first touch: a complex t
    lu[1] = m.a[3];
    const double k = 1.0 / cnorm(m.a[3]);
    tt = cmulc(m.a[2], m.a[3]);
    tt.x *= k;
    tt.y *= k;
    if (below(fabs(tt.y), 1e-17)) tt.y = 0.0;
    if (below(fabs(tt.x), 1e-17)) tt.x = 0.0;
    return tt;
  }
  const double k = rsqrt_d(n00 * n10);
  tt.x = n10 * k;
  const double2 w = cmulc(m.a[3], m.a[2]);
  if (runs_early(F, t)) {         // lu = u, the cosine in rw
    const double c0 = rsqrt_d(n00), s0 = n00 * k * c0, c = n00 * c0;
    lu[0] = c2(m.a[0].x * c0, m.a[0].y * c0);
    lu[1] = c2(m.a[2].x * s0, m.a[2].y * s0);
    T[pv].rw[0] = c2(c, 0.0);
    T[pv].rw[1] = c2(w.x * (k * c), w.y * (k * c));
    return tt;
  }
  lu[1] = c2(m.a[2].x * (n00 * k), m.a[2].y * (n00 * k));
  T[pv].rw[1] = c2(w.x * k, w.y * k);
  return tt;
}

// Stage 4: the diagonal of block b at index z (flips f, one bit per data qubit) for both outcomes.
QEC_HD void block_diagonal(const FactorView& F, int b, int z, int f, const uint8_t* code, const double2 (*fm)[4],
                           const Touch* T, double2& d0, double2& d1) {
  const FBlock& B = F.blocks[b];
  const int zl = z ^ f;
  double2 v0, v1;
  if (B.z_type) {
    v0 = c2(1.0, 0.0);
    v1 = c2(0.0, 0.0);
    for (int k = B.anc_begin; k < B.anc_end; ++k) {
      const FItem it = F.items[k];
      if (it.kind == FI_GATE) {
        const double2* g = fm[FM_G0 + ((zl >> it.arg) & 1)];
        const double2 x = v0, y = v1;
        v0 = cmul2(g[0], x, g[1], y);
        v1 = cmul2(g[2], x, g[3], y);
      } else {
        pauli_rows(item_pauli(it, code, true), v0, v1);
      }
    }
  } else {
    double2 l = c2(1.0, 0.0);
    for (int j = 0; j < B.w; ++j) {
      const double2 lm = fm[FM_LAM][3 * ((zl >> j) & 1)];
      l = cmul(l, c2(lm.x, signed_by(lm.y, T[4 * b + j].flip)));
    }
    v0 = c2(1.0, 0.0);
    v1 = c2(0.0, 0.0);
    // the branch that leaves the preparation with the ancilla in |1> carries l
    for (int k = B.anc_begin; k < B.anc_end; ++k) {
      const FItem it = F.items[k];
      if (it.kind == FI_MAT) {
        const double2* g = fm[it.arg];
        const double2 x = v0, y = v1;
        v0 = cmul2(g[0], x, g[1], y);
        v1 = cmul2(g[2], x, g[3], y);
        if (it.arg == FM_PREP) v1 = cmul(v1, l);
      } else if (it.kind != FI_GATE) {
        pauli_rows(item_pauli(it, code, true), v0, v1);
      }
    }
  }
  double2 e = T[4 * b].ph[z & 1];
  for (int j = 1; j < B.w; ++j) e = cmul(e, T[4 * b + j].ph[(z >> j) & 1]);
  d0 = cmul(v0, e);
  d1 = cmul(v1, e);
}

// Working memory of the rounds compiled together (nr of them, each 4 nstab touches and nsites draws).
struct Rounds {
  int nr;
  uint8_t* code;          // [nr][nsites]
  Touch* T;               // [nr][4 nstab]
  uint8_t* swap;          // [nr][4 nstab]: bit 0 the touch swaps, bits 1, 2 its flips before and after
  uint32_t* mask;         // [nr]: the qubits that the whole round flips (zeroed by the caller)
};

QEC_HD void toggle(uint32_t* w, uint32_t bits) {
#if defined(__CUDA_ARCH__)
  atomicXor(w, bits);
#else
  *w ^= bits;
#endif
}

// A thread group: rank, size, and a barrier over its threads.
struct OneThread {
  int rank = 0, size = 1;
  QEC_HD void sync() const {}
};

// Touch i of nr rounds: all X-stabilizer touches first, those of Z stabilizers from a multiple of 32 on
// (the two kinds are different code: a warp runs one of them).  -1: none.
QEC_HD int touch_count(const FactorView& F, int nr) { return (nr * F.n_x + 31) / 32 * 32 + nr * (F.n_touch - F.n_x); }
QEC_HD int touch_at(const FactorView& F, int nr, int i, int& k) {
  const int zs = (nr * F.n_x + 31) / 32 * 32;
  if (i < nr * F.n_x) {
    k = i / F.n_x;
    return F.order[i - k * F.n_x];
  }
  if (i < zs) return -1;
  i -= zs;
  const int nz = F.n_touch - F.n_x;
  k = i / nz;
  return F.order[F.n_x + i - k * nz];
}

// First half, rounds rnd .. rnd + nr - 1: draws, factors and merged unitaries, and the flips each round
// makes.  event(k, i, code) is called for every draw.
#if defined(__CUDACC__)
#pragma nv_exec_check_disable
#endif
template <class G, class E>
QEC_HD void compile_merge(const G& g, const FactorView& F, const uint64_t* thr, uint64_t seed, uint64_t traj,
                          uint64_t rnd, const double2 (*fm)[4], const Rounds& R, E event) {
  const int nt = 4 * F.nstab, all = touch_count(F, R.nr);
  for (int i = g.rank; i < R.nr * F.nsites; i += g.size) {
    const int k = i / F.nsites, s = i - k * F.nsites;
    const int c = draw_site(F.sites[s], thr, seed, traj, rnd + k);
    R.code[i] = (uint8_t)c;
    event(k, s, c);
  }
  g.sync();
  for (int i = g.rank; i < all; i += g.size) {
    int k = 0;
    const int t = touch_at(F, R.nr, i, k);
    if (t >= 0) touch_factors(F, t, R.code + k * F.nsites, fm, R.T[k * nt + t]);
  }
  g.sync();
  for (int i = g.rank; i < R.nr * F.n_touch; i += g.size) {
    const int k = i / F.n_touch, t = F.order[i - k * F.n_touch];
    Touch* T = R.T + k * nt;
    int s = touch_merge(F, t, T);
    R.swap[k * nt + t] = (uint8_t)s;
    if (F.touches[t].next < 0) s ^= touch_end_swap(T[t]);
    if (s) toggle(R.mask + k, 1u << F.blocks[t >> 2].q[t & 3]);
  }
  g.sync();
}

// Second half, given the flips in force when the first round starts: rotation(k, t, value) per touch and
// diagonal(k, b, z, D_0, D_1) per block and index.
#if defined(__CUDACC__)
#pragma nv_exec_check_disable
#endif
template <class G, class ER, class ED>
QEC_HD void compile_emit(const G& g, const FactorView& F, const double2 (*fm)[4], const Rounds& R, uint32_t flips,
                         ER rotation, ED diagonal) {
  const int nt = 4 * F.nstab;
  for (int i = g.rank; i < R.nr * F.n_touch; i += g.size) {
    const int k = i / F.n_touch, t0 = F.order[i - k * F.n_touch];
    if (F.touches[t0].prev >= 0) continue;
    uint32_t at_start = flips;
    for (int e = 0; e < k; ++e) at_start ^= R.mask[e];
    int f = (int)(at_start >> F.blocks[t0 >> 2].q[t0 & 3]) & 1;
    for (int t = t0; t >= 0; t = F.touches[t].next) {
      uint8_t& w = R.swap[k * nt + t];
      const int s = w & 1;
      w = (uint8_t)(s | (f << 1) | ((f ^ s) << 2));
      f ^= s;
    }
  }
  g.sync();
  for (int i = g.rank; i < R.nr * F.n_touch; i += g.size) {
    const int k = i / F.n_touch, t = F.order[i - k * F.n_touch];
    const int w = R.swap[k * nt + t];
    rotation(k, t, touch_rotation(F, t, R.T + k * nt, (w >> 1) & 1, (w >> 2) & 1));
  }
  g.sync();
  for (int i = g.rank; i < R.nr * F.n_touch; i += g.size) {
    const int k = i / F.n_touch;
    Touch& T = R.T[k * nt + F.order[i - k * F.n_touch]];
    T.ph[0] = cmul(T.ph[0], T.rw[0]);
    T.ph[1] = cmul(T.ph[1], T.rw[1]);
  }
  g.sync();
  for (int i = g.rank; i < 16 * R.nr * F.nstab; i += g.size) {
    const int k = i / (16 * F.nstab), b = (i >> 4) - k * F.nstab, z = i & 15;
    if (z >> F.blocks[b].w) continue;
    int f = 0;
    for (int j = 0; j < F.blocks[b].w; ++j) f |= ((R.swap[k * nt + 4 * b + j] >> 2) & 1) << j;
    double2 d0, d1;
    block_diagonal(F, b, z, f, R.code + k * F.nsites, fm, R.T + k * nt, d0, d1);
    diagonal(k, b, z, d0, d1);
  }
}

}  // namespace fac
}  // namespace qec
