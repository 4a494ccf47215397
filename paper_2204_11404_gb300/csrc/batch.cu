// Batched form: many small-register trajectories at once, one launch per engine.
//
// A trajectory of the d = 3 code runs on chip, its blocks in factored form (factor.hpp).  Reduced
// register (9 data qubits + the reused ancilla, Sec. II.B): one warp per trajectory, 512 amplitudes
// (onchip.cuh).  Unreduced register (all 17 qubits): one CTA per trajectory.  A part's four ancillas
// are active together; the other part's are |0> throughout (reset after their measurement, untouched
// before their part), so a slab of 2^13 amplitudes holds the exact state.  Warps and CTAs take
// trajectories from device work counters, so precisions and noise parameters mix freely in one
// run.  The circuit program is built once with every noise and coherent slot present; a
// trajectory's own matrices and draw thresholds follow from its noise input (a zero angle is the
// identity, a zero probability never fires).
//
// complex64 trajectories of both registers have engines of their own, in dense blocks and gate units
// (batch_dense.cu); each engine is a launch of its own, side by side.
//
// The FP64 pipe bounds the complex128 trajectories.  2048 trajectories of 3 rounds, dense blocks and gate
// units before: reduced register 8.24 -> 1.43 ms, unreduced 33.3 -> 3.58.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include "../../include/qecsv.h"
#include "batch_dense.hpp"
#include "gate_eigen.hpp"
#include "onchip.cuh"
#include "kernels.hpp"
#include "program.hpp"

using namespace qec;

namespace {

constexpr int kD = 3;                    // register of the batched form: d = 3
constexpr int kND = kD * kD;             // 9 data qubits
constexpr int kNAmp = 1 << kND;          // 512 amplitudes
constexpr int kNStab = kND - 1;          // 8 stabilizers
constexpr int kNAnc = kNStab / 2;        // ancillas of one part
constexpr int kTouches = 4 * kNStab;
constexpr int kSites = 224;              // draws of a round, every slot present (checked at creation)
constexpr int kKinds = 4;                // precision + 2 for the unreduced register

struct BatchCtl {
  uint64_t seed;
  uint32_t n[kKinds];             // trajectories of each kind in this run
  unsigned int counter[kKinds];   // their work queue heads (zeroed before every run)
  uint32_t snap_item;             // item whose final data-register state goes to snap (~0u = none)
};

struct BatchArgs {
  FactorView F;               // noisy program (all slots present), or the init program
  const qec_noise* noise;     // [n]
  const uint32_t* idx;        // reduced-register complex128 items of this run
  const uint32_t* idx_u;      // unreduced-register ones
  const uint64_t* traj;       // [n]
  BatchCtl* ctl;
  int rounds, cr;
  int width;                  // unreduced register: slab bits a sweep may hold (see u_sweep)
  const double2* psi0;        // init code state
  uint8_t* syn;               // [n][rounds+1][8]
  uint8_t* bits;              // [n][9]
  uint8_t* logical;           // [n]
  double2* snap;              // [512] data-register state of ctl->snap_item after its last round
  double2* init_out;          // not null: compute the init state into it
};

using namespace oc;

// Shared memory of one trajectory besides its amplitudes; NR rounds are compiled together.
template <int NR>
struct Mem {
  enum : int { kRounds = NR };
  double2 fm[FM_COUNT][4];
  uint64_t thr[PR_COUNT];
  uint32_t bits, mask[NR];
  union {
    struct {
      fac::Touch T[NR * kTouches];
      uint8_t swap[NR * kTouches];
      uint8_t code[NR * kSites];
    } c;                                     // compile
    struct {
      double heap[kNAmp];
      double ur[kND];
    } r;                                     // readout
    double2 cs[16];                          // the trajectory's angles
  };
};

// This trajectory's matrices and draw thresholds (the conventions of the program builder; a twirled
// trajectory's coherent terms are draws, their unitaries the identity).
template <class G, class Mem>
__device__ void trajectory_noise(const G& g, const qec_noise& nz, bool cr, Mem& M) {
  const bool tw = nz.twirl != 0.0;
  const double q = 0.7853981633974483;   // pi / 4
  if (g.rank < 15) {
    const int l = g.rank;
    const double th[6] = {nz.theta_rx, nz.theta_rz, nz.theta_rzx, 2.0 * nz.phi_zz, nz.round_rz, nz.round_rx};
    double a = 0.0;
    if (l >= 9) {
      a = 0.5 * th[l - 9];
    } else {
      const double on = tw ? 0.0 : 0.5;
      const double rx = on * th[0], rz = on * th[1];
      a = l == 0 ? on * th[4] : l == 1 ? on * th[5] : l == 2 ? q + rx : l == 3 ? 2.0 * (q + rx) : l == 4 ? q + rz
        : l == 5 ? 2.0 * (q + rz) : l == 6 ? (nz.overrot_follows != 0.0 ? -q - rx : rx - q) : l == 7 ? q + on * th[2]
        : on * th[3];
    }
    double s, c;
    sincos(a, &s, &c);
    M.cs[l] = make_double2(c, s);
  }
  g.sync();
  if (g.rank < FM_SH) {
    const int id = g.rank;
    auto C = [&](int k) { return M.cs[k].x; };
    auto S = [&](int k) { return M.cs[k].y; };
    double2 m[4];
    auto rx = [&](double c, double s) {
      m[0] = m[3] = make_double2(c, 0.0);
      m[1] = m[2] = make_double2(0.0, -s);
    };
    m[1] = m[2] = make_double2(0.0, 0.0);
    if (id == FM_ROUND) {
      m[0] = make_double2(C(1) * C(0), -C(1) * S(0));
      m[3] = make_double2(C(1) * C(0), C(1) * S(0));
      m[1] = make_double2(S(1) * S(0), -S(1) * C(0));
      m[2] = make_double2(-S(1) * S(0), -S(1) * C(0));
    } else if (id == FM_RX1 || id == FM_RX2) {
      rx(C(id == FM_RX1 ? 2 : 3), S(id == FM_RX1 ? 2 : 3));
    } else if (id == FM_RZ1 || id == FM_RZ2) {
      const int k = id == FM_RZ1 ? 4 : 5;
      m[0] = make_double2(C(k), -S(k));
      m[3] = make_double2(C(k), S(k));
    } else if (id == FM_PREP || id == FM_POST) {
      if (cr) {
        rx(C(id == FM_PREP ? 6 : 2), S(id == FM_PREP ? 6 : 2));
      } else {
        const double h = 0.70710678118654752;
        m[0] = m[1] = m[2] = make_double2(h, 0.0);
        m[3] = make_double2(-h, 0.0);
      }
    } else {   // the gate's block for control 0 / 1, then its ZZ phases
      const double sg = id == FM_G0 ? 1.0 : -1.0;
      if (cr) {
        m[0] = m[3] = make_double2(C(7), 0.0);
        m[1] = m[2] = make_double2(0.0, -sg * S(7));
      } else {
        const bool x = id == FM_G1;
        m[0] = m[3] = make_double2(x ? 0.0 : 1.0, 0.0);
        m[1] = m[2] = make_double2(x ? 1.0 : 0.0, 0.0);
      }
      const double2 p = make_double2(C(8), -sg * S(8)), n = make_double2(C(8), sg * S(8));
      m[0] = fac::cmul(m[0], p);
      m[1] = fac::cmul(m[1], p);
      m[2] = fac::cmul(m[2], n);
      m[3] = fac::cmul(m[3], n);
    }
    for (int k = 0; k < 4; ++k) M.fm[id][k] = m[k];
  }
  if (g.rank < PR_COUNT) {
    // PR_TW_*: sin^2 of the half angle (of phi for the ZZ term), in the order RX, RZ, RZX, ZZ, round RZ, round RX
    const double s = g.rank < 3 ? 0.0 : M.cs[9 + g.rank - 3].y;
    const double p = g.rank == PR_P1 ? nz.p1 : g.rank == PR_P2 ? nz.p2 : g.rank == PR_IDLE ? nz.p_idle : tw ? s * s : 0.0;
    M.thr[g.rank] = fac::draw_threshold(p);
  }
  g.sync();
  if (g.rank == 0) gate_eigen<double2, double>(M.fm[FM_G0], M.fm[FM_G1], M.fm[FM_SH], M.fm[FM_A0], M.fm[FM_A1], M.fm[FM_LAM]);
  g.sync();
}

// Compiles rounds rnd .. rnd + nr - 1 into blk[nr][kNStab]; returns the flips in force after them.
template <class G, class Mem>
__device__ uint32_t compile_rounds(const G& g, const FactorView& F, Mem& M, Compiled<double>* blk, uint64_t seed, uint64_t traj,
                                   int rnd, int nr, uint32_t flips) {
  if (g.rank < nr) M.mask[g.rank] = 0;
  g.sync();
  fac::Rounds R;
  R.nr = nr;
  R.T = M.c.T;
  R.swap = M.c.swap;
  R.code = M.c.code;
  R.mask = M.mask;
  fac::compile_merge(g, F, M.thr, seed, traj, (uint64_t)rnd, M.fm, R, [](int, int, int) {});
  fac::compile_emit(g, F, M.fm, R, flips,
                    [&](int k, int i, double2 v) {
                      Compiled<double>& c = blk[k * kNStab + (i >> 2)];
                      c.rot[i & 3] = v;
                      c.form[i & 3] = rotation_form(v);
                    },
                    [&](int k, int b, int z, double2 d0, double2 d1) {
                      Compiled<double>& c = blk[k * kNStab + b];
                      c.d[0][z] = d0;
                      c.d[1][z] = d1;
                      c.wt[0][z] = fac::cnorm(d0);
                      c.wt[1][z] = fac::cnorm(d1);
                    });
  for (int i = g.rank; i < nr * kNStab; i += g.size)
    blk[i].u = uniform53(draw(seed, traj, (uint64_t)(rnd + i / kNStab), 0u, (uint32_t)(kND + i % kNStab), TAG_MEASURE).v[0]);
  g.sync();
  for (int k = 0; k < nr; ++k) flips ^= M.mask[k];
  return flips;
}

// Samples the final readout and writes the bits and the raw logical; the state to snap where asked.
template <int NT, class Mem>
__device__ void finish(const BatchArgs& a, const double2* psi, uint32_t flips, Mem& M, uint32_t item,
                       uint64_t seed, uint64_t traj, int rank) {
  const Group<NT> g{rank};
  g.sync();   // the compile's memory is reused
  if (rank < kND)
    M.r.ur[rank] = uniform53(draw(seed, traj, (uint64_t)a.rounds + 1, 0u, (uint32_t)rank, TAG_READOUT).v[0]);
  readout<double, NT>(psi, kND, flips, M.r.heap, M.r.ur, &M.bits, rank);
  const uint32_t x = M.bits;
  if (rank < kND) a.bits[(size_t)item * kND + rank] = (uint8_t)((x >> rank) & 1u);
  if (rank == 0) a.logical[item] = (uint8_t)(__popc(x & ((1u << kD) - 1u)) & 1);
  if (item == a.ctl->snap_item)
    for (int i = rank; i < kNAmp; i += NT) a.snap[i] = psi[i ^ flips];
  g.sync();
}

// ---- reduced register: one warp per trajectory, or one CTA of four where there are few ------------------
// What bounds it: the FP64 pipe (per round 1840 FP64 instructions a warp for the blocks, about 700 for their
// compile).  A warp's FP64 instructions issue at its scheduler's rate, a quarter of the SM's, so up to four
// trajectories per SM run on CTAs of four warps (150 trajectories of 5 rounds: 0.30 ms).
using WMem = Mem<1>;
constexpr size_t kGroupSmem = sizeof(WMem) + 16 * (size_t)kNAmp + sizeof(Compiled<double>) * kNStab;
constexpr size_t kWarpSmem = kGroupSmem;
static_assert(sizeof(WMem) % 16 == 0 && kWarpSmem % 16 == 0, "16-byte aligned amplitudes");

template <int NT>
__device__ void run_group(const BatchArgs& a, unsigned char* wsm, double* red, uint32_t item, int rank) {
  const Group<NT> g{rank};
  WMem& M = *reinterpret_cast<WMem*>(wsm);
  double2* psi = reinterpret_cast<double2*>(wsm + sizeof(WMem));
  Compiled<double>* blk = reinterpret_cast<Compiled<double>*>(wsm + sizeof(WMem) + 16 * (size_t)kNAmp);
  const bool init = a.init_out != nullptr;
  const qec_noise nz = init ? qec_noise{} : a.noise[item];
  const uint64_t traj = init ? 0ull : a.traj[item], seed = a.ctl->seed;
  trajectory_noise(g, nz, a.cr != 0, M);
  for (int i = rank; i < kNAmp; i += NT) psi[i] = init ? make_double2(i == 0 ? 1.0 : 0.0, 0.0) : a.psi0[i];
  uint8_t* syn = init ? nullptr : a.syn + (size_t)item * (a.rounds + 1) * kNStab;
  if (syn && rank < kNStab) syn[rank] = 0;
  uint32_t flips = 0;
  int parity = 0;
  for (int rnd = init ? 0 : 1; rnd <= (init ? 0 : a.rounds); ++rnd) {
    flips = compile_rounds(g, a.F, M, blk, seed, traj, rnd, 1, flips);
    for (int b = 0; b < kNStab; ++b) {
      const FBlock B = a.F.blocks[b];
      const int m = run_block<double, NT, kNAmp / (4 * NT)>(psi, B, blk[b], red, parity++, rank, init ? B.offset : -1);
      if (syn && rank == 0) syn[rnd * kNStab + b] = (uint8_t)(m ^ B.offset);
    }
  }
  if (init) {   // one warp
    double s = 0.0;
    for (int i = rank; i < kNAmp; i += NT) s += psi[i].x * psi[i].x + psi[i].y * psi[i].y;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const double sc = rsqrt(s);
    for (int i = rank; i < kNAmp; i += NT) a.init_out[i] = make_double2(psi[i ^ flips].x * sc, psi[i ^ flips].y * sc);
    return;
  }
  finish<NT>(a, psi, flips, M, item, seed, traj, rank);
}

// Warps: the first trajectory of each by its place (warp 0 of every CTA, then warp 1, ...: few
// trajectories then spread over the SMs), the others from the counter.
__global__ void k_batch(const __grid_constant__ BatchArgs a) {
  extern __shared__ __align__(16) unsigned char bsm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* wsm = bsm + (size_t)warp * kWarpSmem;
  if (a.init_out) {
    if (blockIdx.x == 0 && warp == 0) run_group<32>(a, wsm, nullptr, 0, lane);
    return;
  }
  const uint32_t all = gridDim.x * (blockDim.x >> 5), n = a.ctl->n[QEC_C128];
  for (uint32_t pos = (uint32_t)warp * gridDim.x + blockIdx.x; pos < n;) {
    run_group<32>(a, wsm, nullptr, a.idx[pos], lane);
    if (lane == 0) pos = all + atomicAdd(&a.ctl->counter[QEC_C128], 1u);
    pos = __shfl_sync(0xffffffffu, pos, 0);
  }
}

// One trajectory per CTA of 128 threads.
__global__ void __launch_bounds__(128) k_batch_cta(const __grid_constant__ BatchArgs a) {
  extern __shared__ __align__(16) unsigned char bsm[];
  __shared__ double red[2 * 64];
  run_group<128>(a, bsm, red, a.idx[blockIdx.x], (int)threadIdx.x);
}

// ---- unreduced register: one CTA per 17-qubit trajectory ------------------------------------------------
// The slab's index is the data index in its low 9 bits and the part's ancilla j in bit 9 + j.  A
// stabilizer's circuit leaves its ancilla in |m> with the data multiplied by D_m (factor.hpp), so it
// doubles the part of the slab in use: rotations on the 2^(9+j) amplitudes there are, then D_0 times
// them where they lie and D_1 times them at ancilla bit 1.  (Ops of different stabilizers on different
// qubits commute, and each qubit meets its gates in time order.)  When the part's four ancillas have
// entered, the norms of the 16 ancilla configurations give their measurements in order, and the
// measured configuration's data is the register for the next part.
constexpr int kUAmp = kNAmp << kNAnc;          // 8192 amplitudes
struct UMem {
  Mem<4> m;   // one CTA per SM, whose compile nothing else hides: four rounds together
  double norm[1 << kNAnc];
};
static_assert(sizeof(UMem) % 16 == 0, "16-byte aligned amplitudes");
constexpr size_t kUSmem = sizeof(UMem) + sizeof(double2) * kUAmp + sizeof(Compiled<double>) * kNStab * decltype(UMem::m)::kRounds;

// Rotations of data qubits j0 .. j0 + W - 1 of a block on 2^nb amplitudes in groups of 2^W; with `enter`,
// the block's ancilla enters at bit nb.  Two qubits a sweep are the faster choice (2048 complex128
// trajectories of 3 rounds: 3.58 ms, 3.96 with four): the early ancillas' slabs then fill the CTA.
template <int W>
__device__ void u_sweep(double2* slab, int nb, const FBlock& B, const Compiled<double>& C, int j0, bool enter) {
  using T2 = double2;
  constexpr int N = 1 << W;
  int q[W];
#pragma unroll
  for (int j = 0; j < W; ++j) q[j] = B.q[j0 + j];
  uint32_t off[N];
#pragma unroll
  for (int l = 0; l < N; ++l) {
    off[l] = 0;
#pragma unroll
    for (int j = 0; j < W; ++j) off[l] |= (uint32_t)((l >> j) & 1) << q[j];
  }
  for (uint32_t i = threadIdx.x; i < (1u << nb) >> W; i += blockDim.x) {
    uint32_t x = i;
#pragma unroll
    for (int j = 0; j < W; ++j) x = ((x >> q[j]) << (q[j] + 1)) | (x & ((1u << q[j]) - 1u));
    T2 v[N];
#pragma unroll
    for (int l = 0; l < N; ++l) v[l] = slab[x | off[l]];
#pragma unroll
    for (int j = 0; j < W; ++j) {
      const int f = C.form[j0 + j];
      if (f) {
        const T2 t = C.rot[j0 + j];
#pragma unroll
        for (int l = 0; l < N; ++l)
          if (!(l & (1 << j))) rotate(v[l], v[l | (1 << j)], t, f);
      }
    }
    if (!enter) {
#pragma unroll
      for (int l = 0; l < N; ++l) slab[x | off[l]] = v[l];
      continue;
    }
    int z0 = 0;   // the block's data qubits outside this sweep
    for (int j = 0; j < j0; ++j) z0 |= (int)((x >> B.q[j]) & 1u) << j;
#pragma unroll
    for (int l = 0; l < N; ++l) {
      const T2 d0 = C.d[0][z0 | (l << j0)], d1 = C.d[1][z0 | (l << j0)];
      T2 o;
      o.x = fma(-d0.y, v[l].y, d0.x * v[l].x);
      o.y = fma(d0.y, v[l].x, d0.x * v[l].y);
      slab[x | off[l]] = o;
      o.x = fma(-d1.y, v[l].y, d1.x * v[l].x);
      o.y = fma(d1.y, v[l].x, d1.x * v[l].y);
      slab[x | off[l] | (1u << nb)] = o;
    }
  }
  __syncthreads();
}

struct CtaGroup {
  int rank, size;
  __device__ __forceinline__ void sync() const { __syncthreads(); }
};

template <int NT>
__device__ void run_cta_u(const BatchArgs& a, unsigned char* sm, uint32_t item) {
  const int tid = threadIdx.x;
  const CtaGroup g{tid, NT};
  UMem& U = *reinterpret_cast<UMem*>(sm);
  double2* slab = reinterpret_cast<double2*>(sm + sizeof(UMem));
  Compiled<double>* compiled = reinterpret_cast<Compiled<double>*>(sm + sizeof(UMem) + sizeof(double2) * kUAmp);
  constexpr int NR = decltype(UMem::m)::kRounds;
  const qec_noise nz = a.noise[item];
  const uint64_t traj = a.traj[item], seed = a.ctl->seed;
  trajectory_noise(g, nz, a.cr != 0, U.m);
  for (int i = tid; i < kNAmp; i += NT) slab[i] = a.psi0[i];
  uint8_t* syn = a.syn + (size_t)item * (a.rounds + 1) * kNStab;
  if (tid < kNStab) syn[tid] = 0;
  uint32_t flips = 0;
  for (int rnd = 1; rnd <= a.rounds; ++rnd) {
    const int k = (rnd - 1) % NR;
    if (k == 0) flips = compile_rounds(g, a.F, U.m, compiled, seed, traj, rnd, min(NR, a.rounds + 1 - rnd), flips);
    const Compiled<double>* blk = compiled + k * kNStab;
    for (int part = 0; part < 2; ++part) {
      for (int j = 0; j < kNAnc; ++j) {
        const FBlock B = a.F.blocks[part * kNAnc + j];
        const Compiled<double>& C = blk[part * kNAnc + j];
        const int nb = kND + j;
        if (B.w == 2) {
          u_sweep<2>(slab, nb, B, C, 0, true);
        } else if (a.width > 4) {
          u_sweep<4>(slab, nb, B, C, 0, true);
        } else {
          if (C.form[0] | C.form[1]) u_sweep<2>(slab, nb, B, C, 0, false);
          u_sweep<2>(slab, nb, B, C, 2, true);
        }
      }
      // the 16 configurations' norms: 16 lanes each (lane l of a configuration takes data indices l,
      // l + 16, ...: the sums do not depend on the CTA's size)
      for (int c = tid >> 4; c < (1 << kNAnc); c += NT >> 4) {
        double w = 0.0;
        for (int i = tid & 15; i < kNAmp; i += 16) {
          const double2 v = slab[c * kNAmp + i];
          w = fma(v.x, v.x, fma(v.y, v.y, w));
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
        if ((tid & 15) == 0) U.norm[c] = w;
      }
      __syncthreads();
      // each ancilla in order, given the ones before (every thread alike)
      int m = 0;
      double norm = 0.0;
      for (int j = 0; j < kNAnc; ++j) {
        double s0 = 0.0, s1 = 0.0;
        for (int c = 0; c < (1 << kNAnc); ++c) {
          if ((c & ((1 << j) - 1)) != m) continue;
          if ((c >> j) & 1) s1 += U.norm[c];
          else s0 += U.norm[c];
        }
        const bool one = blk[part * kNAnc + j].u * (s0 + s1) < s1;
        m |= (int)one << j;
        norm = one ? s1 : s0;
      }
      const bool rescale = small_norm(norm);
      const double sc = norm_scale<double>(norm);
      if (m || rescale)
        for (int i = tid; i < kNAmp; i += NT) {
          double2 v = slab[m * kNAmp + i];
          if (rescale) {
            v.x *= sc;
            v.y *= sc;
          }
          slab[i] = v;
        }
      if (tid < kNAnc) {
        const int b = part * kNAnc + tid;
        syn[rnd * kNStab + b] = (uint8_t)(((m >> tid) & 1) ^ a.F.blocks[b].offset);
      }
      __syncthreads();
    }
  }
  finish<NT>(a, slab, flips, U.m, item, seed, traj, tid);
}

template <int NT>
__global__ void __launch_bounds__(NT) k_batch_u(const __grid_constant__ BatchArgs a) {
  extern __shared__ __align__(16) unsigned char usm[];
  __shared__ uint32_t s_pos;
  constexpr int kind = QEC_C128 + 2;
  const uint32_t n = a.ctl->n[kind];
  for (;;) {
    if (threadIdx.x == 0) s_pos = atomicAdd(&a.ctl->counter[kind], 1u);
    __syncthreads();
    const uint32_t pos = s_pos;
    __syncthreads();
    if (pos >= n) return;
    run_cta_u<NT>(a, usm, a.idx_u[pos]);
    __syncthreads();
  }
}

const void* u_kernel(int threads) {
  return threads == 128 ? (const void*)k_batch_u<128> : threads == 256 ? (const void*)k_batch_u<256> : (const void*)k_batch_u<512>;
}

}  // namespace

struct qec_batch {
  int rounds = 0, gates = 0, num_sms = 0;
  uint32_t cap = 0;
  cudaStream_t work = nullptr;
  cudaStream_t user = nullptr;
  cudaEvent_t ev_in = nullptr, ev_out = nullptr, t0 = nullptr, t1 = nullptr;
  unsigned char* d_all = nullptr;    // the allocation that holds every device buffer
  FactorProgram fac[2];              // [0] noisy program, every slot present; [1] init program
  unsigned char* d_fac[2] = {nullptr, nullptr};
  size_t fac_off[2][5] = {};
  // the complex64 engines' programs, again noisy and init: ops, blocks, then the unreduced register's ops, items,
  // passes, pass units and folded units at off64
  Program prog[2];
  UProgram uprog[2];
  unsigned char* d_prog64[2] = {nullptr, nullptr};
  size_t off64[2][7] = {};
  int n_upasses[2] = {0, 0}, n_upunits[2] = {0, 0};
  int u_items = 0;                   // unit matrices a CTA of theirs holds
  double* d_mats = nullptr;
  double2* d_psi0 = nullptr;
  float2* d_psi0_64 = nullptr;       // 2^9, then the unreduced register's slab
  uint32_t* d_idx = nullptr;         // a run's items by kind, one kind after the other
  std::vector<uint32_t> h_idx;
  cudaStream_t side[kKinds - 1] = {};   // launches besides the work stream's
  cudaEvent_t fork = nullptr, join[kKinds - 1] = {};
  qec_noise* d_noise = nullptr;
  uint64_t* d_traj = nullptr;
  BatchCtl* d_ctl = nullptr;
  BatchCtl* h_ctl = nullptr;   // pinned
  uint8_t* d_syn = nullptr;
  uint8_t* d_bits = nullptr;
  uint8_t* d_log = nullptr;
  int warps_per_cta = 8;
  int ctas_per_sm[kKinds] = {1, 1, 1, 1};
  float last_ms = 0.f;
  double2* d_snap = nullptr;
  int64_t snap_item = -1;   // for the next run
  bool snap_valid = false;  // a completed run recorded a snapshot
  int fusion_k = 0;         // unreduced engines: slab bits a sweep or pass may hold (0: no plan yet)
  int u_threads = 256;      // unreduced engines: threads per CTA
  bool tuning = false;      // runs use the configured warps however few trajectories they hold
};

namespace {

qec_status bfail(qec_status s, const std::string& m) {
  set_last_error(m);
  return s;
}

#define QEC_BCUDA(call)                                                                   \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess) {                                                              \
      cudaGetLastError(); /* reported here, not by the next launch */                     \
      return bfail(e_ == cudaErrorMemoryAllocation ? QEC_ENOMEM : QEC_ECUDA,              \
                   std::string(#call) + ": " + cudaGetErrorString(e_));                   \
    }                                                                                     \
  } while (0)

void batch_free(qec_batch* b) {
  if (b->d_all) cudaFree(b->d_all);
  if (b->fork) cudaEventDestroy(b->fork);
  for (int i = 0; i < kKinds - 1; ++i) {
    if (b->join[i]) cudaEventDestroy(b->join[i]);
    if (b->side[i]) cudaStreamDestroy(b->side[i]);
  }
  if (b->h_ctl) cudaFreeHost(b->h_ctl);
  cudaEvent_t evs[] = {b->ev_in, b->ev_out, b->t0, b->t1};
  for (cudaEvent_t e : evs) if (e) cudaEventDestroy(e);
  if (b->work) cudaStreamDestroy(b->work);
}

FactorView batch_program(const qec_batch* b, int which) {
  FactorView v = view_of(b->fac[which]);
  const unsigned char* d = b->d_fac[which];
  const size_t* off = b->fac_off[which];
  v.sites = reinterpret_cast<const FSite*>(d + off[0]);
  v.items = reinterpret_cast<const FItem*>(d + off[1]);
  v.touches = reinterpret_cast<const FTouch*>(d + off[2]);
  v.blocks = reinterpret_cast<const FBlock*>(d + off[3]);
  v.order = reinterpret_cast<const uint16_t*>(d + off[4]);
  return v;
}

BatchArgs batch_args(const qec_batch* b) {
  BatchArgs a;
  a.F = batch_program(b, 0);
  a.noise = b->d_noise;
  a.traj = b->d_traj;
  a.ctl = b->d_ctl;
  a.rounds = b->rounds;
  a.cr = b->gates == QEC_GATES_CR;
  a.width = b->fusion_k;
  a.psi0 = b->d_psi0;
  a.idx = a.idx_u = b->d_idx;
  a.syn = b->d_syn;
  a.bits = b->d_bits;
  a.logical = b->d_log;
  a.snap = b->d_snap;
  a.init_out = nullptr;
  return a;
}

// which: the noisy program or the init round's.
Batch64Args batch64_args(const qec_batch* b, int which) {
  const unsigned char* d = b->d_prog64[which];
  const size_t* off = b->off64[which];
  Batch64Args a{};
  a.ops = reinterpret_cast<const ProgOp*>(d + off[0]);
  a.blocks = reinterpret_cast<const BlockInfo*>(d + off[1]);
  a.n_ops = (int)b->prog[which].ops.size();
  a.uops = reinterpret_cast<const ProgOp*>(d + off[2]);
  a.uitems = reinterpret_cast<const UItem*>(d + off[3]);
  a.upasses = reinterpret_cast<const UPass*>(d + off[4]);
  a.upunits = reinterpret_cast<const UPassUnit*>(d + off[5]);
  a.uabs = reinterpret_cast<const UAbs*>(d + off[6]);
  a.n_uitems = (int)b->uprog[which].items.size();
  a.n_upasses = b->n_upasses[which];
  a.n_upunits = b->n_upunits[which];
  a.mats = b->d_mats;
  a.rounds = b->rounds;
  a.snap_item = ~0u;
  if (which) return a;
  a.noise = b->d_noise;
  a.traj = b->d_traj;
  a.seed = b->h_ctl->seed;
  a.snap_item = b->h_ctl->snap_item;
  a.syn = b->d_syn;
  a.bits = b->d_bits;
  a.logical = b->d_log;
  a.snap = b->d_snap;
  return a;
}

// Function attributes are the process's, not a handle's: the ceiling, so that handles of different shapes coexist; the
// largest carveout, so that engines side by side fit the same SMs (batch_dense.cu).
constexpr int kSmemCeiling = 226 * 1024;
cudaError_t set_attributes(const void* fn) {
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCeiling);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
}
size_t smem_for(int warps) { return (size_t)warps * kWarpSmem; }

// The run's launches: each engine that has trajectories, side by side (one CTA wave each at most, pulling
// trajectories from the control word's counters).
qec_status launch_batch(qec_batch* b) {
  const uint32_t* n = b->h_ctl->n;
  BatchArgs a = batch_args(b);
  Batch64Args a64 = batch64_args(b, 0);
  QEC_BCUDA(cudaEventRecord(b->fork, b->work));
  uint32_t base = 0;
  for (int kind = 0, used = 0; kind < kKinds; base += n[kind++]) {
    if (!n[kind]) continue;
    cudaStream_t s = used ? b->side[used - 1] : b->work;
    if (used) QEC_BCUDA(cudaStreamWaitEvent(s, b->fork, 0));
    const uint32_t wave = (uint32_t)(b->num_sms * b->ctas_per_sm[kind]);
    const bool u = kind >= 2;
    const uint32_t ctas = u ? n[kind] : (n[kind] + b->warps_per_cta - 1) / b->warps_per_cta, grid = ctas < wave ? ctas : wave;
    if (kind & 1) {
      a64.idx = b->d_idx + base;
      a64.n = n[kind];
      a64.counter = &b->d_ctl->counter[kind];
      a64.psi0 = u ? b->d_psi0_64 + kNAmp : b->d_psi0_64;
      // few trajectories: fewer warps on an SM each
      const uint32_t per = (n[kind] + b->num_sms - 1) / b->num_sms;
      if (u) QEC_BCUDA(launch_batch64_u(a64, b->u_threads, b->u_items, (int)grid, s));
      else if (per < (uint32_t)b->warps_per_cta && !b->tuning) QEC_BCUDA(launch_batch64(a64, (int)per, (int)((n[kind] + per - 1) / per), s));
      else QEC_BCUDA(launch_batch64(a64, b->warps_per_cta, (int)grid, s));
    } else if (u) {
      a.idx_u = b->d_idx + base;
      void* args[1] = {&a};
      QEC_BCUDA(cudaLaunchKernel(u_kernel(b->u_threads), dim3(grid), dim3((unsigned)b->u_threads), args, kUSmem, s));
    } else {
      a.idx = b->d_idx + base;
      // up to four trajectories per SM: a CTA of four warps each (see above)
      if (n[kind] <= 4u * (uint32_t)b->num_sms && !b->tuning) k_batch_cta<<<n[kind], 128, kGroupSmem, s>>>(a);
      else k_batch<<<grid, 32 * b->warps_per_cta, smem_for(b->warps_per_cta), s>>>(a);
      QEC_BCUDA(cudaGetLastError());
    }
    if (used) {
      QEC_BCUDA(cudaEventRecord(b->join[used - 1], s));
      QEC_BCUDA(cudaStreamWaitEvent(b->work, b->join[used - 1], 0));
    }
    ++used;
  }
  return QEC_OK;
}

// Threads per CTA (128..512) of the unreduced engines and their width in slab bits (2..6): the complex64
// engine's passes hold that many, the complex128 one rotates a weight-4 block's four data qubits in one sweep
// from 5 on, with the ancilla that enters, else two at a time.
qec_status set_fusion(qec_batch* b, int k, int threads) {
  if (k < 2 || k > kUMaxFusion || (threads != 128 && threads != 256 && threads != 512))
    return bfail(QEC_EINVAL, "fusion width must be in [2, 6] and threads 128, 256 or 512");
  int occ[2] = {0, 0};
  QEC_BCUDA(set_attributes(u_kernel(threads)));
  QEC_BCUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[0], u_kernel(threads), threads, kUSmem));
  QEC_BCUDA(setup_batch64_u(threads, b->u_items, &occ[1]));
  if (occ[0] < 1 || occ[1] < 1) return bfail(QEC_EUNSUPPORTED, "unreduced batched kernel does not fit an SM with this shape");
  for (int w = 0; w < 2 && k != b->fusion_k; ++w) {
    std::vector<UPass> passes;
    std::vector<UPassUnit> punits;
    std::vector<UAbs> uabs;
    build_passes(b->uprog[w], k, passes, punits, uabs);
    const void* src[3] = {passes.data(), punits.data(), uabs.data()};
    const size_t bytes[3] = {sizeof(UPass) * passes.size(), sizeof(UPassUnit) * punits.size(), sizeof(UAbs) * uabs.size()};
    for (int i = 0; i < 3; ++i)
      if (bytes[i]) QEC_BCUDA(cudaMemcpy(b->d_prog64[w] + b->off64[w][4 + i], src[i], bytes[i], cudaMemcpyHostToDevice));
    b->n_upasses[w] = (int)passes.size();
    b->n_upunits[w] = (int)punits.size();
  }
  b->fusion_k = k;
  b->u_threads = threads;
  b->ctas_per_sm[QEC_C128 + 2] = occ[0];
  b->ctas_per_sm[QEC_C64 + 2] = occ[1];
  return QEC_OK;
}

qec_status set_shape(qec_batch* b, int warps) {
  if (warps < 1 || warps > 10) return bfail(QEC_EINVAL, "warps per CTA must be in [1, 10]");
  int occ[2] = {0, 0};
  QEC_BCUDA(set_attributes((const void*)k_batch));
  QEC_BCUDA(set_attributes((const void*)k_batch_cta));
  QEC_BCUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[0], k_batch, 32 * warps, smem_for(warps)));
  QEC_BCUDA(setup_batch64(warps, &occ[1]));
  if (occ[0] < 1 || occ[1] < 1) return bfail(QEC_EUNSUPPORTED, "batched kernel does not fit an SM with this shape");
  b->warps_per_cta = warps;
  b->ctas_per_sm[QEC_C128] = occ[0];
  b->ctas_per_sm[QEC_C64] = occ[1];
  return QEC_OK;
}

}  // namespace

// Nothing throws across the C entries: what their host containers or strings may throw becomes a status.
template <class F>
static qec_status guarded(F f) {
  try {
    return f();
  } catch (...) {
    return bfail(QEC_ENOMEM, "host allocation failed");
  }
}

extern "C" {

qec_status qec_debug_unreduced_plan(int32_t gates, int32_t k, int32_t* items, uint32_t cap, uint32_t* n_items,
                                    int32_t* pass_units, uint32_t* n_pass_units, int32_t* absorbs, uint32_t* n_absorbs) {
  return guarded([&]() -> qec_status {
    if (!items || !n_items || !pass_units || !n_pass_units || !absorbs || !n_absorbs)
      return bfail(QEC_EINVAL, "null argument");
    if (k < 2 || k > kUMaxFusion) return bfail(QEC_EINVAL, "fusion width must be in [2, 6]");
    qec_params p{};
    p.d = kD;
    p.rounds = 1;
    p.layout = QEC_LAYOUT_REDUCED;   // the parameters qec_batch_create builds both programs from
    p.gates = gates;
    p.precision = QEC_C128;
    p.noise = qec_noise{1, 1, 1, 1, 1, 1, 1, 1, 1, 0};   // every site and coherent op present
    std::string err;
    UProgram U;
    if (!build_unreduced_program(p, true, U, err, true)) return bfail(QEC_EINVAL, err);
    std::vector<UPass> passes;
    std::vector<UPassUnit> punits;
    std::vector<UAbs> uabs;
    build_passes(U, k, passes, punits, uabs);
    *n_items = (uint32_t)U.items.size();
    if (U.items.size() > cap || punits.size() > cap || uabs.size() > cap)
      return bfail(QEC_EINVAL, "capacity too small");
    for (size_t i = 0; i < U.items.size(); ++i) {
      const UItem& u = U.items[i];
      items[4 * i] = u.kind;
      items[4 * i + 1] = u.nq;
      items[4 * i + 2] = u.qa;
      items[4 * i + 3] = u.kind == 0 && u.nq == 2 ? u.qb : -1;
    }
    uint32_t na = 0;
    for (size_t i = 0; i < punits.size(); ++i) {
      pass_units[i] = punits[i].item;
      for (int e = punits[i].abs0; e < punits[i].abs0 + punits[i].nabs; ++e) {
        absorbs[3 * na] = uabs[e].item1;
        absorbs[3 * na + 1] = punits[i].item;
        absorbs[3 * na + 2] = uabs[e].mode;
        ++na;
      }
    }
    *n_pass_units = (uint32_t)punits.size();
    *n_absorbs = na;
    return QEC_OK;
  });
}

qec_status qec_batch_create(int32_t d, int32_t rounds, int32_t gates, uint32_t max_traj, void* cuda_stream,
                            qec_batch** out) {
  return guarded([&]() -> qec_status {
    if (!out) return bfail(QEC_EINVAL, "null output handle");
    *out = nullptr;
    if (d != kD) return bfail(QEC_EUNSUPPORTED, "the batched form runs the d = 3 reduced register");
    if (rounds < 0 || rounds > 64 || max_traj == 0 || max_traj > (1u << 24))
      return bfail(QEC_EINVAL, "rounds must be in [0, 64] and max_traj in [1, 2^24]");
    qec_params p{};
    p.d = d;
    p.rounds = rounds;
    p.layout = QEC_LAYOUT_REDUCED;
    p.gates = gates;
    p.precision = QEC_C128;
    // every noise site and coherent op present; the per-trajectory values decide what they do
    p.noise = qec_noise{1, 1, 1, 1, 1, 1, 1, 1, 1, 0};
    std::string err;
    qec_batch* b = new (std::nothrow) qec_batch();
    if (!b) return bfail(QEC_ENOMEM, "host allocation failed");
    struct Free {
      void operator()(qec_batch* x) const { batch_free(x); delete x; }
    };
    std::unique_ptr<qec_batch, Free> owner(b);
    b->rounds = rounds;
    b->gates = gates;
    b->cap = max_traj;
    b->user = static_cast<cudaStream_t>(cuda_stream);
    for (int w = 0; w < 2; ++w) {
      Program& P = b->prog[w];
      UProgram& U = b->uprog[w];
      if (!build_program(p, w == 0, P, err, w == 0) || !build_factor(P, b->fac[w], err) ||
          !build_unreduced_program(p, w == 0, U, err, w == 0))
        return bfail(QEC_EINVAL, err);
      if (b->fac[w].sites.size() > (size_t)kSites || P.ops.size() > (size_t)kBatchOps || U.items.size() > (size_t)kUMaxItems)
        return bfail(QEC_EUNSUPPORTED, "a round has more draws, ops or units than the engines' tables");
      if ((int)U.items.size() > b->u_items) b->u_items = (int)U.items.size();
    }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&b->num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->work, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_in, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_out, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreate(&b->t0);
    if (e == cudaSuccess) e = cudaEventCreate(&b->t1);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming);
    for (int i = 0; i < kKinds - 1; ++i) {
      if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->side[i], cudaStreamNonBlocking);
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->join[i], cudaEventDisableTiming);
    }
    if (e != cudaSuccess) return bfail(QEC_ECUDA, std::string("CUDA setup: ") + cudaGetErrorString(e));
    const size_t syn_bytes = (size_t)max_traj * (rounds + 1) * kNStab;
    const void* src[2][12];
    size_t bytes[2][12], total[2] = {0, 0}, total64[2] = {0, 0};
    for (int w = 0; w < 2; ++w) {
      const FactorProgram& F = b->fac[w];
      const Program& P = b->prog[w];
      const UProgram& U = b->uprog[w];
      const size_t items = U.items.size();   // at least as many as there are passes, pass units or folded units
      const void* s[12] = {F.sites.data(), F.items.data(), F.touches.data(), F.blocks.data(), F.order.data(),
                           P.ops.data(), P.blocks.data(), U.ops.data(), U.items.data(), nullptr, nullptr, nullptr};
      const size_t n[12] = {sizeof(FSite) * F.sites.size(), sizeof(FItem) * F.items.size(), sizeof(FTouch) * F.touches.size(),
                            sizeof(FBlock) * F.blocks.size(), sizeof(uint16_t) * F.order.size(),
                            sizeof(ProgOp) * P.ops.size(), sizeof(BlockInfo) * P.blocks.size(), sizeof(ProgOp) * U.ops.size(),
                            sizeof(UItem) * items, sizeof(UPass) * items, sizeof(UPassUnit) * items, sizeof(UAbs) * items};
      for (int i = 0; i < 12; ++i) {
        size_t& at = i < 5 ? total[w] : total64[w];
        src[w][i] = s[i];
        bytes[w][i] = n[i];
        (i < 5 ? b->fac_off[w][i] : b->off64[w][i - 5]) = at;
        at += (n[i] + 255) / 256 * 256;
      }
    }
    void** allocs[] = {(void**)&b->d_fac[0], (void**)&b->d_fac[1], (void**)&b->d_prog64[0], (void**)&b->d_prog64[1],
                       (void**)&b->d_mats, (void**)&b->d_psi0, (void**)&b->d_psi0_64, (void**)&b->d_noise, (void**)&b->d_traj,
                       (void**)&b->d_ctl, (void**)&b->d_syn, (void**)&b->d_bits, (void**)&b->d_log, (void**)&b->d_idx,
                       (void**)&b->d_snap};
    const size_t sizes[] = {total[0], total[1], total64[0], total64[1], sizeof(b->prog[0].mats), sizeof(double2) * kNAmp,
                            sizeof(float2) * (kNAmp + kSlabAmps), sizeof(qec_noise) * max_traj, sizeof(uint64_t) * max_traj,
                            sizeof(BatchCtl), syn_bytes, (size_t)max_traj * kND, (size_t)max_traj, sizeof(uint32_t) * max_traj,
                            sizeof(double2) * kNAmp};
    // one allocation, the programs and matrices (the first five) first: one copy
    constexpr int kUploads = 5, kParts = sizeof(sizes) / sizeof(sizes[0]);
    size_t off[kParts + 1] = {0};
    for (int i = 0; i < kParts; ++i) off[i + 1] = off[i] + (sizes[i] + 255) / 256 * 256;
    e = cudaMalloc((void**)&b->d_all, off[kParts]);
    if (e != cudaSuccess) return bfail(QEC_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    for (int i = 0; i < kParts; ++i) *allocs[i] = b->d_all + off[i];
    std::vector<unsigned char> stage(off[kUploads]);
    for (int w = 0; w < 2; ++w)
      for (int i = 0; i < 12; ++i)
        if (src[w][i] && bytes[w][i])
          std::memcpy(stage.data() + (i < 5 ? off[w] + b->fac_off[w][i] : off[2 + w] + b->off64[w][i - 5]), src[w][i], bytes[w][i]);
    std::memcpy(stage.data() + off[4], b->prog[0].mats, sizeof(b->prog[0].mats));
    e = cudaMemcpy(b->d_all, stage.data(), stage.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return bfail(QEC_ECUDA, std::string("upload: ") + cudaGetErrorString(e));
    e = cudaMallocHost((void**)&b->h_ctl, sizeof(BatchCtl));
    if (e != cudaSuccess) return bfail(QEC_ENOMEM, "pinned allocation failed");
    std::memset(b->h_ctl, 0, sizeof(BatchCtl));
    e = cudaMemcpy(b->d_ctl, b->h_ctl, sizeof(BatchCtl), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return bfail(QEC_ECUDA, cudaGetErrorString(e));
    qec_status st = set_shape(b, 10);
    if (st) return st;
    if ((st = set_fusion(b, 4, 256))) return st;
    // the noise-free init round, once per precision, in complex64 once per register, side by side
    BatchArgs a = batch_args(b);
    a.F = batch_program(b, 1);
    a.init_out = b->d_psi0;
    k_batch<<<1, 32, smem_for(1), b->work>>>(a);
    e = cudaGetLastError();
    Batch64Args a64 = batch64_args(b, 1);
    a64.out = b->d_psi0_64;
    if (e == cudaSuccess) e = launch_batch64(a64, 1, 1, b->side[0]);
    a64.out = b->d_psi0_64 + kNAmp;
    if (e == cudaSuccess) e = launch_batch64_u(a64, 256, b->u_items, 1, b->side[1]);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->work);
    for (int i = 0; i < 2 && e == cudaSuccess; ++i) e = cudaStreamSynchronize(b->side[i]);
    if (e != cudaSuccess) return bfail(QEC_ECUDA, std::string("init round: ") + cudaGetErrorString(e));
    *out = owner.release();
    return QEC_OK;
  });
}

qec_status qec_batch_run(qec_batch* b, uint64_t seed, uint32_t n, const uint64_t* traj, const int32_t* kind,
                         const qec_noise* noise, uint8_t* syndromes, uint8_t* data_bits, uint8_t* raw_logical) {
  return guarded([&]() -> qec_status {
    if (!b) return bfail(QEC_EINVAL, "null handle");
    if (n > b->cap) return bfail(QEC_EINVAL, "n exceeds the batch capacity given at creation");
    if (n == 0) return QEC_OK;
    if (!traj || !kind || !noise) return bfail(QEC_EINVAL, "null input array");
    for (uint32_t i = 0; i < n; ++i) {
      if (kind[i] < 0 || kind[i] > 3)
        return bfail(QEC_EINVAL, "kind must be precision (QEC_C128 or QEC_C64) | 2 * layout (QEC_LAYOUT_*)");
      const qec_noise& z = noise[i];
      const double pr[3] = {z.p1, z.p2, z.p_idle};
      for (double v : pr)
        if (!(v >= 0.0 && v <= 1.0)) return bfail(QEC_EINVAL, "noise probabilities must be in [0, 1]");
      const double an[6] = {z.theta_rx, z.theta_rz, z.theta_rzx, z.phi_zz, z.round_rz, z.round_rx};
      for (double v : an)
        if (!(std::fabs(v) <= 4.0)) return bfail(QEC_EINVAL, "angles must be finite with |angle| <= 4");
      if (z.twirl != 0.0 && z.twirl != 1.0) return bfail(QEC_EINVAL, "twirl must be 0 or 1");
      if (z.overrot_follows != 0.0 && z.overrot_follows != 1.0) return bfail(QEC_EINVAL, "overrot_follows must be 0 or 1");
    }
    if (b->user) {
      QEC_BCUDA(cudaEventRecord(b->ev_in, b->user));
      QEC_BCUDA(cudaStreamWaitEvent(b->work, b->ev_in, 0));
    }
    QEC_BCUDA(cudaMemcpyAsync(b->d_traj, traj, sizeof(uint64_t) * n, cudaMemcpyHostToDevice, b->work));
    QEC_BCUDA(cudaMemcpyAsync(b->d_noise, noise, sizeof(qec_noise) * n, cudaMemcpyHostToDevice, b->work));
    uint32_t count[kKinds] = {0, 0, 0, 0}, at[kKinds];
    for (uint32_t i = 0; i < n; ++i) ++count[kind[i]];
    at[0] = 0;
    for (int k = 1; k < kKinds; ++k) at[k] = at[k - 1] + count[k - 1];
    b->h_idx.resize(n);
    for (uint32_t i = 0; i < n; ++i) b->h_idx[at[kind[i]]++] = i;
    QEC_BCUDA(cudaMemcpyAsync(b->d_idx, b->h_idx.data(), sizeof(uint32_t) * n, cudaMemcpyHostToDevice, b->work));
    QEC_BCUDA(cudaStreamSynchronize(b->work));   // h_ctl is reused
    b->h_ctl->seed = seed;
    for (int k = 0; k < kKinds; ++k) {
      b->h_ctl->n[k] = count[k];
      b->h_ctl->counter[k] = 0;
    }
    const bool snap = b->snap_item >= 0 && b->snap_item < (int64_t)n;
    b->h_ctl->snap_item = snap ? (uint32_t)b->snap_item : ~0u;
    b->snap_valid = false;
    QEC_BCUDA(cudaMemcpyAsync(b->d_ctl, b->h_ctl, sizeof(BatchCtl), cudaMemcpyHostToDevice, b->work));
    QEC_BCUDA(cudaEventRecord(b->t0, b->work));
    qec_status st = launch_batch(b);
    if (st) return st;
    QEC_BCUDA(cudaEventRecord(b->t1, b->work));
    const size_t ss = (size_t)(b->rounds + 1) * kNStab;
    if (syndromes) QEC_BCUDA(cudaMemcpyAsync(syndromes, b->d_syn, n * ss, cudaMemcpyDeviceToHost, b->work));
    if (data_bits) QEC_BCUDA(cudaMemcpyAsync(data_bits, b->d_bits, (size_t)n * kND, cudaMemcpyDeviceToHost, b->work));
    if (raw_logical) QEC_BCUDA(cudaMemcpyAsync(raw_logical, b->d_log, n, cudaMemcpyDeviceToHost, b->work));
    if (b->user) {
      QEC_BCUDA(cudaEventRecord(b->ev_out, b->work));
      QEC_BCUDA(cudaStreamWaitEvent(b->user, b->ev_out, 0));
    }
    QEC_BCUDA(cudaStreamSynchronize(b->work));
    QEC_BCUDA(cudaEventElapsedTime(&b->last_ms, b->t0, b->t1));
    b->snap_valid = snap;
    return QEC_OK;
  });
}

qec_status qec_batch_autotune(qec_batch* b, uint64_t seed, uint32_t n, const uint64_t* traj, const int32_t* kind,
                              const qec_noise* noise, int32_t* chosen_warps, float* best_ms) {
  return guarded([&]() -> qec_status {
    if (!b || !chosen_warps || !best_ms || !traj || !kind || !noise) return bfail(QEC_EINVAL, "null argument");
    // the sample split by register: each engine is tuned on its own trajectories, on the kernels that large runs
    // take, repeated until they fill the GPU twice (or the handle); without any its configuration stays
    std::vector<uint64_t> tr[2];
    std::vector<int32_t> kd[2];
    std::vector<qec_noise> nz[2];
    for (uint32_t i = 0; i < n; ++i) {
      const int u = (kind[i] & 2) ? 1 : 0;
      tr[u].push_back(traj[i]);
      kd[u].push_back(kind[i]);
      nz[u].push_back(noise[i]);
    }
    for (int u = 0; u < 2; ++u) {
      const size_t own = tr[u].size(), want = std::min<size_t>(b->cap, (u ? 4 : 40) * (size_t)b->num_sms);
      for (size_t i = 0; own && i + own < want; ++i) {
        tr[u].push_back(tr[u][i]);
        kd[u].push_back(kd[u][i]);
        nz[u].push_back(nz[u][i]);
      }
    }
    struct Tuning {
      qec_batch* b;
      explicit Tuning(qec_batch* x) : b(x) { b->tuning = true; }
      ~Tuning() { b->tuning = false; }
    };
    auto time_run = [&](int u, float& t) -> qec_status {
      const Tuning on(b);
      for (int rep = 0; rep < 3; ++rep) {   // first run warms up, the faster of the others counts
        qec_status st = qec_batch_run(b, seed, (uint32_t)tr[u].size(), tr[u].data(), kd[u].data(), nz[u].data(),
                                      nullptr, nullptr, nullptr);
        if (st) return st;
        if (rep) t = rep == 1 || b->last_ms < t ? b->last_ms : t;
      }
      return QEC_OK;
    };
    qec_status st;
    if (!tr[0].empty()) {   // reduced register: warps per CTA
      int best = -1;
      float best_t = 0.f;
      for (int w : {2, 4, 6, 8, 10}) {
        if (set_shape(b, w) != QEC_OK) continue;
        float t = 0.f;
        if ((st = time_run(0, t))) return st;
        if (best < 0 || t < best_t) {
          best = w;
          best_t = t;
        }
      }
      if (best < 0) return bfail(QEC_EUNSUPPORTED, "no batched kernel shape fits");
      if ((st = set_shape(b, best))) return st;
    }
    if (!tr[1].empty()) {   // unreduced register: width in slab bits x threads per CTA
      int bk = -1, bthr = 256;
      float bu = 0.f;
      for (int k = 2; k <= kUMaxFusion; ++k)
        for (int thr : {128, 256}) {
          if (set_fusion(b, k, thr) != QEC_OK) continue;
          float t = 0.f;
          if ((st = time_run(1, t))) return st;
          if (bk < 0 || t < bu) {
            bk = k;
            bthr = thr;
            bu = t;
          }
        }
      if (bk < 0) return bfail(QEC_EUNSUPPORTED, "no unreduced engine shape fits");
      if ((st = set_fusion(b, bk, bthr))) return st;
    }
    float t_all = 0.f;   // the whole sample with the chosen configuration
    for (int rep = 0; rep < 2; ++rep) {
      if ((st = qec_batch_run(b, seed, n, traj, kind, noise, nullptr, nullptr, nullptr))) return st;
      t_all = b->last_ms;
    }
    *chosen_warps = b->warps_per_cta;
    *best_ms = t_all;
    return QEC_OK;
  });
}

qec_status qec_batch_config(const qec_batch* b, int32_t* warps_per_cta, int32_t* fusion_width, int32_t* u_threads) {
  if (!b || !warps_per_cta || !fusion_width || !u_threads) return bfail(QEC_EINVAL, "null argument");
  *warps_per_cta = b->warps_per_cta;
  *fusion_width = b->fusion_k;
  *u_threads = b->u_threads;
  return QEC_OK;
}

qec_status qec_batch_set_config(qec_batch* b, int32_t warps_per_cta, int32_t fusion_width, int32_t u_threads) {
  return guarded([&]() -> qec_status {
    if (!b) return bfail(QEC_EINVAL, "null handle");
    qec_status st = set_shape(b, warps_per_cta);
    if (st) return st;
    return set_fusion(b, fusion_width, u_threads);
  });
}

qec_status qec_batch_snapshot(qec_batch* b, int64_t item) {
  if (!b || item < -1) return bfail(QEC_EINVAL, "null handle or item < -1");
  b->snap_item = item;
  return QEC_OK;
}

qec_status qec_batch_get_state(qec_batch* b, void* host_buf, size_t bytes) {
  if (!b || !host_buf) return bfail(QEC_EINVAL, "null argument");
  if (bytes < sizeof(double2) * kNAmp) return bfail(QEC_EINVAL, "host buffer too small");
  if (!b->snap_valid) return bfail(QEC_EINVAL, "no completed run recorded a snapshot");
  double* out = static_cast<double*>(host_buf);
  QEC_BCUDA(cudaMemcpy(out, b->d_snap, sizeof(double2) * kNAmp, cudaMemcpyDeviceToHost));
  double nrm = 0.0;   // the reduced register keeps the norm P(m) of the last outcome; report unit norm
  for (int i = 0; i < 2 * kNAmp; ++i) nrm += out[i] * out[i];
  const double sc = nrm > 0.0 ? 1.0 / std::sqrt(nrm) : 1.0;
  for (int i = 0; i < 2 * kNAmp; ++i) out[i] *= sc;
  return QEC_OK;
}

qec_status qec_batch_last_ms(const qec_batch* b, float* ms) {
  if (!b || !ms) return bfail(QEC_EINVAL, "null argument");
  *ms = b->last_ms;
  return QEC_OK;
}

qec_status qec_batch_destroy(qec_batch* b) {
  if (!b) return QEC_OK;
  if (b->work) cudaStreamSynchronize(b->work);
  batch_free(b);
  delete b;
  return QEC_OK;
}

}  // extern "C"
