// Batched form: many small-register trajectories at once, one launch per engine.
//
// A trajectory of the d = 3 code runs on chip, its blocks in factored form (factor.hpp).  Reduced
// register (9 data qubits + the reused ancilla, Sec. II.B): one warp per trajectory, 512 amplitudes
// (onchip.cuh).  Unreduced register (all 17 qubits): one CTA per trajectory.  A part's four ancillas
// are active together; the other part's are |0> throughout (reset after their measurement, untouched
// before their part), so a slab of 2^13 amplitudes holds the exact state.  Warps and CTAs take
// trajectories from device work counters, so precisions and noise parameters mix freely in one
// launch.  The circuit program is built once with every noise and coherent slot present; a
// trajectory's own matrices and draw thresholds follow from its noise input (a zero angle is the
// identity, a zero probability never fires).
//
// The FP64 pipe bounds the complex128 trajectories, the compile and the sweeps' latency the complex64 ones.
// 2048 trajectories of 3 rounds, dense blocks and gate units before: reduced register 8.24 -> 1.43 ms
// complex128, 2.20 -> 0.61 complex64; unreduced 33.3 -> 3.58 and 10.0 -> 1.17.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "../../include/qecsv.h"
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
constexpr int kUMaxFusionDecl = 6;       // widest sweep a configuration may ask for (slab bits)

struct BatchCtl {
  uint64_t seed;
  uint32_t n;                 // reduced-register (10-qubit) trajectories in this run
  unsigned int counter;       // their work queue head (zeroed before every run)
  uint32_t n_u[2];            // unreduced-register (17-qubit) trajectories in this run: complex128, complex64
  unsigned int counter_u[2];  // their work queue heads
  uint32_t snap_item;         // item whose final data-register state goes to snap (~0u = none)
};

// One pass of the unreduced engine over the slab: kind 0 applies the units punits[u0, u1) (disjoint
// slab bits, together `nbits` bits listed in bits[]); kind 1 measures the ancilla of items[item].
struct UPass {
  int32_t kind;
  int32_t item;
  int32_t u0, u1;
  int32_t nbits;
  int32_t bits[kUMaxFusionDecl];
};

// A unit inside a pass: items[item] on slab bits qa (, qb), and the pass's other bits.  A two-qubit
// unit also carries the one-qubit units folded into its matrix: entries abs0 .. abs0 + nabs - 1 of
// the program's UAbs list.
struct UPassUnit {
  int32_t item;
  int32_t nq, qa, qb;
  int32_t nother;
  int32_t other[kUMaxFusionDecl];
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

struct BatchArgs {
  FactorView F;               // noisy program (all slots present), or the init program
  const qec_noise* noise;     // [n]
  const int32_t* kind;        // [n]: bit 0 = complex64 (else complex128), bit 1 = unreduced register
  const uint32_t* idx;        // reduced-register items of this run
  const uint32_t* idx_u;      // unreduced-register items of this run
  const uint64_t* traj;       // [n]
  BatchCtl* ctl;
  int rounds, cr;
  int width;                  // unreduced register: slab bits a sweep may hold (see u_sweep)
  const void* psi0[2];        // init code state per precision
  uint8_t* syn;               // [n][rounds+1][8]
  uint8_t* bits;              // [n][9]
  uint8_t* logical;           // [n]
  double2* snap;              // [512] data-register state of ctl->snap_item after its last round
  int init_mode;              // 1: compute the init state of precision init_prec into init_out
  int init_prec;
  void* init_out;
};

using namespace oc;

// Shared memory of one trajectory besides its amplitudes; NR rounds are compiled together.
template <int NR>
struct Mem {
  static constexpr int kRounds = NR;
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
  if (g.rank < FM_COUNT) {
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
}

// Compiles rounds rnd .. rnd + nr - 1 into blk[nr][kNStab]; returns the flips in force after them.
template <typename T, class G, class Mem>
__device__ uint32_t compile_rounds(const G& g, const FactorView& F, Mem& M, Compiled<T>* blk, uint64_t seed, uint64_t traj,
                                   int rnd, int nr, uint32_t flips) {
  using T2 = typename V2t<T>::t;
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
                      Compiled<T>& c = blk[k * kNStab + (i >> 2)];
                      c.rot[i & 3] = make2<T2>(v.x, v.y);
                      c.form[i & 3] = rotation_form(v);
                    },
                    [&](int k, int b, int z, double2 d0, double2 d1) {
                      Compiled<T>& c = blk[k * kNStab + b];
                      c.d[0][z] = make2<T2>(d0.x, d0.y);
                      c.d[1][z] = make2<T2>(d1.x, d1.y);
                      c.wt[0][z] = (T)fac::cnorm(d0);
                      c.wt[1][z] = (T)fac::cnorm(d1);
                    });
  for (int i = g.rank; i < nr * kNStab; i += g.size)
    blk[i].u = uniform53(draw(seed, traj, (uint64_t)(rnd + i / kNStab), 0u, (uint32_t)(kND + i % kNStab), TAG_MEASURE).v[0]);
  g.sync();
  for (int k = 0; k < nr; ++k) flips ^= M.mask[k];
  return flips;
}

// Samples the final readout and writes the bits and the raw logical; the state to snap where asked.
template <typename T, int NT, class Mem>
__device__ void finish(const BatchArgs& a, const typename V2t<T>::t* psi, uint32_t flips, Mem& M, uint32_t item,
                       uint64_t seed, uint64_t traj, int rank) {
  const Group<NT> g{rank};
  g.sync();   // the compile's memory is reused
  if (rank < kND)
    M.r.ur[rank] = uniform53(draw(seed, traj, (uint64_t)a.rounds + 1, 0u, (uint32_t)rank, TAG_READOUT).v[0]);
  readout<T, NT>(psi, kND, flips, M.r.heap, M.r.ur, &M.bits, rank);
  const uint32_t x = M.bits;
  if (rank < kND) a.bits[(size_t)item * kND + rank] = (uint8_t)((x >> rank) & 1u);
  if (rank == 0) a.logical[item] = (uint8_t)(__popc(x & ((1u << kD) - 1u)) & 1);
  if (item == a.ctl->snap_item)
    for (int i = rank; i < kNAmp; i += NT) a.snap[i] = make_double2((double)psi[i ^ flips].x, (double)psi[i ^ flips].y);
  g.sync();
}

// ---- reduced register: one warp per trajectory, or one CTA of four where there are few ------------------
// What bounds it: the FP64 pipe (complex128: per round 1840 FP64 instructions a warp for the blocks, about
// 700 for their compile, which complex64 trajectories run too).  A warp's FP64 instructions issue at its
// scheduler's rate, a quarter of the SM's, so up to four trajectories per SM run on CTAs of four warps
// (301 trajectories of 5 rounds, half complex128, with their host copies: 1.84 -> 0.84 ms).
using WMem = Mem<1>;
constexpr size_t kGroupSmem = sizeof(WMem) + 16 * (size_t)kNAmp + sizeof(Compiled<double>) * kNStab;
constexpr size_t kWarpSmem = kGroupSmem;
static_assert(sizeof(WMem) % 16 == 0 && kWarpSmem % 16 == 0, "16-byte aligned amplitudes");

template <typename T, int NT>
__device__ void run_group(const BatchArgs& a, unsigned char* wsm, double* red, uint32_t item, int rank) {
  using T2 = typename V2t<T>::t;
  const Group<NT> g{rank};
  WMem& M = *reinterpret_cast<WMem*>(wsm);
  T2* psi = reinterpret_cast<T2*>(wsm + sizeof(WMem));
  Compiled<T>* blk = reinterpret_cast<Compiled<T>*>(wsm + sizeof(WMem) + 16 * (size_t)kNAmp);
  const bool init = a.init_mode != 0;
  const qec_noise nz = init ? qec_noise{} : a.noise[item];
  const uint64_t traj = init ? 0ull : a.traj[item], seed = a.ctl->seed;
  trajectory_noise(g, nz, a.cr != 0, M);
  const T2* p0 = reinterpret_cast<const T2*>(a.psi0[sizeof(T) == 4]);
  for (int i = rank; i < kNAmp; i += NT) psi[i] = init ? make2<T2>(i == 0 ? 1.0 : 0.0, 0.0) : p0[i];
  uint8_t* syn = init ? nullptr : a.syn + (size_t)item * (a.rounds + 1) * kNStab;
  if (syn && rank < kNStab) syn[rank] = 0;
  uint32_t flips = 0;
  int parity = 0;
  for (int rnd = init ? 0 : 1; rnd <= (init ? 0 : a.rounds); ++rnd) {
    flips = compile_rounds<T>(g, a.F, M, blk, seed, traj, rnd, 1, flips);
    for (int b = 0; b < kNStab; ++b) {
      const FBlock B = a.F.blocks[b];
      const int m = run_block<T, NT, kNAmp / (4 * NT)>(psi, B, blk[b], red, parity++, rank, init ? B.offset : -1);
      if (syn && rank == 0) syn[rnd * kNStab + b] = (uint8_t)(m ^ B.offset);
    }
  }
  if (init) {   // one warp
    double s = 0.0;
    for (int i = rank; i < kNAmp; i += NT) s += (double)psi[i].x * psi[i].x + (double)psi[i].y * psi[i].y;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const double sc = rsqrt(s);
    T2* out = reinterpret_cast<T2*>(a.init_out);
    for (int i = rank; i < kNAmp; i += NT) out[i] = make2<T2>(psi[i ^ flips].x * sc, psi[i ^ flips].y * sc);
    return;
  }
  finish<T, NT>(a, psi, flips, M, item, seed, traj, rank);
}

// Warps: the first trajectory of each by its place (warp 0 of every CTA, then warp 1, ...: few
// trajectories then spread over the SMs), the others from the counter.
__global__ void k_batch(const __grid_constant__ BatchArgs a) {
  extern __shared__ __align__(16) unsigned char bsm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* wsm = bsm + (size_t)warp * kWarpSmem;
  if (a.init_mode) {
    if (blockIdx.x == 0 && warp == 0) {
      if (a.init_prec == 0) run_group<double, 32>(a, wsm, nullptr, 0, lane);
      else run_group<float, 32>(a, wsm, nullptr, 0, lane);
    }
    return;
  }
  const uint32_t all = gridDim.x * (blockDim.x >> 5), n = a.ctl->n;
  for (uint32_t pos = (uint32_t)warp * gridDim.x + blockIdx.x; pos < n;) {
    const uint32_t item = a.idx[pos];
    if ((a.kind[item] & 1) == 0) run_group<double, 32>(a, wsm, nullptr, item, lane);
    else run_group<float, 32>(a, wsm, nullptr, item, lane);
    if (lane == 0) pos = all + atomicAdd(&a.ctl->counter, 1u);
    pos = __shfl_sync(0xffffffffu, pos, 0);
  }
}

// One trajectory per CTA of 128 threads.
__global__ void __launch_bounds__(128) k_batch_cta(const __grid_constant__ BatchArgs a) {
  extern __shared__ __align__(16) unsigned char bsm[];
  __shared__ double red[2 * 64];
  const uint32_t item = a.idx[blockIdx.x];
  if ((a.kind[item] & 1) == 0) run_group<double, 128>(a, bsm, red, item, (int)threadIdx.x);
  else run_group<float, 128>(a, bsm, red, item, (int)threadIdx.x);
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
template <typename T>
struct UMem {
  Mem<sizeof(T) == 8 ? 4 : 1> m;   // complex128: one CTA per SM, whose compile nothing else hides: four rounds together
  double norm[1 << kNAnc];
};
static_assert(sizeof(UMem<double>) % 16 == 0 && sizeof(UMem<float>) % 16 == 0, "16-byte aligned amplitudes");
template <typename T>
constexpr size_t u_smem() {
  return sizeof(UMem<T>) + sizeof(typename V2t<T>::t) * kUAmp + sizeof(Compiled<T>) * kNStab * decltype(UMem<T>::m)::kRounds;
}

// Rotations of data qubits j0 .. j0 + W - 1 of a block on 2^nb amplitudes in groups of 2^W; with `enter`,
// the block's ancilla enters at bit nb.  Two qubits a sweep are the faster choice (2048 complex128
// trajectories of 3 rounds: 3.58 ms, 3.96 with four): the early ancillas' slabs then fill the CTA.
template <typename T, int W>
__device__ void u_sweep(typename V2t<T>::t* slab, int nb, const FBlock& B, const Compiled<T>& C, int j0, bool enter) {
  using T2 = typename V2t<T>::t;
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

template <typename T, int NT>
__device__ void run_cta_u(const BatchArgs& a, unsigned char* sm, uint32_t item) {
  using T2 = typename V2t<T>::t;
  const int tid = threadIdx.x;
  const CtaGroup g{tid, NT};
  UMem<T>& U = *reinterpret_cast<UMem<T>*>(sm);
  T2* slab = reinterpret_cast<T2*>(sm + sizeof(UMem<T>));
  Compiled<T>* compiled = reinterpret_cast<Compiled<T>*>(sm + sizeof(UMem<T>) + sizeof(T2) * kUAmp);
  constexpr int NR = decltype(UMem<T>::m)::kRounds;
  const qec_noise nz = a.noise[item];
  const uint64_t traj = a.traj[item], seed = a.ctl->seed;
  trajectory_noise(g, nz, a.cr != 0, U.m);
  const T2* p0 = reinterpret_cast<const T2*>(a.psi0[sizeof(T) == 4]);
  for (int i = tid; i < kNAmp; i += NT) slab[i] = p0[i];
  uint8_t* syn = a.syn + (size_t)item * (a.rounds + 1) * kNStab;
  if (tid < kNStab) syn[tid] = 0;
  uint32_t flips = 0;
  for (int rnd = 1; rnd <= a.rounds; ++rnd) {
    const int k = (rnd - 1) % NR;
    if (k == 0) flips = compile_rounds<T>(g, a.F, U.m, compiled, seed, traj, rnd, min(NR, a.rounds + 1 - rnd), flips);
    const Compiled<T>* blk = compiled + k * kNStab;
    for (int part = 0; part < 2; ++part) {
      for (int j = 0; j < kNAnc; ++j) {
        const FBlock B = a.F.blocks[part * kNAnc + j];
        const Compiled<T>& C = blk[part * kNAnc + j];
        const int nb = kND + j;
        if (B.w == 2) {
          u_sweep<T, 2>(slab, nb, B, C, 0, true);
        } else if (a.width > 4) {
          u_sweep<T, 4>(slab, nb, B, C, 0, true);
        } else {
          if (C.form[0] | C.form[1]) u_sweep<T, 2>(slab, nb, B, C, 0, false);
          u_sweep<T, 2>(slab, nb, B, C, 2, true);
        }
      }
      // the 16 configurations' norms: 16 lanes each, the squares of a lane's amplitudes in the state's
      // precision, then FP64 (lane l of a configuration takes data indices l, l + 16, ...: the sums do
      // not depend on the CTA's size)
      for (int c = tid >> 4; c < (1 << kNAnc); c += NT >> 4) {
        T s = 0;
        for (int i = tid & 15; i < kNAmp; i += 16) {
          const T2 v = slab[c * kNAmp + i];
          s = fma(v.x, v.x, fma(v.y, v.y, s));
        }
        double w = (double)s;
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
      const T sc = norm_scale<T>(norm);
      if (m || rescale)
        for (int i = tid; i < kNAmp; i += NT) {
          T2 v = slab[m * kNAmp + i];
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
  finish<T, NT>(a, slab, flips, U.m, item, seed, traj, tid);
}

// One precision's trajectories (a launch of its own: a complex64 slab is half the size, so that two or
// three CTAs share an SM).  idx_u lists the complex128 items, then the complex64 ones.
template <typename T, int NT>
__global__ void __launch_bounds__(NT) k_batch_u(const __grid_constant__ BatchArgs a) {
  extern __shared__ __align__(16) unsigned char usm[];
  __shared__ uint32_t s_pos;
  constexpr int P = sizeof(T) == 4;
  const uint32_t n = a.ctl->n_u[P], base = P ? a.ctl->n_u[0] : 0u;
  for (;;) {
    if (threadIdx.x == 0) s_pos = atomicAdd(&a.ctl->counter_u[P], 1u);
    __syncthreads();
    const uint32_t pos = s_pos;
    __syncthreads();
    if (pos >= n) return;
    run_cta_u<T, NT>(a, usm, a.idx_u[base + pos]);
    __syncthreads();
  }
}

const void* u_kernel(int prec, int threads) {
  if (prec) return threads == 128 ? (const void*)k_batch_u<float, 128> : threads == 256 ? (const void*)k_batch_u<float, 256> : (const void*)k_batch_u<float, 512>;
  return threads == 128 ? (const void*)k_batch_u<double, 128> : threads == 256 ? (const void*)k_batch_u<double, 256> : (const void*)k_batch_u<double, 512>;
}
constexpr size_t u_smem_of(int prec) { return prec ? u_smem<float>() : u_smem<double>(); }

}  // namespace

struct qec_batch {
  int rounds = 0, gates = 0, num_sms = 0;
  uint32_t cap = 0;
  cudaStream_t work = nullptr;
  cudaStream_t user = nullptr;
  cudaEvent_t ev_in = nullptr, ev_out = nullptr, t0 = nullptr, t1 = nullptr;
  FactorProgram fac[2];              // [0] noisy program, every slot present; [1] init program
  unsigned char* d_fac[2] = {nullptr, nullptr};
  size_t fac_off[2][5] = {};
  void* d_psi0[2] = {nullptr, nullptr};
  uint32_t* d_idx = nullptr;
  uint32_t* d_idx_u = nullptr;
  std::vector<uint32_t> h_idx, h_idx_u;
  cudaStream_t side[2] = {nullptr, nullptr};   // the unreduced engine's launches, per precision
  cudaEvent_t fork = nullptr, join[2] = {nullptr, nullptr};
  int u_ctas_per_sm[2] = {1, 1};
  qec_noise* d_noise = nullptr;
  int32_t* d_kind = nullptr;
  uint64_t* d_traj = nullptr;
  BatchCtl* d_ctl = nullptr;
  BatchCtl* h_ctl = nullptr;   // pinned
  uint8_t* d_syn = nullptr;
  uint8_t* d_bits = nullptr;
  uint8_t* d_log = nullptr;
  int warps_per_cta = 8;
  int ctas_per_sm = 1;
  float last_ms = 0.f;
  double2* d_snap = nullptr;
  int64_t snap_item = -1;   // for the next run
  bool snap_valid = false;  // a completed run recorded a snapshot
  int fusion_k = 4;         // unreduced engine: slab bits a sweep may hold
  int u_threads = 256;      // unreduced engine: threads per CTA
};

namespace {

qec_status bfail(qec_status s, const std::string& m) {
  set_last_error(m);
  return s;
}

#define QEC_BCUDA(call)                                                                   \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess)                                                                \
      return bfail(e_ == cudaErrorMemoryAllocation ? QEC_ENOMEM : QEC_ECUDA,              \
                   std::string(#call) + ": " + cudaGetErrorString(e_));                   \
  } while (0)

void batch_free(qec_batch* b) {
  void* ptrs[] = {b->d_fac[0], b->d_fac[1], b->d_psi0[0], b->d_psi0[1], b->d_noise, b->d_kind, b->d_traj, b->d_ctl,
                  b->d_syn, b->d_bits, b->d_log, b->d_idx, b->d_idx_u, b->d_snap};
  for (void* p : ptrs) if (p) cudaFree(p);
  if (b->fork) cudaEventDestroy(b->fork);
  for (int i = 0; i < 2; ++i) {
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
  a.kind = b->d_kind;
  a.traj = b->d_traj;
  a.ctl = b->d_ctl;
  a.rounds = b->rounds;
  a.cr = b->gates == QEC_GATES_CR;
  a.width = b->fusion_k;
  a.psi0[0] = b->d_psi0[0];
  a.psi0[1] = b->d_psi0[1];
  a.idx = b->d_idx;
  a.idx_u = b->d_idx_u;
  a.syn = b->d_syn;
  a.bits = b->d_bits;
  a.logical = b->d_log;
  a.snap = b->d_snap;
  a.init_mode = 0;
  a.init_prec = 0;
  a.init_out = nullptr;
  return a;
}

size_t smem_for(int warps) { return (size_t)warps * kWarpSmem; }

// The run's launches: each engine that has trajectories, side by side (one CTA wave each at most, pulling
// trajectories from the control word's counters).
qec_status launch_batch(qec_batch* b, uint32_t n, uint32_t n_u128, uint32_t n_u64) {
  BatchArgs a = batch_args(b);
  const uint32_t n_u[2] = {n_u128, n_u64};
  bool busy = n > 0;   // something runs on the work stream itself
  if (n_u128 || n_u64) QEC_BCUDA(cudaEventRecord(b->fork, b->work));
  if (n > 0) {
    // up to four trajectories per SM: a CTA of four warps each (see above)
    if (n <= 4u * (uint32_t)b->num_sms) {
      k_batch_cta<<<n, 128, kGroupSmem, b->work>>>(a);
    } else {
      const uint32_t ctas = (n + b->warps_per_cta - 1) / b->warps_per_cta, wave = (uint32_t)(b->num_sms * b->ctas_per_sm);
      k_batch<<<ctas < wave ? ctas : wave, 32 * b->warps_per_cta, smem_for(b->warps_per_cta), b->work>>>(a);
    }
    QEC_BCUDA(cudaGetLastError());
  }
  for (int i = 0; i < 2; ++i) {
    if (!n_u[i]) continue;
    cudaStream_t s = busy ? b->side[i] : b->work;
    if (busy) QEC_BCUDA(cudaStreamWaitEvent(s, b->fork, 0));
    const uint32_t wave = (uint32_t)(b->num_sms * b->u_ctas_per_sm[i]);
    void* args[1] = {&a};
    QEC_BCUDA(cudaLaunchKernel(u_kernel(i, b->u_threads), dim3(n_u[i] < wave ? n_u[i] : wave), dim3((unsigned)b->u_threads),
                               args, u_smem_of(i), s));
    if (busy) {
      QEC_BCUDA(cudaEventRecord(b->join[i], s));
      QEC_BCUDA(cudaStreamWaitEvent(b->work, b->join[i], 0));
    }
    busy = true;
  }
  return QEC_OK;
}

// Time-ordered plan of one round of the unreduced register (qec_debug_unreduced_plan) for fusion width k: consecutive units whose slab bits
// are disjoint from those already in the pass (they commute with them) join it while the pass has at
// most k bits; a unit on a bit already in the pass, or a measurement, closes it.
// One-qubit units folded into two-qubit units: on each slab bit, a run of consecutive one-qubit units
// (nothing else on that bit between them) directly before a two-qubit unit on the bit goes into that
// unit's matrix from the right, a run directly after one from the left (between two, into the one
// whose second qubit is the bit).  Moving the run next to the unit is exact: the run acts on its bit alone, and nothing else
// acts on that bit in between.  absorbed[it] marks the folded units; pre/post list them per
// two-qubit unit in program order.
void plan_absorb(const UProgram& U, std::vector<char>& absorbed, std::vector<std::vector<UAbs>>& pre,
                 std::vector<std::vector<UAbs>>& post) {
  const int n = (int)U.items.size();
  absorbed.assign(n, 0);
  pre.assign(n, {});
  post.assign(n, {});
  auto is1 = [&](int it) { return U.items[it].kind == 0 && U.items[it].nq == 1; };
  auto is2 = [&](int it) { return U.items[it].kind == 0 && U.items[it].nq == 2; };
  for (int b = 0; b < U.nbits; ++b) {
    std::vector<int> seq;   // items acting on bit b, in order
    for (int it = 0; it < n; ++it) {
      const UItem& u = U.items[it];
      if (u.qa == b || (u.kind == 0 && u.nq == 2 && u.qb == b)) seq.push_back(it);
    }
    for (size_t i = 0; i < seq.size();) {
      if (!is1(seq[i])) { ++i; continue; }
      size_t j = i;
      while (j < seq.size() && is1(seq[j])) ++j;
      int target = -1;
      bool after = false;
      const bool next2 = j < seq.size() && is2(seq[j]), prev2 = i > 0 && is2(seq[i - 1]);
      // between two two-qubit units, the one in which b is the second qubit (the gate's target) takes
      // the run: a one-qubit matrix there keeps that unit block-diagonal in its first qubit
      if (next2 && (!prev2 || U.items[seq[j]].qb == b || U.items[seq[i - 1]].qb != b)) {
        target = seq[j];
      } else if (prev2) {
        target = seq[i - 1];
        after = true;
      }
      if (target >= 0) {
        const int bit = U.items[target].qa == b ? 2 : 0;
        for (size_t r = i; r < j; ++r) {
          absorbed[seq[r]] = 1;
          (after ? post : pre)[target].push_back({seq[r], bit | (after ? 1 : 0)});
        }
      }
      i = j;
    }
  }
}

void build_passes(const UProgram& U, int k, std::vector<UPass>& passes, std::vector<UPassUnit>& punits,
                  std::vector<UAbs>& uabs) {
  passes.clear();
  punits.clear();
  uabs.clear();
  std::vector<char> absorbed;
  std::vector<std::vector<UAbs>> pre, post;
  plan_absorb(U, absorbed, pre, post);
  UPass cur{};
  uint32_t mask = 0;
  auto close = [&]() {
    if (cur.u1 == cur.u0) return;
    cur.nbits = 0;
    for (int q = 0; q < 32; ++q)
      if (mask & (1u << q)) cur.bits[cur.nbits++] = q;
    for (int i = cur.u0; i < cur.u1; ++i) {
      UPassUnit& pu = punits[i];
      const uint32_t um = (1u << pu.qa) | (pu.nq == 2 ? (1u << pu.qb) : 0u);
      pu.nother = 0;
      for (int j = 0; j < cur.nbits; ++j)
        if (!(um & (1u << cur.bits[j]))) pu.other[pu.nother++] = cur.bits[j];
    }
    passes.push_back(cur);
  };
  auto open = [&]() {
    cur = UPass{};
    cur.kind = 0;
    cur.u0 = cur.u1 = (int32_t)punits.size();
    mask = 0;
  };
  open();
  for (int it = 0; it < (int)U.items.size(); ++it) {
    const UItem& u = U.items[it];
    if (u.kind == 1) {
      close();
      UPass m{};
      m.kind = 1;
      m.item = it;
      passes.push_back(m);
      open();
      continue;
    }
    if (absorbed[it]) continue;
    const uint32_t um = (1u << u.qa) | (u.nq == 2 ? (1u << u.qb) : 0u);
    if ((mask & um) || __builtin_popcount(mask | um) > k) {
      close();
      open();
    }
    UPassUnit pu{};
    pu.item = it;
    pu.nq = u.nq;
    pu.qa = u.qa;
    pu.qb = u.nq == 2 ? u.qb : 0;
    pu.abs0 = (int32_t)uabs.size();
    for (auto r = pre[it].rbegin(); r != pre[it].rend(); ++r) uabs.push_back(*r);   // right factors, latest first
    for (const UAbs& x : post[it]) uabs.push_back(x);                              // left factors, in order
    pu.nabs = (int32_t)uabs.size() - pu.abs0;
    punits.push_back(pu);
    cur.u1 = (int32_t)punits.size();
    mask |= um;
  }
  close();
}

// Sweep width (2..6 slab bits: with more than 4 a weight-4 block's four data qubits go in one sweep, with the
// ancilla that enters; else two at a time) and threads per CTA (128..512)
// of the unreduced engine.
qec_status set_fusion(qec_batch* b, int k, int threads) {
  if (k < 2 || k > kUMaxFusionDecl || (threads != 128 && threads != 256 && threads != 512))
    return bfail(QEC_EINVAL, "fusion width must be in [2, 6] and threads 128, 256 or 512");
  int occ[2] = {0, 0};
  for (int i = 0; i < 2; ++i) {
    QEC_BCUDA(cudaFuncSetAttribute(u_kernel(i, threads), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)u_smem_of(i)));
    QEC_BCUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[i], u_kernel(i, threads), threads, u_smem_of(i)));
    if (occ[i] < 1) return bfail(QEC_EUNSUPPORTED, "unreduced batched kernel does not fit an SM with this shape");
  }
  b->fusion_k = k;
  b->u_threads = threads;
  b->u_ctas_per_sm[0] = occ[0];
  b->u_ctas_per_sm[1] = occ[1];
  return QEC_OK;
}

qec_status set_shape(qec_batch* b, int warps) {
  QEC_BCUDA(cudaFuncSetAttribute(k_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_for(warps)));
  int occ = 0;
  QEC_BCUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_batch, 32 * warps, smem_for(warps)));
  if (occ < 1) return bfail(QEC_EUNSUPPORTED, "batched kernel does not fit an SM with this shape");
  b->warps_per_cta = warps;
  b->ctas_per_sm = occ;
  return QEC_OK;
}

}  // namespace

extern "C" {

qec_status qec_debug_unreduced_plan(int32_t gates, int32_t k, int32_t* items, uint32_t cap, uint32_t* n_items,
                                    int32_t* pass_units, uint32_t* n_pass_units, int32_t* absorbs, uint32_t* n_absorbs) {
  if (!items || !n_items || !pass_units || !n_pass_units || !absorbs || !n_absorbs)
    return bfail(QEC_EINVAL, "null argument");
  if (k < 2 || k > kUMaxFusionDecl) return bfail(QEC_EINVAL, "fusion width must be in [2, 6]");
  try {
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
  } catch (...) {
    return bfail(QEC_ENOMEM, "host allocation failed");
  }
}

qec_status qec_batch_create(int32_t d, int32_t rounds, int32_t gates, uint32_t max_traj, void* cuda_stream,
                            qec_batch** out) {
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
  auto bail = [&](qec_status s) { batch_free(b); delete b; return s; };
  b->rounds = rounds;
  b->gates = gates;
  b->cap = max_traj;
  b->user = static_cast<cudaStream_t>(cuda_stream);
  for (int w = 0; w < 2; ++w) {
    Program P;
    if (!build_program(p, w == 0, P, err, w == 0) || !build_factor(P, b->fac[w], err)) return bail(bfail(QEC_EINVAL, err));
    if (b->fac[w].sites.size() > (size_t)kSites)
      return bail(bfail(QEC_EUNSUPPORTED, "a round has more draws than the engine's table"));
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
  for (int i = 0; i < 2; ++i) {
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->side[i], cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->join[i], cudaEventDisableTiming);
  }
  if (e != cudaSuccess) return bail(bfail(QEC_ECUDA, std::string("CUDA setup: ") + cudaGetErrorString(e)));
  const size_t syn_bytes = (size_t)max_traj * (rounds + 1) * kNStab;
  const void* src[2][5];
  size_t bytes[2][5], total[2];
  for (int w = 0; w < 2; ++w) {
    const FactorProgram& F = b->fac[w];
    const void* s[5] = {F.sites.data(), F.items.data(), F.touches.data(), F.blocks.data(), F.order.data()};
    const size_t n[5] = {sizeof(FSite) * F.sites.size(), sizeof(FItem) * F.items.size(), sizeof(FTouch) * F.touches.size(),
                         sizeof(FBlock) * F.blocks.size(), sizeof(uint16_t) * F.order.size()};
    total[w] = 0;
    for (int i = 0; i < 5; ++i) {
      src[w][i] = s[i];
      bytes[w][i] = n[i];
      b->fac_off[w][i] = total[w];
      total[w] += (n[i] + 255) / 256 * 256;
    }
  }
  void** allocs[] = {(void**)&b->d_fac[0], (void**)&b->d_fac[1], &b->d_psi0[0], &b->d_psi0[1], (void**)&b->d_noise,
                     (void**)&b->d_kind, (void**)&b->d_traj, (void**)&b->d_ctl, (void**)&b->d_syn, (void**)&b->d_bits,
                     (void**)&b->d_log, (void**)&b->d_idx, (void**)&b->d_idx_u, (void**)&b->d_snap};
  const size_t sizes[] = {total[0], total[1], (size_t)kNAmp * 16, (size_t)kNAmp * 8, sizeof(qec_noise) * max_traj,
                          sizeof(int32_t) * max_traj, sizeof(uint64_t) * max_traj, sizeof(BatchCtl), syn_bytes,
                          (size_t)max_traj * kND, (size_t)max_traj, sizeof(uint32_t) * max_traj,
                          sizeof(uint32_t) * max_traj, sizeof(double2) * kNAmp};
  for (size_t i = 0; i < sizeof(sizes) / sizeof(sizes[0]); ++i) {
    e = cudaMalloc(allocs[i], sizes[i]);
    if (e != cudaSuccess) return bail(bfail(QEC_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e)));
  }
  for (int w = 0; w < 2; ++w)
    for (int i = 0; i < 5 && e == cudaSuccess; ++i)
      if (bytes[w][i])
        e = cudaMemcpy(b->d_fac[w] + b->fac_off[w][i], src[w][i], bytes[w][i], cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return bail(bfail(QEC_ECUDA, std::string("upload: ") + cudaGetErrorString(e)));
  e = cudaMallocHost((void**)&b->h_ctl, sizeof(BatchCtl));
  if (e != cudaSuccess) return bail(bfail(QEC_ENOMEM, "pinned allocation failed"));
  std::memset(b->h_ctl, 0, sizeof(BatchCtl));
  e = cudaMemcpy(b->d_ctl, b->h_ctl, sizeof(BatchCtl), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return bail(bfail(QEC_ECUDA, cudaGetErrorString(e)));
  qec_status st = set_shape(b, 10);
  if (st) return bail(st);
  if ((st = set_fusion(b, 4, 256))) return bail(st);
  for (int prec = 0; prec < 2; ++prec) {   // the noise-free init round, once per precision
    BatchArgs a = batch_args(b);
    a.F = batch_program(b, 1);
    a.init_mode = 1;
    a.init_prec = prec;
    a.init_out = b->d_psi0[prec];
    k_batch<<<1, 32, smem_for(1), b->work>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return bail(bfail(QEC_ECUDA, std::string("init round: ") + cudaGetErrorString(e)));
  }
  e = cudaStreamSynchronize(b->work);
  if (e != cudaSuccess) return bail(bfail(QEC_ECUDA, std::string("init round: ") + cudaGetErrorString(e)));
  *out = b;
  return QEC_OK;
}

qec_status qec_batch_run(qec_batch* b, uint64_t seed, uint32_t n, const uint64_t* traj, const int32_t* kind,
                         const qec_noise* noise, uint8_t* syndromes, uint8_t* data_bits, uint8_t* raw_logical) {
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
  QEC_BCUDA(cudaMemcpyAsync(b->d_kind, kind, sizeof(int32_t) * n, cudaMemcpyHostToDevice, b->work));
  QEC_BCUDA(cudaMemcpyAsync(b->d_noise, noise, sizeof(qec_noise) * n, cudaMemcpyHostToDevice, b->work));
  b->h_idx.clear();
  b->h_idx_u.clear();
  // each engine's items complex128 first, then complex64: the warps (CTAs) then run one precision's
  // code at a time instead of interleaving both instantiations, and the longer items start first.
  // Every trajectory's result is independent of the order.
  uint32_t n_u128 = 0;
  for (int prec = 0; prec < 2; ++prec) {
    for (uint32_t i = 0; i < n; ++i)
      if ((kind[i] & 1) == prec) ((kind[i] & 2) ? b->h_idx_u : b->h_idx).push_back(i);
    if (prec == 0) n_u128 = (uint32_t)b->h_idx_u.size();
  }
  if (!b->h_idx.empty())
    QEC_BCUDA(cudaMemcpyAsync(b->d_idx, b->h_idx.data(), sizeof(uint32_t) * b->h_idx.size(), cudaMemcpyHostToDevice, b->work));
  if (!b->h_idx_u.empty())
    QEC_BCUDA(cudaMemcpyAsync(b->d_idx_u, b->h_idx_u.data(), sizeof(uint32_t) * b->h_idx_u.size(),
                              cudaMemcpyHostToDevice, b->work));
  QEC_BCUDA(cudaStreamSynchronize(b->work));   // h_ctl is reused
  b->h_ctl->seed = seed;
  b->h_ctl->n = (uint32_t)b->h_idx.size();
  b->h_ctl->counter = 0;
  b->h_ctl->n_u[0] = n_u128;
  b->h_ctl->n_u[1] = (uint32_t)b->h_idx_u.size() - n_u128;
  b->h_ctl->counter_u[0] = b->h_ctl->counter_u[1] = 0;
  const bool snap = b->snap_item >= 0 && b->snap_item < (int64_t)n;
  b->h_ctl->snap_item = snap ? (uint32_t)b->snap_item : ~0u;
  b->snap_valid = false;
  QEC_BCUDA(cudaMemcpyAsync(b->d_ctl, b->h_ctl, sizeof(BatchCtl), cudaMemcpyHostToDevice, b->work));
  QEC_BCUDA(cudaEventRecord(b->t0, b->work));
  qec_status st = launch_batch(b, b->h_ctl->n, b->h_ctl->n_u[0], b->h_ctl->n_u[1]);
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
}

qec_status qec_batch_autotune(qec_batch* b, uint64_t seed, uint32_t n, const uint64_t* traj, const int32_t* kind,
                              const qec_noise* noise, int32_t* chosen_warps, float* best_ms) {
  if (!b || !chosen_warps || !best_ms || !traj || !kind || !noise) return bfail(QEC_EINVAL, "null argument");
  // the sample split by register: each engine is tuned on its own trajectories
  std::vector<uint64_t> tr[2];
  std::vector<int32_t> kd[2];
  std::vector<qec_noise> nz[2];
  for (uint32_t i = 0; i < n; ++i) {
    const int u = (kind[i] & 2) ? 1 : 0;
    tr[u].push_back(traj[i]);
    kd[u].push_back(kind[i]);
    nz[u].push_back(noise[i]);
  }
  auto time_run = [&](int u, float& t) -> qec_status {
    t = 1e30f;
    if (tr[u].empty()) return QEC_OK;
    for (int rep = 0; rep < 2; ++rep) {   // first run warms up
      qec_status st = qec_batch_run(b, seed, (uint32_t)tr[u].size(), tr[u].data(), kd[u].data(), nz[u].data(),
                                    nullptr, nullptr, nullptr);
      if (st) return st;
      if (rep) t = b->last_ms;
    }
    return QEC_OK;
  };
  // reduced register: warps per CTA
  const int cand[] = {2, 4, 6, 8, 10};
  int best = -1;
  float best_t = 0.f;
  for (int w : cand) {
    if (set_shape(b, w) != QEC_OK) continue;
    float t;
    qec_status st = time_run(0, t);
    if (st) return st;
    if (best < 0 || t < best_t) {
      best = w;
      best_t = t;
    }
  }
  if (best < 0) return bfail(QEC_EUNSUPPORTED, "no batched kernel shape fits");
  qec_status st = set_shape(b, best);
  if (st) return st;
  // unreduced register: sweep width (slab bits) x threads per CTA
  int bk = -1, bthr = 256;
  float bu = 0.f;
  for (int k : {4, 6})
    for (int thr : {128, 256}) {
      if (set_fusion(b, k, thr) != QEC_OK) continue;
      float t;
      if ((st = time_run(1, t))) return st;
      if (bk < 0 || t < bu) {
        bk = k;
        bthr = thr;
        bu = t;
      }
    }
  if (bk < 0) return bfail(QEC_EUNSUPPORTED, "no unreduced engine shape fits");
  if ((st = set_fusion(b, bk, bthr))) return st;
  float t_all = 0.f;   // the whole sample with the chosen configuration
  for (int rep = 0; rep < 2; ++rep) {
    if ((st = qec_batch_run(b, seed, n, traj, kind, noise, nullptr, nullptr, nullptr))) return st;
    t_all = b->last_ms;
  }
  *chosen_warps = best;
  *best_ms = t_all;
  return QEC_OK;
}

qec_status qec_batch_config(const qec_batch* b, int32_t* warps_per_cta, int32_t* fusion_width, int32_t* u_threads) {
  if (!b || !warps_per_cta || !fusion_width || !u_threads) return bfail(QEC_EINVAL, "null argument");
  *warps_per_cta = b->warps_per_cta;
  *fusion_width = b->fusion_k;
  *u_threads = b->u_threads;
  return QEC_OK;
}

qec_status qec_batch_set_config(qec_batch* b, int32_t warps_per_cta, int32_t fusion_width, int32_t u_threads) {
  if (!b) return bfail(QEC_EINVAL, "null handle");
  qec_status st = set_shape(b, warps_per_cta);
  if (st) return st;
  return set_fusion(b, fusion_width, u_threads);
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
