// complex64 engines of the batched form, in one order of evaluation.
//
// An FP32 amplitude carries the rounding of the order that computed it, and probabilities come from FP64
// sums over the FP32 squares, so complex64 trajectories keep dense blocks (reduced register) and gate
// units in time order (unreduced register) where the complex128 ones run in factored form (batch.cu; the same
// in FP32 is 2 to 8 times as fast, but its states differ by up to 7e-7 and its weights were FP32 sums).
// A trajectory's result depends on its inputs alone: not on the other trajectories of a run, nor on warps
// per CTA, threads or fusion width.
//
// What bounds them: reduced register, latency (a chain of small products per block, then FP64 sums and
// conversions); unreduced, the FP64 fusing of the units at a round's start, then the slab's sweeps.  2048
// trajectories of 3 rounds: 1.26 and 5.2 ms.  (2.2 and 10.0 with a block's draws one after the other, units of
// identity matrices multiplied out, one CTA per SM; factored in FP32 0.61 and 1.17.)
#include <cuda_runtime.h>

#include <algorithm>

#include "batch_dense.hpp"
#include "common.cuh"
#include "factor.cuh"
#include "onchip.cuh"

namespace qec {
namespace {

constexpr int kD = 3;                    // register of the batched form: d = 3
constexpr int kND = kD * kD;             // 9 data qubits
constexpr int kNAmp = 1 << kND;          // 512 amplitudes
constexpr int kNStab = kND - 1;          // 8 stabilizers

__device__ __forceinline__ float2 mk(double re, double im) { return make_float2((float)re, (float)im); }

__device__ __forceinline__ float2 cmul_add(float2 acc, float2 a, float2 b) {
  acc.x = fmaf(a.x, b.x, acc.x);
  acc.x = fmaf(-a.y, b.y, acc.x);
  acc.y = fmaf(a.x, b.y, acc.y);
  acc.y = fmaf(a.y, b.x, acc.y);
  return acc;
}

// What a trajectory's noise input makes of the program: draw thresholds and matrices (the conventions of
// the program builder; twirled coherent terms are draws, their unitaries the identity).
struct Noise {
  float2 mats[M_COUNT][16];
  uint64_t thr[PR_COUNT];
  double cs[8][2];
  uint32_t identity;     // bit id: matrix id is the identity
};

template <class G>
__device__ void trajectory_noise(const G& g, const Batch64Args& a, const qec_noise& nz, bool init, Noise& N) {
  for (int i = g.rank; i < M_COUNT * 16; i += g.size) N.mats[i >> 4][i & 15] = mk(a.mats[2 * i], a.mats[2 * i + 1]);
  const bool tw = nz.twirl != 0.0;
  const double th[6] = {nz.theta_rx, nz.theta_rz, nz.theta_rzx, 2.0 * nz.phi_zz, nz.round_rz, nz.round_rx};
  if (g.rank < 6) {   // half angles (of phi itself for the ZZ term)
    const double h = 0.5 * th[g.rank];
    N.cs[g.rank][0] = cos(h);
    N.cs[g.rank][1] = sin(h);
  }
  g.sync();
  if (g.rank < PR_COUNT) {
    const int l = g.rank;
    const double s = l < 3 ? 0.0 : N.cs[l - 3][1];
    const double p = l == PR_P1 ? nz.p1 : l == PR_P2 ? nz.p2 : l == PR_IDLE ? nz.p_idle : tw ? s * s : 0.0;
    N.thr[l] = fac::draw_threshold(p);
  }
  // the coherent matrices: a row of zeros and one or two entries
  if (g.rank == 31) {
    uint32_t id = 1u << M_I;
    const int of[7] = {M_ROT_RX, M_ROT_RXP, M_ROT_RZ, M_ROT_RZX, M_ZZ, M_ROUND_RZ, M_ROUND_RX}, from[7] = {0, 0, 1, 2, 3, 4, 5};
    for (int i = 0; i < 7 && !init; ++i)
      if (tw || th[from[i]] == 0.0) id |= 1u << of[i];
    N.identity = id;
  }
  if (!init && g.rank < 7) {
    const int of[7] = {M_ROT_RX, M_ROT_RXP, M_ROT_RZ, M_ROT_RZX, M_ZZ, M_ROUND_RZ, M_ROUND_RX}, from[7] = {0, 0, 1, 2, 3, 4, 5};
    const int id = of[g.rank];
    const double c = tw ? 1.0 : N.cs[from[g.rank]][0];
    double s = tw ? 0.0 : N.cs[from[g.rank]][1];
    if (id == M_ROT_RXP && nz.overrot_follows != 0.0) s = -s;
    float2* m = N.mats[id];
    for (int i = 0; i < 16; ++i) m[i] = mk(0, 0);
    if (id == M_ROT_RX || id == M_ROT_RXP || id == M_ROUND_RX) {
      m[0] = m[5] = mk(c, 0);
      m[1] = m[4] = mk(0, -s);
    } else if (id == M_ROT_RZ || id == M_ROUND_RZ) {
      m[0] = mk(c, -s);
      m[5] = mk(c, s);
    } else if (id == M_ROT_RZX) {
      for (int r = 0; r < 4; ++r) {
        m[5 * r] = mk(c, 0);
        m[4 * r + (r ^ 1)] = mk(0, r >> 1 ? s : -s);
      }
    } else {
      for (int r = 0; r < 4; ++r) m[5 * r] = mk(c, (r >> 1) ^ (r & 1) ? s : -s);
    }
  }
  g.sync();
}

// The draw of an op (noise_code, or 1 for a twirled term that fires; 0: it does nothing); the thresholds decide as
// uniform53(w) < p does.
__device__ __forceinline__ int draw_op(const ProgOp& op, const uint64_t* thr, uint64_t seed, uint64_t traj, uint64_t rnd) {
  const bool twirl = op.kind == OP_T1 || op.kind == OP_T2;
  if (!twirl && op.kind != OP_N1 && op.kind != OP_N2) return 0;
  const uint64_t t = thr[op.pidx];
  if (t == 0) return 0;
  const U64x4 w = draw(seed, traj, rnd, op.step, op.site, twirl ? TAG_TWIRL : TAG_NOISE);
  if ((w.v[0] >> 11) >= t) return 0;
  return twirl ? 1 : (int)(((w.v[1] >> 32) * (op.kind == OP_N1 ? 3ull : 15ull)) >> 32) + 1;
}

// Final readout (Sec. III.B), bits, raw logical and the recorded state.
template <int NT>
__device__ void finish(const Batch64Args& a, const float2* psi, double* heap, double* ur, uint32_t* bits, uint32_t item,
                       uint64_t traj, int rank) {
  const oc::Group<NT> g{rank};
  if (rank < kND) ur[rank] = uniform53(draw(a.seed, traj, (uint64_t)a.rounds + 1, 0u, (uint32_t)rank, TAG_READOUT).v[0]);
  if (item == a.snap_item)
    for (int i = rank; i < kNAmp; i += NT) a.snap[i] = make_double2((double)psi[i].x, (double)psi[i].y);
  oc::readout<float, NT>(psi, kND, 0u, heap, ur, bits, rank);
  const uint32_t x = *bits;
  if (rank < kND) a.bits[(size_t)item * kND + rank] = (uint8_t)((x >> rank) & 1u);
  if (rank == 0) a.logical[item] = (uint8_t)(__popc(x & ((1u << kD) - 1u)) & 1);
  g.sync();
}

// ---- reduced register: one warp per trajectory -----------------------------------------------------------
__device__ void apply1_w(float2* U, int w, int b, const float2* m, int lane) {
  const int C = 1 << w;
  for (int it = lane; it < C * C; it += 32) {
    const int c = it & (C - 1), pr = it >> w;
    const int r0 = (int)ins0(pr, b), r1 = r0 | (1 << b);
    const float2 x = U[r0 * 16 + c], y = U[r1 * 16 + c];
    float2 o0 = mk(0, 0), o1 = mk(0, 0);
    o0 = cmul_add(o0, m[0], x);
    o0 = cmul_add(o0, m[1], y);
    o1 = cmul_add(o1, m[4], x);
    o1 = cmul_add(o1, m[5], y);
    U[r0 * 16 + c] = o0;
    U[r1 * 16 + c] = o1;
  }
  __syncwarp();
}

__device__ void apply2_w(float2* U, int w, int a, int b, const float2* m, int lane) {
  const int C = 1 << w;
  const int lo = a < b ? a : b, hi = a < b ? b : a;
  for (int it = lane; it < (C / 2) * C; it += 32) {
    const int c = it & (C - 1), qd = it >> w;
    const int base = (int)ins0(ins0(qd, lo), hi);
    int idx[4];
    float2 x[4];
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      idx[l] = base | ((l >> 1) << a) | ((l & 1) << b);
      x[l] = U[idx[l] * 16 + c];
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float2 acc = mk(0, 0);
#pragma unroll
      for (int k = 0; k < 4; ++k) acc = cmul_add(acc, m[4 * r + k], x[k]);
      U[idx[r] * 16 + c] = acc;
    }
  }
  __syncwarp();
}

// Ancilla measurement of one block on the warp's register: A = sum |K1 v|^2, N = sum |v|^2
// (FP64 accumulated), outcome u < A / N (forced to the offset in the init round), then
// v <- K_m v / sqrt(N) in place.  Returns the raw outcome.
template <int W>
__device__ int measure_block(float2* psi, const float2* U, const BlockInfo& bi, bool init, double u, int lane) {
  constexpr int C = 1 << W, G = kNAmp >> W;
  int q[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) q[j] = j < W ? bi.q[j] : 0;
  uint32_t off[C];
#pragma unroll
  for (int l = 0; l < C; ++l) {
    uint32_t o = 0;
#pragma unroll
    for (int j = 0; j < W; ++j) o |= (uint32_t)((l >> j) & 1) << q[j];
    off[l] = o;
  }
  auto base_of = [&](int g) {
    uint32_t base = g;
#pragma unroll
    for (int j = 0; j < W; ++j) base = (uint32_t)ins0(base, q[j]);
    return base;
  };
  double A = 0.0, N = 0.0;
  for (int g = lane; g < G; g += 32) {
    const uint32_t base = base_of(g);
    float2 v[C];
#pragma unroll
    for (int l = 0; l < C; ++l) {
      v[l] = psi[base + off[l]];
      N += (double)v[l].x * v[l].x + (double)v[l].y * v[l].y;
    }
#pragma unroll
    for (int r = 0; r < C; ++r) {
      float2 acc = mk(0, 0);
#pragma unroll
      for (int c = 0; c < C; ++c) acc = cmul_add(acc, U[(C + r) * 16 + c], v[c]);
      A += (double)acc.x * acc.x + (double)acc.y * acc.y;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    A += __shfl_xor_sync(0xffffffffu, A, o);
    N += __shfl_xor_sync(0xffffffffu, N, o);
  }
  const int m = init ? bi.offset : u < A / N ? 1 : 0;
  const double scale = 1.0 / sqrt(N);
  for (int g = lane; g < G; g += 32) {
    const uint32_t base = base_of(g);
    float2 v[C];
#pragma unroll
    for (int l = 0; l < C; ++l) v[l] = psi[base + off[l]];
#pragma unroll
    for (int r = 0; r < C; ++r) {
      float2 acc = mk(0, 0);
#pragma unroll
      for (int c = 0; c < C; ++c) acc = cmul_add(acc, U[(m * C + r) * 16 + c], v[c]);
      psi[base + off[r]] = mk((double)acc.x * scale, (double)acc.y * scale);
    }
  }
  __syncwarp();
  return m;
}

// A block's compile folds consecutive ops on the same qubits into one pending factor before it
// touches the 32 x 16 block matrix U: a 2x2 on one qubit (pb < 0; entries 0, 1, 4, 5 of P) or a 4x4
// on a qubit pair (local index 2 bit(pa) + bit(pb)).  An op on other qubits first applies the
// pending factor to U.  The product is the same operator as the ops applied one at a time.
struct PendingOp {
  float2* P;    // [16], the warp's pending factor
  int pa = -1, pb = -1;
  int lane;
  static __device__ __forceinline__ int sw(int i) { return ((i & 1) << 1) | (i >> 1); }
  // P <- G P for a 4x4 G (qubit order of G swapped against P's when swap)
  __device__ void lmul2(const float2* g, bool swap) {
    float2 acc = mk(0, 0);
    if (lane < 16) {
      const int r = lane >> 2, c = lane & 3;
#pragma unroll
      for (int k = 0; k < 4; ++k) acc = cmul_add(acc, g[4 * (swap ? sw(r) : r) + (swap ? sw(k) : k)], P[4 * k + c]);
    }
    __syncwarp();
    if (lane < 16) P[lane] = acc;
    __syncwarp();
  }
  // P <- (g on local bit) P for a 2x2 g (entries 0, 1, 4, 5), P a 4x4 (dim 4) or a 2x2 (dim 2)
  __device__ void lmul1(const float2* g, int bit, int dim) {
    float2 acc = mk(0, 0);
    const int r = lane >> 2, c = lane & 3;
    const bool on = dim == 4 ? lane < 16 : (r < 2 && c < 2);
    if (on) {
      const int rb = (r >> bit) & 1, r0 = r & ~(1 << bit), r1 = r | (1 << bit);
      acc = cmul_add(acc, g[4 * rb], P[4 * r0 + c]);
      acc = cmul_add(acc, g[4 * rb + 1], P[4 * r1 + c]);
    }
    __syncwarp();
    if (on) P[lane] = acc;
    __syncwarp();
  }
  __device__ void flush(float2* U, int w) {
    if (pa < 0) return;
    if (pb < 0) apply1_w(U, w, pa, P, lane);
    else apply2_w(U, w, pa, pb, P, lane);
    pa = pb = -1;
  }
  __device__ void start(const float2* g, int x, int y) {   // P <- g (a 4x4 on (x, y), or a 2x2 on x when y < 0)
    if (lane < 16) P[lane] = g[lane];
    __syncwarp();
    pa = x;
    pb = y;
  }
  __device__ void one(float2* U, int w, int x, const float2* g) {
    if (pa == x && pb < 0) {
      lmul1(g, 0, 2);
    } else if (pb >= 0 && (x == pa || x == pb)) {
      lmul1(g, x == pa ? 1 : 0, 4);
    } else {
      flush(U, w);
      start(g, x, -1);
    }
  }
  __device__ void two(float2* U, int w, int x, int y, const float2* g) {
    if (pb >= 0 && ((x == pa && y == pb) || (x == pb && y == pa))) {
      lmul2(g, x != pa);
      return;
    }
    if (pb < 0 && pa >= 0 && (x == pa || y == pa)) {
      // the pending one-qubit factor becomes a 4x4 on (x, y): Q on its bit, the identity on the other
      const int bit = x == pa ? 1 : 0;
      const float2 q00 = P[0], q01 = P[1], q10 = P[4], q11 = P[5];
      __syncwarp();
      if (lane < 16) {
        const int r = lane >> 2, c = lane & 3;
        const int ob = 1 - bit;
        float2 v = mk(0, 0);
        if (((r >> ob) & 1) == ((c >> ob) & 1)) {
          const int rb = (r >> bit) & 1, cb = (c >> bit) & 1;
          v = rb ? (cb ? q11 : q10) : (cb ? q01 : q00);
        }
        P[lane] = v;
      }
      __syncwarp();
      pa = x;
      pb = y;
      lmul2(g, false);
      return;
    }
    flush(U, w);
    start(g, x, y);
  }
};

// Shared memory of a warp's trajectory.
struct alignas(16) WarpMem {
  float2 U[32 * 16];     // the block's matrix; at the end the readout's tree
  float2 psi[kNAmp];
  Noise noise;
  float2 pend[16];
  double ur[kND];
  uint32_t bits;
  uint8_t code[kBatchOps];
};
static_assert(sizeof(float2) * 32 * 16 >= sizeof(double) * kNAmp, "layout of a warp's memory");

// One trajectory (or the noise-free init round) on one warp.
__device__ void run_warp(const Batch64Args& a, WarpMem& M, uint32_t item) {
  const int lane = threadIdx.x & 31;
  const oc::Group<32> g{lane};
  const bool init = a.noise == nullptr;
  PendingOp pend;
  pend.P = M.pend;
  pend.lane = lane;
  const qec_noise nz = init ? qec_noise{} : a.noise[item];
  const uint64_t traj = init ? 0ull : a.traj[item];
  trajectory_noise(g, a, nz, init, M.noise);
  for (int i = lane; i < kNAmp; i += 32) M.psi[i] = init ? mk(i == 0 ? 1.0 : 0.0, 0.0) : reinterpret_cast<const float2*>(a.psi0)[i];
  uint8_t* syn = init ? nullptr : a.syn + (size_t)item * (a.rounds + 1) * kNStab;
  if (syn && lane < kNStab) syn[lane] = 0;
  const int r_first = init ? 0 : 1, r_last = init ? 0 : a.rounds;
  for (int rnd = r_first; rnd <= r_last; ++rnd) {
    for (int i = lane; i < a.n_ops; i += 32) M.code[i] = (uint8_t)draw_op(a.ops[i], M.noise.thr, a.seed, traj, (uint64_t)rnd);
    __syncwarp();
    for (int k = 0; k < kNStab; ++k) {
      const BlockInfo bi = a.blocks[k];
      const int w = bi.w, C = 1 << w;
      for (int i = lane; i < 32 * 16; i += 32) M.U[i] = mk((i / 16 < C && i / 16 == i % 16) ? 1.0 : 0.0, 0.0);
      __syncwarp();
      for (int oi = bi.op_begin; oi < bi.op_end; ++oi) {
        const ProgOp op = a.ops[oi];
        const int code = M.code[oi];
        if (op.kind == OP_U1 || op.kind == OP_T1) {
          if (op.kind == OP_U1 || code) pend.one(M.U, w, op.q0, M.noise.mats[op.mat]);
        } else if (op.kind == OP_U2 || op.kind == OP_T2) {
          if (op.kind == OP_U2 || code) pend.two(M.U, w, op.q0, op.q1, M.noise.mats[op.mat]);
        } else if (code) {
          if (op.kind == OP_N1) {
            pend.one(M.U, w, op.q0, M.noise.mats[code]);
          } else {
            if (code >> 2) pend.one(M.U, w, op.q0, M.noise.mats[code >> 2]);
            if (code & 3) pend.one(M.U, w, op.q1, M.noise.mats[code & 3]);
          }
        }
      }
      pend.flush(M.U, w);
      const double u = init ? 0.0 : uniform53(draw(a.seed, traj, (uint64_t)rnd, 0u, (uint32_t)(kND + k), TAG_MEASURE).v[0]);
      const int m = w == 4 ? measure_block<4>(M.psi, M.U, bi, init, u, lane) : measure_block<2>(M.psi, M.U, bi, init, u, lane);
      if (syn && lane == 0) syn[rnd * kNStab + k] = (uint8_t)(m ^ bi.offset);
    }
    __syncwarp();   // the codes are read
  }
  if (init) {
    for (int i = lane; i < kNAmp; i += 32) a.out[i] = M.psi[i];
    return;
  }
  finish<32>(a, M.psi, reinterpret_cast<double*>(M.U), M.ur, &M.bits, item, traj, lane);
}

// The first trajectory of a warp by its place (warp 0 of every CTA, then warp 1, ...), the others from the counter.
__global__ void k_batch64(const __grid_constant__ Batch64Args a) {
  extern __shared__ __align__(16) unsigned char bsm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  WarpMem& M = reinterpret_cast<WarpMem*>(bsm)[warp];
  if (a.noise == nullptr) {
    if (blockIdx.x == 0 && warp == 0) run_warp(a, M, 0);
    return;
  }
  const uint32_t all = gridDim.x * (blockDim.x >> 5);
  for (uint32_t pos = (uint32_t)warp * gridDim.x + blockIdx.x; pos < a.n;) {
    run_warp(a, M, a.idx[pos]);
    if (lane == 0) pos = all + atomicAdd(a.counter, 1u);
    pos = __shfl_sync(0xffffffffu, pos, 0);
  }
}

// ---- unreduced register: one CTA per 17-qubit trajectory --------------------------------
// Each round's gate units (a gate with its coherent terms and sampled Paulis on 1 or 2 slab bits)
// are fused into their matrices at the start of the round, one thread per unit: the noise draws
// depend only on (seed, trajectory, round, step, site), not on the state.  The slab is then
// updated in passes: a pass holds consecutive units on disjoint slab bits (which commute), at most
// `fusion width` bits in all, and each thread applies every unit of the pass to whole groups of
// amplitudes (all combinations of the pass's bits) that it alone touches, so a pass needs one
// barrier however many units it holds.  Measurements are passes of their own.
constexpr int kUChunks = 256;                 // measurement: chunks of the 4096 amplitude pairs

// Left-multiplies the DIM x DIM unit matrix M (row stride 4) by a one-qubit gate g on local bit BIT.
template <int DIM, int BIT, typename T2>
__device__ __forceinline__ void left1(double2 (&M)[16], const T2* g) {
  const double2 g00 = make_double2((double)g[0].x, (double)g[0].y), g01 = make_double2((double)g[1].x, (double)g[1].y);
  const double2 g10 = make_double2((double)g[4].x, (double)g[4].y), g11 = make_double2((double)g[5].x, (double)g[5].y);
#pragma unroll
  for (int r0 = 0; r0 < DIM; ++r0) {
    if (r0 & (1 << BIT)) continue;
    const int r1 = r0 | (1 << BIT);
#pragma unroll
    for (int c = 0; c < DIM; ++c) {
      const double2 x = M[r0 * 4 + c], y = M[r1 * 4 + c];
      M[r0 * 4 + c] = make_double2(g00.x * x.x - g00.y * x.y + g01.x * y.x - g01.y * y.y,
                                   g00.x * x.y + g00.y * x.x + g01.x * y.y + g01.y * y.x);
      M[r1 * 4 + c] = make_double2(g10.x * x.x - g10.y * x.y + g11.x * y.x - g11.y * y.y,
                                   g10.x * x.y + g10.y * x.x + g11.x * y.y + g11.y * y.x);
    }
  }
}

// Left-multiplies the 4x4 unit matrix M by a two-qubit gate g (local index 2 bit(qa) + bit(qb)).
__device__ __forceinline__ void left2(double2 (&M)[16], const float2* g) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    double2 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = M[k * 4 + c];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      double re = 0.0, im = 0.0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (g[r * 4 + k].x == 0.f && g[r * 4 + k].y == 0.f) continue;   // (half of a gate's entries, or more)
        const double gx = (double)g[r * 4 + k].x, gy = (double)g[r * 4 + k].y;
        re += gx * v[k].x - gy * v[k].y;
        im += gx * v[k].y + gy * v[k].x;
      }
      M[r * 4 + c] = make_double2(re, im);
    }
  }
}

// Right-multiplies the 4x4 unit matrix M (row stride 4) by a one-qubit gate g on local bit BIT:
// M <- M (g on BIT), the gate applied before M.
template <int BIT>
__device__ __forceinline__ void right1(double2 (&M)[16], const double2* g) {
  const double2 g00 = g[0], g01 = g[1], g10 = g[4], g11 = g[5];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
#pragma unroll
    for (int c0 = 0; c0 < 4; ++c0) {
      if (c0 & (1 << BIT)) continue;
      const int c1 = c0 | (1 << BIT);
      const double2 x = M[r * 4 + c0], y = M[r * 4 + c1];
      M[r * 4 + c0] = make_double2(x.x * g00.x - x.y * g00.y + y.x * g10.x - y.y * g10.y,
                                   x.x * g00.y + x.y * g00.x + y.x * g10.y + y.y * g10.x);
      M[r * 4 + c1] = make_double2(x.x * g01.x - x.y * g01.y + y.x * g11.x - y.y * g11.y,
                                   x.x * g01.y + x.y * g01.x + y.x * g11.y + y.y * g11.x);
    }
  }
}

// The fused matrix of one unit: the product, in op order, of its gate, coherent terms and the
// Paulis its noise sites draw (DIM 2 or 4; local index 2 bit(qa) + bit(qb), qa the only bit of a
// one-qubit unit), built in place by left multiplications.  Returns 0 when no op of the unit acts
// (every draw came up empty, every angle is 0 and no gate): the unit is then the identity.
template <int DIM>
__device__ int fuse_unit(const UItem& u, const ProgOp* ops, const Noise& N, uint64_t seed, uint64_t traj, int rnd, double2* F) {
  double2 M[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) M[i] = make_double2((i / 4 == i % 4) ? 1.0 : 0.0, 0.0);
  int any = 0;
  auto one = [&](int id, bool on_qa) {   // one-qubit matrix id on qa (local bit 1) or qb (bit 0)
    if ((N.identity >> id) & 1u) return;
    if (DIM == 2) left1<DIM, 0>(M, N.mats[id]);
    else if (on_qa) left1<DIM, 1>(M, N.mats[id]);
    else left1<DIM, 0>(M, N.mats[id]);
  };
  for (int oi = u.op_begin; oi < u.op_end; ++oi) {
    const ProgOp op = ops[oi];
    int code = 0;
    if (op.kind != OP_U1 && op.kind != OP_U2 && !(code = draw_op(op, N.thr, seed, traj, (uint64_t)rnd))) continue;
    if ((op.kind == OP_U1 || op.kind == OP_U2) && ((N.identity >> op.mat) & 1u)) continue;   // an angle of 0
    any = 1;
    if (DIM == 4 && (op.kind == OP_U2 || op.kind == OP_T2)) {
      left2(M, N.mats[op.mat]);
    } else if (op.kind == OP_N2) {   // Pauli code >> 2 on op.q0, code & 3 on op.q1
      one(code >> 2, op.q0 == u.qa);
      one(code & 3, op.q1 == u.qa);
    } else {
      one((op.kind == OP_U1 || op.kind == OP_T1) ? op.mat : code, op.q0 == u.qa);
    }
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) F[i] = M[i];
  return any;
}

// Offset of pass-local combination s over the `n` slab bits in b[] (bit j of s -> slab bit b[j]).
__device__ __forceinline__ int deposit_bits(int s, const int* b, int n) {
  int o = 0;
  for (int j = 0; j < n; ++j) o |= ((s >> j) & 1) << b[j];
  return o;
}

// Slab index of group g of a pass: g's bits spread over the slab bits outside the pass
// (insert a zero at each pass bit, ascending).
__device__ __forceinline__ int group_base_u(int g, const int* bits, int nbits) {
  for (int j = 0; j < nbits; ++j) g = ((g >> bits[j]) << (bits[j] + 1)) | (g & ((1 << bits[j]) - 1));
  return g;
}

// Shared memory of a CTA's trajectory: slab, this, then [items][16] unit matrices and their shapes.
struct alignas(16) UMem64 {
  Noise noise;
  double csum[2][kUChunks];
  double ur[kND + 1];
  uint32_t bits[4];
};
constexpr size_t u_smem(int items) {
  return sizeof(float2) * kSlabAmps + sizeof(UMem64) + (size_t)items * (16 * sizeof(double2) + sizeof(int)) + 16;
}

// One trajectory (or the noise-free init round) of the unreduced register on one CTA.
template <int NT>
__device__ void run_cta_u(const Batch64Args& a, unsigned char* sm, uint32_t item) {
  const int tid = threadIdx.x;
  const oc::Group<NT> g{tid};
  float2* slab = reinterpret_cast<float2*>(sm);
  UMem64& M = *reinterpret_cast<UMem64*>(sm + sizeof(float2) * kSlabAmps);
  double2* Ft = reinterpret_cast<double2*>(sm + sizeof(float2) * kSlabAmps + sizeof(UMem64));   // [items][16]
  int* Fon = reinterpret_cast<int*>(Ft + a.n_uitems * 16);                                      // [items]
  const bool init = a.noise == nullptr;
  const qec_noise nz = init ? qec_noise{} : a.noise[item];
  const uint64_t traj = init ? 0ull : a.traj[item], seed = a.seed;
  trajectory_noise(g, a, nz, init, M.noise);
  for (int i = tid; i < kSlabAmps; i += NT) slab[i] = init ? mk(i == 0 ? 1.0 : 0.0, 0.0) : reinterpret_cast<const float2*>(a.psi0)[i];
  __syncthreads();
  uint8_t* syn = init ? nullptr : a.syn + (size_t)item * (a.rounds + 1) * kNStab;
  if (syn && tid < kNStab) syn[tid] = 0;
  const int r_first = init ? 0 : 1, r_last = init ? 0 : a.rounds;
  for (int rnd = r_first; rnd <= r_last; ++rnd) {
    // every unit of the round, one thread each
    for (int it = tid; it < a.n_uitems; it += NT) {
      const UItem u = a.uitems[it];
      Fon[it] = u.kind != 0 ? 0
                : u.nq == 1 ? fuse_unit<2>(u, a.uops, M.noise, seed, traj, rnd, Ft + 16 * it)
                            : fuse_unit<4>(u, a.uops, M.noise, seed, traj, rnd, Ft + 16 * it);
    }
    __syncthreads();
    // the one-qubit units next to a two-qubit unit on the same qubit, folded into its matrix (one
    // thread per two-qubit unit; each one-qubit unit belongs to at most one); the passes skip them.
    // Then the unit's shape, from exact zeros: Fon = 2 when the matrix is block-diagonal in its first
    // qubit (local bit 1: the two-qubit gates act on the second qubit conditioned on the first), 3
    // when block-antidiagonal (an X or Y drawn on the first qubit), else 1 (dense).
    for (int pu = tid; pu < a.n_upunits; pu += NT) {
      const UPassUnit U = a.upunits[pu];
      if (U.nq != 2) continue;
      double2 m[16];
      double2* F = Ft + 16 * U.item;
#pragma unroll
      for (int i = 0; i < 16; ++i) m[i] = F[i];
      for (int e = U.abs0; e < U.abs0 + U.nabs; ++e) {
        const UAbs A = a.uabs[e];
        if (!Fon[A.item1]) continue;   // the identity
        const double2* h = Ft + 16 * A.item1;
        if (A.mode & 1) {
          if (A.mode & 2) left1<4, 1>(m, h);
          else left1<4, 0>(m, h);
        } else {
          if (A.mode & 2) right1<1>(m, h);
          else right1<0>(m, h);
        }
      }
      bool bd = true, ad = true;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        F[i] = m[i];
        const bool z = m[i].x == 0.0 && m[i].y == 0.0;
        if (((i >> 3) & 1) != ((i >> 1) & 1)) bd = bd && z;   // row bit 1 != column bit 1
        else ad = ad && z;
      }
      if (Fon[U.item]) Fon[U.item] = bd ? 2 : ad ? 3 : 1;
    }
    __syncthreads();
    // each unit's matrix converted once, in place (the first half of its slot)
    for (int it = tid; it < a.n_uitems; it += NT) {
      if (!Fon[it]) continue;
      double2 v[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = Ft[16 * it + i];
      float2* o = reinterpret_cast<float2*>(Ft + 16 * it);
#pragma unroll
      for (int i = 0; i < 16; ++i) o[i] = mk(v[i].x, v[i].y);
    }
    __syncthreads();
    for (int pi = 0; pi < a.n_upasses; ++pi) {
      const UPass P = a.upasses[pi];
      if (P.kind == 1) {
        // measurement of the ancilla at slab bit u.qa: Born rule, collapse, renormalise, reset.  The squares are
        // summed in FP32 over fixed chunks (chunk c: pairs c, c + 256, ..., 16 of them), the chunk sums in
        // FP64 in a fixed order by one warp, so that the sums do not depend on the CTA size
        const UItem u = a.uitems[P.item];
        const int b = u.qa;
        for (int c = tid; c < kUChunks; c += NT) {
          float f0 = 0.f, f1 = 0.f;
          for (int pr = c; pr < kSlabAmps / 2; pr += kUChunks) {
            const int i0 = (int)ins0(pr, b), i1 = i0 | (1 << b);
            f0 = fmaf(slab[i0].x, slab[i0].x, fmaf(slab[i0].y, slab[i0].y, f0));
            f1 = fmaf(slab[i1].x, slab[i1].x, fmaf(slab[i1].y, slab[i1].y, f1));
          }
          M.csum[0][c] = (double)f0;
          M.csum[1][c] = (double)f1;
        }
        __syncthreads();
        if (tid < 32) {
          double a0 = 0.0, a1 = 0.0;
          for (int c = tid; c < kUChunks; c += 32) {
            a0 += M.csum[0][c];
            a1 += M.csum[1][c];
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            a0 += __shfl_xor_sync(0xffffffffu, a0, o);
            a1 += __shfl_xor_sync(0xffffffffu, a1, o);
          }
          if (tid == 0) {
            M.csum[0][0] = a0;
            M.csum[1][0] = a1;
          }
        }
        __syncthreads();
        const double s0 = M.csum[0][0], s1 = M.csum[1][0];
        int m = u.offset;
        if (!init) {
          const double uu = uniform53(draw(seed, traj, (uint64_t)rnd, 0u, (uint32_t)(kND + u.stab), TAG_MEASURE).v[0]);
          m = uu < s1 / (s0 + s1) ? 1 : 0;
        }
        const float sc = (float)(1.0 / sqrt(m ? s1 : s0));   // in FP64, applied in the state's precision
        for (int pr = tid; pr < kSlabAmps / 2; pr += NT) {
          const int i0 = (int)ins0(pr, b), i1 = i0 | (1 << b);
          const float2 kept = m ? slab[i1] : slab[i0];
          slab[i0] = make_float2(kept.x * sc, kept.y * sc);
          slab[i1] = mk(0, 0);
        }
        __syncthreads();
        if (syn && tid == 0) syn[rnd * kNStab + u.stab] = (uint8_t)(m ^ u.offset);
        continue;
      }
      // apply: thread-local groups over the pass's bits, every unit of the pass in turn
      const int G = kSlabAmps >> P.nbits;
      for (int pu = P.u0; pu < P.u1; ++pu) {
        const UPassUnit U = a.upunits[pu];
        const int shape = Fon[U.item];
        if (!shape) continue;
        const float2* Fg = reinterpret_cast<const float2*>(Ft + 16 * U.item);
        const int nsub = 1 << U.nother;
        if (U.nq == 1) {
          const float2 f0 = Fg[0], f1 = Fg[1], f4 = Fg[4], f5 = Fg[5];
          for (int gr = tid; gr < G; gr += NT) {
            const int base = group_base_u(gr, P.bits, P.nbits);
            for (int sub = 0; sub < nsub; ++sub) {
              const int i0 = base | deposit_bits(sub, U.other, U.nother), i1 = i0 | (1 << U.qa);
              const float2 x = slab[i0], y = slab[i1];
              float2 o0 = mk(0, 0), o1 = mk(0, 0);
              o0 = cmul_add(o0, f0, x);
              o0 = cmul_add(o0, f1, y);
              o1 = cmul_add(o1, f4, x);
              o1 = cmul_add(o1, f5, y);
              slab[i0] = o0;
              slab[i1] = o1;
            }
          }
          continue;
        }
        float2 f[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) f[i] = Fg[i];
        // block-(anti)diagonal in the first qubit: rows 0, 1 from one column pair, rows 2, 3 from the
        // other (the nonzero terms of the dense sum, in the same order); selects keep every index a constant
        const bool bd = shape == 2;
        float2 h[8];   // row r, term j: f[r][c(r) + j]
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int j = 0; j < 2; ++j) h[2 * r + j] = ((r < 2) == bd) ? f[r * 4 + j] : f[r * 4 + 2 + j];
        for (int gr = tid; gr < G; gr += NT) {
          const int base = group_base_u(gr, P.bits, P.nbits);
          for (int sub = 0; sub < nsub; ++sub) {
            const int b0 = base | deposit_bits(sub, U.other, U.nother);
            int idx[4];
            float2 x[4];
#pragma unroll
            for (int l = 0; l < 4; ++l) {
              idx[l] = b0 | ((l >> 1) << U.qa) | ((l & 1) << U.qb);
              x[l] = slab[idx[l]];
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              float2 acc = mk(0, 0);
              if (shape != 1) {
                const bool low = (r < 2) == bd;   // this row reads columns 0, 1
                acc = cmul_add(acc, h[2 * r], low ? x[0] : x[2]);
                acc = cmul_add(acc, h[2 * r + 1], low ? x[1] : x[3]);
              } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) acc = cmul_add(acc, f[r * 4 + k], x[k]);
              }
              slab[idx[r]] = acc;
            }
          }
        }
      }
      __syncthreads();
    }
  }
  if (init) {
    for (int i = tid; i < kSlabAmps; i += NT) a.out[i] = slab[i];
    return;
  }
  // the data qubits with every ancilla |0>: slab entries 0..511; the tree takes the ancillas' part
  finish<NT>(a, slab, reinterpret_cast<double*>(slab + kNAmp), M.ur, M.bits, item, traj, tid);
}

template <int NT>
__global__ void __launch_bounds__(NT, NT > 256 ? 1 : 2) k_batch64_u(const __grid_constant__ Batch64Args a) {
  extern __shared__ __align__(16) unsigned char usm[];
  __shared__ uint32_t s_pos;
  if (a.noise == nullptr) {
    if (blockIdx.x == 0) run_cta_u<NT>(a, usm, 0);
    return;
  }
  for (;;) {
    if (threadIdx.x == 0) s_pos = atomicAdd(a.counter, 1u);
    __syncthreads();
    const uint32_t pos = s_pos;
    __syncthreads();
    if (pos >= a.n) return;
    run_cta_u<NT>(a, usm, a.idx[pos]);
    __syncthreads();
  }
}

const void* u_kernel(int threads) {
  return threads == 128 ? (const void*)k_batch64_u<128> : threads == 256 ? (const void*)k_batch64_u<256> : (const void*)k_batch64_u<512>;
}

}  // namespace

// (Function attributes are the process's, not a handle's: always the ceiling, so that handles of different shapes coexist.)
// All engines ask for the largest shared-memory carveout: launches that run side by side then fit the same SMs (150
// trajectories beside 151 complex128 ones otherwise pile up on the few SMs that those leave: 5 rounds 2.05 ms, 0.86 so).
constexpr int kSmemCeiling = 226 * 1024;
static cudaError_t set_attributes(const void* fn) {
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCeiling);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
}

cudaError_t setup_batch64(int warps, int* occ) {
  const size_t smem = sizeof(WarpMem) * (size_t)warps;
  *occ = 0;
  const cudaError_t e = set_attributes((const void*)k_batch64);
  return e != cudaSuccess ? e : cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k_batch64, 32 * warps, smem);
}

cudaError_t launch_batch64(const Batch64Args& a, int warps, int ctas, cudaStream_t s) {
  k_batch64<<<ctas, 32 * warps, sizeof(WarpMem) * (size_t)warps, s>>>(a);
  return cudaGetLastError();
}

cudaError_t setup_batch64_u(int threads, int items, int* occ) {
  *occ = 0;
  const cudaError_t e = set_attributes(u_kernel(threads));
  return e != cudaSuccess ? e : cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, u_kernel(threads), threads, u_smem(items));
}

cudaError_t launch_batch64_u(const Batch64Args& a, int threads, int items, int ctas, cudaStream_t s) {
  Batch64Args b = a;
  void* args[1] = {&b};
  return cudaLaunchKernel(u_kernel(threads), dim3((unsigned)ctas), dim3((unsigned)threads), args, u_smem(items), s);
}

// ---- the unreduced register's plan -------------------------------------------------------------------
// One-qubit units folded into two-qubit units: on each slab bit, a run of consecutive one-qubit units
// (nothing else on that bit between them) directly before a two-qubit unit on the bit goes into that
// unit's matrix from the right, a run directly after one from the left (between two, into the one
// whose second qubit is the bit).  Moving the run next to the unit is exact: the run acts on its bit alone, and nothing else
// acts on that bit in between.  absorbed[it] marks the folded units; pre/post list them per
// two-qubit unit in program order.
static void plan_absorb(const UProgram& U, std::vector<char>& absorbed, std::vector<std::vector<UAbs>>& pre,
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

}  // namespace qec
