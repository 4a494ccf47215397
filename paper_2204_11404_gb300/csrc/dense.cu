// complex64 trajectories of registers of up to 13 data qubits, whole on chip, in dense blocks.
//
// An FP32 amplitude carries the rounding of the order that computed it.  So complex64 keeps one order
// of evaluation on these registers, whose states are read and compared: a block is its dense Kraus pair
// (built in FP64, rounded to FP32 once), an amplitude one row of K_m / sqrt(N) times its group, 4
// multiply-adds per entry in column order, the sums of squares FP32 over the groups of one of 256 places
// and FP64 over those.  (In factored form, factor.hpp, the same block has fewer multiply-adds and
// rounds differently: states then differ by up to 8e-7.)  The guess, the decision and the corrective apply are those of
// the passes over HBM (rounds.cu): the outcome of the same stabilizer one round earlier is applied, and
// the other one, from the untouched input, where the draw says so.
//
// Two launches: the Kraus pairs of all blocks (one CTA each: they depend on the draws only, and their FP64
// arithmetic wants every SM), then one CTA per trajectory with the register in shared memory.
//
// What bounds it: the pairs the FP64 pipe (13 to 17 us of an SM for a block of the d = 3 code), the
// trajectories a chain per block (3 us: K scaled, applied, the sums' FP64 tree, 1 / sqrt(N)).  d = 3, 7
// rounds, 37 trajectories with reconfigure: 0.44 ms (0.2 in factored form; a graph of passes per trajectory,
// the same arithmetic, 34).
#include <cuda_runtime.h>

#include "common.cuh"
#include "dense.hpp"
#include "onchip.cuh"

namespace qec {
namespace {

// ---- Kraus pairs -------------------------------------------------------------------------------------
// U (the block's unitary on inputs with the ancilla in |0>) grows op by op as in inst_block (kernels.cu): the same
// products and sums in FP64, without those that an entry's zero real or imaginary part makes zero.  A
// column sees no other column, so eight lanes carry one and meet at warp barriers only.
// kind of a matrix entry: bit 0 a real part, bit 1 an imaginary one.
constexpr int kCol = 33;   // column stride of U: eight lanes' rows in different banks

__device__ __forceinline__ double2 first_term(const double* m, int kind, double2 x) {
  if (kind == 1) return make_double2(__dmul_rn(m[0], x.x), __dmul_rn(m[0], x.y));
  if (kind == 2) return make_double2(-__dmul_rn(m[1], x.y), __dmul_rn(m[1], x.x));
  return make_double2(m[0] * x.x - m[1] * x.y, m[0] * x.y + m[1] * x.x);
}

// m (a row's two entries, x's and y's) times (x, y).
__device__ __forceinline__ double2 row2(const double (*m)[2], const uint8_t* kind, double2 x, double2 y) {
  double2 o = make_double2(0.0, 0.0);
  if (kind[0]) o = first_term(m[0], kind[0], x);
  if (kind[1] & 1) {
    o.x = __fma_rn(m[1][0], y.x, o.x);
    o.y = __fma_rn(m[1][0], y.y, o.y);
  }
  if (kind[1] & 2) {
    o.x = __fma_rn(-m[1][1], y.y, o.x);
    o.y = __fma_rn(m[1][1], y.x, o.y);
  }
  return o;
}

__global__ void __launch_bounds__(128) k_dense_compile(const __grid_constant__ DenseArgs a) {
  __shared__ double2 U[16 * kCol];
  __shared__ double sm[M_COUNT][16][2];
  __shared__ uint8_t kind[M_COUNT][16];
  __shared__ ProgOp ops[kDenseOps];
  __shared__ uint8_t code[kDenseOps];
  const int tid = threadIdx.x, blk = blockIdx.x, k = blk % a.nstab, rnd = 1 + blk / a.nstab;
  const uint64_t traj = a.first + blockIdx.y;
  const BlockInfo bi = a.blocks[k];
  const int w = bi.w, C = 1 << w, nops = bi.op_end - bi.op_begin;
  for (int i = tid; i < M_COUNT * 16; i += 128) {
    const double re = a.mats[2 * i], im = a.mats[2 * i + 1];
    sm[i >> 4][i & 15][0] = re;
    sm[i >> 4][i & 15][1] = im;
    kind[i >> 4][i & 15] = (uint8_t)((re != 0.0 ? 1 : 0) | (im != 0.0 ? 2 : 0));
  }
  for (int i = tid; i < 16 * kCol; i += 128) U[i] = make_double2(i / kCol == i % kCol ? 1.0 : 0.0, 0.0);
  if (tid < nops) {
    const ProgOp op = a.ops[bi.op_begin + tid];
    int c = 0;
    if (op.kind == OP_T1 || op.kind == OP_T2) {
      c = twirl_fires(op, a.prob[op.pidx], a.seed, traj, (uint64_t)rnd) ? 1 : 0;
    } else if (op.kind == OP_N1 || op.kind == OP_N2) {
      c = noise_code(op, a.prob[op.pidx], a.seed, traj, (uint64_t)rnd);
      if (c && a.events) {
        const unsigned e = atomicAdd(&a.ctl->n_events, 1u);
        if (e < a.ctl->ev_cap) {
          int32_t* ev = a.events + 5 * (size_t)e;
          ev[0] = (int32_t)traj; ev[1] = rnd; ev[2] = op.step; ev[3] = (int32_t)op.site; ev[4] = c;
        }
      }
    }
    ops[tid] = op;
    code[tid] = (uint8_t)c;
  }
  __syncthreads();
  const int col = tid >> 3, lane8 = tid & 7;
  double2* V = U + col * kCol;
  auto one = [&](int id, int b) {   // a one-qubit matrix on local bit b
    if (col < C)
      for (int p = lane8; p < C; p += 8) {
        const int r0 = (int)ins0(p, b), r1 = r0 | (1 << b);
        const double2 x = V[r0], y = V[r1];
        V[r0] = row2(&sm[id][0], &kind[id][0], x, y);
        V[r1] = row2(&sm[id][4], &kind[id][4], x, y);
      }
    __syncwarp();
  };
  auto two = [&](int id, int qa, int qb) {   // a two-qubit matrix on local index 2 bit(qa) + bit(qb)
    const int lo = min(qa, qb), hi = max(qa, qb);
    if (col < C && lane8 < C / 2) {
      const int base = (int)ins0(ins0(lane8, lo), hi);
      double2 x[4];
#pragma unroll
      for (int l = 0; l < 4; ++l) x[l] = V[base | ((l >> 1) << qa) | ((l & 1) << qb)];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        double2 s = make_double2(0.0, 0.0);
        bool any = false;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int kd = kind[id][4 * r + c];
          if (!kd) continue;
          const double2 t = first_term(sm[id][4 * r + c], kd, x[c]);
          s = any ? make_double2(__dadd_rn(s.x, t.x), __dadd_rn(s.y, t.y)) : t;
          any = true;
        }
        V[base | ((r >> 1) << qa) | ((r & 1) << qb)] = s;
      }
    }
    __syncwarp();
  };
  for (int i = 0; i < nops; ++i) {
    const ProgOp op = ops[i];
    const int c = code[i];
    if (op.kind == OP_U1 || op.kind == OP_T1) {
      if (op.kind == OP_U1 || c) one(op.mat, op.q0);
    } else if (op.kind == OP_U2 || op.kind == OP_T2) {
      if (op.kind == OP_U2 || c) two(op.mat, op.q0, op.q1);
    } else if (c) {
      if (op.kind == OP_N1) {
        one(c, op.q0);
      } else {
        if (c >> 2) one(c >> 2, op.q0);
        if (c & 3) one(c & 3, op.q1);
      }
    }
  }
  const size_t at = (size_t)blockIdx.y * gridDim.x + blk;
  float2* out = a.kraus + at * 2 * a.entries;
  if (col < C)
    for (int r = lane8; r < 2 * C; r += 8) {   // row r of K_(r / C)
      const double2 v = V[r];
      out[(r >> w) * a.entries + (r & (C - 1)) * C + col] = make_float2((float)v.x, (float)v.y);
    }
  if (tid == 0) a.u[at] = uniform53(draw(a.seed, traj, (uint64_t)rnd, 0u, (uint32_t)(a.nd + k), TAG_MEASURE).v[0]);
}

// ---- trajectories --------------------------------------------------------------------------------------
template <int D> struct DenseShape { static constexpr int NT = D == 9 ? 128 : D == 11 ? 256 : 512; };

template <int D>
__global__ void __launch_bounds__(DenseShape<D>::NT) k_dense_run(const __grid_constant__ DenseArgs a) {
  constexpr int NT = DenseShape<D>::NT, NW = NT / 32, AMPS = 1 << D;
  constexpr int KE = D == 9 ? 256 : 16, KN = (KE + NT - 1) / NT;   // weight-4 blocks at 9 qubits only
  extern __shared__ __align__(16) unsigned char dsm[];
  float2* const psi = reinterpret_cast<float2*>(dsm);   // two registers: a block reads one, writes the other
  __shared__ __align__(16) float2 sK[KE];
  __shared__ double red[2][16];
  __shared__ double ur[D], s_scale, s_inv[2];   // 1 / sqrt(N) and 1 / N of a block's input
  __shared__ BlockInfo info[D - 1];
  __shared__ uint8_t out[65 * (D - 1)];
  __shared__ int s_m;
  __shared__ uint32_t s_bits;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nstab = a.nstab, blocks = a.rounds * nstab;
  const int syn_len = (a.rounds + 1) * nstab;
  if (tid < nstab) info[tid] = a.blocks[tid];
  for (uint32_t t = blockIdx.x; t < a.n; t += gridDim.x) {
    const float2* K = a.kraus + (size_t)t * blocks * 2 * a.entries;
    const double* u = a.u + (size_t)t * blocks;
    for (int i = tid; i < AMPS; i += NT) psi[i] = reinterpret_cast<const float2*>(a.psi0)[i];
    for (int i = tid; i < nstab; i += NT) out[i] = 0;
    if (tid < D) ur[tid] = uniform53(draw(a.seed, a.first + t, (uint64_t)a.rounds + 1, 0u, (uint32_t)tid, TAG_READOUT).v[0]);
    if (tid == 0) s_scale = s_inv[0] = 1.0;
    __syncthreads();
    unsigned misses = 0;
    int cur = 0;
    float2 mine[KN], next[KN];   // this thread's entries of the block's matrix and of the next one's guess
    double u_next = 0.0;
    auto fetch = [&](float2 (&to)[KN], int b, int m) {
#pragma unroll
      for (int i = 0; i < KN; ++i) {
        const int e = tid + NT * i;
        to[i] = e < a.entries ? K[((size_t)b * 2 + m) * a.entries + e] : make_float2(0.f, 0.f);
      }
    };
    if (blocks) {
      fetch(next, 0, info[0].offset);
      u_next = u[0];
    }
    for (int b = 0; b < blocks; ++b) {
      const BlockInfo& bi = info[b % nstab];
      const int g = out[b] ^ bi.offset;
      const double u_b = u_next;
#pragma unroll
      for (int i = 0; i < KN; ++i) mine[i] = next[i];
      if (b + 1 < blocks) {   // (a stabilizer's outcome of the round before: there since an earlier barrier)
        fetch(next, b + 1, out[b + 1] ^ info[(b + 1) % nstab].offset);
        u_next = u[b + 1];
      }
      const float2* src = psi + cur * AMPS;
      float2* dst = psi + (cur ^ 1) * AMPS;
      // K_m (in `mine`) / sqrt(N) from src to dst; the first lanes of warps 0 and 1 get the sums of squares of both
      auto apply = [&](double& sI, double& sO) {
        const double scale = s_scale;
#pragma unroll
        for (int i = 0; i < KN; ++i) {
          const int e = tid + NT * i;
          if (e < a.entries) sK[e] = make_float2((float)((double)mine[i].x * scale), (float)((double)mine[i].y * scale));
        }
        __syncthreads();
        double nI = 0.0, nO = 0.0;
        if (KE == 256 && bi.w == 4) {
          // 32 groups of 16: a warp takes four rows of each; then warp 0 and 1 sum the squares a group to a lane
          const uint32_t o1 = 1u << bi.q[0], o2 = 1u << bi.q[1], o4 = 1u << bi.q[2], o8 = 1u << bi.q[3];
          uint32_t base = (uint32_t)lane;
#pragma unroll
          for (int j = 0; j < 4; ++j) base = (uint32_t)ins0(base, bi.q[j]);
          float2 v[16];
#pragma unroll
          for (int l = 0; l < 16; ++l)
            v[l] = src[base | (l & 1 ? o1 : 0u) | (l & 2 ? o2 : 0u) | (l & 4 ? o4 : 0u) | (l & 8 ? o8 : 0u)];
          const uint32_t rows = base | (warp & 1 ? o4 : 0u) | (warp & 2 ? o8 : 0u);
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const float4* kr = reinterpret_cast<const float4*>(sK + (4 * warp + r) * 16);
            float sr = 0.f, si = 0.f;
#pragma unroll
            for (int c = 0; c < 16; c += 2) {
              const float4 kk = kr[c >> 1];
              sr = fmaf(kk.x, v[c].x, sr);
              sr = fmaf(-kk.y, v[c].y, sr);
              si = fmaf(kk.x, v[c].y, si);
              si = fmaf(kk.y, v[c].x, si);
              sr = fmaf(kk.z, v[c + 1].x, sr);
              sr = fmaf(-kk.w, v[c + 1].y, sr);
              si = fmaf(kk.z, v[c + 1].y, si);
              si = fmaf(kk.w, v[c + 1].x, si);
            }
            dst[rows | (r & 1 ? o1 : 0u) | (r & 2 ? o2 : 0u)] = make_float2(sr, si);
          }
          __syncthreads();
          if (warp < 2) {
            float s = 0.f;
#pragma unroll
            for (int l = 0; l < 16; ++l) {
              const float2 y = warp ? v[l] : dst[base | (l & 1 ? o1 : 0u) | (l & 2 ? o2 : 0u) | (l & 4 ? o4 : 0u) | (l & 8 ? o8 : 0u)];
              s = fmaf(y.x, y.x, fmaf(y.y, y.y, s));
            }
            if (warp) nI = (double)s;
            else nO = (double)s;
          }
        } else {
          // groups of 4, 256 places; at 13 qubits two tiles of 2^12, one after the other in the sums: without
          // qubit 12, or without qubit 10 where the block has qubit 12
          constexpr int PER = AMPS / 4 / NT;
          const int cut = D == 13 && bi.q[1] == 12 ? 10 : 12;
          const uint32_t place = (uint32_t)tid & 255u;
          float tI = 0.f, tO = 0.f;
#pragma unroll
          for (int j = 0; j < PER; ++j) {
            uint32_t x = place + 256u * j;
            if (D == 13) {
              // the group's bits beside the block's, tile bit (cut) put in at its place among them
              const int at = cut - (bi.q[0] < cut) - (bi.q[1] < cut);
              x = (uint32_t)ins0(x, at) | ((uint32_t)(tid >> 8) << at);
            }
            x = (uint32_t)ins0(ins0(x, bi.q[0]), bi.q[1]);
            float2 v[4];
#pragma unroll
            for (int l = 0; l < 4; ++l) {
              v[l] = src[x | ((l & 1) << bi.q[0]) | ((l >> 1) << bi.q[1])];
              tI = fmaf(v[l].x, v[l].x, fmaf(v[l].y, v[l].y, tI));
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              float sr = 0.f, si = 0.f;
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                const float2 kk = sK[4 * r + c];
                sr = fmaf(kk.x, v[c].x, sr);
                sr = fmaf(-kk.y, v[c].y, sr);
                si = fmaf(kk.x, v[c].y, si);
                si = fmaf(kk.y, v[c].x, si);
              }
              dst[x | ((r & 1) << bi.q[0]) | ((r >> 1) << bi.q[1])] = make_float2(sr, si);
              tO = fmaf(sr, sr, fmaf(si, si, tO));
            }
          }
          nI = (double)tI;
          nO = (double)tO;
        }
        // both sums in one tree: lanes 0..15 fold the inputs', 16..31 the outputs'
        double v2 = lane & 16 ? nO : nI;
        v2 += __shfl_xor_sync(0xffffffffu, lane & 16 ? nI : nO, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v2 += __shfl_xor_sync(0xffffffffu, v2, o);
        if ((lane & 15) == 0) red[lane >> 4][warp] = v2;
        __syncthreads();
        if (warp < 2) {   // eight warps of a tile, then the tiles
          double s = (lane & 15) < NW ? red[lane >> 4][lane & 15] : 0.0;
          s += __shfl_xor_sync(0xffffffffu, s, 4);
          s += __shfl_xor_sync(0xffffffffu, s, 2);
          s += __shfl_xor_sync(0xffffffffu, s, 1);
          s += __shfl_xor_sync(0xffffffffu, s, 8);
          sI = s;
          sO = __shfl_sync(0xffffffffu, s, 16);
        }
      };
      double sI = 0.0, sO = 0.0;
      apply(sI, sO);
      if (tid == 0) {
        const double Np = sI * s_inv[b & 1], A1 = g ? sO : Np - sO;   // |input|^2 and P(1) of it, the input's scale taken out
        const int m = u_b * Np < A1 ? 1 : 0;
        s_m = m;
        out[b + nstab] = (uint8_t)(m ^ bi.offset);
        if (m == g) s_scale = 1.0 / sqrt(sO);
      } else if (tid == 32) {
        s_inv[(b + 1) & 1] = 1.0 / sO;
      }
      __syncthreads();
      const int m = s_m;
      if (m != g) {
        ++misses;
        fetch(mine, b, m);
        apply(sI, sO);
        if (tid == 0) s_scale = 1.0 / sqrt(sO);
        else if (tid == 32) s_inv[(b + 1) & 1] = 1.0 / sO;
      }
      cur ^= 1;
      __syncthreads();   // s_scale; sK and dst are complete
    }
    double* heap = reinterpret_cast<double*>(psi + (cur ^ 1) * AMPS);   // the register that is free
    oc::readout<float, NT>(psi + cur * AMPS, D, 0u, heap, ur, &s_bits, tid);
    const uint32_t x = s_bits;
    if (a.syn)
      for (int i = tid; i < syn_len; i += NT) a.syn[(size_t)t * syn_len + i] = out[i];
    if (a.bits && tid < a.nd) a.bits[(size_t)t * a.nd + tid] = (uint8_t)((x >> tid) & 1u);
    if (tid == 0) {
      if (a.logical) a.logical[t] = (uint8_t)(__popc(x & ((1u << a.nl) - 1u)) & 1);
      if (a.ctl) {
        if (misses) atomicAdd(&a.ctl->spec_misses, (unsigned long long)misses);
        if (t == a.n - 1) a.ctl->final_norm = heap[1];
      }
    }
    if (a.psi_out && t == a.n - 1)
      for (int i = tid; i < AMPS; i += NT) reinterpret_cast<float2*>(a.psi_out)[i] = psi[cur * AMPS + i];
    __syncthreads();   // the tree, out and s_bits are read
  }
}

constexpr size_t dense_smem(int D) { return 16ull << D; }

template <int D>
cudaError_t run_t(const DenseArgs& a, int num_sms, cudaStream_t s) {
  int occ = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_dense_run<D>, DenseShape<D>::NT, dense_smem(D));
  if (e != cudaSuccess) return e;
  const uint32_t wave = (uint32_t)(num_sms * (occ < 1 ? 1 : occ));
  k_dense_run<D><<<a.n < wave ? a.n : wave, DenseShape<D>::NT, dense_smem(D), s>>>(a);
  return cudaGetLastError();
}

template <int D>
cudaError_t attr_t() {
  return cudaFuncSetAttribute(k_dense_run<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dense_smem(D));
}

}  // namespace

bool dense_applies(int precision, int nd) { return !is_f64(precision) && (nd == 9 || nd == 11 || nd == 13); }

cudaError_t setup_dense(int nd) { return nd == 9 ? attr_t<9>() : nd == 11 ? attr_t<11>() : attr_t<13>(); }

cudaError_t launch_dense_runs(const DenseArgs& a, int num_sms, cudaStream_t s) {
  if (a.nd != 9 && a.nd != 11 && a.nd != 13) return cudaErrorInvalidValue;
  if (a.n == 0) return cudaSuccess;
  if (a.n > 65535u) return cudaErrorInvalidValue;
  if (a.rounds > 0) {
    k_dense_compile<<<dim3((unsigned)(a.rounds * a.nstab), a.n), 128, 0, s>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return a.nd == 9 ? run_t<9>(a, num_sms, s) : a.nd == 11 ? run_t<11>(a, num_sms, s) : run_t<13>(a, num_sms, s);
}

}  // namespace qec
