// A whole trajectory of a small register on one thread group, with the register in shared memory.
//
// Per round the group compiles the blocks into factored form (factor.cuh), then runs them: a block's
// rotations on groups of four amplitudes (two data qubits at a time: one sweep for a weight-2 block,
// two for a weight-4 one), the two outcomes' weights sum_x |D_m(z(x)) phi(x)|^2 on the amplitudes in
// registers (phi is already rotated, so a probability is a diagonal sum), the outcome, and the
// multiplication by D_m.  The last sweep's amplitudes stay in registers across the reduction, so a
// block reads and writes shared memory once per sweep and HBM never.
#pragma once
#include "common.cuh"
#include "factor.cuh"

namespace qec {
namespace oc {

template <typename T> struct V2t;
template <> struct V2t<double> { using t = double2; };
template <> struct V2t<float> { using t = float2; };

template <typename T2>
__device__ __forceinline__ T2 make2(double x, double y) {
  T2 r;
  r.x = (decltype(r.x))x;
  r.y = (decltype(r.y))y;
  return r;
}

// NT threads with ranks 0..NT-1: one warp (NT = 32), or a CTA.
template <int NT>
struct Group {
  int rank;
  static constexpr int size = NT;
  __device__ __forceinline__ void sync() const {
    if constexpr (NT == 32) __syncwarp();
    else __syncthreads();
  }
};

// Rotation forms: 0 none (t = 0), 1 a real t, 2 a complex one.  The same for every amplitude, so a
// branch on it is free of divergence, and an integer test keeps it off the FP64 pipe.
__device__ __forceinline__ uint8_t rotation_form(double2 t) {
  return fac::is_zero(t.y) ? (fac::is_zero(t.x) ? 0 : 1) : 2;
}

// o_0 = x - t* y, o_1 = y + t x.
template <typename T2>
__device__ __forceinline__ void rotate(T2& x, T2& y, T2 t, int form) {
  T2 a = x, b = y;
  a.x = fma(-t.x, y.x, a.x);
  a.y = fma(-t.x, y.y, a.y);
  b.x = fma(t.x, x.x, b.x);
  b.y = fma(t.x, x.y, b.y);
  if (form == 2) {
    a.x = fma(-t.y, y.y, a.x);
    a.y = fma(t.y, y.x, a.y);
    b.x = fma(-t.y, x.y, b.x);
    b.y = fma(t.y, x.x, b.y);
  }
  x = a;
  y = b;
}

// Sums a and b over the group; every thread returns the same totals.  A warp folds the two sums in
// one shuffle tree (lanes 0..15 carry a, 16..31 b after the first step), in a fixed order.
template <int NT>
__device__ __forceinline__ void group_sum2(double& a, double& b, double* red, int rank) {
  const int lane = rank & 31, warp = rank >> 5;
  const bool hi = lane & 16;
  double v = hi ? b : a;
  v += __shfl_xor_sync(0xffffffffu, hi ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if constexpr (NT > 32) {
    constexpr int NW = NT / 32;
    if ((lane & 15) == 0) red[(lane >> 4) * 32 + warp] = v;
    __syncthreads();
    constexpr int M = NW < 16 ? NW : 16;   // lanes l and l + 16 take warp l's partials
    v = red[(lane >> 4) * 32 + (lane & (M - 1))];
    if constexpr (NW > 16) v += red[(lane >> 4) * 32 + 16 + (lane & 15)];
#pragma unroll
    for (int o = M / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  a = __shfl_sync(0xffffffffu, v, 0);
  b = __shfl_sync(0xffffffffu, v, 16);
}

// The same sums over 128 places, four on a lane (place 32 i + lane) instead of one on each of 128 threads: the same
// tree as group_sum2<128>, so that one warp and a CTA of four decide alike.  Each step of a warp's tree
// halves the values that a lane carries: 11 additions, 5 for one value each.
__device__ __forceinline__ void warp_sum4(const double (&a)[4], const double (&b)[4], double& A, double& B) {
  const int lane = threadIdx.x & 31;
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
  double r[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) r[i] = (h16 ? b[i] : a[i]) + __shfl_xor_sync(0xffffffffu, h16 ? a[i] : b[i], 16);
  double p0 = (h8 ? r[2] : r[0]) + __shfl_xor_sync(0xffffffffu, h8 ? r[0] : r[2], 8);
  double p1 = (h8 ? r[3] : r[1]) + __shfl_xor_sync(0xffffffffu, h8 ? r[1] : r[3], 8);
  double v = (h4 ? p1 : p0) + __shfl_xor_sync(0xffffffffu, h4 ? p0 : p1, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 8);   // the four warps' sums
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  A = __shfl_sync(0xffffffffu, v, 0);
  B = __shfl_sync(0xffffffffu, v, 16);
}

// The register's scale is free (a probability is a ratio of sums over one state): where the kept part's
// norm gets small, an exact power of two brings it back into range.
__device__ __forceinline__ int norm_exp(double a) { return (int)((__double_as_longlong(a) >> 52) & 0x7FF) - 1023; }
__device__ __forceinline__ bool small_norm(double a) { return norm_exp(a) < -20; }
template <typename T>
__device__ __forceinline__ T norm_scale(double a) {
  const int e = norm_exp(a);
  return (T)__longlong_as_double((long long)(1023 + (-(e < -1022 ? -1022 : e) >> 1)) << 52);
}

// A compiled block in shared memory.
template <typename T>
struct Compiled {
  using T2 = typename V2t<T>::t;
  T2 d[2][16];      // D_0, D_1
  T wt[2][16];      // |D_0|^2, |D_1|^2
  T2 rot[4];
  double u;         // measurement uniform
  uint8_t form[4];  // the rotations' forms
};

// One block on the group's register psi (2^D = 4 NT ITEMS amplitudes); returns the raw outcome (drawn, or
// `forced` where that is not negative).  red: 64 doubles (NT > 32), alternated between calls by `parity`.
template <typename T, int NT, int ITEMS>
__device__ __forceinline__ int run_block(typename V2t<T>::t* psi, const FBlock& B, const Compiled<T>& C, double* red,
                                         int parity, int rank, int forced = -1) {
  using T2 = typename V2t<T>::t;
  T2 v[ITEMS][4];
  uint32_t at[ITEMS];
  auto sweep = [&](int qa, int qb, int j, bool store) {
    const T2 ta = C.rot[j], tb = C.rot[j + 1];
    const int fa = C.form[j], fb = C.form[j + 1];
    const uint32_t ma = 1u << qa, mb = 1u << qb;   // qa < qb
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      uint32_t x = (uint32_t)(rank + NT * i);
      x = ((x >> qa) << (qa + 1)) | (x & (ma - 1u));
      x = ((x >> qb) << (qb + 1)) | (x & (mb - 1u));
      at[i] = x;
#pragma unroll
      for (int l = 0; l < 4; ++l) v[i][l] = psi[x | (l & 1 ? ma : 0u) | (l & 2 ? mb : 0u)];
      if (fa) {
        rotate(v[i][0], v[i][1], ta, fa);
        rotate(v[i][2], v[i][3], ta, fa);
      }
      if (fb) {
        rotate(v[i][0], v[i][2], tb, fb);
        rotate(v[i][1], v[i][3], tb, fb);
      }
      if (store)
#pragma unroll
        for (int l = 0; l < 4; ++l) psi[x | (l & 1 ? ma : 0u) | (l & 2 ? mb : 0u)] = v[i][l];
    }
  };
  const bool w4 = B.w == 4;
  int qa = B.q[0], qb = B.q[1];
  if (w4) {
    if (C.form[0] | C.form[1]) {
      sweep(qa, qb, 0, true);
      if constexpr (NT == 32) __syncwarp();
      else __syncthreads();
    }
    qa = B.q[2];
    qb = B.q[3];
  }
  sweep(qa, qb, w4 ? 2 : 0, false);
  T s0[ITEMS], s1[ITEMS];
  int z0[ITEMS];
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    z0[i] = w4 ? (int)(((at[i] >> B.q[0]) & 1u) | (((at[i] >> B.q[1]) & 1u) << 1)) : 0;
    s0[i] = s1[i] = 0;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int z = w4 ? z0[i] | (l << 2) : l;
      const T sq = fma(v[i][l].x, v[i][l].x, v[i][l].y * v[i][l].y);
      s0[i] = fma(C.wt[0][z], sq, s0[i]);
      s1[i] = fma(C.wt[1][z], sq, s1[i]);
    }
  }
  double A0, A1;
  if constexpr (NT == 32 && ITEMS == 4) {
    warp_sum4(s0, s1, A0, A1);
  } else {
    A0 = (double)s0[0];
    A1 = (double)s1[0];
#pragma unroll
    for (int i = 1; i < ITEMS; ++i) {
      A0 += (double)s0[i];
      A1 += (double)s1[i];
    }
    group_sum2<NT>(A0, A1, red + (parity & 1) * 64, rank);
  }
  const int m = forced >= 0 ? forced : C.u * (A0 + A1) < A1 ? 1 : 0;
  const double A = m ? A1 : A0;
  const bool rescale = small_norm(A);
  const T sc = norm_scale<T>(A);
  const uint32_t ma = 1u << qa, mb = 1u << qb;
#pragma unroll
  for (int i = 0; i < ITEMS; ++i)
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      T2 d = C.d[m][w4 ? z0[i] | (l << 2) : l];
      if (rescale) {
        d.x *= sc;
        d.y *= sc;
      }
      T2 o;
      o.x = fma(-d.y, v[i][l].y, d.x * v[i][l].x);
      o.y = fma(d.y, v[i][l].x, d.x * v[i][l].y);
      psi[at[i] | (l & 1 ? ma : 0u) | (l & 2 ? mb : 0u)] = o;
    }
  if constexpr (NT == 32) __syncwarp();
  else __syncthreads();
  return m;
}

// Final readout (Sec. III.B): qubit j gets [u_j < P(q_j = 1 | outcomes of qubits < j)].  heap (2^D
// doubles) gets, at 2^j + i, the weight of all indices equal to i modulo 2^j (j < D), built from the
// top level down with one addition per entry; the qubits are then sampled by walking it.  ur[j]: the
// uniforms.  psi is read at x ^ flips.  Thread 0 returns the sampled index in *out; heap[1] is the norm.
template <typename T, int NT>
__device__ void readout(const typename V2t<T>::t* psi, int D, uint32_t flips, double* heap, const double* ur,
                        uint32_t* out, int rank) {
  const Group<NT> g{rank};
  auto weight = [&](uint32_t x) {
    const auto a = psi[x ^ flips];
    return (double)a.x * (double)a.x + (double)a.y * (double)a.y;
  };
  for (int j = D - 1; j >= 0; --j) {
    const uint32_t n = 1u << j;
    for (uint32_t i = (uint32_t)rank; i < n; i += NT)
      heap[n + i] = j == D - 1 ? weight(i) + weight(i + n) : heap[2 * n + i] + heap[2 * n + n + i];
    g.sync();
  }
  if (rank == 0) {
    uint32_t x = 0;
    for (int j = 0; j < D; ++j) {
      const uint32_t n = 1u << j;
      const double all = heap[n + x], one = j == D - 1 ? weight(x + n) : heap[2 * n + x + n];
      if (ur[j] * all < one) x |= n;
    }
    *out = x;
  }
  g.sync();
}

}  // namespace oc
}  // namespace qec
