// Trajectories of registers in HBM, in factored passes (factor.hpp), several blocks to a pass.
//
// A block's outcome needs the whole register's sums, so a pass cannot know its blocks' outcomes.  It
// runs them for guesses (Sec. II.B measures a stabilizer once a round, and its outcome changes only at
// a detection event: the guess is its previous outcome) and sums |phi|^2 after every block.  The
// ratio of neighbouring sums is the outcome's probability given the ones before, so one pass decides
// its blocks up to and including the first wrong guess; the pass then runs again on its untouched
// input with those outcomes, until every guess held.  Results are those of measuring one block
// after the other.
//
// Per tile and block a thread holds one group of 16 amplitudes in registers: one rotation per data
// qubit, the diagonal of the outcome, the squares.  Tiles stream through shared memory (16-byte
// asynchronous copies in, whole 128-byte runs out); the register is read and written once per pass.
//
// What bounds them at d = 5 (2^25 amplitudes): in complex64 the shared-memory sweeps and their barriers (52% of issue
// slots, 0.54 of the copy bandwidth; per issue 1.6 cycles fixed latency, 1.4 shared memory, 1.2 barriers): 151 us for a
// pass of four blocks and 44 for one of one, plus 34 until the last CTA arrives.  In complex128 the FP64 pipe: 550 to 946
// us a block, plus 95 to 190 at the barrier, where the CTAs that were scheduled first on an SM wait for the others.  Against a
// dense 16x16 pass per block, five rounds: complex64 19.1 -> 7.6 ms, complex128 359 -> 87; with the Z part
// in diagonal passes 7.0 and 70.5.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "onchip.cuh"
#include "rounds.hpp"

namespace qec {
namespace {

using namespace oc;

template <typename T> struct Shape;
// complex64: 128 threads, 2 buffers, five CTAs per SM.  The pass is bound by its shared-memory sweeps (one
// per block) and their latency, so small CTAs that meet at barriers of four warps beat larger tiles:
// five rounds at d = 5 took 8.92 ms, against 9.00 with three buffers and four CTAs, 10.4 with six CTAs
// (85 registers: spills), 9.7 with runs of 128 bytes (11 passes a round instead of 9) and 9.5 with
// 4096-amplitude tiles on 256 threads.
template <> struct Shape<float> {
  static constexpr int BUF = 2, CTAS = 5, CTAS_POST = 4, CHAIN = 4;
};
// complex128: three CTAs per SM; the FP64 pipe is the bound (one ready warp per scheduler keeps it busy).
template <> struct Shape<double> {
  static constexpr int BUF = 2, CTAS = 3, CTAS_POST = 3, CHAIN = 4;
};

__device__ __forceinline__ void cp16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// ---- amplitudes in registers: packed pairs for complex64 (one instruction per complex axpy) -------------
typedef unsigned long long p2;
__device__ __forceinline__ p2 pk(float a, float b) {
  p2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 upk(p2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ p2 fma2(p2 a, p2 b, p2 c) {
  p2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
template <typename T> struct Reg;
template <> struct Reg<float> {
  using A = p2;
  using S = p2;         // running sum of squares
  static __device__ __forceinline__ A load(const float2* p) { return *reinterpret_cast<const p2*>(p); }
  static __device__ __forceinline__ void store(float2* p, A v) { *reinterpret_cast<p2*>(p) = v; }
  struct R { p2 t, nt, ti, nti; };   // (t, t), (-t, -t), (ti, -ti), (-ti, ti)
  static __device__ __forceinline__ R rot(float2 t) { return {pk(t.x, t.x), pk(-t.x, -t.x), pk(t.y, -t.y), pk(-t.y, t.y)}; }
  static __device__ __forceinline__ A swp(A v) { const float2 f = upk(v); return pk(f.y, f.x); }
  static __device__ __forceinline__ void real(A& x, A& y, const R& r) {
    const A a = fma2(r.nt, y, x);
    y = fma2(r.t, x, y);
    x = a;
  }
  // x - t* y: re: x.re - t.x y.re - t.y y.im, im: x.im - t.x y.im + t.y y.re
  static __device__ __forceinline__ void cplx(A& x, A& y, const R& r) {
    const A a = fma2(r.nti, swp(y), fma2(r.nt, y, x));
    const A a2 = a;
    y = fma2(r.nti, swp(x), fma2(r.t, x, y));
    x = a2;
  }
  static __device__ __forceinline__ void load2(const float2* p, A& a, A& b) {
    const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(p);
    a = w.x;
    b = w.y;
  }
  static __device__ __forceinline__ void store2(float2* p, A a, A b) { *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(a, b); }
  static __device__ __forceinline__ A scale(A v, float x, float y) {
    const float2 f = upk(v);
    return pk(fmaf(-y, f.y, x * f.x), fmaf(y, f.x, x * f.y));
  }
  static __device__ __forceinline__ void scale2(A& a, A& b, const float2* d) {   // d[0], d[1]: 16-byte aligned
    const float4 w = *reinterpret_cast<const float4*>(d);
    a = scale(a, w.x, w.y);
    b = scale(b, w.z, w.w);
  }
  static __device__ __forceinline__ S zero() { return 0ull; }
  static __device__ __forceinline__ void sq(S& s, A v) { s = fma2(v, v, s); }
  // Over the tiles: FP32 pairs (Knuth's two-sum keeps what each addition rounds off), so the FP64 pipe
  // is left out of the tile loop.
  using Acc = float2;
  static __device__ __forceinline__ void add(Acc& acc, S s) {
    const float2 f = upk(s), a = acc;
    const float v = f.x + f.y, h = a.x + v, z = h - a.x;
    acc = make_float2(h, a.y + ((a.x - (h - z)) + (v - z)));
  }
  static __device__ __forceinline__ Acc none() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ double total(Acc a) { return (double)a.x + (double)a.y; }
};
template <> struct Reg<double> {
  using A = double2;
  using S = double;
  static __device__ __forceinline__ A load(const double2* p) { return *p; }
  static __device__ __forceinline__ void store(double2* p, A v) { *p = v; }
  struct R { double2 t; };
  static __device__ __forceinline__ R rot(double2 t) { return {t}; }
  static __device__ __forceinline__ void real(A& x, A& y, const R& r) {
    const A a = make_double2(fma(-r.t.x, y.x, x.x), fma(-r.t.x, y.y, x.y));
    y = make_double2(fma(r.t.x, x.x, y.x), fma(r.t.x, x.y, y.y));
    x = a;
  }
  static __device__ __forceinline__ void cplx(A& x, A& y, const R& r) {
    const A a = make_double2(fma(-r.t.y, y.y, fma(-r.t.x, y.x, x.x)), fma(r.t.y, y.x, fma(-r.t.x, y.y, x.y)));
    y = make_double2(fma(-r.t.y, x.y, fma(r.t.x, x.x, y.x)), fma(r.t.y, x.x, fma(r.t.x, x.y, y.y)));
    x = a;
  }
  static __device__ __forceinline__ A scale(A v, double2 d) {
    return make_double2(fma(-d.y, v.y, d.x * v.x), fma(d.y, v.x, d.x * v.y));
  }
  static __device__ __forceinline__ void scale2(A& a, A& b, const double2* d) {
    a = scale(a, d[0]);
    b = scale(b, d[1]);
  }
  static __device__ __forceinline__ S zero() { return 0.0; }
  static __device__ __forceinline__ void sq(S& s, A v) { s = fma(v.x, v.x, fma(v.y, v.y, s)); }
  using Acc = double;
  static __device__ __forceinline__ void add(Acc& acc, S s) { acc += s; }
  static __device__ __forceinline__ Acc none() { return 0.0; }
  static __device__ __forceinline__ double total(Acc a) { return a; }
};

// Tile slot of amplitude e (ChainDesc::swz): a 16-byte chunk's place among the 8 of a 128-byte line.
// Linear over XOR, and a chunk stays whole.
template <typename T>
__host__ __device__ __forceinline__ uint32_t slot_of(uint32_t e, const uint16_t* swz) {
  constexpr int P = sizeof(T) == 4 ? 1 : 0;
#if defined(__CUDA_ARCH__)
  auto par = [](uint32_t x) { return (uint32_t)__popc(x) & 1u; };
#else
  auto par = [](uint32_t x) { return (uint32_t)__builtin_popcount(x) & 1u; };
#endif
  return e ^ (par(e & swz[0]) << P) ^ (par(e & swz[1]) << (P + 1)) ^ (par(e & swz[2]) << (P + 2));
}

// Groups of 2^GB amplitudes per thread: 16, or 4 on small complex128 registers (weight-2 blocks only), where a
// warp's FP64 instructions, one every 64 cycles, are the pass's time and four times the warps share them.  Eight
// CTAs per SM (15 qubits, five rounds, 128 trajectories: 7.5, 6.9, 6.4 and 5.8 ms with 4, 5, 6 and 8).
__host__ __device__ constexpr int group_bits(int TB) { return TB == 9 ? 2 : 4; }
__host__ __device__ constexpr int round_threads(int TB) { return 1 << (TB - group_bits(TB)); }

template <typename T, int TB>
struct Smem {
  static constexpr int NT = round_threads(TB), TS = 1 << TB;
  using T2 = typename V2t<T>::t;
  T2 tile[Shape<T>::BUF][TS];
  T2 d[Shape<T>::CHAIN][16];
  T2 rot[Shape<T>::CHAIN][8];              // before the diagonal, then (4 ..) after it
  uint32_t gen[Shape<T>::CHAIN][4];        // slots of a group's four tile bits
  typename Reg<T>::Acc acc[Shape<T>::CHAIN][NT];   // a thread's sums over the CTA's tiles
  uint16_t base[Shape<T>::CHAIN][NT];      // slot of a thread's group in each block
  alignas(8) uint8_t form[Shape<T>::CHAIN][8];
};

// One block on the thread's group of 2^GB amplitudes of a tile; returns its sum of squares after it.
// PAIR (complex64): the group's first tile bit is bit 0, so its amplitudes come in 16-byte pairs.
// POST: rotations after the diagonal (those that run early) may be there.
template <typename T, int GB, bool PAIR, bool POST>
__device__ __forceinline__ typename Reg<T>::S run_group(typename V2t<T>::t* tile, uint32_t b0, const uint32_t* gen,
                                                        const typename V2t<T>::t* rot, uint2 forms,
                                                        const typename V2t<T>::t* d) {
  using R = Reg<T>;
  constexpr int NA = 1 << GB;
  typename R::A v[NA];
  uint32_t at[NA];
  at[0] = b0;
#pragma unroll
  for (int j = 0; j < GB; ++j) {
    const uint32_t g = gen[j];
#pragma unroll
    for (int l = 0; l < (1 << j); ++l) at[l | (1 << j)] = at[l] ^ g;
  }
  if constexpr (PAIR) {
#pragma unroll
    for (int l = 0; l < NA; l += 2) R::load2(tile + at[l], v[l], v[l + 1]);
  } else {
#pragma unroll
    for (int l = 0; l < NA; ++l) v[l] = R::load(tile + at[l]);
  }
  auto turn = [&](uint32_t f4, const typename V2t<T>::t* r4) {
#pragma unroll
    for (int j = 0; j < GB; ++j) {
      const uint32_t f = (f4 >> (8 * j)) & 0xFFu;   // 0 also for a spectator
      if (f == 0) continue;
      const auto r = R::rot(r4[j]);
      if (f == 1) {
#pragma unroll
        for (int l = 0; l < NA; ++l)
          if (!(l & (1 << j))) R::real(v[l], v[l | (1 << j)], r);
      } else {
#pragma unroll
        for (int l = 0; l < NA; ++l)
          if (!(l & (1 << j))) R::cplx(v[l], v[l | (1 << j)], r);
      }
    }
  };
  turn(forms.x, rot);
#pragma unroll
  for (int l = 0; l < NA; l += 2) R::scale2(v[l], v[l + 1], d + l);
  if (POST && forms.y) turn(forms.y, rot + 4);
  auto s = R::zero();
#pragma unroll
  for (int l = 0; l < NA; l += 2) {
    R::sq(s, v[l]);
    R::sq(s, v[l + 1]);
    if constexpr (PAIR) {
      R::store2(tile + at[l], v[l], v[l + 1]);
    } else {
      R::store(tile + at[l], v[l]);
      R::store(tile + at[l + 1], v[l + 1]);
    }
  }
  return s;
}

__device__ __forceinline__ double warp_total(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// All CTAs of a group meet.  false: gave up (a bounded wait), reported in ctl->status.
__device__ __forceinline__ bool group_barrier(unsigned int* bar, unsigned int target, Ctl* ctl, int* s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    int ok = 0;
    for (long i = 0; i < 40000000; ++i) {
      if (*(volatile unsigned int*)bar >= target) {
        ok = 1;
        break;
      }
      __nanosleep(32);
    }
    if (!ok) atomicOr(&ctl->status, 1u);
    __threadfence();
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

template <typename T, bool POST, int TB>
__global__ void __launch_bounds__(round_threads(TB), (TB == kSmallTileBits ? 8 : POST ? Shape<T>::CTAS_POST : Shape<T>::CTAS)) k_rounds(const __grid_constant__ RoundArgs a, int r0, int r1) {
  using T2 = typename V2t<T>::t;
  using SH = Shape<T>;
  constexpr int GB = group_bits(TB), NT = round_threads(TB), NW = NT / 32, CH = 16 / sizeof(T2), NCH = (1 << TB) / (NT * CH);
  extern __shared__ __align__(16) unsigned char rsm[];
  Smem<T, TB>& S = *reinterpret_cast<Smem<T, TB>*>(rsm);
  __shared__ double s_sum[kMaxChain];
  __shared__ int s_ok, s_known, s_out;
  __shared__ ChainDesc C;
  __shared__ uint8_t s_prev[64];   // the syndrome bits of the round before, the guesses
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int grp = blockIdx.x / a.G, rank = blockIdx.x - grp * a.G;
  const int nstab = a.F.nstab;
  unsigned int* bar = a.bar + 2 * grp;
  uint8_t* syn = a.syn + (size_t)grp * (a.rounds + 1) * nstab;
  const Compiled<T>* blk = reinterpret_cast<const Compiled<T>*>(a.blocks) + (size_t)grp * a.rounds * nstab;
  const size_t amps = (size_t)1 << a.D;
  T2* buf[2] = {reinterpret_cast<T2*>(a.buf[0]) + grp * amps, reinterpret_cast<T2*>(a.buf[1]) + grp * amps};
  double N = r0 == 1 ? 1.0 : *(volatile double*)(a.norm + grp);
  unsigned int epoch = 0, misses = 0;
  bool ok = true;
  for (int i = tid; i < nstab; i += NT) s_prev[i] = r0 == 1 ? 0 : syn[(r0 - 1) * nstab + i];
  for (int rnd = r0; rnd <= r1 && ok; ++rnd) {
    for (int c = 0; c < a.nc && ok; ++c) {
      __syncthreads();
      for (int i = tid; i < (int)(sizeof(ChainDesc) / 4); i += NT)
        reinterpret_cast<uint32_t*>(&C)[i] = reinterpret_cast<const uint32_t*>(a.chains + c)[i];
      __syncthreads();
      const int step = (rnd - 1) * a.steps + c, nb = C.nb;
      const T2* src = step == 0 ? reinterpret_cast<const T2*>(a.psi0) : buf[(step & 1) ^ 1];
      T2* dst = buf[step & 1];
      const Compiled<T>* cb = blk + (size_t)(rnd - 1) * nstab + C.b0;
      // the group bases, rotations and forms of the chain's blocks
      for (int i = tid; i < nb * NT; i += NT) {
        const int b = i / NT;
        uint32_t x = (uint32_t)(i - b * NT);
#pragma unroll
        for (int j = 0; j < GB; ++j) {
          const int q = C.bits[b][j];
          x = ((x >> q) << (q + 1)) | (x & ((1u << q) - 1u));
        }
        S.base[b][i - b * NT] = (uint16_t)slot_of<T>(x, C.swz);
      }
      if (tid < 4 * nb && (tid & 3) < GB) {
        const int b = tid >> 2, j = tid & 3, q = C.qubit[b][j];
        S.gen[b][j] = slot_of<T>(1u << C.bits[b][j], C.swz);
        if (q < 4) S.rot[b][j] = cb[b].rot[q];
        S.form[b][j] = q < 4 && !fac::runs_early(a.F, 4 * (C.b0 + b) + q) ? cb[b].form[q] : (uint8_t)0;
        const int nx = q < 4 ? a.F.touches[4 * (C.b0 + b) + q].next : -1;
        const bool after = POST && nx >= 0 && fac::runs_early(a.F, nx);
        const Compiled<T>& cn = blk[(size_t)(rnd - 1) * nstab + (after ? nx >> 2 : 0)];
        if (after) S.rot[b][4 + j] = cn.rot[nx & 3];
        S.form[b][4 + j] = after ? cn.form[nx & 3] : (uint8_t)0;
      }
      // this thread's 16-byte chunks e = CH (tid + NT i): register offset and tile slot, both linear over XOR
      auto t2g = [&](uint32_t e) {
        const uint32_t h = e >> C.lb;
        uint32_t o = 0;
        for (int j = 0; j < C.nh; ++j) o |= ((h >> j) & 1u) << C.hbits[j];
        return o | (e & ((1u << C.lb) - 1u));
      };
      uint32_t coff[NCH];
#pragma unroll
      for (int i = 0; i < NCH; ++i) coff[i] = t2g((uint32_t)(CH * (tid + NT * i)));
      const uint32_t cslot = slot_of<T>((uint32_t)(CH * tid), C.swz);
      auto cdst = [&](int i) { return cslot ^ slot_of<T>((uint32_t)(CH * NT * i), C.swz); };
      const int obit = lane < C.nout ? C.obits[lane] : 0, nout = C.nout;
      auto tile_base = [&](uint32_t t) {
        return __reduce_or_sync(0xffffffffu, lane < nout ? ((t >> lane) & 1u) << obit : 0u);
      };
      const uint32_t ntile = 1u << C.nout;
      auto load_tile = [&](uint32_t t, T2* b) {
        if (t < ntile) {
          const T2* p = src + tile_base(t);
#pragma unroll
          for (int i = 0; i < NCH; ++i) cp16(b + cdst(i), p + coff[i]);
        }
        cp_commit();
      };
      int known = 0, out = 0;   // outcomes decided so far: bits 0 .. known - 1 of out
      for (;;) {
        // the chosen outcomes' diagonals; the input's scale goes into the first
        for (int i = tid; i < (nb << GB); i += NT) {
          const int b = i >> GB, l = i & ((1 << GB) - 1);
          const int off = a.F.blocks[C.b0 + b].offset;
          const int m = b < known ? (out >> b) & 1 : s_prev[C.b0 + b] ^ off;
          int z = 0;
#pragma unroll
          for (int j = 0; j < GB; ++j)
            if (C.qubit[b][j] < 4) z |= ((l >> j) & 1) << C.qubit[b][j];
          T2 v = cb[b].d[m][z];
          if (b == 0) {
            const double sc = rsqrt(N);
            v.x = (T)((double)v.x * sc);
            v.y = (T)((double)v.y * sc);
          }
          S.d[b][l] = v;
        }
        __syncthreads();
        for (int b = 0; b < nb; ++b) S.acc[b][tid] = Reg<T>::none();   // read by this thread alone, then after the last sync
        uint32_t t = (uint32_t)rank, cur = 0;
#pragma unroll
        for (int i = 0; i < SH::BUF - 1; ++i) load_tile(t + i * a.G, S.tile[i]);
        for (; t < ntile; t += a.G) {
          T2* tile = S.tile[cur];
          cp_wait<SH::BUF - 2>();
          __syncthreads();   // the tile is in; the previous one has left its buffer
          const uint32_t nxt = cur == 0 ? SH::BUF - 1 : cur - 1;
          load_tile(t + (SH::BUF - 1) * a.G, S.tile[nxt]);
          for (int b = 0; b < nb; ++b) {
            const uint2 forms = *reinterpret_cast<const uint2*>(S.form[b]);
            typename Reg<T>::S s;
            if (sizeof(T) == 4 && C.bits[b][0] == 0)
              s = run_group<T, GB, sizeof(T) == 4, POST>(tile, S.base[b][tid], S.gen[b], S.rot[b], forms, S.d[b]);
            else
              s = run_group<T, GB, false, POST>(tile, S.base[b][tid], S.gen[b], S.rot[b], forms, S.d[b]);
            Reg<T>::add(S.acc[b][tid], s);
            __syncthreads();
          }
          T2* p = dst + tile_base(t);
#pragma unroll
          for (int i = 0; i < NCH; ++i)
            *reinterpret_cast<float4*>(p + coff[i]) = *reinterpret_cast<const float4*>(tile + cdst(i));
          cur = cur + 1 == SH::BUF ? 0 : cur + 1;
        }
        cp_wait<0>();
        __syncthreads();
        for (int b = warp; b < nb; b += NW) {   // block b's sum over the CTA
          double acc = 0.0;
#pragma unroll
          for (int i = 0; i < NW; ++i) acc += Reg<T>::total(S.acc[b][lane + 32 * i]);
          acc = warp_total(acc);
          if (lane == 0) a.partials[((size_t)(epoch & 1) * gridDim.x + blockIdx.x) * kMaxChain + b] = acc;
        }
        ++epoch;
        ok = group_barrier(bar, epoch * a.G, a.ctl, &s_ok);
        if (!ok) break;
        // every CTA sums the group's partials in the same order and decides alike
        for (int b = warp; b < nb; b += NW) {
          const double* p = a.partials + ((size_t)((epoch - 1) & 1) * gridDim.x + grp * a.G) * kMaxChain + b;
          double s = 0.0;
          for (int i = lane; i < a.G; i += 32) s += __ldcg(p + (size_t)i * kMaxChain);
          s = warp_total(s);
          if (lane == 0) s_sum[b] = s;
        }
        __syncthreads();
        if (tid == 0) {
          double before = known ? s_sum[known - 1] : 1.0;
          int k = known, o = out;
          bool hit = true;
          while (k < nb && hit) {
            const int off = a.F.blocks[C.b0 + k].offset;
            const int gss = s_prev[C.b0 + k] ^ off;
            const double p1 = gss ? s_sum[k] : before - s_sum[k];
            const int m = cb[k].u * before < p1 ? 1 : 0;
            o |= m << k;
            hit = m == gss;
            before = s_sum[k];
            ++k;
            misses += !hit;
          }
          s_known = hit ? -k : k;   // negative: every guess held
          s_out = o;
        }
        __syncthreads();
        out = s_out;
        const int k = s_known;
        if (k < 0) {
          N = s_sum[nb - 1];
          break;
        }
        known = k;
        __syncthreads();   // s_known, s_out, s_sum are read before the next pass writes them
      }
      if (!ok) break;
      if (tid < nb) {
        const uint8_t bit = (uint8_t)(((out >> tid) & 1) ^ a.F.blocks[C.b0 + tid].offset);
        s_prev[C.b0 + tid] = bit;
        if (rank == 0) syn[rnd * nstab + C.b0 + tid] = bit;
      }
    }
  }
  if (tid == 0) {
    if (rank == 0) {
      a.norm[grp] = N;
      if (misses) atomicAdd(&a.ctl->spec_misses, (unsigned long long)misses);
    }
    // the last CTA to leave returns the barrier to 0 (none waits on it any more)
    __threadfence();
    if (atomicAdd(bar + 1, 1u) == (unsigned)a.G - 1) {
      bar[0] = 0;
      bar[1] = 0;
    }
  }
}

// ---- diagonal passes ------------------------------------------------------------------------------------
// A pass of blocks without rotations is phi(x) <- E(z(x)) phi(x), z the pass's data bits and E the product
// of the chosen outcomes' diagonals, and every sum it needs is a weighted sum of h(z) = sum |phi|^2 over
// the amplitudes with bits z.  A thread keeps the same tile positions in every tile, so its E and h are
// in registers; amplitudes stream through a ring of thread-private 16-byte copies, without barriers: 6
// multiply-adds each however many blocks the pass holds.  When the tiles are done, the sums for the
// guessed outcomes decide the blocks up to the first wrong guess; those for the corrected path come
// from the same h.  So the outcomes cost one pass whatever the guesses, and wrong ones one more without
// sums.
//
// At 2^25 amplitudes a complex64 pass takes 68 to 93 us (memory: 512 MiB are 79 at the copy rate) and 17 to 37
// to decide, a complex128 one 350 (the FP64 pipe: 6 multiply-adds an amplitude are 320; 1 GiB 158) and 8
// to 15.  The Z part of a d = 5 round, complex128, went from 12 dense tensor-core passes of 0.39 ms to 1.7-2.0.
constexpr int kDiagThreads = 512;
__host__ __device__ constexpr int diag_bits(bool f64) { return f64 ? 12 : 13; }

template <typename T>
struct DiagSmem {
  using T2 = typename V2t<T>::t;
  static constexpr int TB = diag_bits(sizeof(T) == 8), P = (1 << TB) / kDiagThreads;   // positions per thread
  static constexpr int CH = 16 / sizeof(T2), NCH = P / CH, STAGES = 2;
  union {
    float4 ring[STAGES][NCH][kDiagThreads];
    struct {                                   // after a pass
      double pos[1 << TB];                     // h per tile position
      double sum[kMaxDiag + 1][kDiagThreads];
    } r;
  };
  T2 E[1 << kDiagUnion];
  double h[1 << kDiagUnion];
  double wd[kMaxDiag][2][16];                  // |D_m|^2
  T2 d[kMaxDiag][2][16];
  double u[kMaxDiag];
  double scale;                                // of the input
  uint8_t guess[kMaxDiag];
};

template <typename T>
__global__ void __launch_bounds__(kDiagThreads) k_diagonals(const __grid_constant__ RoundArgs a, int rnd) {
  using T2 = typename V2t<T>::t;
  using SM = DiagSmem<T>;
  constexpr int NT = kDiagThreads, P = SM::P, CH = SM::CH, NCH = SM::NCH, ST = SM::STAGES;
  extern __shared__ __align__(16) unsigned char dsm[];
  SM& S = *reinterpret_cast<SM*>(dsm);
  __shared__ double s_sum[kMaxDiag + 1];
  __shared__ int s_ok, s_known, s_out;
  __shared__ DiagDesc C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nstab = a.F.nstab, G = (int)gridDim.x;
  uint8_t* syn = a.syn;
  const Compiled<T>* blk = reinterpret_cast<const Compiled<T>*>(a.blocks) + (size_t)(rnd - 1) * nstab;
  double N = a.diag_in ? *(volatile const double*)(a.diag_in + (size_t)(rnd - 1) * a.diag_stride)
                       : rnd == 1 && a.step0 == 0 ? 1.0 : *(volatile double*)a.norm;
  unsigned int epoch = 0, misses = 0;
  bool ok = true;
  for (int c = 0; c < a.nd && ok; ++c) {
    __syncthreads();
    for (int i = tid; i < (int)(sizeof(DiagDesc) / 4); i += NT)
      reinterpret_cast<uint32_t*>(&C)[i] = reinterpret_cast<const uint32_t*>(a.diags + c)[i];
    __syncthreads();
    const int step = (rnd - 1) * a.steps + a.step0 + c, nb = C.nb;
    const T2* src = reinterpret_cast<const T2*>(step == 0 ? a.psi0 : a.buf[(step & 1) ^ 1]);
    T2* dst = reinterpret_cast<T2*>(a.buf[step & 1]);
    const Compiled<T>* cb = blk + C.b0;
    if (tid < nb) {
      const int b = C.b0 + tid;
      S.u[tid] = cb[tid].u;
      S.guess[tid] = (uint8_t)((rnd == 1 ? 0 : syn[(rnd - 1) * nstab + b]) ^ a.F.blocks[b].offset);
    }
    if (tid == NT - 1) S.scale = rsqrt(N);
    for (int i = tid; i < 32 * nb; i += NT) {
      const int b = i >> 5, m = (i >> 4) & 1, z = i & 15;
      if (z >> C.w[b]) continue;
      const T2 d = cb[b].d[m][z];
      S.d[b][m][z] = d;
      S.wd[b][m][z] = fma((double)d.x, (double)d.x, (double)d.y * (double)d.y);
    }
    uint32_t coff[NCH];
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      const uint32_t e = (uint32_t)(CH * (tid + NT * i)), hi = e >> C.lb;
      uint32_t o = 0;
      for (int j = 0; j < C.nh; ++j) o |= ((hi >> j) & 1u) << C.hbits[j];
      coff[i] = o | (e & ((1u << C.lb) - 1u));
    }
    auto bin_of = [&](uint32_t e) {   // the pass's data bits at tile index e
      uint32_t z = 0;
      for (int j = 0; j < C.nu; ++j) z |= ((e >> C.ubits[j]) & 1u) << j;
      return z;
    };
    auto z_of = [&](int b, uint32_t bin) {   // block b's data bits
      int z = 0;
      for (int j = 0; j < C.w[b]; ++j) z |= (int)((bin >> C.at[b][j]) & 1u) << j;
      return z;
    };
    const int nout = C.nout, obit = lane < nout ? C.obits[lane] : 0;
    auto tile_base = [&](uint32_t t) {
      return __reduce_or_sync(0xffffffffu, lane < nout ? ((t >> lane) & 1u) << obit : 0u);
    };
    const uint32_t ntile = 1u << nout, bins = 1u << C.nu;
    auto load = [&](uint32_t t, int st) {
      if (t < ntile) {
        const T2* p = src + tile_base(t);
#pragma unroll
        for (int i = 0; i < NCH; ++i) cp16(&S.ring[st][i][tid], p + coff[i]);
      }
      cp_commit();
    };
    double h[P];
    // one pass for the outcomes in `out`; SUM: |phi|^2 goes into h
    auto pass = [&](int out, auto with_sums) {
      constexpr bool SUM = decltype(with_sums)::value;
      __syncthreads();   // S.d, S.wd are there; the ring's memory is free
#pragma unroll
      for (int i = 0; i < ST; ++i) load(blockIdx.x + i * G, i);
      for (uint32_t z = tid; z < bins; z += NT) {
        T2 e = make2<T2>(S.scale, 0.0);
        for (int b = 0; b < nb; ++b) {
          const T2 d = S.d[b][(out >> b) & 1][z_of(b, z)], x = e;
          e.x = fma(-d.y, x.y, d.x * x.x);
          e.y = fma(d.y, x.x, d.x * x.y);
        }
        S.E[z] = e;
      }
      __syncthreads();
      T2 E[P];
#pragma unroll
      for (int k = 0; k < P; ++k) E[k] = S.E[bin_of((uint32_t)(CH * (tid + NT * (k / CH)) + k % CH))];
      T part[P];   // complex64: FP32 over up to 16 tiles, then FP64
      int run = 0, st = 0;
#pragma unroll
      for (int k = 0; k < P; ++k) {
        part[k] = 0;
        h[k] = SUM ? 0.0 : h[k];
      }
      for (uint32_t t = blockIdx.x; t < ntile; t += G) {
        T2* o = dst + tile_base(t);
        cp_wait<ST - 1>();
#pragma unroll
        for (int i = 0; i < NCH; ++i) {
          T2 v[CH];
          *reinterpret_cast<float4*>(v) = S.ring[st][i][tid];
#pragma unroll
          for (int k = 0; k < CH; ++k) {
            const T2 x = v[k], e = E[CH * i + k];
            if (SUM) part[CH * i + k] = fma(x.x, x.x, fma(x.y, x.y, part[CH * i + k]));
            v[k].x = fma(-e.y, x.y, e.x * x.x);
            v[k].y = fma(e.y, x.x, e.x * x.y);
          }
          *reinterpret_cast<float4*>(o + coff[i]) = *reinterpret_cast<const float4*>(v);
        }
        load(t + ST * G, st);   // this thread has consumed its copies of the stage
        st = st + 1 == ST ? 0 : st + 1;
        if (SUM && sizeof(T) == 4 && ++run == 16) {
          run = 0;
#pragma unroll
          for (int k = 0; k < P; ++k) {
            h[k] += (double)part[k];
            part[k] = 0;
          }
        }
      }
      cp_wait<0>();
      if (SUM)
#pragma unroll
        for (int k = 0; k < P; ++k) h[k] += (double)part[k];
    };
    int out = 0, known = 0;   // chosen outcomes; the first `known` are decided
    __syncthreads();
    for (int b = 0; b < nb; ++b) out |= S.guess[b] << b;
    const int guess = out;
    pass(out, std::true_type{});
    __syncthreads();
#pragma unroll
    for (int k = 0; k < P; ++k) S.r.pos[CH * (tid + NT * (k / CH)) + k % CH] = h[k];
    __syncthreads();
    for (uint32_t z = tid; z < bins; z += NT) {
      uint32_t e0 = 0;
      for (int j = 0; j < C.nu; ++j) e0 |= ((z >> j) & 1u) << C.ubits[j];
      double s = 0.0;
      for (uint32_t i = 0; i < (1u << (SM::TB - C.nu)); ++i) {
        uint32_t e = e0;
        for (int j = 0; j < SM::TB - C.nu; ++j) e |= ((i >> j) & 1u) << C.rbits[j];
        s += S.r.pos[e];
      }
      S.h[z] = s;   // read by this thread alone
    }
    for (;;) {
      // S_i of the chosen path, i = 0 (the input's norm) .. nb
      double s[kMaxDiag + 1];
#pragma unroll
      for (int i = 0; i <= kMaxDiag; ++i) s[i] = 0.0;
      for (uint32_t z = tid; z < bins; z += NT) {
        double w = S.h[z];
        s[0] += w;
#pragma unroll
        for (int b = 0; b < kMaxDiag; ++b)
          if (b < nb) {
            w *= S.wd[b][(out >> b) & 1][z_of(b, z)];
            s[b + 1] += w;
          }
      }
#pragma unroll
      for (int i = 0; i <= kMaxDiag; ++i)
        if (i <= nb) S.r.sum[i][tid] = s[i];
      __syncthreads();
      if (warp <= nb) {
        double t = 0.0;
        const uint32_t n = bins < NT ? bins : NT;
        for (uint32_t i = lane; i < n; i += 32) t += S.r.sum[warp][i];
        t = warp_total(t);
        if (lane == 0) a.partials[((size_t)(epoch & 1) * G + blockIdx.x) * (kMaxDiag + 1) + warp] = t;
      }
      ++epoch;
      ok = group_barrier(a.bar, epoch * G, a.ctl, &s_ok);
      if (!ok) break;
      if (warp <= nb) {
        const double* p = a.partials + (size_t)((epoch - 1) & 1) * G * (kMaxDiag + 1) + warp;
        double t = 0.0;
        for (int i = lane; i < G; i += 32) t += __ldcg(p + (size_t)i * (kMaxDiag + 1));
        t = warp_total(t);
        if (lane == 0) s_sum[warp] = t;
      }
      __syncthreads();
      if (tid == 0) {
        int k = known, o = out;
        bool hit = true;
        while (k < nb && hit) {
          const int g = (out >> k) & 1;
          const double p1 = g ? s_sum[k + 1] : s_sum[k] - s_sum[k + 1];
          const int m = S.u[k] * s_sum[k] < p1 ? 1 : 0;
          hit = m == g;
          if (!hit) o ^= 1 << k;
          ++k;
          misses += !hit;
        }
        s_known = hit ? nb + 1 : k;
        s_out = o;
      }
      __syncthreads();
      known = s_known;
      out = s_out;
      if (known > nb) break;   // the whole path holds
    }
    if (!ok) break;
    const double total = s_sum[nb];
    if (out != guess) pass(out, std::false_type{});
    N = total / N;
    if (blockIdx.x == 0 && tid < nb)
      syn[rnd * nstab + C.b0 + tid] = (uint8_t)(((out >> tid) & 1) ^ a.F.blocks[C.b0 + tid].offset);
    if (c + 1 < a.nd) {   // the next pass reads what every CTA wrote
      ++epoch;
      ok = group_barrier(a.bar, epoch * G, a.ctl, &s_ok);
    }
  }
  if (tid == 0) {
    if (blockIdx.x == 0) {
      if (a.diag_out) a.diag_out[(size_t)(rnd - 1) * a.diag_stride] = N;
      else a.norm[0] = N;
      if (misses) atomicAdd(&a.ctl->spec_misses, (unsigned long long)misses);
      if (a.ctl->prob_force_exact) {   // these sums are the exact evaluation that hook asks for
        int n = 0;
        for (int c = 0; c < a.nd; ++c) n += a.diags[c].nb;
        atomicAdd(&a.ctl->prob_fallbacks, (unsigned long long)n);
      }
    }
    __threadfence();
    if (atomicAdd(a.bar + 1, 1u) == (unsigned)G - 1) {
      a.bar[0] = 0;
      a.bar[1] = 0;
    }
  }
}

// ---- dense blocks for the tensor-core passes ---------------------------------------------------------------
// K_m = R_after D_m R_before of block b (the factored register's gauge), R the products of the rotations
// before it and of those after it that run early (their cosines are in D_m).  One CTA per block, a
// thread per entry.
__global__ void __launch_bounds__(256) k_dense(const __grid_constant__ RoundArgs a, int nb, double2* kraus, double* u) {
  const int b = blockIdx.x % nb, r = blockIdx.x / nb, nstab = a.F.nstab;
  const Compiled<double>* blk = reinterpret_cast<const Compiled<double>*>(a.blocks) + (size_t)r * nstab;
  const Compiled<double>& C = blk[b];
  const FBlock B = a.F.blocks[b];
  const int w = B.w, n = 1 << w, row = threadIdx.x >> 4, col = threadIdx.x & 15;
  __shared__ double2 pre[4][4], post[4][4];
  if (threadIdx.x < 8) {
    const int j = threadIdx.x & 3;
    const bool after = threadIdx.x >= 4;
    double2 t = make_double2(0.0, 0.0);
    if (j < w) {
      const int tc = 4 * b + j, nx = a.F.touches[tc].next;
      if (!after) {
        if (!fac::runs_early(a.F, tc)) t = C.rot[j];
      } else if (nx >= 0 && fac::runs_early(a.F, nx)) {
        // the cosine is in D_m: the t form itself
        t = blk[nx >> 2].rot[nx & 3];
      }
    }
    double2* m = after ? post[j] : pre[j];
    m[0] = m[3] = make_double2(1.0, 0.0);
    m[1] = make_double2(-t.x, t.y);
    m[2] = t;
  }
  __syncthreads();
  double2 k0 = make_double2(0.0, 0.0), k1 = k0;
  if (row < n && col < n)
    for (int l = 0; l < n; ++l) {
      double2 x = make_double2(1.0, 0.0);
      for (int j = 0; j < w; ++j)
        x = fac::cmul(x, fac::cmul(post[j][2 * ((row >> j) & 1) + ((l >> j) & 1)], pre[j][2 * ((l >> j) & 1) + ((col >> j) & 1)]));
      const double2 x0 = fac::cmul(x, C.d[0][l]), x1 = fac::cmul(x, C.d[1][l]);
      k0 = make_double2(k0.x + x0.x, k0.y + x0.y);
      k1 = make_double2(k1.x + x1.x, k1.y + x1.y);
    }
  double2* out = kraus + ((size_t)r * nstab + b) * KRAUS_STRIDE;
  out[threadIdx.x] = k0;
  out[256 + threadIdx.x] = k1;
  if (threadIdx.x == 0) u[(size_t)r * nstab + b] = C.u;
}

// ---- compile ------------------------------------------------------------------------------------------
__host__ __device__ inline size_t scratch_bytes(int nstab, int nsites) {
  return (sizeof(fac::Touch) * 4 * nstab + 4 * nstab + nsites + 255) / 256 * 256;
}

struct CtaGroup {
  int rank, size;
  __device__ __forceinline__ void sync() const { __syncthreads(); }
};

__device__ __forceinline__ fac::Rounds round_scratch(const RoundArgs& a, size_t stride, int grp, int r) {
  unsigned char* w = a.scratch + ((size_t)grp * a.rounds + r) * stride;
  fac::Rounds R;
  R.nr = 1;
  R.T = reinterpret_cast<fac::Touch*>(w);
  R.swap = w + sizeof(fac::Touch) * 4 * a.F.nstab;
  R.code = R.swap + 4 * a.F.nstab;
  R.mask = a.masks + (size_t)grp * a.rounds + r;
  return R;
}

__device__ __forceinline__ void load_mats(const RoundArgs& a, double2 (*fm)[4]) {
  for (int i = threadIdx.x; i < FM_COUNT * 4; i += blockDim.x)
    fm[i >> 2][i & 3] = make_double2(a.fm[i >> 2][i & 3][0], a.fm[i >> 2][i & 3][1]);
}

__global__ void __launch_bounds__(128) k_compile_merge(const __grid_constant__ RoundArgs a, size_t stride) {
  __shared__ double2 fm[FM_COUNT][4];
  const int r = blockIdx.x, grp = blockIdx.y;
  const fac::Rounds R = round_scratch(a, stride, grp, r);
  load_mats(a, fm);
  if (threadIdx.x == 0) *R.mask = 0;
  __syncthreads();
  const uint64_t traj = a.first + grp;
  fac::compile_merge(CtaGroup{(int)threadIdx.x, (int)blockDim.x}, a.F, a.thr, a.seed, traj, (uint64_t)(r + 1), fm, R,
                     [&](int, int i, int c) {
                       const FSite& s = a.F.sites[i];
                       if (!a.events || !c || s.kind == OP_T1 || s.kind == OP_T2) return;
                       const unsigned e = atomicAdd(&a.ctl->n_events, 1u);
                       if (e >= a.ctl->ev_cap) return;
                       int32_t* ev = a.events + 5 * (size_t)e;
                       ev[0] = (int32_t)traj; ev[1] = r + 1; ev[2] = s.step; ev[3] = (int32_t)s.site; ev[4] = c;
                     });
}

template <typename T>
__global__ void __launch_bounds__(128) k_compile_emit(const __grid_constant__ RoundArgs a, size_t stride) {
  using T2 = typename V2t<T>::t;
  __shared__ double2 fm[FM_COUNT][4];
  const int r = blockIdx.x, grp = blockIdx.y;
  const fac::Rounds R = round_scratch(a, stride, grp, r);
  load_mats(a, fm);
  __syncthreads();
  uint32_t flips = 0;
  for (int i = 0; i < r; ++i) flips ^= a.masks[(size_t)grp * a.rounds + i];
  Compiled<T>* out = reinterpret_cast<Compiled<T>*>(a.blocks) + ((size_t)grp * a.rounds + r) * a.F.nstab;
  fac::compile_emit(CtaGroup{(int)threadIdx.x, (int)blockDim.x}, a.F, fm, R, flips,
                    [&](int, int i, double2 v) {
                      out[i >> 2].rot[i & 3] = make2<T2>(v.x, v.y);
                      out[i >> 2].form[i & 3] = rotation_form(v);
                    },
                    [&](int, int b, int z, double2 d0, double2 d1) {
                      out[b].d[0][z] = make2<T2>(d0.x, d0.y);
                      out[b].d[1][z] = make2<T2>(d1.x, d1.y);
                    });
  for (int b = threadIdx.x; b < a.F.nstab; b += blockDim.x)
    out[b].u = uniform53(draw(a.seed, a.first + grp, (uint64_t)(r + 1), 0u, (uint32_t)(a.F.nd + b), TAG_MEASURE).v[0]);
}

}  // namespace

// The kernel for a pass's tile bits and its shared memory; early: with the rotations that run early (large
// registers only).
struct RoundKernel {
  const void* fn;
  size_t smem;
};
template <typename T>
static RoundKernel round_kernel_t(int tb, bool early) {
  if constexpr (sizeof(T) == 8)
    if (tb == kSmallTileBits) return {(const void*)k_rounds<T, false, kSmallTileBits>, sizeof(Smem<T, kSmallTileBits>)};
  return {early ? (const void*)k_rounds<T, true, 11> : (const void*)k_rounds<T, false, 11>, sizeof(Smem<T, 11>)};
}
static RoundKernel round_kernel(int precision, int tb, bool early) {
  return is_f64(precision) ? round_kernel_t<double>(tb, early) : round_kernel_t<float>(tb, early);
}

size_t compile_scratch_bytes(const FactorProgram& F) { return scratch_bytes(F.nstab, (int)F.sites.size()); }
size_t compiled_block_bytes(int precision) { return is_f64(precision) ? sizeof(Compiled<double>) : sizeof(Compiled<float>); }

// Shared-memory wavefronts of a warp's 16 group loads (32-bit banks; `wide`: bytes of one load), summed
// over the pass's blocks.
static int conflict_cost(const ChainDesc& c, int precision, int gb) {
  const bool f64 = is_f64(precision);
  int cost = 0;
  for (int i = 0; i < c.nb; ++i) {
    const bool pair = !f64 && c.bits[i][0] == 0;
    const int wide = f64 || pair ? 16 : 8, lanes = 128 / wide, unit = f64 ? 16 : 8;
    for (int w = 0; w < 32; w += lanes) {
      int per_slot[16] = {}, worst = 0;
      for (int l = w; l < w + lanes; ++l) {
        uint32_t x = (uint32_t)l;
        for (int j = 0; j < gb; ++j) {
          const int q = c.bits[i][j];
          x = ((x >> q) << (q + 1)) | (x & ((1u << q) - 1u));
        }
        const uint32_t s = f64 ? slot_of<double>(x, c.swz) : slot_of<float>(x, c.swz);
        worst = std::max(worst, ++per_slot[(s * unit % 128) / wide]);
      }
      cost += worst * (pair ? 1 : 2);   // half as many loads for pairs
    }
  }
  return cost;
}

// Swizzle masks over the tile bits above a line's chunk bits: the default fold, or a better one of a
// fixed pseudo-random sequence (the same for every handle).
static void choose_swizzle(ChainDesc& c, int precision, int TB) {
  const int lo = is_f64(precision) ? 3 : 4;
  const uint32_t all = ((1u << TB) - 1u) & ~((1u << lo) - 1u);
  uint16_t best[3];
  for (int k = 0; k < 3; ++k) {
    uint32_t m = 0;
    for (int b = lo + k; b < TB; b += 3) m |= 1u << b;
    c.swz[k] = best[k] = (uint16_t)m;
  }
  int cost = conflict_cost(c, precision, group_bits(TB)), floor = 0;
  for (int i = 0; i < c.nb; ++i) floor += !is_f64(precision) && c.bits[i][0] != 0 ? 4 : is_f64(precision) ? 8 : 4;
  uint64_t x = 0x9E3779B97F4A7C15ull;
  for (int t = 0; t < 100 && cost > floor; ++t) {
    for (int k = 0; k < 3; ++k) {
      x ^= x << 13;
      x ^= x >> 7;
      x ^= x << 17;
      c.swz[k] = (uint16_t)(x & all);
    }
    const int n = conflict_cost(c, precision, group_bits(TB));
    if (n < cost) {
      cost = n;
      std::copy(c.swz, c.swz + 3, best);
    }
  }
  std::copy(best, best + 3, c.swz);
}

std::vector<ChainDesc> plan_chains(const FactorProgram& F, int precision, int TB, int most, int b0, int b1) {
  constexpr int low = 3;
  most = std::min(most, is_f64(precision) ? Shape<double>::CHAIN : Shape<float>::CHAIN);
  std::vector<ChainDesc> out;
  for (int b = b0; b < b1;) {
    uint32_t mask = 0;
    int nb = 0;
    while (b + nb < b1 && nb < most) {
      uint32_t m = mask;
      for (int j = 0; j < F.blocks[b + nb].w; ++j) m |= 1u << F.blocks[b + nb].q[j];
      if (nb && __builtin_popcount(m | ((1u << low) - 1u)) > TB) break;
      mask = m;
      ++nb;
    }
    ChainDesc c{};
    c.b0 = b;
    c.nb = nb;
    int lb = low;
    while (__builtin_popcount(mask | ((1u << lb) - 1u)) < TB) ++lb;   // registers of more than TB qubits only
    c.lb = lb;
    int tile_bit[32];
    for (int q = 0; q < F.nd; ++q) {
      if (q < lb) tile_bit[q] = q;
      else if (mask & (1u << q)) {
        tile_bit[q] = lb + c.nh;
        c.hbits[c.nh++] = (uint8_t)q;
      } else {
        tile_bit[q] = -1;
        c.obits[c.nout++] = (uint8_t)q;
      }
    }
    for (int i = 0; i < nb; ++i) {
      const FBlock& B = F.blocks[b + i];
      c.w[i] = B.w;
      int q[4], which[4], n = B.w;
      for (int j = 0; j < n; ++j) {
        q[j] = tile_bit[B.q[j]];
        which[j] = j;
      }
      // spectators: tile bit 0 (complex64 amplitudes then come in pairs), then the highest tile bits
      // outside the block (a warp's groups lie side by side)
      auto used = [&](int x) { return std::find(q, q + n, x) != q + n; };
      const int gb = group_bits(TB);
      for (int x = TB; n < gb; --x) {
        const int y = x == TB ? 0 : x;
        if (used(y)) continue;
        q[n] = y;
        which[n++] = 4;
      }
      for (int j = 0; j < gb; ++j) {   // ascending
        int at = 0;
        for (int k = 0; k < gb; ++k) at += q[k] < q[j];
        c.bits[i][at] = (uint8_t)q[j];
        c.qubit[i][at] = (uint8_t)which[j];
      }
    }
    choose_swizzle(c, precision, TB);
    out.push_back(c);
    b += nb;
  }
  return out;
}

std::vector<DiagDesc> plan_diagonals(const FactorProgram& F, int precision, int b0, int b1) {
  const int TB = diag_bits(is_f64(precision)), low = is_f64(precision) ? 3 : 4;
  std::vector<DiagDesc> out;
  for (int b = b0; b < b1;) {
    uint32_t mask = 0;
    int nb = 0;
    while (b + nb < b1 && nb < kMaxDiag) {
      uint32_t m = mask;
      for (int j = 0; j < F.blocks[b + nb].w; ++j) m |= 1u << F.blocks[b + nb].q[j];
      if (nb && (__builtin_popcount(m | ((1u << low) - 1u)) > TB || __builtin_popcount(m) > kDiagUnion)) break;
      mask = m;
      ++nb;
    }
    DiagDesc c{};
    c.b0 = b;
    c.nb = nb;
    int lb = low;
    while (__builtin_popcount(mask | ((1u << lb) - 1u)) < TB) ++lb;
    c.lb = lb;
    int tile_bit[32];
    for (int q = 0; q < F.nd; ++q) {
      if (q < lb) tile_bit[q] = q;
      else if (mask & (1u << q)) {
        tile_bit[q] = lb + c.nh;
        c.hbits[c.nh++] = (uint8_t)q;
      } else {
        c.obits[c.nout++] = (uint8_t)q;
      }
    }
    int index[32], nr = 0;   // a data qubit's place among the pass's
    uint32_t in_union = 0;
    for (int q = 0; q < F.nd; ++q)
      if (mask & (1u << q)) {
        index[q] = c.nu;
        c.ubits[c.nu++] = (uint8_t)tile_bit[q];
        in_union |= 1u << tile_bit[q];
      }
    for (int t = 0; t < TB; ++t)
      if (!(in_union & (1u << t))) c.rbits[nr++] = (uint8_t)t;
    for (int i = 0; i < nb; ++i) {
      c.w[i] = F.blocks[b + i].w;
      for (int j = 0; j < c.w[i]; ++j) c.at[i][j] = (uint8_t)index[F.blocks[b + i].q[j]];
    }
    out.push_back(c);
    b += nb;
  }
  return out;
}

cudaError_t setup_rounds(int precision) {
  cudaError_t e = cudaSuccess;
  for (int v = is_f64(precision) ? 0 : 1; v < 3 && e == cudaSuccess; ++v) {
    const RoundKernel k = round_kernel(precision, v == 0 ? kSmallTileBits : kTileBits, v == 2);
    e = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k.fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  }
  const void* dg = is_f64(precision) ? (const void*)k_diagonals<double> : (const void*)k_diagonals<float>;
  const int dsmem = is_f64(precision) ? (int)sizeof(DiagSmem<double>) : (int)sizeof(DiagSmem<float>);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(dg, cudaFuncAttributeMaxDynamicSharedMemorySize, dsmem);
  return e;
}

int round_wave(int precision, int tb, bool early, int num_sms) {
  int occ = 0;
  const RoundKernel k = round_kernel(precision, tb, early);
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k.fn, round_threads(tb), k.smem);
  return e == cudaSuccess && occ > 0 ? occ * num_sms : 0;
}

cudaError_t launch_compile(int precision, const RoundArgs& a, cudaStream_t s) {
  const size_t stride = scratch_bytes(a.F.nstab, a.F.nsites);
  const dim3 grid((unsigned)a.rounds, (unsigned)a.groups);
  k_compile_merge<<<grid, 128, 0, s>>>(a, stride);
  if (is_f64(precision)) k_compile_emit<double><<<grid, 128, 0, s>>>(a, stride);
  else k_compile_emit<float><<<grid, 128, 0, s>>>(a, stride);
  return cudaGetLastError();
}

cudaError_t launch_diagonals(int precision, const RoundArgs& a, int r, int num_sms, cudaStream_t s) {
  RoundArgs b = a;
  void* args[2] = {&b, &r};
  const int64_t tiles = 1ll << (a.D - diag_bits(is_f64(precision)));
  const dim3 grid((unsigned)(tiles < num_sms ? tiles : num_sms));
  const void* fn = is_f64(precision) ? (const void*)k_diagonals<double> : (const void*)k_diagonals<float>;
  return cudaLaunchCooperativeKernel(fn, grid, dim3(kDiagThreads), args, is_f64(precision) ? sizeof(DiagSmem<double>) : sizeof(DiagSmem<float>), s);
}

cudaError_t launch_dense(const RoundArgs& a, int nb, void* kraus, double* u, cudaStream_t s) {
  k_dense<<<nb * a.rounds, 256, 0, s>>>(a, nb, static_cast<double2*>(kraus), u);
  return cudaGetLastError();
}

cudaError_t launch_rounds(int precision, const RoundArgs& a, int r0, int r1, cudaStream_t s) {
  RoundArgs b = a;
  void* args[3] = {&b, &r0, &r1};
  const dim3 grid((unsigned)(a.groups * a.G));
  const RoundKernel k = round_kernel(precision, a.tb, a.F.early != 0);
  return cudaLaunchCooperativeKernel(k.fn, grid, dim3((unsigned)round_threads(a.tb)), args, k.smem, s);
}

}  // namespace qec
