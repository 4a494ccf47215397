// On-chip complex128 trajectories: registers of 9 and 11 data qubits (the d = 3 surface code, the
// repetition code of d = 9 and 11), one CTA per trajectory, the whole trajectory in one launch.
//
// What bounds it: for one trajectory latency (FP64 instructions issue at 64 cycles per warp and
// scheduler on this chip, then barriers and the reduction trees of 8 blocks a round), for many the
// FP64 pipe: per weight-4 block 8 rotation, 4 weight and 4 diagonal multiply-adds per amplitude,
// against 136 for the dense probability and apply, plus the compile, about a quarter of the work.
// Measured against a graph of dense probability and apply passes per trajectory (d = 3, 3 rounds,
// complex128): one trajectory 849 -> 145 us, 1000 of them 797 ms -> 0.67 ms.
#include <cuda_runtime.h>

#include "onchip.cuh"
#include "onchip.hpp"

namespace qec {
namespace {

using namespace oc;

// Rounds compiled together, and the shared memory of one trajectory.
template <int NT, int ITEMS>
struct Layout {
  static constexpr int kAmps = 4 * NT * ITEMS;
  static constexpr int kD = kAmps == 512 ? 9 : 11;
  static constexpr int kStab = kD - 1;                        // 8 (both codes), 10
  static constexpr int kRounds = 4;
  static constexpr int kTouches = 4 * kStab;
  static constexpr int kSites = 384;                          // draws of a round, at most
  static constexpr size_t kScratch = kRounds * (sizeof(fac::Touch) * kTouches + kTouches + kSites);
  static constexpr size_t kUnion = ((kScratch > 8 * (size_t)kAmps ? kScratch : 8 * (size_t)kAmps) + 15) / 16 * 16;
  static constexpr size_t kPsi = sizeof(double2) * (size_t)kAmps;
  static constexpr size_t kBlocks = sizeof(Compiled<double>) * kRounds * kStab;
  static constexpr size_t kSmem = kPsi + kUnion + kBlocks;
};

template <int NT, int ITEMS>
__global__ void __launch_bounds__(NT) k_onchip(const __grid_constant__ OnchipArgs a) {
  using T = double;
  using T2 = double2;
  using L = Layout<NT, ITEMS>;
  constexpr int D = L::kD;
  extern __shared__ __align__(16) unsigned char osm[];
  T2* psi = reinterpret_cast<T2*>(osm);
  unsigned char* un = osm + L::kPsi;                       // compile scratch, then the readout's tree
  Compiled<T>* blk = reinterpret_cast<Compiled<T>*>(un + L::kUnion);
  __shared__ double red[2 * 64];
  __shared__ double2 fm[FM_COUNT][4];
  __shared__ uint32_t mask[L::kRounds];
  __shared__ double ur[D];
  __shared__ uint8_t out[65 * L::kStab];
  __shared__ uint32_t s_bits;
  const int tid = threadIdx.x;
  const FactorView& F = a.F;
  const int nstab = F.nstab, syn_len = (a.rounds + 1) * nstab;
  for (int i = tid; i < FM_COUNT * 4; i += NT) fm[i >> 2][i & 3] = make_double2(a.fm[i >> 2][i & 3][0], a.fm[i >> 2][i & 3][1]);
  for (uint32_t t = blockIdx.x; t < a.n; t += gridDim.x) {
    const uint64_t traj = a.first + t;
    const T2* p0 = reinterpret_cast<const T2*>(a.psi0);
    for (int i = tid; i < L::kAmps; i += NT) psi[i] = p0[i];
    for (int i = tid; i < nstab; i += NT) out[i] = 0;
    if (tid < D) ur[tid] = uniform53(draw(a.seed, traj, (uint64_t)a.rounds + 1, 0u, (uint32_t)tid, TAG_READOUT).v[0]);
    uint32_t flips = 0;
    unsigned misses = 0;
    int parity = 0;
    for (int r0 = 1; r0 <= a.rounds; r0 += L::kRounds) {
      const int nr = min(L::kRounds, a.rounds + 1 - r0);
      if (tid < L::kRounds) mask[tid] = 0;
      __syncthreads();
      const Group<NT> g{tid};
      fac::Rounds R;
      R.nr = nr;
      R.T = reinterpret_cast<fac::Touch*>(un);
      R.swap = un + sizeof(fac::Touch) * L::kRounds * L::kTouches;
      R.code = R.swap + L::kRounds * L::kTouches;
      R.mask = mask;
      fac::compile_merge(g, F, a.thr, a.seed, traj, (uint64_t)r0, fm, R, [&](int k, int i, int c) {
        const FSite& s = F.sites[i];
        if (!a.events || !c || s.kind == OP_T1 || s.kind == OP_T2) return;
        const unsigned e = atomicAdd(&a.ctl->n_events, 1u);
        if (e >= a.ctl->ev_cap) return;
        int32_t* ev = a.events + 5 * (size_t)e;
        ev[0] = (int32_t)traj; ev[1] = r0 + k; ev[2] = s.step; ev[3] = (int32_t)s.site; ev[4] = c;
      });
      fac::compile_emit(g, F, fm, R, flips,
                        [&](int k, int i, double2 v) {
                          Compiled<T>& c = blk[k * L::kStab + (i >> 2)];
                          c.rot[i & 3] = make2<T2>(v.x, v.y);
                          c.form[i & 3] = rotation_form(v);
                        },
                        [&](int k, int b, int z, double2 d0, double2 d1) {
                          Compiled<T>& c = blk[k * L::kStab + b];
                          c.d[0][z] = make2<T2>(d0.x, d0.y);
                          c.d[1][z] = make2<T2>(d1.x, d1.y);
                          c.wt[0][z] = (T)fac::cnorm(d0);
                          c.wt[1][z] = (T)fac::cnorm(d1);
                        });
      for (int i = tid; i < nr * nstab; i += NT) {
        const int k = i / nstab, b = i - k * nstab;
        blk[k * L::kStab + b].u =
            uniform53(draw(a.seed, traj, (uint64_t)(r0 + k), 0u, (uint32_t)(F.nd + b), TAG_MEASURE).v[0]);
      }
      __syncthreads();
      for (int k = 0; k < nr; ++k) {
        flips ^= mask[k];
        for (int b = 0; b < nstab; ++b) {
          const FBlock B = F.blocks[b];
          const int m = run_block<T, NT, ITEMS>(psi, B, blk[k * L::kStab + b], red, parity++, tid);
          if (tid == 0) {
            uint8_t* o = out + (r0 + k) * nstab + b;
            *o = (uint8_t)(m ^ B.offset);
            misses += *o != o[-nstab];
          }
        }
      }
      __syncthreads();   // mask and the compiled blocks are read
    }
    double* heap = reinterpret_cast<double*>(un);
    readout<T, NT>(psi, D, flips, heap, ur, &s_bits, tid);
    const uint32_t x = s_bits;
    if (a.syn)
      for (int i = tid; i < syn_len; i += NT) a.syn[(size_t)t * syn_len + i] = out[i];
    if (a.bits && tid < F.nd) a.bits[(size_t)t * F.nd + tid] = (uint8_t)((x >> tid) & 1u);
    if (tid == 0) {
      if (a.logical) a.logical[t] = (uint8_t)(__popc(x & ((1u << a.nl) - 1u)) & 1);
      if (a.ctl) {
        if (misses) atomicAdd(&a.ctl->spec_misses, (unsigned long long)misses);
        if (t == a.n - 1) a.ctl->final_norm = heap[1];
      }
    }
    if (a.psi_out && t == a.n - 1)
      for (int i = tid; i < L::kAmps; i += NT) reinterpret_cast<T2*>(a.psi_out)[i] = psi[i ^ flips];
    __syncthreads();   // the tree and s_bits are read
  }
}

template <int NT, int ITEMS>
cudaError_t launch_t(const OnchipArgs& a, int num_sms, cudaStream_t s) {
  constexpr size_t smem = Layout<NT, ITEMS>::kSmem;
  int occ = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_onchip<NT, ITEMS>, NT, smem);
  if (e != cudaSuccess) return e;
  const uint32_t wave = (uint32_t)(num_sms * (occ < 1 ? 1 : occ));
  k_onchip<NT, ITEMS><<<a.n < wave ? a.n : wave, NT, smem, s>>>(a);
  return cudaGetLastError();
}

template <int NT, int ITEMS>
cudaError_t attr_t() {
  return cudaFuncSetAttribute(k_onchip<NT, ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)Layout<NT, ITEMS>::kSmem);
}

}  // namespace

bool onchip_applies(int nd) { return nd == 9 || nd == 11; }

cudaError_t setup_onchip() {
  cudaError_t e = attr_t<128, 1>();
  if (e == cudaSuccess) e = attr_t<512, 1>();
  return e;
}

// Threads: one group of four amplitudes each: a single trajectory's latency is a chain of sweeps, and its
// FP64 work spreads over the SM's four schedulers.
cudaError_t launch_onchip(const OnchipArgs& a, int num_sms, cudaStream_t s) {
  if (!onchip_applies(a.F.nd) || a.F.nsites > Layout<128, 1>::kSites) return cudaErrorInvalidValue;
  if (a.n == 0) return cudaSuccess;
  return a.F.nd == 9 ? launch_t<128, 1>(a, num_sms, s) : launch_t<512, 1>(a, num_sms, s);
}

}  // namespace qec
