// Trajectory entry point that makes no device allocation.
//
// For callers that cannot call cudaMalloc: code that runs while its framework
// owns every byte of device memory through its own pool or arena, code on a
// latency-critical path where cudaMalloc's implicit device synchronisation is
// not acceptable, or plug-ins that are handed a stream and output buffers but
// no allocator.  All device working memory of the call (circuit program, init
// state, the init round's Kraus blocks and reduction partials, the Kraus blocks of a few
// complex64 trajectories, control word) lives in one file-scope static device array below; the caller passes
// only the inputs (parameters, seed, trajectory range) and the device output
// buffers.  The array is sized for the d = 3 register (2^9 amplitudes) with at
// most kNoAllocMaxRounds noisy rounds, and every GPU that loads this library
// holds it until the process exits.
#include <cuda_runtime.h>

#include <cstddef>
#include <cstring>
#include <mutex>
#include <string>

#include "../../include/qecsv.h"
#include "common.cuh"
#include "dense.hpp"
#include "factor.cuh"
#include "kernels.hpp"
#include "onchip.hpp"
#include "program.hpp"

using namespace qec;

namespace {

constexpr size_t kNoAllocBytes = (size_t)2 << 20;   // 2 MiB
constexpr int kNoAllocMaxD = 3;
constexpr int kNoAllocMaxRounds = 16;
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// Device address of g_noalloc_scratch per device (host code must not use the symbol itself:
// in host code its name is only a host-side stand-in).
std::mutex g_mu;
void* g_scratch_ptr[kMaxDevices] = {};

qec_status nfail(qec_status s, const std::string& m) {
  set_last_error(m);   // reported by qec_last_error()
  return s;
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

struct Carve {
  size_t off = 0;
  size_t take(size_t bytes) {
    size_t o = off;
    off = up256(off + bytes);
    return o;
  }
};

qec_status run_noalloc(const qec_params* params, uint64_t seed, uint64_t first_traj, uint32_t n,
                       uint8_t* d_syndromes, uint8_t* d_data_bits, uint8_t* d_raw_logical, void* cuda_stream) {
  if (!params) return nfail(QEC_EINVAL, "null params");
  std::string err;
  if (!validate_params(*params, err)) return nfail(QEC_EINVAL, err);
  if (params->layout != QEC_LAYOUT_REDUCED) return nfail(QEC_EUNSUPPORTED, "only the reduced register runs on the GPU");
  if (params->d > kNoAllocMaxD || params->rounds > kNoAllocMaxRounds)
    return nfail(QEC_EINVAL, "qec_run_trajectories_noalloc: its static device scratch (2 MiB) holds at most d = 3 "
                             "and 16 noisy rounds; use qec_create/qec_run_trajectories for larger runs");
  if (n == 0) return QEC_OK;
  if (!d_syndromes || !d_data_bits || !d_raw_logical) return nfail(QEC_EINVAL, "null output buffer");

  Program init_prog, prog;
  if (!build_program(*params, false, init_prog, err) || !build_program(*params, true, prog, err))
    return nfail(QEC_EINVAL, err);
  const int D = prog.nd, nstab = prog.nstab, R = params->rounds;
  const int prec = params->precision;
  const size_t amp = is_f64(prec) ? 16 : 8;

  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return nfail(QEC_ECUDA, std::string("device query: ") + cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return nfail(QEC_EUNSUPPORTED, "device index too large");
  unsigned char* base = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_scratch_ptr[dev]) {   // once per device, with that device current
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess || !p)
        return nfail(QEC_ECUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
      g_scratch_ptr[dev] = p;
    }
    base = static_cast<unsigned char*>(g_scratch_ptr[dev]);
  }

  FactorProgram fprog;
  if (!build_factor(prog, fprog, err)) return nfail(QEC_EINVAL, err);
  int pgrid = pass_grid(D, 2, sms);
  const int pg4 = pass_grid(D, 4, sms);
  if (pg4 > pgrid) pgrid = pg4;
  const bool dense = dense_applies(prec, D);   // complex64: blocks' Kraus pairs, for as many trajectories as 1 MiB holds
  if (dense && !dense_fits(prog)) return nfail(QEC_EUNSUPPORTED, "a block has more ops than the engine's table");
  const size_t entries = (size_t)dense_entries(prog), blocks = (size_t)nstab * R;
  const uint32_t most = blocks ? (uint32_t)((1u << 20) / (blocks * 2 * entries * sizeof(float2))) : 65535u;
  Carve c;
  const size_t o_psi0 = c.take(((size_t)1 << D) * amp);
  const size_t o_ops = c.take(sizeof(ProgOp) * (init_prog.ops.size() + 1));
  const size_t o_blk = c.take(sizeof(BlockInfo) * nstab), o_mat = c.take(sizeof(prog.mats));
  const void* fac_src[5] = {fprog.sites.data(), fprog.items.data(), fprog.touches.data(), fprog.blocks.data(),
                            fprog.order.data()};
  const size_t fac_bytes[5] = {sizeof(FSite) * fprog.sites.size(), sizeof(FItem) * fprog.items.size(),
                               sizeof(FTouch) * fprog.touches.size(), sizeof(FBlock) * fprog.blocks.size(),
                               sizeof(uint16_t) * fprog.order.size()};
  size_t o_fac[5];
  for (int i = 0; i < 5; ++i) o_fac[i] = c.take(fac_bytes[i]);
  const size_t o_kraus = c.take((size_t)nstab * KRAUS_STRIDE * amp);
  const size_t o_u = c.take(sizeof(double) * nstab), o_A = c.take(sizeof(double) * nstab);
  const size_t o_N = c.take(sizeof(double) * nstab), o_m = c.take(sizeof(int) * nstab);
  const size_t o_part = c.take(sizeof(double) * 2 * (pgrid > MAX_PASS_GRID ? pgrid : MAX_PASS_GRID));
  const size_t o_ctl = c.take(sizeof(Ctl));
  const size_t o_nops = c.take(dense ? sizeof(ProgOp) * (prog.ops.size() + 1) : 0);
  const size_t o_nblk = c.take(dense ? sizeof(BlockInfo) * nstab : 0), o_nmat = c.take(dense ? sizeof(prog.mats) : 0);
  const size_t o_pair = c.take(dense ? most * blocks * 2 * entries * sizeof(float2) : 0);
  const size_t o_nu = c.take(dense ? most * blocks * sizeof(double) : 0);
  if (c.off > kNoAllocBytes) return nfail(QEC_EINVAL, "request does not fit the 2 MiB static scratch");

  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  void* psi0 = base + o_psi0;
  ProgOp* ops = reinterpret_cast<ProgOp*>(base + o_ops);
  BlockInfo* blks = reinterpret_cast<BlockInfo*>(base + o_blk);
  double* mats = reinterpret_cast<double*>(base + o_mat);
  if (!init_prog.ops.empty())
    e = cudaMemcpyAsync(ops, init_prog.ops.data(), sizeof(ProgOp) * init_prog.ops.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(blks, init_prog.blocks.data(), sizeof(BlockInfo) * nstab, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(mats, init_prog.mats, sizeof(init_prog.mats), cudaMemcpyHostToDevice, st);
  for (int i = 0; i < 5 && e == cudaSuccess; ++i)
    if (fac_bytes[i]) e = cudaMemcpyAsync(base + o_fac[i], fac_src[i], fac_bytes[i], cudaMemcpyHostToDevice, st);
  if (dense) {
    if (e == cudaSuccess && !prog.ops.empty())
      e = cudaMemcpyAsync(base + o_nops, prog.ops.data(), sizeof(ProgOp) * prog.ops.size(), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(base + o_nblk, prog.blocks.data(), sizeof(BlockInfo) * nstab, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(base + o_nmat, prog.mats, sizeof(prog.mats), cudaMemcpyHostToDevice, st);
  }
  // The control word is the only scratch that must start from known values (the reduction
  // ticket at 0); everything else is written before it is read.
  Ctl h_ctl;
  std::memset(&h_ctl, 0, sizeof(h_ctl));
  h_ctl.seed = seed;
  h_ctl.first = first_traj;
  h_ctl.traj = first_traj;
  Ctl* ctl = reinterpret_cast<Ctl*>(base + o_ctl);
  if (e == cudaSuccess) e = cudaMemcpyAsync(ctl, &h_ctl, sizeof(Ctl), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return nfail(QEC_ECUDA, std::string("scratch upload: ") + cudaGetErrorString(e));

  auto inst = [&]() {
    const Program& P = init_prog;
    InstArgs a;
    a.ops = ops;
    a.blocks = blks;
    a.mats = mats;
    for (int i = 0; i < PR_COUNT; ++i) a.prob[i] = P.prob[i];
    a.nstab = nstab;
    a.nd = D;
    a.round_base = 0;
    a.nblk = nstab;
    a.kraus = base + o_kraus;
    a.u = reinterpret_cast<double*>(base + o_u);
    a.ctl = nullptr;
    a.events = nullptr;
    return a;
  };
  auto pass = [&](int blk) {
    const BlockInfo& bi = init_prog.blocks[blk];
    PassArgs a;
    a.src = psi0;
    a.dst = psi0;
    a.D = D;
    a.w = bi.w;
    for (int j = 0; j < 4; ++j) a.q[j] = bi.q[j] < 0 ? 0 : bi.q[j];
    a.kraus = base + o_kraus + (size_t)blk * KRAUS_STRIDE * amp;
    a.u = reinterpret_cast<double*>(base + o_u) + blk;
    a.forced = bi.offset;
    a.A = reinterpret_cast<double*>(base + o_A) + blk;
    a.N = reinterpret_cast<double*>(base + o_N) + blk;
    a.m = reinterpret_cast<int*>(base + o_m) + blk;
    a.ctl = ctl;
    a.partials = reinterpret_cast<double*>(base + o_part);
    a.syn = nullptr;
    a.syn_stride = (R + 1) * nstab;
    a.syn_idx = 0;
    a.offset = bi.offset;
    return a;
  };

  // The same launches and kernels as qec_create / qec_run_trajectories, so that the results are
  // identical: the init round's passes, then every trajectory on chip.
  auto prob = [&](const PassArgs& a) { return launch_prob(prec, a, pass_grid_for(prec, true, D, a.w, sms), st); };
  auto apply = [&](const PassArgs& a) { return launch_apply(prec, a, pass_grid_for(prec, false, D, a.w, sms), st); };
  // Noise-free init round with outcomes forced to the zero syndrome (Sec. III.B), in psi0.
  e = launch_set_basis0(prec, psi0, D, st);
  if (e == cudaSuccess) e = launch_instantiate(prec, inst(), st);
  for (int k = 0; k < nstab && e == cudaSuccess; ++k) {
    const PassArgs a = pass(k);
    e = prob(a);
    if (e == cudaSuccess) e = apply(a);
  }
  if (e == cudaSuccess) e = dense ? setup_dense(D) : setup_onchip();
  if (e == cudaSuccess && dense) {
    DenseArgs a;
    a.ops = reinterpret_cast<const ProgOp*>(base + o_nops);
    a.blocks = reinterpret_cast<const BlockInfo*>(base + o_nblk);
    a.mats = reinterpret_cast<const double*>(base + o_nmat);
    for (int i = 0; i < PR_COUNT; ++i) a.prob[i] = prog.prob[i];
    a.nstab = nstab;
    a.nd = D;
    a.rounds = R;
    a.nl = params->d;
    a.entries = (int)entries;
    a.seed = seed;
    a.psi0 = psi0;
    a.kraus = reinterpret_cast<float2*>(base + o_pair);
    a.u = reinterpret_cast<double*>(base + o_nu);
    a.psi_out = nullptr;
    a.ctl = nullptr;
    a.events = nullptr;
    for (uint32_t at = 0; at < n && e == cudaSuccess; at += a.n) {
      a.n = n - at < most ? n - at : most;
      a.first = first_traj + at;
      a.syn = d_syndromes + (size_t)at * (R + 1) * nstab;
      a.bits = d_data_bits + (size_t)at * D;
      a.logical = d_raw_logical + at;
      e = launch_dense_runs(a, sms, st);
    }
  } else if (e == cudaSuccess) {
    OnchipArgs a;
    a.F = view_of(fprog);
    a.F.sites = reinterpret_cast<const FSite*>(base + o_fac[0]);
    a.F.items = reinterpret_cast<const FItem*>(base + o_fac[1]);
    a.F.touches = reinterpret_cast<const FTouch*>(base + o_fac[2]);
    a.F.blocks = reinterpret_cast<const FBlock*>(base + o_fac[3]);
    a.F.order = reinterpret_cast<const uint16_t*>(base + o_fac[4]);
    for (int i = 0; i < PR_COUNT; ++i) a.thr[i] = fac::draw_threshold(prog.prob[i]);
    factor_mats(prog.mats, params->gates == QEC_GATES_CR, params->noise.twirl != 0.0, a.fm);
    a.seed = seed;
    a.first = first_traj;
    a.n = n;
    a.rounds = R;
    a.nl = params->d;
    a.psi0 = psi0;
    a.psi_out = nullptr;
    a.syn = d_syndromes;
    a.bits = d_data_bits;
    a.logical = d_raw_logical;
    a.ctl = nullptr;
    a.events = nullptr;
    e = launch_onchip(a, sms, st);
  }
  if (e != cudaSuccess) return nfail(QEC_ECUDA, std::string("launch: ") + cudaGetErrorString(e));
  return QEC_OK;
}

}  // namespace

extern "C" qec_status qec_run_trajectories_noalloc(const qec_params* params, uint64_t seed, uint64_t first_traj,
                                                   uint32_t n, uint8_t* d_syndromes, uint8_t* d_data_bits,
                                                   uint8_t* d_raw_logical, void* cuda_stream) {
  try {
    return run_noalloc(params, seed, first_traj, n, d_syndromes, d_data_bits, d_raw_logical, cuda_stream);
  } catch (...) {   // a host allocation of the circuit program failed: nothing crosses the C ABI
    return nfail(QEC_ENOMEM, "exception in qec_run_trajectories_noalloc");
  }
}
