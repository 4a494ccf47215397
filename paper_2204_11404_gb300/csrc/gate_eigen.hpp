// The gate's eigenbasis in an X stabilizer (factor.hpp), in any real type: once per handle in extended precision
// on the host (a rounding error there is in every block of a trajectory, alike in every round), per trajectory
// on the device where a batch's trajectories have their own angles.
#pragma once
#include <cmath>

namespace qec {

#if defined(__CUDACC__)
#define QEC_EIGEN_HD __host__ __device__
#else
#define QEC_EIGEN_HD
#endif

// C: a complex type with members x, y; R: its real type.  g0, g1: 2x2 unitaries, row-major.  lam gets Lambda as a 2x2.
template <class C, class R>
QEC_EIGEN_HD inline void gate_eigen(const C* g0, const C* g1, C* sh, C* a0, C* a1, C* lam) {
  auto c = [](R x, R y) { C r; r.x = x; r.y = y; return r; };
  // a* b + d* e, and a b + d e
  auto dotc = [&](C a, C b, C d, C e) {
    return c(a.x * b.x + a.y * b.y + d.x * e.x + d.y * e.y, a.x * b.y - a.y * b.x + d.x * e.y - d.y * e.x);
  };
  auto dot = [&](C a, C b, C d, C e) {
    return c(a.x * b.x - a.y * b.y + d.x * e.x - d.y * e.y, a.x * b.y + a.y * b.x + d.x * e.y + d.y * e.x);
  };
  auto norm = [](C a) { return a.x * a.x + a.y * a.y; };
  // T = G_0+ G_1.  Its traceless part is a phase times n . sigma with a real n; the phase is read off its
  // largest component.
  const C t0 = dotc(g0[0], g1[0], g0[2], g1[2]), t1 = dotc(g0[0], g1[1], g0[2], g1[3]);
  const C t2 = dotc(g0[1], g1[0], g0[3], g1[2]), t3 = dotc(g0[1], g1[1], g0[3], g1[3]);
  const R half = (R)0.5;
  const C vz = c(half * (t0.x - t3.x), half * (t0.y - t3.y)), vx = c(half * (t1.x + t2.x), half * (t1.y + t2.y));
  const C vy = c(-half * (t1.y - t2.y), half * (t1.x - t2.x));
  const R lx = norm(vx), ly = norm(vy), lz = norm(vz);
  const C ph = lx < ly ? (ly < lz ? vz : vy) : (lx < lz ? vz : vx);
  R nx = vx.x * ph.x + vx.y * ph.y, ny = vy.x * ph.x + vy.y * ph.y, nz = vz.x * ph.x + vz.y * ph.y;
  const R len2 = nx * nx + ny * ny + nz * nz;
  R p = 1;
  C q = c(0, 0);
  if (len2 > (R)1e-280) {   // (else T is a phase: any basis)
    const R k0 = 1 / std::sqrt(len2), s = nz < 0 ? -k0 : k0;
    nx *= s;
    ny *= s;
    nz *= s;
    const R k = 1 / std::sqrt(2 * (1 + nz));
    p = (1 + nz) * k;
    q = c(nx * k, ny * k);
  }
  const C s0 = c(p, 0), s1 = c(-q.x, q.y), s2 = q;   // S = [[s0, s1], [s2, s0]], columns the eigenvectors
  sh[0] = s0;
  sh[1] = c(q.x, -q.y);
  sh[2] = c(-q.x, -q.y);
  sh[3] = s0;
  for (int r = 0; r < 2; ++r) {
    a0[2 * r] = dot(g0[2 * r], s0, g0[2 * r + 1], s2);
    a0[2 * r + 1] = dot(g0[2 * r], s1, g0[2 * r + 1], s0);
    a1[2 * r] = dot(g1[2 * r], s0, g1[2 * r + 1], s2);
    a1[2 * r + 1] = dot(g1[2 * r], s1, g1[2 * r + 1], s0);
  }
  // lambda: the eigenvectors' products with T, A_0+ A_1
  lam[0] = dotc(a0[0], a1[0], a0[2], a1[2]);
  lam[3] = dotc(a0[1], a1[1], a0[3], a1[3]);
  lam[1] = lam[2] = c(0, 0);
}

}  // namespace qec
