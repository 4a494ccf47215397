"""The factored form of the stabilizer blocks (one rotation per data qubit, then a diagonal per
outcome), compiled on the CPU by the code the device runs, against the dense Kraus blocks: the same
trajectories, outcome by outcome, for every gate set, code and noise option."""
import numpy as np
import pytest

import workloads as W
from paper_2204_11404_gb300 import capi

COHERENT = dict(theta_rx=0.3, theta_rz=0.2, theta_rzx=0.25, phi_zz=0.15, round_rz=0.2, round_rx=0.1)
NOISE = [
    {},
    dict(p1=0.2, p2=0.3, p_idle=0.2),
    dict(W.STRESS),
    dict(COHERENT, p1=0.1, p2=0.1, p_idle=0.1, overrot_follows=1),
    dict(COHERENT, twirl=1, p1=0.05, p2=0.05),
    dict(p1=1.0, p2=1.0, p_idle=1.0, theta_rx=4.0, theta_rz=-3.0, theta_rzx=2.0, phi_zz=-1.5, round_rz=3.0, round_rx=-2.5),
    dict(p1=1e-3, p2=1e-3, round_rz=0.02),
    dict(phi_zz=0.02),
]


def members(nd, q):
    """Register indices [groups][2^w] of a block's groups, bit j of the second index = data bit q[j]."""
    w = len(q)
    g = np.arange(1 << (nd - w))
    for b in sorted(q):
        g = ((g >> b) << (b + 1)) | (g & ((1 << b) - 1))
    off = np.array([sum(((l >> j) & 1) << q[j] for j in range(w)) for l in range(1 << w)])
    return g[:, None] + off[None, :]


def dense_step(psi, idx, k):
    return psi[idx] @ k.T


def factored_step(phi, idx, t, d):
    v = phi[idx].copy()
    w = idx.shape[1].bit_length() - 1
    for j in range(w):
        v = v.reshape(len(v), -1, 2, 1 << j)
        x, y = v[:, :, 0].copy(), v[:, :, 1].copy()
        v[:, :, 0] = x - np.conj(t[j]) * y
        v[:, :, 1] = y + t[j] * x
        v = v.reshape(len(v), -1)
    return v, v * d[0][: 1 << w], v * d[1][: 1 << w]


@pytest.mark.parametrize("code,d", [("surface", 3), ("repetition", 9)])
@pytest.mark.parametrize("gates", ["cr", "cnot"])
@pytest.mark.parametrize("noise", range(len(NOISE)))
def test_factored_blocks_follow_the_dense_ones(code, d, gates, noise):
    rounds, traj, seed = 3, 5, 17
    params = capi.make_params(d, rounds, gates, code=code, **NOISE[noise])
    nd = 9
    info = np.zeros((64, 6), np.int32)
    _, nb = capi.qec_debug_program(params, None, 0, info.ctypes.data, 64)
    rng = np.random.default_rng(noise)
    psi = rng.normal(size=1 << nd) + 1j * rng.normal(size=1 << nd)   # any state: K acts the same on all
    psi /= np.linalg.norm(psi)
    phi, flips = psi.copy(), 0
    worst = 0.0
    for rnd in range(1, rounds + 1):
        kraus, u = np.zeros((nb, 2, 16, 16), np.complex128), np.zeros(nb)
        capi.qec_debug_blocks(params, seed, traj, rnd, kraus.ctypes.data, u.ctypes.data)
        flips, rot, diag = capi.qec_debug_factors(params, seed, traj, rnd, flips, nb)
        assert np.abs(rot).max() <= 1 + 1e-12          # the larger entry of a column leads
        for b in range(nb):
            w = info[b, 0]
            idx = members(nd, [int(q) for q in info[b, 1:1 + w]])
            v = [dense_step(psi, idx, kraus[b, m][: 1 << w, : 1 << w]) for m in (0, 1)]
            _, f0, f1 = factored_step(phi, idx, rot[b], diag[b])
            p = [np.vdot(x, x).real for x in v]
            pf = [np.vdot(x, x).real for x in (f0, f1)]
            worst = max(worst, abs(p[0] - pf[0]), abs(p[1] - pf[1]))
            m = int(u[b] < p[1] / (p[0] + p[1]))
            psi = psi.copy()
            psi[idx] = v[m] / np.sqrt(p[m])
            phi = phi.copy()
            phi[idx] = (f0, f1)[m] / np.sqrt(pf[m])
        err = np.abs(psi - phi[np.arange(1 << nd) ^ flips]).max()
        worst = max(worst, err)
    # about 20 roundings per amplitude and block, 24 blocks, amplitudes below 1; an unlikely outcome
    # divides by its probability's root, which the draws above keep over 1e-3
    assert worst < 24 * 20 * 2.3e-16 * 30, worst


def test_every_program_factors():
    """All codes and sizes, with every noise site present: the block form holds."""
    for code, d in [("surface", 3), ("surface", 5)] + [("repetition", d) for d in range(9, 26, 2)]:
        for gates in ("cr", "cnot"):
            for tw in (0, 1):
                params = capi.make_params(d, 1, gates, code=code, twirl=tw, **W.STRESS)
                nb = (d * d if code == "surface" else d) - 1
                _, rot, diag = capi.qec_debug_factors(params, 3, 1, 1, 0, nb)
                assert np.isfinite(rot).all() and np.isfinite(diag).all()
                w = 2 if code == "repetition" else 4
                # outcome pairs are complete: |D_0|^2 + |D_1|^2 is 1 up to the rotations' cosines
                assert (np.abs(diag[:, :, : 1 << min(w, 2)]) ** 2).sum(1).max() <= 1 + 1e-12
