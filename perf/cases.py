"""The work that users of this library have it do, as timed cases.

A case is one call of a public entry point: `Simulator.run` (a handle of one register, trajectories
with host outputs), the same after `Simulator.reconfigure` (what a job server does for every job) or
`BatchSimulator.run` (many d = 3 trajectories with their own precision and noise).  Fields:
  form        "sim" | "job" | "batch"
  code, d     "surface" 3 or 5, "repetition" odd 9..25 (registers of 9 to 25 data qubits)
  rounds, n   noisy rounds and trajectories of one call
  gates, precision
  noise       which coherent terms are on (see `noise_of`), p the depolarizing rate, theta the angle
  state       also read the final state (Simulator.state, BatchSimulator.state)
  kinds       batch: the registers and precisions that are mixed
"""
import math
import random

import numpy as np

from paper_2204_11404_gb300.simulator import BatchSimulator, Simulator

KINDS = {"mix": ("c128", "c64", "c128u", "c64u"), "reduced": ("c128", "c64"), "c64": ("c64",), "unreduced": ("c128u", "c64u")}


def sim(name, code, d, rounds, n, gates, precision, noise="cr", p=3e-3, theta=0.01, state=False, form="sim"):
    return {"name": name, "form": form, "code": code, "d": d, "rounds": rounds, "n": n, "gates": gates,
            "precision": precision, "noise": noise, "p": p, "theta": theta, "state": state}


def batch(name, rounds, n, kinds, gates="cr", state=False):
    return {"name": name, "form": "batch", "rounds": rounds, "n": n, "kinds": kinds, "gates": gates, "state": state}


def listed():
    return [
        # one trajectory of the smallest register: the latency of a call
        sim("d3_one", "surface", 3, 3, 1, "cnot", "c128", "round", p=1e-3, theta=0.02),
        # a logical error rate of the d = 3 code: 1000 trajectories of one noise point
        sim("d3_thousand", "surface", 3, 3, 1000, "cnot", "c128", "round", p=1e-3, theta=0.02),
        # a served d = 3 job: new noise and rounds on a resident handle, then its trajectories
        sim("d3_job", "surface", 3, 7, 37, "cr", "c64", "plain", p=4e-3, theta=0.06, form="job"),
        # one d = 5 trajectory (26-qubit register, five rounds) in each form, the default first
        sim("d5_c128tc", "surface", 5, 5, 1, "cr", "c128tc"),
        sim("d5_c64tc", "surface", 5, 5, 1, "cr", "c64tc"),
        sim("d5_c64", "surface", 5, 5, 1, "cr", "c64"),
        sim("d5_c128", "surface", 5, 5, 1, "cr", "c128"),
        # the repetition code at the largest register, and at a middle and a small one whose
        # final state is studied too
        sim("rep25_c128tc", "repetition", 25, 5, 1, "cr", "c128tc"),
        sim("rep17_c64", "repetition", 17, 5, 6, "cr", "c64", "all", theta=0.05),
        sim("rep13_c128_state", "repetition", 13, 4, 1, "cr", "c128", "all", theta=0.05, state=True),
        # the batched form: its full mix, and a small batch of the 10-qubit registers
        batch("batch_mix_8192", 3, 8192, "mix"),
        batch("batch_reduced_301", 5, 301, "reduced", state=True),
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["d3", "d3", "d5", "rep", "rep", "batch"])
    gates = rng.choice(["cr", "cr", "cnot"])
    noise = rng.choice(["cr", "plain", "all", "round", "sweep", "twirl"])
    p, theta = math.exp(rng.uniform(math.log(5e-4), math.log(1e-2))), rng.uniform(0.0, 0.1)
    if what == "batch":
        kinds, rounds = rng.choice(["mix", "reduced", "c64", "unreduced"]), rng.randint(1, 6)
        n = log_int(rng, 16, 8192 * 3 // rounds // (4 if kinds == "unreduced" else 2))
        return {k: v for k, v in batch("", rounds, n, kinds, gates, rng.random() < 0.3).items() if k != "name"}
    precision = rng.choice(["c128", "c64", "c64tc", "c128tc"])
    if what == "d3":
        rounds = rng.randint(1, 10)
        c = sim("", "surface", 3, rounds, log_int(rng, 1, 2000 // rounds), gates, precision, noise, p, theta, rng.random() < 0.5,
                rng.choice(["sim", "job"]))
    elif what == "d5":
        rounds = rng.randint(1, 4)
        c = sim("", "surface", 5, rounds, rng.randint(1, 4 // rounds), gates, precision, noise, p, theta)
    else:
        d, rounds = rng.randrange(9, 26, 2), rng.randint(1, 6)
        if d == 25:
            rounds = min(rounds, 4)
        most = max(1, min(64, 2 ** (25 - d) * 4 // rounds))
        c = sim("", "repetition", d, rounds, log_int(rng, 1, most), gates, precision, noise, p, theta, d <= 13 and rng.random() < 0.5)
    return {k: v for k, v in c.items() if k != "name"}


def noise_of(c):
    """Depolarizing rate p on every step (one-qubit gates, two-qubit gates, waits; "round": gates
    only) and the coherent terms: "cr" Rx over-rotation and ZZ crosstalk, "plain" Rx over-rotation,
    "sweep" one over-rotation angle after every rotation gate, "all" every term, "round" an Rz on
    every data qubit per round, "twirl" the Pauli twirl of "sweep"."""
    p, th = c["p"], c["theta"]
    nz = {"p1": p, "p2": p, "p_idle": p}
    if c["noise"] == "round":
        return {"p1": p, "p2": p, "round_rz": th}
    if c["noise"] in ("sweep", "twirl"):
        return dict(nz, theta_rx=th, theta_rz=th, theta_rzx=th, twirl=float(c["noise"] == "twirl"))
    if c["noise"] == "all":
        return dict(nz, theta_rx=th, theta_rz=th, theta_rzx=th, phi_zz=0.02, round_rz=th / 2, round_rx=th / 2)
    return dict(nz, theta_rx=th, phi_zz=0.02) if c["noise"] == "cr" else dict(nz, theta_rx=th)


def batch_inputs(c, seed):
    """Trajectory indices, kinds (interleaved) and each trajectory's own noise."""
    rng = np.random.default_rng(seed)
    p, th = rng.uniform(1e-4, 1e-2, c["n"]), rng.uniform(0.0, 0.1, c["n"])
    kinds = [KINDS[c["kinds"]][i % len(KINDS[c["kinds"]])] for i in range(c["n"])]
    first = int(rng.integers(0, 1 << 20))
    noise = [dict(p1=a, p2=a, p_idle=a, theta_rx=b) for a, b in zip(p.tolist(), th.tolist())]
    return list(range(first, first + c["n"])), kinds, noise


def prepare(case, seed):
    if case["form"] == "batch":
        traj, kinds, noise = batch_inputs(case, seed)
        return case, seed, BatchSimulator(case["rounds"], case["gates"], max_traj=case["n"]), (traj, kinds, noise)
    nz = noise_of(case)
    h = Simulator(case["d"], case["rounds"], case["gates"], case["precision"], code=case["code"],
                  **(nz if case["form"] == "sim" else {}))
    return case, seed, h, nz


def run(state):
    case, seed, h, inputs = state
    if case["form"] == "batch":
        if case["state"]:
            h.snapshot(case["n"] - 1)
        syn, bits, logical = h.run(seed, *inputs)
    else:
        if case["form"] == "job":
            h.reconfigure(case["rounds"], **inputs)
        syn, bits, logical = h.run(seed, 3 * seed, case["n"])
    out = {"syndromes": syn, "data_bits": bits, "raw_logical": logical}
    if case["state"]:
        out["state"] = h.state()
    return out


def geometry(case):
    """Data qubits and the weights of one round's stabilizers."""
    if case["form"] == "batch":
        return 9, [2] * 4 + [4] * 4
    d = case["d"]
    if case["code"] == "repetition":
        return d, [2] * (d - 1)
    return d * d, [2] * (2 * (d - 1)) + [4] * ((d - 1) * (d - 1))


def work(case):
    """Registers that outgrow the chip's shared memory: one read and one write per noisy round, since a
    round's outcomes depend on the whole register; the smaller ones stay on the chip.  Arithmetic
    per amplitude and stabilizer: one rotation per qubit of the stabilizer, one complex factor (the
    collapse) and one square."""
    nd, weights = geometry(case)
    amps, traj = 1 << nd, case["n"] * case["rounds"]
    flops = amps * traj * sum(4 * w + 10 for w in weights)
    out = case["n"] * ((case["rounds"] + 1) * len(weights) + nd + 1) + (16 * amps if case["state"] else 0)
    if case["form"] == "batch":
        return {"bytes": out + case["n"] * 100, "flops": flops}
    amp = 16 if case["precision"].startswith("c128") else 8
    return {"bytes": out + (2 * amp * amps * traj if amps * amp > (32 << 20) else 0), "flops": flops}


# ---- the final state in 64 bits, gate by gate (registers of up to 13 data qubits) ---------------------

def philox(counter, seed):
    mask = (1 << 64) - 1
    c0, c1, c2, c3 = (x & mask for x in counter)
    k0, k1 = seed & mask, 0
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B97F4A7C15) & mask, (k1 + 0xBB67AE8584CAA73B) & mask
        a, b = 0xD2E7470EE14C6C93 * c0, 0xCA5A826395121157 * c2
        c0, c1, c2, c3 = (b >> 64) ^ c1 ^ k0, b & mask, (a >> 64) ^ c3 ^ k1, a & mask
    return c0, c1


PAULI = [np.eye(2, dtype=complex), np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]]),
         np.diag([1.0 + 0j, -1.0])]
X, Z = PAULI[1], PAULI[3]


def rot(a, angle):
    return math.cos(angle / 2) * np.eye(len(a)) - 1j * math.sin(angle / 2) * a


class Exact:
    """One trajectory on the data qubits and one reused ancilla (bit nd)."""

    def __init__(self, code, d, rounds, gates, noise, seed, traj):
        self.cr, self.seed, self.traj = gates == "cr", seed, traj
        self.nz = dict({k: 0.0 for k in ("p1", "p2", "p_idle", "theta_rx", "theta_rz", "theta_rzx", "phi_zz", "round_rz",
                                         "round_rx", "twirl")}, **noise)
        self.stabs = []
        if code == "repetition":
            self.nd = d
            self.stabs = [("Z", [k + 1, k, None, None]) for k in range(d - 1)]
        else:
            self.nd = d * d
            at = lambda r, c: r * d + c if 0 <= r < d and 0 <= c < d else None  # noqa: E731
            found = {"X": [], "Z": []}
            for r in range(-1, d):
                for c in range(-1, d):
                    tl, tr, bl, br = at(r, c), at(r, c + 1), at(r + 1, c), at(r + 1, c + 1)
                    kind = "X" if (r + c) % 2 else "Z"
                    w = sum(q is not None for q in (tl, tr, bl, br))
                    edge = (r in (-1, d - 1)) if kind == "X" else (c in (-1, d - 1))
                    if w == 4 or (w == 2 and edge):
                        found[kind].append(((r, c), [br, bl, tl, tr]) if kind == "X" else ((c, -r), [tr, br, bl, tl]))
            for kind in "XZ":
                self.stabs += [(kind, slots) for _, slots in sorted(found[kind], key=lambda e: e[0])]
        self.n_of = {k: [sum(q in s for kk, s in self.stabs if kk == k) for q in range(self.nd)] for k in "XZ"}
        self.psi = np.zeros(2 << self.nd, complex)
        self.psi[0] = 1.0
        for rnd in range(rounds + 1):
            self.round(rnd)

    def uniform(self, rnd, step, site, tag):
        w = philox((self.traj, rnd, (step << 32) | site, tag), self.seed)
        return (w[0] >> 11) * 2.0 ** -53, w[1] >> 32

    def one(self, q, m):
        v = self.psi.reshape(-1, 2, 1 << q)
        self.psi = np.einsum("ab,xby->xay", m, v).reshape(-1)

    def two(self, a, b, m):
        """m on the local index 2 bit(a) + bit(b)."""
        hi, lo = max(a, b), min(a, b)
        v = self.psi.reshape(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
        t = m.reshape(2, 2, 2, 2)   # out a, out b, in a, in b
        self.psi = np.einsum("abcd,xcydz->xaybz" if a > b else "abcd,xdycz->xbyaz", t, v).reshape(-1)

    def pauli1(self, rnd, step, site, q, p):
        if rnd and p > 0:
            u, k = self.uniform(rnd, step, site, 0)
            if u < p:
                self.one(q, PAULI[(k * 3 >> 32) + 1])

    def term(self, rnd, step, site, factor, qs, a, angle, full=False):
        """exp(-i angle/2 a), or twirled a itself with its probability (`full`: exp(-i angle a))."""
        angle = 2 * angle if full else angle
        if not rnd or not angle:
            return
        if not self.nz["twirl"]:
            m = rot(a, angle)
        elif self.uniform(rnd, step, factor << 24 | site, 4)[0] < math.sin(angle / 2) ** 2:
            m = a
        else:
            return
        self.one(qs[0], m) if len(qs) == 1 else self.two(qs[0], qs[1], m)

    def data_step(self, rnd, q, t):
        nz = self.nz
        if t == 0:
            self.term(rnd, t, q, 6, [q], Z, nz["round_rz"])
            self.term(rnd, t, q, 7, [q], X, nz["round_rx"])
        elif self.cr and t in (6, 11):
            a, angle, times = (X, nz["theta_rx"], self.n_of["X"][q]) if t == 6 else (Z, nz["theta_rz"], self.n_of["Z"][q])
            for f in range(times):
                self.one(q, rot(a, math.pi / 2))
                self.term(rnd, t, q, f, [q], a, angle)
            self.pauli1(rnd, t, q, q, nz["p1"] if times else nz["p_idle"])
        else:
            self.pauli1(rnd, t, q, q, nz["p_idle"])

    def round(self, rnd):
        nz, nd, clock = self.nz, self.nd, [-1] * self.nd

        def until(q, t):
            for s in range(clock[q] + 1, t + 1):
                self.data_step(rnd, q, s)
            clock[q] = t

        for part, steps in (("X", range(1, 7)), ("Z", range(7, 12))):
            for k, (kind, slots) in enumerate(self.stabs):
                if kind != part:
                    continue
                for t in steps:
                    if kind == "X" and t in (1, 6):
                        if self.cr:
                            self.one(nd, rot(X, -math.pi / 2 if t == 1 else math.pi / 2))
                            self.term(rnd, t, nd + k, 0, [nd], X, nz["theta_rx"])
                        else:
                            self.one(nd, (X + Z) / math.sqrt(2))
                        self.pauli1(rnd, t, nd + k, nd, nz["p1"])
                        continue
                    q = None if t == 11 else slots[t - 2 if kind == "X" else t - 7]
                    if q is None:
                        self.pauli1(rnd, t, nd + k, nd, nz["p_idle"])
                        continue
                    until(q, t - 1)
                    clock[q] = t
                    pair = [nd, q] if kind == "X" else [q, nd]
                    if self.cr:
                        self.two(*pair, rot(np.kron(Z, X), math.pi / 2))
                        self.term(rnd, t, q, 4, pair, np.kron(Z, X), nz["theta_rzx"])
                    else:
                        self.two(*pair, np.eye(4)[[0, 1, 3, 2]].astype(complex))
                    self.term(rnd, t, q, 5, pair, np.kron(Z, Z), nz["phi_zz"], full=True)
                    if rnd and nz["p2"] > 0:
                        u, w = self.uniform(rnd, t, q, 0)
                        if u < nz["p2"]:
                            c = (w * 15 >> 32) + 1
                            self.one(nd, PAULI[c >> 2])
                            self.one(q, PAULI[c & 3])
                self.measure(rnd, k, slots)
            for q in range(nd):
                until(q, 6 if part == "X" else 11)

    def measure(self, rnd, k, slots):
        v = self.psi.reshape(2, -1)
        p = [float(np.vdot(x, x).real) for x in v]
        if rnd:
            m = int(self.uniform(rnd, 0, self.nd + k, 1)[0] < p[1] / (p[0] + p[1]))
        else:
            m = int(self.cr and sum(q is not None for q in slots) == 2)
        self.psi = np.concatenate([v[m] / math.sqrt(p[m]), np.zeros_like(v[0])])


def exact(case, seed):
    if not case["state"]:
        return None
    if case["form"] == "batch":
        traj, _, noise = batch_inputs(case, seed)
        e = Exact("surface", 3, case["rounds"], case["gates"], noise[-1], seed, traj[-1])
    else:
        e = Exact(case["code"], case["d"], case["rounds"], case["gates"], noise_of(case), seed, 3 * seed + case["n"] - 1)
    return {"syndromes": None, "data_bits": None, "raw_logical": None, "state": e.psi[: 1 << e.nd]}


if __name__ == "__main__":
    for c in listed() + [draw(random.Random(7)) for _ in range(3)]:
        print(c, work(c))
