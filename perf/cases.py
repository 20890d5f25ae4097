"""Performance cases of the Parallel-Tempering engine: the calls a simulation program makes, over the sizes it
makes them at.

Every case goes through the public binding (`PT`, `fmc_graph`).  A pass advances an ensemble by some sweeps, or
recomputes its energies, or trains / applies the learned proposal, and returns what the call leaves behind: all
amplitudes, all energies, the accumulators, the network parameters.

Two notes on values:

- A Metropolis chain is chaotic: one decision taken differently changes everything after it.  FP32 fields carry a
  relative rounding error of about 1e-7, and about one decision in 5e7 lies that close to its threshold.  The FP32
  passes therefore take at most a few hundred thousand decisions, from a start that does not depend on the sweep
  kernel (the exact beta = 0 draws that a new ensemble begins with).
- The ABI widens everything to FP64.  Energies of an FP32 ensemble hold FP32 sums, so they are returned in FP32
  (FP64 ones in FP64).  Amplitudes never pass through a sum and are returned as they come.

`exact` is the plain FP64 restatement: Philox4x32-10 counters, pair moves by recomputing every quadruplet that
holds a moved mode, swaps of configurations.  It uses none of the engine's code.
"""
import math

import numpy as np
import torch

import paper_2511_13508_gb300 as pt
from paper_2511_13508_gb300 import workload

DECISIONS = 1 << 17  # pair decisions of a drawn FP32 pass


def listed():
    return [
        # The smallest ensemble of the repository's workloads (n16_fp64): one swap interval of the FP64 path with its
        # measurements, resync and swap pass; a test run, or the exact check beside an FP32 run.
        dict(name="n16_fp64_interval", kind="comb", precision="fp64", N=16, S=4, nT=8, R=2, t_min=0.4, sweeps=64, observe=True),
        # One disorder sample at the smallest size of the paper's production runs (N = 18: 42 temperatures, 4
        # replicas), one swap interval: little work per update, so launches and latency count.
        dict(name="n18_sample_interval", kind="comb", precision="fp32", N=18, S=1, nT=42, R=4, t_min=0.3, sweeps=64, observe=True),
        # Batched disorder average at the middle size (n64_batched): the throughput workload.
        dict(name="n64_batch", kind="comb", precision="fp32", N=64, S=64, nT=32, R=2, t_min=0.3, sweeps=2, observe=False),
        # Samples of different sizes in one launch, as finite-size scaling wants them (ragged).
        dict(name="ragged_batch", kind="ragged", precision="fp32", N=128, S=96, nT=24, R=2, t_min=0.3, sweeps=1, observe=False),
        # The largest workload (n256_large): the headline benchmark's ensemble.
        dict(name="n256_batch", kind="comb", precision="fp32", N=256, S=16, nT=48, R=2, t_min=0.25, sweeps=2, observe=False),
        # One disorder sample at the largest size: what a user has who looks at a single sample.
        dict(name="n256_sample", kind="comb", precision="fp32", N=256, S=1, nT=48, R=2, t_min=0.25, sweeps=4, observe=False),
        # The FP64 path at the middle size: the precision reference of the FP32 runs.
        dict(name="n64_fp64", kind="comb", precision="fp64", N=64, S=16, nT=32, R=2, t_min=0.3, sweeps=2, observe=False),
        # The paper's own graph: random frequencies, matching condition with a linewidth (benchmark leg random_graph).
        dict(name="random_graph_n64", kind="random", precision="fp32", N=64, S=16, nT=32, R=2, t_min=0.3, sweeps=4, observe=False),
        # A sparse mode-locked graph at the largest mode count the engine takes (benchmark leg sparse_n2048_z16).
        dict(name="sparse_n2048", kind="sparse", precision="fp32", N=2048, S=4, nT=32, R=2, z=16, t_min=0.3, sweeps=1, observe=False),
        # Full recomputation of every chain's energy: the resync of a run, and the check of a restored state.
        dict(name="n256_energy", kind="energy", precision="fp32", N=256, S=8, nT=48, R=2, t_min=0.25),
        # Learned proposal: training steps on collected configurations (n64_learned).
        dict(name="n64_train", kind="train", N=64, S=16, n_cold=8, R=2, batch=512, steps=4),
        # Learned proposal in use: sweeps with a round of global moves at their end (n64_learned, every 8 sweeps
        # there).
        dict(name="n64_global_moves", kind="global", precision="fp32", N=64, S=16, nT=32, R=2, t_min=0.3, n_cold=8, sweeps=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(n):
    return max(4, n - n % 2)


def _ensemble(rng, N, most_samples, decisions):
    """Samples, temperatures, replicas and sweeps with about `decisions` pair decisions at most."""
    nT, R = rng.randint(8, 48), rng.choice((1, 2, 2, 3, 4))
    room = max(1, decisions // (nT * R * (N // 2)))
    S = _log_int(rng, 1, max(1, min(most_samples, room)))
    sweeps = max(1, min(64, decisions // (S * nT * R * (N // 2))))
    return dict(N=N, S=S, nT=nT, R=R, t_min=round(rng.uniform(0.2, 0.5), 3), sweeps=sweeps)


def draw(rng):
    """Ensembles of the listed kinds, sizes spread over their logarithm, odd group counts and sizes among them."""
    kind = rng.choice(("comb", "comb", "comb", "ragged", "fp64", "random", "sparse", "energy", "train", "global"))
    D = _log_int(rng, DECISIONS // 16, DECISIONS)
    if kind == "comb":
        N = _even(_log_int(rng, 16, 256))
        return dict(kind="comb", precision="fp32", observe=rng.random() < 0.5, **_ensemble(rng, N, min(64, 65536 // (N * N) * 8 + 8), D))
    if kind == "ragged":
        e = _ensemble(rng, _even(_log_int(rng, 48, 160)), 64, D)
        e["S"] = max(2, e["S"])
        return dict(kind="ragged", precision="fp32", observe=False, **e)
    if kind == "fp64":
        N = _even(_log_int(rng, 16, 64))
        e = _ensemble(rng, N, 32, D // 8)
        return dict(kind="comb", precision="fp64", observe=rng.random() < 0.5, **e)
    if kind == "random":
        return dict(kind="random", precision="fp32", observe=rng.random() < 0.5, **_ensemble(rng, _even(_log_int(rng, 16, 96)), 24, D))
    if kind == "sparse":
        return dict(kind="sparse", precision="fp32", observe=False, z=rng.randint(8, 24), **_ensemble(rng, _even(_log_int(rng, 256, 2048)), 8, D))
    if kind == "energy":
        N = _even(_log_int(rng, 16, 256))
        e = _ensemble(rng, N, min(64, 65536 // (N * N) * 8 + 8), 4 * D)
        del e["sweeps"]
        return dict(kind="energy", precision=rng.choice(("fp32", "fp32", "fp64")) if N <= 64 else "fp32", **e)
    N = rng.choice((16, 32, 48, 64))
    if kind == "train":
        return dict(kind="train", N=N, S=rng.randint(1, 16), n_cold=rng.randint(2, 8), R=rng.choice((1, 2, 4)), batch=rng.choice((128, 256, 512)), steps=rng.randint(1, 4))
    e = _ensemble(rng, N, 16, D)
    e["sweeps"] = min(8, e["sweeps"])
    return dict(kind="global", precision=rng.choice(("fp32", "fp32", "fp64")) if N == 16 else "fp32", n_cold=rng.randint(2, min(8, e["nT"])), **e)


# ---------------------------------------------------------------------------------------------- inputs
def _rng(seed, *more):
    return np.random.Generator(np.random.PCG64([int(seed) & 0x7FFFFFFF, *more]))


def _sizes(case):
    if case["kind"] != "ragged":
        return [case["N"]] * case["S"]
    # sizes between a quarter of the largest and the largest (32, 48, 64, 96, 128 for the listed case)
    top = case["N"]
    choices = sorted({_even(top * k // 8) for k in (2, 3, 4, 6, 8)})
    sizes = [choices[i] for i in _rng(case["S"], 1).integers(0, len(choices), size=case["S"])]
    sizes[0] = top
    return sizes


def _sparse_graph(N, z, rng):
    """round(z N / 4) quadruplets of the comb, uniformly without replacement (workload.sparse_comb_graph's law)."""
    M = int(round(z * N / 4))
    got = np.zeros((0, 4), np.int64)
    while len(got) < M:
        x = np.sort(rng.integers(0, N, size=(16 * M, 3)), axis=1)
        d = x[:, 1] + x[:, 2] - x[:, 0]
        ok = (x[:, 0] < x[:, 1]) & (x[:, 1] < x[:, 2]) & (d < N)
        got = np.unique(np.concatenate([got, np.column_stack([x[ok], d[ok]])]), axis=0)
    return got[np.sort(rng.permutation(len(got))[:M])].astype(np.int32)


def _couplings(case, seed, s, n, N):
    g = _rng(seed, 2, s).standard_normal(n)
    return g if case["kind"] == "sparse" else g / N  # sigma_J = 1 at finite connectivity, 1/N otherwise


def _temps(case):
    return workload.geometric_ladder(case["t_min"], 1.6, case["nT"])


def _configurations(rng, shape, N):
    """Configurations on the constraint surface with a wide spread of intensities."""
    g = rng.standard_normal((*shape, N))
    s = g * g / (g * g).sum(-1, keepdims=True)
    return (N * s) ** 0.25 * np.exp(2j * np.pi * rng.random((*shape, N)))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        N, S, R, nT = case["N"], case["S"], case["R"], case["n_cold"]
        n = len(pt.enumerate_quads(N))
        sim = pt.PT([N] * S, [_couplings(case, seed, s, n, N) for s in range(S)], workload.geometric_ladder(0.3, 1.6, nT), R, seed)
        sim.learn_init(n_cold=nT, batch=case["batch"], data_per_sample=1 << 12, seed=seed)
        rng = _rng(seed, 3)
        for _ in range(16):  # collected configurations, here given ones: nT * R rows per sample each time
            sim.set_state(_configurations(rng, (S * R * nT,), N).reshape(-1))
            sim.collect(0, 1)
        return dict(case, sim=sim)
    sizes = _sizes(case)
    if kind == "random":
        graphs = [pt.fmc_graph(workload.random_frequencies(N, int(seed) % (1 << 30) + s)) for s, N in enumerate(sizes)]
    elif kind == "sparse":
        graphs = [_sparse_graph(N, case["z"], _rng(seed, 4, s)) for s, N in enumerate(sizes)]
    else:
        graphs = None
    counts = [len(g) for g in graphs] if graphs else None
    if counts is None:
        by = {N: len(pt.enumerate_quads(N)) for N in set(sizes)}
        counts = [by[N] for N in sizes]
    J = [_couplings(case, seed, s, n, N) for s, (n, N) in enumerate(zip(counts, sizes))]
    sim = pt.PT(sizes, J, _temps(case), case["R"], int(seed), precision=case["precision"], graphs=graphs)
    if kind == "global":
        sim.learn_init(n_cold=case["n_cold"], batch=128, data_per_sample=1 << 10, seed=seed)
        sim.set_global_every(case["sweeps"])
    return dict(case, sim=sim)


def run(state):
    sim, kind = state["sim"], state["kind"]
    if kind == "train":
        losses = sim.train(state["steps"], lr=1e-3)
        return dict(losses=losses.astype(np.float32), parameters=sim.learn_params())
    fp32 = state["precision"] == "fp32"
    if kind == "energy":
        E = sim.energy()
        return dict(E=E.astype(np.float32) if fp32 else E)
    sim.sweep(state["sweeps"])
    a, E = sim.state()
    out = dict(a=a, E=E.astype(np.float32) if fp32 else E)
    if kind == "global" or state["observe"]:
        for k, v in sim.observables().items():
            out[k] = v.astype(np.float32) if fp32 and v.dtype == np.float64 else v.astype(np.int64) if v.dtype == np.uint64 else v
    return out


# ---------------------------------------------------------------------------------------------- work
def _comb_count(N):
    return sum(m * (m - 1) // 2 for m in ((s + 1) // 2 - max(0, s - N + 1) for s in range(1, 2 * N - 2)))


def work(case):
    """A pair update needs the coupling terms of its two modes: 4 |Q| per chain-sweep on average, each a real coupling
    times a complex pair product (4 flops, and 3 for its share of the product, which serves both fields).
    Couplings are read once, amplitudes and energies read and written once."""
    if case["kind"] == "train":
        N, S = case["N"], case["S"]
        P = 256 * 3 * N + 256 * (case["n_cold"] + 2) + 256 * 256 + 4 * N * 257
        return dict(bytes=24 * P * S + 4 * S * case["batch"] * 2 * N * case["steps"], flops=6 * P * case["batch"] * S * case["steps"])
    z = 4 if case.get("precision") == "fp32" else 8
    sizes = _sizes(case)
    Q = sum(round(case["z"] * N / 4) if case["kind"] == "sparse" else _comb_count(N) for N in sizes) / len(sizes)
    N, chains = sum(sizes) / len(sizes), case["nT"] * case["R"]
    if case["kind"] == "energy":
        return dict(bytes=case["S"] * (z * Q + chains * (2 * z * N + 8)), flops=case["S"] * chains * Q * 7)
    flops = case["S"] * chains * case["sweeps"] * 4 * Q * 7
    if case["kind"] == "global":  # forward passes: both configurations, and 8 mode blocks of the sampler
        P = 256 * 3 * N + 256 * 256 + 4 * N * 256
        flops += 2 * P * case["S"] * case["n_cold"] * case["R"] * 10 + 2 * 9 * Q * case["S"] * case["n_cold"] * case["R"]
    return dict(bytes=case["S"] * (z * Q + chains * 2 * (2 * z * N + 8)), flops=flops)


# ---------------------------------------------------------------------------------------------- exact
def _philox(seed, c0, c1, c2, tag):
    """Philox4x32-10 words [4, ...] of the counters (c0, c1, c2, tag) under the key `seed`."""
    c0, c1, c2 = (np.asarray(c, np.uint64) for c in (c0, c1, c2))
    shape = np.broadcast_shapes(c0.shape, c1.shape, c2.shape)
    x = [np.broadcast_to(c, shape).astype(np.uint64) for c in (c0, c1, c2)] + [np.full(shape, tag, np.uint64)]
    low, sh = np.uint64(0xFFFFFFFF), np.uint64(32)
    k0, k1 = int(seed) & 0xFFFFFFFF, (int(seed) >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * x[0], np.uint64(0xCD9E8D57) * x[2]
        x = [(p1 >> sh) ^ x[1] ^ np.uint64(k0), p1 & low, (p0 >> sh) ^ x[3] ^ np.uint64(k1), p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return np.stack(x)


def _u01(w):
    return (w.astype(np.float64) + 0.5) / 4294967296.0


def _comb(N):
    out = []
    for a in range(N):
        for b in range(a + 1, N):
            c = np.arange(b + 1, N - (b - a))
            if len(c):
                out.append(np.column_stack([np.full_like(c, a), np.full_like(c, b), c, b + c - a]))
    return np.concatenate(out) if out else np.zeros((0, 4), np.int64)


def _matching(w):
    """Random-frequency graph: every splitting of every 4-subset that meets the matching condition."""
    N = len(w)
    gamma, out = 1.0 / (2 * (N - 1)), []
    for a in range(N):
        i, j, k = (x.reshape(-1) for x in np.meshgrid(*[np.arange(a + 1, N)] * 3, indexing="ij"))
        ok = (i < j) & (j < k)
        i, j, k = i[ok], j[ok], k[ok]
        rows = []
        for n, (p, u, v, q) in enumerate(((a, i, j, k), (a, j, k, i), (a, i, k, j))):
            hit = np.abs(w[p] + w[q] - w[u] - w[v]) < gamma
            full = np.broadcast_arrays(p, u, v, q)
            rows.append(np.column_stack([f[hit] for f in (*full, i, j, k)] + [np.full(hit.sum(), n)]))
        rows = np.concatenate(rows)
        out.append(rows[np.lexsort((rows[:, 7], rows[:, 6], rows[:, 5], rows[:, 4]))][:, :4])
    return np.concatenate(out)


class _Sample:
    """One disorder sample in FP64: configurations [N, R * nT] in (r, t) order."""

    def __init__(self, s, N, quads, J, temps, R, seed, dev):
        self.s, self.N, self.R, self.nT, self.seed, self.dev = s, N, R, len(temps), int(seed), dev
        self.q = torch.from_numpy(np.ascontiguousarray(quads, np.int64)).to(dev)
        self.J = torch.from_numpy(J).to(dev)
        self.beta_np = 1.0 / temps
        self.beta = torch.from_numpy(np.tile(self.beta_np, R)).to(dev)
        order = np.argsort(quads.reshape(-1), kind="stable")
        at = np.searchsorted(quads.reshape(-1)[order], np.arange(N + 1))
        self.inc = [torch.from_numpy(order[at[i]:at[i + 1]] // 4).to(dev) for i in range(N)]
        self.cid = s * R * self.nT + np.arange(R * self.nT)
        w = _philox(seed, self.cid[None, :], np.arange(N)[:, None], 0, 1)
        g = np.sqrt(-2 * np.log(_u01(w[0]))) * np.cos(2 * np.pi * _u01(w[1]))
        u = math.sqrt(N) * np.abs(g) / np.linalg.norm(g, axis=0)
        self.a = torch.from_numpy(np.sqrt(u) * np.exp(2j * np.pi * _u01(w[2]))).to(dev)
        self.acc = np.zeros(R * self.nT, np.int64)
        self.E = self.energy()

    def terms(self, a, q):
        return ((a[q[:, 0]].conj() * a[q[:, 1]]) * (a[q[:, 2]] * a[q[:, 3]].conj())).real

    def energy(self):
        E = torch.zeros(self.a.shape[1], dtype=torch.float64, device=self.dev)
        for i in range(0, len(self.q), 1 << 16):
            E -= 2.0 * (self.J[i:i + (1 << 16)] @ self.terms(self.a, self.q[i:i + (1 << 16)]))
        return E

    def sweep(self, t):
        N, half = self.N, self.N // 2
        w = _philox(self.seed, self.s, t, np.arange(half), 2)
        j = (w[0] * np.uint64(N)) >> np.uint64(32)
        k = (j + np.uint64(1) + ((w[1] * np.uint64(N - 1)) >> np.uint64(32))) % np.uint64(N)
        p = _philox(self.seed, self.cid[None, :], t, np.arange(half)[:, None], 3)
        ph = torch.from_numpy(np.exp(2j * np.pi * _u01(p[:2]))).to(self.dev)
        th = 0.5 * np.pi * _u01(p[2])
        amp = torch.from_numpy(np.sqrt(np.stack([np.cos(th), np.sin(th)]))).to(self.dev)
        U = torch.from_numpy(_u01(p[3])).to(self.dev)
        for i, (x, y) in enumerate(zip(j.tolist(), k.tolist())):
            K = (self.a[x].abs() ** 4 + self.a[y].abs() ** 4) ** 0.25
            new = self.a.clone()
            new[x], new[y] = K * amp[0, i] * ph[0, i], K * amp[1, i] * ph[1, i]
            rest = self.inc[y]
            idx = torch.cat([self.inc[x], rest[(self.q[rest] != x).all(1)]])
            q = self.q[idx]
            dH = -2.0 * (self.J[idx] @ (self.terms(new, q) - self.terms(self.a, q)))
            ok = (dH <= 0) | (U[i] < torch.exp(-self.beta * dH))
            self.a = torch.where(ok, new, self.a)
            self.E = torch.where(ok, self.E + dH, self.E)

    def resync(self):
        self.a = self.a * (self.N / (self.a.abs() ** 4).sum(0)) ** 0.25
        self.E = self.energy()

    def measure(self, stat, qstat):
        u = self.a.abs().cpu().numpy() ** 2
        i2, i4, i8 = (u ** n for n in (1, 2, 4))
        i2, i4, i8, E = i2.sum(0), i4.sum(0), i8.sum(0), self.E.cpu().numpy()
        v = np.stack([np.ones_like(E), E, E * E, i4 / i2 ** 2, i8 / i4 ** 2, i2, i2 * i2], -1)
        stat += v.reshape(self.R, self.nT, 7).sum(0)
        a = self.a.cpu().numpy().reshape(self.N, self.R, self.nT)
        for r in range(self.R):
            for o in range(r + 1, self.R):
                q = (a[:, r].conj() * a[:, o]).real.sum(0) / self.N
                qstat += np.stack([q ** n for n in range(5)], -1)

    def swap(self, done):
        perm, E = np.arange(self.R * self.nT).reshape(self.R, self.nT), self.E.cpu().numpy()
        for r in range(self.R):
            U = _u01(_philox(self.seed, self.s * self.R + r, done, np.arange(self.nT - 1), 4)[0])
            for i in range(self.nT - 1):
                D = (self.beta_np[i] - self.beta_np[i + 1]) * (E[perm[r, i]] - E[perm[r, i + 1]])
                if D >= 0 or U[i] < math.exp(D):
                    perm[r, i], perm[r, i + 1] = perm[r, i + 1], perm[r, i]
        at = torch.from_numpy(perm.reshape(-1)).to(self.dev)
        self.a, self.E = self.a[:, at], self.E[at]


def exact(case, seed):
    """The pass in FP64.  None for the learned proposal (the network runs in BF16 by design), and for the counters of
    whole numbers."""
    if case["kind"] in ("train", "global"):
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    temps, a, E, stat, qstat = _temps(case), [], [], [], []
    cache = {}
    for s, N in enumerate(_sizes(case)):
        if case["kind"] == "random":
            w = np.sort(np.random.Generator(np.random.PCG64(int(seed) % (1 << 30) + s)).uniform(0.0, 1.0, size=N))
            quads = _matching(w)
        elif case["kind"] == "sparse":
            quads = _sparse_graph(N, case["z"], _rng(seed, 4, s)).astype(np.int64)
        else:
            quads = cache[N] = cache[N] if N in cache else _comb(N)
        x = _Sample(s, N, quads, _couplings(case, seed, s, len(quads), N), temps, case["R"], seed, dev)
        st, qs = np.zeros((case["nT"], 7)), np.zeros((case["nT"], 5))
        for t in range(case.get("sweeps", 0)):
            x.sweep(t)
            if (t + 1) % 64 == 0:
                x.resync()
            if (t + 1) % 16 == 0:
                x.measure(st, qs)
            if (t + 1) % 64 == 0 and case["nT"] > 1:
                x.swap((t + 1) // 64 - 1)
        a.append(x.a.T.reshape(-1).cpu().numpy())
        E.append(x.E.cpu().numpy())
        stat.append(st)
        qstat.append(qs)
    if case["kind"] == "energy":
        return dict(E=np.concatenate(E))
    out = dict(a=np.concatenate(a), E=np.concatenate(E))
    if case["observe"]:
        out.update(stat=np.stack(stat), qstat=np.stack(qstat))
    return out
