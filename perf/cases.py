"""The calls that a user's PTHR program makes, as measurable cases.

Every case goes through the package's public classes (`Batch`, `Group`).  A
case's "kind" says which calls one pass makes:

  emcs             `Batch.emcs`: whole elementary Monte Carlo steps
  sweep            `Batch.sweep`: local sweeps alone
  moves            `Batch.houdayer`, `Batch.measure`, `Batch.read_observables`
  autocorrelation  `Batch.reservoir_autocorrelation`
  serve            `Batch.reset_samples`, then EMCS of the whole pool
  group            `Group.emcs`: several lattice sizes together

Batches are prepared as a run has them between two calls: couplings drawn
from N(0,1) (on the 2^-18 grid, or off it as a user's own float32 file may
be), and some EMCS done, so that spins, overlaps and clusters look as they do
in a run and not as they do at a random start.
"""
import math

import numpy as np
import torch

from paper_2605_25872_gb300 import Batch, BatchConfig, Group, _lib, buffer_info

GROUP_SIZES = (6, 8, 10, 12, 16)     # lattice sizes of the serving mix
_FIELDS = ("L", "n_samples", "n_temps", "t_min", "t_max", "n_replicas", "n_res", "sweeps_per_emcs",
           "res_sweeps_per_emcs", "acu_interval", "rule", "cluster", "er_on", "acu_t_below", "spin_layout")


def listed():
    return [
        # plain PTHR of one small sample: every launch is far from filling the GPU
        dict(name="emcs-L4-plain", kind="emcs", L=4, n_samples=1, n_temps=12, sweeps_per_emcs=1, n=4, warm=64),
        # many small samples, one sweep and one cluster move per step, replayed as a graph
        dict(name="emcs-L8-batched", kind="emcs", L=8, n_samples=256, n_temps=16, n_res=0, sweeps_per_emcs=1, er_on=False,
             n=4, warm=200),
        # the same at L = 12, where each colour row is padded (6 sites in 2 words)
        dict(name="emcs-L12-batched", kind="emcs", L=12, n_samples=1024, n_temps=24, n_res=0, sweeps_per_emcs=1,
             er_on=False, n=1, warm=100),
        # the flagship: the paper's EMCS (10 sweeps, ACU, PT, ER with 240 reservoir sweeps) at L = 16
        dict(name="emcs-L16-paper", kind="emcs", L=16, n_samples=512, n_temps=32, n=1, warm=16),
        # the paper's L = 14 grid (rows of 7 sites), few samples, called without a graph
        dict(name="emcs-L14-few", kind="emcs", L=14, n_samples=20, n_temps=48, t_max=2.0, n=1, graph=False, warm=12),
        # the paper's late bins: the MicSA walker at L = 18 (rows of 9 sites), spins stored as bits
        dict(name="emcs-L18-micsa-bits", kind="emcs", L=18, n_samples=24, n_temps=72, t_max=2.0, rule="micsa",
             spin_layout="bits", n=1, warm=8),
        # heat bath and the single-cluster move on odd counts
        dict(name="emcs-L10-heatbath", kind="emcs", L=10, n_samples=37, n_temps=13, n_res=3, rule="heatbath",
             cluster="single", sweeps_per_emcs=3, res_sweeps_per_emcs=40, n=2, warm=30),
        # the largest lattice, with a user's couplings that are not on the grid
        dict(name="sweep-L24-offgrid", kind="sweep", L=24, n_samples=19, n_temps=8, n_res=2, on_grid=False,
             n_pt=10, n_sweep_res=10, warm=2),
        # cluster move, measurement with the chaos overlap and a read of the accumulators
        dict(name="moves-L12-chaos", kind="moves", L=12, n_samples=64, n_temps=24, n_res=0, er_on=False),
        # C(tau) of the reservoir at T_max
        dict(name="autocorrelation-L16", kind="autocorrelation", L=16, n_samples=64, n_temps=8, t_max=2.0,
             points=4, per_point=60, warm=2),
        # a serving pool: new requests into free slots (pre-thermalised at admission), then a chunk of EMCS
        dict(name="serve-L10-admit", kind="serve", L=10, n_samples=64, n_temps=24, first=5, count=7, pretherm=960,
             n=2, warm=12),
        # the serving mix of five sizes advanced together
        dict(name="group-mixed", kind="group", n_samples=32, n_temps=24, n=1, warm=6),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """A case of the listed ranges, no dearer than the listed L = 16 EMCS."""
    while True:
        kind = rng.choices(("emcs", "sweep", "moves", "autocorrelation", "serve", "group"), (10, 2, 3, 2, 2, 1))[0]
        c = dict(kind=kind, L=2 * rng.randint(2, 9), n_samples=_log_int(rng, 1, 1024), n_temps=rng.randint(5, 72),
                 t_max=rng.choice((1.6, 1.8, 2.0)), spin_layout=rng.choice(("bytes", "bytes", "bits")))
        if kind == "emcs":
            c.update(n=rng.randint(1, 4), warm=rng.randint(8, 24), graph=rng.random() < 0.7,
                     sweeps_per_emcs=rng.choice((1, 1, 3, 10)),
                     rule=rng.choice(("metropolis", "metropolis", "metropolis", "micsa", "heatbath")),
                     cluster=rng.choice(("acu", "acu", "acu", "single")), er_on=rng.random() < 0.6)
            c.update(n_res=rng.randint(1, 5) if c["er_on"] else 0, res_sweeps_per_emcs=rng.choice((40, 240)))
        elif kind == "sweep":
            c.update(L=2 * rng.randint(2, 12), n_res=rng.randint(1, 4), on_grid=rng.random() < 0.5,
                     n_pt=rng.randint(1, 12), n_sweep_res=rng.randint(0, 60), warm=2)
        elif kind == "moves":
            c.update(L=2 * rng.randint(2, 8), n_samples=_log_int(rng, 1, 128), n_temps=rng.randint(5, 32), n_res=0,
                     er_on=False)
        elif kind == "autocorrelation":
            c.update(n_temps=rng.randint(2, 8), points=rng.randint(1, 4), per_point=rng.randint(20, 120), warm=2)
        elif kind == "serve":
            c.update(n_samples=rng.randint(8, 128), n_temps=rng.randint(8, 32), pretherm=rng.choice((0, 240, 960)),
                     n=rng.randint(1, 4), warm=6)
            c["count"] = rng.randint(1, 8)
            c["first"] = rng.randint(0, c["n_samples"] - c["count"])
        else:
            del c["L"]
            c.update(n_samples=rng.randint(8, 48), n_temps=rng.randint(8, 32), n=rng.randint(1, 2), warm=4)
        most = {"moves": 2 * 64 * 24 * 4 * 12 ** 3 * 4.0}.get(kind, work(listed()[3])["flops"])
        if work(c)["flops"] <= most:
            return c


def _config(c, L=None):
    return BatchConfig(seed=0, **{**{k: c[k] for k in _FIELDS if k in c},
                                  **({"n_temps": c["n_temps"], "L": L} if L else {})})


def _inputs(c, L, seed):
    """Philox keys [S] and couplings [S, 3, L^3] of a batch, from the seed."""
    rng = np.random.Generator(np.random.PCG64([seed, L]))
    keys = rng.integers(0, 2 ** 63, c["n_samples"], dtype=np.uint64)
    gen = torch.Generator(device="cuda").manual_seed(seed * 64 + L)
    J = torch.randn((c["n_samples"], 3, L ** 3), dtype=torch.float64, device="cuda", generator=gen)
    if c.get("on_grid", True):
        J = (torch.round(J * 2.0 ** 18) / 2.0 ** 18).clamp_(-8.0, 8.0)
    return keys, J.to(torch.float32)


def _pair_spins(c, seed):
    """Spins of every clone [S, n_lat, V] whose replica pairs overlap in large
    domains with small islands, the overlap growing towards T_min."""
    cfg = _config(c)
    S, N, NT, L = cfg.n_samples, cfg.n_lat, cfg.n_slot, cfg.L
    gen = torch.Generator(device="cuda").manual_seed(seed * 64 + 63)

    def rand(*shape):
        return torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)

    s = rand(S, cfg.n_replicas, NT, L, L, L).sign()
    f = rand(S, cfg.n_replicas // 2, NT, L, L, L)
    for _ in range(3):                                   # smooth: domains of a few sites
        for d in (3, 4, 5):
            f = f + 0.5 * (f.roll(1, d) + f.roll(-1, d))
        f = f / f.std()
    cold = torch.linspace(1.3, 0.1, NT, device="cuda", dtype=torch.float64).view(1, 1, NT, 1, 1, 1)
    q = torch.where(f + cold < 0, -1.0, 1.0) * torch.where(rand(*f.shape) > 2.0, -1.0, 1.0)
    s[:, 1::2] = s[:, 0::2] * q
    return s.to(torch.int8).reshape(S, N, L ** 3)


def _outputs(b):
    """The batch's whole state in its own buffers."""
    off, n = buffer_info(b.cfg, _lib.BUF_SPINS)
    return {"spins": b.ws[off:off + n], "energies": b.energies, "perm": b.perm, "age": b.age,
            "round_trips": b.round_trips, "pt_accepted": b.pt_accepted, "flips": b.flips, "obs": b.obs,
            "cluster_stats": b.cluster_stats, "emcs": b.emcs_counter}


def _batch(c, L, seed):
    keys, J = _inputs(c, L, seed)
    return Batch(_config(c, L), couplings=J, seeds=keys, stream=torch.cuda.Stream())


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "group":
        batches = [_batch(c, L, seed) for L in GROUP_SIZES]
        g = Group(batches, stream=torch.cuda.Stream())
        g.emcs(c["warm"])
        g.synchronize()
        return {"case": c, "group": g, "out": [{k: _outputs(b)[k] for k in ("spins", "energies", "obs", "flips",
                                                                            "cluster_stats", "perm")}
                                               for b in batches]}
    b = _batch(c, c["L"], seed)
    st = {"case": c, "batch": b}
    if kind == "moves":
        b.import_spins(_pair_spins(c, seed))
    else:
        if b.cfg.n_res and kind != "serve":
            b.prethermalize(100)
        b.emcs(c["warm"])
    b.synchronize()
    st["out"] = _outputs(b)
    if kind == "moves":
        st["out"]["chaos"] = b.chaos
        st["host"] = np.zeros(tuple(b.obs.shape))
    if kind == "serve":     # the requests' own seeds and couplings, on the host
        rng = np.random.Generator(np.random.PCG64([seed, 7]))
        st["keys"] = rng.integers(0, 2 ** 63, c["count"], dtype=np.uint64)
        z = rng.standard_normal((c["count"], 3, b.cfg.V))
        st["J"] = np.clip(np.rint(z * 2.0 ** 18) / 2.0 ** 18, -8.0, 8.0).astype(np.float32)
    return st


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "group":
        state["group"].emcs(c["n"])
        return state["out"]
    b = state["batch"]
    if kind == "emcs":
        b.emcs(c["n"], graph=c.get("graph", True))
    elif kind == "sweep":
        b.sweep(c["n_pt"], c["n_sweep_res"])
        b.swap(pt=False, er=False)
    elif kind == "moves":
        b.houdayer()
        b.measure(chaos=True)
        return {**state["out"], "read": b.read_observables(state["host"])}
    elif kind == "autocorrelation":
        return {**state["out"], "sums": b.reservoir_autocorrelation(c["points"], c["per_point"])}
    else:
        b.reset_samples(c["first"], c["count"], state["keys"], couplings=state["J"], pretherm_sweeps=c["pretherm"])
        b.emcs(c["n"], graph=True)
    return state["out"]


def _updates(c, L=None):
    """Spin updates, spins held and replica pairs moved in one pass of one batch."""
    cfg = _config(c, L)
    SV = cfg.n_samples * cfg.n_replicas * cfg.V
    kind = c["kind"]
    res = cfg.n_res * (cfg.res_sweeps_per_emcs if cfg.er_on else 0)
    if kind == "sweep":
        return SV * (cfg.n_temps * c["n_pt"] + cfg.n_res * c["n_sweep_res"])
    if kind == "autocorrelation":
        return SV * cfg.n_res * c["points"] * c["per_point"]
    if kind == "moves":
        return SV * cfg.n_temps
    n = c["n"] * SV * (cfg.n_temps * cfg.sweeps_per_emcs + res)
    if kind == "serve":
        n += c["count"] * cfg.n_replicas * cfg.V * cfg.n_res * c["pretherm"]
    return n


def work(case):
    """Each coupling and spin read and each spin written once, and the
    arithmetic of a local update: a quarter of a Philox call (15), the uniform
    (2), the field (6), the exponent and its exponential (3), the comparison
    and the flip (3)."""
    sizes = GROUP_SIZES if case["kind"] == "group" else (case["L"],)
    nbytes = flops = 0.0
    for L in sizes:
        cfg = _config(case, L)
        per_spin = 0.125 if cfg.spin_layout == "bits" else 1.0
        lattices = cfg.n_replicas * cfg.n_res if case["kind"] == "autocorrelation" else cfg.n_lat
        nbytes += cfg.n_samples * cfg.V * (12.0 + 2.0 * per_spin * lattices)
        flops += _updates(case, L) * (29.0 if case["kind"] != "moves" else 4.0)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- 64-bit values
def _philox_word0(key, c0, c1, c2, c3):
    """Word 0 of Philox4x32-10 (Salmon et al., SC'11)."""
    m, lo32 = (np.uint64(0xD2511F53), np.uint64(0xCD9E8D57)), np.uint64(0xFFFFFFFF)
    c0, c1, c2, c3, key = (np.asarray(v, dtype=np.uint64) for v in (c0, c1, c2, c3, key))
    k0, k1 = key & lo32, key >> np.uint64(32)
    for _ in range(10):
        p0, p1 = m[0] * c0, m[1] * c2
        c0, c1, c2, c3 = ((p1 >> np.uint64(32)) ^ c1 ^ k0, p1 & lo32, (p0 >> np.uint64(32)) ^ c3 ^ k1, p0 & lo32)
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & lo32, (k1 + np.uint64(0xBB67AE85)) & lo32
    return c0


def _labels(q):
    """Smallest site index of every cluster {i ~ j: neighbours, q_i = q_j}; q [n, L, L, L] (z, y, x)."""
    n, L = q.shape[0], q.shape[1]
    lab = np.broadcast_to(np.arange(L ** 3, dtype=np.int64).reshape(1, L, L, L), q.shape).copy()
    same = [(d, sh, q == np.roll(q, sh, d)) for d in (1, 2, 3) for sh in (1, -1)]
    while True:
        new = lab
        for d, sh, eq in same:
            new = np.where(eq, np.minimum(new, np.roll(new, sh, d)), new)
        flat = new.reshape(n, -1)
        flat = np.take_along_axis(flat, flat, 1)         # pointer jumping
        if np.array_equal(flat.reshape(lab.shape), lab):
            return lab
        lab = flat.reshape(lab.shape)


def exact(case, seed):
    """The cluster move, the energies and the observables of the "moves" kind
    in 64 bits.  The others are Markov chains whose every step decides on the
    one before: their spins and counts are whole numbers, and their energies
    follow from those."""
    if case["kind"] != "moves":
        return None
    c, cfg = dict(case), _config(case)
    S, NR, N, L, V, NP = cfg.n_samples, cfg.n_replicas, cfg.n_slot, cfg.L, cfg.V, cfg.n_replicas // 2
    NT = cfg.n_temps
    keys, J = _inputs(c, L, seed)
    J = J.cpu().numpy().astype(np.float64).reshape(S, 3, L, L, L)
    s = _pair_spins(c, seed).cpu().numpy().reshape(S, NR, N, L, L, L)
    T = cfg.t_min + np.arange(NT) * (cfg.t_max - cfg.t_min) / (NT - 1)
    for k in range(NT):
        if T[k] >= cfg.acu_t_below:
            break
        q = s[:, 0::2, k] * s[:, 1::2, k]
        lab = _labels(q.reshape(S * NP, L, L, L)).reshape(S, NP, -1)
        pair = (np.arange(NP) * NT + k).reshape(1, NP, 1)
        w = _philox_word0(keys.reshape(S, 1, 1), lab, pair, 0, 2)
        eta = np.where(w >> np.uint64(31), -1, 1).astype(np.int8).reshape(q.shape)
        s[:, 0::2, k] *= eta
        s[:, 1::2, k] *= eta
    E = np.zeros((S, NR, N))
    for mu, axis in ((0, -1), (1, -2), (2, -3)):
        for k in range(N):
            E[:, :, k] -= (J[:, None, mu] * (s[:, :, k] * np.roll(s[:, :, k], -1, axis))).sum((-1, -2, -3))
    obs, chaos = np.zeros((S, NT, 8)), np.zeros((S, NT, 2))
    for k in range(NT):
        q = s[:, 0::2, k] * s[:, 1::2, k]
        qm = q.mean((-1, -2, -3), dtype=np.float64)
        ql = sum((q * np.roll(q, -1, a)).sum((-1, -2, -3), dtype=np.float64) for a in (-1, -2, -3)) / (3.0 * V)
        e = E[:, :, k] / V
        Sv = E[:, 0::2, k] / (3.0 * V) + (1.0 - ql) / T[k]
        for i, v in enumerate((np.ones((S, 1)), e, e * e, qm, qm ** 2, ql, Sv, qm ** 4)):
            obs[:, k, i] = v.sum(1)
        qc = (s[:, 0::2, 0] * s[:, 1::2, k]).mean((-1, -2, -3), dtype=np.float64)
        chaos[:, k] = np.stack((np.full(S, float(NP)), (qc ** 2).sum(1)), 1)
    none = {k: None for k in ("spins", "perm", "age", "round_trips", "pt_accepted", "flips", "cluster_stats", "emcs")}
    return {**none, "energies": E.reshape(S, NR * N), "obs": obs, "chaos": chaos, "read": obs}
