"""Workloads that a user of this library has it do, for measuring it.

``listed()`` names twelve of them and ``draw(rng)`` makes more of the same
ranges; a case is a dict of plain values.  ``prepare(case, seed)`` makes what
a program holds before the call (inputs on the GPU or in host memory, a
context with the melt loaded), ``run(state)`` is one pass through the public
entry points, ``work(case)`` the bytes and operations such a pass cannot do
without, and ``exact(case, seed)`` its outputs in 64 bits, from torch alone.

Inputs.  Melts come from the seeded generator ``kg_inputs``.  The softest
stage of the schedule (n = 2) starts from them as they are, as a real run
does; the harder stages, the analyses and the primitive paths need a melt
without overlaps, which ``_relax`` makes here by a capped steepest descent in
torch (gathers and fixed-order sums only, so a seed always gives the same
bits).  The library itself takes no part in making inputs.

Types.  A mixed-precision context carries velocities, forces and displacements
in binary32, so its positions and velocities are returned as binary32; a
binary64 context returns binary64.
"""
import math

import numpy as np
import torch

import kg_inputs as KI
import paper_2109_11001_gb300 as kg

RHO = 0.85
RC = 2.0 ** (1.0 / 6.0)
R0, L0 = 1.5, 0.960897
GAMMA, TEMP = 1.0, 1.0
QMIN = 0.01                  # FENE continuation, as every run of the soft stages at scale uses it
SCAN = [(0.0, 100, 200), (0.5, 200, 150), (1.0, 400, 100), (1.5, 800, 50),
        (2.0, 100, 250), (2.5, 200, 250), (3.0, 400, 200), (3.5, 800, 250)]   # (kappa, N, chains)
XI = [2.0, 3.0, 4.0, 5.0, 5.75, 6.5, 7.0, 8.0, 9.0, 10.0, 11.0, 12.0]


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _md(chains, length, kappa, n, dt, **more):
    c = {"kind": "md", "chains": chains, "length": length, "kappa": kappa, "n": n, "dt": dt, "steps": 50,
         "fp64": False, "skin": 0.3, "tpm": 1, "block": 128, "sweep": False}
    c.update(more)
    return c


def listed():
    return [
        # the smallest melt (20 x 50): a single melt followed step by step, where launches are all the time
        _md(20, 50, 1.5, 12.0, 0.01, name="md_1k"),
        # a user's mid-size melt (200 x 400) in the production stage, default settings
        _md(200, 400, 2.5, 12.0, 0.01, name="md_80k"),
        # the same melt all in binary64, the setting for reference trajectories
        _md(200, 400, 2.5, 12.0, 0.01, name="md_80k_fp64", fp64=True),
        # the flagship melt (1000 x 1600) in the first and longest stage, at the tuned skin: 50 MD steps and one
        # double-bridging sweep at the paper's rate, the loop that equilibration consists of
        _md(1000, 1600, 3.5, 2.0, 0.005, name="dbh_1600k", sweep=True, skin=0.5),
        # sixteen small melts in one context: many samples of one state point, equilibrated together
        {"name": "batch_16x1k", "kind": "batch", "melts": 16, "chains": 20, "length": 50, "kappa": 1.5, "scan": False,
         "n": 2.0, "dt": 0.005, "steps": 50, "skin": 0.3},
        # eight uneven melts in one context: a scan of the stiffness
        {"name": "scan_485k", "kind": "batch", "melts": 8, "chains": 0, "length": 0, "kappa": 0.0, "scan": True,
         "n": 2.0, "dt": 0.005, "steps": 50, "skin": 0.3},
        # a caller that keeps the state in host memory: load, 50 steps, read back (ragged chains, a stage between)
        {"name": "host_200k", "kind": "host", "chains": 457, "length": 437, "kappa": 3.0, "n": 7.0, "dt": 0.005,
         "steps": 50, "skin": 0.4},
        # a large double-bridging budget on the flagship melt
        {"name": "db_1600k", "kind": "db", "chains": 1000, "length": 1600, "kappa": 3.5, "attempts": 160000},
        # the learned proposal with online training: one logged sweep, then a few optimiser steps
        {"name": "learned_400k", "kind": "learned", "chains": 500, "length": 800, "kappa": 3.0, "attempts": 80000,
         "iters": 20, "batch": 2048},
        # energies, chain statistics and histograms of a sample
        {"name": "observables_400k", "kind": "observables", "chains": 500, "length": 800, "kappa": 3.0, "bins": 100},
        # structure of a sample: S(q) over a shell of wave vectors and g(r)
        {"name": "structure_80k", "kind": "structure", "chains": 200, "length": 400, "kappa": 2.5, "nq": 256,
         "hmax": 24, "rmax": 3.0, "bins": 300},
        # primitive paths of a melt: the first contraction, where the list is rebuilt most
        {"name": "paths_200k", "kind": "paths", "chains": 250, "length": 800, "kappa": 2.0, "steps": 200,
         "fp64": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _melt_size(rng, lo, hi, nmax=1600):
    m = _log_int(rng, lo, hi)
    length = min(_log_int(rng, 20, nmax), m // 4)
    return max(2, m // length), length


def draw(rng):
    kind = rng.choice(["md", "md", "md", "md", "batch", "batch", "host", "db", "learned", "observables", "structure",
                       "paths"])
    kappa = round(rng.uniform(0.0, 3.5), 2)
    if kind == "md":
        fp64 = rng.random() < 0.2
        n = rng.choice(XI)
        chains, length = _melt_size(rng, 1000, 60000 if fp64 else 800000)
        return _md(chains, length, kappa, n, rng.choice([0.004, 0.005] if n < 5.0 else [0.005, 0.008, 0.01]),
                   fp64=fp64, skin=rng.choice([0.3, 0.3, 0.4, 0.5, 0.6]), tpm=1 if fp64 else rng.choice([1, 1, 1, 2]),
                   block=rng.choice([64, 128, 256]), sweep=rng.random() < 0.5)
    if kind == "batch":
        chains, length = _melt_size(rng, 1000, 20000, 400)
        return {"kind": "batch", "melts": rng.randint(2, 16), "chains": chains, "length": length, "kappa": kappa,
                "scan": False, "n": 2.0, "dt": 0.005, "steps": 50, "skin": rng.choice([0.3, 0.4, 0.5])}
    if kind == "host":
        chains, length = _melt_size(rng, 2000, 200000)
        return {"kind": "host", "chains": chains, "length": length, "kappa": kappa, "n": rng.choice(XI), "dt": 0.005,
                "steps": 50, "skin": rng.choice([0.3, 0.4, 0.5])}
    if kind == "db":
        chains, length = _melt_size(rng, 10000, 800000)
        return {"kind": "db", "chains": chains, "length": length, "kappa": kappa,
                "attempts": max(100, chains * length // rng.randint(10, 100))}
    if kind == "learned":
        chains, length = _melt_size(rng, 10000, 200000, 800)
        return {"kind": "learned", "chains": chains, "length": length, "kappa": kappa,
                "attempts": max(1000, chains * length // rng.randint(5, 20)), "iters": rng.randint(1, 20),
                "batch": rng.choice([256, 1000, 2048])}
    if kind == "observables":
        chains, length = _melt_size(rng, 2000, 300000, 1000)
        return {"kind": "observables", "chains": chains, "length": length, "kappa": kappa,
                "bins": rng.randint(20, 400)}
    if kind == "structure":
        chains, length = _melt_size(rng, 2000, 80000, 800)
        return {"kind": "structure", "chains": chains, "length": length, "kappa": kappa, "nq": rng.randint(1, 256),
                "hmax": rng.randint(2, 24), "rmax": round(rng.uniform(1.5, 4.0), 2), "bins": rng.randint(50, 500)}
    chains, length = _melt_size(rng, 4000, 150000, 800)
    return {"kind": "paths", "chains": chains, "length": length, "kappa": kappa, "steps": rng.randint(20, 200),
            "fp64": chains * length < 20000 and rng.random() < 0.3}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _table(x, box, r):
    """Cell grid of side >= r: (cells per axis, cell of each point (3, M), members of every cell (cells, cap))."""
    n = max(1, int(box / r))
    c = torch.floor(x * (n / box)).to(torch.int64) % n
    flat = (c[2] * n + c[1]) * n + c[0]
    order = torch.argsort(flat, stable=True)
    count = torch.bincount(flat, minlength=n ** 3)
    first = torch.cumsum(count, 0) - count
    table = torch.full((n ** 3, int(count.max())), -1, dtype=torch.int64, device=x.device)
    sorted_cell = flat[order]
    table[sorted_cell, torch.arange(len(order), device=x.device) - first[sorted_cell]] = order
    return n, c, table


def _candidates(x, box, r, chunk):
    """For chunks of points: (rows, candidates (m, 27 cap), -1 for none, and their minimum-image vectors (3, m, 27 cap))."""
    n, c, table = _table(x, box, r)
    span = [0] if n == 1 else [0, 1] if n == 2 else [-1, 0, 1]
    for lo in range(0, x.shape[1], chunk):
        rows = torch.arange(lo, min(lo + chunk, x.shape[1]), device=x.device)
        cand = torch.cat([table[((c[2, rows] + dz) % n * n + (c[1, rows] + dy) % n) * n + (c[0, rows] + dx) % n]
                          for dz in span for dy in span for dx in span], 1)
        d = x[:, cand.clamp(min=0)] - x[:, rows, None]
        yield rows, cand, d - box * torch.round(d / box)


def _neighbours(x, box, length, r, interchain=False):
    """(M, K) points within r that are not 1-2 bonded (or, with interchain, of another chain), padded with the point itself."""
    found = []
    for rows, cand, d in _candidates(x, box, r, 100000):
        keep = (cand >= 0) & (cand != rows[:, None]) & ((d * d).sum(0) < r * r)
        same = cand // length == (rows // length)[:, None]
        keep &= ~(same if interchain else same & ((cand - rows[:, None]).abs() == 1))
        i, j = keep.nonzero(as_tuple=True)
        nbr = rows[:, None].repeat(1, max(1, int(keep.sum(1).max())))
        nbr[i, (keep.cumsum(1) - 1)[i, j]] = cand[i, j]
        found.append(nbr)
    width = max(f.shape[1] for f in found)
    pad = [torch.cat([f, f[:, :1].repeat(1, width - f.shape[1])], 1) if f.shape[1] < width else f for f in found]
    own = torch.arange(x.shape[1], device=x.device)[:, None]
    out = torch.cat(pad, 0)
    if any(f.shape[1] < width for f in found):     # repeated entries of the padding become the point itself
        lengths = torch.cat([torch.full((len(f), 1), f.shape[1], device=x.device) for f in found], 0)
        out = torch.where(torch.arange(width, device=x.device)[None, :] < lengths, out, own)
    return out


def _mlj(r2, n):
    """U_MLJ^n (Eqs. 5-6, shifted) and (dU/dr)/r at r^2, zero past the cutoff."""
    c1, c2 = 6.0 * 2.0 ** (n / 6.0) / (n - 6.0), 2.0 * n / (n - 6.0)
    inside = (r2 > 0) & (r2 < RC * RC)
    r2 = torch.where(inside, r2, torch.ones_like(r2))
    i6 = r2 ** -3
    rn = i6 * i6 if n == 12.0 else r2 ** (-0.5 * n)
    zero = torch.zeros_like(r2)
    return torch.where(inside, c1 * rn - c2 * i6 + 1.0, zero), torch.where(inside, (6.0 * c2 * i6 - n * c1 * rn) / r2, zero)


def _k_fene(n):
    """k_n of Eq. 9."""
    return 6.0 * n * (R0 * R0 - L0 * L0) * (2.0 ** (n / 6.0) * L0 ** -n - 2.0 * L0 ** -6.0) / ((n - 6.0) * R0 * R0 * L0 * L0)


def _pairs(x, box, nbr, n):
    """Pair forces (3, M), pair energy, pair virial."""
    d = x[:, nbr] - x[:, :, None]
    d -= box * torch.round(d / box)
    r2 = (d * d).sum(0)
    u, f = _mlj(r2, n)
    return (f * d).sum(-1), 0.5 * u.sum(), -0.5 * (f * r2).sum()


def _bonded(x, box, length, kappa, n, qmin=QMIN, cap=None):
    """Bond (Eq. 10) and bending (Eq. 4) forces with their energies and virial."""
    p = x.reshape(3, -1, length)
    b = p[:, :, 1:] - p[:, :, :-1]
    b = b - box * torch.round(b / box)
    r2 = (b * b).sum(0)
    q, k = 1.0 - r2 / (R0 * R0), _k_fene(n)
    if cap is not None:
        q = q.clamp(min=cap)
    soft = q < qmin
    qs = torch.where(soft, torch.full_like(q, max(qmin, 1e-30)), q)
    u, f = _mlj(r2, n)
    f = f + k / qs
    e = u - 0.5 * k * R0 * R0 * torch.log(qs) + torch.where(soft, k * (r2 - (1 - qmin) * R0 * R0) / (2 * max(qmin, 1e-30)),
                                                            torch.zeros_like(q))
    force = torch.zeros_like(p)
    force[:, :, :-1] += f * b
    force[:, :, 1:] -= f * b
    b1, b2 = b[:, :, :-1], b[:, :, 1:]
    l1, l2 = r2[:, :-1], r2[:, 1:]
    inv = 1.0 / torch.sqrt(l1 * l2)
    cs = (b1 * b2).sum(0) * inv
    g1, g2 = b2 * inv - cs / l1 * b1, b1 * inv - cs / l2 * b2
    force[:, :, :-2] -= kappa * g1
    force[:, :, 1:-1] += kappa * (g1 - g2)
    force[:, :, 2:] += kappa * g2
    return force.reshape(3, -1), e.sum(), kappa * (1.0 - cs).sum(), -(f * r2).sum()


def _relax(x, box, length, kappa):
    """The melt pushed apart: 160 capped steps down the n = 12 energy, in binary32."""
    x = x.float()
    for it in range(160):
        if it % 8 == 0:
            nbr = _neighbours(x, box, length, RC + 0.45)
        f = _pairs(x, box, nbr, 12.0)[0] + _bonded(x, box, length, kappa, 12.0, cap=0.05)[0]
        s = 2e-4 * f
        x = x + s * (0.03 / torch.sqrt((s * s).sum(0)).clamp(min=0.03))
    return x.double()


def _melt(chains, length, kappa, seed, relaxed):
    """(box, x, v) on the GPU."""
    m = KI.random_walk_melt(chains, length, RHO, kappa, seed)
    x, v = torch.from_numpy(m.x).cuda(), torch.from_numpy(m.v).cuda()
    return m.box, _relax(x, m.box, length, kappa) if relaxed else x, v


def _melts(case, seed):
    """[(chains, length, kappa, box, x, v)] of a case."""
    if case["kind"] == "batch":
        sizes = ([(c, n, k) for k, n, c in SCAN] if case["scan"] else
                 [(case["chains"], case["length"], case["kappa"])] * case["melts"])
        return [(c, n, k) + _melt(c, n, k, 1000 * seed + i, False) for i, (c, n, k) in enumerate(sizes)]
    soft = case["kind"] in ("db", "learned") or case.get("n", 12.0) < 5.0
    if case["kind"] == "paths":
        soft = False
    c, n, k = case["chains"], case["length"], case["kappa"]
    return [(c, n, k) + _melt(c, n, k, 1000 * seed, not soft)]


class _State:
    """A context and the buffers that a program reads its results into."""

    def __init__(self, case, seed):
        self.case = case
        self.melts = _melts(case, seed)
        fp64 = case.get("fp64", False) and case["kind"] == "md"
        p = kg.make_params([(c, n, box, k) for c, n, k, box, _, _ in self.melts],
                           precision=kg.KG_FP64 if fp64 else kg.KG_MIXED, seed=seed + 7, fene_qmin=QMIN,
                           skin=case.get("skin", 0.3), block_size=case.get("block", 0),
                           threads_per_monomer=case.get("tpm", 0))
        self.ctx = None
        self.ctx = kg.kg_create(p, 0, torch.cuda.current_stream().cuda_stream, kg.torch_allocator())
        stage = case.get("n", 2.0 if case["kind"] in ("db", "learned") else 12.0)
        kg.kg_set_potential_schedule(self.ctx, [kg.stage(stage, 10 ** 15, case.get("dt", 0.005))])
        host = case["kind"] == "host"
        self.out = []
        for i, (_, _, _, _, x, v) in enumerate(self.melts):
            m = x.shape[1]
            if host:
                self.host_in = [x.cpu().pin_memory(), v.cpu().pin_memory()]
                self.out.append([torch.empty(3, m, dtype=torch.float64, pin_memory=True) for _ in range(2)])
            else:
                kg.kg_load_config(self.ctx, i, x, v)
                self.out.append([torch.empty(3, m, dtype=torch.float64, device="cuda"),
                                 torch.empty(3, m, dtype=torch.float64, device="cuda"),
                                 torch.empty(m, dtype=torch.int32, device="cuda")])
        self.melts = [t[:4] for t in self.melts]       # the program lets go of the inputs it has loaded
        if case["kind"] == "learned":
            g = np.random.default_rng(seed)
            w = np.concatenate([(g.standard_normal(64 * 24) * math.sqrt(2 / 24)), np.zeros(64),
                                (g.standard_normal(64 * 64) * math.sqrt(2 / 64)), np.zeros(64),
                                g.standard_normal(64) * 0.1, np.zeros(1)])
            kg.kg_mlp_log(self.ctx, 1 << 18)
            kg.kg_mlp_set_weights(self.ctx, w)
        if case["kind"] == "structure":
            self.hkl = _wave_vectors(case, seed)

    def __del__(self):
        if self.ctx is not None:
            kg.kg_destroy(self.ctx)
            self.ctx = None


def _wave_vectors(case, seed):
    hkl = np.random.default_rng(seed).integers(-case["hmax"], case["hmax"] + 1, size=(case["nq"], 3))
    hkl[np.all(hkl == 0, axis=1), 0] = 1
    return hkl.astype(np.int32)


def prepare(case, seed):
    return _State(case, seed)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    case, ctx = s.case, s.ctx
    kind = case["kind"]
    if kind in ("md", "batch"):
        kg.kg_step(ctx, case["steps"])
        if case.get("sweep", True):
            kg.kg_db_sweep(ctx, -1.0)
        for i, (x, v, pid) in enumerate(s.out):
            kg.kg_get_config(ctx, i, x, v, pid)
        if case.get("fp64", False):
            return {"x": s.out[0][0], "v": s.out[0][1], "pid": s.out[0][2]}
        return [{"x": x.float(), "v": v.float(), "pid": pid} for x, v, pid in s.out]
    if kind == "host":
        kg.kg_load_config(ctx, 0, s.host_in[0], s.host_in[1])
        kg.kg_set_counters(ctx, 0, 0)
        kg.kg_step(ctx, case["steps"])
        kg.kg_get_config(ctx, 0, s.out[0][0], s.out[0][1])
        return {"x": s.out[0][0].float(), "v": s.out[0][1].float()}
    if kind == "db":
        st = kg.kg_db_sweep_k(ctx, [case["attempts"]])
        x, _, pid = s.out[0]
        kg.kg_get_config(ctx, 0, x, None, pid)
        return {"x": x, "pid": pid, "attempted": st.attempted, "empty": st.empty, "accepted": st.accepted}
    if kind == "learned":
        st = kg.kg_db_sweep_learned_k(ctx, [case["attempts"]], 0.1)
        loss = kg.kg_mlp_train(ctx, case["iters"], case["batch"], 2e-3)
        x, _, pid = s.out[0]
        kg.kg_get_config(ctx, 0, x, None, pid)
        return {"x": x, "pid": pid, "attempted": st.attempted, "empty": st.empty, "accepted": st.accepted,
                "weights": kg.kg_mlp_get_weights(ctx).astype(np.float32), "loss": loss}
    if kind == "observables":
        r2n, bond, cos = np.zeros(case["length"]), np.zeros(case["bins"]), np.zeros(case["bins"])
        o = kg.kg_observables(ctx, 0, r2n, bond, cos, case["bins"])
        return {"r2n": r2n, "bond": bond, "cos": cos, "e_pair": o.e_pair, "e_bond": o.e_bond, "e_angle": o.e_angle,
                "e_kin": o.e_kin, "virial": o.virial, "pressure": o.pressure}
    if kind == "structure":
        sq = kg.kg_structure_factor(ctx, 0, s.hkl)
        # S(q) is a sum of binary32 phase factors; g(r) holds exact counts
        return {"sq": sq.astype(np.float32), "gr": kg.kg_pair_distribution(ctx, 0, case["rmax"], case["bins"])}
    fp64 = case["fp64"]
    x = s.out[0][0]
    lpp, res = kg.kg_primitive_path(ctx, 0, case["chains"], case["steps"], x_out=x,
                                    precision=kg.KG_FP64 if fp64 else kg.KG_MIXED)
    if fp64:
        return {"x": x, "lpp": lpp, "lpp_mean": res["lpp_mean"], "fmax": res["fmax"]}
    return {"x": x.float(), "lpp": lpp.astype(np.float32), "lpp_mean": res["lpp_mean"], "fmax": res["fmax"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Positions in 24 bytes; velocities in 12 (mixed) or 24 (binary64).  A step reads and writes both and computes
    about five pair terms within the cutoff, two bonds, three angles and three normals per monomer."""
    kind = case["kind"]
    if kind == "batch":
        m = sum(c * n for _, n, c in SCAN) if case["scan"] else case["melts"] * case["chains"] * case["length"]
    else:
        m = case["chains"] * case["length"]
    vel = 24 if case.get("fp64", False) else 12
    if kind in ("md", "batch"):
        return {"bytes": m * case["steps"] * 2.0 * (24 + vel), "flops": m * case["steps"] * 375.0}
    if kind == "host":
        return {"bytes": m * (case["steps"] * 2.0 * (24 + vel) + 96.0), "flops": m * case["steps"] * 375.0}
    if kind == "db":     # positions and ids once; 27 cells of two monomers per drawn bond
        return {"bytes": m * 28.0 + case["attempts"] * 54 * 16.0, "flops": case["attempts"] * 54 * 10.0}
    if kind == "learned":
        rows = case["iters"] * case["batch"]
        return {"bytes": m * 28.0 + case["attempts"] * 54 * 16.0 + rows * 200.0,
                "flops": case["attempts"] * 54 * 10.0 + rows * 3 * 2 * 5700.0}
    if kind == "observables":
        return {"bytes": m * (24.0 + 12.0), "flops": m * (300.0 + 8.0 * (case["length"] - 1) / 2.0)}
    if kind == "structure":
        shell = RHO * 4.0 / 3.0 * math.pi * case["rmax"] ** 3
        return {"bytes": m * 24.0 * 2, "flops": m * (case["nq"] * 20.0 + shell * 10.0)}
    return {"bytes": m * case["steps"] * 2.0 * (24 + vel), "flops": m * case["steps"] * 150.0}


# ---------------------------------------------------------------------------
# the outputs in 64 bits
# ---------------------------------------------------------------------------
_MASK = 0xFFFFFFFF


def _philox(counter, key):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors that hold 32-bit words."""
    c, (k0, k1) = list(counter), key
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & _MASK) ^ c[1] ^ k0, p1 & _MASK, ((p0 >> 32) & _MASK) ^ c[3] ^ k1, p0 & _MASK]
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return c


def _normals(seed, melt, step, m):
    """(3, m) standard normals of the Langevin noise."""
    i = torch.arange(m, dtype=torch.int64, device="cuda")
    z = torch.zeros_like(i)
    w = _philox([i, z + (step & _MASK), z + (step >> 32), z + (melt << 4)], (seed & _MASK, seed >> 32))
    u = [(2 * (t >> 9) + 1).double() * 2.0 ** -24 for t in w]
    a, b = torch.sqrt(-2.0 * torch.log(u[0])), torch.sqrt(-2.0 * torch.log(u[2]))
    return torch.stack([a * torch.cos(2 * math.pi * u[1]), a * torch.sin(2 * math.pi * u[1]),
                        b * torch.cos(2 * math.pi * u[3])])


def _trajectory(case, seed, melt, t):
    """(x, v) of a melt after the case's steps."""
    _, length, kappa, box, x, v = t
    n, dt, nbr, ref = case["n"], case["dt"], None, None
    amp = math.sqrt(2.0 * GAMMA * TEMP / dt)
    for step in range(case["steps"]):
        if nbr is None or float(((x - ref) ** 2).sum(0).max()) > 0.25 ** 2:
            nbr, ref = _neighbours(x, box, length, RC + 0.5), x
        f = _pairs(x, box, nbr, n)[0] + _bonded(x, box, length, kappa, n)[0]
        v = v + dt * (f - GAMMA * v + amp * _normals(seed + 7, melt, step, x.shape[1]))
        x = x + dt * v
    return x, v


def _paths(case, t):
    chains, length, _, box, x, _ = t
    dt, skin = 0.005, 0.3
    m = x.shape[1]
    mobile = torch.ones(chains, length, dtype=torch.float64, device="cuda")
    mobile[:, 0] = mobile[:, -1] = 0.0
    mobile = mobile.reshape(-1)
    k = _k_fene(12.0)

    def conservative(x, nbr):
        f = _pairs(x, box, nbr, 12.0)[0]
        p = x.reshape(3, chains, length)
        b = p[:, :, 1:] - p[:, :, :-1]
        g = k / (1.0 - (b * b).sum(0) / (R0 * R0)) * b
        f = f.reshape(3, chains, length)
        f[:, :, :-1] += g
        f[:, :, 1:] -= g
        return f.reshape(3, m) * mobile

    v, ref, nbr = torch.zeros_like(x), x, _neighbours(x, box, length, RC + skin, True)
    f = conservative(x, nbr)
    for _ in range(case["steps"]):
        v = v + 0.5 * dt * f
        x = x + dt * v
        if float(((x - ref) ** 2).sum(0).max()) > (0.5 * skin) ** 2:
            nbr, ref = _neighbours(x, box, length, RC + skin, True), x
        f = conservative(x, nbr) - GAMMA * v
        v = v + 0.5 * dt * f
    p = x.reshape(3, chains, length)
    lpp = torch.sqrt(((p[:, :, 1:] - p[:, :, :-1]) ** 2).sum(0)).sum(1)
    return {"x": x, "lpp": lpp, "lpp_mean": float(lpp.mean()), "fmax": float(torch.sqrt((f * f).sum(0)).max())}


def _observables(case, seed, t):
    chains, length, kappa, box, x, v = t
    m = x.shape[1]
    fp, ep, wp = _pairs(x, box, _neighbours(x, box, length, RC), 12.0)
    fb, eb, ea, wb = _bonded(x, box, length, kappa, 12.0)
    dt = 0.005
    vn = v + 0.5 * dt * (fp + fb - GAMMA * v + math.sqrt(2.0 * GAMMA * TEMP / dt) * _normals(seed + 7, 0, 0, m))
    ek, w = float(0.5 * (vn * vn).sum()), float(wp + wb)
    p = x.reshape(3, chains, length)
    r2n = np.zeros(length)
    for i in range(1, length):
        r2n[i] = float(((p[:, :, i:] - p[:, :, :-i]) ** 2).sum()) / (chains * (length - i))
    b = p[:, :, 1:] - p[:, :, :-1]
    size = torch.sqrt((b * b).sum(0))
    cs = (b[:, :, 1:] * b[:, :, :-1]).sum(0) / (size[:, 1:] * size[:, :-1])
    bins = case["bins"]
    ib = torch.floor(size / R0 * bins).to(torch.int64).reshape(-1)
    ic = torch.floor((cs + 1.0) * 0.5 * bins).to(torch.int64).clamp(0, bins - 1).reshape(-1)
    hist = [torch.bincount(i[(i >= 0) & (i < bins)], minlength=bins).double().cpu().numpy() for i in (ib, ic)]
    return {"r2n": r2n, "bond": hist[0], "cos": hist[1], "e_pair": float(ep), "e_bond": float(eb),
            "e_angle": float(ea), "e_kin": ek, "virial": w, "pressure": (2.0 * ek + w) / (3.0 * box ** 3)}


def _structure(case, seed, t):
    chains, length, _, box, x, _ = t
    m = x.shape[1]
    q = torch.from_numpy(_wave_vectors(case, seed)).double().cuda()
    sq = []
    for lo in range(0, len(q), 32):
        turns = (q[lo:lo + 32] @ x) / box
        turns = 2.0 * math.pi * (turns - torch.floor(turns))
        sq.append((torch.cos(turns).sum(1) ** 2 + torch.sin(turns).sum(1) ** 2) / m)
    rmax, bins = case["rmax"], case["bins"]
    dr = rmax / bins
    hist = torch.zeros(bins, dtype=torch.int64, device="cuda")
    for rows, cand, d in _candidates(x, box, rmax, 10000):
        r = torch.sqrt((d * d).sum(0))
        keep = (cand >= 0) & (cand != rows[:, None]) & (r < rmax)
        i = torch.floor(r[keep] / dr).to(torch.int64)
        hist += torch.bincount(i[i < bins], minlength=bins)
    edge = np.arange(bins + 1) * dr
    shell = m * (m / box ** 3) * (4.0 / 3.0 * math.pi * (edge[1:] ** 3 - edge[:-1] ** 3))
    return {"sq": torch.cat(sq), "gr": hist.double().cpu().numpy() / shell}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("db", "learned") or case.get("sweep", kind == "batch"):
        return None          # swaps are whole numbers; a trajectory through them has no value of its own
    t = _melts(case, seed)[0]
    if kind in ("md", "host"):
        x, v = _trajectory(case, seed, 0, t)
        if kind == "host":
            return {"x": x, "v": v}
        out = {"x": x, "v": v, "pid": None}
        return out if case["fp64"] else [out]
    if kind == "observables":
        return _observables(case, seed, t)
    if kind == "structure":
        return _structure(case, seed, t)
    return _paths(case, t)
