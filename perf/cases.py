"""The framework's work in the forms a user calls it, with sizes, inputs and reference values.

Three families, all through the public binding (paper_1812_00367_gb300.nb):

* evaluations: predict to a time and sum acceleration, jerk, snap and potential of a list of
  active particles (`Simulation.predict` + `Simulation.evaluate`, or the allocation-free entry),
  in each arithmetic and for both integration orders;
* integrations: restore a state (a checkpoint) and advance it (`nb_set_state` + `Simulation.run`),
  with shared steps, with block steps, and with many clusters together;
* diagnostics: the energy of the whole system (`Simulation.energy`).

Inputs are Plummer spheres in Henon units (paper_1812_00367_gb300.ic), equal masses or a
Kroupa-like spectrum, softening 1e-4 (1e-5 with the spectrum).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1812_00367_gb300 import ic, nb

DEV = "cuda"
ETA = {6: 0.4, 4: 0.02}            # the step criteria's usual coefficients
DT_MIN, DT_MAX = 2.0 ** -20, 2.0 ** -3
PAIR_FLOPS = {6: 79, 4: 43, "pot": 14}
STATE_DOUBLES = 23                 # m, t, dt, pot and six vectors


def listed():
    return [
        # the smallest integration: one small cluster on shared steps, where launches and latency count
        {"name": "shared_fp64_n1024", "kind": "shared", "n": 1024, "precision": "fp64", "order": 6,
         "kroupa": False, "steps": 16, "h": 2.0 ** -8},
        # the usual integration: block steps, most of them with few active particles
        {"name": "block_fp64_n16384", "kind": "block", "n": 16384, "precision": "fp64", "order": 6,
         "kroupa": False, "t0": 2.0 ** -7, "t1": 2.0 ** -6},
        # an ensemble of small clusters of uneven sizes, advanced together on their own block steps
        {"name": "batch_fp64_96", "kind": "batch", "clusters": 96, "n_min": 256, "n_max": 4096,
         "precision": "fp64", "order": 6, "kroupa": False, "t0": 2.0 ** -7, "t1": 2.0 ** -6},
        # a block step's evaluation with a small active set against a large system
        {"name": "eval_fp64_n65536_a48", "kind": "eval", "n": 65536, "active": 48,
         "precision": "fp64", "order": 6, "kroupa": False},
        # a middling active set that fills no whole tile
        {"name": "eval_fp64_n65536_a1000", "kind": "eval", "n": 65536, "active": 1000,
         "precision": "fp64", "order": 6, "kroupa": False},
        # every particle active: the start-up, the coarse block steps, the headline's bulk
        {"name": "eval_fp64_n65536_all", "kind": "eval", "n": 65536, "active": 65536,
         "precision": "fp64", "order": 6, "kroupa": False},
        # the 4th-order scheme's pair terms, an odd size
        {"name": "eval4_fp64_n30011_all", "kind": "eval", "n": 30011, "active": 30011,
         "precision": "fp64", "order": 4, "kroupa": False},
        # extended precision (pairs of singles), every particle active
        {"name": "eval_ex_n65536_all", "kind": "eval", "n": 65536, "active": 65536,
         "precision": "ex", "order": 6, "kroupa": False},
        # extended precision, a mass spectrum, ragged sizes
        {"name": "eval_ex_n10007_a513", "kind": "eval", "n": 10007, "active": 513,
         "precision": "ex", "order": 6, "kroupa": True},
        # accelerations in pairs of singles, jerk and snap in single precision
        {"name": "eval_fp32x_n65536_a8192", "kind": "eval", "n": 65536, "active": 8192,
         "precision": "fp32x", "order": 6, "kroupa": False},
        # single precision, the arithmetic the 4th-order scheme can use
        {"name": "eval4_fp32_n65536_all", "kind": "eval", "n": 65536, "active": 65536,
         "precision": "fp32", "order": 4, "kroupa": False},
        # energy bookkeeping between slices of a run
        {"name": "energy_n65536", "kind": "energy", "n": 65536, "precision": "fp64", "order": 6,
         "kroupa": False},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "eval", "noalloc", "shared", "block", "batch", "energy"])
    if kind == "eval":
        n = _log_int(rng, 300, 65536)
        active = n if rng.random() < 0.3 else _log_int(rng, 1, n)
        return {"kind": kind, "n": n, "active": active,
                "precision": rng.choice(["fp64", "fp64", "ex", "fp32x", "fp32"]),
                "order": rng.choice([6, 6, 4]), "kroupa": rng.random() < 0.3}
    if kind == "noalloc":
        n = _log_int(rng, 300, 32768)
        return {"kind": kind, "n": n, "active": _log_int(rng, 1, n), "precision": "fp64", "order": 6,
                "kroupa": rng.random() < 0.3}
    if kind == "shared":
        return {"kind": kind, "n": _log_int(rng, 256, 4096), "precision": "fp64",
                "order": rng.choice([6, 4]), "kroupa": False, "steps": rng.randint(8, 32),
                "h": 2.0 ** -8}
    if kind == "block":
        return {"kind": kind, "n": _log_int(rng, 2000, 16384), "precision": "fp64", "order": 6,
                "kroupa": False, "t0": 2.0 ** -7, "t1": 2.0 ** -6}
    if kind == "batch":
        return {"kind": kind, "clusters": rng.randint(8, 96), "n_min": 256, "n_max": _log_int(rng, 1000, 4096),
                "precision": "fp64", "order": 6, "kroupa": False, "t0": 2.0 ** -7, "t1": 2.0 ** -6}
    return {"kind": kind, "n": _log_int(rng, 1024, 65536), "precision": "fp64", "order": 6,
            "kroupa": rng.random() < 0.3}


def _eps(case):
    return 1e-5 if case["kroupa"] else 1e-4


def _system(case, seed):
    """(m, x, v, offsets) on the host; offsets is None for one cluster."""
    if case["kind"] == "batch":
        # the sizes belong to the case, the particles to the seed
        sizes = ic.cluster_sizes(case["clusters"], case["clusters"], case["n_min"], case["n_max"])
        b = ic.plummer_batch(sizes=sizes, seed=seed % 20011 + 1)
        return b.m, b.x, b.v, b.offsets
    masses = ic.kroupa_masses(case["n"], seed=seed + 1) if case["kroupa"] else None
    m, x, v = ic.plummer(case["n"], seed=seed, masses=masses)
    return m, x, v, None


def _mean_field(x):
    """Acceleration of the smooth Plummer model: realistic a_j - a_i for the snap terms."""
    b2 = ic.HENON_PLUMMER_SCALE ** 2
    return -x / ((x * x).sum(axis=1) + b2)[:, None] ** 1.5


def _active(case, seed):
    """The active list as a block step has it: increasing indices."""
    if case["active"] >= case["n"]:
        return np.arange(case["n"], dtype=np.int32)
    rng = np.random.default_rng(seed + 77)
    return np.sort(rng.choice(case["n"], size=case["active"], replace=False)).astype(np.int32)


def prepare(case, seed):
    m, x, v, offsets = _system(case, seed)
    n, eps, order = len(m), _eps(case), case["order"]
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "noalloc":
        a = _mean_field(x)
        st["jpred"] = torch.as_tensor(np.concatenate([x.T, v.T, a.T, m[None]])).to(DEV).contiguous()
        st["active"] = torch.as_tensor(_active(case, seed)).to(DEV)
        st["out"] = torch.empty((10, case["active"]), dtype=torch.float64, device=DEV)
        st["n"], st["eps"] = n, eps
        return st
    if kind in ("eval", "energy"):
        sim = nb.Simulation(m, x, v, eps=eps, eta=ETA[order], precision=case["precision"],
                            keep_state=True, order=order)
        zero = np.zeros((n, 3))
        sim.set_state_numpy({"m": m, "x": x, "v": v, "a": _mean_field(x), "j": zero, "s": zero, "c": zero,
                             "t": np.zeros(n), "dt": np.full(n, 2.0 ** -6), "pot": np.zeros(n)})
        st["t"] = 2.0 ** -8
        if kind == "eval":
            st["active"] = torch.as_tensor(_active(case, seed)).to(DEV)
    else:
        h = case.get("h")
        sim = nb.Simulation(m, x, v, eps=eps, eta=ETA[order], precision=case["precision"], offsets=offsets,
                            dt_min=h or DT_MIN, dt_max=h or DT_MAX, order=order)
        if kind != "shared":
            sim.run(case["t0"])
        st["t"] = case["steps"] * h if kind == "shared" else case["t1"]
        # the checkpoint that every pass starts from
        st["saved"] = {f: t.clone() for f, t in sim.buf.items()}
        st["saved_state"] = nb.make_state(st["saved"])
    st["sim"] = sim
    return st


def run(state):
    kind = state["kind"]
    if kind == "noalloc":
        out = state["out"]
        status = nb.load().nb_evaluate_noalloc(
            state["jpred"].data_ptr(), state["n"], state["eps"], state["active"].data_ptr(),
            state["active"].numel(), out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        if status:
            raise nb.NbError(status, "nb_evaluate_noalloc")
        return out
    sim = state["sim"]
    if kind == "eval":
        sim.predict(state["t"], out=False)
        return sim.evaluate(state["active"])
    if kind == "energy":
        ekin, epot, P, L = sim.energy(state["t"])
        return {"ekin": ekin, "epot": epot, "L": L}
    nb.nb_set_state(sim.ctx, state["saved_state"])
    block_steps, interactions = sim.run(state["t"])
    return {"block_steps": block_steps, "interactions": int(interactions),
            **{f: sim.buf[f] for f in ("x", "v", "a", "j", "s", "c", "t", "dt", "pot")}}


def work(case):
    kind, order = case["kind"], case["order"]
    if kind == "batch":
        # sizes are log-uniform between n_min and n_max
        span = math.log(case["n_max"] / case["n_min"])
        n = case["clusters"] * (case["n_max"] - case["n_min"]) / span
        n2 = case["clusters"] * (case["n_max"] ** 2 - case["n_min"] ** 2) / (2 * span)
    else:
        n, n2 = case["n"], case["n"] ** 2
    state = 8 * STATE_DOUBLES * n
    if kind in ("eval", "noalloc"):
        return {"bytes": 8 * 20 * n + 84 * case["active"],
                "flops": PAIR_FLOPS[order] * float(case["active"]) * n}
    if kind == "energy":
        return {"bytes": 8 * 20 * n, "flops": PAIR_FLOPS["pot"] * float(n2)}
    if kind == "shared":
        return {"bytes": 2 * state, "flops": PAIR_FLOPS[order] * float(n2) * case["steps"]}
    # block steps: a particle is corrected about 250 times per time unit at these sizes
    return {"bytes": 2 * state, "flops": PAIR_FLOPS[order] * float(n2) * 250.0 * (case["t1"] - case["t0"])}


# ------------------------------------------------------------------ values in 64 bits
def _force(m, x, v, a, eps, idx, order):
    """[10][len(idx)] sums over all j != i, in rows of at most 2^25 pairs."""
    n = len(m)
    out = torch.zeros((10, len(idx)), dtype=torch.float64, device=DEV)
    rows = max(1, (1 << 25) // n)
    for b in range(0, len(idx), rows):
        i = idx[b:b + rows]
        r = [x[None, :, k] - x[i, None, k] for k in range(3)]
        y2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2] + eps * eps
        mm = m[None, :].expand(len(i), n).clone()
        mm.scatter_(1, i[:, None], 0.0)
        y2.scatter_(1, i[:, None], 1.0)
        y2 = 1.0 / y2
        my = mm * torch.sqrt(y2)
        o = out[:, b:b + rows]
        o[9] = -my.sum(1)
        if order == 0:  # the potential alone
            continue
        q = my * y2
        dv = [v[None, :, k] - v[i, None, k] for k in range(3)]
        al = (r[0] * dv[0] + r[1] * dv[1] + r[2] * dv[2]) * y2
        w1 = [dv[k] - 3.0 * al * r[k] for k in range(3)]
        for k in range(3):
            o[k] = (q * r[k]).sum(1)
            o[3 + k] = (q * w1[k]).sum(1)
        if order == 6:
            da = [a[None, :, k] - a[i, None, k] for k in range(3)]
            w = sum(dv[k] * dv[k] + r[k] * da[k] for k in range(3))
            be = w * y2 + al * al
            for k in range(3):
                o[6 + k] = (q * (da[k] - 6.0 * al * w1[k] - 3.0 * be * r[k])).sum(1)
    return out


def _norm(u):
    return torch.sqrt((u * u).sum(1))


class _Hermite:
    """One cluster on block steps in plain torch (6th order after Nitadori & Makino 2008, 4th order
    after Makino & Aarseth 1992; power-of-two steps)."""

    def __init__(self, m, x, v, eps, order, dt_min, dt_max):
        t64 = lambda u: torch.as_tensor(np.ascontiguousarray(u), dtype=torch.float64).to(DEV)  # noqa: E731
        self.m, self.x, self.v, self.eps, self.order = t64(m), t64(x), t64(v), eps, order
        self.dt_min, self.dt_max, self.eta = dt_min, dt_max, ETA[order]
        n = len(m)
        every = torch.arange(n, device=DEV)
        zero = torch.zeros_like(self.x)
        o = _force(self.m, self.x, self.v, zero, eps, every, 4)
        self.a, self.j, self.pot = o[0:3].T.clone(), o[3:6].T.clone(), o[9].clone()
        self.s, self.c = zero.clone(), zero.clone()
        if order == 6:
            o = _force(self.m, self.x, self.v, self.a, eps, every, 6)
            self.a, self.j, self.s, self.pot = (o[0:3].T.clone(), o[3:6].T.clone(), o[6:9].T.clone(),
                                                o[9].clone())
        an, jn, sn = _norm(self.a), _norm(self.j), _norm(self.s)
        r = an / jn
        if order == 6:
            r = torch.minimum(r, torch.sqrt(an / sn))
        self.t = torch.zeros(n, dtype=torch.float64, device=DEV)
        self.dt = torch.exp2(torch.floor(torch.log2(0.01 * r))).clamp(dt_min, dt_max)
        self.steps, self.inter = 0, 0

    def step_until(self, t_end):
        n = len(self.m)
        while True:
            tn = float((self.t + self.dt).min())
            if tn > t_end:
                return
            act = torch.nonzero(self.t + self.dt == tn)[:, 0]
            h = (tn - self.t)[:, None]
            s, c = (self.s, self.c) if self.order == 6 else (0.0 * self.s, 0.0 * self.c)
            xp = self.x + h * (self.v + h / 2 * (self.a + h / 3 * (self.j + h / 4 * (s + h / 5 * c))))
            vp = self.v + h * (self.a + h / 2 * (self.j + h / 3 * (s + h / 4 * c)))
            ap = self.a + h * (self.j + h / 2 * (s + h / 3 * c))
            o = _force(self.m, xp, vp, ap, self.eps, act, self.order)
            self._correct(act, tn, o)
            self.steps += 1
            self.inter += len(act) * (n - 1)

    def _correct(self, act, tn, o):
        h = (tn - self.t[act])[:, None]
        x0, v0, a0, j0, s0 = (u[act] for u in (self.x, self.v, self.a, self.j, self.s))
        a1, j1, s1 = o[0:3].T, o[3:6].T, o[6:9].T
        if self.order == 6:
            v1 = v0 + h / 2 * (a1 + a0) - h * h / 10 * (j1 - j0) + h ** 3 / 120 * (s1 + s0)
            x1 = x0 + h / 2 * (v1 + v0) - h * h / 10 * (a1 - a0) + h ** 3 / 120 * (j1 + j0)
            c5 = (6 * (a1 - a0) - 3 * h * (j1 + j0) + h * h / 2 * (s1 - s0)) / h ** 5
            c4 = (h / 4 * (s1 + s0) - (j1 - j0) / 2) / h ** 3
            d5, d4 = 120 * c5, 24 * c4 + 60 * h * c5
            d3 = (s1 - s0) / h + 12 * h * c4 + 10 * h * h * c5
            A1 = torch.sqrt(_norm(a1) * _norm(s1)) + _norm(j1)
            A4 = torch.sqrt(_norm(d3) * _norm(d5)) + _norm(d4)
            crit = self.eta * (A1 / A4) ** (1.0 / 3.0)
            s_new, c_new = s1, d3
        else:
            v1 = v0 + h / 2 * (a0 + a1) + h * h / 12 * (j0 - j1)
            x1 = x0 + h / 2 * (v0 + v1) + h * h / 12 * (a0 - a1)
            d2 = (6 * (a0 - a1) + 2 * h * (j0 + 2 * j1)) / h ** 2
            d3 = (12 * (a0 - a1) + 6 * h * (j0 + j1)) / h ** 3
            crit = torch.sqrt(self.eta * (_norm(a1) * _norm(d2) + _norm(j1) ** 2)
                              / (_norm(j1) * _norm(d3) + _norm(d2) ** 2))
            s_new, c_new = d2, d3
        old = self.dt[act]
        q = tn / (2 * old)
        new = torch.where(crit < old, torch.exp2(torch.floor(torch.log2(crit))),
                          torch.where((crit >= 2 * old) & (q == torch.floor(q)), 2 * old, old))
        self.dt[act] = new.clamp(self.dt_min, self.dt_max)
        self.t[act] = tn
        self.x[act], self.v[act], self.a[act], self.j[act] = x1, v1, a1, j1
        self.s[act], self.c[act], self.pot[act] = s_new, c_new, o[9]


def exact(case, seed):
    m, x, v, offsets = _system(case, seed)
    eps, order, kind = _eps(case), case["order"], case["kind"]
    t64 = lambda u: torch.as_tensor(np.ascontiguousarray(u), dtype=torch.float64).to(DEV)  # noqa: E731
    if kind in ("eval", "noalloc", "energy"):
        a = _mean_field(x)
        h = 0.0 if kind == "noalloc" else 2.0 ** -8
        M, X, V, A = t64(m), t64(x), t64(v), t64(a)
        X, V = X + h * (V + h / 2 * A), V + h * A
        if kind == "energy":
            pot = _force(M, X, V, A, eps, torch.arange(len(m), device=DEV), 0)[9]
            L = (M[:, None] * torch.cross(X, V, dim=1)).sum(0)
            return {"ekin": float(0.5 * (M * (V * V).sum(1)).sum()), "epot": float(0.5 * (M * pot).sum()),
                    "L": L.cpu().numpy()}
        return _force(M, X, V, A, eps, torch.as_tensor(_active(case, seed)).to(DEV).long(), order)
    if kind == "batch":
        return None  # a hundred clusters one by one in plain torch take minutes
    h = case.get("h")
    sim = _Hermite(m, x, v, eps, order, h or DT_MIN, h or DT_MAX)
    if kind == "block":
        sim.step_until(case["t0"])
        steps0, inter0 = sim.steps, sim.inter
        sim.step_until(case["t1"])
    else:
        steps0 = inter0 = 0
        sim.step_until(case["steps"] * h)
    return {"block_steps": sim.steps - steps0, "interactions": sim.inter - inter0,
            "x": sim.x.T.contiguous(), "v": sim.v.T.contiguous(), "a": sim.a.T.contiguous(),
            "j": sim.j.T.contiguous(), "s": sim.s.T.contiguous(), "c": sim.c.T.contiguous(),
            "t": sim.t, "dt": sim.dt, "pot": sim.pot}
