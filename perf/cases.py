"""The work this library is measured on: solves, batches and training as a program calls them.

Every case goes through the public entry points of ``paper_2403_04578_gb300.tpf`` on the synthetic feeders and
loads of ``paper_2403_04578_gb300.inputs``, at the sizes of the repository's own configurations, benchmark
and tests.  A case's ``feeder`` seeds the network (a user keeps one), the seed given to ``prepare`` the loads.

Returned are the voltages and the whole-number results of each call.  The power mismatch that a solve also
writes is left out: at convergence it is the size of the rounding left in V (1e-12 to 1e-10 pu), so its digits
carry no result that V, which is returned whole, does not.
"""
import functools
import math

import numpy as np
import torch

from paper_2403_04578_gb300 import inputs as G
from paper_2403_04578_gb300 import tpf

TOL = 1e-10
YEAR = 525_600  # minutes
SWEEPS = 8      # sweeps of a flat-start column (7.1 to 8.3 on these feeders); the learned start takes 5 to 6
BATCH = 1024    # columns of a training step


def listed():
    return [
        # One feeder, one day at one-minute steps: the smallest call, answered while a user waits.
        {"name": "small_day", "kind": "sparse", "n_bus": 34, "columns": 1440, "feeder": 1, "loads": "constant"},
        # The headline workload: a 1,000-bus feeder over the one-minute year, from the flat start.
        {"name": "year_flat", "kind": "sparse", "n_bus": 1000, "columns": YEAR, "feeder": 1, "loads": "constant"},
        # The same year from the learned start (prediction and solve in one call).
        {"name": "year_learned", "kind": "learned", "n_bus": 1000, "columns": YEAR, "feeder": 1},
        # Two weeks of one-minute loads that live in the host's pinned memory, results back there.
        {"name": "host_fortnight", "kind": "host", "n_bus": 1000, "columns": 20_160, "feeder": 1},
        # Feeder.solve with its defaults: Algorithm 1's dense product on the tensor cores.
        {"name": "dense_default", "kind": "dense", "n_bus": 1000, "columns": 65_536, "feeder": 1,
         "precision": "mixed", "topology": "radial"},
        # An hourly year of a meshed 200-bus network in plain double precision (meshed networks have the dense form only).
        {"name": "fp64_meshed", "kind": "dense", "n_bus": 200, "columns": 8760, "feeder": 5, "precision": "fp64",
         "topology": "meshed"},
        # The sparse form in plain double precision.
        {"name": "fp64_sparse", "kind": "tree64", "n_bus": 1000, "columns": 16_384, "feeder": 1},
        # Scenario x hour tensor of single-precision loads with PV, voltage-band statistics beside V.
        {"name": "scenarios", "kind": "scenarios", "n_bus": 500, "scenarios": 20, "hours": 8760, "feeder": 3},
        # Many feeders of different sizes, prepared once and solved again and again with new loads.
        {"name": "feeder_batch", "kind": "batch", "feeders": 256, "feeder": 1000},
        # Voltage-dependent (ZIP) loads.
        {"name": "zip_loads", "kind": "sparse", "n_bus": 1000, "columns": 65_536, "feeder": 1, "loads": "zip"},
        # An unbalanced three-phase feeder.
        {"name": "three_phase", "kind": "poly", "n_bus": 500, "columns": 16_384, "feeder": 1},
        # Training the learned start: an epoch of 32 steps for a 200-bus feeder, the updated weights read back.
        {"name": "train_epoch", "kind": "train", "n_bus": 200, "steps": 32, "hidden": 256, "layers": 3, "feeder": 5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sparse", "sparse", "learned", "host", "dense", "dense", "tree64", "scenarios", "batch", "poly",
                       "train"])
    c = {"kind": kind, "feeder": rng.randrange(1, 1000)}
    if kind == "sparse":
        c["n_bus"] = _log(rng, 20, 2000)
        c["columns"] = _log(rng, 96, min(YEAR, 400_000_000 // c["n_bus"]))
        c["loads"] = rng.choice(["constant", "constant", "zip"])
    elif kind == "learned":
        c["n_bus"] = _log(rng, 100, 1000)
        c["columns"] = _log(rng, 1440, min(YEAR, 400_000_000 // c["n_bus"]))
    elif kind == "host":
        c["n_bus"] = _log(rng, 100, 1000)
        c["columns"] = _log(rng, 1440, min(86_400, 20_000_000 // c["n_bus"]))
    elif kind == "dense":
        c["n_bus"] = _log(rng, 34, 1000)
        c["precision"] = rng.choice(["mixed", "fp64"])
        c["topology"] = rng.choice(["radial", "meshed"])
        most = 65_536 if c["precision"] == "mixed" else 2_000_000_000 // c["n_bus"] ** 2
        c["columns"] = _log(rng, 288, min(65_536, most))
    elif kind == "tree64":
        c["n_bus"] = _log(rng, 34, 1000)
        c["columns"] = _log(rng, 288, 16_384)
    elif kind == "scenarios":
        c["n_bus"] = _log(rng, 100, 500)
        c["scenarios"] = _log(rng, 2, 20)
        c["hours"] = _log(rng, 24, 8760)
    elif kind == "batch":
        c["feeders"] = _log(rng, 16, 256)
    elif kind == "poly":
        c["n_bus"] = _log(rng, 34, 500)
        c["columns"] = _log(rng, 96, 16_384)
    else:
        c["n_bus"] = _log(rng, 34, 500)
        c["steps"] = _log(rng, 8, 32)
        c["hidden"] = rng.choice([128, 256])
        c["layers"] = rng.choice([1, 2, 3])
    return c


# ------------------------------------------------------------------------------------------- inputs

def _dev():
    return torch.device("cuda", torch.cuda.current_device())


@functools.lru_cache(maxsize=600)
def _make(n_bus, seed, peak_factor=1.0):
    return G.make_feeder(n_bus, seed, peak_factor=peak_factor)


def _network(case):
    """The feeder's data; a scenario tensor's feeder is scaled for its largest scenario factor."""
    return _make(case["n_bus"], case["feeder"], 1.8 if case["kind"] == "scenarios" else 1.0)


def _branches(case, f):
    """Branch list (from, to, z); a meshed network closes two to twenty loops with tie lines."""
    fr, to, z = f.from_bus, f.to_bus, f.z_pu
    if case.get("topology") == "meshed":
        r = np.random.default_rng(case["feeder"])
        ties = max(2, min(20, case["n_bus"] // 20))
        a = r.choice(np.arange(1, case["n_bus"] // 2), ties)
        b = r.choice(np.arange(case["n_bus"] // 2, case["n_bus"]), ties, replace=False)
        zt = z[r.integers(0, len(z), ties)] * r.uniform(1.0, 3.0, ties)
        fr, to, z = np.r_[fr, a], np.r_[to, b], np.r_[z, zt]
    return fr.astype(np.int32), to.astype(np.int32), z


def _loads(case, f, seed, columns=None):
    T = columns or case["columns"]
    # Columns are consecutive minutes; short tensors spread over the day.
    return G.load_tensor_device(f, T, seed, _dev(), step_minutes=max(1.0, 1440.0 / T))


def _alpha(case):
    return np.random.default_rng(case["feeder"]).dirichlet([2, 1, 1], case["n_bus"] - 1).T.copy()


def _poly_loads(f, T, seed):
    """The recipe of inputs.load_tensor_poly, drawn on the device: S[T][n_pq * phases]."""
    d = _dev()
    g = torch.Generator(device=d)
    g.manual_seed(seed)
    base = torch.tensor(f.load_scale * f.base_kw[1:] / G.S_BASE_KW, device=d)
    tanphi = torch.tensor(np.tan(np.arccos(f.pf[1:])), device=d)
    hours = (np.arange(T) * max(1.0, 1440.0 / T) / 60.0) % 24.0
    shape = torch.tensor(G.daily_shape(hours), device=d)
    p = torch.randn((T,) + tuple(base.shape), generator=g, device=d, dtype=torch.float64).mul_(0.2).exp_()
    p.mul_(base[None]).mul_(shape[:, None, None])
    return torch.complex(p, p * tanphi[None]).reshape(T, -1)


def _batch_specs(case):
    return G.batch_specs(case["feeders"], seed0=case["feeder"], seed=case["feeder"] + 7)


def _train_network(fd, f, seed, columns=16_384, epochs=20):
    """The learned start's network, trained on other loads as a user trains it once per feeder."""
    S = G.load_tensor_device(f, columns, seed, _dev())
    V, _, _, _ = fd.solve(S, tol=TOL, method="sparse")
    net = tpf.LearnedStart(f.n_pq, hidden=256, hidden_layers=3, max_batch=BATCH, seed=1)
    net.fit_normalization(S, V)
    gen = torch.Generator(device="cpu").manual_seed(seed)
    for ep in range(epochs):
        lr = 1e-3 * (0.5 * (1 + math.cos(math.pi * ep / epochs)) * 0.9 + 0.1)
        order = torch.randperm(columns, generator=gen).to(S.device)
        Sp, Vp = S[order].contiguous(), V[order].contiguous()
        for k in range(columns // BATCH):
            net.train_step(Sp[k * BATCH:(k + 1) * BATCH], Vp[k * BATCH:(k + 1) * BATCH], lr=lr, want_loss=False)
    return net


def _first_weights(case):
    """Xavier-uniform weights, zero biases: per layer W [out][in], then b."""
    n = case["n_bus"] - 1
    sizes = [2 * n] + [case["hidden"]] * case["layers"] + [2 * n]
    r = np.random.default_rng(case["feeder"])
    parts = []
    for i, o in zip(sizes[:-1], sizes[1:]):
        a = math.sqrt(6.0 / (i + o))
        parts += [r.uniform(-a, a, o * i).astype(np.float32), np.zeros(o, np.float32)]
    return sizes, np.concatenate(parts)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        fds, offs, loads = [], [0], []
        for k, (nb, T, sd) in enumerate(_batch_specs(case)):
            f = _make(nb, sd)
            fds.append(tpf.Feeder.from_inputs(f))
            loads.append(G.load_tensor_device(f, T, seed + k, _dev(), step_minutes=G.step_minutes_for(T)))
            offs.append(offs[-1] + T * (nb - 1))
        cols = np.concatenate([[0], np.cumsum([s.shape[0] for s in loads])])
        V = torch.empty(offs[-1], dtype=torch.complex128, device=_dev())
        it = torch.empty(int(cols[-1]), dtype=torch.int32, device=_dev())
        mm = torch.empty(int(cols[-1]), dtype=torch.float64, device=_dev())
        cut = lambda x, k: x[int(cols[k]):int(cols[k + 1])]  # noqa: E731
        plan = tpf.BatchGraph(fds, loads, [V[offs[k]:offs[k + 1]].view(s.shape) for k, s in enumerate(loads)],
                              [cut(it, k) for k in range(len(fds))], [cut(mm, k) for k in range(len(fds))],
                              tol=TOL, start="flat")
        return {"kind": kind, "plan": plan, "V": V, "iters": it}
    if kind == "poly":
        f = G.make_feeder_poly(case["n_bus"], case["feeder"])
        fd = tpf.Feeder.poly(f.n_bus, f.from_bus, f.to_bus, f.z_blocks, f.phases, f.slack, f.v0, f.pq_bus)
        return {"kind": kind, "feeder": fd, "S": _poly_loads(f, case["columns"], seed)}
    f = _network(case)
    if kind == "scenarios":
        return {"kind": kind, "feeder": tpf.Feeder.from_inputs(f),
                "S": G.scenario_tensor_device(f, case["scenarios"], case["hours"], seed, _dev())}
    if kind == "train":
        S = _loads(case, f, seed, case["steps"] * BATCH)
        with tpf.Feeder.from_inputs(f) as fd:
            V, _, _, _ = fd.solve(S, tol=TOL, method="sparse")
        net = tpf.LearnedStart(f.n_pq, hidden=case["hidden"], hidden_layers=case["layers"], max_batch=BATCH)
        net.set_params(_first_weights(case)[1])
        net.fit_normalization(S, V)
        order = torch.randperm(S.shape[0], generator=torch.Generator(device="cpu").manual_seed(seed)).to(S.device)
        return {"kind": kind, "net": net, "S": S[order].contiguous(), "V": V[order].contiguous()}
    fr, to, z = _branches(case, f)
    fd = tpf.Feeder(f.n_bus, fr, to, z, f.slack, f.v0, f.pq_bus)
    state = {"kind": kind, "feeder": fd, "S": _loads(case, f, seed), "precision": case.get("precision")}
    if kind == "learned":
        state["net"] = _train_network(fd, f, seed + 100)
    if kind == "host":
        T, n = state["S"].shape
        state["S"] = torch.empty((T, n), dtype=torch.complex128, pin_memory=True).copy_(state["S"])
        state["out"] = (torch.empty((T, n), dtype=torch.complex128, pin_memory=True),
                        torch.empty(T, dtype=torch.int32, pin_memory=True),
                        torch.empty(T, dtype=torch.float64, pin_memory=True))
    if case.get("loads") == "zip":
        fd.set_zip(_alpha(case))
    return state


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["plan"].launch()
        conv, _, _ = state["plan"].wait()
        return {"V": state["V"], "iters": state["iters"], "converged": conv}
    if kind == "train":
        net, S, V = state["net"], state["S"], state["V"]
        for k in range(S.shape[0] // BATCH):
            net.train_step(S[k * BATCH:(k + 1) * BATCH], V[k * BATCH:(k + 1) * BATCH], lr=1e-3, want_loss=False)
        return {"weights": net.params()}
    fd, S = state["feeder"], state["S"]
    if kind == "scenarios":
        r = fd.solve_tensor(S, tol=TOL)
        return {k: r[k] for k in ("V", "iters", "vmin", "vmax", "viol", "bus_under", "bus_over", "status")}
    if kind == "learned":
        V, it, _, fallback, st = fd.solve_learned(state["net"], S, tol=TOL)
        return {"V": V, "iters": it, "fallback": fallback, "status": st}
    if kind == "host":
        V, it, _, st = fd.solve_host(S, tol=TOL, method="sparse", out=state["out"])
    elif kind == "dense":
        V, it, _, st = fd.solve(S, tol=TOL, precision=state["precision"])
    else:
        V, it, _, st = fd.solve(S, tol=TOL, precision="fp64" if kind == "tree64" else "mixed", method="sparse")
    return {"V": V, "iters": it, "status": st}


def work(case):
    """Bytes: loads in, voltages (and counts) out, once.  Operations: per bus and sweep a division-based current
    and the tree substitution's two passes (36), or the dense product (8 n^2 per column and sweep)."""
    kind = case["kind"]
    if kind == "batch":
        el = sum((nb - 1) * T for nb, T, _ in _batch_specs(case))
        return {"bytes": 32 * el, "flops": 36 * el * SWEEPS}
    if kind == "scenarios":
        el = (case["n_bus"] - 1) * case["scenarios"] * case["hours"]
        return {"bytes": 16 * el, "flops": 36 * el * SWEEPS}
    n = case["n_bus"] - 1
    if kind == "train":
        sizes, w = _first_weights(case)
        cols = case["steps"] * BATCH
        # forward, weight and input gradients; weights and Adam moments read and written at every step
        macs = sum(i * o for i, o in zip(sizes[:-1], sizes[1:]))
        return {"bytes": 32 * n * cols + case["steps"] * 24 * w.size, "flops": 6 * macs * cols}
    if kind == "poly":
        el = 3 * n * case["columns"]
        return {"bytes": 32 * el, "flops": 52 * el * SWEEPS}  # 3 x 3 branch blocks
    el = n * case["columns"]
    if kind == "dense":
        return {"bytes": 32 * el, "flops": 8 * n * el * SWEEPS}
    if kind == "learned":
        macs = 2 * n * 256 * 2 + 2 * 256 * 256
        return {"bytes": 32 * el, "flops": 36 * el * 6 + 2 * macs * case["columns"]}
    return {"bytes": 32 * el, "flops": (46 if case.get("loads") == "zip" else 36) * el * SWEEPS}


# ------------------------------------------------------------------------ the same in 64 bits, plain torch

def _levels(fr, to, n_bus):
    """Per tree level below the slack's children: the demand buses (row index) and their parents' rows."""
    depth, parent = np.zeros(n_bus, int), np.zeros(n_bus, int)
    for a, b in zip(fr, to):  # parents come before children in these feeders
        depth[b], parent[b] = depth[a] + 1, a
    out = []
    for d in range(2, int(depth.max()) + 1):
        kids = np.flatnonzero(depth == d)
        out.append((torch.tensor(kids - 1, device=_dev()), torch.tensor(parent[kids] - 1, device=_dev())))
    return out


def _tree_map(levels, z, vs):
    """I -> v_s - (sum over the path of z_b times the subtree sum of I), rows = buses (x phases) x columns."""
    def apply(I):
        L = torch.view_as_real(I).clone()
        for kids, par in reversed(levels):
            L.index_add_(0, par, L[kids])
        L = torch.view_as_complex(L)
        D = torch.einsum("bpq,bqt->bpt", z, L) if z.dim() == 3 else z[:, None] * L
        for kids, par in levels:
            D[kids] += D[par]
        return vs - D
    return apply


def _iterate(step, S, tol, alpha=None, max_iter=100):
    """Algorithm 1 column by column: V_0 = 1 (or the given source phasors), stop at max |step| <= tol."""
    apply, V0 = step
    T = S.shape[0]
    rows = S.shape[1] if V0.dim() == 0 else None
    out = torch.empty((T, S.shape[1]), dtype=torch.complex128, device=S.device)
    for a in range(0, T, 16_384):
        s = S[a:a + 16_384].to(torch.complex128).T.contiguous()
        if rows is None:  # polyphase: [bus][phase][column]
            s = s.view(-1, V0.shape[0], s.shape[1])
        V = torch.ones_like(s) if V0.dim() == 0 else torch.ones_like(s) * V0[None, :, None]
        live = torch.ones(s.shape[-1], dtype=torch.bool, device=s.device)
        for _ in range(max_iter):
            I = torch.conj(s / V)
            if alpha is not None:
                I = alpha[0][:, None] * I + alpha[1][:, None] * torch.conj(s) + alpha[2][:, None] * torch.conj(s) * V
            Vn = apply(I.resolve_conj())
            d = (Vn - V).abs().reshape(-1, s.shape[-1]).amax(0)
            V = torch.where(live, Vn, V)
            live &= d > tol
            if not bool(live.any()):
                break
        out[a:a + 16_384] = V.reshape(-1, s.shape[-1]).T
    return out


def _t(x):
    return torch.tensor(np.asarray(x), device=_dev())


def _exact_feeder(case, f, S, tol, alpha=None):
    fr, to, z = _branches(case, f)
    one = torch.ones((), dtype=torch.complex128, device=_dev())
    if case.get("topology") == "meshed":
        Y = np.zeros((f.n_bus, f.n_bus), complex)
        y = 1.0 / z
        for a, b, v in zip(fr, to, y):
            Y[a, a] += v
            Y[b, b] += v
            Y[a, b] -= v
            Y[b, a] -= v
        K = -np.linalg.inv(Y[1:, 1:])
        K, W = _t(K), _t(K @ Y[1:, 0] * f.v0)
        return _iterate((lambda I: K @ I + W[:, None], one), S, tol, alpha)
    return _iterate((_tree_map(_levels(fr, to, f.n_bus), _t(z), f.v0), one), S, tol, alpha)


def _exact_train(case, seed):
    f = _network(case)
    S = _loads(case, f, seed, case["steps"] * BATCH)
    V = _exact_feeder(case, f, S, 1e-13)
    order = torch.randperm(S.shape[0], generator=torch.Generator(device="cpu").manual_seed(seed)).to(S.device)
    x = torch.cat([S.real, S.imag], 1)
    y = torch.cat([V.real - 1.0, V.imag], 1)
    x = ((x - x.mean(0)) / x.std(0, unbiased=False))[order]
    y = ((y - y.mean(0)) / y.std(0, unbiased=False))[order]
    sizes, w = _first_weights(case)
    p, at = [], 0
    for i, o in zip(sizes[:-1], sizes[1:]):
        p += [_t(w[at:at + o * i].astype(np.float64)).reshape(o, i), _t(w[at + o * i:at + o * i + o].astype(np.float64))]
        at += o * i + o
    m, v = [torch.zeros_like(q) for q in p], [torch.zeros_like(q) for q in p]
    for k in range(case["steps"]):
        q = [t.clone().requires_grad_(True) for t in p]
        a = x[k * BATCH:(k + 1) * BATCH]
        for layer in range(0, len(q), 2):
            a = a @ q[layer].T + q[layer + 1]
            if layer + 2 < len(q):
                a = torch.nn.functional.gelu(a)
        g = torch.autograd.grad(((a - y[k * BATCH:(k + 1) * BATCH]) ** 2).mean(), q)
        for j in range(len(p)):
            m[j] = 0.9 * m[j] + 0.1 * g[j]
            v[j] = 0.999 * v[j] + 0.001 * g[j] ** 2
            p[j] = p[j] - 1e-3 * (m[j] / (1 - 0.9 ** (k + 1))) / ((v[j] / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    return {"weights": torch.cat([t.reshape(-1) for t in p])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "batch":
        Vs = []
        for k, (nb, T, sd) in enumerate(_batch_specs(case)):
            f = _make(nb, sd)
            S = G.load_tensor_device(f, T, seed + k, _dev(), step_minutes=G.step_minutes_for(T))
            Vs.append(_exact_feeder(case, f, S, TOL).reshape(-1))
        return {"V": torch.cat(Vs), "iters": None, "converged": None}
    if kind == "poly":
        f = G.make_feeder_poly(case["n_bus"], case["feeder"])
        v0 = _t(f.v0)
        step = _tree_map(_levels(f.from_bus, f.to_bus, f.n_bus), _t(f.z_blocks), v0[None, :, None])
        V0 = torch.ones(f.phases, dtype=torch.complex128, device=_dev())
        return {"V": _iterate((step, V0), _poly_loads(f, case["columns"], seed), 1e-13), "iters": None, "status": 0}
    f = _network(case)
    if kind == "scenarios":
        S = G.scenario_tensor_device(f, case["scenarios"], case["hours"], seed, _dev())
        V = _exact_feeder(case, f, S.reshape(-1, f.n_pq), TOL).reshape(S.shape)
        return {"V": V, "iters": None, "vmin": V.abs().amin(-1), "vmax": V.abs().amax(-1), "viol": None,
                "bus_under": None, "bus_over": None, "status": 0}
    S = _loads(case, f, seed)
    alpha = _t(_alpha(case)) if case.get("loads") == "zip" else None
    if kind == "learned":  # the iterates depend on the network's start: the point they end at
        return {"V": _exact_feeder(case, f, S, 1e-13), "iters": None, "fallback": None, "status": 0}
    V = _exact_feeder(case, f, S, TOL, alpha)
    return {"V": V.cpu() if kind == "host" else V, "iters": None, "status": 0}
