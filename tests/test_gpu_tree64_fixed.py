"""The FP64 sparse kernel's fixed-point sums (csrc/tpf_tree64.cu) against the FP64 dense path.

Both iterate the same map with every result rounded near 2^-53 (V is about 1 pu, sums of up to 1,023 terms of a
voltage drop of at most 0.3 pu), so iterates agree within 2e-14 pu and counts are equal.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04578_gb300 import inputs as G  # noqa: E402
from paper_2403_04578_gb300 import tpf  # noqa: E402

pytestmark = pytest.mark.gpu
BOUND = 2e-14


def _pair(fd, S, V0=None, **kw):
    out = []
    for method in ("sparse", "dense"):
        V = None if V0 is None else V0.clone()
        out.append(fd.solve(S, V=V, precision="fp64", method=method, start=None if V0 is None else "given", **kw))
    return out


@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 127, 128, 129, 255, 500, 1023])
@pytest.mark.parametrize("zip_loads", [False, True])
def test_sizes(n, zip_loads):
    f = G.make_feeder(n + 1, n)
    S = torch.from_numpy(np.ascontiguousarray(G.load_tensor(f, 65, 3))).cuda()
    with tpf.Feeder.from_inputs(f) as fd:
        if zip_loads:
            fd.set_zip(np.random.default_rng(n).dirichlet([2, 1, 1], n).T.copy())
        (V, it, mm, st), (Vd, itd, _, std) = _pair(fd, S, tol=1e-10)
        assert st == tpf.OK and std == tpf.OK
        assert float((V - Vd).abs().max()) <= BOUND and bool((it == itd).all())
        assert float(mm.max()) <= 1e-8
        for k in (1, 3):  # iterates on the way
            (V, it, _, _), (Vd, itd, _, _) = _pair(fd, S, tol=0.0, max_iter=k)
            assert float((V - Vd).abs().max()) <= BOUND and bool((it == itd).all())


@pytest.mark.parametrize("n", [2049, 4096])
def test_eight_buses_per_thread(n):
    f = G.make_feeder(n + 1, 7)
    S = torch.from_numpy(np.ascontiguousarray(G.load_tensor(f, 20, 3))).cuda()
    with tpf.Feeder.from_inputs(f) as fd:
        V, it, mm, st = fd.solve(S, tol=1e-12, precision="fp64", method="sparse")
        Vm, itm, _, stm = fd.solve(S, tol=1e-10, precision="mixed", method="sparse")
    assert st == tpf.OK and stm == tpf.OK
    # The mixed path's bound; the power balance of FP64 voltages: 1e-16 pu times admittances below 1e4 pu.
    assert float((V - Vm).abs().max()) <= 1e-8 and float(mm.max()) <= 1e-9


def test_out_of_range():
    """What leaves the integers' range goes back to FP64 throughout, column by column."""
    f = G.make_feeder(130, 4)
    S = torch.from_numpy(np.ascontiguousarray(G.load_tensor(f, 40, 3))).cuda()
    S[3, 5] = float("nan")
    S[4, 100] = float("inf")
    S[5, 20] = 1e300
    S[6] *= 40.0       # no solution
    S[7] *= 1e-290
    S[8] = 0.0
    V0 = torch.full_like(S, 1.0)
    V0[10] *= 0.1      # currents ten times the loads
    V0[11] *= 2.5      # beyond 2 pu
    V0[12] *= -1.0
    V0[13, 7] = 0.0    # an infinite current
    bad = torch.zeros(40, dtype=torch.bool)
    bad[[3, 4, 5, 6, 13]] = True
    with tpf.Feeder.from_inputs(f) as fd:
        (V, it, _, st), (Vd, itd, _, std) = _pair(fd, S, V0=V0, tol=1e-10, max_iter=40)
    assert st == tpf.ENOCONV and std == tpf.ENOCONV
    assert bool((it == itd).all()) and bool((it.cpu()[bad] == -40).all()) and bool((it.cpu()[~bad] > 0).all())
    assert float((V - Vd).abs().cpu()[~bad].max()) <= BOUND


@pytest.mark.parametrize("v0", [1.9, 2.5, 30.0])
def test_source_voltage(v0):
    f = G.make_feeder(60, 4)
    S = torch.from_numpy(np.ascontiguousarray(G.load_tensor(f, 40, 3))).cuda()
    with tpf.Feeder(f.n_bus, f.from_bus, f.to_bus, f.z_pu, f.slack, v0 + 0.1j, f.pq_bus) as fd:
        (V, it, _, st), (Vd, itd, _, _) = _pair(fd, S, tol=1e-10)
    assert st == tpf.OK and bool((it == itd).all())
    assert float((V - Vd).abs().max()) <= BOUND * v0
