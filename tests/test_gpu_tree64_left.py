"""Columns that leave the FP64 sparse kernel's integers: in place up to 64 buses and from 513 on, at two buses per
thread between these by a second launch.

Against the FP64 dense path, with the bound of test_gpu_tree64_fixed.py (2e-14 pu).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04578_gb300 import inputs as G  # noqa: E402
from paper_2403_04578_gb300 import tpf  # noqa: E402
from plain64 import BOUND  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 64, 65, 130, 512, 513])
@pytest.mark.parametrize("zip_loads", [False, True])
@pytest.mark.parametrize("leaving", [[], [0], [3, 4, 69], list(range(70))])
def test_columns_that_leave(n, zip_loads, leaving):
    f = G.make_feeder(n + 1, n)
    S = torch.from_numpy(np.ascontiguousarray(G.load_tensor(f, 70, 3))).cuda()
    V0 = torch.full_like(S, 1.0)
    V0[leaving, n // 2] *= 0.4  # below half a pu
    with tpf.Feeder.from_inputs(f) as fd:
        if zip_loads:
            fd.set_zip(np.random.default_rng(n).dirichlet([2, 1, 1], n).T.copy())
        Vd, itd, _, _ = fd.solve(S, V=V0.clone(), precision="fp64", method="dense", start="given", tol=1e-10)
        V, it, mm, st = fd.solve(S, V=V0.clone(), precision="fp64", method="sparse", start="given", tol=1e-10)
        s = fd.stats()
    assert st == tpf.OK and s["converged"] == 70 and s["kernel_launches"] == 1 + (bool(leaving) and 64 < n <= 512)
    assert s["sweeps"] == int(it.max())
    assert float((V - Vd).abs().max()) <= BOUND and bool((it == itd).all()) and float(mm.max()) <= 1e-8
