"""Lightly loaded buses near zero voltage in the FP64 kernels, against plain FP64 sweeps (plain64.py).

Every load is at most half of |V_0| times the column's largest, so no current is far above that of a column at
1 pu, and the bound of plain64.py holds.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04578_gb300 import inputs as G  # noqa: E402
from paper_2403_04578_gb300 import tpf  # noqa: E402
from plain64 import BOUND, check_plain, net_of  # noqa: E402

pytestmark = pytest.mark.gpu


LOW = [0.6, 0.3, 0.1, 1e-2, 1e-4, 3e-5, 1e-6, 1e-8]


def _case(low):
    f = G.make_feeder(150, 9)
    S = G.load_tensor(f, 40, 3)
    r = np.random.default_rng(4)
    V0 = np.ones(S.shape, complex)
    at = np.arange(5, S.shape[1], 12)
    V0[:, at] = low * np.exp(1j * r.uniform(-3.0, 3.0, (40, len(at))))
    S[:, at] *= 0.5 * low
    return f, S, V0


@pytest.mark.parametrize("method", ["dense", "sparse"])
@pytest.mark.parametrize("low", LOW)
def test_low_voltage(low, method):
    f, S, V0 = _case(low)
    for k in (1, 2):
        check_plain(net_of(f), S, method, tol=0.0, max_iter=k, V0=V0)


@pytest.mark.parametrize("low", LOW)
def test_low_voltage_zip(low):
    # The dense path's ZIP currents are FP64 divisions at every voltage.
    f, S, V0 = _case(low)
    S, V0 = (torch.from_numpy(x).cuda() for x in (S, V0))
    with tpf.Feeder.from_inputs(f) as fd:
        fd.set_zip(np.random.default_rng(2).dirichlet([2, 1, 1], f.n_pq).T.copy())
        V, Vd = (fd.solve(S, V=V0.clone(), precision="fp64", method=m, start="given", tol=0.0, max_iter=1)[0]
                 for m in ("sparse", "dense"))
    assert float((V - Vd).abs().max()) <= BOUND
