"""The FP64 sparse kernel on networks and loads that lie many decades apart (bound and plain side: plain64.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04578_gb300 import inputs as G  # noqa: E402
from paper_2403_04578_gb300 import tpf  # noqa: E402
from plain64 import check_plain, net_of  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("z", [1e3, 1e6, 1e9, 1e12])
def test_large_impedance(z):
    # An unloaded stub of a large impedance (an open switch).
    f = G.make_feeder(200, 5)
    S = G.load_tensor(f, 70, 3)
    S = np.concatenate([S, np.zeros((70, 1))], 1)
    assert bool((check_plain(net_of(f, [(77, z * (1 + 1j))]), S, "sparse") > 0).all())


@pytest.mark.parametrize("big", [1.0, 30.0, 1e3, 1e6])
def test_one_large_load(big):
    # One load of thousands of times the others, 0.01 pu below the source.
    f = G.make_feeder(400, 6)
    S = G.load_tensor(f, 66, 3)
    S = np.concatenate([S, np.full((66, 1), big * (1 + 0.3j))], 1)
    check_plain(net_of(f, [(0, 0.01 / big * (0.6 + 0.8j))]), S, "sparse")


@pytest.mark.parametrize("share", [0.5, 0.7])
def test_couplers(share):
    # More than half of the branches next to zero: the lines are no large impedances, and no column leaves the
    # integers (at this size a second launch would solve it).
    f = G.make_feeder(300, 8)
    z = f.z_pu.copy()
    z[np.random.default_rng(1).permutation(len(z))[:int(share * len(z))]] *= 1e-5
    S = G.load_tensor(f, 70, 3)
    f.z_pu[:] = z
    check_plain(net_of(f), S, "sparse")
    with tpf.Feeder(*net_of(f), 0, 1.0 + 0j, np.arange(1, f.n_bus, dtype=np.int32)) as fd:
        fd.solve(torch.from_numpy(np.ascontiguousarray(S)).cuda(), precision="fp64", method="sparse", tol=1e-12)
        assert fd.stats()["kernel_launches"] == 1
