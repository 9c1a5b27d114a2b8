"""The FP64 sparse kernel on networks and loads that lie many decades apart (bound and plain side: plain64.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04578_gb300 import inputs as G  # noqa: E402
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
