"""The power mismatch that the FP64 sparse kernel reports, against its definition at the returned V.

max_i |V_i conj((Y V)_i) + S_i| with the branch currents y (V_parent - V).  Differences of neighbouring voltages
are exact; the products, sums and the last product round to at most 16 2^-53 of the currents that meet at a bus, on
either side, and the kernel's integers to 2^-49 of the largest load for each of them (at most sixteen).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04578_gb300 import inputs as G  # noqa: E402
from paper_2403_04578_gb300 import tpf  # noqa: E402

pytestmark = pytest.mark.gpu


def _mismatch(fr, to, z, V, S):
    Vb = np.concatenate([np.ones((V.shape[0], 1), complex), V], 1)
    y = (z.real - 1j * z.imag) / (z.real ** 2 + z.imag ** 2)
    J = y * (Vb[:, fr] - Vb[:, to])  # into bus to
    bal = np.zeros_like(Vb)
    for b in range(len(fr)):
        bal[:, to[b]] -= J[:, b]
        bal[:, fr[b]] += J[:, b]
    size = np.zeros(Vb.shape)
    for b in range(len(fr)):
        size[:, to[b]] += np.abs(J[:, b])
        size[:, fr[b]] += np.abs(J[:, b])
    bound = 2.0 ** -48 * (size[:, 1:] + np.abs(S)).max(1) + 2.0 ** -45 * np.abs(S).max(1)
    return np.abs(V * np.conj(bal[:, 1:]) + S).max(1), bound


@pytest.mark.parametrize("n_bus", [12, 200, 700])
@pytest.mark.parametrize("z_scale", [1.0, 1e-6, 1e-12, 1e-14, 1e-16])
def test_mismatch(n_bus, z_scale):
    f = G.make_feeder(n_bus, 3)
    z = f.z_pu.copy()
    stiff = np.arange(len(z)) % 3 == 1
    z[stiff] *= z_scale
    S = G.load_tensor(f, 600, 5)
    with tpf.Feeder(f.n_bus, f.from_bus, f.to_bus, z, f.slack, f.v0, f.pq_bus) as fd:
        V, it, mm, st = fd.solve(torch.from_numpy(np.ascontiguousarray(S)).cuda(), precision="fp64", method="sparse",
                                 tol=1e-10)
    assert st == tpf.OK
    ref, bound = _mismatch(f.from_bus, f.to_bus, z, V.cpu().numpy(), S)
    assert (np.abs(mm.cpu().numpy() - ref) <= bound).all()
