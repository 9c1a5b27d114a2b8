"""The mixed dense path's residual kernels (csrc/tpf_residual.cu) at the edges of their blocks.

Mixed results agree with the FP64 path within 1e-8 pu (the bound of every mixed test here), whatever the
shape of the tree: a star puts all buses into one list of children, a chain gives every bus one child.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04578_gb300 import inputs as G  # noqa: E402
from paper_2403_04578_gb300 import tpf  # noqa: E402

pytestmark = pytest.mark.gpu


def _tree(shape, n, seed):
    r = np.random.default_rng(seed)
    if shape == "random":
        f = G.make_feeder(n + 1, seed)
        return f.from_bus, f.to_bus, f.z_pu
    to = np.arange(1, n + 1, dtype=np.int32)
    # A star below bus 1; a chain.  Impedances such that the drops stay near 0.05 pu.
    fr = np.where(to == 1, 0, 1 if shape == "star" else to - 1).astype(np.int32)
    z = (r.uniform(0.5, 1.0, n) + 1j * r.uniform(0.5, 1.0, n)) * (0.05 / n if shape == "star" else 0.1 / n)
    order = r.permutation(n)  # branches in any order, in either direction
    flip = r.random(n) < 0.5
    fr, to = np.where(flip, to, fr)[order], np.where(flip, fr, to)[order]
    return fr.astype(np.int32), to.astype(np.int32), z[order]


# Chains of a thousand and more branches of 1e-4 pu are past the mixed path's reach (rounding V to FP32
# times admittances of 1e4 pu keeps the step above switch_tol), so chains end at 511.
SIZES = [1, 2, 63, 64, 127, 128, 129, 255, 256, 257, 511, 1023, 1025, 2047, 2048]


@pytest.mark.parametrize("n,shape", [(n, s) for s in ("random", "star", "chain") for n in SIZES
                                     if s != "chain" or n <= 511])
def test_edges(n, shape):
    fr, to, z = _tree(shape, n, n)
    r = np.random.default_rng(1)
    T = 37
    p = r.uniform(0.2, 1.0, (T, n)) * (1.0 if shape != "random" else 0.01) / n
    S = torch.from_numpy(p + 0.3j * p).cuda()
    with tpf.Feeder(n + 1, fr, to, z, 0, 1.02 + 0.01j, np.arange(1, n + 1, dtype=np.int32)) as fd:
        Vx, itx, _, stx = fd.solve(S, tol=1e-11, precision="fp64", method="dense")
        V, it, mm, st = fd.solve(S, tol=1e-10, precision="mixed", method="dense")
        assert stx == tpf.OK and st == tpf.OK
        assert float((V - Vx).abs().max()) <= 1e-8 and bool((it > 0).all())
        assert float(mm.max()) <= 1e-6
        for start in ("given", "warm"):
            V0 = Vx * (1.0 + 2e-3)
            Vg, itg, _, st = fd.solve(S, V=V0, tol=1e-10, precision="mixed", method="dense", start=start)
            assert st == tpf.OK and float((Vg - Vx).abs().max()) <= 1e-8


def test_unconverged_columns():
    f = G.make_feeder(200, 3)
    S = torch.from_numpy(np.ascontiguousarray(G.load_tensor(f, 130, 2))).cuda()
    S[5] *= 1e3
    S[6, 3] = float("nan")
    with tpf.Feeder.from_inputs(f) as fd:
        V, it, mm, st = fd.solve(S, tol=1e-10, max_iter=25, precision="mixed", method="dense")
        Vx, itx, _, _ = fd.solve(S, tol=1e-11, max_iter=25, precision="fp64", method="dense")
    assert st == tpf.ENOCONV and it[5] == -25 and it[6] == -25
    ok = torch.ones(130, dtype=torch.bool)
    ok[[5, 6]] = False
    assert bool((it.cpu()[ok] > 0).all()) and float((V - Vx).abs().cpu()[ok].max()) <= 1e-8
