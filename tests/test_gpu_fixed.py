"""The FP64 dense path's fixed-point sweeps (csrc/tpf_fixed.cu) against the plain FP64 kernels.

The plain side is the allocation-free solve, whose sweeps are FP64 FMAs whatever the size.  Both iterate the
same map; a plain sweep's rounding is at most n 2^-53 sum_j |K_ij| |I_j| (n <= 400, the sum a voltage drop of
at most 0.2 pu: 9e-15 pu) and the map contracts, so 2e-14 pu bounds the difference of the iterates.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04578_gb300 import inputs as G  # noqa: E402
from paper_2403_04578_gb300 import tpf  # noqa: E402

pytestmark = pytest.mark.gpu
BOUND = 2e-14


def _both(f, S, tol=1e-10, max_iter=100, V0=None):
    dev = torch.device("cuda")
    Sd = torch.from_numpy(np.ascontiguousarray(S)).to(dev)
    K, W = tpf.precompute_host(f.n_bus, f.from_bus, f.to_bus, f.z_pu, f.slack, f.v0, f.pq_bus)
    Kd = torch.from_numpy(np.ascontiguousarray(K)).to(dev).reshape(f.n_pq, f.n_pq)
    Wd = torch.from_numpy(np.ascontiguousarray(W)).to(dev).reshape(-1)
    start = torch.empty_like(Sd) if V0 is None else torch.from_numpy(V0).to(dev)
    Vp = start.clone()
    itp = torch.empty(S.shape[0], dtype=torch.int32, device=dev)
    tpf.solve_fp64_noalloc(Kd, Wd, Sd, Vp, iters=itp, tol=tol, max_iter=max_iter, given_start=V0 is not None)
    with tpf.Feeder.from_inputs(f) as fd:
        V, it, mm, st = fd.solve(Sd, V=start.clone() if V0 is not None else None, precision="fp64", method="dense",
                                 tol=tol, max_iter=max_iter, start="given" if V0 is not None else None)
    return [x.cpu().numpy() for x in (V, it, mm, Vp, itp)]


# Demand buses around the rule's line (17), the K steps of 16, the chunks of 64 and the tiles of 128;
# columns around the tiles of 64; and more tiles than two per SM.
@pytest.mark.parametrize("n_pq,T", [(17, 1), (31, 63), (33, 64), (63, 65), (64, 130), (65, 1), (127, 64), (128, 200),
                                    (129, 65), (255, 64), (257, 129), (399, 66), (33, 40_000), (130, 10_000)])
def test_sizes(n_pq, T):
    f = G.make_feeder(n_pq + 1, n_pq)
    V, it, mm, Vp, itp = _both(f, G.load_tensor(f, T, 7))
    assert np.abs(V - Vp).max() <= BOUND
    assert (it == itp).all() and (it > 0).all()
    assert mm.max() <= 1e-8


@pytest.mark.parametrize("max_iter", [1, 2, 5])
def test_every_iterate(max_iter):
    # The iterates before convergence, from a start far from the solution, at loads of twelve decades.
    f = G.make_feeder(130, 4)
    r = np.random.default_rng(1)
    S = G.load_tensor(f, 70, 3)
    S = S * 10.0 ** r.uniform(-12, 0, S.shape)
    V0 = (1.0 + 0.1 * r.standard_normal(S.shape)) + 0.1j * r.standard_normal(S.shape)
    V, it, _, Vp, itp = _both(f, S, tol=0.0, max_iter=max_iter, V0=V0)
    assert np.abs(V - Vp).max() <= BOUND
    assert (it == itp).all()


def test_columns_without_fixed_point_form():
    f = G.make_feeder(100, 2)
    S = G.load_tensor(f, 80, 5)
    S[3, 7] = np.nan
    S[10, 0] = np.inf
    S[11, 50] = 1e303          # above 2^1000: plain FP64
    S[12, 50] = 1e300          # below: fixed point, and a step beyond 1e30
    S[20] = 0.0
    S[21] *= 1e-300
    S[30] *= 1e4               # no solution
    V, it, _, Vp, itp = _both(f, S, max_iter=30)
    bad = np.zeros(80, bool)
    bad[[3, 10, 11, 12, 30]] = True
    assert (it == itp).all() and (it[bad] == -30).all() and (it[~bad] > 0).all()
    assert np.abs(V[~bad] - Vp[~bad]).max() <= BOUND
    for t in (3, 10):
        np.testing.assert_array_equal(np.isfinite(V[t]), np.isfinite(Vp[t]))
    for t in (11, 12):
        np.testing.assert_allclose(V[t], Vp[t], rtol=1e-12, atol=1e-13 * np.abs(Vp[t]).max())


@pytest.mark.parametrize("scale", [0.1, 0.4, 1.9, 3.0])
def test_currents_beyond_the_integer_quotient(scale):
    # Voltages of 2 pu and more, or currents above four times the largest load, take FP64 divisions; loads ten
    # times larger in a drop of up to 3 pu round to 15 times the bound of a sweep (3e-13 pu).
    f = G.make_feeder(150, 9)
    S = G.load_tensor(f, 70, 3)
    r = np.random.default_rng(2)
    V0 = np.ones(S.shape, complex)
    V0[::2] = scale * np.exp(1j * r.uniform(-3.0, 3.0, (35, S.shape[1])))
    for k in (1, 2):
        V, it, _, Vp, itp = _both(f, S, tol=0.0, max_iter=k, V0=V0)
        assert np.abs(V - Vp).max() <= 15 * BOUND
        assert (it == itp).all()
