"""Host-buffer solves in the sparse form: cut into chunks by bytes where copies overlap, and with the device
solve's results however they are cut.

64 MB of loads are several chunks of about 16 MB in page-locked memory, and one in pageable memory, which the host
thread copies itself.  A chunk is one kernel launch, and columns do not depend on one another.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04578_gb300 import inputs as G  # noqa: E402
from paper_2403_04578_gb300 import tpf  # noqa: E402

pytestmark = pytest.mark.gpu


def _feeder(kind):
    if kind == "poly":
        f = G.make_feeder_poly(67, 3)
        fd = tpf.Feeder.poly(f.n_bus, f.from_bus, f.to_bus, f.z_blocks, f.phases, f.slack, f.v0, f.pq_bus)
        return fd, G.load_tensor_poly(f, 20_201, 3).reshape(20_201, -1)
    f = G.make_feeder(200, 3)
    fd = tpf.Feeder.from_inputs(f)
    if kind == "zip":
        fd.set_zip(np.random.default_rng(1).dirichlet([2, 1, 1], f.n_pq).T.copy())
    return fd, G.load_tensor(f, 20_201, 3)


@pytest.mark.parametrize("kind", ["mixed", "fp64", "zip", "poly"])
# page-locked: loads, results, counts and mismatches
@pytest.mark.parametrize("pinned,cut", [((1, 1, 1), True), ((1, 1, 0), True), ((0, 1, 1), True), ((0, 1, 0), False),
                                        ((1, 0, 0), False), ((0, 0, 0), False)])
def test_chunks(kind, pinned, cut):
    fd, S = _feeder(kind)
    S = torch.from_numpy(np.ascontiguousarray(S))
    T, n = S.shape
    kw = dict(precision="fp64" if kind == "fp64" else "mixed", method="sparse", tol=1e-10)

    def host(shape, dtype, pin):
        return torch.empty(shape, dtype=dtype, pin_memory=bool(pin))

    Sh = host((T, n), torch.complex128, pinned[0]).copy_(S)
    out = (host((T, n), torch.complex128, pinned[1]), host((T,), torch.int32, pinned[2]),
           host((T,), torch.float64, pinned[2]))
    with fd:
        V, it, mm, st = fd.solve(S.cuda(), **kw)
        Vh, ith, mmh, sth = fd.solve_host(Sh, out=out, **kw)
        assert (fd.stats()["kernel_launches"] > 1) == cut and fd.stats()["columns"] == T
    assert st == sth == tpf.OK
    assert torch.equal(Vh, V.cpu()) and torch.equal(ith, it.cpu()) and torch.equal(mmh, mm.cpu())
