"""Solves that meet a full device: TPF_ENOMEM or another way to the same result, and a handle that works afterwards.

The rest of the device's memory is held in one allocation while a call runs.  Kernels that the call may take have
run before, so that nothing but the library's buffers is allocated in between.
"""
import contextlib

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04578_gb300 import inputs as G  # noqa: E402
from paper_2403_04578_gb300 import tpf  # noqa: E402

pytestmark = pytest.mark.gpu
MB = 1 << 20
# Bounds the difference of two kernels' results: n 2^-53 times a drop of 0.05 pu, n = 999, and the map contracts.
BOUND = 2e-14


@contextlib.contextmanager
def _leave(bytes_):
    """At most about `bytes_` of device memory left inside."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = []
    for step in (1 << 30, 32 * MB, 2 * MB):
        while torch.cuda.mem_get_info()[0] >= bytes_ + step:
            n = (torch.cuda.mem_get_info()[0] - bytes_) // step * step
            held.append(torch.empty(n, dtype=torch.uint8, device="cuda"))
    try:
        yield
    finally:
        torch.cuda.synchronize()
        held.clear()
        torch.cuda.empty_cache()


def _warm(T):
    """Every FP64 dense kernel has run; the loads and outputs of a 999-bus solve, and its handle with K in place."""
    for n in (10, 40):
        f = G.make_feeder(n, 1)
        with tpf.Feeder.from_inputs(f) as fd:
            fd.solve(torch.from_numpy(G.load_tensor(f, 8, 1)).cuda(), precision="fp64", method="dense")
    f = G.make_feeder(1000, 1)
    S = torch.from_numpy(np.ascontiguousarray(G.load_tensor(f, T, 3))).cuda()
    fd = tpf.Feeder.from_inputs(f)
    fd.solve(S, precision="mixed", method="dense", tol=1e-10)
    return fd, S, (torch.empty_like(S), torch.empty(T, dtype=torch.int32, device="cuda"),
                   torch.empty(T, dtype=torch.float64, device="cuda"))


# K's digit planes take 29 MB; those of 2,000 columns' currents 88 MB.
@pytest.mark.parametrize("T,left", [(64, 20 * MB), (2000, 72 * MB)])
def test_solve_after_a_full_device(T, left):
    fd, S, (V, it, mm) = _warm(T)
    with fd:
        with _leave(left):
            try:
                fd.solve(S, V=V, iters=it, mismatch=mm, start="flat", precision="fp64",
                         method="dense", tol=1e-10)
            except tpf.TpfError as e:
                assert e.status == tpf.ENOMEM
        other = torch.cuda.Stream()
        V2, it2, _, st = fd.solve(S, precision="fp64", method="dense", tol=1e-10, stream=other)
        Vs, its, _, _ = fd.solve(S, precision="fp64", method="sparse", tol=1e-10)
    assert st == tpf.OK and bool((it2 == its).all())
    assert float((V2 - Vs).abs().max()) <= BOUND


@pytest.mark.parametrize("T,left", [(64, 20 * MB), (2000, 72 * MB)])
def test_fp64_dense_without_room_for_digit_planes(T, left):
    fd, S, (V, it, mm) = _warm(T)
    with fd:
        with _leave(left):
            _, _, _, st = fd.solve(S, V=V, iters=it, mismatch=mm, start="flat", precision="fp64",
                                   method="dense", tol=1e-10)
            plain = fd.stats()["kernel_launches"]
        V2, it2, mm2, st2 = fd.solve(S, precision="fp64", method="dense", tol=1e-10)
        assert fd.stats()["kernel_launches"] > plain  # four kernels a sweep instead of two
    assert st == st2 == tpf.OK and bool((it == it2).all())
    assert float((V - V2).abs().max()) <= BOUND
    assert float(mm.max()) <= 1e-8 and float(mm2.max()) <= 1e-8


def _expect_error(call):
    with pytest.raises(tpf.TpfError) as e:
        call()
    assert e.value.status in (tpf.ENOMEM, tpf.ECUDA)


def test_dense_form_after_a_full_device():
    # K (16 MB) is built by the first dense solve, which fails; the next one has to build all of it.
    f = G.make_feeder(1000, 1)
    S = torch.from_numpy(np.ascontiguousarray(G.load_tensor(f, 64, 3))).cuda()
    _warm(64)[0].close()
    with tpf.Feeder.from_inputs(f) as fd:
        Vs, its, _, _ = fd.solve(S, precision="fp64", method="sparse", tol=1e-10)
        for left in (8 * MB, 20 * MB):
            with _leave(left):
                _expect_error(lambda: fd.solve(S, precision="mixed", method="dense", tol=1e-10))
        V, it, _, st = fd.solve(S, precision="mixed", method="dense", tol=1e-10)
    assert st == tpf.OK and bool((it > 0).all())
    assert float((V - Vs).abs().max()) <= 1e-8  # the mixed path's bound


def test_workspace_after_a_full_device():
    # 20,000 columns need seven planes of 82 to 164 MB; the second one finds no room.
    fd, S, _ = _warm(128)
    with fd:
        V, it, _, _ = fd.solve(S, precision="mixed", method="dense", tol=1e-10)
        big = S.repeat(157, 1)[:20_000].contiguous()
        out = torch.empty_like(big)
        with _leave(240 * MB):
            _expect_error(lambda: fd.solve(big, V=out, start="flat", precision="mixed", method="dense", tol=1e-10))
        V2, it2, _, st = fd.solve(S, precision="mixed", method="dense", tol=1e-10)
    assert st == tpf.OK and torch.equal(V, V2) and torch.equal(it, it2)
