"""Plain FP64 sweeps beside the FP64 dense and sparse kernels (used by the tests of these).

The FP64 dense and sparse kernels work in fixed point; the plain side is the allocation-free solve, whose sweeps
are FP64 FMAs.  All iterate the same map.  A plain sweep's rounding is at most n 2^-53 sum_j |K_ij| |I_j| (up to
400 buses and a voltage drop of at most 0.2 pu: 9e-15 pu) and the map contracts, so 2e-14 pu bounds the
difference of the iterates.
"""
import numpy as np
import torch

from paper_2403_04578_gb300 import tpf

BOUND = 2e-14


def net_of(f, extra=()):
    """Feeder.__init__'s first four arguments, with extra branches (bus, z), each to a new last bus."""
    fr, to, z = list(f.from_bus), list(f.to_bus), list(f.z_pu)
    n_bus = f.n_bus
    for bus, zz in extra:
        fr.append(bus)
        to.append(n_bus)
        z.append(zz)
        n_bus += 1
    return n_bus, np.array(fr, np.int32), np.array(to, np.int32), np.array(z, complex)


def _plain(net, S, tol, max_iter, V0):
    n = net[0] - 1
    K, W = tpf.precompute_host(*net, 0, 1.0 + 0j, np.arange(1, net[0], dtype=np.int32))
    K = torch.from_numpy(np.ascontiguousarray(K)).cuda().reshape(n, n)
    W = torch.from_numpy(np.ascontiguousarray(W)).cuda().reshape(-1)
    V = torch.empty_like(S) if V0 is None else V0.clone()
    it = torch.empty(S.shape[0], dtype=torch.int32, device=S.device)
    tpf.solve_fp64_noalloc(K, W, S, V, iters=it, tol=tol, max_iter=max_iter, given_start=V0 is not None)
    return V, it


def check_plain(net, S, method, tol=1e-12, max_iter=100, V0=None):
    """The FP64 solve gives the plain sweeps' iterates and counts; returns the counts."""
    S = torch.from_numpy(np.ascontiguousarray(S)).cuda()
    V0 = None if V0 is None else torch.from_numpy(np.ascontiguousarray(V0)).cuda()
    Vp, itp = _plain(net, S, tol, max_iter, V0)
    with tpf.Feeder(*net, 0, 1.0 + 0j, np.arange(1, net[0], dtype=np.int32)) as fd:
        V, it, _, _ = fd.solve(S, V=None if V0 is None else V0.clone(), precision="fp64", method=method, tol=tol,
                               max_iter=max_iter, start=None if V0 is None else "given")
    assert float((V - Vp).abs().max()) <= BOUND
    assert bool((it == itp).all())
    return it
