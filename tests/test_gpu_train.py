"""The training kernels (csrc/tpf_mlp_train.cu) at the edges of their tiles: gradients against the FP64
reference, and the first Adam step against its closed form.

A gradient is compared as in test_gpu_mlp: relative L2 error <= 2e-2 with up to four weight layers.  Every
product rounds both operands to BF16 (rms 1.1e-3), so ten layers, 19 products in a chain, come to 7e-3 rms of
their own; 5e-2 bounds them.  From zero moments Adam moves a weight by lr g / (|g| + eps) exactly.
"""
import numpy as np
import pytest

from oracle import mlp as OM
from paper_2403_04578_gb300 import tpf

pytestmark = pytest.mark.gpu


def _norm(A):
    mu, sd = A.mean(axis=0), A.std(axis=0)
    return (A - mu) / sd


# (demand buses, units, hidden layers, columns): features that fill their padding exactly, exceed it by two
# and leave most of it; widths that are no multiple of 32; more layers than one launch of the weight
# gradients takes; batches of two to sixteen K chunks (the splits of the weight gradients).
@pytest.mark.parametrize("n,hidden,layers,B", [(64, 128, 1, 128), (65, 100, 2, 256), (16, 64, 9, 384),
                                               (199, 256, 3, 1024), (299, 384, 2, 640)])
def test_gradients_and_adam(n, hidden, layers, B):
    import torch

    r = np.random.default_rng(n)
    S = r.uniform(0.01, 0.1, (B, n)) + 1j * r.uniform(0.0, 0.03, (B, n))
    V = 1.0 - 0.05 * r.random((B, n)) - 0.03j * r.random((B, n))
    Sd, Vd = torch.from_numpy(S).cuda(), torch.from_numpy(V).cuda()
    net = tpf.LearnedStart(n, hidden=hidden, hidden_layers=layers, max_batch=1024, seed=3)
    net.fit_normalization(Sd, Vd)
    sizes = net.sizes
    Ws = [r.uniform(-1, 1, (o, i)).astype(np.float32) * np.float32(np.sqrt(6.0 / (i + o)))
          for i, o in zip(sizes[:-1], sizes[1:])]
    bs = [r.normal(0, 0.05, o).astype(np.float32) for o in sizes[1:]]
    flat = np.concatenate([np.concatenate([w.ravel(), b]) for w, b in zip(Ws, bs)])
    net.set_params(flat)
    assert np.array_equal(net.params(), flat)
    loss, g = net.gradients(Sd, Vd)
    ref = OM.MLP([w.astype(np.float64) for w in Ws], [b.astype(np.float64) for b in bs])
    X = _norm(np.concatenate([S.real, S.imag], axis=1))
    Y = _norm(np.concatenate([V.real - 1.0, V.imag], axis=1))
    loss_ref, gW, gb = ref.gradients(X, Y)
    g_ref = np.concatenate([np.concatenate([w.ravel(), b]) for w, b in zip(gW, gb)])
    assert loss == pytest.approx(loss_ref, rel=2e-2)
    assert np.linalg.norm(g - g_ref) <= (2e-2 if layers < 4 else 5e-2) * np.linalg.norm(g_ref)
    # Another batch size in between must leave nothing behind.
    net.gradients(Sd[:128], Vd[:128])
    lr = 1e-3
    assert net.train_step(Sd, Vd, lr=lr) == pytest.approx(loss, rel=1e-6)
    step = flat.astype(np.float64) - net.params()
    want = lr * g / (np.abs(g) + 1e-8)
    big = np.abs(g) > 1e-6
    # FP32 rounding of w - step: 2^-24 |w| <= 6e-8 against steps of 1e-3.
    assert big.mean() > 0.5 and np.abs(step - want)[big].max() <= 1e-6
    net.close()
