"""Training batches of more columns than a grid has rows of 32 (csrc/tpf_mlp_train.cu).

The batch repeats 128 columns, so that its mean gradient is theirs.  Differences: every dZ is rounded to BF16 at
another scale (2^-9 each, in two factors), and FP32 sums of 131,080 products of 16 columns lose at most 2^-24 each,
of the mean absolute product: taken as four times the largest gradient (loads and voltages go together).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2403_04578_gb300 import inputs as G  # noqa: E402
from paper_2403_04578_gb300 import tpf  # noqa: E402

pytestmark = pytest.mark.gpu


def test_two_million_columns():
    B = 65_536 * 32 + 128
    f = G.make_feeder(3, 1)
    S = torch.from_numpy(np.ascontiguousarray(G.load_tensor(f, 128, 1, step_minutes=11.0))).cuda()
    with tpf.Feeder.from_inputs(f) as fd:
        V = fd.solve(S, tol=1e-10, method="sparse")[0]
    net = tpf.LearnedStart(f.n_pq, hidden=128, hidden_layers=1, max_batch=B)
    net.fit_normalization(S, V)
    loss, grad = net.gradients(S, V)
    big = [x.repeat(B // 128, 1) for x in (S, V)]
    loss_b, grad_b = net.gradients(*big)
    assert loss_b == pytest.approx(loss, rel=1e-3)
    assert np.abs(grad_b - grad).max() <= (2.0 ** -8 + 131_080 * 2.0 ** -24) * 4 * np.abs(grad).max()
    w = net.params()
    net.train_step(*big, want_loss=False)
    assert not np.array_equal(net.params(), w)
    net.close()
