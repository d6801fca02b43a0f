"""Gradients of the width-128 network where the tensor-core weight-gradient
kernel's tiles end: sequences of 1, 127, 128, 129 and 300 coarse positions, one
and several sequences, with one and several shares of the tiles per layer.
Against the oracle with BF16-rounded operands, with the bars of the other
gradient tests (up to 11 contractions in series: 3e-3 in L2 per tensor, every
element within 1.5e-2 of the tensor's largest)."""
import numpy as np
import pytest

import paper_2201_05280_gb300 as rpk
from oracle import surrogate as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,nseq,lq", [(1, 1, 1), (1, 5, 127), (2, 2, 128), (2, 3, 129), (1, 1, 300)])
def test_gradients_at_tile_edges(nb, nseq, lq):
    import torch
    cin, cout, width = 3, 2, 128
    rng = np.random.default_rng(100 * nb + lq)
    p = S.init_params(cin, cout, width, nb, seed=nb)
    v = S.flatten(p, nb).astype(np.float32)
    p = S.unflatten(v.astype(np.float64), cin, cout, width, nb)
    x = rng.normal(size=(nseq, 4 * lq, cin)).astype(np.float32)
    t = rng.normal(size=(nseq, 4 * lq, cout)).astype(np.float32)
    m = (rng.uniform(size=(nseq, 4 * lq)) < 0.75).astype(np.float32)
    net = rpk.Net(cin, cout, width, nb, seed=5)
    net.set_params(v)
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    loss = net.loss_grad(dev(x), dev(t), dev(m))
    g = S.unflatten(net.params(grads=True).astype(np.float64), cin, cout, width, nb)
    net.close()
    ref_loss, ref, _ = S.loss_and_grad(p, x.astype(np.float64), t.astype(np.float64), m.astype(np.float64), nb, cout,
                                       rnd=S.bf16)
    assert abs(loss - ref_loss) <= 1e-4 * ref_loss
    for k in ref:
        d = g[k] - ref[k]
        assert np.linalg.norm(d) <= 3e-3 * np.linalg.norm(ref[k]), k
        assert np.abs(d).max() <= 1.5e-2 * np.abs(ref[k]).max(), k
