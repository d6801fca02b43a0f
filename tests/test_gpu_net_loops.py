"""Width-128 network passes in which a thread block takes several tiles: the residual-block
kernel's buffers, accumulators and weight ring across tiles, the tile list of ragged
sequences (tiles end at 124 positions), the weight-gradient kernel's two staging buffers
and sums over tiles. Against the oracle with BF16-rounded operands and the bars of the
other network tests: forward 1e-3 in L2 and 3e-3 per element, gradients 3e-3 and 1.5e-2.
(More (layer, half) pairs than SMs: test_gpu_net_memory.py, 64 blocks.)"""
import numpy as np
import pytest

import paper_2201_05280_gb300 as rpk
from oracle import surrogate as S

pytestmark = pytest.mark.gpu

WIDTH = 128


def _net(cin, cout, nb, seed):
    rng = np.random.default_rng(seed)
    p = S.init_params(cin, cout, WIDTH, nb, seed=seed)
    for k in p:
        if "_b" in k:
            p[k] = rng.normal(0, 0.1, p[k].shape)
    v = S.flatten(p, nb).astype(np.float32)
    net = rpk.Net(cin, cout, WIDTH, nb, seed=1)
    net.set_params(v)
    return net, S.unflatten(v.astype(np.float64), cin, cout, WIDTH, nb), rng


def test_ragged_forward_of_many_tiles():
    import torch
    cin, cout = 3, 2
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    net, p, rng = _net(cin, cout, 1, 21)
    lens = np.array([1, 123, 124, 125, 248, 249] * 12 + [1, 2, 3, 4, 5, 6, 7] * (3 * sms // 7 + 1))
    rng.shuffle(lens)  # at least 3 tiles for every block, long and short ones among them
    assert sum(-(-n // 124) for n in lens) > 3 * sms
    x = rng.normal(size=(4 * int(lens.sum()), cin)).astype(np.float32)
    y = net.forward_ragged(torch.tensor(x, device="cuda"), [4 * int(n) for n in lens]).cpu().numpy()
    net.close()
    at = np.concatenate([[0], np.cumsum(4 * lens)])
    ref = np.zeros(y.shape)
    for n in np.unique(lens):
        which = np.flatnonzero(lens == n)
        out, _ = S.forward(p, np.stack([x[at[i]:at[i + 1]] for i in which]).astype(np.float64), 1, cout, S.bf16)
        for i, o in zip(which, out):
            ref[at[i]:at[i + 1]] = o
    assert np.linalg.norm(y - ref) <= 1e-3 * np.linalg.norm(ref)
    assert np.abs(y - ref).max() <= 3e-3 * np.abs(ref).max()


@pytest.mark.parametrize("nb,nseq,lq", [(1, 500, 5), (2, 40, 126)])
def test_gradients_over_many_tiles(nb, nseq, lq):
    import torch
    cin, cout = 3, 2
    net, p, rng = _net(cin, cout, nb, 22)
    x = rng.normal(size=(nseq, 4 * lq, cin)).astype(np.float32)
    t = rng.normal(size=(nseq, 4 * lq, cout)).astype(np.float32)
    m = (rng.uniform(size=(nseq, 4 * lq)) < 0.75).astype(np.float32)
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    loss = net.loss_grad(dev(x), dev(t), dev(m))
    g = S.unflatten(net.params(grads=True).astype(np.float64), cin, cout, WIDTH, nb)
    net.close()
    ref_loss, ref, _ = S.loss_and_grad(p, x.astype(np.float64), t.astype(np.float64), m.astype(np.float64), nb, cout,
                                       rnd=S.bf16)
    assert abs(loss - ref_loss) <= 1e-4 * ref_loss
    for k in ref:
        d = g[k] - ref[k]
        assert np.linalg.norm(d) <= 3e-3 * np.linalg.norm(ref[k]), k
        assert np.abs(d).max() <= 1.5e-2 * np.abs(ref[k]).max(), k
