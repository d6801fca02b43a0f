"""Training batches whose output gradients would need more than 4 GiB at a slot per
layer keep two slots and take each block's weight gradients after its input gradient.
64 blocks, 133,120 coarse positions: the memory of the step stays within what the
activations, two slots or 4 GiB, inputs and outputs need, and the gradient is the mean of
those of eight parts that do have a slot per layer. Mask sums of the parts and the whole
differ by a power of two, so every operand rounds alike and only the order of FP32 sums
differs: at most 133,120 terms accumulated in any order, errors adding up as a random
walk, sqrt(133120) x 2^-24 = 2.2e-5 of a tensor's L2 norm at full cancellation-free
magnitude; 1e-4 leaves room for cancellation in the biases' sums."""
import numpy as np
import pytest

import paper_2201_05280_gb300 as rpk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [128, 16])
def test_large_batches(width):
    import torch
    cin, cout, nb, lq, parts, seqs = 3, 2, 64, 130, 8, 128
    if width == 16:  # the other widths' kernels: an eighth of the slots' size
        seqs = 1024
    rng = np.random.default_rng(1)
    net = rpk.Net(cin, cout, width, nb, seed=2)
    v = net.params()
    at = width * 4 * cin + width
    n = nb * 2 * (5 * width * width + width)
    v[at:at + n] *= 0.05  # 64 blocks of order-one branches would diverge
    net.set_params(v)
    gen = torch.Generator(device="cuda").manual_seed(3)
    shape = (parts * seqs, 4 * lq)
    x = torch.randn(shape + (cin,), generator=gen, device="cuda")
    t = torch.randn(shape + (cout,), generator=gen, device="cuda")
    m = torch.ones(shape, device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    net.loss_grad(x, t, m)
    used = free - torch.cuda.mem_get_info()[0]
    whole = net.params(grads=True).astype(np.float64)
    net.close()
    slot = 4 * width * lq * parts * seqs
    assert (2 * nb + 1) * slot > 4 << 30  # this batch is over the limit
    assert used <= (2 * nb + 1) * slot + max(2 * slot, 4 << 30) + (128 << 20), used / 2**30
    net = rpk.Net(cin, cout, width, nb, seed=2)
    net.set_params(v)
    total = np.zeros_like(whole)
    for k in range(parts):
        s = slice(k * seqs, (k + 1) * seqs)
        net.loss_grad(x[s], t[s], m[s])
        total += net.params(grads=True)
    net.close()
    total /= parts
    assert np.linalg.norm(whole) > 0
    assert np.linalg.norm(whole - total) <= 1e-4 * np.linalg.norm(total)
