"""Kernels that may start while the one before still runs, against the same kernels one after
the other: equal bits. Lattices with ordinary launches throughout (rpk_timing 2) and with
overlapping ones, at sizes of both transport forms; the network's residual blocks for a
few sequences, whose blocks of threads leave SMs for the next launch's, and for so many
that every SM is taken until a launch ends."""
import numpy as np
import pytest

import paper_2201_05280_gb300 as rpk
import rpk_inputs as I

pytestmark = pytest.mark.gpu

T0 = 0.2948964908710633
WALLS = ([0.03, 0.0, -0.02, T0 * 1.02], [-0.04, 0.0, 0.01, T0 * 0.97])


def _run(shape, precision, mode, walls, nsub, f, apart):
    lat = rpk.Lattice(*shape, precision=precision)
    lat.set_relax(delta=2.0, tau=0.6, tau1=0.8, b=0.3, k_r=0.9, nsub=nsub)
    lat.set_rot_mode(mode)
    if walls:
        lat.set_walls(*WALLS)
    lat.init_fields(f["rho"], f["u"], f["T"], f["R"])
    if apart:
        rpk._check(rpk.load_library().rpk_timing(lat._h, 2))
    out = lat.step(30).read_moments()
    lat.close()
    return out


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("precision,mode", [("f32", "conservative"), ("f32", "paper"), ("bf16dev", "conservative"),
                                            ("f64", "conservative")])
@pytest.mark.parametrize("shape,nsub", [((42, 4, 2), 3), ((21, 5, 3), 2), ((300, 1, 1), 20), ((64, 64, 48), 2)])
def test_lattice_launches(shape, nsub, precision, mode, walls):
    if walls and shape[1] < 2:
        pytest.skip("walls need ny >= 2")
    f = I.random_smooth(*shape, T0, seed=13)
    want = _run(shape, precision, mode, walls, nsub, f, True)
    for _ in range(4):
        got = _run(shape, precision, mode, walls, nsub, f, False)
        for k in want:
            assert np.array_equal(got[k], want[k]), k


def test_network_blocks():
    import torch
    net = rpk.Net(3, 2, 128, 6, seed=4)
    x = torch.randn((1000, 4 * 130, 3), generator=torch.Generator(device="cuda").manual_seed(7), device="cuda")
    want = net.forward(x)
    for n in (1, 3, 40, 75, 120):
        for first in (0, 200, 777):
            assert torch.equal(net.forward(x[first:first + n].contiguous()), want[first:first + n]), (n, first)
    net.close()
