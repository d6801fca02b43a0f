"""The kernels of a step may start while the one before still runs (programmatic
dependent launch). Event records between the launches keep them apart: a run with
kernel timing on and runs without give the same bits, on lattices small enough for
blocks of several launches to share an SM."""
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
    lat.timing(apart)
    out = lat.step(40).read_moments()
    lat.close()
    return out


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("precision,mode", [("f32", "conservative"), ("f32", "paper"), ("f16dev", "conservative"),
                                            ("f64", "conservative")])
@pytest.mark.parametrize("shape,nsub", [((42, 4, 2), 2), ((21, 4, 2), 3), ((16, 16, 16), 1), ((33, 9, 5), 12),
                                        ((300, 1, 1), 20), ((64, 64, 48), 2)])
def test_overlapping_launches(shape, nsub, precision, mode, walls):
    if walls and shape[1] < 2:
        pytest.skip("walls need ny >= 2")
    f = I.random_smooth(*shape, T0, seed=11)
    want = _run(shape, precision, mode, walls, nsub, f, True)
    for _ in range(6):
        got = _run(shape, precision, mode, walls, nsub, f, False)
        for k in want:
            assert np.array_equal(got[k], want[k]), k
