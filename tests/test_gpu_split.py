"""FP64 lattices of at most two warps of points per SM (152) collide with four warps per
32 points. Against the same state repeated along x until a thread takes a point again:
sizes below, at and above a warp of points and the line between the two, in both
rotational solvers. FP64 rounding in another order: the parity bound of the other FP64
tests, 1e-12."""
import numpy as np
import pytest

import paper_2201_05280_gb300 as rpk
import rpk_inputs as I

pytestmark = pytest.mark.gpu

T0 = 0.2948964908710633
CS = np.sqrt(1.4 * T0)


def _run(f, shape, mode):
    lat = rpk.Lattice(*shape, precision="f64").set_relax(delta=2.0, tau=0.6, tau1=0.8, b=0.3, k_r=0.9, nsub=2)
    lat.set_rot_mode(mode)
    out = lat.init_fields(f["rho"], f["u"], f["T"], f["R"]).step(5).read_moments()
    lat.close()
    return out


@pytest.mark.parametrize("mode", ["conservative", "paper"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (31, 1, 1), (8, 2, 2), (33, 1, 1), (4864, 1, 1), (4865, 1, 1), (5, 4, 3),
                                   (12, 13, 14)])
def test_four_warps_a_point_group(shape, mode):
    nx, ny, nz = shape
    f = I.random_smooth(nx, ny, nz, T0, seed=17)
    reps = -(-10000 // (nx * ny * nz))
    got = _run(f, shape, mode)
    big = _run(I.tile(f, nx, ny, nz, (reps, 1, 1)), (reps * nx, ny, nz), mode)
    for k in got:
        a = np.asarray(got[k]).reshape(-1, 2, nz, ny, nx)
        b = np.asarray(big[k]).reshape(-1, 2, nz, ny, reps, nx)
        scale = max(np.abs(a).max(), CS if k == "u" else 0.0)
        assert np.abs(b - a[:, :, :, :, None, :]).max() <= 1e-12 * scale, k
