"""Small FP32 lattices take the rotational transport in 3-D tiles with a recomputed
halo, several passes a launch. Their sizes at the edges (axes shorter than the halo,
of one point, tiles +- 1, more sub-steps than one launch takes; every boundary)
against the FP64 lattice, which takes a launch per pass. Each of the 4 steps rounds
41 populations' deviations (<= 0.1, 2^-24 relative) and their sums: 4 x 41 x 0.1 x
6e-8 = 1e-6; a sub-step adds two roundings of e (<= 2^-24 of 0.3), 4 x 20 x 2 x 2e-8 =
3e-6 at most. A layer missing from a halo shows as about 1e-3."""
import numpy as np
import pytest

import paper_2201_05280_gb300 as rpk
import rpk_inputs as I

pytestmark = pytest.mark.gpu

T0 = 0.2948964908710633
CS = np.sqrt(1.4 * T0)
WALLS = ([0.03, 0.0, -0.02, T0 * 1.02], [-0.04, 0.0, 0.01, T0 * 0.97])
XWALLS = ([0.0, 0.02, -0.01, T0 * 1.02], [0.0, -0.03, 0.02, T0 * 0.98])
KEYS = ("rho", "u", "T", "R", "Erot")


def _run(precision, nx, ny, nz, bc, nsub, f, res):
    lat = rpk.Lattice(nx, ny, nz, precision=precision, bc_x="reservoir" if bc == "ends" else "periodic")
    lat.set_relax(delta=2.0, tau=0.6, tau1=0.8, b=0.3, k_r=0.9, nsub=nsub)
    if bc == "ends":
        lat.set_reservoirs(res)
    if "y" in bc:
        lat.set_walls(*WALLS)
    if "x" in bc:
        lat.set_x_walls(*XWALLS)
    lat.timing()
    out = lat.init_fields(f["rho"], f["u"], f["T"], f["R"]).step(4).read_moments()
    launches = lat.timing_read()["transport"][1]
    lat.close()
    return out, launches


@pytest.mark.parametrize("nsub", [1, 3, 8, 20])
@pytest.mark.parametrize("nx,ny,nz,bc", [
    (1, 2, 3, ""), (2, 1, 1, "x"), (3, 5, 2, ""), (17, 9, 4, ""), (32, 32, 32, ""), (33, 31, 29, ""), (200, 7, 1, ""),
    (4, 2, 1, "y"), (23, 40, 3, "y"), (61, 33, 8, "y"), (2, 6, 5, "x"), (40, 11, 6, "x"), (2, 2, 2, "xy"),
    (37, 30, 4, "xy"), (2, 3, 1, "ends"), (45, 12, 7, "ends")])
def test_tiles_against_fp64(nx, ny, nz, bc, nsub):
    f, res = I.random_smooth(nx, ny, nz, T0, seed=5), None
    rng = np.random.default_rng(nx + ny)
    f["R"] = f["R"] * (1.0 + 0.02 * rng.uniform(-1, 1, f["R"].shape))
    if bc == "ends":
        res = [1.01, 0.01, 0.0, 0.0, T0 * 1.01, T0 * 0.99, 0.99, -0.01, 0.0, 0.0, T0 * 0.99, T0 * 1.01]
    got, launches = _run("f32", nx, ny, nz, bc, nsub, f, res)
    ref, passes = _run("f64", nx, ny, nz, bc, nsub, f, res)
    assert passes == 4 * (2 + nsub)
    assert launches < passes or nx * ny * nz > 20000
    for k in KEYS:
        scale = max(np.abs(ref[k]).max(), CS if k == "u" else 0.0)
        assert np.abs(got[k] - ref[k]).max() <= 4e-6 * scale, k
