"""Quasi-1-D lattices take the rotational transport in tiles of one sublattice
line (MacCormack and up to 16 FTCS sub-steps in one launch, halo recomputed).
Sizes at its edges against the FP64 oracle: lines shorter than the halo (the
periodic wrap goes round more than once), one tile, tile +- 1, and sub-step
counts below, at and above one launch's 16. FP64 differs from the oracle in
rounding order only: the parity bound of the other FP64 tests, 1e-12."""
import numpy as np
import pytest

import oracle as O
import paper_2201_05280_gb300 as rpk
import rpk_inputs as I

pytestmark = pytest.mark.gpu

T0 = 0.2948964908710633


@pytest.mark.parametrize("nsub", [1, 2, 16, 17, 40])
@pytest.mark.parametrize("nx,bcx", [(1, 0), (3, 0), (2, 1), (5, 1), (30, 0), (31, 1), (94, 0), (95, 1), (2500, 1),
                                    (6001, 0)])
def test_line_transport(nx, bcx, nsub):
    relax = dict(delta=2.0, tau=0.6, tau1=0.8, b=0.3, k_r=0.9, nsub=nsub)
    if bcx:
        f, res = I.shock_tube(nx, T0, rho_r=1 / 1.1, p_r=0.85)
        f["R"] = f["R"] * (1.0 + 0.01 * np.cos(np.arange(f["R"].size)))
    else:
        f, res = I.random_smooth(nx, 1, 1, T0), None
    lat = rpk.Lattice(nx, 1, 1, precision="f64", bc_x="reservoir" if bcx else "periodic").set_relax(**relax)
    if bcx:
        lat.set_reservoirs(res)
    got = lat.init_fields(f["rho"], f["u"], f["T"], f["R"]).step(6).read_moments()
    lat.close()
    P = O.make_params(2.0, 0.6, 0.8, 0.3, 0.9, 1.0, nsub, bcx)
    ref = O.State(P, nx, 1, 1, reservoirs=res).init_fields(f["rho"], f["u"], f["T"], f["R"]).step(6).fields()
    for k in ("rho", "u", "T", "R", "Erot"):
        scale = max(np.abs(ref[k]).max(), np.sqrt(1.4 * T0) if k == "u" else 0.0)
        assert np.abs(got[k] - ref[k]).max() <= 1e-12 * scale, k
