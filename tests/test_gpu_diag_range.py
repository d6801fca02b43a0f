"""The diagnostics sum in FP64: totals far above FP32's largest value stay finite
and exact to the rounding of a point's own FP32 values. A uniform gas at rest with
rho = R keeps every h at R - 1, so M = N R, E = N (3 + delta)/2 R theta0 and H1 =
N (R ln R - R - (delta/2) R ln theta0). Two points per thread (nx even, both
rotational solvers) and one (nx odd). A point's value takes fewer than 64 FP32
roundings: 64 x 2^-24 < 4e-6 of the sum of magnitudes."""
import numpy as np
import pytest

import paper_2201_05280_gb300 as rpk

pytestmark = pytest.mark.gpu

T0 = 0.2948964908710633


@pytest.mark.parametrize("mode", ["conservative", "paper"])
@pytest.mark.parametrize("nx", [128, 127])
def test_totals_beyond_fp32(nx, mode):
    R, delta = 1e36, 2.0
    lat = rpk.Lattice(nx, 128, 128, precision="f32")
    lat.set_relax(delta=delta, tau=0.6, tau1=0.8, b=0.0, k_r=0.1, nsub=1).set_rot_mode(mode)
    n = lat.npts
    one = np.ones(n)
    d = lat.init_fields(R * one, np.zeros((3, n)), T0 * one, T0 * one).step(1).diagnostics()
    lat.close()
    want = {"M": n * R, "E": n * 0.5 * (3.0 + delta) * R * T0,
            "H1": n * (R * np.log(R) - R - 0.5 * delta * R * np.log(T0))}
    for k, v in want.items():
        assert abs(d[k] - v) <= 4e-6 * abs(v), (k, d[k], v)
