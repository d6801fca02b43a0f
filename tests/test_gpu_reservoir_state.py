"""A tube at rest with its reservoirs: the reservoirs' populations are those that the same
state gives a point, bit for bit. With relaxation times of 1e30 the collision leaves
every stored population as it is, so after one step each point pulls initial populations
from the tube or from a reservoir, and the density and velocity of all points are equal
bits."""
import numpy as np
import pytest

import paper_2201_05280_gb300 as rpk

pytestmark = pytest.mark.gpu

T0 = 0.2948964908710633
RELAX = dict(delta=2.0, tau=1e30, tau1=1e30, b=0.0, k_r=0.0, nsub=1)


@pytest.mark.parametrize("kind,precision", [("batch", "f32"), ("batch", "f64"), ("lattice", "f32"), ("lattice", "f64")])
def test_uniform_tube(kind, precision):
    rng = np.random.default_rng(5)
    nx = 9
    for _ in range(8):
        s = [rng.uniform(0.5, 2.0), *rng.uniform(-0.1, 0.1, 3), T0 * rng.uniform(0.8, 1.2), T0 * rng.uniform(0.8, 1.2)]
        one = np.ones(2 * nx)
        f = s[0] * one, np.stack([u * one for u in s[1:4]]), s[4] * one, s[5] * one
        if kind == "batch":
            b = rpk.Batch([dict(nx=nx, nsteps=1, relax=RELAX, res=s + s)], precision=precision, save_every=100)
            got = b.init_fields(*f).run().read_moments()
            b.close()
        else:
            lat = rpk.Lattice(nx, 1, 1, precision=precision, bc_x="reservoir").set_relax(**RELAX).set_reservoirs(s + s)
            got = lat.init_fields(*f).step(1).read_moments()
            lat.close()
        # a point 2 cells and more from the ends pulls from the tube alone
        for sub in (slice(0, nx), slice(nx, 2 * nx)):
            assert np.array_equal(got["rho"][sub], np.full(nx, got["rho"][sub][4])), s
            assert np.array_equal(got["u"][:, sub], np.repeat(got["u"][:, sub][:, 4:5], nx, 1)), s
