"""Rotational diffusion of the batched tubes at the sizes where its pieces
end, FP64 against the oracle tube by tube (rounding order differs: the 1e-12 of
the other FP64 tests). FTCS takes 5 points per lane of a warp in FP64 (pieces of
150 points, up to 5 sub-steps per barrier); the backward-Euler solve takes
blocks of 9 points and 32 lanes of separators per line, so 9 n and 288 n + 1
are the ends of a block, of a lane's share and of a line with one separator
more than lanes."""
import numpy as np
import pytest

import oracle as O
import paper_2201_05280_gb300 as rpk
import rpk_inputs as I

pytestmark = pytest.mark.gpu

T0 = 0.2948964908710633
NX = (2, 3, 9, 10, 11, 18, 19, 149, 150, 151, 287, 288, 289, 297, 298, 577, 1025, 2049)


@pytest.mark.parametrize("threads", [128, 512])
@pytest.mark.parametrize("diffusion,nsub", [("implicit", 1), ("ftcs", 1), ("ftcs", 4), ("ftcs", 5), ("ftcs", 13)])
def test_tube_diffusion(diffusion, nsub, threads):
    relax = dict(delta=2.0, tau=0.6, tau1=0.8, b=0.3, k_r=2.0, nsub=nsub + 1)
    tubes, parts, refs = [], [], []
    for i, nx in enumerate(NX):
        f, res = I.shock_tube(nx, T0, rho_r=1 / 1.2, p_r=0.7)
        f["R"] = f["R"] * (1.0 + 0.02 * np.sin(0.7 * np.arange(2 * nx) + i))
        tubes.append(dict(nx=nx, nsteps=4, relax=relax, res=res))
        parts.append(f)
        P = O.make_params(2.0, 0.6, 0.8, 0.3, 2.0, 1.0, nsub + 1, 1, 1 if diffusion == "implicit" else 0)
        refs.append(O.State(P, nx, 1, 1, reservoirs=res).init_fields(f["rho"], f["u"], f["T"], f["R"]).step(4).fields())
    B = rpk.Batch(tubes, precision="f64", save_every=100).set_diffusion(diffusion)
    cat = {k: np.concatenate([p[k] for p in parts], axis=-1) for k in ("rho", "u", "T", "R")}
    got = B.init_fields(cat["rho"], cat["u"], cat["T"], cat["R"]).set_config(threads).run().read_moments()
    B.close()
    at = 0
    for nx, ref in zip(NX, refs):
        for k in ("rho", "u", "T", "R", "Erot"):
            scale = max(np.abs(ref[k]).max(), np.sqrt(1.4 * T0) if k == "u" else 0.0)
            assert np.abs(got[k][..., at:at + 2 * nx] - ref[k]).max() <= 1e-12 * scale, (nx, k)
        at += 2 * nx
