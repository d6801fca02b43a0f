"""FP32 tubes at the lengths where the points per lane of the FTCS pieces change. A piece
is 30 lanes of w = 5, 7, 9 or 13 points; two lines of pieces fit a block of n warps up to
15 n w cells, the first w that fits keeps the pieces in registers, and longer tubes take
them in passes. 128, 256 and 512 threads, 256 also in the form for two blocks per SM;
sub-step counts of a barrier's w, one more, and three barriers and one; the
backward-Euler solve at the same lengths (several separators per lane). Against the FP64
oracle with the 5e-5 of the other FP32 tubes: at most 4 steps x 40 sub-steps of four
roundings of 2^-24 in sequence make 4e-5."""
import functools

import numpy as np
import pytest

import oracle as O
import paper_2201_05280_gb300 as rpk
import rpk_inputs as I

pytestmark = pytest.mark.gpu

T0 = 0.2948964908710633
CS = np.sqrt(1.4 * T0)
SHORT = (19, 150, 151, 271, 599, 600, 601, 839, 841, 1000)  # two blocks per SM: up to 1000 cells
NX = {128: (209, 210, 211, 300, 301, 420, 421, 540, 541, 780, 781),
      256: (270, 600, 601, 840, 841, 1080, 1081, 1560, 1561, 1900),
      512: (389, 391, 1200, 1201, 1680, 1681, 2160, 2161, 3120, 3121, 4132)}


@functools.lru_cache(maxsize=None)
def _tube(nx, implicit, nsub):
    f, res = I.shock_tube(nx, T0, rho_r=1 / 1.2, p_r=0.7)
    f["R"] = f["R"] * (1.0 + 0.02 * np.sin(0.7 * np.arange(2 * nx) + nx))
    P = O.make_params(2.0, 0.6, 0.8, 0.3, 2.0, 1.0, nsub, 1, implicit)
    return f, res, O.State(P, nx, 1, 1, reservoirs=res).init_fields(f["rho"], f["u"], f["T"], f["R"]).step(4).fields()


@pytest.mark.parametrize("threads,ctas", [(128, 1), (256, 1), (256, 2), (512, 1)])
@pytest.mark.parametrize("nsub", [0, 5, 6, 7, 8, 9, 10, 13, 14, 16, 22, 28, 40])
def test_fp32_tubes(threads, ctas, nsub):
    """nsub 0: backward Euler."""
    relax = dict(delta=2.0, tau=0.6, tau1=0.8, b=0.3, k_r=2.0, nsub=max(nsub, 2))
    lengths = SHORT if ctas == 2 else NX[threads]
    parts = [_tube(nx, 0 if nsub else 1, max(nsub, 2)) for nx in lengths]
    tubes = [dict(nx=nx, nsteps=4, relax=relax, res=p[1]) for nx, p in zip(lengths, parts)]
    B = rpk.Batch(tubes, precision="f32", save_every=100).set_diffusion("ftcs" if nsub else "implicit")
    cat = {k: np.concatenate([p[0][k] for p in parts], axis=-1) for k in ("rho", "u", "T", "R")}
    got = B.init_fields(cat["rho"], cat["u"], cat["T"], cat["R"]).set_config(threads, ctas).run().read_moments()
    B.close()
    at = 0
    for nx, (_, _, ref) in zip(lengths, parts):
        for k in ("rho", "u", "T", "R", "Erot"):
            scale = max(np.abs(ref[k]).max(), CS if k == "u" else 0.0)
            assert np.abs(got[k][..., at:at + 2 * nx] - ref[k]).max() <= 5e-5 * scale, (nx, k)
        at += 2 * nx
