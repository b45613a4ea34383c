"""The sloppy multi-shift solver's windowed update when a solve ends inside its first window: residual slots that it
never wrote may hold anything, NaN included, and must not reach the solutions."""
import numpy as np
import pytest

import synth
from gpu_common import EPS, KAPPA, MU, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 6, 2, 6), (4, 4, 4, 4)])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_unwritten_slots_do_not_matter(dims, nrhs):
    """With shifts of 1e8 and 1e6 |Qhat^2 x| is below 3e-6 |sigma x| and CG needs one or two iterations.  16-bit
    rounding moves x by a few 1e-5 of that: x = b / sigma to 1e-5, and equal whatever the workspace held."""
    tm = require_gpu()
    g = tm.Gauge(synth.random_su3_field(dims, 0.5, 33), dims, KAPPA, MU, EPS)
    b = synth.gaussian_rhs(dims, 34, nrhs=nrhs)
    bi = g.pack(torch.from_numpy(b).cuda(), nrhs=nrhs)
    sigma = [1e8, 1e6]
    f = g.convert(g.pack(torch.from_numpy(synth.gaussian_rhs(dims, 35, nrhs=24)).cuda(), nrhs=24), tm.TMND_F64,
                  tm.TMND_F32, nrhs=24)
    o = g.spinor(24, prec=tm.TMND_F32)
    xs = [g.spinor(nrhs) for _ in sigma]
    got = []
    for bad in (1.0, float("nan"), float("inf")):
        # the FP32 operator leaves its temporaries for 24 right-hand sides in the same workspace
        tm.tm_nd_apply(g.handle, o, f * bad, tm.OP_QHAT2 | tm.OP_F32, 0.25, nrhs=24)
        info = tm.mms_cg_solve(g.handle, bi, nrhs, sigma, xs, rho=1e-4, rho_inner=1e-4, prec=tm.TMND_S16, batch=nrhs)
        assert info["iters"] < 8
        got.append([g.unpack(x, nrhs=nrhs).cpu().numpy() for x in xs])
    for x in got:
        for v, w, s in zip(x, got[0], sigma):
            assert np.array_equal(v, w)
            assert np.linalg.norm(v * s - b) <= 1e-5 * np.linalg.norm(b)
    g.close()
