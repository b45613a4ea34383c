"""The FP64 multi-shift solver's windowed update of the shifted vectors (8 iterations per pass, sums in 58-bit words)
where it could go wrong: windows cut short at every length, shifts whose coefficients are too small for words,
sites where the residual is still zero, lattices that do not fill a block.

Powers of two only move exponents: solutions must follow bit for bit.  Against the oracle: the certified residual
of a converged shift (1e-10, 5 % for the two sides' own rounding)."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import EPS, KAPPA, MU, require_gpu, torch

pytestmark = pytest.mark.gpu


def _solve(tm, g, b, sigma):
    bi = g.pack(torch.from_numpy(np.ascontiguousarray(b[None])).cuda())
    xs = [g.spinor() for _ in sigma]
    tm.mms_cg_solve(g.handle, bi, 1, sigma, xs, rho=1e-10)
    return [g.unpack(x)[0].cpu().numpy() for x in xs]


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 2, 2, 6), (4, 4, 4, 6)])
@pytest.mark.parametrize("source", ["gaussian", "point"])
def test_windowed_update(dims, source):
    tm = require_gpu()
    U = synth.random_su3_field(dims, 0.5, 21)
    g = tm.Gauge(U, dims, KAPPA, MU, EPS)
    act = oracle.action(dims, KAPPA, MU, EPS)
    b = synth.gaussian_rhs(dims, 8)[0]
    if source == "point":
        b = np.zeros_like(b)
        b[1, 0, 2, 1] = 1.0
    # bases from 1e-3 to 1e2 end after different numbers of iterations; 1e40's coefficients have no words
    for base in (1e-3, 0.03, 0.3, 1.0, 3.0, 10.0, 1e2):
        sigma = sorted([1e40, 2e2, 7 * base, base], reverse=True)
        x = _solve(tm, g, b, sigma)
        for s, v in zip(sigma, x):
            r = oracle.qhat2(act, U, v, s) - b
            assert np.linalg.norm(r) <= 1.05e-10 * np.linalg.norm(b), (base, s)
        for k in (-60, 47):
            for v, w in zip(x, _solve(tm, g, b * 2.0 ** k, sigma)):
                assert np.array_equal(w, v * 2.0 ** k)
    g.close()
