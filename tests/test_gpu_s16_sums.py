"""The sums |p|^2, |y|^2 and |r'|^2 of the 16-bit stencil, which set alpha and beta of the sloppy multi-shift
solver: a site's squares are added in FP32, the sites in FP64, for every launch variant, lattices that end inside
a tile, odd numbers of right-hand sides and right-hand sides that have stopped.

alpha_0 = |r|^2 / (|y|^2 + sigma |p|^2).  With sigma = 1e14, r = p = b and components that are integers times the
site's power of two (so that p is b exactly in 16 bits, and both add a site's squares in the same order),
alpha_0 sigma = 1 - |y|^2 / (sigma |p|^2), which is 1 to 2e-14 (|y|^2 < 2 |p|^2, tested), up to
the rounding of two FP64 sums of V/2 <= 432 positive terms, 432 2^-53 = 5e-14 each at most: bound 2e-13.  FP32 sums
over several sites miss it by a few 1e-9."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import EPS, KAPPA, MU, require_gpu, torch

pytestmark = pytest.mark.gpu

SIGMA = 1e14


def _gauge(dims):
    tm = require_gpu()
    U = synth.random_su3_field(dims, 0.5, 91)
    return tm, U, tm.Gauge(U, dims, KAPPA, MU, EPS)


def _integers(dims, nrhs, seed):
    """[nrhs][V/2][2][4][3]: per site three real components of the first flavour, integers up to 32767 (reached)
    times the site's power of two, the rest zero."""
    rng = np.random.default_rng(seed)
    vh = int(np.prod(dims)) // 2
    b = np.zeros((nrhs, vh, 2, 4, 3), dtype=np.complex128)
    n = rng.integers(1, 32768, (3, nrhs, vh)).astype(float)
    n[0] = 32767.0
    scale = 2.0 ** rng.integers(-6, 7, (nrhs, vh))
    for q, (s, c) in enumerate(((0, 0), (1, 2), (3, 1))):
        b[:, :, 0, s, c] = n[q] * scale
    return b


def _solve(tm, g, b, sigma, variant, rho, rho_inner, hist):
    n = len(b)
    bi = g.pack(torch.from_numpy(np.ascontiguousarray(b)).cuda(), nrhs=n)
    xs = [g.spinor(n) for _ in sigma]
    try:
        tm.tmnd_s16_force_shape(variant)
        info = tm.mms_cg_solve(g.handle, bi, n, sigma, xs, rho=rho, rho_inner=rho_inner, prec=tm.TMND_S16, batch=n, ab_hist=hist)
    finally:
        tm.tmnd_s16_force_shape(-1)
    return [g.unpack(x, nrhs=n).cpu().numpy() for x in xs], info


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 6, 6, 4), (2, 6, 2, 6)])
@pytest.mark.parametrize("nrhs", [1, 3, 5, 16])
def test_norms_are_fp64_sums_over_sites(dims, nrhs):
    tm, U, g = _gauge(dims)
    b = _integers(dims, nrhs, 17)
    y = oracle.schur(oracle.action(dims, KAPPA, MU, EPS), U, b[0])
    assert np.linalg.norm(y) ** 2 < 2.0 * np.linalg.norm(b[0]) ** 2
    if nrhs > 1:
        b[1] = 0.0  # stopped before the first iteration, in one pass with the first
    for v in range(tm.S16_SHAPES):
        hist = np.zeros(4)
        (x,), info = _solve(tm, g, b, [SIGMA], v, 0.5, 0.5, hist)
        assert info["iters"] == 1 and info["refine_iters"] == 0
        assert abs(hist[0] * SIGMA - 1.0) <= 2e-13, (v, hist[0] * SIGMA - 1.0)
        # the other right-hand sides' alpha_0 from their solutions, x = (float)alpha_0 b in FP32
        assert np.all(np.abs(x * SIGMA - b) <= 2.0 ** -22 * np.abs(b)), v
    g.close()


@pytest.mark.parametrize("dims", [(6, 6, 6, 4), (2, 6, 2, 6)])
@pytest.mark.parametrize("nrhs", [1, 3, 5])
def test_recursion_is_the_same_for_every_variant(dims, nrhs):
    """Vectors are the same bit for bit as long as alpha and beta round to the same floats, which sums that differ by
    V/2 2^-53 leave alone; then the histories agree to that times the few terms of alpha and beta, and the
    solutions of all right-hand sides (no defect correction at this tolerance) are equal."""
    tm, U, g = _gauge(dims)
    b = synth.gaussian_rhs(dims, 23, nrhs=nrhs)
    if nrhs > 1:
        b[1] = 0.0
    sigma = [1.0, 0.3, 0.1]
    ref = None
    for v in range(tm.S16_SHAPES):
        hist = np.zeros(64)
        x, info = _solve(tm, g, b, sigma, v, 2e-2, 1e-2, hist)
        assert info["refine_iters"] == 0 and 2 < info["iters"] < 32
        if ref is None:
            ref = hist, x, info["iters"]
            continue
        assert info["iters"] == ref[2], v
        assert np.allclose(hist, ref[0], rtol=1e-12, atol=0), (v, np.max(np.abs(hist - ref[0])))
        for p, q in zip(x, ref[1]):
            assert np.array_equal(p, q), v
    g.close()
