"""The FP64 operator's contract per output site: results are as accurate as FP64 arithmetic relative to the largest
component of the sites they are made of, wherever else the field is large.

Sites are scaled by 2^-45 .. 2^44, some are zero.  Tolerance: that of the operator tests, 1e-13, times the largest
input component among the sites within the operator's reach (the site itself and two hops for Mhat and its dagger,
four for Qhat^2 + sigma); the rows of these operators at kappa = 0.16 have absolute sums below 8."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import EPS, KAPPA, MU, require_gpu, torch

pytestmark = pytest.mark.gpu


def _reach(m, dims, hops):
    """m: a value per odd site, in the order of the vectors; the largest value within an even number of hops."""
    odd = np.indices(dims).sum(axis=0) % 2 == 1
    f = np.zeros(dims)
    f[odd] = m
    for _ in range(hops):
        f = np.max([f] + [np.roll(f, d, axis=a) for a in range(4) for d in (1, -1)], axis=0)
    return f[odd]


@pytest.mark.parametrize("dims", [(6, 6, 6, 8), (4, 2, 2, 6), (12, 4, 4, 6)])
def test_error_is_small_at_every_site(dims):
    tm = require_gpu()
    U = synth.random_su3_field(dims, 0.5, 78)
    act = oracle.action(dims, KAPPA, MU, EPS)
    g = tm.Gauge(U, dims, KAPPA, MU, EPS)
    b = synth.gaussian_rhs(dims, 16)[0]
    rng = np.random.default_rng(4)
    b *= (2.0 ** rng.integers(-45, 45, b.shape[0]))[:, None, None, None]
    b[rng.integers(0, len(b), 3)] = 0.0
    bi = g.pack(torch.from_numpy(b[None].copy()).cuda())
    largest = np.abs(b).reshape(len(b), -1).max(axis=1)
    for op, ref, hops in ((tm.OP_MHAT, oracle.schur(act, U, b), 2),
                          (tm.OP_QHAT2, oracle.qhat2(act, U, b, 0.25), 4)):
        out = g.spinor()
        tm.tm_nd_apply(g.handle, out, bi, op, 0.25)
        err = np.abs(g.unpack(out).cpu().numpy()[0] - ref).reshape(len(b), -1).max(axis=1)
        bound = 1e-13 * _reach(largest, dims, hops)
        assert np.all(err <= bound), (op, np.max(err / bound))
    g.close()
