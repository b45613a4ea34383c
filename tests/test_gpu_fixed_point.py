"""The FP64 operator's fixed-point arithmetic where it could go wrong: lattices that do not fill a run of
16 sites or a block, fields far from 1, sites that are zero, point sources, NaN, and several right-hand
sides per launch.

Scaling by a power of two only moves the sites' exponents, so the results must follow bit for bit.
Against the oracle the tolerance is that of the operator tests (1e-13 of the largest component)."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import EPS, KAPPA, MU, require_gpu, torch

pytestmark = pytest.mark.gpu

# V/2 = 8 (half a run), 16, 24 (a run and a half), 864, and 3 runs with extents of 2
DIMS = [(2, 2, 2, 2), (2, 2, 2, 4), (2, 2, 2, 6), (6, 6, 6, 8), (4, 2, 2, 6)]


def _gauge(dims):
    tm = require_gpu()
    U = synth.random_su3_field(dims, 0.5, 77)
    return tm, U, tm.Gauge(U, dims, KAPPA, MU, EPS)


def _apply(tm, g, x, op, nrhs=1):
    bi = g.pack(torch.from_numpy(np.ascontiguousarray(x)).cuda(), nrhs=nrhs)
    out = g.spinor(nrhs)
    tm.tm_nd_apply(g.handle, out, bi, op, 0.25, nrhs=nrhs)
    return g.unpack(out, nrhs=nrhs).cpu().numpy()


@pytest.mark.parametrize("dims", DIMS)
def test_powers_of_two_scale_exactly(dims):
    tm, U, g = _gauge(dims)
    b = synth.gaussian_rhs(dims, 5)
    for op in (tm.OP_MHAT_DAG, tm.OP_QHAT2, tm.OP_QHAT):
        ref = _apply(tm, g, b, op)
        for k in (-930, -40, 3, 900):
            assert np.array_equal(_apply(tm, g, b * 2.0 ** k, op), ref * 2.0 ** k), (op, k)
    g.close()


@pytest.mark.parametrize("dims", DIMS)
def test_point_source_and_uneven_sites_match_oracle(dims):
    tm, U, g = _gauge(dims)
    act = oracle.action(dims, KAPPA, MU, EPS)
    b = synth.gaussian_rhs(dims, 6)[0]
    point = np.zeros_like(b)
    point[3, 1, 2, 0] = 1.0 - 2.0 ** -53          # all bits of the mantissa set
    uneven = b * (2.0 ** np.random.default_rng(3).integers(-45, 45, b.shape[0]))[:, None, None, None]
    uneven[1] = 0.0
    for x in (point, uneven, np.zeros_like(b)):
        ref = oracle.qhat2(act, U, x, 0.25)
        got = _apply(tm, g, x[None], tm.OP_QHAT2)[0]
        assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref))
    g.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_component_reaches_its_stencil_only(bad):
    dims = (6, 6, 6, 8)
    tm, U, g = _gauge(dims)
    act = oracle.action(dims, KAPPA, MU, EPS)
    b = synth.gaussian_rhs(dims, 8)
    b[0, 100] = 0.0
    clean = _apply(tm, g, b, tm.OP_MHAT)[0]
    probe = np.zeros_like(b[0])
    probe[100] = 1.0 + 0.5j
    reach = np.abs(oracle.schur(act, U, probe)).reshape(len(probe), -1).max(axis=1) > 0
    b[0, 100, 1, 2, 1] = bad
    got = _apply(tm, g, b, tm.OP_MHAT)[0]
    nan = np.isnan(got).reshape(len(probe), -1)
    assert np.array_equal(nan.all(axis=1), reach) and np.array_equal(nan.any(axis=1), reach)
    assert np.array_equal(got[~reach], clean[~reach])
    g.close()


@pytest.mark.parametrize("dims", [(2, 2, 2, 6), (6, 6, 6, 8), (16, 8, 16, 16)])
def test_right_hand_sides_in_one_launch(dims):
    tm, U, g = _gauge(dims)
    b = synth.gaussian_rhs(dims, 9, nrhs=7)
    for op in (tm.OP_MHAT, tm.OP_QHAT2, tm.OP_QHAT):
        got = _apply(tm, g, b, op, nrhs=7)
        for k in range(7):
            assert np.array_equal(got[k], _apply(tm, g, b[k:k + 1], op)[0])
    g.close()
