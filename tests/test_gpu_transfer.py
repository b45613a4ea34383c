"""Restriction and prolongation at the edges of their tiles: aggregates with and without whole groups of 4
sites along z, fewer sites than a chunk and ragged chunks, 1 to 32 vectors, 1 to 9 right-hand sides, and
vectors on an 8-byte boundary only.  Reference: numpy in complex128 with the handle's own P.  FP32 sums of
up to 1536 products: 2e-5 of the largest output, as in the multigrid parity tests."""
import numpy as np
import pytest

import synth
from gpu_common import EPS, KAPPA, MU, require_gpu, torch

pytestmark = pytest.mark.gpu

# dims, aggregate, vectors per chirality
CASES = [((4, 4, 4, 8), (4, 4, 4, 4), 24), ((4, 4, 4, 4), (1, 1, 2, 4), 9), ((4, 4, 4, 8), (2, 2, 2, 8), 32),
         ((6, 4, 6, 4), (3, 2, 3, 2), 5), ((2, 2, 2, 4), (1, 1, 1, 2), 1), ((6, 2, 4, 12), (2, 1, 2, 6), 17)]


def _sites(dims, bd):
    """(parity, half-index) of [block][local site], both lexicographic"""
    t, x, y, z = np.meshgrid(*[np.arange(d) for d in dims], indexing="ij")
    par = (t + x + y + z) & 1
    h = np.ravel_multi_index((t, x, y, z), dims) >> 1
    nb = [d // b for d, b in zip(dims, bd)]

    def blocks(a):
        a = a.reshape(nb[0], bd[0], nb[1], bd[1], nb[2], bd[2], nb[3], bd[3])
        return a.transpose(0, 2, 4, 6, 1, 3, 5, 7).reshape(int(np.prod(nb)), -1)
    return blocks(par), blocks(h)


@pytest.mark.parametrize("dims,bd,nv", CASES)
def test_restrict_and_prolong(dims, bd, nv):
    tm = require_gpu()
    V = int(np.prod(dims))
    par, h = _sites(dims, bd)
    nb, nsb = par.shape
    rng = np.random.default_rng(5)

    def gauss(*shape):
        return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)
    g = tm.Gauge(synth.random_su3_field(dims, 0.5, 3), dims, KAPPA, MU, EPS)
    mg = tm.tmnd_mg_create(g.handle, bd, nv, torch.from_numpy(gauss(nv, 2, 12, V // 2)).cuda())
    P = np.zeros((nb, 2, nv, nsb, 6), np.complex64)
    tm.tmnd_mg_export(mg, P_host=P)
    P = P.astype(np.complex128)
    for nrhs in (1, 2, 3, 5, 8, 9):
        fine, coarse = gauss(nrhs, 2, 24, V // 2), gauss(nrhs, nb, 2, 2, nv)
        # [rhs][block][site][24] from [rhs][parity][24][V/2]
        vb = np.moveaxis(fine, 2, 3)[:, par, h].astype(np.complex128)
        vb = vb.reshape(nrhs, nb, nsb, 2, 2, 6)                      # flavour, chirality, 6
        ref_c = np.einsum("bckse,rbsfce->rbfck", P.conj(), vb)
        ref_f = np.zeros((nrhs, 2, V // 2, 24), np.complex128)
        ref_f[:, par, h] = np.einsum("bckse,rbfck->rbsfce", P, coarse.astype(np.complex128)).reshape(nrhs, nb, nsb, 24)
        ref_f = np.moveaxis(ref_f, 3, 2)
        for shift in (0, 1):  # one complex64 off the 16-byte boundary
            buf = torch.zeros(fine.size + 2, dtype=torch.complex64, device="cuda")
            fv = buf[shift:shift + fine.size]
            fv.copy_(torch.from_numpy(fine.reshape(-1)))
            out = torch.full((coarse.size,), float("nan"), dtype=torch.complex64, device="cuda")
            tm.tmnd_mg_restrict(mg, out, fv, nrhs)
            got = out.cpu().numpy().reshape(ref_c.shape)
            assert np.abs(got - ref_c).max() <= 2e-5 * np.abs(ref_c).max(), (nrhs, shift)
            fv.fill_(float("nan"))
            tm.tmnd_mg_prolong(mg, fv, torch.from_numpy(coarse).cuda(), nrhs)
            got = fv.cpu().numpy().reshape(ref_f.shape)
            assert np.abs(got - ref_f).max() <= 2e-5 * np.abs(ref_f).max(), (nrhs, shift)
    tm.tmnd_mg_destroy(mg)
    g.close()
