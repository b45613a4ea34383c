"""What is measured: the work that a user of libtmnd has it do, through its public entry points.

A case is one of five kinds, after the calls that a program makes:

  apply    the operator (Mhat, its dagger, Qhat^2 + sigma) on vectors in the library's own layout, in
           FP64, FP32 or on 16-bit data: the step of every Krylov method written around the library
  solve    pack, the multi-shift solve of all shifts, unpack: one call of a force or heat-bath step
  hybrid   the same with the smallest shifts taken from Lagrange guesses instead of the recursion
  layers   the multigrid's layers once each: the fine operator, restriction, the coarse operator on the
           tensor cores and prolongation
  guess    the interpolated initial guess of a new shift from the solved ones

Lattices, shift sets, right-hand-side counts, aggregates and test-vector counts are those of the
repository's configurations and tests (4^4, 16^3x32, 24^3x48, 32^3x64; 10 shifts in 1e-4..1, 12 in
1e-5..2; 1, 2 and 8 right-hand sides; 4^4 aggregates, 24 vectors); ragged lattices stand between them.
The solves stop at 1e-11 of |b|, the tolerance of acceptance and heat-bath steps.
"""
import math

import numpy as np
import torch

import paper_1805_09584_gb300 as tm

KAPPA, MU, EPS = 0.16, 0.1, 0.11
ROUGHNESS = 0.5
RHO = 1e-11
S_ODD = 0.1          # case-C shift of the multigrid layers, sqrt(sigma) at sigma = 0.01
OPS = {"mhat": tm.OP_MHAT, "mhat_dag": tm.OP_MHAT_DAG, "qhat2": tm.OP_QHAT2}
PRECS = {"f64": (tm.TMND_F64, 0), "f32": (tm.TMND_F32, tm.OP_F32), "s16": (tm.TMND_S16, tm.OP_S16)}


# ------------------------------------------------------------------ the cases
def _case(kind, dims, **more):
    return {"kind": kind, "T": dims[0], "X": dims[1], "Y": dims[2], "Z": dims[3], **more}


def _dims(case):
    return case["T"], case["X"], case["Y"], case["Z"]


def _shifts(n):
    """The repository's shift sets, descending: n = 10 in 1e-4..1, else n in 1e-5..2."""
    lo, hi = (1e-4, 1.0) if n == 10 else (1e-5, 2.0)
    return np.exp(np.linspace(math.log(hi), math.log(lo), n))


def listed():
    return [
        # the smallest call: one operator application on the lattice of a unit test or a first try
        {"name": "qhat2_f64_4", **_case("apply", (4, 4, 4, 4), prec="f64", op="qhat2", nrhs=1)},
        # an ordinary double-precision application (the 16^3x32 configuration)
        {"name": "qhat2_f64_16", **_case("apply", (32, 16, 16, 16), prec="f64", op="qhat2", nrhs=1)},
        # a lattice that fits no tile, three right-hand sides, the daggered operator
        {"name": "mhat_dag_f64_ragged", **_case("apply", (10, 6, 14, 22), prec="f64", op="mhat_dag", nrhs=3)},
        # the largest lattice of the repository, one double-precision residual
        {"name": "qhat2_f64_32", **_case("apply", (64, 32, 32, 32), prec="f64", op="qhat2", nrhs=1)},
        # a single-precision preconditioner's operator (the 24^3x48 configuration)
        {"name": "qhat2_f32_24", **_case("apply", (48, 24, 24, 24), prec="f32", op="qhat2", nrhs=1)},
        # the sloppy operator on a batch, its result read back in single precision
        {"name": "qhat2_s16_24_r8", **_case("apply", (48, 24, 24, 24), prec="s16", op="qhat2", nrhs=8)},
        # a small solve, where launches and latencies count
        {"name": "solve_f64_8", **_case("solve", (16, 8, 8, 8), prec="f64", nshift=10, nrhs=1)},
        # the double-precision configuration
        {"name": "solve_f64_16", **_case("solve", (32, 16, 16, 16), prec="f64", nshift=12, nrhs=1)},
        # the mixed-precision configuration: 12 shifts, two right-hand sides
        {"name": "solve_mixed_24", **_case("solve", (48, 24, 24, 24), prec="s16", nshift=12, nrhs=2)},
        # the batched hybrid of the headline at the 16^3x32 volume: 8 shifts by recursion, 4 by guesses, 8 right-hand sides
        {"name": "hybrid_16_r8", **_case("hybrid", (32, 16, 16, 16), prec="s16", nshift=12, nrhs=8, n_mms=8)},
        # one pass through the multigrid's layers for 8 right-hand sides
        {"name": "layers_16_r8", **_case("layers", (32, 16, 16, 16), block=4, nvec=24, nrhs=8)},
        # the guess of the next shift from 8 solved ones, two right-hand sides
        {"name": "guess_24", **_case("guess", (48, 24, 24, 24), nodes=8, nrhs=2)},
    ]


def _draw_dims(rng, vmin, vmax, step=2):
    """Even extents (multiples of `step`) with a volume spread over the logarithm of vmin..vmax."""
    v = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
    while True:
        e = [math.exp(rng.uniform(-0.35, 0.35)) * v ** 0.25 for _ in range(4)]
        d = [max(step if step > 2 else 4, step * round(x / step)) for x in e]
        if vmin <= d[0] * d[1] * d[2] * d[3] <= vmax:
            return tuple(d)


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "solve", "solve", "hybrid", "layers", "guess"])
    if kind == "apply":
        prec = rng.choice(["f64", "f64", "f32", "s16"])
        nrhs = rng.choice([1, 1, 2, 3, 5, 8])
        return _case("apply", _draw_dims(rng, 256, 700000), prec=prec, op=rng.choice(["qhat2", "qhat2", "mhat", "mhat_dag"]), nrhs=nrhs)
    if kind == "solve":
        prec = rng.choice(["f64", "s16"])
        return _case("solve", _draw_dims(rng, 256, 140000), prec=prec, nshift=rng.choice([1, 5, 10, 12]), nrhs=rng.choice([1, 1, 2, 3]))
    if kind == "hybrid":
        return _case("hybrid", _draw_dims(rng, 4096, 140000), prec="s16", nshift=rng.choice([10, 12]), nrhs=rng.choice([1, 2, 4, 8]), n_mms=rng.choice([8, 9]))
    if kind == "layers":
        block = rng.choice([2, 4])
        dims = _draw_dims(rng, 512, 16384) if block == 2 else _draw_dims(rng, 4096, 140000, 4)
        return _case("layers", dims, block=block, nvec=rng.choice([8, 12]) if block == 2 else rng.choice([12, 16, 20, 24]), nrhs=rng.choice([1, 2, 3, 8]))
    return _case("guess", _draw_dims(rng, 4096, 700000), nodes=rng.choice([2, 3, 5, 8]), nrhs=rng.choice([1, 2, 3]))


# ------------------------------------------------------------------ inputs
def _links(dims, seed):
    """Seeded SU(3) links U ~ exp(i r H), H a Gaussian traceless hermitian matrix, [4,T,X,Y,Z,3,3] on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = 4 * math.prod(dims)
    a = torch.randn((8, n), generator=gen, device="cuda", dtype=torch.float64) * (0.5 * ROUGHNESS)
    h = torch.zeros((n, 3, 3), device="cuda", dtype=torch.complex128)
    for k, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
        h[:, i, j] = torch.complex(a[2 * k], -a[2 * k + 1])
        h[:, j, i] = torch.complex(a[2 * k], a[2 * k + 1])
    d8 = a[7] / math.sqrt(3.0)
    h[:, 0, 0], h[:, 1, 1], h[:, 2, 2] = a[6] + d8, d8 - a[6], -2 * d8
    # rows 0 and 1 of 1 + iH - H^2/2 - iH^3/6, then Gram-Schmidt and row 2 = conj(row 0 x row 1)
    rows = []
    for r in (0, 1):
        e = torch.zeros((n, 3), device="cuda", dtype=torch.complex128)
        e[:, r] = 1.0
        acc, p = e.clone(), e
        for m in (1, 2, 3):
            p = (1j / m) * sum(p[:, k:k + 1] * h[:, k, :] for k in range(3))
            acc += p
        rows.append(acc)
    del h, p, e, acc
    r0 = rows[0] / rows[0].abs().square().sum(-1, keepdim=True).sqrt()
    for _ in range(2):
        rows[1] = rows[1] - (r0.conj() * rows[1]).sum(-1, keepdim=True) * r0
        rows[1] = rows[1] / rows[1].abs().square().sum(-1, keepdim=True).sqrt()
    r1 = rows[1]
    r2 = torch.stack([(r0[:, 1] * r1[:, 2] - r0[:, 2] * r1[:, 1]).conj(), (r0[:, 2] * r1[:, 0] - r0[:, 0] * r1[:, 2]).conj(),
                      (r0[:, 0] * r1[:, 1] - r0[:, 1] * r1[:, 0]).conj()], dim=-1)
    return torch.stack([r0, r1, r2], dim=1).reshape(4, *dims, 3, 3)


def _gauss(shape, seed, dtype=torch.complex128):
    """Seeded complex Gaussian numbers (real and imaginary part of variance 1) on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    return torch.view_as_complex(torch.randn((*shape, 2), generator=gen, device="cuda", dtype=real))


def _rhs(case, seed):
    """Canonical right-hand sides [nrhs][V/2][2][4][3] on the odd sites."""
    return _gauss((case["nrhs"], math.prod(_dims(case)) // 2, 2, 4, 3), seed + 7919)


class _Multigrid:
    """Owns a multigrid handle; released before the gauge handle that it refers to."""

    def __init__(self, gauge, block, nvec, vectors):
        self.gauge = gauge
        self.handle = tm.tmnd_mg_create(gauge.handle, block, nvec, vectors)

    def __del__(self):
        tm.tmnd_mg_destroy(self.handle)


def prepare(case, seed):
    dims, kind = _dims(case), case["kind"]
    vh = math.prod(dims) // 2
    g = tm.Gauge(_links(dims, seed).cpu().numpy(), dims, KAPPA, MU, EPS)
    s = {"case": case, "g": g}
    if kind == "apply":
        n, prec = case["nrhs"], PRECS[case["prec"]][0]
        x = g.pack(_rhs(case, seed), n)
        s["x"] = x if prec == tm.TMND_F64 else g.convert(x, tm.TMND_F64, prec, n)
        s["y"] = g.spinor(n, prec=prec)
        if prec == tm.TMND_S16:  # the way from 16-bit data to single precision that the entry points have
            s["y64"], s["y32"] = g.spinor(n), g.spinor(n, prec=tm.TMND_F32)
    elif kind in ("solve", "hybrid"):
        n = case["nrhs"]
        s["sigma"] = _shifts(case["nshift"])
        s["b"] = _rhs(case, seed)
        s["bi"] = g.spinor(n)
        s["x"] = [g.spinor(n) for _ in s["sigma"]]
        s["out"] = [torch.empty_like(s["b"]) for _ in s["sigma"]]
    elif kind == "layers":
        n, nv = case["nrhs"], case["nvec"]
        s["mg"] = _Multigrid(g, (case["block"],) * 4, nv, _gauss((nv, 2, 12, vh), seed + 31, torch.complex64))
        s["x"] = _gauss((n, 2, 24, vh), seed + 7919, torch.complex64)
        s["y"], s["z"] = torch.empty_like(s["x"]), torch.empty_like(s["x"])
        nb = math.prod(dims) // case["block"] ** 4
        s["xc"] = torch.empty((n, nb, 2, 2 * nv), dtype=torch.complex64, device="cuda")
        s["yc"] = torch.empty_like(s["xc"])
    else:
        s["nodes"] = _shifts(12)[:case["nodes"]][::-1].copy()
        s["target"] = _shifts(12)[case["nodes"]]
        s["xs"] = [g.pack(_rhs(case, seed + k), case["nrhs"]) for k in range(case["nodes"])]
        s["out"] = g.spinor(case["nrhs"])
    return s


def run(s):
    case, g = s["case"], s["g"]
    kind, h = case["kind"], s["g"].handle
    if kind == "apply":
        n, flag = case["nrhs"], PRECS[case["prec"]][1]
        tm.tm_nd_apply(h, s["y"], s["x"], OPS[case["op"]] | flag, 0.01, n)
        if case["prec"] != "s16":
            return s["y"]
        tm.tmnd_spinor_convert(h, s["y64"], tm.TMND_F64, s["y"], tm.TMND_S16, n)
        tm.tmnd_spinor_convert(h, s["y32"], tm.TMND_F32, s["y64"], tm.TMND_F64, n)
        return s["y32"]
    if kind in ("solve", "hybrid"):
        n, prec = case["nrhs"], PRECS[case["prec"]][0]
        tm.tmnd_spinor_pack(h, s["bi"], s["b"], n)
        if kind == "solve":
            tm.mms_cg_solve(h, s["bi"], n, s["sigma"], s["x"], rho=RHO, prec=prec)
        else:
            tm.tmnd_hybrid_solve(h, None, s["bi"], n, s["sigma"], case["n_mms"], s["x"], rho=RHO, prec=prec, n_guess=0, guess=1)
        for x, out in zip(s["x"], s["out"]):
            tm.tmnd_spinor_unpack(h, out, x, n)
        return s["out"]
    if kind == "layers":
        n, mg = case["nrhs"], s["mg"].handle
        for k in range(n):
            tm.tmnd_dnd_full_apply(h, s["y"][k], s["x"][k], S_ODD)
        tm.tmnd_mg_restrict(mg, s["xc"], s["x"], n)
        tm.mg_coarse_apply(mg, s["yc"], s["xc"], n, S_ODD)
        tm.tmnd_mg_prolong(mg, s["z"], s["yc"], n)
        return s["y"], s["xc"], s["yc"], s["z"]
    tm.lagrange_guess(h, s["nodes"], s["xs"], s["target"], s["out"], case["nrhs"])
    return s["out"]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """Inputs (vectors, links, operators) read once and outputs written once, in the precision of the case; the
    hops at 1320 operations per site and flavour and 240 of the site term for both.  A solve is
    counted with the iterations that CG needs on the smallest shift (spectrum about 0.011..2.4)."""
    kind, v, n = case["kind"], math.prod(_dims(case)), case.get("nrhs", 1)
    vh = v // 2
    half = (2 * 1320 + 240) * vh  # one stencil launch for one right-hand side
    if kind == "apply":
        vec, link = {"f64": (384, 144), "f32": (192, 72), "s16": (100, 24)}[case["prec"]]
        out = 192 if case["prec"] == "s16" else vec
        return {"bytes": n * vh * (vec + out) + 4 * v * link, "flops": n * half * (4 if case["op"] == "qhat2" else 2)}
    if kind in ("solve", "hybrid"):
        s = float(_shifts(case["nshift"])[-1])
        iters = 0.5 * math.sqrt((2.4 + s) / (0.011 + s)) * math.log(2 / RHO)
        return {"bytes": n * vh * 384 * (1 + case["nshift"]) + 4 * v * 144, "flops": n * iters * 4 * half}
    if kind == "layers":
        nv, nb = case["nvec"], v // case["block"] ** 4
        fine, coarse, p = n * v * 192, n * nb * 4 * nv * 8, v * 12 * nv * 8
        return {"bytes": 3 * fine + 2 * coarse + 4 * v * 72 + p + nb * 10 * (2 * nv) ** 2 * 8,
                "flops": n * (2 * half + 2 * v * 24 * nv * 8 + nb * 20 * (2 * nv) ** 2 * 8)}
    return {"bytes": n * vh * 384 * (case["nodes"] + 1), "flops": n * vh * 96 * case["nodes"]}


# ------------------------------------------------------------------ the same in 64 bits, by plain torch
class _Exact:
    """The doublet operator on the full lattice, fields [..., 2, 4, 3, T, X, Y, Z] in complex128."""

    def __init__(self, dims, seed):
        self.dims, self.v = dims, math.prod(dims)
        self.u = _links(dims, seed).permute(0, 5, 6, 1, 2, 3, 4).contiguous()
        t, x, y, z = torch.meshgrid(*(torch.arange(d, device="cuda") for d in dims), indexing="ij")
        self.odd = ((t + x + y + z) & 1).to(torch.float64)
        flat = self.odd.reshape(-1)
        self.sites = (torch.nonzero(flat == 0)[:, 0], torch.nonzero(flat == 1)[:, 0])  # by parity, in order of lex >> 1
        self.kp, self.kpp = 2 * KAPPA * MU, 2 * KAPPA * EPS

    def full(self, half, parity):
        """[..., comp, V/2] on one parity to the full lattice, zero elsewhere."""
        out = torch.zeros((*half.shape[:-1], self.v), dtype=torch.complex128, device="cuda")
        out[..., self.sites[parity]] = half.to(torch.complex128)
        return out.reshape(*half.shape[:-2], 2, 4, 3, *self.dims)

    def half(self, field, parity):
        return field.reshape(*field.shape[:-7], 24, self.v)[..., self.sites[parity]]

    def hop(self, psi):
        """H psi: sum over mu of (1 - gamma_mu) U psi(x + mu) + (1 + gamma_mu) U^+ psi(x - mu)."""
        out = torch.zeros_like(psi)
        for mu in range(4):
            for sign in (-1, 1):  # forward, backward
                p = psi
                if sign < 0:
                    p = self.shift(psi, mu, -1)
                up, lo = p[..., 0:2, :, :, :, :, :], p[..., 2:4, :, :, :, :, :]
                chi = up + sign * self.b(lo, mu)
                w = torch.empty_like(chi)
                for i in range(3):
                    def link(j):
                        return self.u[mu, i, j] if sign < 0 else self.u[mu, j, i].conj().resolve_conj()
                    acc = link(0) * chi[..., 0, :, :, :, :]
                    for j in (1, 2):
                        acc = torch.addcmul(acc, link(j).expand_as(acc), chi[..., j, :, :, :, :])
                    w[..., i, :, :, :, :] = acc
                if sign > 0:
                    w = self.shift(w, mu, 1)
                out[..., 0:2, :, :, :, :, :] += w
                out[..., 2:4, :, :, :, :, :] += sign * self.b(w, mu, dagger=True)
        return out

    def shift(self, f, mu, by):
        f = torch.roll(f, by, dims=mu - 4)
        if mu == 0:  # antiperiodic in time
            f[..., self.dims[0] - 1 if by < 0 else 0, :, :, :] *= -1
        return f

    @staticmethod
    def b(v, mu, dagger=False):
        """B v or B^+ v of gamma_mu = [[0, B], [B^+, 0]]: B_0 = -1, B_k = -i sigma_k."""
        a, c = v[..., 0:1, :, :, :, :, :], v[..., 1:2, :, :, :, :, :]
        if mu == 0:
            return -v
        w = torch.cat((c, a) if mu == 1 else (-1j * c, 1j * a) if mu == 2 else (a, -c), dim=-6)
        return (1j if dagger else -1j) * w

    def site(self, psi, sign=1.0, inverse=False):
        """A psi or A^-1 psi, A = 1 + i sign kp gamma_5 tau_3 - kpp tau_1."""
        kp, kpp = sign * self.kp, self.kpp
        g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device="cuda").reshape(4, 1, 1, 1, 1, 1)
        t3 = torch.tensor([1.0, -1.0], dtype=torch.float64, device="cuda").reshape(2, 1, 1, 1, 1, 1, 1)
        other = psi.flip(-7)
        if not inverse:
            return psi + (1j * kp) * (t3 * g5) * psi - kpp * other
        return (psi - (1j * kp) * (t3 * g5) * psi + kpp * other) / (1 + kp * kp - kpp * kpp)

    def g5(self, psi):
        out = psi.clone()
        out[..., 2:4, :, :, :, :, :] *= -1
        return out

    def mhat(self, x, dagger=False):
        """Odd-site fields to odd-site fields."""
        if dagger:  # gamma_5 Mhat(-mu) gamma_5
            x = self.g5(x)
        sign = -1.0 if dagger else 1.0
        y = self.site(x, sign) - KAPPA ** 2 * self.hop(self.site(self.hop(x), sign, inverse=True))
        return self.g5(y) if dagger else y

    def qhat2(self, x, sigma):
        return self.mhat(self.mhat(x), dagger=True) + sigma * x

    def dnd(self, x, s):
        """The full operator with the case-C term i s gamma_5 tau_1 on odd sites."""
        return self.site(x) - KAPPA * self.hop(x) + (1j * s) * self.odd * self.g5(x.flip(-7))

    def solve(self, b, sigma):
        """x_i of (Qhat^2 + sigma_i) x_i = b for one field b, by the multi-shift recursion to rounding."""
        n = len(sigma)
        s0 = float(sigma[-1])
        x = [torch.zeros_like(b) for _ in sigma]
        ps = [b.clone() for _ in sigma]
        r, p = b.clone(), b.clone()
        z, zo = [1.0] * n, [1.0] * n
        live = [True] * n
        rr = bb = float(torch.linalg.vector_norm(b).item()) ** 2
        ao, bo = 1.0, 0.0
        for _ in range(2000):
            w = self.qhat2(p, s0)
            al = rr / float(torch.vdot(p.reshape(-1), w.reshape(-1)).real.item())
            r -= al * w
            rn = float(torch.linalg.vector_norm(r).item()) ** 2
            be = rn / rr
            for i in range(n):
                if not live[i]:
                    continue
                zn = z[i] * zo[i] * ao / (al * bo * (zo[i] - z[i]) + zo[i] * ao * (1 + al * (float(sigma[i]) - s0)))
                x[i].add_(ps[i], alpha=al * zn / z[i])
                ps[i].mul_(be * (zn / z[i]) ** 2).add_(r, alpha=zn)
                zo[i], z[i] = z[i], zn
                live[i] = zn * zn * rn > 1e-30 * bb
            p.mul_(be).add_(r)
            rr, ao, bo = rn, al, be
            if not live[-1]:
                break
        return x


def _blocks(f, dims, b):
    """[..., T, X, Y, Z] -> [..., block, site of the block], both lexicographic."""
    lead, k = f.shape[:-4], len(f.shape) - 4
    f = f.reshape(*lead, *(q for d in dims for q in (d // b, b)))
    f = f.permute(*range(k), *(k + 2 * i for i in range(4)), *(k + 2 * i + 1 for i in range(4)))
    return f.reshape(*lead, math.prod(dims) // b ** 4, b ** 4)


def _unblocks(f, dims, b):
    lead, k = f.shape[:-2], len(f.shape) - 2
    f = f.reshape(*lead, *(d // b for d in dims), b, b, b, b)
    f = f.permute(*range(k), *(q for i in range(4) for q in (k + i, k + 4 + i)))
    return f.reshape(*lead, *dims)


def exact(case, seed):
    dims, kind = _dims(case), case["kind"]
    e = _Exact(dims, seed)
    if kind == "apply":
        x = e.full(_rhs(case, seed).reshape(case["nrhs"], -1, 24).transpose(-1, -2), 1)
        y = []
        for k in range(case["nrhs"]):
            f = e.qhat2(x[k], 0.01) if case["op"] == "qhat2" else e.mhat(x[k], case["op"] == "mhat_dag")
            y.append(e.half(f, 1).reshape(-1))
        return torch.cat(y)
    if kind in ("solve", "hybrid"):
        if math.prod(dims) * case["nrhs"] > 600000:
            return None  # minutes of plain torch
        b = e.full(_rhs(case, seed).reshape(case["nrhs"], -1, 24).transpose(-1, -2), 1)
        cols = [[e.half(x, 1).transpose(-1, -2).reshape(-1, 2, 4, 3) for x in e.solve(b[k], _shifts(case["nshift"]))]
                for k in range(case["nrhs"])]
        return [torch.stack([c[i] for c in cols]) for i in range(case["nshift"])]
    if kind == "layers":
        nv, bl, vh = case["nvec"], case["block"], e.v // 2
        tv = _gauss((nv, 2, 12, vh), seed + 31, torch.complex64).to(torch.complex128)
        flat = torch.empty((nv, 12, e.v), dtype=torch.complex128, device="cuda")
        for q in (0, 1):
            flat[..., e.sites[q]] = tv[:, q]
        # [block][chirality][vector][6 * site], orthonormal in the given order
        v = _blocks(flat.reshape(nv, 2, 6, *dims), dims, bl).permute(3, 1, 0, 2, 4).reshape(-1, 2, nv, 6 * bl ** 4).clone()
        for k in range(nv):
            for _ in range(2):
                if k:
                    c = (v[:, :, :k].conj() * v[:, :, k:k + 1]).sum(-1, keepdim=True)
                    v[:, :, k] -= (c * v[:, :, :k]).sum(2)
            v[:, :, k] /= v[:, :, k].abs().square().sum(-1, keepdim=True).sqrt()

        def restrict(f):  # [2, 4, 3, dims] -> [block, 2, 2 nv]
            a = _blocks(f.reshape(2, 2, 6, *dims), dims, bl).permute(3, 0, 1, 2, 4).reshape(-1, 2, 2, 6 * bl ** 4)
            return torch.einsum("bckx,bfcx->bfck", v.conj(), a).reshape(a.shape[0], 2, 2 * nv)

        def prolong(c):
            a = torch.einsum("bckx,bfck->bfcx", v, c.reshape(-1, 2, 2, nv))
            return _unblocks(a.reshape(-1, 2, 2, 6, bl ** 4).permute(1, 2, 3, 0, 4), dims, bl).reshape(2, 4, 3, *dims)

        x = _gauss((case["nrhs"], 2, 24, vh), seed + 7919, torch.complex64)
        ys, xcs, ycs, zs = [], [], [], []

        def mg(f):
            return torch.stack([e.half(f, 0), e.half(f, 1)])
        for k in range(case["nrhs"]):
            f = e.full(x[k, 0], 0) + e.full(x[k, 1], 1)
            c = restrict(f)
            d = restrict(e.dnd(prolong(c), S_ODD))
            ys.append(mg(e.dnd(f, S_ODD)))
            xcs.append(c)
            ycs.append(d)
            zs.append(mg(prolong(d)))
        return torch.stack(ys), torch.stack(xcs), torch.stack(ycs), torch.stack(zs)
    nodes, t = _shifts(12)[:case["nodes"]][::-1], float(_shifts(12)[case["nodes"]])
    out = 0
    for k, m in enumerate(nodes):
        w = math.prod((t - float(o)) / (float(m) - float(o)) for j, o in enumerate(nodes) if j != k)
        out = out + w * _rhs(case, seed + k).reshape(case["nrhs"], -1, 24).transpose(-1, -2)
    return out.reshape(-1)
