"""The work that users of this engine have it do, as measurable cases.

Every case goes through the public entry points of ``paper_1909_03948_gb300`` (``Problem``,
``Batch``, ``UNet``).  The problems are the repository's own: the log-coefficient Poisson
inverse problem on the unit square or cube with a bilaplacian prior and pointwise
observations, at the sizes of its workloads (small2d 32^2, medium2d 256^2, cube3d 64^3, the
uneven 2D batch) and at other sizes of the same ranges.  The log-coefficient m is a prior
draw (its expansion in cosines, truncated), the observation points are uniform in
[0.05, 0.95]^d, the noise level is 1 % of the largest state.  Solves run to the tolerances at
which the repository's tests compare results (1e-10 in 2D, 1e-11 in 3D, 1e-12 for samples):
there two runs that round differently agree to about ten digits.

``exact`` evaluates the same maps in 64 bits with plain torch: the finite-element operators
as sums over the mesh's simplices, and every linear solve by conjugate gradients to
rounding level.
"""
from __future__ import annotations

import math
import os

# one hardware work queue per stream for the uneven batch; read when CUDA starts
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

import numpy as np  # noqa: E402
import torch  # noqa: E402

from paper_1909_03948_gb300 import Batch, Problem, UNet  # noqa: E402
from paper_1909_03948_gb300.warmstart import he_init  # noqa: E402

DEV = "cuda"
MAX_VALUES = 65 ** 3 * 120  # the largest listed block: no drawn case has a larger one


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: one Hessian column with the prior term, as the CG of a Newton step
        # on the 32^2 workload applies it
        {"name": "column_small2d", "kind": "action", "rtol": 1e-10, "dim": 2, "N": 32, "nobs": 50, "gamma": 0.1, "delta": 0.5,
         "columns": 1, "prior": True, "full": False, "tiles": False},
        # the same on the 256^2 workload: every CG iteration of Newton's method is one of these
        {"name": "column_medium2d", "kind": "action", "rtol": 1e-10, "dim": 2, "N": 256, "nobs": 400, "gamma": 0.1, "delta": 0.5,
         "columns": 1, "prior": True, "full": False, "tiles": False},
        # one pass of the randomized eigensolver on 256^2: k + p = 60 random directions
        {"name": "block_medium2d", "kind": "action", "rtol": 1e-10, "dim": 2, "N": 256, "nobs": 400, "gamma": 0.1, "delta": 0.5,
         "columns": 60, "prior": False, "full": False, "tiles": False},
        # the largest: one pass of the eigensolver on 64^3, k + p = 120, with the settings the
        # autotuner picks there
        {"name": "block_cube3d", "kind": "action", "rtol": 1e-11, "dim": 3, "N": 64, "nobs": 1000, "gamma": 0.05, "delta": 0.5,
         "columns": 120, "prior": False, "full": False, "tiles": True},
        # full-Newton directions on a 3D grid that is no multiple of a tile, in a ragged block
        {"name": "full_ragged3d", "kind": "action", "rtol": 1e-11, "dim": 3, "N": 48, "nobs": 300, "gamma": 0.05, "delta": 0.5,
         "columns": 7, "prior": False, "full": True, "tiles": False},
        # between two Newton steps: the cost at a trial point, then the gradient at the next one
        {"name": "gradient_medium2d", "kind": "gradient", "rtol": 1e-10, "dim": 2, "N": 256, "nobs": 400, "gamma": 0.1,
         "delta": 0.5},
        # the eigensolver's inner product: R on a block of 120 on 64^3
        {"name": "precision_cube3d", "kind": "precision", "rtol": 1e-11, "dim": 3, "N": 64, "gamma": 0.05, "delta": 0.5,
         "columns": 120},
        # Laplace sampling on 64^3 with 100 eigenpairs, normals drawn on the device
        {"name": "samples_cube3d", "kind": "samples", "rtol": 1e-12, "dim": 3, "N": 64, "gamma": 0.05, "delta": 0.5, "k": 100,
         "nsamples": 64},
        # the prior's and the posterior's pointwise variance on 256^2 by the randomized method
        {"name": "variance_medium2d", "kind": "variance", "rtol": 1e-10, "dim": 2, "N": 256, "gamma": 0.1, "delta": 0.5, "r": 60,
         "k": 50},
        # the uneven batch: independent 2D problems, blocks of k + p = 40
        {"name": "batch_uneven2d", "kind": "batch", "rtol": 1e-10, "sizes": "64,64,96,96,128,160,192,256,320,384,448,512",
         "columns": 40},
        # the warm start's guesses for a block of 60 on 256^2 (a 264^2 padded grid)
        {"name": "unet_forward_264", "kind": "unet_forward", "H": 264, "W": 264, "batch": 60},
        # one training batch of the warm start on 64^2 problems (a 72^2 padded grid)
        {"name": "unet_gradient_72", "kind": "unet_gradient", "H": 72, "W": 72, "batch": 16},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _cells(rng, dim, lo, hi):
    """Cells per axis the multigrid takes: a small factor times a power of two."""
    fac = range(9, 17) if dim == 2 else (3, 4, 5)
    ok = sorted({f << k for f in fac for k in range(8) if lo <= f << k <= hi})
    return min(ok, key=lambda n: abs(math.log(n / math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["action", "action", "action", "action", "gradient", "precision", "samples", "variance",
                       "batch", "unet_forward", "unet_gradient"])
    if kind == "batch":
        sizes = [_cells(rng, 2, 48, 512) for _ in range(rng.randint(3, 14))]
        cols = min(_log_int(rng, 1, 48), MAX_VALUES // sum((N + 1) ** 2 for N in sizes))
        return {"kind": kind, "rtol": 1e-10, "sizes": ",".join(map(str, sizes)), "columns": cols}
    if kind == "unet_forward":
        return {"kind": kind, "H": 8 * rng.randint(3, 33), "W": 8 * rng.randint(3, 33), "batch": _log_int(rng, 1, 60)}
    if kind == "unet_gradient":
        return {"kind": kind, "H": 8 * rng.randint(3, 17), "W": 8 * rng.randint(3, 17), "batch": _log_int(rng, 1, 32)}
    dim = rng.choice([2, 2, 3])
    N = _cells(rng, dim, 24, 512) if dim == 2 else _cells(rng, dim, 12, 64)
    n = (N + 1) ** dim
    rtol = 1e-12 if kind == "samples" else 1e-10 if dim == 2 else 1e-11
    base = {"kind": kind, "rtol": rtol, "dim": dim, "N": N, "gamma": round(rng.uniform(0.05, 0.2), 3),
            "delta": round(rng.uniform(0.3, 1.0), 3)}
    cols = max(1, min(_log_int(rng, 1, 120), MAX_VALUES // n))
    if kind == "action":
        full, prior = rng.random() < 0.2, rng.random() < 0.4
        cols = max(1, min(cols, MAX_VALUES // (2 * n)))
        base |= {"nobs": _log_int(rng, 20, 1000), "columns": cols, "prior": prior, "full": full,
                 "tiles": dim == 3 and N % 32 == 0 and rng.random() < 0.5}
    elif kind == "gradient":
        base |= {"nobs": _log_int(rng, 20, 1000)}
    elif kind == "precision":
        base |= {"columns": cols}
    elif kind == "samples":
        base |= {"k": rng.randint(1, 100), "nsamples": max(1, min(64, cols))}
    else:
        base |= {"r": min(n, max(8, min(cols, 100, MAX_VALUES // (4 * n)))), "k": rng.randint(1, 60)}
    return base


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cpu").manual_seed(int(seed))


def _cosines(np_, modes):
    i = torch.arange(np_, dtype=torch.float64)
    c = torch.cos(math.pi * i[:, None] * torch.arange(modes, dtype=torch.float64)[None, :] / (np_ - 1))
    return c / c.square().mean(0).sqrt()


def _spectrum(dim, modes, gamma, delta):
    k2 = torch.arange(modes, dtype=torch.float64).square()
    lam = k2[:, None] + k2[None, :] if dim == 2 else k2[:, None, None] + k2[None, :, None] + k2[None, None, :]
    return gamma * math.pi ** 2 * lam + delta


def _prior_fields(dim, np_, gamma, delta, s, g):
    """(s, n) draws of the prior N(0, A^-2): its cosine expansion up to 24 (12) modes per axis."""
    modes = min(np_, 24 if dim == 2 else 12)
    c = _cosines(np_, modes).to(DEV)
    xi = torch.randn((s,) + (modes,) * dim, generator=g, dtype=torch.float64) / _spectrum(dim, modes, gamma, delta)
    xi = xi.to(DEV)
    if dim == 2:
        return torch.einsum("sab,ia,jb->sij", xi, c, c).reshape(s, -1).contiguous()
    t = torch.einsum("sabc,kc->sabk", xi, c)
    t = torch.einsum("sabk,jb->sajk", t, c)
    return torch.einsum("sajk,ia->sijk", t, c).reshape(s, -1).contiguous()


def _noise_block(s, n, g):
    gd = torch.Generator(device=DEV).manual_seed(int(torch.randint(1 << 40, (1,), generator=g)))
    return torch.randn((s, n), generator=gd, dtype=torch.float64, device=DEV)


def _eigenpairs(dim, np_, gamma, delta, k, g):
    """k R-orthonormal cosine modes (scaled by the prior's spectrum, with random signs) and
    eigenvalues that decay through 1 as the informed directions of the misfit Hessian do."""
    modes = min(np_, 16 if dim == 2 else 8)
    sp = _spectrum(dim, modes, gamma, delta).reshape(-1)
    idx = torch.argsort(sp, stable=True)[:k]
    k = idx.numel()
    c = _cosines(np_, modes).to(DEV)
    sgn = (torch.randint(0, 2, (k,), generator=g) * 2 - 1).to(torch.float64)
    out = torch.empty((k, np_ ** dim), dtype=torch.float64, device=DEV)
    for j, q in enumerate(idx.tolist()):
        a = [(q // modes ** (dim - 1 - t)) % modes for t in range(dim)]
        v = torch.einsum("i,j->ij", c[:, a[0]], c[:, a[1]])
        if dim == 3:
            v = torch.einsum("ij,k->ijk", v, c[:, a[2]])
        out[j] = (sgn[j] / sp[q]).item() * v.reshape(-1)
    lam = 20.0 / (1.0 + torch.arange(k, dtype=torch.float64)) ** 1.2
    return lam.to(DEV), out


def _observations(case, g):
    xyz = 0.05 + 0.9 * torch.rand((case["nobs"], case["dim"]), generator=g, dtype=torch.float64)
    d = xyz[:, -1] + 0.01 * torch.randn(case["nobs"], generator=g, dtype=torch.float64)  # u = x_last at m = 0
    return xyz.numpy(), d.numpy()


def _problem(case, xyz, d):
    P = Problem(case["dim"], case["N"], case["gamma"], case["delta"], 0.01, xyz, d_obs=d, rtol=case["rtol"])
    if case.get("tiles"):
        P.set_tuning(nu=2, cheb_alpha=12.0, tma_tiles=1)
    return P


def _inputs(case, seed):
    """Everything random of a case, from the seed alone."""
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("unet_forward", "unet_gradient"):
        H, W, B = case["H"], case["W"], case["batch"]
        np_ = max(H, W)
        f = _prior_fields(2, np_, 0.1, 0.5, 2 * B, g).reshape(2 * B, np_, np_)[:, :H, :W]
        node = torch.zeros((H, W), device=DEV, dtype=torch.float64)
        node[:H - 7, :W - 7] = 1.0  # the nodal grid in its padding
        mask = node.clone()
        mask[0] = mask[H - 8] = 0.0  # the Dirichlet rows
        m = f[:B] * node
        z = (f[B:] + 0.3 * _noise_block(B, H * W, g).reshape(B, H, W)) * mask
        z = z / z.square().sum((1, 2), keepdim=True).div(mask.sum()).sqrt()
        x = torch.stack([m, z, mask.expand(B, H, W)], 1).float().contiguous()
        E = torch.exp(m)
        cx, cy = torch.zeros_like(E), torch.zeros_like(E)
        cx[:, :, :-1] = -0.5 * (E[:, :, :-1] + E[:, :, 1:])
        cy[:, :-1, :] = -0.5 * (E[:, :-1, :] + E[:, 1:, :])
        diag = -cx - cy
        diag[:, :, 1:] -= cx[:, :, :-1]
        diag[:, 1:, :] -= cy[:, :-1, :]
        aux = torch.stack([z * diag, diag, cx, cy], 1).float().contiguous()
        params = he_init(int(torch.randint(1 << 30, (1,), generator=g)))
        bias = 0.02 * torch.randn(params.size, generator=g, dtype=torch.float32).numpy()
        params = np.where(params == 0.0, bias, params).astype(np.float32)  # biases of a trained net are not zero
        return {"x": x, "aux": aux, "params": params}
    if kind == "batch":
        out = []
        for N in map(int, case["sizes"].split(",")):
            u = torch.rand(3, generator=g, dtype=torch.float64).tolist()
            c = {"rtol": case["rtol"], "dim": 2, "N": N, "nobs": 100 + int(700 * u[0]), "gamma": 0.05 + 0.15 * u[1],
                 "delta": 0.2 + 0.8 * u[2], "columns": case["columns"]}
            xyz, d = _observations(c, g)
            m = _prior_fields(2, N + 1, c["gamma"], c["delta"], 1, g)[0]
            out.append({"case": c, "xyz": xyz, "d": d, "m": m, "X": _noise_block(c["columns"], (N + 1) ** 2, g)})
        return {"problems": out}
    dim, np_ = case["dim"], case["N"] + 1
    n = np_ ** dim
    pr = (dim, np_, case["gamma"], case["delta"])
    if kind == "action":
        xyz, d = _observations(case, g)
        s = case["columns"]
        # single columns are search directions (smooth), blocks are random test matrices
        X = _prior_fields(*pr, 1, g) if s == 1 else _noise_block(s, n, g)
        return {"xyz": xyz, "d": d, "m": _prior_fields(*pr, 1, g)[0], "X": X}
    if kind == "gradient":
        xyz, d = _observations(case, g)
        return {"xyz": xyz, "d": d, "m": _prior_fields(*pr, 3, g)}
    if kind == "precision":
        return {"X": _prior_fields(*pr, case["columns"], g)}
    lam, V = _eigenpairs(*pr, case["k"], g)
    if kind == "samples":
        return {"lam": lam, "V": V, "m": _prior_fields(*pr, 1, g)[0], "rng": int(torch.randint(1 << 40, (1,), generator=g))}
    return {"lam": lam, "V": V, "Z": _noise_block(case["r"], n, g)}


def prepare(case, seed):
    a = _inputs(case, seed)
    kind = case["kind"]
    if kind in ("unet_forward", "unet_gradient"):
        net = UNet(case["H"], case["W"], batch_cap=case["batch"])
        net.set_params(a["params"])
        return {"case": case, "net": net, "x": a["x"], "aux": a["aux"]}
    if kind == "batch":
        ps = [_problem(q["case"], q["xyz"], q["d"]) for q in a["problems"]]
        b = Batch(ps)
        b.set_point([q["m"] for q in a["problems"]])
        return {"case": case, "batch": b, "problems": ps, "X": [q["X"] for q in a["problems"]]}
    P = _problem(case, a.pop("xyz", np.zeros((0, case["dim"]))), a.pop("d", None))
    if kind == "action":
        P.set_point(a["m"])  # the linearisation point stays for many actions
    elif kind == "gradient":
        P.set_point(a["m"][0])
    return {"case": case, "P": P, **a}


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "action":
        return state["P"].hessian_apply(state["X"], with_prior=c["prior"], full=c["full"])[0]
    if kind == "gradient":
        P, m = state["P"], state["m"]
        J1 = P.set_point(m[1])
        g, J2 = P.gradient(m[2])
        return {"J_trial": list(J1), "J": list(J2), "g": g}
    if kind == "precision":
        return state["P"].R_apply(state["X"])
    if kind == "samples":
        prior, post, _ = state["P"].laplace_sample(state["m"], state["lam"], state["V"], seed=state["rng"],
                                                   nsamples=c["nsamples"])
        return {"prior": prior, "post": post}
    if kind == "variance":
        prior, post = state["P"].pointwise_variance(state["Z"], "randomized", state["lam"], state["V"])
        return {"prior": prior, "post": post}
    if kind == "batch":
        return state["batch"].hessian_apply(state["X"])
    if kind == "unet_forward":
        return state["net"].forward(state["x"])
    loss, grad = state["net"].loss_grad(state["x"], state["aux"])
    return {"loss": loss, "grad": grad}


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------
_UNET = ((3, 16, 0), (16, 16, 0), (16, 32, 1), (32, 32, 1), (32, 64, 2), (64, 64, 2), (64, 128, 3), (128, 128, 3),
         (192, 64, 2), (64, 64, 2), (96, 32, 1), (32, 32, 1), (48, 16, 0), (16, 16, 0))  # c_in, c_out, level


def _action_work(dim, n, s, full, prior):
    nc = 7 if dim == 2 else 15
    # X in, Y out, the coefficients of K (diagonal and forward couplings) and of C
    by = 16.0 * n * s + 8.0 * n * (nc + 1 + dim)
    # C, C^T and one application of K for each of the two solves, in each pass twice the couplings
    fl = 2.0 * n * s * (2 * nc + 2 * (2 * dim + 1)) * (1.5 if full else 1.0)
    if prior:
        fl += 2.0 * n * s * 3 * nc
    return by, fl


def work(case):
    kind = case["kind"]
    if kind in ("unet_forward", "unet_gradient"):
        px = case["H"] * case["W"] * case["batch"]
        mac = sum(9 * a * b * px / 4 ** lv for a, b, lv in _UNET) + 16 * px
        if kind == "unet_forward":
            return {"bytes": 16.0 * px, "flops": 2.0 * mac}
        return {"bytes": 28.0 * px + 8.0 * 487665, "flops": 6.0 * mac}
    if kind == "batch":
        b = f = 0.0
        for N in map(int, case["sizes"].split(",")):
            x, y = _action_work(2, (N + 1) ** 2, case["columns"], False, False)
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    dim = case["dim"]
    n = (case["N"] + 1) ** dim
    nf = (1 << (dim + 1)) - 1  # couplings of the prior and the mass
    if kind == "action":
        b, f = _action_work(dim, n, case["columns"], case["full"], case["prior"])
    elif kind == "gradient":
        b, f = 24.0 * n, 2.0 * n * (2 * nf + 3 * nf + 3 * (2 * dim + 1))
    elif kind == "precision":
        b, f = 16.0 * n * case["columns"], 2.0 * n * case["columns"] * 3 * nf
    elif kind == "samples":
        b = 16.0 * n * case["nsamples"] + 8.0 * n * case["k"]
        f = 2.0 * n * case["nsamples"] * (3 * nf + 2 * case["k"])
    else:
        r = case["r"]
        b, f = 8.0 * n * (r + case["k"] + 2), 2.0 * n * r * (6 * nf + 2 * r)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same maps in 64 bits
# ---------------------------------------------------------------------------
class _Fem:
    """P1 finite elements on the Kuhn triangulation of the unit square / cube: blocks are
    (s, np, .., np) with the first space axis last."""

    def __init__(self, dim, N, gamma, delta):
        self.D, self.N, self.np, self.h = dim, N, N + 1, 1.0 / N
        self.n = self.np ** dim
        self.vol = self.h ** dim / math.factorial(dim)
        self.chains = []
        axes = list(range(dim))

        def perms(p, rest):
            if not rest:
                self.chains.append([0] + [sum(1 << a for a in p[:k + 1]) for k in range(dim)])
            for a in rest:
                perms(p + [a], [b for b in rest if b != a])
        perms([], axes)
        mass = self.vol / ((dim + 1) * (dim + 2))
        one = torch.ones((1,) + (N,) * dim, dtype=torch.float64, device=DEV)
        self.M = self._assemble(lambda c, i, j: one * (mass * (2.0 if i == j else 1.0)))
        self.K1 = self._assemble(lambda c, i, j: one * (self.vol / self.h ** 2 * self._lap(i, j)))
        self.A = {b: gamma * self.K1.get(b, 0.0) + delta * self.M[b] for b in self.M}
        self.gamma, self.delta = gamma, delta

    def _lap(self, i, j):  # grad(lambda_i) . grad(lambda_j) h^2 on a chain of D + 1 vertices
        if i == j:
            return 1.0 if i in (0, self.D) else 2.0
        return -1.0 if abs(i - j) == 1 else 0.0

    def grid(self, x):
        return x.reshape((-1,) + (self.np,) * self.D)

    def corner(self, x, b):
        """x at the corner b of every cell."""
        for a in range(self.D):
            x = x.narrow(x.dim() - 1 - a, (b >> a) & 1, self.N)
        return x

    def _assemble(self, entry):
        out = {}
        for c in self.chains:
            for i in range(self.D + 1):
                for j in range(i, self.D + 1):
                    b = c[j] ^ c[i]
                    e = entry(c, i, j)
                    if b not in out:
                        out[b] = torch.zeros((1,) + (self.np,) * self.D, dtype=torch.float64, device=DEV)
                    self.corner(out[b], c[i]).add_(e)
        return out

    def apply(self, S, x):
        """The symmetric stencil S = {edge mask b: coupling of node i with node i + b}."""
        y = S[0] * x
        for b, w in S.items():
            if b == 0:
                continue
            lo, hi = [slice(None)], [slice(None)]
            for a in reversed(range(self.D)):
                bit = (b >> a) & 1
                lo.append(slice(0, self.N) if bit else slice(None))
                hi.append(slice(1, None) if bit else slice(None))
            lo, hi = tuple(lo), tuple(hi)
            y[lo] += w[lo] * x[hi]
            y[hi] += w[lo] * x[lo]
        return y

    def stiffness(self, E):
        kap = [sum(self.corner(E, b) for b in c) / (self.D + 1) for c in self.chains]
        return self._assemble(lambda c, i, j: kap[self.chains.index(c)] * (self.vol / self.h ** 2 * self._lap(i, j))
                              if self._lap(i, j) else 0.0 * kap[0])

    def clamp(self, x):
        """Zero on the two Dirichlet faces (the last axis is dimension 1)."""
        x = x.clone()
        x[:, 0] = 0.0
        x[:, -1] = 0.0
        return x

    def C(self, E, u, x):
        out = torch.zeros_like(x)
        v = E * x
        for c in self.chains:
            kap = sum(self.corner(v, b) for b in c) / (self.D + 1) * (self.vol / self.h ** 2)
            for k in range(self.D):
                f = kap * (self.corner(u, c[k + 1]) - self.corner(u, c[k]))
                self.corner(out, c[k]).sub_(f)
                self.corner(out, c[k + 1]).add_(f)
        return out

    def Ct(self, E, u, w):
        out = torch.zeros_like(w)
        for c in self.chains:
            g = sum((self.corner(u, c[k + 1]) - self.corner(u, c[k])) * (self.corner(w, c[k + 1]) - self.corner(w, c[k]))
                    for k in range(self.D)) * (self.vol / self.h ** 2)
            for b in c:
                self.corner(out, b).add_(g)
        return E * out / (self.D + 1)

    def _modes(self, dirichlet):
        """Per space axis the eigenvectors of the 1D stiffness in the lumped mass and their
        eigenvalues; the last space axis with Dirichlet ends if asked."""
        i = torch.arange(self.np, dtype=torch.float64, device=DEV)
        lam = 2.0 - 2.0 * torch.cos(math.pi * i / self.N)
        out = []
        for a in range(self.D):
            if dirichlet and a == self.D - 1:
                q = torch.sin(math.pi * i[:, None] * i[None, :] / self.N)
            else:
                q = torch.cos(math.pi * i[:, None] * i[None, :] / self.N)
            w = torch.ones_like(i)
            w[0] = w[-1] = 0.5
            nrm = (w[:, None] * q.square()).sum(0)
            q = q / nrm.clamp(min=1e-8).sqrt()
            out.append((q.float(), lam))
        return out

    def _spectral(self, dirichlet, a, b, scale=None):
        """x -> s (a K1 + b lumped M)^-1 s x in 32 bits (s = scale, a field), a preconditioner."""
        md = self._modes(dirichlet)
        lam = 0.0
        for ax in range(self.D):
            sh = [1] * (self.D + 1)
            sh[self.D - ax] = self.np
            lam = lam + md[ax][1].reshape(sh)
        den = (a * self.h ** (self.D - 2) * lam + b * self.h ** self.D).float()
        inv = torch.where(den > 0, 1.0 / den, torch.zeros_like(den))

        def go(x, t):
            for ax in range(self.D):
                q = md[ax][0]
                x = torch.movedim(torch.movedim(x, self.D - ax, -1) @ (q if t else q.T), -1, self.D - ax)
            return x

        def apply(r):
            r = r if scale is None else r * scale
            nr = r.flatten(1).norm(dim=1).clamp(min=1e-300).reshape((-1,) + (1,) * self.D)
            z = go(inv * go((r / nr).float(), True), False).double() * nr
            return z if scale is None else z * scale
        return apply

    def solve(self, S, b, dirichlet=False, prec=None):
        """S x = b by preconditioned conjugate gradients to rounding level, column by column."""
        op = (lambda x: self.clamp(self.apply(S, self.clamp(x)))) if dirichlet else (lambda x: self.apply(S, x))
        if dirichlet:
            b = self.clamp(b)
        sh = (-1,) + (1,) * self.D
        dot = lambda p, q: (p.flatten(1) * q.flatten(1)).sum(1)  # noqa: E731
        nb = dot(b, b).sqrt().clamp(min=1e-300)
        x = torch.zeros_like(b)
        for _ in range(3):
            r = b - op(x)
            if float((dot(r, r).sqrt() / nb).max()) < 2e-15:
                break
            z = prec(r)
            p, rz = z.clone(), dot(r, z)
            d = torch.zeros_like(b)
            for it in range(600):
                q = op(p)
                pq = dot(p, q)
                al = torch.where(pq > 0, rz / pq.clamp(min=1e-300), torch.zeros_like(rz)).reshape(sh)
                d += al * p
                r -= al * q
                if it % 8 == 7 and float((dot(r, r).sqrt() / nb).max()) < 1e-15:
                    break
                z = prec(r)
                rzn = dot(r, z)
                p = z + torch.where(rz > 0, rzn / rz.clamp(min=1e-300), torch.zeros_like(rz)).reshape(sh) * p
                rz = rzn
            x = x + d
        return x

    def A_solve(self, b):
        return self.solve(self.A, b, prec=self._spectral(False, self.gamma, self.delta))

    def M_solve(self, b):
        return self.solve(self.M, b, prec=lambda r: r / self.M[0])

    def R(self, x):
        return self.apply(self.A, self.M_solve(self.apply(self.A, x)))

    def Rinv(self, x):
        return self.A_solve(self.apply(self.M, self.A_solve(x)))

    def observe(self, xyz):
        """(index, weight) of the P1 interpolation at the points."""
        t = torch.as_tensor(xyz, dtype=torch.float64, device=DEV).clamp(0, 1) * self.N
        c = t.floor().clamp(max=self.N - 1)
        loc, pi = torch.sort(t - c, dim=1, descending=True, stable=True)
        q = t.shape[0]
        one, zero = torch.ones((q, 1), device=DEV, dtype=torch.float64), torch.zeros((q, 1), device=DEV, dtype=torch.float64)
        ext = torch.cat([one, loc, zero], 1)
        w = ext[:, :-1] - ext[:, 1:]
        stride = torch.tensor([self.np ** a for a in range(self.D)], device=DEV)
        base = (c.long() * stride).sum(1, keepdim=True)
        idx = base + torch.cat([torch.zeros((q, 1), device=DEV, dtype=torch.long), stride[pi].cumsum(1)], 1)
        return idx, w


class _Point:
    """The linearisation point m: state, observation operator and the solves at it."""

    def __init__(self, case, xyz, d, m):
        self.f = f = _Fem(case["dim"], case["N"], case["gamma"], case["delta"])
        self.m = f.grid(m.double())
        self.E = torch.exp(self.m)
        self.K = f.stiffness(self.E)
        self.prec = f._spectral(True, 1.0, 0.0, torch.exp(-0.5 * self.m))
        lift = torch.zeros_like(self.m)
        lift[:, -1] = 1.0
        self.u = lift + self.Kinv(-f.apply(self.K, lift))
        self.idx, self.w = f.observe(xyz)
        self.d = torch.as_tensor(d, dtype=torch.float64, device=DEV)
        self.is2 = 1.0 / 0.01 ** 2

    def Kinv(self, b):
        return self.f.solve(self.K, b, dirichlet=True, prec=self.prec)

    def B(self, u):
        return (u.flatten(1)[:, self.idx] * self.w).sum(-1)

    def Bt(self, y):
        out = torch.zeros((y.shape[0], self.f.n), dtype=torch.float64, device=DEV)
        out.index_add_(1, self.idx.reshape(-1), (y[:, :, None] * self.w).flatten(1))
        return self.f.grid(out)

    def adjoint(self):
        return self.Kinv(-self.is2 * self.Bt(self.B(self.u) - self.d))

    def action(self, X, prior, full):
        f, x = self.f, self.f.grid(X)
        uh = self.Kinv(-f.C(self.E, self.u, x))
        rhs = -self.is2 * self.Bt(self.B(uh))
        if full:
            p = self.adjoint()
            rhs = rhs - f.C(self.E, p, x)
        y = f.Ct(self.E, self.u, self.Kinv(rhs))
        if full:
            y = y + f.Ct(self.E, p, uh) + x * f.Ct(self.E, self.u, p)
        if prior:
            y = y + f.R(x)
        return y.flatten(1)

    def cost(self):
        r = self.B(self.u) - self.d
        mis = 0.5 * self.is2 * float(r.square().sum())
        reg = 0.5 * float((self.m * self.f.R(self.m)).sum())
        return [mis + reg, mis, reg]

    def gradient(self):
        return (self.f.R(self.m) + self.f.Ct(self.E, self.u, self.adjoint())).reshape(-1)


def _philox(seed, sample, ncalls):
    """The sampler's normals (Philox4x32-10 and Box-Muller) of one sample, in 64 bits."""
    lo32 = (1 << 32) - 1
    g = torch.arange(ncalls, device=DEV, dtype=torch.int64)
    c = [g & lo32, g >> 32, torch.full_like(g, sample & lo32), torch.full_like(g, sample >> 32)]
    k = [seed & lo32, seed >> 32]

    def mul(a, b):  # (high, low) words of a 32 x 32-bit product
        t = a * (b & 0xffff)
        u = a * (b >> 16) + (t >> 16)
        return u >> 16, ((u & 0xffff) << 16) | (t & 0xffff)
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k[0], l1, h0 ^ c[3] ^ k[1], l0]
        k = [(k[0] + 0x9E3779B9) & lo32, (k[1] + 0xBB67AE85) & lo32]
    u = [((w >> 8).double() + 0.5) / (1 << 24) for w in c]
    out = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        r = torch.sqrt(-2.0 * torch.log(a))
        out += [r * torch.cos(2.0 * math.pi * b), r * torch.sin(2.0 * math.pi * b)]
    return torch.stack(out, 1).reshape(-1)


def _samples_exact(case, a):
    f = _Fem(case["dim"], case["N"], case["gamma"], case["delta"])
    D, ns = case["dim"], case["nsamples"]
    nq, nc = D + 1, len(f.chains)
    nper = f.N ** D * nc * nq
    q2 = [[0.5, 0.5, 0.0], [0.0, 0.5, 0.5], [0.5, 0.0, 0.5]]
    s5 = math.sqrt(5.0)
    W = torch.zeros((ns,) + (f.np,) * D, dtype=torch.float64, device=DEV)
    for j in range(ns):
        eta = _philox(a["rng"], j, (nper + 3) // 4)[:nper].reshape((1,) + (f.N,) * D + (nc, nq))
        for p, c in enumerate(f.chains):
            for k, b in enumerate(c):
                for q in range(nq):
                    lam = q2[q][k] if D == 2 else ((5 + 3 * s5) / 20 if q == k else (5 - s5) / 20)
                    if lam:
                        f.corner(W[j:j + 1], b).add_(eta[..., p, q], alpha=lam * math.sqrt(f.vol / (D + 1)))
    x = f.A_solve(W)
    RX = f.apply(f.A, f.M_solve(W)).flatten(1)
    x = x.flatten(1)
    S = 1.0 - 1.0 / torch.sqrt(1.0 + a["lam"])
    return {"prior": x, "post": a["m"][None] + x - ((RX @ a["V"].T) * S) @ a["V"]}


def _variance_exact(case, a):
    f = _Fem(case["dim"], case["N"], case["gamma"], case["delta"])
    Q = torch.linalg.qr(f.Rinv(f.grid(a["Z"])).flatten(1).T)[0].T.contiguous()
    T = Q @ f.Rinv(f.grid(Q)).flatten(1).T
    prior = ((0.5 * (T + T.T)) @ Q * Q).sum(0)
    post = prior - ((a["lam"] / (1.0 + a["lam"]))[:, None] * a["V"].square()).sum(0)
    return {"prior": prior, "post": post}


def _unet_layers(params):
    spec = [(a, b, 3) for a, b, _ in _UNET] + [(16, 1, 1)]
    p, off, out = torch.as_tensor(params), 0, []
    for ci, co, k in spec:
        w = p[off:off + co * ci * k * k].reshape(co, ci, k, k)
        off += w.numel()
        out.append((w.bfloat16().double().to(DEV).requires_grad_(True), p[off:off + co].double().to(DEV).requires_grad_(True)))
        off += co
    return out


def _conv(x, wb, relu=True):
    w, b = wb
    N, _, H, W = x.shape
    k = w.shape[-1]
    cols = torch.nn.functional.unfold(x, k, padding=k // 2)
    y = (w.reshape(w.shape[0], -1) @ cols + b[:, None]).reshape(N, -1, H, W)
    return torch.relu(y) if relu else y


def _unet_exact(L, x):
    pool = lambda t: torch.nn.functional.avg_pool2d(t, 2)  # noqa: E731
    up = lambda t: t.repeat_interleave(2, 2).repeat_interleave(2, 3)  # noqa: E731
    e1 = _conv(_conv(x, L[0]), L[1])
    e2 = _conv(_conv(pool(e1), L[2]), L[3])
    e3 = _conv(_conv(pool(e2), L[4]), L[5])
    t = _conv(_conv(pool(e3), L[6]), L[7])
    for i, e in ((8, e3), (10, e2), (12, e1)):
        t = _conv(_conv(torch.cat([up(t), e], 1), L[i]), L[i + 1])
    return _conv(t, L[14], relu=False)


def _unet_loss(y, x, aux):
    """1/(2N) sum_n |mask b - S y|^2 / |mask b|^2 with S = mask K mask, K the 5-point stencil."""
    mask = x[:, 2]
    b, diag, cx, cy = aux.unbind(1)
    v = y[:, 0] * mask
    Kv = diag * v
    Kv = Kv + torch.nn.functional.pad(cx[:, :, :-1] * v[:, :, 1:], (0, 1)) + torch.nn.functional.pad(cx[:, :, :-1] * v[:, :, :-1], (1, 0))
    Kv = Kv + torch.nn.functional.pad(cy[:, :-1] * v[:, 1:], (0, 0, 0, 1)) + torch.nn.functional.pad(cy[:, :-1] * v[:, :-1], (0, 0, 1, 0))
    r = mask * b - mask * Kv
    return 0.5 * (r.square().sum((1, 2)) / (mask * b).square().sum((1, 2))).sum()


def exact(case, seed):
    a = _inputs(case, seed)
    kind = case["kind"]
    if kind == "action":
        return _Point(case, a["xyz"], a["d"], a["m"]).action(a["X"], case["prior"], case["full"])
    if kind == "gradient":
        J1 = _Point(case, a["xyz"], a["d"], a["m"][1]).cost()
        p = _Point(case, a["xyz"], a["d"], a["m"][2])
        return {"J_trial": J1, "J": p.cost(), "g": p.gradient()}
    if kind == "precision":
        f = _Fem(case["dim"], case["N"], case["gamma"], case["delta"])
        return f.R(f.grid(a["X"])).flatten(1)
    if kind == "samples":
        return _samples_exact(case, a)
    if kind == "variance":
        return _variance_exact(case, a)
    if kind == "batch":
        return [_Point(q["case"], q["xyz"], q["d"], q["m"]).action(q["X"], False, False) for q in a["problems"]]
    L = _unet_layers(a["params"])
    N = case["batch"]
    if kind == "unet_forward":
        with torch.no_grad():
            return torch.cat([_unet_exact(L, a["x"][i:i + 1].double()) for i in range(N)])
    loss = 0.0
    for i in range(N):
        x, aux = a["x"][i:i + 1].double(), a["aux"][i:i + 1].double()
        li = _unet_loss(_unet_exact(L, x), x, aux) / N
        li.backward()
        loss += float(li.detach())
    grad = torch.cat([t.grad.reshape(-1) for wb in L for t in wb])
    return {"loss": loss, "grad": grad.cpu().numpy()}
