"""What a user of this library runs: whole solves, eigenvalue runs, batches of systems, single
applications of the preconditioner and the training gradient, each through the public binding.

A case is a dict of plain values; `kind` says which entry point it calls:
  solve   krylov_solve on one brick (variant, cycle, storage precision, preconditioner on or off)
  eig     lobpcg_solve, the m smallest eigenpairs of one brick
  batch   smg_batched_solve, many uneven systems together
  apply   smg_apply_batched, one V-cycle on nb right-hand sides
  grad    smg_net_loss_grad, one training step's loss and gradient of the learned correction
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1212_6680_gb300 import inputs, smg

TOL = 1e-8


def _solve(name, nx, ny, nz, variant="fpcg", npost=0, prec="fp32", precond=True):
    return {"name": name, "kind": "solve", "nx": nx, "ny": ny, "nz": nz, "variant": variant, "npre": 1,
            "npost": npost, "prec": prec, "precond": precond}


def listed():
    return [
        # the smallest grid solved in earnest: launches and latency only
        _solve("solve-24x20x16", 24, 20, 16),
        # the library's headline: flexible PCG without post-smoothing, FP32 cycle
        _solve("solve-128", 128, 128, 128),
        # eight times the headline: the vectors no longer fit in L2
        _solve("solve-256", 256, 256, 256),
        # everything in FP64 with the balanced cycle, for users who want no mixed precision
        _solve("solve-128-fp64", 128, 128, 128, variant="pcg", npost=1, prec="fp64"),
        # the paper's largest brick, 16n x n x n with n = 80: long x-lines
        _solve("solve-1280x80x80", 1280, 80, 80),
        # no side a multiple of anything, the balanced cycle under standard PCG
        _solve("solve-101x75x53", 101, 75, 53, variant="pcg", npost=1),
        # no preconditioner (the paper's first figures): the Krylov kernels alone
        _solve("cg-128", 128, 128, 128, variant="pcg", prec="fp64", precond=False),
        # a block of eigenpairs; unequal sides, so that the eigenvectors are determined
        {"name": "eig-16", "kind": "eig", "nx": 112, "ny": 97, "nz": 83, "npost": 0, "m": 16},
        # one eigenpair on the paper's 4n x 2n x 2n brick, n = 40
        {"name": "eig-1", "kind": "eig", "nx": 160, "ny": 80, "nz": 80, "npost": 0, "m": 1},
        # many uneven systems at once (sides 32..96): the serving load
        {"name": "batch-64", "kind": "batch", "nsys": 64, "lo": 32, "hi": 96, "dims_seed": 1000},
        # the preconditioner alone on a block, as a user's own block solver calls it
        {"name": "apply-8", "kind": "apply", "nx": 96, "ny": 96, "nz": 96, "npost": 0, "prec": "fp32", "nb": 8},
        # one step of training the learned correction (sides 64..128 in the shipped recipe)
        {"name": "grad-96", "kind": "grad", "nx": 96, "ny": 80, "nz": 64},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "cg", "eig", "batch", "apply", "grad"])
    if kind in ("solve", "cg"):
        prec = rng.choice(["fp32", "fp32", "fp64"]) if kind == "solve" else "fp64"
        most = {"fp32": 8e6, "fp64": 2e6}[prec]
        while True:
            nx, ny, nz = _log(rng, 12, 1280 if kind == "solve" else 160), _log(rng, 10, 256), _log(rng, 10, 256)
            if 4e3 <= nx * ny * nz <= most:
                break
        npost = rng.choice([0, 0, 1])
        variant = rng.choice(["pcg", "fpcg", "psd"]) if npost else rng.choice(["fpcg", "fpcg", "psd"])
        if kind == "cg":
            npost, variant = 0, rng.choice(["pcg", "fpcg"])
        c = _solve("", nx, ny, nz, variant, npost, prec, kind == "solve")
        del c["name"]
        return c
    if kind == "eig":
        while True:  # sides whose m + 1 smallest eigenvalues are apart: the eigenvectors are then determined
            m = rng.choice([1, 1, 2, 4, 8])
            nx, ny, nz = _log(rng, 24, 320), _log(rng, 20, 120), _log(rng, 20, 120)
            if not 2e4 <= nx * ny * nz <= 1e6:
                continue
            w = _eigenvalues(nx, ny, nz, m + 1)
            if np.min(np.diff(w) / w[1:]) > 0.02:
                return {"kind": "eig", "nx": nx, "ny": ny, "nz": nz, "npost": rng.choice([0, 1]), "m": m}
    if kind == "batch":
        lo = _log(rng, 20, 48)
        return {"kind": "batch", "nsys": _log(rng, 4, 48), "lo": lo, "hi": min(112, 2 * lo + rng.randrange(24)),
                "dims_seed": rng.randrange(1 << 20)}
    if kind == "apply":
        while True:
            nx, ny, nz, nb = _log(rng, 12, 512), _log(rng, 10, 160), _log(rng, 10, 160), _log(rng, 1, 16)
            if 4e3 <= nx * ny * nz * nb <= 4e6:
                return {"kind": "apply", "nx": nx, "ny": ny, "nz": nz, "npost": rng.choice([0, 1]),
                        "prec": rng.choice(["fp32", "fp32", "fp64"]), "nb": nb}
    return {"kind": "grad", "nx": _log(rng, 48, 112), "ny": _log(rng, 48, 112), "nz": _log(rng, 48, 112)}


def _rand(seed, shape, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 17)
    return torch.rand(shape, generator=g, dtype=dtype, device="cuda") * 2 - 1


def _dims(case):
    return inputs.uneven_dims(case["nsys"], case["lo"], case["hi"], seed=case["dims_seed"])


def _offsets(dims):
    """Where each system's vector starts in one buffer (multiples of 32 values), and its length."""
    n = np.prod(dims, axis=1)
    pad = (n + 31) // 32 * 32
    return np.concatenate([[0], np.cumsum(pad)]), n


class _Batched:
    """Owns a batched handle."""

    def __init__(self, dims):
        self.h = smg.smg_batched_setup(dims, 1, 0, "fp32")

    def __del__(self):
        smg.smg_batched_destroy(self.h)


def prepare(case, seed):
    k = case["kind"]
    if k == "batch":
        dims = _dims(case)
        off, n = _offsets(dims)
        b, x = _rand(seed, (int(off[-1]),)), torch.zeros(int(off[-1]), dtype=torch.float64, device="cuda")
        cut = lambda v: [v[int(o):int(o) + int(m)] for o, m in zip(off, n)]  # noqa: E731
        return {"case": case, "H": _Batched(dims), "x": x, "b_list": cut(b), "x_list": cut(x)}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    N = nx * ny * nz
    if k == "grad":
        w = inputs.net_init_weights(seed=77)
        return {"case": case, "w": w, "rho": _rand(2 * seed, (N,)), "e": _rand(2 * seed + 1, (N,))}
    H = smg.Handle(nx, ny, nz, case.get("npre", 1), case["npost"], case.get("prec", "fp32"))
    s = {"case": case, "H": H}
    if k == "solve":
        if not case["precond"]:
            smg.smg_set_option(H.h, smg.SMG_OPT_PRECOND, 0)
        s["b"] = _rand(seed, (N,))
        s["x"] = torch.zeros(N, dtype=torch.float64, device="cuda")
    elif k == "eig":
        g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 17)
        s["X0"] = torch.randn((case["m"], N), generator=g, dtype=torch.float64, device="cuda")
        s["X"] = torch.empty_like(s["X0"])
    else:
        s["R"] = _rand(seed, (case["nb"], N))
        s["S"] = torch.empty_like(s["R"])
    return s


def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "solve":
        s["x"].zero_()
        _, it, _ = smg.krylov_solve(s["H"].h, case["variant"], s["b"], s["x"], TOL, 5000)
        return {"x": s["x"], "iters": it}
    if k == "eig":
        s["X"].copy_(s["X0"])
        _, it, lam = smg.lobpcg_solve(s["H"].h, case["m"], s["X"], TOL, 200)
        # an eigenvector's sign is arbitrary: the first component positive
        return {"X": s["X"] * s["X"][:, :1].sign(), "lambda": lam, "iters": it}
    if k == "batch":
        s["x"].zero_()
        _, it, _ = smg.smg_batched_solve(s["H"].h, "fpcg", s["b_list"], s["x_list"], TOL, 100)
        return {"x": s["x"], "iters": it}
    if k == "apply":
        smg.smg_apply_batched(s["H"].h, case["nb"], s["R"], s["S"])
        # an FP32 cycle stores its result in 32 bits and widens it exactly: they are 32-bit numbers
        return {"s": s["S"] if case["prec"] == "fp64" else s["S"].float()}
    loss, g = smg.smg_net_loss_grad((case["nx"], case["ny"], case["nz"]), "bf16", s["w"], s["rho"], s["e"])
    return {"loss": loss, "grad": g}


def work(case):
    """Inputs read and outputs written once.  Operations: the stencils and line solves of the
    cycles (about 60 per point and relaxation sweep, all levels) and the recurrences (30 per point)
    over the iterations such a solve takes to 1e-8."""
    k = case["kind"]
    if k == "batch":
        N = int(np.sum(np.prod(_dims(case), axis=1)))
        return {"bytes": 16 * N, "flops": N * 11 * 250}
    N = case["nx"] * case["ny"] * case["nz"]
    if k == "grad":
        return {"bytes": 16 * N, "flops": N * 3 * 2 * 27 * 288}
    cycle = 120 * (1 + case["npost"]) + 60
    if k == "solve":
        if not case["precond"]:
            return {"bytes": 16 * N, "flops": N * 30 * int(3.5 * max(case["nx"], case["ny"], case["nz"]))}
        it = 7 if case["npost"] else 11
        return {"bytes": 16 * N, "flops": N * it * (cycle + 30)}
    if k == "eig":
        m = case["m"]
        return {"bytes": 16 * N * m, "flops": N * 35 * (m * (cycle + 30) + 36 * m * m)}
    return {"bytes": 16 * N * case["nb"], "flops": N * case["nb"] * cycle}


# ---- the same results in 64 bits, by plain torch and numpy ------------------------------------------

def _sines(n):
    j = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
    # the argument is reduced in integers first, so that the table is accurate to the last bits
    a = torch.remainder(torch.outer(j, j), 2 * (n + 1))
    return torch.sin(a * (math.pi / (n + 1))) * math.sqrt(2.0 / (n + 1))


def _lam(n):
    j = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
    return 4 * torch.sin(j * (math.pi / (2 * (n + 1)))) ** 2


def _eigenvalues(nx, ny, nz, count):
    """The `count` smallest eigenvalues of the 7-point operator (closed form)."""
    w = [4 * np.sin(np.arange(1, min(n, 32) + 1) * np.pi / (2 * (n + 1))) ** 2 for n in (nx, ny, nz)]
    return np.sort((w[0][:, None, None] + w[1][None, :, None] + w[2][None, None, :]).ravel())[:count]


def _eigenvectors(nx, ny, nz, count):
    """Their unit eigenvectors, products of sines (positive at the first point), one per row."""
    w = [4 * np.sin(np.arange(1, min(n, 32) + 1) * np.pi / (2 * (n + 1))) ** 2 for n in (nx, ny, nz)]
    s = w[0][:, None, None] + w[1][None, :, None] + w[2][None, None, :]
    V = [_sines(n) for n in (nx, ny, nz)]
    rows = []
    for q in np.argsort(s, axis=None)[:count]:
        i, j, k = (int(v) for v in np.unravel_index(q, s.shape))
        rows.append(torch.einsum("z,y,x->zyx", V[2][k], V[1][j], V[0][i]).reshape(-1))
    return torch.stack(rows)


def _poisson(b, nx, ny, nz):
    """A^-1 b by the sine eigenvectors of the three directions."""
    Vx, Vy, Vz = _sines(nx), _sines(ny), _sines(nz)

    def both(u):
        u = u @ Vx
        u = torch.einsum("zyx,yk->zkx", u, Vy)
        return (Vz @ u.reshape(nz, -1)).reshape(nz, ny, nx)

    d = _lam(nz)[:, None, None] + _lam(ny)[None, :, None] + _lam(nx)[None, None, :]
    return both(both(b.reshape(nz, ny, nx)) / d).reshape(-1)


def _prolongation(X):
    """Injection of the odd points, the even ones weighted by the collapsed couplings X."""
    n = X.shape[0]
    P = np.zeros((n, n // 2))
    for i in range(n):
        if i % 2:
            P[i, i // 2] = 1.0
        else:
            if i > 0:
                P[i, i // 2 - 1] = -X[i, i - 1] / X[i, i]
            if i + 1 < n:
                P[i, i // 2] = -X[i, i + 1] / X[i, i]
    return P


def _plane_cycle(c, d, ny, lam, g):
    """One 2D cycle with zero initial guess for planes with operators c L2D + d; g is
    [batch, plane, line, mode], the x-line matrices being diagonal in their sine eigenvectors."""
    S = [c[p] * np.eye(ny) for p in range(len(c))]
    T = [c[p] * (2 * np.eye(ny) - np.eye(ny, k=1) - np.eye(ny, k=-1)) + d[p] * np.eye(ny) for p in range(len(c))]

    def level(S, T, g):
        n = S[0].shape[0]
        dev = lambda M: torch.tensor(np.stack(M), device="cuda")  # noqa: E731
        St, Tt = dev(S), dev(T)
        diag = torch.diagonal(St, dim1=1, dim2=2)[:, :, None] * lam + torch.diagonal(Tt, dim1=1, dim2=2)[:, :, None]
        if n == 1:
            return g / diag

        def mul(u):  # B u
            return torch.einsum("pij,bpjk->bpik", St, u * lam) + torch.einsum("pij,bpjk->bpik", Tt, u)

        u = torch.zeros_like(g)

        def relax(u, odd):
            r = g - mul(u)
            u = u.clone()
            u[:, :, odd::2] += r[:, :, odd::2] / diag[:, odd::2]
            return u

        u = relax(relax(u, 0), 1)
        P = [_prolongation(t) for t in T]
        Pt = dev(P)
        coarse = level([p.T @ s @ p for p, s in zip(P, S)], [p.T @ t @ p for p, t in zip(P, T)],
                       torch.einsum("pij,bpik->bpjk", Pt, g - mul(u)))
        u = u + torch.einsum("pij,bpjk->bpik", Pt, coarse)
        return relax(relax(u, 1), 0)

    return level(S, T, g)


def _vcycle(r, nx, ny, nz, npre, npost):
    """The V-cycle on r [batch, z, y, x], in the sine eigenvectors of the x-lines."""
    V, lam = _sines(nx), _lam(nx)

    def lap(u):  # (lambda + Ly) u
        w = (lam + 2) * u
        w[:, :, 1:] -= u[:, :, :-1]
        w[:, :, :-1] -= u[:, :, 1:]
        return w

    def level(M, K, f):
        n = M.shape[0]
        Mt, Kt = torch.tensor(M, device="cuda"), torch.tensor(K, device="cuda")

        def mul(u):
            return torch.einsum("zw,bwyk->bzyk", Mt, lap(u)) + torch.einsum("zw,bwyk->bzyk", Kt, u)

        def sweep(u, odd):
            g = (f - mul(u))[:, odd::2]
            u = u.clone()
            u[:, odd::2] += _plane_cycle(np.diag(M)[odd::2], np.diag(K)[odd::2], ny, lam, g)
            return u

        u = torch.zeros_like(f)
        if n == 1:
            return sweep(u, 0)
        for _ in range(npre):
            u = sweep(sweep(u, 0), 1)
        P = _prolongation(K)
        Pt = torch.tensor(P, device="cuda")
        e = level(P.T @ M @ P, P.T @ K @ P, torch.einsum("zc,bzyk->bcyk", Pt, f - mul(u)))
        u = u + torch.einsum("zc,bcyk->bzyk", Pt, e)
        for _ in range(npost):
            u = sweep(sweep(u, 1), 0)
        return u

    K = 2 * np.eye(nz) - np.eye(nz, k=1) - np.eye(nz, k=-1)
    return level(np.eye(nz), K, r @ V) @ V


def _net(w, rho, nx, ny, nz):
    conv = torch.nn.functional.conv3d
    w1, w2, w3 = w[:432].view(16, 1, 3, 3, 3), w[432:7344].view(16, 16, 3, 3, 3), w[7344:].view(1, 16, 3, 3, 3)
    rms = rho.square().mean().sqrt()
    a = (rho / rms).view(1, 1, nz, ny, nx)
    a = torch.relu(conv(a, w1, padding=1))
    a = torch.relu(conv(a, w2, padding=1))
    return conv(a, w3, padding=1).view(-1) * rms


def _apply_A(u, nx, ny, nz):
    p = torch.nn.functional.pad(u.view(nz, ny, nx), (1, 1, 1, 1, 1, 1))
    c = p[1:-1, 1:-1, 1:-1]
    return (6 * c - p[1:-1, 1:-1, :-2] - p[1:-1, 1:-1, 2:] - p[1:-1, :-2, 1:-1] - p[1:-1, 2:, 1:-1]
            - p[:-2, 1:-1, 1:-1] - p[2:, 1:-1, 1:-1]).reshape(-1)


def exact(case, seed):
    k = case["kind"]
    if k == "batch":
        dims = _dims(case)
        off, n = _offsets(dims)
        b, x = _rand(seed, (int(off[-1]),)), torch.zeros(int(off[-1]), dtype=torch.float64, device="cuda")
        for o, m, (nx, ny, nz) in zip(off, n, dims):
            x[int(o):int(o) + int(m)] = _poisson(b[int(o):int(o) + int(m)], int(nx), int(ny), int(nz))
        return {"x": x, "iters": None}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    N = nx * ny * nz
    if k == "solve":
        return {"x": _poisson(_rand(seed, (N,)), nx, ny, nz), "iters": None}
    if k == "eig":
        return {"X": _eigenvectors(nx, ny, nz, case["m"]), "lambda": _eigenvalues(nx, ny, nz, case["m"]), "iters": None}
    if k == "apply":
        r = _rand(seed, (case["nb"], N)).view(case["nb"], nz, ny, nx)
        return {"s": _vcycle(r, nx, ny, nz, 1, case["npost"]).reshape(case["nb"], N)}
    w = torch.tensor(inputs.net_init_weights(seed=77), device="cuda").bfloat16().double().requires_grad_(True)
    rho, e = _rand(2 * seed, (N,)), _rand(2 * seed + 1, (N,))
    d = e - _net(w, rho, nx, ny, nz)
    loss = torch.dot(d, _apply_A(d, nx, ny, nz)) / torch.dot(e, _apply_A(e, nx, ny, nz))
    loss.backward()
    return {"loss": loss.item(), "grad": w.grad.detach()}
