"""The V-cycle in the sine eigenvectors of the x-lines is the same operator as the cycle with exact line
solves: a numpy restatement of the mode-space kernels' arithmetic (right-hand sides over the diagonals,
folded transforms, restrictions merged over five planes) from the set-up's own coefficients
(smg_setup_coefs), against the oracle's cycle over odd, even and degenerate sizes."""
import numpy as np
import pytest

from paper_1212_6680_gb300 import inputs


@pytest.fixture(scope="module")
def smg():
    from paper_1212_6680_gb300 import build

    build.build()
    from paper_1212_6680_gb300 import smg as m

    return m


def fold_matrices(n):
    h = (n + 1) // 2
    x = np.arange(1, h + 1)[:, None]
    s = lambda k: np.sqrt(2 / (n + 1)) * np.sin(np.pi * (x * k % (2 * (n + 1))) / (n + 1))  # noqa: E731
    return s(2 * np.arange(h) + 1), s(2 * np.arange(n // 2) + 2)


def to_modes(r, n):
    odd, even = fold_matrices(n)
    h, ne = (n + 1) // 2, n // 2
    a, m = r[..., :h], r[..., ::-1][..., :h]
    s = a + m
    if n % 2:
        s = s.copy()
        s[..., -1] = a[..., -1]
    return np.concatenate([s @ odd, (a - m)[..., :ne] @ even[:ne]], axis=-1)


def from_modes(f, n):
    odd, even = fold_matrices(n)
    h = (n + 1) // 2
    e, o = f[..., :h] @ odd.T, f[..., h:] @ even.T
    out = np.empty(f.shape)
    out[..., :h] = e + o
    out[..., ::-1][..., : n // 2] = (e - o)[..., : n // 2]
    return out


class Cycle:
    def __init__(self, smg, nx, ny, nz, npre, npost):
        self.npre, self.npost = npre, npost
        self.nx = nx
        lvl = lambda n: 1 if n == 1 else 1 + lvl(n // 2)  # noqa: E731
        self.L, self.P = lvl(nz), lvl(ny)
        k = np.arange(nx)
        h = (nx + 1) // 2
        kk = np.where(k < h, 2 * k + 1, 2 * (k - h) + 2)
        self.lam = 4 * np.sin(np.pi * kk / (2 * (nx + 1))) ** 2
        self.nz = [nz >> l for l in range(self.L)]
        self.zc = [[smg.smg_setup_coefs(nx, ny, nz, l, z, 0)[0] for z in range(self.nz[l])] for l in range(self.L)]
        self.lines = {(l, z, m): smg.smg_setup_coefs(nx, ny, nz, l, z, m)[1]
                      for l in range(self.L) for z in range(self.nz[l]) for m in range(self.P)}

    def at(self, c, s, t):
        return c[s] * self.lam + c[t]

    def ycycle(self, l, z, m, g):
        """g: right-hand sides over the diagonals."""
        c = self.lines[l, z, m]
        n = len(c)
        if n == 1:
            return g
        am = [self.at(c[y], 0, 3) / self.at(c[y], 1, 4) for y in range(n)]
        ap = [self.at(c[y], 2, 5) / self.at(c[y], 1, 4) for y in range(n)]
        nb = lambda u, y: (am[y] * u[y - 1] if y > 0 else 0.0) + (ap[y] * u[y + 1] if y + 1 < n else 0.0)  # noqa: E731
        u = [v.copy() for v in g]
        for y in range(1, n, 2):
            u[y] = g[y] - nb(g, y)
        d = self.lines[l, z, m + 1]
        gc = []
        for j in range(n // 2):
            o = 2 * j + 1
            w0, w1 = c[o - 1][7], (c[o + 1][6] if o + 1 < n else 0.0)
            v = -(w0 * self.at(c[o - 1], 2, 5) + (w1 * self.at(c[o + 1], 0, 3) if o + 1 < n else 0.0)) * u[o]
            if o - 2 >= 0:
                v = v - w0 * self.at(c[o - 1], 0, 3) * u[o - 2]
            if o + 2 < n:
                v = v - w1 * self.at(c[o + 1], 2, 5) * u[o + 2]
            gc.append(v / self.at(d[j], 1, 4))
        e = self.ycycle(l, z, m + 1, gc)
        v = [x.copy() for x in g]
        for y in range(0, n, 2):
            if y > 0:
                v[y] += c[y][6] * e[y // 2 - 1]
            if y + 1 < n:
                v[y] += c[y][7] * e[y // 2]
        for y in range(1, n, 2):
            v[y] = g[y] - nb(v, y)
        for y in range(0, n, 2):
            v[y] = g[y] - nb(v, y)
        return v

    def couple(self, u, M, K):
        d = 2 * u
        d[1:] -= u[:-1]
        d[:-1] -= u[1:]
        return K * u + M * (self.lam * u + d)

    def relax(self, l, f, u, colour, mode):
        n = self.nz[l]
        for z in range(colour, n, 2):
            c, g = self.zc[l][z], f[z].copy()
            if mode > 0:
                if z > 0:
                    g -= self.couple(u[z - 1], c[0], c[3])
                if z + 1 < n:
                    g -= self.couple(u[z + 1], c[2], c[5])
                if mode == 2:
                    g -= self.couple(u[z], c[1], c[4])
            line = self.lines[l, z, 0]
            v = np.stack(self.ycycle(l, z, 0, [g[y] / self.at(line[y], 1, 4) for y in range(len(line))]))
            u[z] = u[z] + v if mode == 2 else v

    def restrict(self, l, f, u):
        n, zc = self.nz[l], self.zc[l]
        out = []
        for Z in range(n // 2):
            o = 2 * Z + 1
            h1, h2 = o + 1 < n, o + 2 < n
            w0, w1 = zc[o - 1][7], (zc[o + 1][6] if h1 else 0.0)
            g = f[o] + w0 * f[o - 1] + (w1 * f[o + 1] if h1 else 0.0)
            get = lambda z, i: zc[z][i] if z < n else 0.0  # noqa: E731
            if Z > 0:
                g = g - self.couple(u[o - 2], w0 * zc[o - 1][0], w0 * zc[o - 1][3])
            g = g - self.couple(u[o - 1], zc[o][0] + w0 * zc[o - 1][1], zc[o][3] + w0 * zc[o - 1][4])
            g = g - self.couple(u[o], zc[o][1] + w0 * zc[o - 1][2] + w1 * get(o + 1, 0),
                                zc[o][4] + w0 * zc[o - 1][5] + w1 * get(o + 1, 3))
            if h1:
                g = g - self.couple(u[o + 1], zc[o][2] + w1 * zc[o + 1][1], zc[o][5] + w1 * zc[o + 1][4])
            if h2:
                g = g - self.couple(u[o + 2], w1 * zc[o + 1][2], w1 * zc[o + 1][5])
            out.append(g)
        return np.stack(out)

    def level(self, l, f):
        u = np.zeros_like(f)
        if l == self.L - 1:
            self.relax(l, f, u, 0, 0)
            return u
        for s in range(self.npre):
            self.relax(l, f, u, 0, 0 if s == 0 else 2)
            self.relax(l, f, u, 1, 1 if s == 0 else 2)
        e = self.level(l + 1, self.restrict(l, f, u))
        for z in range(self.nz[l]):
            if z % 2:
                u[z] += e[z // 2]
            else:
                if z > 0:
                    u[z] += self.zc[l][z][6] * e[z // 2 - 1]
                if z // 2 < len(e):
                    u[z] += self.zc[l][z][7] * e[z // 2]
        for _ in range(self.npost):
            self.relax(l, f, u, 1, 2)
            self.relax(l, f, u, 0, 2)
        return u

    def apply(self, r):
        return from_modes(self.level(0, to_modes(r, self.nx)), self.nx)


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 4), (7, 1, 5), (6, 5, 1), (9, 8, 7), (8, 16, 16), (13, 12, 10), (5, 33, 6),
                                   (16, 6, 21)])
@pytest.mark.parametrize("cycle", [(1, 0), (1, 1), (2, 2)])
def test_mode_space_cycle_is_the_line_solve_cycle(smg, orc, shape, cycle):
    nx, ny, nz = shape
    r = inputs.rhs(nx, ny, nz, seed=11)
    ref = orc.SMG(nx, ny, nz, *cycle).apply(r)
    s = Cycle(smg, nx, ny, nz, *cycle).apply(r)
    assert np.max(np.abs(s - ref)) <= 1e-12 * np.max(np.abs(ref))
