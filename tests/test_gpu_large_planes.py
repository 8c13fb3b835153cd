"""Planes of 2^32 nodes, whose offsets do not fit 32 bits: a 2-D field is one
plane.  The transform is a tensor product of 1-D operators, so the result for a
sum of outer products a b^T is a sum of outer products of O(n) vectors, formed
here in binary64 and compared at every node of the finest level."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

N = 65537                       # N * N = 2^32 + 2^17 + 1: only the last two rows lie past 2^32
TOL = 1e-5                      # the parity bar of this path in binary32


def levels(n):
    """Fine node coordinates of every level, finest first."""
    x = [np.arange(n, dtype=np.float64)]
    while x[-1].size > 2:
        m = x[-1].size
        x.append(x[-1][np.append(np.arange(0, m - 1, 2), m - 1)])
    return x


class Ops:
    """1-D operators of one level (fine coordinates x)."""

    def __init__(self, x):
        m = x.size
        self.kept = np.append(np.arange(0, m - 1, 2), m - 1)
        self.new = np.setdiff1d(np.arange(m), self.kept)
        h = x[self.new + 1] - x[self.new - 1]
        self.wl, self.wr = (x[self.new + 1] - x[self.new]) / h, (x[self.new] - x[self.new - 1]) / h
        self.fine, self.coarse = self.bands(x), self.bands(x[self.kept])

    @staticmethod
    def bands(x):
        h = np.diff(x)
        return (np.append(h, 0.0) + np.append(0.0, h)) / 3.0, h / 6.0

    def restrict(self, v):                       # P^T
        full = v.copy()
        np.add.at(full, self.new - 1, self.wl * v[self.new])
        np.add.at(full, self.new + 1, self.wr * v[self.new])
        return full[self.kept]

    def prolong(self, c):                        # P
        v = self.inject(c)
        v[self.new] = self.wl * v[self.new - 1] + self.wr * v[self.new + 1]
        return v

    def mass(self, v):                           # M
        d, o = self.fine
        r = d * v
        r[1:] += o * v[:-1]
        r[:-1] += o * v[1:]
        return r

    def prolong_mass(self, c):                   # M P
        return self.mass(self.prolong(c))

    def project(self, v):                        # the coarse values of a decomposition
        return self.solve(self.restrict(self.mass(v)))

    def solve(self, b):                          # the coarse mass matrix
        from scipy.linalg import solveh_banded
        d, o = self.coarse
        return solveh_banded(np.stack([d, np.append(o, 0.0)]), b, lower=True)

    def inject(self, c):                         # coarse values at the kept nodes
        v = np.zeros(self.kept.size + self.new.size)
        v[self.kept] = c
        return v


def outer(terms, rows, cols=slice(None)):
    """sum of c a b^T over (c, a, b) at the rows and columns, on the GPU"""
    out = 0
    for c, a, b in terms:
        out = out + c * torch.outer(torch.from_numpy(a[rows]).cuda(), torch.from_numpy(b[cols]).cuda())
    return out


def recompose_adjoint_terms(a, b, ops):
    """Coefficient gradient of the finest level (terms, at its new nodes) of the gradient a b^T."""
    ya, yb = (ops.prolong_mass(ops.solve(ops.restrict(v))) for v in (a, b))
    return [(1.0, a, b), (-1.0, ya, yb)]


def decompose_adjoint_terms(a, b, s, t, ops, below):
    """Field gradient of the coefficient gradients a b^T at the new nodes of the
    finest level and s t^T at those of the level below: terms at the new nodes of
    the finest level, and at its kept nodes (coarse vectors)."""
    gv = [(1.0, s, t), (-1.0, below.inject(below.restrict(s)), below.inject(below.restrict(t)))]
    h = [(1.0, a, b)] + [(c, *(ops.prolong_mass(ops.solve(v)) for v in p)) for c, *p in gv]
    kept = list(gv)
    for c, x, y in h:
        kept += [(-c, ops.restrict(x), ops.restrict(y)), (c, x[ops.kept], y[ops.kept])]
    return h, kept


def split(stream, n):
    """The finest level's section of a coefficient stream of an n x n field (n
    odd), as rows: the kept ones' new nodes with the new row after each, and the
    last kept row's."""
    mc, pairs = (n + 1) // 2, (n - 1) // 2
    s = stream[mc * mc:]
    body = s[:pairs * (2 * n - mc)].view(pairs, 2 * n - mc)
    return body[:, :n - mc], body[:, n - mc:], s[pairs * (2 * n - mc):]


def check_section(stream, terms, n, step=2048):
    kept, new, last = split(stream, n)
    ops_new, scale, err = slice(1, None, 2), 0.0, 0.0
    for r in range(0, new.shape[0], step):
        e = min(r + step, new.shape[0])
        for got, rows, cols in ((kept, slice(2 * r, 2 * e, 2), ops_new), (new, slice(2 * r + 1, 2 * e, 2), slice(None))):
            ref = outer(terms, rows, cols)
            scale = max(scale, ref.abs().max().item())
            err = max(err, (got[r:e] - ref).abs().max().item())
    ref = outer(terms, slice(n - 1, n), ops_new)[0]
    scale = max(scale, ref.abs().max().item())
    err = max(err, (last - ref).abs().max().item())
    assert err <= TOL * scale, (err, scale)


def vectors(n, seed, count):
    rng = np.random.default_rng(seed)
    return [rng.standard_normal(n).astype(np.float32).astype(np.float64) for _ in range(count)]


def product(a, b, out):
    """out[i, j] = a[i] b[j] in binary32"""
    x, y = (torch.from_numpy(v).cuda().float() for v in (a, b))
    return torch.mul(x[:, None], y[None, :], out=out)


@pytest.mark.parametrize("n", [129, N])
def test_adjoints(n):
    from paper_2503_06322_gb300 import hpdr as H
    x = levels(n)
    ops, below = Ops(x[0]), Ops(x[1])
    g = torch.empty(n, n, dtype=torch.float32, device="cuda")
    out = torch.empty(n * n, dtype=torch.float32, device="cuda")
    a, b = vectors(n, 1, 2)
    H.hpdr_recompose_adjoint(product(a, b, g), out=out)
    check_section(out, recompose_adjoint_terms(a, b, ops), n)

    # coefficients of the two finest levels; the others are zero
    s, t = vectors((n + 1) // 2, 2, 2)
    out.zero_()
    for m, (p, q) in ((n, (a, b)), ((n + 1) // 2, (s, t))):
        kept, new, last = split(out[:m * m], m)
        P, Q = (torch.from_numpy(v).cuda().float() for v in (p, q))
        torch.mul(P[:-1:2, None], Q[None, 1::2], out=kept)
        torch.mul(P[1::2, None], Q[None, :], out=new)
        last.copy_(P[-1] * Q[1::2])
    H.hpdr_decompose_adjoint(out, (n, n), out=g)
    h, k = decompose_adjoint_terms(a, b, s, t, ops, below)
    scale = err = 0.0
    for r in range(0, n, 2048):
        e = min(r + 2048, n)
        ref = outer(h, slice(r, e))
        ref[::2, ::2] = outer(k, slice(r // 2, (e + 1) // 2))
        scale = max(scale, ref.abs().max().item())
        err = max(err, (g[r:e] - ref).abs().max().item())
    assert err <= TOL * scale, (err, scale)


@pytest.mark.parametrize("n", [129, N])
def test_transforms(n):
    from paper_2503_06322_gb300 import hpdr as H
    x = levels(n)
    a, b = vectors(n, 3, 2)
    u = product(a, b, torch.empty(n, n, dtype=torch.float32, device="cuda"))
    coef = H.hpdr_decompose(u)
    m, p, q = n, a, b
    for grid in x[:2]:
        ops = Ops(grid)
        check_section(coef[:m * m], [(1.0, p, q), (-1.0, ops.prolong(p[ops.kept]), ops.prolong(q[ops.kept]))], m)
        m, p, q = (m + 1) // 2, ops.project(p), ops.project(q)
    back = H.hpdr_recompose(coef, (n, n))
    del coef
    err = max((back[r:r + 4096] - u[r:r + 4096]).abs().max().item() for r in range(0, n, 4096))
    assert err <= TOL * np.abs(a).max() * np.abs(b).max()


@pytest.mark.parametrize("n", [129, N])
def test_containers(n):
    from paper_2503_06322_gb300 import hpdr as H
    a, b = vectors(n, 4, 2)
    u = product(a, b, torch.empty(n, n, dtype=torch.float32, device="cuda"))
    buf = H.hpdr_compress(u, 1e-2)
    back = H.hpdr_decompress(buf)
    del buf
    err = max((back[r:r + 4096].double() - u[r:r + 4096]).abs().max().item() for r in range(0, n, 4096))
    del back
    torch.cuda.empty_cache()
    assert err <= 1e-2 * u.abs().max().item()
