"""The FP64 operator's line contractions (csrc/nsk_fx.cuh) where the values of a line differ by many orders
of magnitude, where they are tiny, infinite or NaN, and on Gauss-Lobatto nodes.

Reference: the operator in extended precision (numpy.longdouble). Bound of a row, derived before any run: sums in
FP64 with W = N + 3 products make at most W + 2 roundings of 2^-53 (the last for mu), table entries are
within 4 more, a diagonal entry (formed from the others of its column) within 2 of the largest row sum R; the
fixed-point form is within 10 (W + 1) units of 2^-61 M R, M the line's largest value, and is used for a row only
while M is at most 2^4 times the largest value M_i that enters the row. So
  |error_i| <= (W + 6) 2^-53 (sum_j |a_ij x_j| + R |x_i|) + 10 (W + 1) 2^-57 M_i R,
with a value "entering" a row unless its entry is an exact zero of the FP64 operator (the R |x_i| term and x_i itself
only where the diagonal entry is not one).
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1912_12059_gb300 import inputs, nsk
from tolerances import rhs_tolerance

pytestmark = pytest.mark.gpu
L = np.longdouble
GAUSS, LOBATTO = nsk.NSK_NODES_GAUSS, nsk.NSK_NODES_GAUSS_LOBATTO


def _legendre(n, x):
    a, b = L(1), x
    for k in range(2, n + 1):
        a, b = b, ((2 * k - 1) * x * b - (k - 1) * a) / L(k)
    return b, a


def _operator(N, nt):
    """(T [np][np + 2] rows (l_i(-1) / (2 w_i), (w_j / w_i) l_i'(x_j), -l_i(1) / (2 w_i)), l [2][np], exact zeros [np][np + 2])."""
    n = N + 1
    x, w = np.zeros(n, L), np.zeros(n, L)
    for i in range(n):
        if nt == GAUSS:
            z = np.cos(L(np.pi) * (4 * (n - i) - 1) / (4 * n + 2))
            for _ in range(60):
                p, q = _legendre(n, z)
                z -= p * (1 - z * z) / (n * (q - z * p))
            p, q = _legendre(n, z)
            x[i], w[i] = z, 2 * (1 - z * z) / (n * q) ** 2
        else:
            z = -np.cos(L(np.pi) * i / N)
            if 0 < i < N:
                for _ in range(60):
                    p, q = _legendre(N, z)
                    d1 = N * (q - z * p) / (1 - z * z)
                    z -= d1 / ((2 * z * d1 - N * (N + 1) * p) / (1 - z * z))
            else:
                z = L(-1 if i == 0 else 1)
            p, _ = _legendre(N, z)
            x[i], w[i] = z, 2 / (N * (N + 1) * p * p)
    lam = [1 / np.prod([x[j] - x[m] for m in range(n) if m != j]) for j in range(n)]
    T, l = np.zeros((n, n + 2), L), np.zeros((2, n), L)
    for i in range(n):
        for j in range(n):
            if i != j:
                T[i, 1 + j] = w[j] / w[i] * (lam[i] / lam[j] / (x[j] - x[i]))  # l_i'(x_j)
        if nt == GAUSS:
            for s, x0 in enumerate((L(-1), L(1))):
                l[s, i] = lam[i] / (x0 - x[i]) / sum(lam[m] / (x0 - x[m]) for m in range(n))
        T[i, 1 + i] = -sum(lam[j] / lam[i] / (x[i] - x[j]) for j in range(n) if j != i)
    if nt == LOBATTO:
        l[0, 0] = l[1, N] = 1
    T[:, 0], T[:, n + 1] = l[0] / (2 * w), -l[1] / (2 * w)
    zero = np.zeros((n, n + 2), bool)
    if nt == LOBATTO:
        zero[1:, 0] = zero[:-1, n + 1] = True
    if N == 2:
        zero[1, 2] = True
    if nt == LOBATTO and N == 3:
        zero[1, 2] = zero[2, 3] = True
    T[zero] = 0
    return T, l, zero


def _rows(T, zero, g):
    """(exact sums, bounds) of the lines g [K][np + 2] with the operator T (metric and mu folded in)."""
    n = T.shape[0]
    x, W = g.astype(L), n + 2
    R = np.abs(T).sum(1).max()
    ex = x @ T.T
    A = np.abs(x) @ np.abs(T).T
    Mi = np.stack([np.abs(np.where(zero[i], 0, x)).max(1) for i in range(n)], axis=1)
    own = np.stack([np.zeros(len(g), L) if zero[i, 1 + i] else np.abs(x[:, 1 + i]) for i in range(n)], axis=1)
    return ex, L(2) ** -53 * (W + 6) * (A + R * own) + 10 * (W + 1) * L(2) ** -57 * Mi * R


def _solver(N, nt, mu=0.0173):
    s = nsk.Solver(2, (4, 2), N, node_type=nt)  # 2/h = 8 and 4
    s.set_params(mu=mu)
    return s


@pytest.mark.parametrize("nt", [GAUSS, LOBATTO])
@pytest.mark.parametrize("N", [2, 3, 4, 5])
@pytest.mark.parametrize("scale", [1.0, 1e-291, 3e250])
def test_graded_lines(gpu, N, nt, scale):
    T, l, zero = _operator(N, nt)
    g = np.random.Generator(np.random.PCG64(10 * N + nt))
    K, W = 4000, N + 3
    lines = g.uniform(0.5, 1.0, (K, W)) * g.choice((-1.0, 1.0), (K, W)) * 10.0 ** -g.uniform(0.0, 14.0, (K, W))
    lines[:500] = g.uniform(0.5, 1.0, (500, W)) * g.choice((-1.0, 1.0), (500, W))
    for i in range(500, 1000):  # one large value among small ones, zeros too
        lines[i] = 1e-9 * g.standard_normal(W) * (g.random(W) < 0.8)
        lines[i, g.integers(W)] = g.standard_normal()
    lines *= scale
    s = _solver(N, nt)
    for k, rh, mu in ((0, 8.0, False), (1, 4.0, False), (0, 8.0, True)):
        f = L(rh) * (L(0.0173) if mu else L(1))
        sums, ends = s._test_hook_lines(torch.from_numpy(lines).cuda(), k, mu)
        ex, tol = _rows(f * T, zero, lines)
        err = np.abs(sums.cpu().numpy().astype(L) - ex)
        assert (err <= tol + L(2) ** -1040).all(), (k, mu, float((err / (tol + L(2) ** -1040)).max()))
        x, e = lines[:, 1:-1], ends.cpu().numpy()
        if nt == LOBATTO:
            assert (e == x[:, [0, -1]]).all()
        else:
            xl, n = x.astype(L), N + 1
            bound = (np.abs(xl) @ np.abs(l).T * (n + 6) * L(2) ** -53
                     + 10 * (n + 1) * L(2) ** -61 * np.abs(xl).max(1)[:, None] * np.abs(l).sum(1).max() * 2)
            assert (np.abs(e.astype(L) - xl @ l.T) <= bound + L(2) ** -1040).all()
    s.close()


@pytest.mark.parametrize("nt", [GAUSS, LOBATTO])
@pytest.mark.parametrize("N", [2, 3, 4, 5])
def test_lines_with_an_infinity_or_nan(gpu, N, nt):
    """As FP64 sums give them: an infinity times every entry that is not zero, NaN everywhere."""
    T, l, zero = _operator(N, nt)
    n, W = N + 1, N + 3
    g = np.random.Generator(np.random.PCG64(N))
    lines = np.repeat(g.uniform(0.5, 1.0, (1, W)), 2 * W, axis=0)
    for j in range(W):
        lines[j, j], lines[W + j, j] = -np.inf, np.nan
    s = _solver(N, nt)
    sums, ends = (t.cpu().numpy() for t in s._test_hook_lines(torch.from_numpy(lines).cuda()))
    big = np.abs(T) > 1e-6
    for j in range(W):
        for i in range(n):
            assert np.isnan(sums[W + j, i])
            if big[i, j]:
                assert sums[j, i] == -np.sign(float(T[i, j])) * np.inf
            else:
                assert not np.isfinite(sums[j, i])
        if 1 <= j <= n:
            if nt == LOBATTO:
                assert np.array_equal(ends[[j, W + j]], lines[[j, W + j]][:, [1, n]], equal_nan=True)
            else:
                assert (ends[j] == -np.sign(l[:, j - 1].astype(float)) * np.inf).all() and np.isnan(ends[W + j]).all()
    s.close()


@pytest.mark.parametrize("dim,N", [(2, 2), (2, 3), (2, 4), (2, 5), (3, 2), (3, 3), (3, 4), (3, 5)])
def test_fluid_at_rest_beside_a_moving_one(gpu, dim, N):
    """Gauss-Lobatto: the density residual at the interior nodes of an element whose momentum is 1e-10 of its
    neighbours' is formed from its own values alone, to their precision."""
    ne, n = (4,) * dim, N + 1
    E, npe = 4**dim, n**dim
    s = nsk.Solver(dim, ne, N, node_type=LOBATTO)
    s.set_params()
    T, _, zero = _operator(N, LOBATTO)
    g = np.random.Generator(np.random.PCG64(dim * 10 + N))
    U = np.ones((dim + 2, E, npe))
    e0 = sum(1 * 4**k for k in range(dim))  # element (1, 1(, 1))
    for k in range(dim):
        U[1 + k] = g.uniform(0.1, 0.3, (E, npe))
        U[1 + k, e0] = 1e-10 * g.standard_normal(npe)
    s.set_state(U)
    R = s.rhs()[0, e0].reshape((n,) * dim)
    ex, tol = np.zeros((n,) * dim, L), np.zeros((n,) * dim, L)
    for k in range(dim):
        ax = dim - 1 - k
        m = np.moveaxis(U[1 + k, e0].reshape((n,) * dim), ax, -1)
        lines = np.zeros((m.size // n, n + 2))
        lines[:, 1:-1] = m.reshape(-1, n)  # face values enter no interior row
        a, b = _rows(8 * T, zero, lines)
        ex += np.moveaxis(a.reshape(m.shape), -1, ax)
        tol += np.moveaxis(b.reshape(m.shape), -1, ax)
    inside = (slice(1, -1),) * dim
    err = np.abs(R.astype(L) - ex)[inside]
    assert (err <= tol[inside]).all(), float((err / tol[inside]).max())
    s.close()


@pytest.mark.parametrize("dim,ne,N", [(2, (6, 5), 3), (2, (4, 7), 4), (2, (5, 3), 5), (3, (5, 3, 3), 3), (3, (3, 3, 2), 4),
                                      (3, (2, 3, 2), 5)])
@pytest.mark.parametrize("flux", [nsk.NSK_FLUX_LF, nsk.NSK_FLUX_HLLC])
def test_lobatto_residual_parity(gpu, dim, ne, N, flux):
    prm = dict(T=0.85, kappa=1e-3, alpha=1e3, beta=1e-3, mu=2e-2)
    hi = [1.0, 0.8, 1.3][:dim]
    s = nsk.Solver(dim, ne, N, [0.0] * dim, hi, LOBATTO, nsk.NSK_FP64)
    s.set_params(**prm)
    s.set_flux(flux)
    o = O.Oracle(dim, ne, (0.0,) * dim, tuple(hi), N, O.NODES_LOBATTO, flux=flux, **prm)
    U = inputs.random_state(o.shape, seed=60 + 10 * dim + N)
    s.set_state(U)
    Qg, Qo = s.lift(), o.lift(U)
    for c in range(o.nq):
        assert np.abs(Qg[c] - Qo[c]).max() <= 1e-12 * (np.abs(Qo[c]).max() + 1e-3 * np.abs(Qo).max()), c
    Rg, Ro = s.rhs(), o.rhs(U)
    tol = rhs_tolerance(o, U, Ro)
    for v in range(o.nvar):
        err = np.abs(Rg[v] - Ro[v]).max()
        assert err <= tol[v], (v, err, tol[v])
    s.close()
