"""Sizes at which the kernels' rules and tiles have their edges: the FP64 integer contractions on
meshes of one or a few elements, the FP32 line sums, the training kernels' column slices and ragged
row tiles, and the limit of the implicit integrator's small-system kernels.
"""
import numpy as np
import pytest

import oracle as O
from oracle import esdirk as ES
from oracle import mlp as omlp
from paper_1912_12059_gb300 import inputs, nsk
from tolerances import rhs_tolerance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,ne,N", [(2, (1, 1), 2), (2, (1, 1), 5), (2, (33, 1), 3), (2, (1, 6), 4), (3, (1, 1, 1), 3),
                                      (3, (1, 2, 1), 2), (3, (2, 1, 3), 4), (3, (7, 1, 1), 5)])
@pytest.mark.parametrize("mu", [0.0, 2e-2])
def test_integer_contractions_on_few_elements(gpu, dim, ne, N, mu):
    """Residual parity where an element is its own neighbour and groups of elements are partly
    empty, with and without viscosity, on boxes with sides of a ratio of up to 60."""
    prm = dict(T=0.85, kappa=1e-3, alpha=1e3, beta=1e-3, mu=mu)
    hi = [3.0, 0.05, 1.3][:dim]
    s = nsk.Solver(dim, ne, N, [0.0] * dim, hi, 0, nsk.NSK_FP64)
    s.set_params(**prm)
    o = O.Oracle(dim, ne, (0.0,) * dim, tuple(hi), N, O.NODES_GAUSS, **prm)
    U = inputs.random_state(o.shape, seed=10 * dim + N)
    s.set_state(U)
    Rg, Ro = s.rhs(), o.rhs(U)
    tol = rhs_tolerance(o, U, Ro)
    for v in range(o.nvar):
        err = np.abs(Rg[v] - Ro[v]).max()
        assert err <= tol[v], (v, err, tol[v])
    s.close()


@pytest.mark.parametrize("tpb", [128, 256])
@pytest.mark.parametrize("ne,N", [((1, 1, 1), 4), ((3, 1, 1), 4), ((5, 3, 1), 4), ((1, 2, 1), 5), ((3, 1, 3), 5),
                                  ((3, 1, 3), 2)])
def test_fp32_line_sums_on_few_elements(gpu, tpb, ne, N):
    """FP32 lines of 5 and 6 nodes (and 3, on the other side of the rule), groups of one and two elements
    with a remainder: residual and gradients within the FP64 tests' bounds in FP32's units in the last
    place (2^-23 for 2^-52)."""
    prm = dict(T=0.85, kappa=1e-3, alpha=1e3, beta=1e-3, mu=2e-2)
    hi = [1.0, 0.8, 1.3]
    s = nsk.Solver(3, ne, N, [0.0] * 3, hi, 0, nsk.NSK_FP32_MIXED)
    s.set_params(**prm)
    s.set_schedule(tpb, 0)
    o = O.Oracle(3, ne, (0.0,) * 3, tuple(hi), N, O.NODES_GAUSS, **prm)
    U = inputs.random_state(o.shape, seed=40 + N).astype(np.float32).astype(np.float64)
    s.set_state(U)
    Qg, Qo = s.lift(), o.lift(U)
    for c in range(o.nq):
        scale = np.abs(Qo[c]).max() + 1e-3 * np.abs(Qo).max()
        assert np.abs(Qg[c] - Qo[c]).max() <= 2.0**29 * 1e-12 * scale, c
    Rg, Ro = s.rhs(), o.rhs(U)
    tol = rhs_tolerance(o, U, Ro)
    for v in range(o.nvar):
        err = np.abs(Rg[v] - Ro[v]).max()
        assert err <= 2.0**29 * tol[v], (v, err, tol[v])
    s.close()


@pytest.mark.parametrize("n_in,h1,h2,n_out,B", [(16, 16, 16, 16, 16), (33, 80, 48, 48, 144), (70, 208, 112, 96, 272),
                                                (250, 256, 16, 64, 400), (40, 96, 256, 256, 1040)])
def test_training_gradients_at_tile_edges(gpu, n_in, h1, h2, n_out, B):
    """Widths in slices of 64, 32 and 16 columns, rows that leave a ragged last tile. The activations
    and their gradients are rounded to BF16 (2^-9 each) at most five times along a path: 5 x 2^-9
    = 1e-2 of a sum's terms, and 4e-2 where terms cancel to a quarter of their size."""
    import torch

    m = nsk.MLP(n_in, h1, h2, n_out, max_batch=B, max_rows=B)
    m.init_params(seed=5)
    p = omlp.unflatten(m.get_params().astype(np.float64), m.n_in_pad, h1, h2, n_out)
    for k in ("W1", "W2", "W3"):
        p[k] = torch.from_numpy(p[k].astype(np.float32)).to(torch.bfloat16).double().numpy()
    rng = np.random.default_rng(6)
    Xn = np.zeros((B, m.n_in_pad))
    Xn[:, :n_in] = rng.uniform(-1, 1, size=(B, n_in))
    Xt = torch.from_numpy(Xn).to(torch.bfloat16)
    Tn = rng.normal(size=(B, n_out))
    g_gpu, loss = m.gradients(Xt.to(gpu), torch.from_numpy(Tn).float().to(gpu))
    L_ref, g_ref = omlp.loss_and_grad(p, Xt.double().numpy(), Tn)
    assert abs(loss - L_ref) <= 1e-2 * L_ref
    gg = m.unflatten(g_gpu.astype(np.float64))
    for k in ("W1", "b1", "W2", "b2", "W3", "b3"):
        a, b = gg[k], g_ref[k]
        if k == "W1":
            assert np.abs(a[:, n_in:]).max(initial=0.0) == 0.0
            a, b = a[:, :n_in], b[:, :n_in]
        assert np.linalg.norm(a - b) <= 4e-2 * np.linalg.norm(b), k
    m.close()


@pytest.mark.parametrize("E,krylov_dim,precond", [(341, 30, False), (342, 30, False), (24, 3, False), (24, 5, True),
                                                  (24, 1, True), (31, 64, True), (9, 30, False)])
def test_implicit_step_around_the_small_system_limit(gpu, E, krylov_dim, precond):
    """341 elements of 12 unknowns are the largest mesh of the small-system kernels (4092 of 4096
    unknowns) and 342 the first beyond; Krylov dimensions below, off and above the captured four
    steps, with restarts. Both sides solve to the same Newton tolerance: 1e-8 as in the other parity
    tests."""
    prm = dict(T=0.85, kappa=1e-4, alpha=100.0, beta=1e-2, mu=1e-2)
    s = nsk.Solver(1, (E,), 3, [0.0], [1.0], 0, nsk.NSK_FP64)
    s.set_params(**prm)
    o = O.Oracle(1, (E,), (0.0,), (1.0,), 3, O.NODES_GAUSS, **prm)
    rv, rl, _ = O.maxwell(0.85)
    U = inputs.slab_1d(o.coords(), rv, rl, 1e-4)
    dt = 5.0 * o.timestep(U, 0.5)
    s.set_state(U)
    st = s.step_esdirk(dt, 1, newton_tol=1e-11, krylov_tol=1e-8, krylov_dim=krylov_dim, block_precond=precond)
    Ug = s.get_state()
    Uo, sto = ES.step(o.rhs, U, dt, newton_tol=1e-11, krylov_tol=1e-8, m=krylov_dim, nelem=(E,) if precond else None)
    assert st["failed"] == 0 and sto["failed"] == 0
    for v in range(o.nvar):
        assert np.abs(Ug[v] - Uo[v]).max() <= 1e-8 * np.abs(Uo[v]).max() + 1e-12, v
    s.close()
