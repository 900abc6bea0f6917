"""The spectral solves behind the staggered composite grid's projection and the
exact Stokes velocity: every split of rows between the fine and the base part
(none, one, all but one, all refined), the grid beside them that is not a power
of two (diagonal preconditioner, FAC), and right-hand sides that are rounding."""

import numpy as np
import pytest
import torch

from oracle.composite_mac import CompositeMAC

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_2680_gb300 import selm as mod
    return mod


@pytest.mark.parametrize("n,K", [(4, 0), (4, 1), (4, 4), (8, 7), (16, 3), (12, 4)])
@pytest.mark.parametrize("adjoint", [0, 1])
def test_projection(S, n, K, adjoint):
    """P~ u (or W P~ W^-1 u) against the oracle's direct solve at 1e-11: the
    pressure to a relative residual of 1e-14, times the operator's condition (a
    few hundred at these sizes).  Projecting the result again moves it by
    rounding only, and a zero field stays zero."""
    g = CompositeMAC(n, K, 3)
    h = S.selm_mac_create(S.make_mac_desc(3, n, K, projection=1, proj_tol=1e-14))
    u = np.random.default_rng(n + K).standard_normal(g.n_faces)
    want = g.weight * g.project(u / g.weight) if adjoint else g.project(u)
    ud = torch.tensor(u, device="cuda")
    out = torch.empty_like(ud)
    S.selm_mac_project(h, ud, out, adjoint=bool(adjoint))
    got = out.cpu().numpy()
    assert np.linalg.norm(got - want) <= 1e-11 * np.linalg.norm(want)
    again = torch.empty_like(out)
    S.selm_mac_project(h, out, again, adjoint=bool(adjoint))
    assert ((again - out).norm() / out.norm()).item() <= 1e-11
    zero = torch.zeros_like(ud)
    assert S.selm_mac_project(h, zero, out, adjoint=bool(adjoint)) == (0, 0.0)
    assert not out.any()
    S.selm_mac_destroy(h)


@pytest.mark.parametrize("n", [4, 16, 32, 24])
def test_stokes_velocity(S, n):
    """The Stokes velocity of an FP32 handle (spectral, except at 24) against the
    FP64 handle's FAC solves, both to 1e-11: 1e-9, the tolerance over the Schur
    complement's smallest eigenvalue."""
    us = []
    for prec in (0, 1):
        h = S.selm_mg_create(S.make_desc(dim=3, n=n, mu=0.9, precision=prec, tol=1e-11))
        size = S.selm_mg_layout(h, 0, 0, 0)[2]
        f = torch.tensor(np.random.default_rng(n).standard_normal(size), device="cuda")
        u = torch.empty_like(f)
        iters, res = S.selm_mg_stokes_solve(h, f, u)
        assert res <= 1e-11
        us.append(u)
        torch.cuda.synchronize()
        S.selm_mg_destroy(h)
    assert ((us[0] - us[1]).norm() / us[0].norm()).item() <= 1e-9


def test_projection_past_the_spectral_range(S):
    """A field whose divergence has r.r within FP64 but r.S^-1 r beyond it: the
    spectral preconditioner breaks down, and the projection falls back to the
    diagonal one instead of returning what came out.  u = G phi + w with w free of
    divergence, phi one mode along z (S^-1 of which is the largest): P~ u = w, to
    proj_tol times the condition number (a few thousand)."""
    n, K = 32, 8
    h = S.selm_mac_create(S.make_mac_desc(3, n, K, projection=1))
    nf, nc, fine = S.selm_mac_faces(h), S.selm_mac_cells(h), 2 * K * (2 * n) ** 2
    z = torch.cat([(torch.arange(2 * K, device="cuda", dtype=torch.float64).repeat_interleave(4 * n * n) + 0.5) / (2 * n),
                   (torch.arange(K, n, device="cuda", dtype=torch.float64).repeat_interleave(n * n) + 0.5) / n])
    vol = torch.full((nc,), 1.0 / n ** 3, dtype=torch.float64, device="cuda")
    vol[:fine] /= 8
    g, w, div = (torch.empty(k, dtype=torch.float64, device="cuda") for k in (nf, nf, nc))
    S.selm_mac_gradient(h, torch.cos(torch.pi * z), g)
    S.selm_mac_project(h, torch.tensor(np.random.default_rng(3).standard_normal(nf), device="cuda"), w)
    S.selm_mac_divergence(h, g + w, div)
    rr = ((vol * div) ** 2).sum().item()
    scale = 2.0 ** np.floor(0.5 * (np.log2(4e305) - np.log2(rr)))
    out = torch.empty_like(w)
    iters, res = S.selm_mac_project(h, (g + w) * scale, out)
    assert iters > 16 and res <= 1e-13
    assert ((out / scale - w).norm() / w.norm()).item() <= 1e-9
    S.selm_mac_destroy(h)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,K", [(4, 2), (16, 3), (32, 0), (32, 9), (32, 32), (64, 0), (64, 8), (64, 64)])
def test_projection_iterations(S, n, K, prec):
    """The spectral solve preconditions conjugate gradients, which would hide a wrong
    one behind more iterations or the diagonal fallback.  It is the operator's
    inverse to about five digits (FP32), so 1e-12 takes at most 4 iterations: all
    splits of rows, one to four rows per lane of the constant mode's scan and two
    blocks of columns per row (n = 64).  The result is free of divergence to the
    tolerance and is its own projection."""
    h = S.selm_mac_create(S.make_mac_desc(3, n, K, projection=1, proj_tol=1e-12, precision=prec))
    nf, nc, fine = S.selm_mac_faces(h), S.selm_mac_cells(h), 2 * K * (2 * n) ** 2
    u = torch.tensor(np.random.default_rng(n + K).standard_normal(nf), device="cuda")
    out, again = torch.empty_like(u), torch.empty_like(u)
    div = torch.empty((2, nc), dtype=torch.float64, device="cuda")
    iters, res = S.selm_mac_project(h, u, out)
    assert iters <= 4 and res <= 1e-12
    S.selm_mac_divergence(h, u, div[0])
    S.selm_mac_divergence(h, out, div[1])
    div[:, :fine] /= 8                                      # times the cells' volumes, as the solve measures it
    assert (div[1].norm() / div[0].norm()).item() <= 1e-11
    S.selm_mac_project(h, out, again)
    assert ((again - out).norm() / out.norm()).item() <= 1e-10
    S.selm_mac_destroy(h)


@pytest.mark.parametrize("n", [64, 128])
def test_stokes_velocity_of_large_grids(S, n):
    """test_stokes_velocity's comparison up to the largest grid of the spectral solve
    (FP64 handle: FAC), to 1e-9 from solves to 1e-11."""
    us = []
    for prec in (0, 1):
        h = S.selm_mg_create(S.make_desc(dim=3, n=n, mu=0.9, precision=prec, tol=1e-11))
        f = torch.tensor(np.random.default_rng(n).standard_normal(S.selm_mg_layout(h, 0, 0, 0)[2]), device="cuda")
        u = torch.empty_like(f)
        assert S.selm_mg_stokes_solve(h, f, u)[1] <= 1e-11
        us.append(u)
        torch.cuda.synchronize()
        S.selm_mg_destroy(h)
    assert ((us[0] - us[1]).norm() / us[0].norm()).item() <= 1e-9


@pytest.mark.parametrize("n,K", [(8, 3), (16, 5), (32, 0), (32, 9)])
def test_projection_error(S, n, K):
    """The default tolerance (1e-13) on a white field against a solve to 1e-17: 1e-14,
    three times the residual of 1e-13 / 32 at which the spectral iteration stops
    (error over residual: 1.3 on such fields)."""
    out = []
    for tol in (0.0, 1e-17):
        h = S.selm_mac_create(S.make_mac_desc(3, n, K, projection=1, proj_tol=tol))
        u = torch.tensor(np.random.default_rng(1).standard_normal(S.selm_mac_faces(h)), device="cuda")
        out.append(torch.empty_like(u))
        S.selm_mac_project(h, u, out[-1])
        torch.cuda.synchronize()
        S.selm_mac_destroy(h)
    assert ((out[0] - out[1]).norm() / out[1].norm()).item() <= 1e-14
