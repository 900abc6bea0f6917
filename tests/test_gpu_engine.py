"""The coarse engine where its slabs, classes and buffers of normals come out
uneven: odd class extents, a last slab with fewer planes, normals that do not
fit beside the level (96^3 in FP32), CTA 0 alone with helpers drawing for it
(2-D in FP64).  One stochastic V-cycle against the oracle at the parity tests'
field tolerances (1e-12 in FP64, 1e-5 in FP32)."""

import pytest
import torch

import selm_inputs
from oracle import grid, multigrid, philox
from tests.gpu_util import comps, from_dev, rel, round_like, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,prec,mode", [(3, 40, "fp32", 0), (3, 40, "fp64", 0), (3, 72, "fp32", 0),
                                             (3, 96, "fp32", 0), (2, 96, "fp64", 0), (2, 160, "fp32", 0),
                                             (3, 24, "fp32", 1), (2, 48, "fp64", 1)])
def test_uneven_vcycle(dim, n, prec, mode):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_2680_gb300 import selm as S
    dt, tol = (torch.float64, 1e-12) if prec == "fp64" else (torch.float32, 1e-5)
    m = S.SelmMG(dim=dim, n=n, levels=3 if mode else 0, precision=0 if prec == "fp64" else 1, coarse_mode=mode,
                 seed=11, instance=3)
    assert S.selm_mg_engine_info(m.h)[0] >= 1
    osys = grid.velocity_system(n, dim, levels=S.selm_mg_levels(m.h))
    v0 = round_like(selm_inputs.fields(osys.shapes(0), seed=1), dt)
    b0 = round_like(selm_inputs.fields(osys.shapes(0), seed=2), dt)
    v, b = to_dev(m.h, v0, dt), to_dev(m.h, b0, dt)
    S.selm_mg_vcycle(m.h, 0, v, b, 7, 1)
    want = [x.copy() for x in v0]
    multigrid.vcycle(osys, 0, want, b0, philox.PhiloxNoise(11, 3, 7), 1.0,
                     coarse_mode="smooth" if mode else "cholesky")
    assert rel(from_dev(m.h, v), want) < tol


@pytest.mark.parametrize("noise", [0, 1])
def test_full_passes_keep_dataflow_values(noise):
    """Level 1 of 72^3 (144^3 grid): one launch per colour pass with the dataflow
    order's parity bits, against the plain per-pass form: every stored value
    within an ulp, so the V-cycles agree to the FP32 tolerance."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_2680_gb300 import selm as S
    m = S.SelmMG(dim=3, n=144, precision=1, seed=11, instance=3)
    b = torch.randn(comps(m.h, 0, 0)[1], device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    out = []
    for coop in (1, 0):
        S.selm_mg_set_option(m.h, S.SELM_OPT_LEVEL_COOP, coop)
        v = torch.zeros_like(b)
        S.selm_mg_vcycle(m.h, 0, v, b, 7, noise)
        out.append(v)
    assert ((out[0] - out[1]).norm() / out[1].norm()).item() < 1e-5
    assert not torch.equal(out[0], out[1])


@pytest.mark.parametrize("dim,n", [(3, 48), (3, 80), (2, 208), (2, 1024)])
@pytest.mark.parametrize("noise", [0, 1])
def test_row_pairs(dim, n, noise):
    """Both x colours of a row in one launch: rows of 3, 5, 13 and 64 segments (a
    block's last threads idle, the neighbour segment wraps), one sweep of level 1."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import gibbs
    from paper_1003_2680_gb300 import selm as S
    m = S.SelmMG(dim=dim, n=n, precision=1, seed=11, instance=3)
    osys = grid.velocity_system(n, dim, levels=S.selm_mg_levels(m.h))
    v0 = round_like(selm_inputs.fields(osys.shapes(1), seed=1), torch.float32)
    b0 = round_like(selm_inputs.fields(osys.shapes(1), seed=2), torch.float32)
    v, b = to_dev(m.h, v0, torch.float32, level=1), to_dev(m.h, b0, torch.float32, level=1)
    S.selm_mg_smooth(m.h, 0, 1, v, b, sweep=1, cycle=7, noise=noise)
    want = gibbs.sweep(osys, 1, [x.copy() for x in v0], b0, 1, philox.PhiloxNoise(11, 3, 7), float(noise))
    assert rel(from_dev(m.h, v, level=1), want) < 1e-5


@pytest.mark.parametrize("n", [768, 2048])
def test_2d_levels_by_launches(n):
    """2-D levels above the engine: launches of row pairs by default; the cooperative
    option set explicitly or off makes no difference to any value."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_2680_gb300 import selm as S
    m = S.SelmMG(dim=2, n=n, precision=1, seed=11, instance=3)
    assert S.selm_mg_engine_info(m.h)[0] >= 2
    b = torch.randn(comps(m.h, 0, 0)[1], device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    out = []
    for coop in (1, 0):
        S.selm_mg_set_option(m.h, S.SELM_OPT_LEVEL_COOP, coop)
        S.selm_mg_set_option(m.h, S.SELM_OPT_ENGINE_LEVEL, 2)
        v = torch.zeros_like(b)
        S.selm_mg_vcycle(m.h, 0, v, b, 7, 1)
        out.append(v)
    assert ((out[0] - out[1]).norm() / out[1].norm()).item() < 1e-5


@pytest.mark.parametrize("dim,n,prec", [(2, 32, "fp64"), (2, 32, "fp32"), (2, 64, "fp64"), (3, 48, "fp32")])
def test_normals_drawn_into_another_block(dim, n, prec):
    """The engine's normals reach the block that holds a level from the other blocks
    of its cluster: with no level divided over the cluster (2-D, 16^2 and below: the
    others are there to draw only) and beside levels that are.  Many launches one
    after another, each with its own counter, against the oracle."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_2680_gb300 import selm as S
    dt, tol = (torch.float64, 1e-12) if prec == "fp64" else (torch.float32, 1e-5)
    m = S.SelmMG(dim=dim, n=n, precision=0 if prec == "fp64" else 1, seed=11, instance=3)
    assert S.selm_mg_engine_info(m.h)[0] == 1
    osys = grid.velocity_system(n, dim, levels=S.selm_mg_levels(m.h))
    v0 = round_like(selm_inputs.fields(osys.shapes(0), seed=1), dt)
    b0 = round_like(selm_inputs.fields(osys.shapes(0), seed=2), dt)
    b = to_dev(m.h, b0, dt)
    out = []
    for cycle in range(64):
        v = to_dev(m.h, v0, dt)
        S.selm_mg_vcycle(m.h, 0, v, b, cycle, 1)
        out.append(v)
    for cycle in (0, 31, 63):
        want = [x.copy() for x in v0]
        multigrid.vcycle(osys, 0, want, b0, philox.PhiloxNoise(11, 3, cycle), 1.0)
        assert rel(from_dev(m.h, out[cycle]), want) < tol


@pytest.mark.parametrize("dim,n", [(2, 768), (2, 160), (3, 144)])
@pytest.mark.parametrize("noise", [0, 1])
def test_grid_barriers_on_request(dim, n, noise):
    """SELM_OPT_LEVEL_COOP = 2: level 1 as two cooperative launches, also where the
    default takes row-pair launches (as many launches as without the option, less the
    memory operations).  2-D levels admit no dataflow order, so there the default
    stores no parity bits and gives the cooperative form's values bit by bit; in 3-D
    it does, within the FP32 tolerance."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_2680_gb300 import selm as S
    m = S.SelmMG(dim=dim, n=n, precision=1, seed=11, instance=3)
    b = torch.randn(comps(m.h, 0, 0)[1], device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    out, launches = {}, {}
    for coop in (0, 1, 2):
        S.selm_mg_set_option(m.h, S.SELM_OPT_LEVEL_COOP, coop)
        S.selm_mg_set_option(m.h, S.SELM_OPT_ENGINE_LEVEL, 2)
        v = torch.zeros_like(b)
        before = S.selm_kernel_launches()
        S.selm_mg_vcycle(m.h, 0, v, b, 7, noise)
        launches[coop] = S.selm_kernel_launches() - before
        out[coop] = v
    # level 1: 6 class pairs (3-D; 3 in 2-D) x 4 sweeps, residual, restriction, prolongation, against 2
    assert launches[0] == launches[1] == launches[2] + (24 if dim == 3 else 12) + 1
    if dim == 2:
        assert torch.equal(out[1], out[2])
    assert ((out[1] - out[2]).norm() / out[2].norm()).item() < 1e-5


@pytest.mark.parametrize("dim,n", [(3, 80), (2, 512)])
def test_engine_level_on_request(dim, n):
    """SELM_OPT_ENGINE_LEVEL on an FP64 handle: the engine starts at the level asked
    for (40^3, 256^2: levels that the library's own choice leaves to cooperative
    launches), with the same V-cycle to 1e-12."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_2680_gb300 import selm as S
    m = S.SelmMG(dim=dim, n=n, precision=0, seed=11, instance=3)
    b = torch.randn(comps(m.h, 0, 0)[1], device="cuda", dtype=torch.float64,
                    generator=torch.Generator("cuda").manual_seed(5))
    assert S.selm_mg_engine_info(m.h)[0] == 2
    out = []
    for level in (0, 1):
        S.selm_mg_set_option(m.h, S.SELM_OPT_ENGINE_LEVEL, level)
        assert S.selm_mg_engine_info(m.h)[0] == (level or 2)
        v = torch.zeros_like(b)
        S.selm_mg_vcycle(m.h, 0, v, b, 7, 1)
        out.append(v)
    assert ((out[0] - out[1]).norm() / out[1].norm()).item() < 1e-12


@pytest.mark.parametrize("span,zeros", [(0, False), (20, False), (31, False), (40, False), (70, False), (20, True)])
def test_fixed_point_residual_rounding(span, zeros):
    """The FP32 outer residual's integer sum, bit by bit: every value of a window
    (4 sites of a row, their neighbours) becomes floor(z 2^(1080 - emax)), emax the
    window's largest exponent, whatever the spread of the exponents (up to 31 bits
    and beyond are separate code) and the signs.  b = s RN(sum), so any other
    rounding of a value leaves a residual: r = 0 exactly."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import math
    from fractions import Fraction

    import numpy as np
    from paper_1003_2680_gb300 import selm as S
    n = 8
    m = S.SelmMG(dim=3, n=n, precision=1, seed=11)
    lay, size = comps(m.h, 0, 0)
    rng = np.random.default_rng(span)
    z = rng.choice([-1.0, 1.0], size) * rng.uniform(0.5, 1.0, size) * 2.0 ** rng.integers(-span, 1, size)
    if zeros:
        z[rng.random(size) < 0.05] = 0.0
    r = torch.empty(size, dtype=torch.float32, device="cuda")
    probe = np.zeros(size)
    (nz, ny, nx), off = lay[0]
    centre = off + (3 * ny + 3) * nx + 3
    probe[centre] = 1.0
    S.selm_mg_outer_residual(m.h, 0, torch.tensor(probe, device="cuda"), torch.zeros(size, dtype=torch.float64, device="cuda"), r)
    s = -r[centre].item() / 6
    assert s > 0 and math.frexp(s)[0] == 0.5          # a power of two: s RN(sum) is exact
    b = np.zeros(size)
    for ci, ((nz, ny, nx), off) in enumerate(lay):
        f = z[off:off + nz * ny * nx].reshape(nz, ny, nx)
        g = b[off:off + nz * ny * nx].reshape(nz, ny, nx)
        for k in range(nz):
            dg = 6 + ((k == 0) + (k == nz - 1) if ci < 2 else 0)      # no-slip ghost on cell centres
            for j in range(ny):
                rows = [f[k, j - 1], f[k, (j + 1) % ny]] + ([f[k - 1, j]] if k > 0 else []) + ([f[k + 1, j]] if k + 1 < nz else [])
                for x0 in range(0, nx, 4):
                    own = f[k, j].take(range(x0 - 1, x0 + 5), mode="wrap")
                    win = np.concatenate([own] + [q[x0:x0 + 4] for q in rows])
                    emax = max(math.frexp(v)[1] for v in win if v != 0.0) + 1022    # biased exponent
                    fix = lambda v: math.floor(Fraction(v) * Fraction(2) ** (1080 - emax))
                    for e in range(4):
                        t = dg * fix(own[1 + e]) - fix(own[e]) - fix(own[2 + e]) - sum(fix(q[x0 + e]) for q in rows)
                        g[k, j, x0 + e] = s * float(Fraction(t) * Fraction(2) ** (emax - 1080))
    norm = torch.zeros(1, dtype=torch.float64, device="cuda")
    S.selm_mg_outer_residual(m.h, 0, torch.tensor(z, device="cuda"), torch.tensor(b, device="cuda"), r, norm)
    assert not r.any() and norm.item() == 0.0
