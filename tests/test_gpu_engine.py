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
