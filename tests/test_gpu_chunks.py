"""Level-0 sweeps and residuals where the z-marching kernels split the rows into
chunks of more than one row, the last one short (the wall-normal component has
n - 1 rows): same inputs and counters as the oracle, at the field tolerances of
the parity tests (1e-12 in FP64, 1e-5 in FP32)."""

import pytest
import torch

import selm_inputs
from oracle import gibbs, grid, philox
from tests.gpu_util import empty, from_dev, rel, round_like, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [("fp64", 96), ("fp64", 128), ("fp32", 80), ("fp32", 96)])
def test_level0_chunks(prec, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_2680_gb300 import selm as S
    dt, tol = (torch.float64, 1e-12) if prec == "fp64" else (torch.float32, 1e-5)
    m = S.SelmMG(dim=3, n=n, precision=0 if prec == "fp64" else 1, seed=11, instance=3)
    osys = grid.velocity_system(n, 3, levels=S.selm_mg_levels(m.h))
    v0 = round_like(selm_inputs.fields(osys.shapes(0), seed=1), dt)
    b0 = round_like(selm_inputs.fields(osys.shapes(0), seed=2), dt)
    v, b = to_dev(m.h, v0, dt), to_dev(m.h, b0, dt)
    bc = empty(m.h, dt, level=1)
    S.selm_mg_residual_restrict(m.h, 0, 0, v, b, bc)
    r = [x - a for x, a in zip(b0, osys.apply(0, v0))]
    assert rel(from_dev(m.h, bc, level=1), osys.restrict(0, r)) < tol
    S.selm_mg_smooth(m.h, 0, 0, v, b, sweep=1, cycle=7, noise=1)
    want = gibbs.sweep(osys, 0, [x.copy() for x in v0], b0, 1, philox.PhiloxNoise(11, 3, 7), 1.0)
    assert rel(from_dev(m.h, v), want) < tol
