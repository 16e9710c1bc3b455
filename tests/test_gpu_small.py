"""Transforms of 16 ... 256 points with four values per thread (radix 4, closing
radix 2), in every kernel that runs them: the column schedules of the general and
the zero-rim path, the nest kernels, the potential; whole grids against the oracle
within the bounds of tests/_gpu.py."""
import numpy as np
import pytest

import oracle
from paper_1603_03142_gb300 import workloads as W
from tests._gpu import rel_linf_levels, run_gpu, sgf, tol, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    return sgf()


@pytest.mark.parametrize("n", [16, 32, 64, 128])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_small_general_and_nest(lib, n, prec):
    levels = 3 if n <= 64 else 2
    nest = W.Nest(n=n, levels=levels, off=[(0, 0), (n // 4 + 1, n // 2), (n // 8, 3)][:levels])
    sigma = W.dn_density(nest, 2, 0.9)
    ox, oy = oracle.force(nest, sigma)
    plan = lib.Plan(nest, prec)
    for inv, c3 in ((0, 0), (1, 1), (2, 0)):
        plan.set_schedule(0, inv, c3)
        gx, gy = run_gpu(plan, sigma)
        assert max(rel_linf_levels(nest, gx, gy, ox, oy)) <= tol(prec, n), (inv, c3)
    dt = torch.float64 if prec == "fp64" else torch.float32
    phi = lib.Plan(nest, prec, potential=True).solve_potential(
        [torch.from_numpy(s).to(device="cuda", dtype=dt) for s in sigma])
    ref = oracle.potential(nest, sigma)
    for l in range(levels):
        keep = ~nest.covered_mask(l)
        d = np.abs(phi[l].double().cpu().numpy() - ref[l])[keep].max()
        assert d <= tol(prec, n) * np.abs(ref[l][keep]).max()


@pytest.mark.parametrize("n", [16, 64, 128, 256])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_small_zero_rim(lib, n, prec):
    nest = W.Nest(n=n)
    s = W.dn_density(nest, 2, 0.85)[0]
    s[:2], s[-2:], s[:, :2], s[:, -2:] = 0, 0, 0, 0
    plan = lib.Plan(nest, prec, zero_rim=True)
    if n <= 128:
        ox, oy = oracle.force(nest, [s])
        rows = slice(None)
    else:
        rows = n // 2
        ox, oy = ([np.asarray(v)[None]] for v in oracle.force_row(nest, [s], rows))
    for col in (0, 1, 2):
        for inv in (0, 1, 2):
            plan.set_schedule(col, inv)
            gx, gy = run_gpu(plan, [s])
            plan.check()
            scale = max(np.abs(ox[0]).max(), np.abs(oy[0]).max())
            d = max(np.abs(gx[0][rows] - ox[0]).max(), np.abs(gy[0][rows] - oy[0]).max())
            assert d <= tol(prec, n) * scale, (col, inv, d / scale)
