"""The M-apply on layer grids of every size and depth: tiles that are the whole layer, tiles
with halos that wrap, few and many levels, layers finer and coarser than the apertures."""
import numpy as np
import pytest

import oracle as O
import synth
from tests.gpu_common import TOL_OP, assert_close, to_dev, to_np

pytestmark = pytest.mark.gpu

# (grid side, wavelet levels, grid spacing [m]) of the three layers; apertures are 0.5 m
GRIDS = [
    [(16, 1, 0.5), (16, 2, 0.5), (16, 3, 0.5)],
    [(8, 3, 2.0), (16, 4, 1.0), (32, 5, 0.5)],
    [(8, 1, 2.0), (32, 1, 0.5), (64, 1, 0.25)],
    [(64, 2, 0.5), (64, 6, 0.25), (32, 4, 0.3)],
    [(128, 7, 0.5), (128, 3, 0.125), (128, 5, 0.2)],
    [(64, 5, 1.0), (128, 6, 1.0), (16, 3, 1.7)],
]


def workload(grid):
    wl = synth.tiny_mcao_elongated()
    wl["layers"] = [dict(L, n=n, levels=lev, delta=d) for L, (n, lev, d) in zip(wl["layers"], grid)]
    return wl


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("case", range(len(GRIDS)))
def test_apply_matches_oracle_on_every_grid(case, prec):
    from paper_2202_11945_gb300 import Reconstructor
    wl = workload(GRIDS[case])
    geo = O.Geometry(wl)
    R = Reconstructor(wl, precision=prec)
    rng = np.random.default_rng(100 + case)
    c = rng.standard_normal(geo.n_c).astype(np.float32).astype(float)
    assert_close(to_np(R.apply_M(to_dev(c, prec))), O.apply_M(geo, c), TOL_OP[prec], "M c")
    assert_close(to_np(R.rhs(to_dev(c[:geo.n_s], prec))), O.rhs(geo, c[:geo.n_s]), TOL_OP[prec], "b")


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("case", range(len(GRIDS)))
def test_iterations_match_oracle_on_every_grid(case, prec):
    """Three PCG iterations: the direction update, whose tiles form their halos themselves."""
    from paper_2202_11945_gb300 import Reconstructor
    wl = workload(GRIDS[case])
    geo = O.Geometry(wl)
    D = O.prior_diag(geo)
    b = O.rhs(geo, np.random.default_rng(200 + case).standard_normal(geo.n_s))
    ref, _ = O.pcg(geo, b, np.zeros(geo.n_c), 1.0 / O.precond_diag(geo, D), 3, D)
    R = Reconstructor(wl, precision=prec)
    c = R.pcg(to_dev(b, prec), to_dev(np.zeros(geo.n_c), prec), 3)
    # a few times the operators' bound: three applications, the sums of alpha and beta
    assert_close(to_np(c), ref, 100 * TOL_OP[64] if prec == 64 else 10 * TOL_OP[32], "c")
