"""The least-squares fit's kernels beyond the shapes of their fast paths, on systems of the same
condition as those of test_gpu_lsfit and so within its bounds:
- more directions than warps with a direction of their own (9): every direction several times,
  its weight shared among the copies, is the same system;
- actuators under more pupil rows than are held in registers (6): five times as many nodes a side
  with 25 times the regularisation scales the system by 25."""
import numpy as np
import pytest

import oracle as O
import synth
from tests.gpu_common import rel_l2, to_dev, to_np
from tests.test_gpu_lsfit import CASES, SOLVE_TOL, TOL, oracle_fit, recon

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("copies", [2, 6])
@pytest.mark.parametrize("prec", [64, 32])
def test_many_directions(copies, prec):
    wl = synth.tiny_mcao()
    geo = O.Geometry(wl)
    c = np.random.default_rng(31).standard_normal(geo.n_c)
    dirs, w, n_fit, eps = CASES["tiny_mcao"]
    ref = oracle_fit(geo, c, (dirs, w, n_fit, eps))
    R = recon(wl, prec)
    a, _, rel = R.fit_ls(to_dev(c, prec), dirs * copies, [x / copies for x in w] * copies, n_fit, eps, tol=SOLVE_TOL[prec])
    assert rel <= SOLVE_TOL[prec]
    assert rel_l2(to_np(a), ref) <= TOL[prec], rel_l2(to_np(a), ref)
    R.close()


@pytest.mark.parametrize("name", ["tiny_scao", "tiny_mcao"])
@pytest.mark.parametrize("prec", [64, 32])
def test_many_pupil_rows_an_actuator(name, prec):
    wl = synth.workload_by_name(name)
    geo = O.Geometry(wl)
    c = np.random.default_rng(32).standard_normal(geo.n_c)
    dirs, w, n_fit, eps = CASES[name]
    ref = oracle_fit(geo, c, (dirs, w, 5 * n_fit, 25 * eps))
    R = recon(wl, prec)
    a, _, rel = R.fit_ls(to_dev(c, prec), dirs, w, 5 * n_fit, 25 * eps, tol=SOLVE_TOL[prec])
    assert rel <= SOLVE_TOL[prec]
    assert rel_l2(to_np(a), ref) <= TOL[prec], rel_l2(to_np(a), ref)
    R.close()
