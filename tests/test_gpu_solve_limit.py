"""The iteration limit of the converged solves only ends the recurrence: a solve given as many
iterations as it needs does the same ones as a solve given far more."""
import numpy as np
import pytest

import synth
from tests.gpu_common import recon, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["tiny_scao", "tiny_mcao"])
@pytest.mark.parametrize("prec", [32, 64])
def test_limit_does_not_change_the_recurrence(name, prec):
    s = to_dev(synth.simulate_slopes(synth.workload_by_name(name), 0), prec)
    tol = 1e-8
    R = recon(name, prec)
    b = R.rhs(s)
    x, it, rel = R.solve(b, tol=tol, max_iters=60000)
    assert rel <= tol and it < 60000
    y, it2, rel2 = R.solve(b, tol=tol, max_iters=it)
    assert (it2, rel2) == (it, rel) and np.array_equal(to_np(x), to_np(y))
    dm, it, rel = R.reconstruct_converged(s, tol=tol, max_iters=60000)
    assert rel <= tol
    R.close()
    R = recon(name, prec)                     # no solution held to start from
    dm2, it2, rel2 = R.reconstruct_converged(s, tol=tol, max_iters=it)
    assert (it2, rel2) == (it, rel) and np.array_equal(to_np(dm), to_np(dm2))
    R.close()
