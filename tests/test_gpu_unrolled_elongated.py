"""Reverse mode through the frame with spot elongation (Eq. 3): the noise weights of its last step,
where the means of the elongated stars' weighted slopes nearly cancel, against the FP64 oracle's
reverse pass.  The bounds are those of the plain geometries, from the same arithmetic."""
import pytest

from tests.gpu_common import TOL_FRAME, rel_l2, to_dev, to_np
from tests.test_gpu_unrolled import TOL_GRAD, case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,prec", [("tiny_mcao_elongated", 64), ("tiny_mcao_elongated", 32), ("paper_mcao", 32)], ids=str)
def test_elongated_frame_vjp_matches_oracle(name, prec):
    from paper_2202_11945_gb300 import Reconstructor
    wl, s, c0, g_a, a_ref, gs_ref = case(name)
    R = Reconstructor(wl, precision=prec, graph=False)
    a, gs = R.frame_vjp(to_dev(s, prec), to_dev(c0, prec), to_dev(g_a, prec))
    assert rel_l2(to_np(a), a_ref) <= TOL_FRAME[prec]
    assert rel_l2(to_np(gs), gs_ref) <= TOL_GRAD[prec]
    R.close()
