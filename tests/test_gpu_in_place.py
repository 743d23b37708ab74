"""Operators whose output is their input: the coefficient and layer vectors have one length, so a
caller may pass one buffer for both."""
import numpy as np
import pytest
import torch

import synth
from tests.gpu_common import TOL_OP, assert_close, to_np

pytestmark = pytest.mark.gpu


def workload(n, levels):
    wl = synth.tiny_mcao()
    wl["layers"] = [dict(L, n=n, levels=levels, delta=0.5) for L in wl["layers"]]
    return wl


# layers of one tile, of four and of sixteen, few and all levels
@pytest.mark.parametrize("n,levels", [(32, 5), (64, 2), (64, 6), (128, 3), (128, 7)])
@pytest.mark.parametrize("prec", [32, 64])
def test_in_place_equals_out_of_place(n, levels, prec):
    from paper_2202_11945_gb300 import Reconstructor
    R = Reconstructor(workload(n, levels), precision=prec)
    gen = torch.Generator(device="cuda").manual_seed(n + levels)
    for name in ("idwt", "dwt", "apply_M"):
        for rep in range(20):
            x = torch.randn(R.n_coeffs, dtype=R.dtype, device="cuda", generator=gen)
            want = to_np(getattr(R, name)(x))
            assert_close(to_np(getattr(R, name)(x, out=x)), want, 2 * TOL_OP[prec], name)
    # an output right behind its input does not overlap it
    buf = torch.randn(2 * R.n_coeffs, dtype=R.dtype, device="cuda", generator=gen)
    want = to_np(R.idwt(buf[:R.n_coeffs]))
    got = R.idwt(buf[:R.n_coeffs], out=buf[R.n_coeffs:])
    assert np.array_equal(to_np(got), want)
    R.close()
