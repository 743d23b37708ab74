"""The largest instances: sixteen sensors of 80 x 80 subapertures (fifteen elongated laser stars and
a coarse 4 x 4 one), in single precision sixteen 128 x 128 layers.  The functionals of a tile exceed
the shared memory set aside for them, so part of them is read from device memory, and the shares
exceed a round of their loops; in double precision the aperture rows under a band of a grid coarser
than the apertures (4 to 8 rows a layer row) are staged in two passes.  The M-apply against the one with a kernel per layer and sensor,
which shares none of this; both round as an operator does, so twice its bound."""
import numpy as np
import pytest

import synth
from tests.gpu_common import TOL_OP, assert_close, to_np

pytestmark = pytest.mark.gpu


def workload(n_layers, delta):
    arc = synth.arcsec(1.0)
    wfs = []
    for k in range(15):
        az = 2 * np.pi * k / 15
        wfs.append(dict(n_sub=80, nb=1, lgs=True, theta=(20 * arc * np.cos(az), 20 * arc * np.sin(az)), H=90e3, sigma=0.1,
                        launch=(20.0 * np.cos(az), 20.0 * np.sin(az)), na_fwhm=11.4e3, spot_fwhm=1.1 * arc))
    wfs.append(dict(n_sub=4, nb=20, lgs=False, theta=(0.0, 0.0), H=0.0, sigma=0.02))
    layers = [dict(h=600.0 * k, w=1.0 / n_layers, delta=delta, n=128, levels=7 - k % 7) for k in range(n_layers)]
    dms = [dict(h=0.0, spacing=0.5, n_act=81)]
    return dict(name="limits", D=40.0, obs=0.28, wfs=wfs, layers=layers, dms=dms,
                params=dict(alpha=1.0, tau=0.0, gain=1.0, iters=2, r0=0.157, L0=25.0, alpha_eta=0.2))


@pytest.mark.parametrize("prec,n_layers,delta", [(32, 16, 0.5), (64, 6, 0.5), (64, 6, 1.1), (64, 6, 1.9)])
def test_largest_instances(prec, n_layers, delta):
    import torch
    from paper_2202_11945_gb300 import Reconstructor
    R = Reconstructor(workload(n_layers, delta), precision=prec)
    gen = torch.Generator(device="cuda").manual_seed(prec)
    c = torch.randn(R.n_coeffs, dtype=R.dtype, device="cuda", generator=gen)
    assert_close(to_np(R.apply_M(c)), to_np(R.apply_M_noalloc(c)), 2 * TOL_OP[prec], "M c")
    s = torch.randn(R.n_slopes, dtype=R.dtype, device="cuda", generator=gen)
    a = to_np(R.reconstruct(s))
    r = R.rhs(s) - R.apply_M(R.get_state()[0])
    assert np.all(np.isfinite(a)) and float(r.norm()) < float(R.rhs(s).norm())
    R.close()
