"""Batched frames against the instances' own, bit by bit, on the instances whose sums over a
sensor have many nodes per tile (rings of the 24 m geometries inside one tile, spot elongation):
the branch of the inverse kernel that reduces them together."""
import numpy as np
import pytest

import synth
from tests.gpu_common import to_dev, to_np

pytestmark = pytest.mark.gpu


def workloads():
    uneven = synth.batched_instances(64)
    return [uneven[19], uneven[48], uneven[57], synth.tiny_mcao_elongated(), synth.paper_mcao()]


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("warm", [False, True])
def test_batched_frames_with_dense_sums_equal_single_frames(prec, warm):
    from paper_2202_11945_gb300 import Batch, Reconstructor
    wls = workloads()
    for wl in wls:
        wl["params"] = dict(wl["params"], iters=4)
    one = [Reconstructor(wl, precision=prec, warm_residual=warm) for wl in wls]
    many = [Reconstructor(wl, precision=prec, warm_residual=warm) for wl in wls]
    B = Batch(many)
    atm = [synth.TruthAtmosphere(wl["truth"]) for wl in wls]
    for t in range(4):
        s = [to_dev(synth.simulate_slopes(wl, t, atm=a), prec) for wl, a in zip(wls, atm)]
        got = B.reconstruct(s)
        for wl, R, Rb, x, b in zip(wls, one, many, s, got):
            a = R.reconstruct(x)
            assert np.array_equal(to_np(a), to_np(b)), (wl["name"], t)
            assert np.array_equal(to_np(R.get_state()[0]), to_np(Rb.get_state()[0])), (wl["name"], t)
    B.close()
    for R in one + many:
        R.close()
