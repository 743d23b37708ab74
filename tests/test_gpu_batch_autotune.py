"""The autotuner tries the vector kernel's shapes only where the frames launch it."""
import pytest

import synth
from tests.gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warm", [False, True])
def test_vector_shapes_are_tried_for_the_warm_recurrence_only(warm):
    from paper_2202_11945_gb300 import Batch, Reconstructor
    wls = synth.batched_instances(6)[2:]
    rs = [Reconstructor(wl, precision=32, warm_residual=warm) for wl in wls]
    B = Batch(rs)
    s = [to_dev(synth.simulate_slopes(wl, 0), 32) for wl in wls]
    seen = set()
    for _ in range(4 if warm else 8):
        cfg, us = B.autotune(s, reps=2)
        assert us > 0
        seen.add((cfg["vec_passes"], cfg["vec_threads"]))
    allowed = {(p, t) for p in (1, 4) for t in (0, 256, 512)} if warm else {(1, 0)}
    assert seen <= allowed, seen
    B.close()
    for r in rs:
        r.close()
