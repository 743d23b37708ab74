"""Stage launches back to back do what the same launches one at a time do: the layer stage updates
c and the residual on every launch, so a launch that read either too early would leave others."""
import numpy as np
import pytest
import torch

import synth
from tests.gpu_common import recon, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["tiny_scao", "tiny_mcao", "maory"])
@pytest.mark.parametrize("prec", [32, 64])
def test_repeated_stages_equal_single_ones(name, prec):
    s = to_dev(synth.simulate_slopes(synth.workload_by_name(name), 0), prec)
    out = []
    for together in (True, False):
        R = recon(name, prec)
        R.reconstruct(s)
        for stage in ("idwt", "sensor", "layer"):
            for k in range(1 if together else 25):
                R.bench_stage(stage, 25 if together else 1)
                if not together:
                    torch.cuda.synchronize()
        out.append([to_np(x) for x in (R.get_state()[0], R.residual(False)[0])])
        R.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
