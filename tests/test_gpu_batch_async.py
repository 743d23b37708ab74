"""A batched frame given other slope and command tensors than the one before is enqueued like any
other: the call returns while the stream still works on what was there, and the frames come out
right."""
import time

import numpy as np
import pytest
import torch

import synth
from tests.gpu_common import to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [3, 16, 48])
def test_fresh_tensors_do_not_wait_for_the_stream(count):
    from paper_2202_11945_gb300 import Batch, Reconstructor
    wls = synth.batched_instances(count)
    rs, ref = ([Reconstructor(wl, precision=32) for wl in wls] for _ in range(2))
    B, Bref = Batch(rs), Batch(ref)
    gen = torch.Generator(device="cuda").manual_seed(count)
    sets = [[torch.randn(r.n_slopes, device="cuda", generator=gen) for r in rs] for _ in range(6)]
    want = []
    same = [torch.empty_like(x) for x in sets[0]]              # one buffer for every frame's slopes
    for s in sets:
        for a, b in zip(same, s):
            a.copy_(b)
        want.append([to_np(d) for d in Bref.reconstruct(same)])
    B.reconstruct(sets[0])                                     # builds the plan
    for r in rs:
        r.reset()
    torch.cuda.synchronize()
    torch.cuda._sleep(400_000_000)                             # some 0.2 s of the stream
    t0 = time.perf_counter()
    got = [B.reconstruct(s) for s in sets]
    host = time.perf_counter() - t0
    busy = not torch.cuda.current_stream().query()
    for g, w in zip(got, want):
        for a, b in zip(g, w):
            assert np.array_equal(to_np(a), b)
    assert busy and host < 0.1, host
    B.close()
    Bref.close()
    for r in rs + ref:
        r.close()
