"""A handle whose spot elongation is switched on, off and to other values by update_params: the
frame's kernels, single and batched, against the oracle after every switch.  The switch allocates
nothing, so a device without free memory cannot leave a handle half changed."""
import numpy as np
import pytest

import oracle as O
import synth
from paper_2202_11945_gb300 import Batch, FewhaError, Reconstructor, lib
from tests.gpu_common import TOL_FRAME, TOL_OP, assert_close, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


def elongated(wl, alpha_eta):
    return dict(wl, params=dict(wl["params"], alpha_eta=alpha_eta))


@pytest.mark.parametrize("start", [0.0, 0.2])
@pytest.mark.parametrize("prec", [32, 64])
def test_switched_elongation_matches_the_oracle(prec, start):
    wl = synth.tiny_mcao_elongated()
    atm = synth.TruthAtmosphere(wl["truth"])
    s = synth.simulate_slopes(wl, 0, atm=atm)
    R, Rb = (Reconstructor(elongated(wl, start), precision=prec) for _ in range(2))
    B = Batch([Rb])
    before = R.device_bytes()
    for alpha_eta in (0.2, 0.0, 0.35, 0.2, 0.0):
        for r in (R, Rb):
            lib().fewha_test_fail_alloc(0)              # any allocation would fail
            try:
                r.update_params(alpha_eta=alpha_eta)
            finally:
                lib().fewha_test_fail_alloc(-1)
            r.reset()
        assert R.device_bytes() == before
        w = elongated(wl, alpha_eta)
        geo, ref = O.Geometry(w), O.Reconstructor(w)
        c = np.random.default_rng(3).standard_normal(geo.n_c).astype(np.float32).astype(float)
        assert_close(to_np(R.apply_M(to_dev(c, prec))), O.apply_M(geo, c), TOL_OP[prec], "M c")
        assert_close(to_np(R.rhs(to_dev(s, prec))), O.rhs(geo, s), TOL_OP[prec], "b")
        for t in range(2):
            x = to_dev(synth.simulate_slopes(wl, t, atm=atm), prec)
            a = to_np(R.reconstruct(x))
            assert rel_l2(a, ref.frame(to_np(x))) <= TOL_FRAME[prec], (alpha_eta, t)
            assert np.array_equal(a, to_np(B.reconstruct([x])[0])), (alpha_eta, t)
    B.close()
    R.close()
    Rb.close()


def test_dense_sums_of_a_switched_handle():
    """The 37 m geometry, whose elongation sums are weights per node, made without elongation."""
    wl = synth.paper_mcao()
    geo = O.Geometry(wl)
    R = Reconstructor(elongated(wl, 0.0), precision=32)
    c = np.random.default_rng(4).standard_normal(geo.n_c).astype(np.float32).astype(float)
    plain = O.Geometry(elongated(wl, 0.0))
    assert_close(to_np(R.apply_M(to_dev(c, 32))), O.apply_M(plain, c), TOL_OP[32], "plain")
    R.update_params(alpha_eta=wl["params"]["alpha_eta"])
    assert_close(to_np(R.apply_M(to_dev(c, 32))), O.apply_M(geo, c), TOL_OP[32], "elongated")
    R.close()


def test_creation_with_both_noise_models_fails_cleanly():
    wl = elongated(synth.tiny_mcao_elongated(), 0.0)
    failures = 0
    for after in range(400):
        lib().fewha_test_fail_alloc(after)
        try:
            R = Reconstructor(wl, precision=32)
        except FewhaError as e:
            assert e.code == -3, e
            failures += 1
            continue
        finally:
            lib().fewha_test_fail_alloc(-1)
        R.close()
        break
    assert failures >= 20
