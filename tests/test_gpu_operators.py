"""The operators beside the frame on every form their kernels accept, against the per-sensor
and per-layer kernels (slope maps, projections)."""

import pytest
import torch

from tests.gpu_common import recon

pytestmark = pytest.mark.gpu


def _rel(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("name", ["tiny_scao", "tiny_mcao", "paper_mcao"])
@pytest.mark.parametrize("prec", [32, 64])
def test_model_and_its_adjoint(name, prec):
    """Gamma P phi and P^T Gamma^T s against the two-step forms.  Both sides round O(10)
    operations of one precision on values that do not cancel beyond the slopes' own
    differences (a factor of about 100 on smooth layers): 1e3 eps."""
    R = recon(name, prec)
    tol = 1e3 * (1.2e-7 if prec == 32 else 2.3e-16)
    gen = torch.Generator(device="cuda").manual_seed(5)
    phi = torch.randn(R.n_coeffs, dtype=R.dtype, device="cuda", generator=gen)
    s = torch.randn(R.n_slopes, dtype=R.dtype, device="cuda", generator=gen)
    assert _rel(R.forward(phi), R.slopes(R.project(phi))) <= tol
    assert _rel(R.forward_adj(s), R.project_adj(R.slopes_adj(s))) <= tol
    # <G phi, s> = <phi, G^T s>
    lhs = float((R.forward(phi).double() * s.double()).sum())
    rhs = float((phi.double() * R.forward_adj(s).double()).sum())
    scale = float(R.forward(phi).double().norm() * s.double().norm())
    assert abs(lhs - rhs) <= tol * scale
