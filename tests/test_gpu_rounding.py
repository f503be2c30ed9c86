"""Outputs whose rounding is part of what the kernels promise."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_00098_gb300 as p
    from paper_1609_00098_gb300 import build as b
    b.build()
    return p


@pytest.mark.parametrize("flux", [0, 1])
@pytest.mark.parametrize("n", [3, 4, 5, 6, 7, 8])
def test_relativistic_volume_term_of_a_uniform_flow_is_zero(pkg, n, flux):
    """The fluxes enter the mixed relativistic contraction as differences to node 0's, each flux
    and the difference rounded on their own: equal fluxes differ by zero, and the right-hand side
    of a uniform flow is zero at every node that no face lifts into.  (A product fused with the
    subtraction leaves its rounding error, 1e-8 of the flux, times the sum of |D|.)"""
    import torch
    m = pkg.Mesh(system=1, K=(3, 2, 2), n=n, flux=flux, limiter=0, gamma=5.0 / 3.0, lo=(0, 0, 0), hi=(1, 1, 1),
                 precision=1)
    prim = torch.tensor([1.3, 0.31, -0.23, 0.17, 0.7], dtype=torch.float64, device="cuda")
    R = m.rhs(m.from_prim(prim[:, None].expand(5, m.E * n ** 3).contiguous())).cpu().numpy()
    inner = R.reshape(m.E, 5, n, n, n)[:, :, 1:-1, 1:-1, 1:-1]
    assert inner.size and np.abs(inner).max() == 0.0
