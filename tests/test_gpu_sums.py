"""The sums of squares of the GPU path -- the step's loss 1/2 ||R||^2 and LSQR's norms -- against float64.

Both are sums of positive terms, so the error of any order of summation in float64 is at most its depth (additions on
the longest path) times 2^-53 relative; the square root of a norm halves it.  The bars below are that depth, counted
for the smallest case and rounded up, and hold for every way of splitting the sum that is no less exact."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2202_04486_gb300 import binding, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    binding.load_library()


def _lsqr(D, U, nv, n_iter):
    ns, nr, nt = D.shape
    plan = binding.MDCPlan(D, nv, nb_max=ns)
    X = torch.zeros((nv, nr, nt), device="cuda")
    norms = torch.zeros(n_iter + 1, device="cuda", dtype=torch.float64)
    binding.smdd_lsqr(plan.handle, X, U, n_iter, 0, None, norms)
    assert plan.sync_status() == binding.MDC_OK
    plan.close()
    return X.double().cpu().numpy(), norms.cpu().numpy()


def test_lsqr_norm_of_large_amplitudes():
    """8.2e7 samples of magnitude 1e18: every square (1e36) is inside the FP32 range, a thread's share of them (about
    1000) is not.  LSQR is linear in U: the run scaled by a power of two must give the scaled norms and solution, to the
    FP32 operator bound (1e-5)."""
    nt, nr, nv, ns = 512, 2, 400, 400
    g = torch.Generator(device="cuda").manual_seed(11)
    D = torch.randn((ns, nr, nt), device="cuda", generator=g)
    U = torch.where(torch.rand((ns, nv, nt), device="cuda", generator=g) < 0.5, -1e18, 1e18).float()
    X, norms = _lsqr(D, U, nv, 2)
    U.mul_(2.0 ** -59)
    X_small, n_small = _lsqr(D, U, nv, 2)
    assert np.isfinite(norms).all() and np.isfinite(X).all()
    exact = float(np.float32(1e18)) * math.sqrt(ns * nv * nt)
    assert abs(norms[0] - exact) <= 1e-12 * exact
    np.testing.assert_allclose(norms, n_small * 2.0 ** 59, rtol=1e-5)
    assert oracle.rel_l2(X, X_small * 2.0 ** 59) <= 1e-5
