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


DEPTH = 64   # additions on the longest path of a step's sum: 32 in a thread, 5 + 8 in its CTA, the CTAs' partials


def _loss(U, nt, nv):
    """loss of a step from X = 0: the residual is -U exactly"""
    ns = U.shape[0]
    D = torch.ones((ns, 2, nt), device="cuda")
    plan = binding.MDCPlan(D, nv, nb_max=ns)
    X = torch.zeros((nv, 2, nt), device="cuda")
    loss = torch.zeros((), device="cuda", dtype=torch.float64)
    plan.step(X, U, torch.arange(ns, device="cuda", dtype=torch.int32), 0.0, loss=loss)
    assert plan.sync_status() == binding.MDC_OK
    plan.close()
    return float(loss)


def _half_sumsq(U):
    return 0.5 * math.fsum(np.square(U.double().cpu().numpy().ravel()))


@pytest.mark.parametrize("nt", [1024, 750, 501, 1500, 128])
def test_loss_is_a_float64_sum(nt):
    """Equal values are the worst case of a sum in FP32 words: every addition rounds the same way."""
    ns, nv = 3, 5
    g = torch.Generator(device="cuda").manual_seed(2)
    for U in (torch.full((ns, nv, nt), 1.78918, device="cuda"), torch.randn((ns, nv, nt), device="cuda", generator=g)):
        exact = _half_sumsq(U)
        assert abs(_loss(U, nt, nv) - exact) <= DEPTH * 2.0 ** -53 * exact


@pytest.mark.parametrize("scale", [2.0 ** 80, 2.0 ** 59, 2.0 ** -43, 2.0 ** -46, 2.0 ** -70])
def test_loss_of_large_and_small_amplitudes(scale):
    """Magnitudes whose squares, or the rounding errors of these, leave the FP32 range; with samples of every smaller
    magnitude beside them."""
    ns, nv, nt = 2, 4, 256
    g = torch.Generator(device="cuda").manual_seed(3)
    U = torch.randn((ns, nv, nt), device="cuda", generator=g) * torch.exp2(torch.randint(-30, 1, (ns, nv, nt), device="cuda", generator=g).float())
    U = U * scale
    exact = _half_sumsq(U)
    assert abs(_loss(U, nt, nv) - exact) <= DEPTH * 2.0 ** -53 * exact


def test_loss_of_infinities_and_nan():
    ns, nv, nt = 2, 4, 256
    U = torch.ones((ns, nv, nt), device="cuda")
    U[1, 2, 77] = float("-inf")
    assert _loss(U, nt, nv) == math.inf
    U[1, 3, 5] = float("nan")
    assert math.isnan(_loss(U, nt, nv))


@pytest.mark.parametrize("offset", [0, 1])
def test_lsqr_norm_is_a_float64_sum(offset):
    """2.6e7 samples, from an aligned and from an unaligned base address; 330 elements a thread, 13 additions in its
    CTA and 2 + 13 over the CTAs."""
    nt, nr, nv, ns = 512, 2, 225, 225
    n = ns * nv * nt
    D = torch.ones((ns, nr, nt), device="cuda")
    g = torch.Generator(device="cuda").manual_seed(4)
    buf = torch.empty(n + 1, device="cuda")
    U = buf[offset:offset + n].view(ns, nv, nt)
    for fill in (lambda: U.fill_(1.116925), lambda: U.normal_(generator=g)):
        fill()
        _, norms = _lsqr(D, U, nv, 1)
        exact = math.sqrt(float(np.sum(np.square(U.double().cpu().numpy()).astype(np.longdouble))))
        assert abs(norms[0] - exact) <= 0.5 * 360 * 2.0 ** -53 * exact
