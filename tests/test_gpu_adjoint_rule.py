"""The split-BF16 adjoint on both sides of the rule that picks its kernel (tile kernel or persistent kernel): bit-identical
to the product that splits its operands itself (a plan for batches above 64 holds no operand images), and, for a
symmetric model, to the step without the flag."""
import numpy as np
import pytest
import torch

from paper_2202_04486_gb300 import binding, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    binding.load_library()


def _randn(shape, seed):
    return torch.randn(shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))


@pytest.mark.parametrize("nt,nr,nv,nb,band", [
    (128, 129, 128, 16, 0),      # 2 tiles a bin, 258 in all: tile kernel
    (128, 260, 129, 16, 0),      # 6 tiles a bin, 774: persistent
    (128, 129, 257, 33, 0),      # two K chunks
    (128, 300, 200, 64, 5), (128, 300, 200, 9, 128),
    (1024, 256, 256, 8, 0),      # images larger than the L2, tiles without padding: tile kernel
    (1024, 256, 256, 40, 0),     # the same with two K chunks: persistent
    (1024, 300, 150, 8, 0),      # the same images with padded tiles: persistent
])
def test_same_bits_as_the_inline_split(nt, nr, nv, nb, band):
    ns = 70
    D, R = _randn((ns, nr, nt), 1), _randn((nb, nv, nt), 2)
    idx = (torch.arange(nb, device="cuda") * 7 % ns).int()
    out = []
    for nb_max in (nb, 65):
        plan = binding.MDCPlan(D, nv, nb_max=nb_max, precision=binding.MDC_PREC_BF16X3)
        if band:
            plan.set_band(band)
        out.append(plan.adjoint(R, idx).cpu().numpy())
        assert plan.sync_status() == binding.MDC_OK
        plan.close()
    assert np.isfinite(out[0]).all() and out[0].any()
    np.testing.assert_array_equal(out[0], out[1])


@pytest.mark.parametrize("nt,n,nb", [
    (256, 300, 16),              # 3 tiles above the diagonal a bin, 771 in all: tile kernel
    (1024, 300, 8),              # 3075, padded tiles: persistent
    (1024, 384, 8),              # without padding, one K chunk a half: tile kernel
    (1024, 384, 20),             # two: persistent
])
def test_symmetric_model(nt, n, nb):
    ns = 40
    D, U = _randn((ns, n, nt), 3), _randn((ns, n, nt), 4)
    X0 = _randn((n, n, nt), 5)
    X0 = X0 + X0.transpose(0, 1)
    idx = (torch.arange(nb, device="cuda") * 3 % ns).int()
    out = []
    for sym in (0, binding.SMDD_SYMMETRIC):
        plan = binding.MDCPlan(D, n, nb_max=nb, precision=binding.MDC_PREC_BF16X3)
        X = X0.clone()
        for k in range(2):
            plan.step(X, U, idx, 1e-6, sym | binding.SMDD_RECIPROCITY | binding.SMDD_KEEP_XHAT | (binding.SMDD_REUSE_XHAT if k else 0))
        assert plan.sync_status() == binding.MDC_OK
        out.append(X.cpu().numpy())
        plan.close()
    assert not np.array_equal(out[0], X0.cpu().numpy())
    np.testing.assert_array_equal(out[0], out[1])
