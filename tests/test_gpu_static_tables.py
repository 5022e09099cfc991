"""The allocation-free forward product at every FFT length: its twiddle tables lie at the start of the static scratch, in a
reserve whose size decides, with the spectra, which problems fit."""
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


def _static(D, X, idx):
    U = torch.full((idx.numel(), X.shape[0], D.shape[2]), float("nan"), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    binding.mdc_forward_static(D, X, idx, U, 1.0, status)
    assert int(status) == 0
    return U


@pytest.mark.parametrize("nt", [31, 60, 127, 250, 511, 1000, 1500, 2000, 4000])
def test_every_length_matches_the_plan(nt):
    D, X = _randn((5, 9, nt), 1), _randn((6, 9, nt), 2)
    idx = torch.tensor([4, 0, 3], device="cuda", dtype=torch.int32)
    plan = binding.MDCPlan(D, 6, nb_max=3)
    ref = plan.forward(X, idx).double()
    err = _static(D, X, idx).double() - ref
    assert (err.norm() / ref.norm()).item() <= 1e-5


@pytest.mark.parametrize("nt,nf,reserve", [(250, 257, 7168), (1000, 1025, 28672), (1500, 1537, 40960), (4000, 4097, 107776)])
def test_largest_problem_that_fits(nt, nf, reserve):
    """8 nf (ns ldr + nv ldr + nv ldb) bytes beside the reserve: the last source that fits is accepted, one more refused."""
    nr, nv, nb = 2, 8, 8
    room = (64 << 20) - reserve - 3 * 256     # (each array is rounded up to 256 bytes)
    ns = (room // (8 * nf) - nv * nr - nv * nb) // nr
    X = _randn((nv, nr, nt), 3)
    idx = torch.arange(nb, device="cuda", dtype=torch.int32)
    D = _randn((ns, nr, nt), 4)
    U = _static(D, X, idx)
    plan = binding.MDCPlan(D[:nb].contiguous(), nv, nb_max=nb)
    ref = plan.forward(X, idx).double()
    assert ((U.double() - ref).norm() / ref.norm()).item() <= 1e-5
    with pytest.raises(binding.MDCError) as e:
        _static(_randn((ns + 2, nr, nt), 4), X, idx)
    assert e.value.status == binding.MDC_ERR_UNSUPPORTED
