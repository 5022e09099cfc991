"""Arrays whose base address is only 4- or 8-byte aligned, at record lengths that would allow 16-byte accesses: the operator,
its adjoint and the update read and write the same bits as on aligned arrays."""
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


def _shifted(t, offset):
    buf = torch.zeros(t.numel() + 4, device="cuda")
    out = buf[offset:offset + t.numel()].view(t.shape)
    out.copy_(t)
    return out


def _randn(shape, seed):
    return torch.randn(shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))


@pytest.mark.parametrize("offset", [1, 2])
@pytest.mark.parametrize("nt", [64, 128, 256, 512, 1024, 1500, 2000, 4096])
def test_same_bits_from_shifted_arrays(nt, offset):
    nr, nv, ns, nb = 11, 5, 6, 4
    D, X0, U, R = _randn((ns, nr, nt), 1), _randn((nv, nr, nt), 2), _randn((ns, nv, nt), 3), _randn((nb, nv, nt), 4)
    idx = torch.tensor([5, 0, 2, 2], device="cuda", dtype=torch.int32)
    out = []
    for o in (0, offset):
        s = lambda t: _shifted(t, o)   # noqa: E731
        plan = binding.MDCPlan(s(D), nv, nb_max=nb)
        res = [plan.forward(s(X0), idx, out=s(R)), plan.adjoint(s(R), idx, out=s(X0))]
        for solver in ("sgd", "nsgd", "adam"):
            X, V, S = s(X0), s(torch.zeros_like(X0)), s(torch.zeros_like(X0))
            for k in range(2):
                fl = binding.SMDD_REUSE_XHAT if k else binding.SMDD_KEEP_XHAT
                if solver == "sgd":
                    plan.step(X, s(U), idx, 1e-7, fl)
                elif solver == "nsgd":
                    plan.step_nsgd(X, V, s(U), idx, 1e-7, flags=fl)
                else:
                    plan.step_adam(X, V, S, s(U), idx, 1e-3, k + 1, eps=1.0, flags=fl)
            res += [X, V, S]
        assert plan.sync_status() == binding.MDC_OK
        plan.close()
        out.append([t.cpu().numpy() for t in res])
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
