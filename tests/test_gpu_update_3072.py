"""The update kernels at FFT length 3072, whose momentum / Adam form has a register split of its own: N-SGD, Adam and the
mute alone, with and without the new model's spectra, at record lengths of every alignment class and at the largest
one, against the FP64 oracle.

Tolerance: the gradient's FP32 bound (1e-5 relative L2); Adam with eps = max|g| carries it to at most 2e-5 a step."""
import numpy as np
import pytest
import torch

import oracle
from paper_2202_04486_gb300 import binding, build, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    binding.load_library()


def _cuda(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=dtype)


@pytest.mark.parametrize("nt", [1025, 1402, 1536])
@pytest.mark.parametrize("solver", ["nsgd", "adam", "mute"])
def test_two_steps(nt, solver):
    nr, nv, ns, nb = 11, 7, 6, 5   # (11 receivers: two CTAs along the row, the second with three traces)
    D = synth.random_traces((ns, nr, nt), nt).astype(np.float32).astype(np.float64)
    U = synth.random_traces((ns, nv, nt), nt + 1).astype(np.float32).astype(np.float64)
    mute = (np.arange(nv * nr).reshape(nv, nr) * 19 % nt).astype(np.int32)
    X, V, S = (np.zeros((nv, nr, nt)) for _ in range(3))
    plan = binding.MDCPlan(_cuda(D), nv, nb_max=nb)
    Xg, Vg, Sg, Ug, mg = _cuda(X), _cuda(V), _cuda(S), _cuda(U), _cuda(mute, torch.int32)
    g0 = oracle.precondition(oracle.gradient(D, X, U, np.arange(nb), fft=True)[0], mute=mute)
    eps, alpha = float(np.abs(g0).max()), 0.2 / oracle.sigma2_max(D)
    for k in range(2):
        idx = synth.random_indices(ns, nb, nt + k)
        fl = binding.SMDD_REUSE_XHAT if k else binding.SMDD_KEEP_XHAT
        ti = _cuda(idx, torch.int32)
        if solver == "nsgd":
            plan.step_nsgd(Xg, Vg, Ug, ti, alpha, mu=0.9, flags=fl, mute=mg)
            X, V, _ = oracle.nsgd_step(D, X, V, U, idx, alpha, 0.9, mute=mute, fft=True)
        elif solver == "adam":
            plan.step_adam(Xg, Vg, Sg, Ug, ti, 1e-3, k + 1, eps=eps, flags=fl, mute=mg)
            X, V, S, _ = oracle.adam_step(D, X, V, S, U, idx, 1e-3, k + 1, eps=eps, mute=mute, fft=True)
        else:
            binding.smdd_step_ex(plan.handle, Xg, Ug, ti, alpha, fl, mute=mg)
            X = X - alpha * oracle.precondition(oracle.gradient(D, X, U, idx, fft=True)[0], mute=mute)
    assert plan.sync_status() == binding.MDC_OK
    assert oracle.rel_l2(Xg.double().cpu().numpy(), X) <= (4e-5 if solver == "adam" else 1e-5)
    if solver != "mute":
        assert oracle.rel_l2(Vg.double().cpu().numpy(), V) <= 1e-5
    muted = np.arange(nt)[None, None, :] < mute[:, :, None]
    assert not Xg.cpu().numpy()[muted].any()
    plan.close()
