"""The FP32 products with every tile geometry that their rules pick, at ragged sizes, against the oracle: rows around 32,
64 and 128, batches around 16, 32, 48, 64 and 96, columns that are no multiple of the chunks; the forward product also in
the layout of the allocation-free entry point.

Tolerance: the FP32 operator's (1e-5 relative L2, 2e-5 of max|ref| elementwise)."""
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


def _f32(shape, seed):
    return synth.random_traces(shape, seed).astype(np.float32).astype(np.float64)


def _check(a, ref):
    a = a.double().cpu().numpy()
    assert oracle.rel_l2(a, ref) <= 1e-5 and np.max(np.abs(a - ref)) <= 2e-5 * np.max(np.abs(ref))


@pytest.mark.parametrize("nv,nb", [
    (5, 3), (128, 16), (97, 9),          # scalar
    (129, 16), (200, 5),                 # 128 x 16
    (32, 17), (7, 70),                   # 64 x 64, few rows
    (33, 17), (64, 32), (129, 31),       # 64 x 32
    (65, 32), (128, 20),                 # 128 x 32
    (100, 48), (256, 80),                # larger batches: 16 columns
    (301, 96),                           # 32 columns
    (65, 64), (200, 49), (140, 128),     # 64 columns
])
def test_forward_geometries(nv, nb):
    nt, nr, ns = 20, 21, 40
    D, X = _f32((ns, nr, nt), 1), _f32((nv, nr, nt), 2)
    idx = synth.random_indices(ns, nb, 3, replace=True)
    ref = oracle.mdc_forward_fft(D, X, idx)
    Dg, Xg, ti = _cuda(D), _cuda(X), _cuda(idx, torch.int32)
    plan = binding.MDCPlan(Dg, nv, nb_max=nb)
    U = plan.forward(Xg, ti)
    assert plan.sync_status() == binding.MDC_OK
    plan.close()
    _check(U, ref)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    U = binding.mdc_forward_static(Dg, Xg, ti, torch.empty_like(U), 1.0, status)
    assert int(status) == 0
    _check(U, ref)


@pytest.mark.parametrize("nr,nv,nb", [
    (513, 1, 5), (530, 9, 33), (700, 16, 17),             # up to 16 rows, more than 512 columns: 64-wide scalar
    (64, 64, 7), (70, 150, 20), (512, 16, 40),            # 32-wide scalar
    (130, 61, 33), (300, 90, 18), (65, 300, 64),          # packed
])
def test_adjoint_geometries(nr, nv, nb):
    nt, ns = 20, 40
    D, R = _f32((ns, nr, nt), 4), _f32((nb, nv, nt), 5)
    idx = synth.random_indices(ns, nb, 6, replace=True)
    plan = binding.MDCPlan(_cuda(D), nv, nb_max=nb)
    G = plan.adjoint(_cuda(R), _cuda(idx, torch.int32))
    assert plan.sync_status() == binding.MDC_OK
    plan.close()
    _check(G, oracle.mdc_adjoint(D, R, idx))


@pytest.mark.parametrize("n", [33, 64, 96, 100, 128, 130, 192, 201])   # upper triangles of 32-wide and of 64-wide tiles
@pytest.mark.parametrize("nb", [5, 33])
def test_reciprocity_geometries(n, nb):
    nt, ns = 20, 40
    D, X, U = _f32((ns, n, nt), 7), _f32((n, n, nt), 8), _f32((ns, n, nt), 9)
    idx = synth.random_indices(ns, nb, 10, replace=True)
    alpha = 0.3 / oracle.sigma2_max(D)
    plan = binding.MDCPlan(_cuda(D), n, nb_max=nb)
    Xg = _cuda(X)
    binding.smdd_step(plan.handle, Xg, _cuda(U), _cuda(idx, torch.int32), alpha, binding.SMDD_RECIPROCITY)
    assert plan.sync_status() == binding.MDC_OK
    plan.close()
    ref, _ = oracle.sgd_step(D, X, U, idx, alpha, recip=True, fft=True)
    _check(Xg, ref)
