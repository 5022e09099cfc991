"""The matrix-vector products (MDC_GEMM_GEMV) at the edges of what they stage: columns around the chunk of 256 of the
forward product, batches around its 8 warps and around the chunk of 128 of the adjoint, every row count of the
instantiations, and an index out of range among good ones.

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


@pytest.mark.parametrize("nr,nv,nb", [(1, 1, 1), (255, 2, 7), (256, 3, 8), (257, 4, 9), (515, 5, 127), (31, 6, 128), (300, 7, 129), (513, 8, 300)])
def test_chunk_edges(nr, nv, nb):
    nt, ns = 40, 50
    D, X, R = _f32((ns, nr, nt), 1), _f32((nv, nr, nt), 2), _f32((nb, nv, nt), 3)
    idx = synth.random_indices(ns, nb, 4, replace=True)
    plan = binding.MDCPlan(_cuda(D), nv, nb_max=nb)
    plan.set_config(gemm_fwd=binding.MDC_GEMM_GEMV, gemm_adj=binding.MDC_GEMM_GEMV)
    ti = _cuda(idx, torch.int32)
    U, G = plan.forward(_cuda(X), ti), plan.adjoint(_cuda(R), ti)
    assert plan.sync_status() == binding.MDC_OK
    _check(U, oracle.mdc_forward_fft(D, X, idx))
    _check(G, oracle.mdc_adjoint(D, R, idx))
    plan.close()


def test_index_out_of_range():
    nt, nr, nv, ns, nb = 33, 20, 3, 12, 11
    D, X, R = _f32((ns, nr, nt), 5), _f32((nv, nr, nt), 6), _f32((nb, nv, nt), 7)
    idx = synth.random_indices(ns, nb, 8, replace=True)
    plan = binding.MDCPlan(_cuda(D), nv, nb_max=nb)
    plan.set_config(gemm_fwd=binding.MDC_GEMM_GEMV, gemm_adj=binding.MDC_GEMM_GEMV)
    bad = idx.copy()
    bad[4], bad[9] = ns, -1
    good = np.array([k for k in range(nb) if k not in (4, 9)])
    U = plan.forward(_cuda(X), _cuda(bad, torch.int32))
    assert plan.sync_status() == binding.MDC_ERR_INDEX_RANGE
    assert not U[4].any() and not U[9].any()
    _check(U[_cuda(good, torch.int64)], oracle.mdc_forward_fft(D, X, idx[good]))
    G = plan.adjoint(_cuda(R), _cuda(bad, torch.int32))
    assert plan.sync_status() == binding.MDC_ERR_INDEX_RANGE
    _check(G, oracle.mdc_adjoint(D, R[good], idx[good]))
    plan.close()
