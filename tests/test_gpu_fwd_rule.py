"""The split-BF16 forward product's two kernels (tile kernel and persistent kernel) give the same bits: rows of a model
are independent, so a model of few rows and at most 64 columns, whose tiles all run at once (tile kernel), is compared with a larger one that
holds the same rows (persistent kernel); and whole epochs on the work queues (tile kernels) with the same epochs on graph
branches, for members of several row tiles, batch blocks of 64 and many K chunks."""
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


def _forward(D, X, idx, nb, band, cfg):
    plan = binding.MDCPlan(D, X.shape[0], nb_max=nb, precision=binding.MDC_PREC_BF16X3)
    plan.set_config(gemm_fwd=cfg, gemm_adj=binding.MDC_GEMM_TC)
    if band:
        plan.set_band(band)
    U = plan.forward(X, idx)
    assert plan.sync_status() == binding.MDC_OK
    plan.close()
    return U


@pytest.mark.parametrize("nr,nb,band", [(1, 1, 0), (31, 16, 0), (64, 17, 0), (50, 32, 7), (63, 33, 0), (33, 64, 64), (65, 20, 0), (40, 100, 0)])
def test_rows_of_a_larger_model(nr, nb, band):
    nt, ns, few, many = 100, 60, 100, 300    # nf 129: 129 (258 with a batch above 64) and 387 tiles
    D, X = _randn((ns, nr, nt), 1), _randn((many, nr, nt), 2)
    idx = (torch.arange(nb, device="cuda") * 11 % ns).int()
    U = _forward(D, X, idx, nb, band, binding.MDC_GEMM_TC)
    U_few = _forward(D, X[:few].contiguous(), idx, nb, band, binding.MDC_GEMM_TC)
    U_stream = _forward(D, X[:few].contiguous(), idx, nb, band, binding.MDC_GEMM_TC_STREAM)
    assert U.any() and torch.isfinite(U).all()
    np.testing.assert_array_equal(U_few.cpu().numpy(), U[:, :few].cpu().numpy())
    np.testing.assert_array_equal(U_stream.cpu().numpy(), U[:, :few].cpu().numpy())


def test_queue_epochs_equal_branch_epochs_for_large_members():
    shapes = [(128, 150, 300, 130, 64, 0), (256, 260, 140, 100, 40, 0), (100, 200, 200, 90, 33, binding.SMDD_RECIPROCITY),
              (256, 140, 140, 70, 16, binding.SMDD_RECIPROCITY | binding.SMDD_SYMMETRIC)]
    out = []
    for mode in (binding.MDC_BATCH_BRANCHES, binding.MDC_BATCH_QUEUE):
        members = []
        for k, (nt, nr, nv, ns, nb, flags) in enumerate(shapes):
            plan = binding.MDCPlan(_randn((ns, nr, nt), 10 * k), nv, nb_max=nb, precision=binding.MDC_PREC_BF16X3)
            perm = torch.stack([torch.randperm(ns, generator=torch.Generator().manual_seed(k + e)) for e in range(2)]).int().cuda()
            members.append(dict(plan=plan, X=torch.zeros((nv, nr, nt), device="cuda"), U_obs=_randn((ns, nv, nt), 10 * k + 1), perm=perm,
                                nb=nb, alpha=1e-7, flags=flags, loss=None))
        batch = binding.MDCBatch(members, n_branches=2, mode=mode)
        batch.run(0, 2)
        torch.cuda.synchronize()
        out.append([m["X"].cpu().numpy() for m in members])
        assert all(m["plan"].sync_status() == binding.MDC_OK for m in members)
        batch.close()
        for m in members:
            m["plan"].close()
    for a, b in zip(*out):
        assert a.any()
        np.testing.assert_array_equal(a, b)
