"""The persistent split-BF16 products at the edges of its tiles: rows around 128, columns around the chunk of
32 and the block of 8, batch blocks of 16 / 32 / 64 and beyond, the last pair of bins and band limits that cut a pair,
and the transposed read of a symmetric model (chunks below, across and above the block diagonal).

Tolerances: a split operand carries 16 significant bits, so a product has a relative error of order 2^-16 and a sum
of K of them, with independent signs, at most that of its largest terms: 1e-4 relative L2 (the bound of the
split-BF16 path) covers it with a factor of several.  The symmetric step reads the same values from the mirrored
position and is bit-identical."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2202_04486_gb300 import binding, build, synth  # noqa: E402

pytestmark = pytest.mark.gpu

REL_L2 = 1e-4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    binding.load_library()


def _cuda(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=dtype)


@pytest.mark.parametrize("nt,nr,nv,ns,nb", [
    (33, 1, 1, 3, 1), (64, 7, 127, 9, 16), (100, 31, 128, 40, 17), (128, 32, 129, 40, 32), (130, 33, 257, 70, 33),
    (200, 100, 130, 80, 64), (64, 65, 60, 90, 65), (257, 129, 384, 150, 130),
])
def test_forward_at_tile_edges(nt, nr, nv, ns, nb):
    seed = nt + nr + nv
    D = synth.random_traces((ns, nr, nt), seed).astype(np.float32).astype(np.float64)
    X = synth.random_traces((nv, nr, nt), seed + 1).astype(np.float32).astype(np.float64)
    idx = synth.random_indices(ns, nb, seed + 2, replace=True)
    plan = binding.MDCPlan(_cuda(D), nv, nb_max=nb, precision=binding.MDC_PREC_BF16X3)
    U = plan.forward(_cuda(X), _cuda(idx, torch.int32)).double().cpu().numpy()
    assert plan.sync_status() == binding.MDC_OK
    assert oracle.rel_l2(U, oracle.mdc_forward_fft(D, X, idx)) <= REL_L2
    plan.close()


@pytest.mark.parametrize("band", [1, 2, 7, 8, 64])
def test_band_limit_that_cuts_a_pair_of_bins(band):
    nt, nr, nv, ns, nb = 64, 40, 140, 30, 20
    D, X = synth.random_traces((ns, nr, nt), 5), synth.random_traces((nv, nr, nt), 6)
    idx = _cuda(synth.random_indices(ns, nb, 7), torch.int32)
    out = []
    for prec in (binding.MDC_PREC_BF16X3, binding.MDC_PREC_FP32):
        plan = binding.MDCPlan(_cuda(D), nv, nb_max=nb, precision=prec)
        plan.set_band(band)
        out.append(plan.forward(_cuda(X), idx).double().cpu().numpy())
        plan.close()
    assert oracle.rel_l2(out[0], out[1]) <= REL_L2


@pytest.mark.parametrize("n,nb", [(161, 16), (200, 32), (300, 48)])
def test_transposed_read_of_a_symmetric_model(n, nb):
    nt, ns = 64, 60
    D, U = synth.random_traces((ns, n, nt), n), synth.random_traces((ns, n, nt), n + 1)
    flags = binding.SMDD_RECIPROCITY | binding.SMDD_KEEP_XHAT | binding.SMDD_REUSE_XHAT
    out = []
    for sym in (0, binding.SMDD_SYMMETRIC):
        plan = binding.MDCPlan(_cuda(D), n, nb_max=nb, precision=binding.MDC_PREC_BF16X3)
        X, Ug = torch.zeros((n, n, nt), device="cuda"), _cuda(U)
        for k in range(3):
            plan.step(X, Ug, _cuda(synth.random_indices(ns, nb, k), torch.int32), 1e-6, flags | sym)
        assert plan.sync_status() == binding.MDC_OK
        out.append(X.cpu().numpy())
        plan.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("nt,nr,nv,ns,nb", [
    (33, 1, 1, 3, 1), (64, 127, 7, 9, 16), (100, 128, 31, 40, 17), (128, 129, 130, 40, 32), (130, 257, 33, 70, 33),
    (64, 300, 400, 80, 64), (64, 65, 60, 90, 65),
])
def test_adjoint_at_tile_edges(nt, nr, nv, ns, nb):
    """The persistent adjoint (tiles of 128 x 128, one or two K chunks of 32; batch 65 runs on the tile kernel)."""
    seed = nt + nr + nv
    D = synth.random_traces((ns, nr, nt), seed).astype(np.float32).astype(np.float64)
    R = synth.random_traces((nb, nv, nt), seed + 1).astype(np.float32).astype(np.float64)
    idx = synth.random_indices(ns, nb, seed + 2, replace=True)
    plan = binding.MDCPlan(_cuda(D), nv, nb_max=nb, precision=binding.MDC_PREC_BF16X3)
    G = plan.adjoint(_cuda(R), _cuda(idx, torch.int32)).double().cpu().numpy()
    assert plan.sync_status() == binding.MDC_OK
    assert oracle.rel_l2(G, oracle.mdc_adjoint_fft(D, R, idx)) <= REL_L2
    plan.close()
