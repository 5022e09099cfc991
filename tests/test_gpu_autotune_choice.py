"""The autotuner does not let timing noise choose between names of one kernel: for the split-BF16 forward product it picks
MDC_GEMM_TC, never MDC_GEMM_TC_STREAM (the same persistent kernel, without the failure-path check), so a tuned plan still
reports a bounded wait that gives up."""
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


def test_tuned_plans_keep_the_failure_path_check():
    nt, ns, nb = 512, 40, 32
    for n in (120, 128, 130, 140, 150, 160, 170, 180):
        g = torch.Generator(device="cuda").manual_seed(n)
        D = torch.randn((ns, n, nt), device="cuda", generator=g)
        X = torch.randn((n, n, nt), device="cuda", generator=g)
        plan = binding.MDCPlan(D, n, nb_max=nb, precision=binding.MDC_PREC_BF16X3)
        best = plan.autotune(nb, 0, reps=3)
        assert best["gemm_fwd"] != binding.MDC_GEMM_TC_STREAM
        if best["gemm_fwd"] == binding.MDC_GEMM_TC:
            binding.mdc_plan_set_wait_probe(plan.handle, 20000)
            plan.forward(X, torch.arange(nb, device="cuda").int())
            assert plan.sync_status() == binding.MDC_ERR_TIMEOUT
        plan.close()
