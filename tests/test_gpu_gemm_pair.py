"""The GEMM's paired form (two CTAs on one 256 x 256 tile) at its edges: an odd CTA with no rows or a
few, ragged N and K, a last round split over K, B as [N, K] and as stored [K, N], every epilogue; the
gate|up epilogues through a decoder step whose last pair is half empty."""
import pytest

import synth
from gpu_helpers import GpuStepper, check_step, oracle_full
from test_gpu_gemm_splitk import check_epilogues

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("kn", [False, True])
@pytest.mark.parametrize("M,N,K", [(7941, 1000, 3080), (8069, 1024, 1544), (8192, 3000, 1032)])
def test_epilogues(M, N, K, kn):
    check_epilogues(M, N, K, kn)


def test_gate_up_epilogues():
    cfg = synth._dec(1, 2048, 16, 5632, 128, 96, 2, 650, "bf16")
    w = synth.make_workload(cfg, 0)
    ref = oracle_full(cfg, w)
    run = GpuStepper(cfg, w)
    try:
        loss = run.step(1)
        check_step(cfg, loss, run.logits.double().cpu().numpy(), run.grads(0), run.head_grads(), ref, 0)
    finally:
        run.close()
