"""The norm backward with several warps to a row (H = 2048: two rows a CTA) at one row, an odd number of rows
and a whole last CTA: LayerNorm in both types and RMSNorm, through the step against the fp64 oracle."""
import pytest

import synth
from gpu_helpers import GpuStepper, check_step, oracle_full

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("T", [1, 2, 7, 77])
@pytest.mark.parametrize("make", [lambda T: synth._enc(2, 2048, 16, 64, 32, T, 1, "bf16"),
                                  lambda T: synth._enc(2, 2048, 16, 64, 32, T, 1, "f32"),
                                  lambda T: synth._dec(2, 2048, 16, 64, 32, 40, 1, T, "bf16")],
                         ids=["layernorm-bf16", "layernorm-f32", "rmsnorm"])
def test_rows(make, T):
    cfg = make(T)
    w = synth.make_workload(cfg, 0)
    ref = oracle_full(cfg, w)
    run = GpuStepper(cfg, w)
    try:
        for d in (1, 2):
            loss = run.step(d)
            check_step(cfg, loss, run.logits.double().cpu().numpy(), run.grads(2 - d), run.head_grads(), ref, 2 - d)
    finally:
        run.close()
