"""The vocabulary cross-entropy at the edges of its forms, through the decoder step against the fp64
oracle: one vector of logits, one more than 512 threads hold (bf16 4096, fp32 2048), the widest that the
registers hold (fp32 16384) and wider or ragged rows, which take the form that re-reads the row."""
import pytest

import synth
from gpu_helpers import GpuStepper, check_step, oracle_full

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("dtype,V", [("bf16", 8), ("bf16", 4096), ("bf16", 4104), ("bf16", 9000), ("bf16", 20000),
                                     ("bf16", 32776), ("f32", 4), ("f32", 37), ("f32", 2052), ("f32", 16384),
                                     ("f32", 16388)])
def test_widths(dtype, V):
    cfg = synth._dec(1, 128, 2, 128, 32 if dtype == "bf16" else 16, V, 1, 5, dtype)
    w = synth.make_workload(cfg, 0)
    ref = oracle_full(cfg, w)
    run = GpuStepper(cfg, w)
    try:
        loss = run.step(1)
        check_step(cfg, loss, run.logits.double().cpu().numpy(), run.grads(0), run.head_grads(), ref, 0)
    finally:
        run.close()
