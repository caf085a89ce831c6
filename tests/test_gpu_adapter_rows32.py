"""The bf16 adapter kernels on 32-row CTAs (more than 16 rows an SM, H <= 1024) with a last CTA of 1, 15, 16
or 17 rows, both placements, the three bottlenecks of that path, through the step at every depth against
the fp64 oracle; the span head gives every token a gradient."""
import dataclasses

import pytest

import synth
from gpu_helpers import GpuStepper, check_step, oracle_full

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


# 16 x 152 SMs = 2432 rows: 2433 (1 past a whole CTA), 2447 (15), 2448 (16), 2449 (17)
@pytest.mark.parametrize("make,L,H,m,B,S", [
    (synth._span, 1, 768, 64, 3, 811), (synth._span, 1, 1024, 128, 31, 79), (synth._span, 1, 1024, 32, 24, 102),
    (synth._span, 1, 128, 128, 1, 2447), (synth._paper, 2, 768, 128, 31, 79), (synth._paper, 2, 1024, 64, 1, 2447),
    (synth._paper, 2, 256, 32, 3, 811)])
def test_ragged_last_cta(make, L, H, m, B, S):
    cfg = dataclasses.replace(make(L, H, H // 64, 64, m, B, S, "bf16"), head="span")
    w = synth.make_workload(cfg, 0)
    ref = oracle_full(cfg, w)
    run = GpuStepper(cfg, w)
    try:
        assert run.model.stats()["num_sms"] * 16 < cfg.tokens
        for d in range(1, L + 1):
            loss = run.step(d)
            check_step(cfg, loss, run.logits.double().cpu().numpy(), run.grads(L - d), run.head_grads(), ref, L - d)
    finally:
        run.close()
