"""The fp32-arithmetic attention at the edges of its tiles (16 rows a CTA, streamed blocks of 64, four
rows a warp), head dims 32 to 128, causal with RoPE and not, fp32 and the bf16 head dims of that path,
through the step at every depth against the fp64 oracle at the repository's parity bar."""
import pytest

import synth
from gpu_helpers import GpuStepper, check_step, oracle_full

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("cfg", [
    synth._enc(2, 64, 2, 128, 16, 2, 1, "f32"), synth._enc(2, 64, 2, 128, 16, 1, 15, "f32"),
    synth._enc(2, 192, 2, 128, 16, 1, 65, "f32"), synth._enc(2, 128, 1, 128, 16, 1, 130, "f32"),
    synth._dec(2, 64, 2, 128, 16, 40, 1, 17, "f32"), synth._dec(2, 64, 1, 128, 16, 40, 2, 64, "f32"),
    synth._dec(2, 192, 2, 128, 16, 40, 1, 81, "f32"), synth._dec(2, 128, 1, 128, 16, 40, 1, 129, "f32"),
    synth._enc(2, 128, 4, 128, 32, 2, 70, "bf16"), synth._dec(2, 192, 2, 128, 32, 40, 1, 66, "bf16")], ids=str)
def test_tile_edges(cfg):
    w = synth.make_workload(cfg, 0)
    ref = oracle_full(cfg, w)
    run = GpuStepper(cfg, w)
    try:
        for d in range(1, cfg.n_layers + 1):
            k = cfg.n_layers - d
            loss = run.step(d)
            check_step(cfg, loss, run.logits.double().cpu().numpy(), run.grads(k), run.head_grads(), ref, k)
    finally:
        run.close()
