"""The attention backward whose key passes also give dQ (head dim 64, sequences to 256), at the edges of
its blocks: one row, a block, a row more, two blocks, and one row past them (two passes again); plain
and causal with RoPE; through the step at every depth against the fp64 oracle."""
import pytest

import synth
from gpu_helpers import GpuStepper, check_step, oracle_full

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("S", [1, 128, 129, 256, 257])
@pytest.mark.parametrize("decoder", [False, True])
def test_block_edges(decoder, S):
    check_every_depth(synth._dec(2, 128, 2, 128, 32, 40, 2, S, "bf16") if decoder else
                      synth._enc(2, 128, 2, 256, 32, 3, S, "bf16"))


@pytest.mark.parametrize("S", [127, 128, 256, 257])
@pytest.mark.parametrize("decoder", [False, True])
def test_head_dim_128(decoder, S):
    """Two passes, with the copies of whole blocks (S a multiple of 128) and of blocks that a sequence ends in."""
    check_every_depth(synth._dec(2, 256, 2, 128, 32, 40, 2, S, "bf16") if decoder else
                      synth._span(2, 256, 2, 256, 32, 2, S, "bf16"))


def check_every_depth(cfg):
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
