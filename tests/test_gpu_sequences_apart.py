"""A sequence's outputs do not depend on what the other sequences of the batch hold, NaN and infinities
among it: the kernels work on blocks of rows that the next sequence's rows may fill up, and a probability
of 0 times a value that is not finite is not 0.  The first sequence's logits are those of the clean batch bit
for bit; sequences that end inside a block, for every form of the bf16 attention forward (one block of 64,
128 and 256 keys; blocks of 128 with head dim 64 and 128, plain and causal)."""
import numpy as np
import pytest

import synth
from gpu_helpers import GpuStepper

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def check_apart(cfg):
    w = synth.make_workload(cfg, 0)
    run = GpuStepper(cfg, w)
    rows = cfg.seq if cfg.arch == "decoder" else 1
    try:
        run.forward(1)
        clean = run.logits.cpu()
        assert bool(clean.isfinite().all())
        for bad in (np.nan, np.inf):
            x = w["x"].copy()
            x[1] = bad
            run.set_batch(x, w["labels"])
            run.forward(1)
            got = run.logits.cpu()
            assert not bool(got[rows:].isfinite().any())
            assert bool((got[:rows] == clean[:rows]).all()), bad
    finally:
        run.close()


@pytest.mark.parametrize("cfg", [
    synth._dec(2, 128, 2, 128, 32, 40, 2, 100, "bf16"), synth._dec(2, 256, 2, 128, 32, 40, 2, 129, "bf16"),
    synth._enc(2, 128, 2, 256, 32, 2, 300, "bf16"), synth._enc(2, 256, 2, 256, 32, 2, 77, "bf16")], ids=str)
def test_blocks_of_128(cfg):
    check_apart(cfg)


@pytest.mark.parametrize("S", [1, 33, 100, 200])
def test_one_block(S):
    check_apart(synth._enc(2, 128, 2, 256, 32, 2, S, "bf16"))
