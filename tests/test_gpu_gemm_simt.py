"""The fp32 GEMM at the edges of its tiles and of its split of K: one row to a row past a tile, K of one
chunk to many, K and N tails, and rows that TMA does not take (a vocabulary of 37), through the fp32
encoder and decoder steps at every depth against the fp64 oracle."""
import pytest

import synth
from gpu_helpers import GpuStepper, check_step, oracle_full

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("cfg", [
    synth._enc(2, 64, 2, 64, 16, 1, 1, "f32"), synth._enc(2, 64, 2, 192, 16, 3, 11, "f32"),
    synth._enc(2, 64, 2, 1088, 16, 2, 32, "f32"), synth._enc(2, 192, 3, 832, 16, 1, 33, "f32"),
    synth._dec(2, 64, 2, 192, 16, 37, 1, 65, "f32"), synth._dec(2, 128, 2, 832, 16, 40, 2, 31, "f32")], ids=str)
def test_tile_and_split_edges(cfg):
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
