"""fp32 models of more tokens than a grid dimension has 32-row tiles (65535 x 32): the first, a middle and the
last sequences' logits are those that a small batch of the same sequences gives, bit for bit."""
import pytest

import synth
from paper_2502_19864_gb300 import ringada as R
from gpu_helpers import ra_cfg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def test_more_than_65535_row_tiles():
    import dataclasses
    import torch
    small = synth._span(1, 64, 1, 64, 8, 6, 128, "f32")
    big = dataclasses.replace(small, batch=16400)
    assert big.tokens > 65535 * 32
    w = synth.make_workload(small, 0)
    gen = torch.Generator(device="cuda").manual_seed(0)
    x = torch.randn(big.batch, big.seq, big.hidden, generator=gen, device="cuda")
    labels = torch.zeros(big.batch, 2, dtype=torch.int32, device="cuda")
    at = [0, 1, 8191, 16383, 16384, 16399]

    def logits(cfg, x):
        model = R.Model(ra_cfg(cfg), cfg.adapter_dim, device="cuda:0")
        model.set_weights(w["layers"], w["head"])
        out = torch.full((cfg.batch, cfg.seq, 2), float("nan"), device="cuda")
        loss = torch.zeros(1, device="cuda")
        R.ra_forward(model.ctx, x.data_ptr(), labels.data_ptr(), cfg.batch, cfg.seq, loss.data_ptr(), out.data_ptr())
        R.ra_sync_status(model.ctx)
        model.close()
        return out

    assert torch.equal(logits(big, x)[at], logits(small, x[at].contiguous()))
