"""The vocabulary cross-entropy at the edges of its forms, through the decoder step against the fp64
oracle: one vector of logits, one more than 512 threads hold (bf16 4096, fp32 2048), the widest that the
registers hold (fp32 16384) and wider or ragged rows, which take the form that re-reads the row."""
import numpy as np
import pytest
import torch

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


@pytest.mark.parametrize("dtype,V", [("f32", 16), ("f32", 18), ("bf16", 16), ("bf16", 32776)])
def test_probabilities_below_the_normal_range(dtype, V):
    """A class of probability 2^-128 or so still gets its gradient.  The final norm's input is zero in column
    1, whose gradient comes through Wh[:, 1] alone: 2^80 for that class and zero for all others.

    Tolerance: half a step of the stored gradient, at 2^-128.5 or more 2^-21.5 of it (fp32) or 2^-5.5 = 2.2e-2
    (bf16), with the exponent's 2^-17 (a logit of 90 in fp32) or the bf16 models' 5e-2."""
    cfg = synth._dec(1, 64, 1, 64, 8, V, 1, 1, dtype)
    w = synth.make_workload(cfg, 0)
    p = w["layers"][0]
    for key in ("Wo", "Wd"):
        p[key][1] = 0
    for key in ("WuA", "WuF"):
        p[key][:, 1] = 0
    w["x"][..., 1] = 0
    w["x"][..., 0] = 1
    w["head"]["rmsf_g"][:2] = 1
    w["head"]["rmsf_g"][2:] = 0
    Wh = np.zeros_like(w["head"]["Wh"])
    Wh[1:, 0] = -1
    w["labels"][:] = 2
    # the class's logit, by the oracle's final norm: ln 2^-128 below the others' sum
    z = oracle_full(cfg, dict(w, head=dict(w["head"], Wh=Wh)))["logits"].reshape(-1)
    to = (np.log(np.exp(z).sum()) - 128 * np.log(2)) / -z[1]
    Wh[3, 0] = synth.round_to(torch.tensor([to]), dtype)[0]
    Wh[3, 1] = 2.0 ** 80
    w["head"]["Wh"] = Wh
    ref = oracle_full(cfg, w)
    run = GpuStepper(cfg, w)
    try:
        run.step(1)
        z = run.logits.double().cpu().numpy().reshape(-1)
        lse, lse_ref = (np.log(np.exp(v - v.max()).sum()) + v.max() for v in (z, ref["logits"].reshape(-1)))
        prob, prob_ref = np.exp(z[3] - lse), np.exp(ref["logits"].reshape(-1)[3] - lse_ref)
        assert 2.0 ** -128.5 < prob < 2.0 ** -126
        got = run.grads(0)[0]["WuF"][:, 1]
        want = ref["grads"][0]["WuF"][:, 1] * (prob / prob_ref)  # (a bf16 logit is off by up to a quarter)
        assert np.linalg.norm(got - want) <= (1e-3 if dtype == "f32" else 7e-2) * np.linalg.norm(want)
    finally:
        run.close()
