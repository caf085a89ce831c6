"""The fp32-arithmetic adapter kernels at the edges of their tiles, through the C ABI against the
fp64 oracle: rows around the row tiles (4 to 32 rows a CTA) and the weight-gradient chunks, widths
and bottlenecks that are no multiple of the 4-element accesses or of the 32- and 64-column tiles,
the largest bottleneck, and misaligned operands.

Bound: the sums are fp32 fused multiply-adds of T, H or m terms in a fixed order, so each result is
within n u |terms| of exact with u = 2^-24; over at most 2304 terms of random sign that is far
inside the 1e-4 of the tensor's maximum that the fp32 parity bar asks for (about 1e-6 is seen)."""
import numpy as np
import pytest

import synth
from oracle import ringada_oracle as O
from paper_2502_19864_gb300 import ringada as R
from gpu_helpers import F32_TOL, GpuStepper, check_step, oracle_full, rel_max

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("T,H,m,shift,dh", [
    (1, 64, 8, 0, True), (3, 1, 1, 0, True), (5, 130, 5, 0, True), (33, 257, 33, 0, True),
    (31, 128, 32, 1, True), (257, 200, 64, 0, False), (700, 96, 65, 0, True), (2304, 64, 96, 0, True),
    (130, 2304, 128, 0, True), (4700, 36, 24, 3, True)])
def test_adapter_backward_edges(T, H, m, shift, dh):
    import torch
    rng = np.random.default_rng(T + H + m)

    def dev(a):   # `shift` floats after the start of an allocation
        t = torch.empty(a.size + shift, device="cuda")
        t[shift:].copy_(torch.tensor(a, dtype=torch.float32).flatten())
        return t[shift:]

    h, Wd = rng.normal(size=(T, H)), rng.normal(size=(H, m)) * 0.05
    x = dict(g=rng.normal(size=(T, H)), h=h, z=h @ Wd, Wd=Wd, Wu=rng.normal(size=(m, H)) * 0.05)
    x = {k: v.astype(np.float32) for k, v in x.items()}
    d = {k: dev(v) for k, v in x.items()}
    out = [dev(np.full(n, np.nan)) for n in (H * m, m * H, T * H)]
    nb = R.ra_adapter_backward_scratch_bytes(T, H, m)
    scratch = torch.empty(nb, dtype=torch.uint8, device="cuda")
    R.ra_adapter_backward(*(d[k].data_ptr() for k in ("g", "h", "z", "Wd", "Wu")), T, H, m,
                          out[0].data_ptr(), out[1].data_ptr(), out[2].data_ptr() if dh else None,
                          scratch.data_ptr(), nb)
    torch.cuda.synchronize()
    f = {k: v.astype(np.float64) for k, v in x.items()}
    rdh, rWd, rWu = O.adapter_backward(f["g"], f["h"], f["z"], f["Wd"], f["Wu"])
    for got, ref in zip(out, (rWd, rWu) + ((rdh,) if dh else ())):
        assert rel_max(got.double().cpu().numpy().reshape(ref.shape), ref) <= F32_TOL


@pytest.mark.parametrize("cfg", [
    synth._enc(2, 320, 5, 640, 40, 3, 37, "bf16"), synth._enc(2, 192, 3, 384, 64, 2, 70, "bf16"),
    synth._paper(2, 256, 4, 512, 72, 2, 33, "bf16"), synth._dec(2, 256, 4, 512, 48, 96, 3, 50, "bf16"),
    synth._dec(2, 192, 2, 384, 104, 101, 2, 19, "f32"), synth._enc(2, 64, 2, 128, 8, 1, 1, "f32"),
    synth._paper(2, 320, 5, 640, 128, 3, 11, "f32")], ids=str)
def test_models_of_other_widths(cfg):
    """Models whose adapters run these kernels, at every depth (the repository's parity bar)."""
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
