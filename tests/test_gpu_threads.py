"""Contexts on their own host threads and streams: one context belongs to one thread at a time, but several
contexts of other shapes may step at once.  The shapes differ in what they ask of the same kernels (dynamic
shared memory among it), so a launch that goes by process-wide state fails or gives other results."""
import os
import subprocess
import sys
import threading

import pytest

import synth
from paper_2502_19864_gb300 import ringada as R
from gpu_helpers import GpuStepper

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("cfgs", [
    (synth._enc(1, 64, 2, 64, 8, 2, 8, "f32"), synth._enc(1, 384, 3, 384, 16, 2, 40, "f32"),
     synth._paper(1, 512, 16, 512, 16, 2, 24, "f32")),
    (synth._enc(1, 256, 4, 256, 32, 2, 40, "bf16"), synth._enc(1, 768, 12, 768, 32, 2, 40, "bf16"),
     synth._dec(1, 320, 5, 320, 40, 40, 2, 40, "bf16"))], ids=["f32", "bf16"])
def test_contexts_of_other_shapes_at_once(cfgs, steps=400):
    import torch
    runs = [GpuStepper(cfg, synth.make_workload(cfg, 0)) for cfg in cfgs]
    try:
        alone = []
        for run in runs:
            run.step(1)
            alone.append((run.logits.cpu(), run.model.grad(0, "WdF").cpu()))
        torch.cuda.synchronize()
        failed = []

        def work(run, want):
            try:
                stream = torch.cuda.Stream()
                for _ in range(steps):
                    R.ra_forward(run.ctx, run.x.data_ptr(), run.labels.data_ptr(), run.cfg.batch, run.cfg.seq,
                                 run.loss.data_ptr(), run.logits.data_ptr(), stream)
                    R.ra_backward_truncated(run.ctx, run.cfg.n_layers - 1, stream)
                R.ra_sync_status(run.ctx, stream)
                if not (torch.equal(run.logits.cpu(), want[0]) and torch.equal(run.model.grad(0, "WdF").cpu(), want[1])):
                    failed.append("%s: other results" % (run.cfg,))
            except Exception as e:
                failed.append("%s: %s" % (run.cfg, e))

        threads = [threading.Thread(target=work, args=a) for a in zip(runs, alone)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not failed, failed
    finally:
        for run in runs:
            run.close()


FIRST_CALLS = """
import sys, threading
sys.path.insert(0, %r)
import torch
from paper_2502_19864_gb300 import ringada as R
A, B = (torch.randn(256, 256, device="cuda").bfloat16() for _ in range(2))
C = [torch.empty(256, 256, device="cuda") for _ in range(16)]
R.lib(); torch.cuda.synchronize()
at_once, failed = threading.Barrier(16), []
def work(c):
    torch.zeros(1, device="cuda")
    at_once.wait()
    try:
        R.ra_gemm_bf16_epi(A.data_ptr(), B.data_ptr(), 256, 256, 256, R.RA_EPI_STORE, C_ptr=c.data_ptr(), c_dtype=R.RA_F32)
    except Exception as e:
        failed.append(str(e))
threads = [threading.Thread(target=work, args=(c,)) for c in C]
for t in threads: t.start()
for t in threads: t.join()
torch.cuda.synchronize()
assert not failed, failed
assert all(torch.equal(c, C[0]) for c in C)
"""


def test_first_calls_of_a_process_at_once():
    """What is looked up once per process (a driver entry point, the device's kind) is there for every thread
    that asks for it, also while another is still looking it up."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    for _ in range(3):
        subprocess.run([sys.executable, "-c", FIRST_CALLS % root], check=True, timeout=300)


def test_stand_alone_call_on_a_thread_new_to_cuda():
    import torch
    A, B = (torch.randn(128, 128, device="cuda").bfloat16() for _ in range(2))
    C, failed = torch.empty(128, 128, device="cuda"), []
    torch.cuda.synchronize()

    def work():
        try:
            R.ra_gemm_bf16_epi(A.data_ptr(), B.data_ptr(), 128, 128, 128, R.RA_EPI_STORE, C_ptr=C.data_ptr(),
                               c_dtype=R.RA_F32)
        except Exception as e:
            failed.append(str(e))

    thread = threading.Thread(target=work)
    thread.start()
    thread.join()
    assert not failed, failed
    torch.cuda.synchronize()
    assert (C.double() - A.double() @ B.double().T).abs().max().item() < 1e-4
