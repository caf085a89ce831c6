"""The split-K tcgen05 GEMM of few output tiles at its edges: one row, one k-block, K and N tails, a
k-block more or less than the shares divide, one to eight CTAs to a tile, every epilogue, B as [N, K] and as
stored [K, N]; against a 64-bit matmul of the same bf16 operands, and bitwise repeatable (the gate|up
epilogues through a decoder step)."""
import pytest

import synth
from gpu_helpers import GpuStepper, check_step, oracle_full
from paper_2502_19864_gb300 import ringada as R

pytestmark = pytest.mark.gpu

SHAPES = [(1, 8, 8), (16, 64, 64), (128, 768, 3072), (129, 72, 1096), (300, 1024, 256), (37, 2304, 776),
          (512, 768, 768), (640, 520, 2056)]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def check_epilogues(M, N, K, kn):
    """Every epilogue of the C ABI's GEMM against 64 bits, twice, with a guard row."""
    import torch
    g = torch.Generator().manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g).to(torch.bfloat16)
    B = (torch.randn(N, K, generator=g) * 0.05).to(torch.bfloat16)
    bias = torch.randn(N, generator=g) * 0.1
    aux = torch.randn(M, N, generator=g)
    acc = (A.cuda().double() @ B.cuda().double().T).cpu()
    u = acc + bias.double()
    cdf = 0.5 * (1 + torch.erf(u / 2 ** 0.5))
    auxb = aux.to(torch.bfloat16)
    Ad, Bd, bd = A.cuda(), (B.T.contiguous() if kn else B).cuda(), bias.cuda()
    ax = {R.RA_EPI_MUL: auxb.cuda(), R.RA_EPI_RESID: aux.cuda()}
    want = {R.RA_EPI_STORE: (u, None), R.RA_EPI_BIAS_GELU: (u, u * cdf), R.RA_EPI_MUL: (acc * auxb.double(), None),
            R.RA_EPI_RESID: (acc + aux.double(), None),
            R.RA_EPI_BIAS_GELU_G: (cdf + u * torch.exp(-u * u / 2) / (2 * torch.pi) ** 0.5, u * cdf)}
    for epi, refs in want.items():
        f32 = epi in (R.RA_EPI_STORE, R.RA_EPI_RESID)
        dt = torch.float32 if f32 else torch.bfloat16
        twice = []
        for _ in range(2):
            # (a guard row behind each output: nothing is written past M rows)
            C = torch.full((M + 1, N), float("nan"), dtype=dt, device="cuda")
            C2 = torch.full((M + 1, N), float("nan"), dtype=torch.bfloat16, device="cuda")
            R.ra_gemm_bf16_epi(Ad.data_ptr(), Bd.data_ptr(), M, N, K, epi | (R.RA_EPI_B_KN if kn else 0),
                               bd.data_ptr() if refs[1] is not None or epi == R.RA_EPI_STORE else None,
                               ax[epi].data_ptr() if epi in ax else None, C.data_ptr(), R.RA_F32 if f32 else R.RA_BF16,
                               C2.data_ptr() if refs[1] is not None else None)
            torch.cuda.synchronize()
            twice.append((C.cpu(), C2.cpu()))
        for got, again, ref, wide in zip(twice[0], twice[1], refs, (f32, False)):
            if ref is None:
                continue
            assert bool(got[M].isnan().all()), "written past the last row"
            assert torch.equal(got[:M], again[:M])
            err = (got[:M].double() - ref).abs().max().item()
            # fp32 sums of K products (the tensor cores truncate at each of K / 16 additions:
            # K / 16 2^-23 of the sum at most), bf16 results half a unit in the 8th bit (2^-9) of the largest value
            assert err <= (1e-5 + K / 16 * 2.0 ** -23 if wide else 2.0 ** -8) * max(ref.abs().max().item(), 1.0), (epi, err)


@pytest.mark.parametrize("kn", [False, True])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_epilogues(M, N, K, kn):
    check_epilogues(M, N, K, kn)


@pytest.mark.parametrize("H,heads,F,S", [(1024, 16, 2816, 120), (2048, 16, 512, 100), (2048, 16, 1024, 77),
                                         (2112, 33, 2560, 33)])
def test_gate_up_epilogues(H, heads, F, S):
    """The gate|up epilogues through a decoder step: SwiGLU' on 64-wide tiles (H 1024: two CTAs to a tile; H
    2048: eight) and SwiGLU on 128-wide ones (H 2048: eight and four CTAs to a tile; H 2112: two)."""
    cfg = synth._dec(1, H, heads, F, 64, 96, 1, S, "bf16")
    w = synth.make_workload(cfg, 0)
    ref = oracle_full(cfg, w)
    run = GpuStepper(cfg, w)
    try:
        loss = run.step(1)
        check_step(cfg, loss, run.logits.double().cpu().numpy(), run.grads(0), run.head_grads(), ref, 0)
    finally:
        run.close()
