"""The CUDA-core GEMM, the logits row statistics and the no-scratch GEMV at the edges of their tiles
and splits.

GEMM, through whole passes against the oracle: K ranges of less than one 32-wide step, with a
remainder and of many steps (d_ffn is the down projection's K), row counts around its 32-row
tiles, float32 and the bf16 shapes the tensor cores do not take (K % 64 != 0). fp32 sums of a
few hundred products of magnitude below 1 err by less than 1e-5; the tolerances are those of the
two precisions (1e-4, and 1e-3 with bf16 hi/lo activations).

GEMV: one output row, one K step, warps without a K range, uneven row ranges per block, the
largest sizes; its products and sums are fp32, K / 256 + 13 roundings deep per sum, so 1e-6 of
sum |x||w| holds at K <= 8192 with a factor of three to spare."""
import pytest

import synth
from cdsl_parity import make_setup, run_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2412_10418_gb300 import build
    build.build()


@pytest.mark.parametrize("dtype,tol", [(synth.DTYPE_F32, 1e-4), (synth.DTYPE_BF16, 1e-3)],
                         ids=["f32", "bf16"])
@pytest.mark.parametrize("d_ffn,batch,k,d", [(8, 1, 1, 1), (72, 3, 11, 1), (1304, 2, 16, 2)])
def test_k_ranges_and_row_tiles(dtype, tol, d_ffn, batch, k, d):
    mk = lambda L, D, h, kv: synth.ModelShape(n_layers=L, d_model=D, n_heads=h, n_kv_heads=kv,
                                              d_ffn=d_ffn, vocab=264)
    wl = synth.scaled(synth.TINY, dtype=dtype, target=mk(2, 192, 3, 1), draft=mk(1, 64, 1, 1),
                      batch=batch, k=k, d=d, prompt_len=37, max_new=6, reward_head=True)
    run_parity(make_setup(wl), steps=2, tol=tol, tol_r=tol)


@pytest.mark.parametrize("vocab,batch,k", [(16, 1, 16), (8, 2, 3), (512, 3, 16), (4104, 6, 5)])
def test_row_statistics_slices(vocab, batch, k):
    """A logits row over clusters of eight, four, two and one blocks (verify rows 2 k batch): more
    beams than logits in a slice, empty slices, uneven ones."""
    mk = lambda: synth.ModelShape(n_layers=1, d_model=128, n_heads=2, n_kv_heads=1, d_ffn=96,
                                  vocab=vocab)
    wl = synth.scaled(synth.TINY, target=mk(), draft=mk(), batch=batch, k=k, d=1, prompt_len=5,
                      max_new=6, n_keywords=2)
    run_parity(make_setup(wl), steps=2, tol=1e-4, tol_r=1e-4)


@pytest.mark.parametrize("R,K,N", [(1, 8, 1), (2, 264, 7), (3, 2056, 305), (4, 1024, 1217),
                                   (5, 8192, 32768), (8, 2048, 609), (8, 4104, 1215)])
def test_gemv_rows(R, K, N):
    import torch
    import paper_2412_10418_gb300 as cdsl

    g = torch.Generator(device="cpu").manual_seed(17 * R + K)
    w = (0.02 * torch.randn((N, K), generator=g)).to(torch.bfloat16).cuda()
    x = torch.randn((R, K), generator=g).cuda()
    y = torch.full((R, N), float("nan"), device="cuda")
    s = torch.cuda.current_stream()
    cdsl.cdsl_gemv_noalloc(w, x, y, s.cuda_stream)
    s.synchronize()
    err = (y.double() - x.double() @ w.double().t()).abs()
    assert bool((err <= 1e-6 * (x.double().abs() @ w.double().abs().t())).all())
