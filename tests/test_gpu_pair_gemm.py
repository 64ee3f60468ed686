"""The paired-SM projection GEMM (more than 64 activation rows) at the edges of its tiles, through
whole passes against the oracle: verify rows just above the threshold, at and past one 256-row
tile, ragged feature counts (d_model, d_ffn, vocabulary and head counts that are no multiples of
the 256-row weight tiles), both head sizes, and prefill passes of more than 256 rows.

Tolerance: activations enter as bf16 hi + lo planes (relative error at most 2^-17 per product)
and everything else is fp32; with logits of magnitude below 10 over two layers 1e-3 leaves a
factor of about ten over the sum of those errors, while a wrong row or feature is off by O(1)."""
import pytest

import synth
from cdsl_parity import make_setup, run_parity

pytestmark = pytest.mark.gpu

TOL = 1e-3

HD64 = synth.ModelShape(n_layers=2, d_model=320, n_heads=5, n_kv_heads=1, d_ffn=704, vocab=1032)
HD128 = synth.ModelShape(n_layers=2, d_model=384, n_heads=3, n_kv_heads=3, d_ffn=576, vocab=520)
DRAFT = dict(n_layers=1, d_model=128, n_heads=2, n_kv_heads=1, d_ffn=192)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2412_10418_gb300 import build
    build.build()


@pytest.mark.parametrize("shape", [HD64, HD128], ids=["hd64", "hd128"])
@pytest.mark.parametrize("batch,k,d", [(1, 13, 4), (2, 16, 7), (4, 13, 4), (8, 16, 4)],
                         ids=["65rows", "256rows", "260rows", "640rows"])
def test_verify_rows_at_tile_edges(shape, batch, k, d):
    wl = synth.scaled(synth.TINY, dtype=synth.DTYPE_BF16, target=shape,
                      draft=synth.ModelShape(vocab=shape.vocab, **DRAFT), batch=batch, k=k, d=d,
                      prompt_len=9, max_new=8, reward_head=True)
    run_parity(make_setup(wl), steps=2, tol=TOL, tol_r=TOL)


@pytest.mark.parametrize("shape", [HD64, HD128], ids=["hd64", "hd128"])
@pytest.mark.parametrize("batch,k,d", [(1, 15, 1), (1, 12, 2), (1, 16, 3)],
                         ids=["30rows", "36rows", "64rows"])
def test_cluster_rows_finished_on_registers(shape, batch, k, d):
    """At most 64 rows, enough of them per block of a cluster that QKV and the residual projections
    are finished on registers: shares of two to eight rows, uneven ones, both head sizes."""
    wl = synth.scaled(synth.TINY, dtype=synth.DTYPE_BF16, target=shape,
                      draft=synth.ModelShape(vocab=shape.vocab, **DRAFT), batch=batch, k=k, d=d,
                      prompt_len=9, max_new=8, reward_head=True)
    run_parity(make_setup(wl), steps=2, tol=TOL, tol_r=TOL)


@pytest.mark.parametrize("shape", [HD64, HD128], ids=["hd64", "hd128"])
@pytest.mark.parametrize("prompt_len", [952, 1016], ids=["16chunks", "17chunks"])
def test_verify_attention_with_a_block_per_chunk_and_past_it(shape, prompt_len):
    """65 verify rows whose 64-key chunks just fit one cluster (a chunk per block, one group of
    warps) and are one too many for it (blocks with two chunks, two groups)."""
    wl = synth.scaled(synth.TINY, dtype=synth.DTYPE_BF16, target=shape,
                      draft=synth.ModelShape(vocab=shape.vocab, **DRAFT), batch=1, k=13, d=4,
                      prompt_len=prompt_len, max_new=8, reward_head=True)
    run_parity(make_setup(wl), steps=2, tol=TOL, tol_r=TOL)


@pytest.mark.parametrize("max_chunk", [0, 65, 300])
def test_prefill_passes_above_256_rows(max_chunk):
    """Ragged prompts of 523 tokens in all, in passes of the default size, of 65 rows (remainder
    3) and of 300 rows."""
    wl = synth.scaled(synth.TINY, dtype=synth.DTYPE_BF16, target=HD64,
                      draft=synth.ModelShape(vocab=HD64.vocab, **DRAFT), batch=3, k=4, d=3,
                      prompt_len=260, max_new=8)
    run_parity(make_setup(wl, lens=[260, 63, 200]), steps=2, tol=TOL, tol_r=TOL,
               max_chunk=max_chunk)


@pytest.mark.parametrize("lens", [[240] * 7 + [241], [260] * 8], ids=["1921rows", "2080rows"])
def test_prefill_passes_of_many_row_tiles(lens):
    """One pass of more than 15 x 128 rows: gate/up and QKV, whose two accumulators are not allowed
    tiles of more than 128 rows here, need 16 and 17 row tiles where 256 rows would need 8 and 9."""
    wl = synth.scaled(synth.TINY, dtype=synth.DTYPE_BF16, target=HD64,
                      draft=synth.ModelShape(vocab=HD64.vocab, **DRAFT), batch=8, k=2, d=2,
                      prompt_len=260, max_new=8)
    run_parity(make_setup(wl, lens=lens), steps=1, tol=TOL, tol_r=TOL, max_chunk=4096)
