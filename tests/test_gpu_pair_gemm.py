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


def ragged(hd, heads, kv_heads, d_ffn):
    return synth.ModelShape(n_layers=2, d_model=hd * heads, n_heads=heads, n_kv_heads=kv_heads,
                            d_ffn=d_ffn, vocab=1032)


@pytest.mark.parametrize("shape,batch", [(ragged(64, 30, 3, 3136), 1), (ragged(64, 30, 3, 3136), 2),
                                         (ragged(64, 30, 3, 3136), 4), (ragged(64, 30, 3, 3136), 8),
                                         (ragged(128, 15, 5, 3136), 1), (ragged(128, 15, 5, 3136), 4),
                                         (ragged(64, 17, 17, 8512), 1), (ragged(64, 17, 17, 8512), 4)],
                         ids=lambda v: f"{v.d_model}x{v.d_ffn}" if hasattr(v, "d_ffn") else f"{65 * v}rows")
def test_chains_and_splits_on_ragged_shapes(shape, batch):
    """K ranges of 17 to 133 blocks, whole and split over two to four pairs, in one chain and in
    several of uneven lengths, their lo planes apart and not; features and rows that fill neither
    the weight tiles nor the row tiles. (On 152 SMs: gate/up whole in chains of 4, 5 and 10 blocks, in
    two in chains of 4 and 5 and in four; down in two to four with chains of 7, 12 and 24 and without;
    QKV and O in two with chains, in three and four without.)"""
    wl = synth.scaled(synth.TINY, dtype=synth.DTYPE_BF16, target=shape,
                      draft=synth.ModelShape(vocab=shape.vocab, **DRAFT), batch=batch, k=13, d=4,
                      prompt_len=9, max_new=8, reward_head=True)
    run_parity(make_setup(wl), steps=1, tol=TOL, tol_r=TOL)


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


def exactness_engine(D, d_ffn, batch, k, d, ffn_scale):
    """One layer of zero attention output; the FFN's output ffn_scale times the embedding's norm (0:
    none). Returns the engine after verify, its logits and the same in float64."""
    import torch
    import paper_2412_10418_gb300 as cdsl

    V = 32000
    shape = synth.ModelShape(n_layers=1, d_model=D, n_heads=D // 128, n_kv_heads=2 if D == 768 else 4,
                             d_ffn=d_ffn, vocab=V)
    small = synth.ModelShape(n_layers=1, d_model=128, n_heads=2, n_kv_heads=1, d_ffn=192, vocab=V)
    g = torch.Generator(device="cuda").manual_seed(D + d_ffn + batch * k * d)

    def weights(sh):
        out = {}
        for name, s in sh.weight_specs():
            w = torch.ones(s, device="cuda") if len(s) == 1 else torch.randn(
                s, generator=g, device="cuda")
            out[name] = (w if len(s) == 1 else w * s[1] ** -0.5).bfloat16()
        return out

    tw, dw = weights(shape), weights(small)
    for name in ("l0.ffn_norm", "final_norm"):
        tw[name] = (1 + 0.1 * torch.randn(D, generator=g, device="cuda")).bfloat16()
    tw["l0.wo"].zero_()
    tw["embed"].mul_(D ** 0.5)          # of unit rms; the FFN's output: about 0.35 before the scale
    tw["l0.w_down"].mul_(ffn_scale / 0.35)
    eng = cdsl.Engine(shape, small, synth.DTYPE_BF16, [tw[n] for n, _ in shape.weight_specs()],
                      [dw[n] for n, _ in small.weight_specs()], batch=batch, k=k, d=d, max_prompt=8,
                      max_new=4, n_keywords=1, a_t=0.3, r_t=0.3)
    prompts = torch.randint(0, V, (batch, 8), generator=g, device="cuda")
    torch.cuda.synchronize()   # (the engine works on a stream of its own)
    eng.prefill(prompts, [8] * batch, torch.zeros(batch, 1, dtype=torch.int32))
    eng.lookahead()
    got = torch.empty(batch, k, d + 1, V, device="cuda")
    eng.verify(got)
    eng.stream.synchronize()
    assert eng.status() == 0
    tok = torch.cat([eng.roots[..., None], eng.draft_tok], -1).long()
    norm = lambda x: x * torch.rsqrt(x.pow(2).mean(-1, keepdim=True) + shape.norm_eps)
    h = tw["embed"][tok].double()
    x = norm(h) * tw["l0.ffn_norm"].double()
    a = torch.nn.functional.silu(x @ tw["l0.w_gate"].double().T) * (x @ tw["l0.w_up"].double().T)
    h = h + a @ tw["l0.w_down"].double().T
    return got, norm(h) * tw["final_norm"].double() @ tw["lm_head"].double().T


@pytest.mark.parametrize("D", [768, 4096])
@pytest.mark.parametrize("batch,k,d", [(1, 13, 4), (1, 16, 9), (1, 16, 13), (2, 16, 9), (4, 16, 15)],
                         ids=["65rows", "160rows", "224rows", "320rows", "1024rows"])
def test_sums_are_as_exact_as_a_serial_fp32_sum(D, batch, k, d):
    """Logits of a model that is its embedding and its LM head: a bf16 embedding times a bf16 gain has
    16 bits, which the hi and lo planes hold exactly, so what is off is the sum over K alone (and the
    row's scale, 1e-7). The bound is the rounding of a serial fp32 sum, 1.8e-8 sqrt(K), or the 5.6e-7
    that chains of four K blocks may take."""
    got, want = exactness_engine(D, 64, batch, k, d, 0.0)
    rel = float((got.double() - want).norm() / want.norm())
    bound = max(1.8e-8 * D ** 0.5, 5.6e-7) + 1e-7
    print(f"K {D}, {batch * k * (d + 1)} rows: {rel:.2e}, bound {bound:.2e}")
    assert rel <= bound


@pytest.mark.parametrize("batch,k,d", [(1, 13, 4), (1, 16, 9), (1, 16, 13), (4, 16, 15)],
                         ids=["65rows", "160rows", "224rows", "1024rows"])
def test_gate_up_sums_do_not_shrink(batch, k, d):
    """An FFN whose output is as large as the embedding that it is added to: where gate and up fall
    short by s each, the hidden state turns by about s. Two roundings to hi and lo planes (the
    activation, 2.4e-6 of half of the state's square, and the LM head's input, 2.4e-6) leave 3e-6;
    5e-6 is the bound. Gate and up in one chain over K = 4096 are 7e-6 off and more."""
    got, want = exactness_engine(4096, 11008, batch, k, d, 1.0)
    rel = float((got.double() - want).norm() / want.norm())
    print(f"{batch * k * (d + 1)} rows: {rel:.2e}")
    assert rel <= 5e-6
