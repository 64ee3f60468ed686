"""Precision of the prefill attention of bf16 models, seen in the K/V cache that it fills.

A two-layer target whose first layer is attention alone (zero down projection): the second layer's V
rows are Wv RMSNorm(E[token] + Wo attention), and E, with gains of one, enters the first layer's
projections exactly (a bf16 value has no lo plane). So two roundings to hi and lo planes lie
between the prompt and the cache's second layer: the attention's output and the second layer's
input. Each is 2.4e-6 of the values' norm (2^-18 of a value at most), 3.4e-6 the two, and 4e-6
with an fp32 attention's own rounding (up to 2e-6 at scores of standard deviation 25). Queries and
keys in two bf16 planes, or a value sum that truncates over all chunks, are 6e-6 to 2.5e-5 off."""
import math

import numpy as np
import pytest

import synth
from cdsl_parity import Setup, make_engine

pytestmark = pytest.mark.gpu

REL = 5e-6


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2412_10418_gb300 import build
    build.build()


def setup(H, KVH, hd, lens, score):
    D = H * hd
    shape = synth.ModelShape(n_layers=2, d_model=D, n_heads=H, n_kv_heads=KVH, d_ffn=64, vocab=1024)
    small = synth.ModelShape(n_layers=1, d_model=64, n_heads=1, n_kv_heads=1, d_ffn=64, vocab=1024)
    wl = synth.scaled(synth.TINY, dtype=synth.DTYPE_BF16, target=shape, draft=small, batch=len(lens),
                      k=2, d=1, prompt_len=max(lens), max_new=4)
    t = synth.model_weights(wl, "target", device="host")
    rng = np.random.default_rng(11)
    # q and k of variance `score` each: scores of standard deviation `score`
    qk = math.sqrt(score) / math.sqrt(D)
    for name, std in (("wq", qk), ("wk", qk), ("wv", 1 / math.sqrt(D)), ("wo", 1 / math.sqrt(D))):
        for l in range(2):
            w = rng.normal(0, std, t[f"l{l}.{name}"].shape).astype(np.float32)
            t[f"l{l}.{name}"][:] = synth.f32_to_bf16_bits(w).reshape(w.shape)
    t["l0.w_down"][:] = 0
    return Setup(wl, t, synth.model_weights(wl, "draft", device="host"), synth.prompts(wl),
                 list(lens), synth.keywords(wl), synth.reward_head(wl))


def second_layer_v(s, b):
    """V of the second layer of prompt b in float64: [positions, KVH, hd]."""
    import torch
    sh = s.wl.target
    w = {n: v.double() for n, v in synth.to_torch(s.t_host, s.wl.dtype).items()}
    H, KVH, hd, n = sh.n_heads, sh.n_kv_heads, sh.head_dim, s.lens[b]
    norm = lambda x: x * torch.rsqrt(x.pow(2).mean(-1, keepdim=True) + sh.norm_eps)
    h = w["embed"][torch.from_numpy(s.prompts[b, :n].astype(np.int64)).cuda()]
    x = norm(h)
    half = hd // 2
    ang = (torch.arange(n, device="cuda", dtype=torch.float64)[:, None]
           * sh.rope_theta ** (-torch.arange(half, device="cuda", dtype=torch.float64) / half))
    cos, sin = ang.cos()[:, None], ang.sin()[:, None]

    def rope(y):
        a, c = y[..., :half], y[..., half:]
        return torch.cat([a * cos - c * sin, c * cos + a * sin], -1)

    q = rope((x @ w["l0.wq"].T).view(n, H, hd))
    k = rope((x @ w["l0.wk"].T).view(n, KVH, hd))
    v = (x @ w["l0.wv"].T).view(n, KVH, hd)
    mask = torch.ones(n, n, device="cuda", dtype=torch.bool).triu(1)
    out = torch.empty(n, H, hd, device="cuda", dtype=torch.float64)
    for i in range(H):
        g = i // (H // KVH)
        p = (q[:, i] @ k[:, g].T / math.sqrt(hd)).masked_fill(mask, -math.inf).softmax(-1)
        out[:, i] = p @ v[:, g]
    h = h + out.view(n, H * hd) @ w["l0.wo"].T
    return (norm(h) @ w["l1.wv"].T).view(n, KVH, hd)


@pytest.mark.parametrize("H,KVH,hd", [(4, 4, 64), (4, 1, 128)], ids=["hd64", "hd128"])
@pytest.mark.parametrize("lens,score", [([1000], 1.5), ([1000], 25.0), ([640, 333, 65], 5.0),
                                        ([3300], 1.5), ([384], 1.5), ([416], 1.5),
                                        ([160] * 8, 1.5), ([70] * 8, 1.5), ([3], 1.5)],
                         ids=["1000", "1000_peaked", "ragged", "3300", "384", "416", "8x160", "8x70",
                              "3"])
def test_prefill_attention_keeps_fp32_precision(H, KVH, hd, lens, score):
    """On both sides of the line between the CUDA-core and the tensor-core kernel (both head counts:
    384 and 416 rows, eight prompts of 70 and 160), full and ragged passes, continued ones (more
    than 1024 rows)."""
    s = setup(H, KVH, hd, lens, score)
    page = 64
    eng = make_engine(s, page_size=page)
    assert eng.status() == 0
    # the workspace begins with the target's pool [layer][page][K, V][kv head][slot][hd]; the
    # prompts' pages are handed out in order
    max_pages = (s.wl.prompt_len + s.wl.max_new + 1 + page - 1) // page
    n_pages = len(lens) * max_pages
    import torch
    pool = eng.ws[:4 * 2 * n_pages * 2 * KVH * page * hd].view(torch.float32)
    pool = pool.view(2, n_pages, 2, KVH, page, hd)
    first = 0
    for b, n in enumerate(lens):
        pages = (n + page - 1) // page
        got = pool[1, first:first + pages, 1].permute(0, 2, 1, 3).reshape(pages * page, KVH, hd)[:n]
        first += pages
        want = second_layer_v(s, b)
        rel = float((got.double() - want).norm() / want.norm())
        print(f"hd {hd} prompt of {n}, scores {score}: {rel:.2e}")
        assert rel <= REL, f"prompt {b}: {rel:.2e} off"
    eng.close()
