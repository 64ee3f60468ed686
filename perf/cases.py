"""What a user of the CDSL lookahead step has it do, as measurable cases.

Every case goes through the package's public entry points: an ``Engine`` (prefill, lookahead,
verify, select, step, tokens) over a target and a draft model, or ``cdsl_gemv_noalloc``. Kinds:

* ``generate``: a whole short request: prefill the prompts, run ``steps`` CDSL-k steps, read the
  tokens back (a service answering requests, or one with small models).
* ``first``: prefill the prompts, then the first step by its three calls with the logits
  returned (time to first token, and what an evaluation of the prompts' next tokens runs).
* ``split``: one step by its three calls on prefilled prompts, with the logits returned (a
  caller that looks at the verify pass, or brings its own reward).
* ``step``: one ``step`` on prefilled prompts (the decoding loop's body: one CUDA graph).
* ``gemv``: one weight-streaming product without device allocation.

Model shapes are the repository's own workloads: the tiny fp32 pair, the small bf16 pair (12
layers of 768 and 4 of 512), the 7B- and 13B-shaped targets with the 1B-shaped draft, at full
depth or as two-layer slices (the same launches, a tenth of the weights). Weights are N(0, 0.02),
gains near 1, prompt ids Zipf(1.1) as in natural text.
"""
import math

import torch

import paper_2412_10418_gb300 as cdsl

DEV = "cuda"


class Shape:
    """A pre-norm decoder's shape, as ``cdsl.model_cfg`` reads it."""

    rope_theta = 10000.0
    norm_eps = 1e-5

    def __init__(self, n_layers, d_model, n_heads, n_kv_heads, d_ffn, vocab):
        self.n_layers, self.d_model, self.n_heads = n_layers, d_model, n_heads
        self.n_kv_heads, self.d_ffn, self.vocab = n_kv_heads, d_ffn, vocab

    @property
    def head_dim(self):
        return self.d_model // self.n_heads

    def weight_shapes(self):
        """In the C ABI's order: embed, nine per layer, final norm, LM head."""
        D, F, hd = self.d_model, self.d_ffn, self.head_dim
        layer = [(D,), (self.n_heads * hd, D), (self.n_kv_heads * hd, D), (self.n_kv_heads * hd, D),
                 (D, self.n_heads * hd), (D,), (F, D), (F, D), (D, F)]
        return [(self.vocab, D)] + layer * self.n_layers + [(D,), (self.vocab, D)]

    def layer_params(self):
        D, hd = self.d_model, self.head_dim
        return self.n_layers * (2 * D * (self.n_heads + self.n_kv_heads) * hd + 3 * D * self.d_ffn)


# family: (target, draft, dtype, the repository's vocabulary and shapes)
FAMILIES = {
    "tiny": (Shape(2, 256, 4, 4, 688, 512), Shape(1, 128, 2, 2, 344, 512), "f32"),
    "small": (Shape(12, 768, 12, 12, 3072, 32000), Shape(4, 512, 8, 8, 2048, 32000), "bf16"),
    "7b": (Shape(32, 4096, 32, 8, 11008, 32000), Shape(16, 2048, 16, 4, 5504, 32000), "bf16"),
    "7b-2layer": (Shape(2, 4096, 32, 8, 11008, 32000), Shape(2, 2048, 16, 4, 5504, 32000), "bf16"),
    "13b": (Shape(40, 5120, 40, 8, 13824, 32000), Shape(16, 2048, 16, 4, 5504, 32000), "bf16"),
    "13b-2layer": (Shape(2, 5120, 40, 8, 13824, 32000), Shape(2, 2048, 16, 4, 5504, 32000), "bf16"),
}
NK = 5   # keywords per prompt


def engine_case(kind, family, batch, k, d, prompt, new, **more):
    """ragged: prompts of different lengths up to `prompt`; head: the composite reward;
    accept: 1 for speculative sampling; step1: the Step-1 budget; same: the draft is the target
    itself and every reward passes, so that whole lookaheads are emitted."""
    c = dict(kind=kind, family=family, batch=batch, k=k, d=d, prompt=prompt, new=new, steps=1,
             ragged=False, head=True, accept=0, step1=0, page=0, same=False)
    c.update(more)
    return c


def named(name, c):
    c["name"] = name
    return c


def listed():
    return [
        # a layer's product in a host framework that must not allocate (4096 -> 11008, 4 rows)
        named("gemv-4096x11008-r4", dict(kind="gemv", n=11008, k=4096, rows=4)),
        # the smallest request: fp32 models, 16 tokens after a 32-token prompt
        named("generate-tiny-fp32", engine_case("generate", "tiny", 1, 4, 4, 32, 16, steps=16, head=False)),
        # one interactive user of a small model whose drafts are accepted: several tokens a step
        named("generate-small-accepted", engine_case("generate", "small", 1, 4, 4, 128, 64, steps=12, same=True)),
        # the small model's decoding loop at the repository's batch
        named("step-small-b8", engine_case("step", "small", 8, 4, 4, 128, 256)),
        # a served batch of 32 ragged prompts: 640 verify rows, and their prefill
        named("first-small-b32", engine_case("first", "small", 32, 4, 4, 128, 64, ragged=True)),
        # the headline workload's decoding loop, full depth
        named("step-7b", engine_case("step", "7b", 1, 4, 4, 512, 128)),
        # time to first token of the headline workload
        named("first-7b", engine_case("first", "7b", 1, 4, 4, 512, 128)),
        # a wide verify pass (16 beams of 11 rows) over a long document
        named("split-7b-2layer-4k", engine_case("split", "7b-2layer", 1, 16, 10, 4096, 128)),
        # every decoding option at once: two prompts of different lengths, k = 3, d = 5 as in the
        # paper's HH-RLHF runs, speculative sampling, Step-1 budget 2, 16-token pages
        named("step-7b-2layer-options", engine_case("step", "7b-2layer", 2, 3, 5, 700, 128, ragged=True,
                                                    accept=1, step1=2, page=16)),
        # four long prompts and 224 verify rows on the largest model, full depth
        named("step-13b", engine_case("step", "13b", 4, 8, 6, 1024, 256)),
        # the same launches with ragged prompts: prefill of about 3,500 tokens and the first step
        named("first-13b-2layer", engine_case("first", "13b-2layer", 4, 8, 6, 1024, 256, ragged=True)),
    ]


def log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    family = rng.choice(["gemv", "tiny", "small", "small", "7b-2layer", "7b-2layer", "13b-2layer"])
    if family == "gemv":
        return dict(kind="gemv", n=log_int(rng, 500, 32768), k=8 * log_int(rng, 32, 1024),
                    rows=rng.randint(1, 8))
    kind = rng.choice(["generate", "step", "first", "split"])
    rows = {"tiny": 160, "small": 640, "7b-2layer": 320, "13b-2layer": 256}[family]
    if kind == "generate":
        rows = min(rows, 256)
    tokens = {"tiny": 256, "small": 4096, "7b-2layer": 8192, "13b-2layer": 4096}[family]
    while True:
        batch, k, d = log_int(rng, 1, 32), rng.randint(1, 16), rng.randint(1, 10)
        if batch * k * (d + 1) <= rows:
            break
    prompt = log_int(rng, 16, max(17, min(4096, tokens // batch)))
    more = {}
    if kind == "generate":
        more["steps"] = rng.randint(2, 8)
    return engine_case(kind, family, batch, k, d, prompt, rng.choice([32, 64, 128]),
                       ragged=rng.random() < 0.5, head=kind != "generate" or rng.random() < 0.5,
                       accept=int(rng.random() < 0.25), step1=rng.choice([0, 0, 0, 1, 2]) if kind == "step" else 0,
                       page=rng.choice([0, 0, 16, 128]), same=kind == "generate" and rng.random() < 0.3, **more)


# ---------------------------------------------------------------------------- inputs

def models(case):
    target, draft, dtype = FAMILIES[case["family"]]
    return target, (target if case["same"] else draft), dtype


def weights_of(shape, dtype, g):
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    out = []
    for s in shape.weight_shapes():
        w = torch.empty(s, dtype=dt, device=DEV)
        out.append(w.normal_(1.0, 0.05, generator=g) if len(s) == 1 else w.normal_(0.0, 0.02, generator=g))
    return out


def lengths_of(case):
    P = case["prompt"]
    if not case["ragged"]:
        return [P] * case["batch"]
    return [P - (b * 37) % (P // 2 + 1) for b in range(case["batch"])]


def zipf_cdf(V):
    """Of ids in [0, V), made on the host: a sum in a fixed order."""
    cdf = torch.arange(1, V + 1, dtype=torch.float64).pow(-1.1).cumsum(0)
    return cdf / cdf[-1]


def inputs(case, seed):
    """The models' weights, the prompts and their keywords, from the seed alone."""
    target, draft, dtype = models(case)
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    tw = weights_of(target, dtype, g)
    dw = tw if case["same"] else weights_of(draft, dtype, g)
    V, B = target.vocab, case["batch"]
    u = torch.rand(B * case["prompt"], generator=g, device=DEV, dtype=torch.float64)
    prompts = torch.searchsorted(zipf_cdf(V).to(DEV), u).clamp_(max=V - 1)
    kw = torch.rand(B, V, generator=g, device=DEV).topk(NK, dim=1).indices
    head = torch.empty(target.d_model, device=DEV).normal_(0.0, 0.02, generator=g)
    return tw, dw, prompts.view(B, -1).int().contiguous(), kw.int().contiguous(), head


_stream = []   # one for all engines, as a program has that serves one request after another


def prepare(case, seed):
    if case["kind"] == "gemv":
        g = torch.Generator(device=DEV)
        g.manual_seed(int(seed))
        w = torch.empty(case["n"], case["k"], dtype=torch.bfloat16, device=DEV).normal_(0.0, 0.02, generator=g)
        x = torch.randn(case["rows"], case["k"], generator=g, device=DEV)
        return dict(case=case, w=w, x=x, y=torch.empty(case["rows"], case["n"], device=DEV),
                    stream=torch.cuda.current_stream().cuda_stream)
    target, draft, dtype = models(case)
    tw, dw, prompts, kw, head = inputs(case, seed)
    a_t, r_t = (0.3, 0.0) if case["same"] else (0.3, 0.3)
    if not _stream:
        _stream.append(torch.cuda.Stream(device=DEV))
    eng = cdsl.Engine(target, draft, dtype, tw, dw, batch=case["batch"], k=case["k"], d=case["d"],
                      max_prompt=case["prompt"], max_new=case["new"], n_keywords=NK, a_t=a_t, r_t=r_t,
                      reward_head=head if case["head"] else None, page_size=case["page"],
                      acceptance=case["accept"], seed=int(seed) & 0xFFFF, step1_budget=case["step1"],
                      stream=_stream[0])
    s = dict(case=case, eng=eng, prompts=prompts, kw=kw, lens=lengths_of(case))
    if case["kind"] in ("first", "split"):
        s["logits"] = torch.zeros(case["batch"], case["k"], case["d"] + 1, target.vocab, device=DEV)
    torch.cuda.synchronize()   # the engine works on a stream of its own
    if case["kind"] in ("step", "split"):
        eng.prefill(prompts, s["lens"], kw)
    return s


# ---------------------------------------------------------------------------- one pass

def decided(eng):
    return dict(beam=eng.beam, state=eng.state, emitted=eng.emitted, n_emitted=eng.n_emitted,
                reward=eng.reward)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "gemv":
        cdsl.cdsl_gemv_noalloc(s["w"], s["x"], s["y"], s["stream"])
        return s["y"]
    eng = s["eng"]
    if kind == "step":
        eng.step()
        return decided(eng)
    if kind == "generate":
        eng.prefill(s["prompts"], s["lens"], s["kw"])
        for _ in range(case["steps"]):
            eng.step()
        tokens, lengths = eng.tokens()
        return dict(decided(eng), tokens=tokens, lengths=lengths)
    if kind == "first":
        eng.prefill(s["prompts"], s["lens"], s["kw"])
    eng.lookahead()
    eng.verify(s["logits"])
    eng.select()
    return dict(decided(eng), roots=eng.roots, draft_tok=eng.draft_tok, logq=eng.logq, logp=eng.logp,
                argmax=eng.argmax, n_accept=eng.n_accept, logits=s["logits"])


# ---------------------------------------------------------------------------- its work

def work(case):
    """Each weight that a pass needs once per forward pass (the d draft calls are serial), the
    fp32 K/V cache read once per forward pass, logits written where they are returned."""
    if case["kind"] == "gemv":
        n, k, r = case["n"], case["k"], case["rows"]
        return dict(bytes=2 * n * k + 4 * r * (n + k), flops=2 * n * k * r)
    target, draft, dtype = models(case)
    size = 2 if dtype == "bf16" else 4
    B, k, d = case["batch"], case["k"], case["d"]
    keys = sum(lengths_of(case))

    def forward(m, rows, lm_rows, keys):
        lm = m.vocab * m.d_model
        by = size * (m.layer_params() + (lm if lm_rows else 0))
        by += 8 * keys * m.n_layers * m.n_kv_heads * m.head_dim
        fl = 2 * rows * m.layer_params() + 2 * lm_rows * lm
        fl += 4 * rows * (keys / B) * m.n_layers * m.n_heads * m.head_dim
        return by, fl

    passes = []
    if case["kind"] in ("first", "generate"):
        passes += [forward(target, keys, B, keys), forward(draft, keys, 0, keys)]
        half = 2 * keys * (keys / B)   # causal: half of the keys
        passes += [(0, -half * m.n_layers * m.n_heads * m.head_dim) for m in (target, draft)]
    for _ in range(case["steps"]):
        passes += [forward(draft, B * k, B * k, keys)] * d + [forward(target, B * k * (d + 1), B * k * (d + 1), keys)]
        if case["step1"] == 2:
            passes += [forward(draft, B, B, keys)] * d + [forward(target, B * (d + 2), B, keys)]
    out = 4 * B * k * (d + 1) * target.vocab if case["kind"] in ("first", "split") else 0
    return dict(bytes=sum(p[0] for p in passes) + out, flops=sum(p[1] for p in passes))


# ---------------------------------------------------------------------------- how near is right

def tolerance(case):
    """Four times what was measured against 64 bits. The gemv's activations are bf16 hi and lo
    planes: 2.5e-6. fp32 models: below 2e-6. bf16 models run their activations as hi and lo planes
    too: logits 6e-6 (two layers) to 5.5e-5 (32 layers). Whole values are tokens and counts: the
    share is one flipped near tie of a verify pass's argmax."""
    if case["kind"] == "gemv":
        return dict(rel=1e-5)
    if case["family"] == "tiny":
        return dict(rel=1e-5, differ=0.005)
    return dict(rel=2.4e-4, differ=0.005)


# ---------------------------------------------------------------------------- in 64 bits

class Decoder:
    """The decoder in float64: plain torch, weights widened where they are used."""

    def __init__(self, shape, weights):
        self.s, self.w = shape, weights

    def norm(self, x, g):
        return x * torch.rsqrt(x.pow(2).mean(-1, keepdim=True) + self.s.norm_eps) * g.double()

    def rope(self, x, start):
        half = x.shape[-1] // 2
        inv = self.s.rope_theta ** (-torch.arange(half, device=DEV, dtype=torch.float64) / half)
        ang = (start + torch.arange(x.shape[1], device=DEV, dtype=torch.float64))[:, None] * inv
        cos, sin = ang.cos()[None, :, None, :], ang.sin()[None, :, None, :]
        a, b = x[..., :half], x[..., half:]
        return torch.cat([a * cos - b * sin, b * cos + a * sin], dim=-1)

    def extend(self, tokens, past=None):
        """tokens [n, t] after the cached positions; past: per layer (K, V) of one sequence (shared
        by all n) or of each. Returns the final-normed hidden states [n, t, D] and the new cache."""
        s, w = self.s, self.w
        n, t = tokens.shape
        H, KVH, hd = s.n_heads, s.n_kv_heads, s.head_dim
        start = past[0][0].shape[1] if past else 0
        h = w[0][tokens].double()
        new = []
        for l in range(s.n_layers):
            g1, wq, wk, wv, wo, g2, wg, wu, wd = w[1 + 9 * l: 10 + 9 * l]
            a = self.norm(h, g1)
            q = self.rope((a @ wq.double().T).view(n, t, H, hd), start)
            K = self.rope((a @ wk.double().T).view(n, t, KVH, hd), start)
            V = (a @ wv.double().T).view(n, t, KVH, hd)
            if past:
                K = torch.cat([past[l][0].expand(n, -1, -1, -1), K], dim=1)
                V = torch.cat([past[l][1].expand(n, -1, -1, -1), V], dim=1)
            new.append((K, V))
            T = K.shape[1]
            hidden = torch.arange(T, device=DEV)[None, :] > start + torch.arange(t, device=DEV)[:, None]
            att = torch.empty(n, t, H, hd, device=DEV, dtype=torch.float64)
            for kv in range(KVH):
                hs = slice(kv * (H // KVH), (kv + 1) * (H // KVH))
                sc = torch.einsum("nthd,nTd->nhtT", q[:, :, hs], K[:, :, kv]) / math.sqrt(hd)
                p = sc.masked_fill(hidden, -math.inf).softmax(-1)
                att[:, :, hs] = torch.einsum("nhtT,nTd->nthd", p, V[:, :, kv])
            h = h + att.view(n, t, H * hd) @ wo.double().T
            a = self.norm(h, g2)
            h = h + (torch.nn.functional.silu(a @ wg.double().T) * (a @ wu.double().T)) @ wd.double().T
        return self.norm(h, w[-2]), new

    def logits(self, hf):
        return hf @ self.w[-1].double().T


def uniform24(seed, c):
    """Draw c of SplitMix64 (Steele, Lea, Flood 2014), its top 24 bits over 2^24."""
    m = (1 << 64) - 1
    z = (seed + (c + 1) * 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return ((z ^ (z >> 31)) >> 40) / float(1 << 24)


def exact_step(case, seed, tgt, drf, head, kw, prompts, states, step):
    """One CDSL-k step of every prompt; states[b]: dict(T, tc, dc, roots). Returns the step's
    outputs, or the float ones alone with a Step-1 budget (which changes emissions only)."""
    B, k, d, same = case["batch"], case["k"], case["d"], case["same"]
    a_t, r_t = (0.3, 0.0) if same else (0.3, 0.3)
    n_min = next(n for n in range(d + 1) if torch.tensor(n / d).float() >= torch.tensor(a_t).float())
    rows = {q: [] for q in ("roots", "draft_tok", "logq", "logp", "argmax", "n_accept", "logits", "reward",
                            "beam", "state", "emitted", "n_emitted")}
    for b, st in enumerate(states):
        left = case["new"] - len(st["T"])
        if left <= 0:
            rows["reward"].append(torch.zeros(k, 2, device=DEV, dtype=torch.float64))
            rows["beam"].append(-1), rows["state"].append(0), rows["n_emitted"].append(0)
            rows["emitted"].append([-1] * (d + 1))
            continue
        roots = st["roots"]
        x, logq, past, tok = [], [], st["dc"], roots[:, None]
        for _ in range(d):
            hf, past = drf.extend(tok, past)
            lq = drf.logits(hf[:, -1]).log_softmax(-1)
            best = lq.max(-1)
            logq.append(best.values), x.append(best.indices)
            tok = best.indices[:, None]
        x, logq = torch.stack(x, 1), torch.stack(logq, 1)
        hf, _ = tgt.extend(torch.cat([roots[:, None], x], 1), st["tc"])
        lg = tgt.logits(hf)
        logp = lg[:, :d].log_softmax(-1).gather(-1, x[..., None])[..., 0]
        amax = lg.argmax(-1)
        n_acc, reward = [], torch.zeros(k, 2, device=DEV, dtype=torch.float64)
        score = torch.sigmoid(hf @ head.double())
        words = set(kw[b].tolist())
        for i in range(k):
            n = 0
            while n < d:
                if case["accept"]:
                    u = uniform24(seed & 0xFFFF, ((step * B + b) * k + i) * d + n)
                    ok = u == 0.0 or math.log(u) <= float(logp[i, n] - logq[i, n])
                else:
                    ok = bool(amax[i, n] == x[i, n])
                if not ok:
                    break
                n += 1
            n_acc.append(n)
            for q, upto in ((0, d), (1, n)):
                said = set(st["T"]) | {int(roots[i])} | set(x[i, :upto].tolist())
                reward[i, q] = len(words & said) / NK
                if case["head"]:
                    reward[i, q] = 0.5 * reward[i, q] + 0.5 * score[i, upto]
        win = int(reward[:, 0].argmax())
        s1 = n_acc[win] >= n_min and float(reward[win, 1]) >= r_t
        emit = [int(roots[win])] + (x[win, :n_acc[win]].tolist() if s1 else [])
        emit = emit[:left]
        rows["roots"].append(roots), rows["draft_tok"].append(x), rows["logq"].append(logq)
        rows["logp"].append(logp), rows["argmax"].append(amax), rows["logits"].append(lg)
        rows["n_accept"].append(torch.tensor(n_acc)), rows["reward"].append(reward), rows["beam"].append(win)
        rows["state"].append(1 if s1 else 2 if n_acc[win] < n_min else 4)
        rows["emitted"].append(emit + [-1] * (d + 1 - len(emit))), rows["n_emitted"].append(len(emit))
        st["T"] += emit
        more = torch.tensor([emit], device=DEV)
        if case["steps"] > 1:
            hf, st["tc"] = tgt.extend(more, st["tc"])
            _, st["dc"] = drf.extend(more, st["dc"])
            st["roots"] = tgt.logits(hf[:, -1]).topk(k, dim=-1).indices[0]
    out = {q: (torch.stack(v) if isinstance(v[0], torch.Tensor) else torch.tensor(v)) for q, v in rows.items() if v}
    return {q: (v if v.is_floating_point() else None) for q, v in out.items()} if case["step1"] else out


@torch.no_grad()
def exact(case, seed):
    if case["kind"] == "gemv":
        s = prepare(case, seed)
        return s["x"].double() @ s["w"].double().T
    target, draft, _ = models(case)
    keys = sum(lengths_of(case))
    if 2 * keys * (target.layer_params() + draft.layer_params()) > 1.2e13:
        return None   # more than about 20 seconds at the card's 64-bit rate
    tw, dw, prompts, kw, head = inputs(case, seed)
    tgt, drf = Decoder(target, tw), Decoder(draft, dw)
    states = []
    for b, n in enumerate(lengths_of(case)):
        ids = prompts[b: b + 1, :n].long()
        hf, tc = tgt.extend(ids)
        _, dc = drf.extend(ids)
        states.append(dict(T=[], tc=tc, dc=dc, roots=tgt.logits(hf[:, -1]).topk(case["k"], dim=-1).indices[0]))
    for step in range(case["steps"]):
        out = exact_step(case, int(seed), tgt, drf, head, kw, prompts, states, step)
    want = ["beam", "state", "emitted", "n_emitted", "reward"]
    if case["kind"] in ("first", "split"):
        want += ["roots", "draft_tok", "logq", "logp", "argmax", "n_accept", "logits"]
    out = {q: out[q] for q in want}
    if case["kind"] == "generate":
        W = case["prompt"] + case["new"]
        out["tokens"] = torch.full((case["batch"], W), -1)
        for b, n in enumerate(lengths_of(case)):
            ids = prompts[b, :n].tolist() + states[b]["T"]
            out["tokens"][b, :len(ids)] = torch.tensor(ids)
        out["lengths"] = torch.tensor([n + len(states[b]["T"]) for b, n in enumerate(lengths_of(case))])
    return out
