"""Performance cases of the LSP decoder: what a program that decodes with this library has it do.

Three kinds of case, all through the public binding:

  decode   one whole decode from host memory (LSPDecoder.generate_host): prompt in, finished tokens out
  pass     one step of the decode loop (LSPDecoder.denoise_step + scores) in the state a decode reaches: the prompt's own
           first pass, or a later one with `pend` rows of the last committed block and `left` positions still masked
  head     the fused LM head + confidence reduction + scan alone on hidden states (LSPDecoder.head_scan)

Model shapes are the benchmark's (the two 7-8B-parameter shapes, bf16), its tiny fp32 model, and the small bf16 models of
the tests.  Weights are random and fixed; the prompts come from the seed.

A random model's predictions hang on rounding: among 126464 nearly equal logits bf16 noise alone decides one argmax in
twenty, and a decode's trajectory with it.  A trained model's do not.  So the weights here carry what induction heads give
a trained model: a few heads of the first layer look `gen` positions back (through the rotary phases), and the LM head
knows the code they write, so a masked position predicts the token `gen` positions earlier.  Seven of eight ids are
predicted with confidence well above the threshold and one of eight well below it, and 12 % of the text are delimiters:
blocks of a few tokens, ended by a delimiter or by the first doubtful position, as on text.  Every other weight is random
with the usual 1/sqrt(2 n_layers) on the projections that write the residual stream.
"""
import math
from types import SimpleNamespace

import torch

from paper_2603_05454_b200 import LSPDecoder, SchedCfg

DEV = "cuda:0"

# n_layers, d_model, n_heads, n_kv_heads, head_dim, d_ffn, vocab, rope_theta, dtype
SHAPES = {
    "llada": (32, 4096, 32, 32, 128, 12288, 126464, 1e4, "bf16"),
    "dream": (28, 3584, 28, 4, 128, 18944, 152064, 1e6, "bf16"),
    "tiny": (2, 256, 4, 4, 64, 1024, 2048, 1e4, "fp32"),
    "small": (2, 512, 4, 2, 128, 1024, 4096, 1e4, "bf16"),
    "small64": (3, 512, 8, 4, 64, 1024, 4096, 1e4, "bf16"),
    # head-only: the LM heads of the two large shapes (layers are never run)
    "llada_head": (1, 4096, 1, 1, 128, 64, 126464, 1e4, "bf16"),
    "dream_head": (1, 3584, 1, 1, 128, 64, 152064, 1e6, "bf16"),
}
DELIMS = (1, 32)          # delimiter ids
BLOCK = 3.2               # mean committed block of a decode (measured on the large model), for work()


def listed():
    return [
        # the smallest use: a tiny fp32 model, batch 1, some thirty passes in which launches and latency are everything
        dict(name="tiny_decode", kind="decode", model="tiny", batch=1, prompt=64, gen=64, topology=0, inplace=0, lagged=0),
        # a small grouped-query bf16 model serving a ragged batch of three short sequences, K/V written in place, block
        # lengths kept on the device
        dict(name="small_decode", kind="decode", model="small", batch=3, prompt=75, gen=53, topology=0, inplace=1, lagged=1),
        # the tail of a batch-1 decode: a handful of rows, every pass streams all weights
        dict(name="llada_tail", kind="pass", model="llada", batch=1, prompt=256, gen=256, pend=3, left=6),
        # the second half of a batch-1 decode
        dict(name="llada_late", kind="pass", model="llada", batch=1, prompt=256, gen=256, pend=5, left=96),
        # the first half of a batch-1 decode
        dict(name="llada_mid", kind="pass", model="llada", batch=1, prompt=256, gen=256, pend=8, left=179),
        # the first pass of a batch-1 decode: prompt and all masked positions
        dict(name="llada_first", kind="pass", model="llada", batch=1, prompt=256, gen=256, pend=256, left=256),
        # the whole batch-1 decode, from host memory to host memory
        dict(name="llada_decode", kind="decode", model="llada", batch=1, prompt=256, gen=256, topology=0, inplace=0, lagged=0),
        # the scattered-acceptance baseline the method is compared with: top-32 acceptance, the region recomputed each pass
        dict(name="llada_scattered", kind="decode", model="llada", batch=1, prompt=256, gen=256, topology=1, inplace=0, lagged=0),
        # a ragged batch of four in the middle of its decode, grouped-query attention, about a thousand rows
        dict(name="dream_mid", kind="pass", model="dream", batch=4, prompt=512, gen=512, pend=7, left=251),
        # the first pass of that batch: four times 512 prompt and 512 masked positions
        dict(name="dream_first", kind="pass", model="dream", batch=4, prompt=512, gen=512, pend=512, left=512),
        # a long batch of sixteen half-way through: eight thousand rows over two thousand keys each
        dict(name="llada_batch16", kind="pass", model="llada", batch=16, prompt=1070, gen=1024, pend=6, left=509),
        # the fused head alone on eight times 1024 hidden states
        dict(name="head_8x1024", kind="head", model="llada_head", batch=8, rows=1024),
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["pass", "pass", "pass", "decode", "decode", "head"])
    if kind == "head":
        return dict(kind="head", model=rng.choice(["llada_head", "dream_head"]), batch=rng.randint(1, 8), rows=_logint(rng, 1, 900))
    if kind == "decode":
        model = rng.choice(["tiny", "small", "small64", "llada"])
        top = 1 if rng.random() < 0.2 else 0
        gen = rng.randint(16, 80)
        batch = 1 if model == "llada" else rng.randint(1, 6)
        return dict(kind="decode", model=model, batch=batch, prompt=gen + rng.randint(0, 120), gen=gen, topology=top,
                    inplace=rng.randint(0, 1), lagged=0 if top else rng.randint(0, 1))
    model = rng.choice(["llada", "llada", "dream"])
    first = rng.random() < 0.2
    batch = _logint(rng, 1, 4 if first else 8)
    gen = 16 * batch + _logint(rng, 24, 512)
    prompt = gen + rng.randint(0, 512)
    if first:
        return dict(kind="pass", model=model, batch=batch, prompt=prompt, gen=gen, pend=prompt, left=gen)
    pend = rng.randint(1, 16)
    return dict(kind="pass", model=model, batch=batch, prompt=prompt, gen=gen, pend=pend, left=_logint(rng, 2, gen - 5 * (batch - 1) - pend - 1))


# ---- model -----------------------------------------------------------------------------------------------------
_models = {}              # the last model built: a serving process holds one model and many decodes


def _shape(name):
    L, d, hq, hkv, dh, f, v, theta, dt = SHAPES[name]
    return SimpleNamespace(n_layers=L, d_model=d, n_heads=hq, n_kv_heads=hkv, head_dim=dh, d_ffn=f, vocab=v, rms_eps=1e-5,
                           rope_theta=theta, dtype=dt, mask_id=v - 1)


def _unsure(v):
    """Ids the model predicts with low confidence: one in eight."""
    return torch.arange(v, device=DEV) % 8 == 5


def _model(name):
    if name in _models:
        return _models[name]
    _models.clear()
    sh = _shape(name)
    dt = torch.float32 if sh.dtype == "fp32" else torch.bfloat16
    gen = torch.Generator(device=DEV).manual_seed(1)

    def rnd(*size, std):
        return torch.empty(*size, dtype=dt, device=DEV).normal_(0.0, std, generator=gen)

    d, hq, hkv, dh, f, v = sh.d_model, sh.n_heads, sh.n_kv_heads, sh.head_dim, sh.d_ffn, sh.vocab
    one = torch.ones(d, dtype=dt, device=DEV)
    if name.endswith("_head"):
        z = lambda *s: torch.zeros(*s, dtype=dt, device=DEV)  # noqa: E731
        w = dict(embed=z(8, d), w_head=rnd(v, d, std=0.12), final_norm=one,
                 layers=[dict(attn_norm=one, w_qkv=z((hq + 2 * hkv) * dh, d), w_o=z(d, hq * dh), ffn_norm=one, w_gate=z(f, d),
                              w_up=z(f, d), w_down=z(d, f))])
        _models[name] = (sh, w)
        return _models[name]
    std = 1.28 / math.sqrt(d)                             # 0.02 at d_model 4096
    res = std / math.sqrt(2 * sh.n_layers)
    embed = rnd(v, d, std=0.02)
    embed[:, 0] = 8 * 0.02                                # a constant feature, as trained models have
    layers = [dict(attn_norm=one, ffn_norm=one, w_qkv=rnd((hq + 2 * hkv) * dh, d, std=std), w_o=rnd(d, hq * dh, std=res),
                   w_gate=rnd(f, d, std=std), w_up=rnd(f, d, std=std), w_down=rnd(d, f, std=res)) for _ in range(sh.n_layers)]
    # copying heads of layer 0: query head 0 of the first KV heads' groups (their query / key rows are set in _copy_heads,
    # which needs the distance); what they write, per token id, is the code the LM head reads
    nc = min(4, hkv)
    w_o = layers[0]["w_o"]
    w_v = layers[0]["w_qkv"][(hq + hkv) * dh:]
    cols = torch.cat([torch.arange(dh, device=DEV) + h * (hq // hkv) * dh for h in range(nc)])
    w_o[:, cols] = rnd(d, nc * dh, std=2.0 / (1.28 * math.sqrt(nc * dh)))
    head = torch.empty(v, d, dtype=dt, device=DEV)
    lse = math.log(v) + 0.7                               # of the other ids' logits
    b = torch.where(_unsure(v), lse - 2.3, lse + 9.0) / 0.8
    for i in range(0, v, 16384):
        e = embed[i:i + 16384].float()
        e = (e / e.square().mean(1, keepdim=True).sqrt()).to(dt)
        code = ((e @ w_v[:nc * dh].t()) @ w_o[:, cols].t()).float()
        code = code / code.square().mean(1, keepdim=True).sqrt()
        head[i:i + 16384] = (code * (b[i:i + 16384, None] / d) + rnd(len(e), d, std=0.6 / math.sqrt(d)).float()).to(dt)
    w = dict(embed=embed, w_head=head, final_norm=one, layers=layers)
    _models[name] = (sh, w)
    return _models[name]


def _copy_heads(sh, w, dist):
    """The weights with layer 0's copying heads set to look `dist` positions back: constant query and key vectors (they read
    the constant feature only) whose rotary phases meet at that distance."""
    hq, hkv, dh = sh.n_heads, sh.n_kv_heads, sh.head_dim
    first = dict(w["layers"][0])
    wq = first["w_qkv"] = first["w_qkv"].clone()
    g = 9.5 / 8.0
    for h in range(min(4, hkv)):
        q0, k0 = h * (hq // hkv) * dh, (hq + h) * dh
        wq[q0:q0 + dh] = 0
        wq[k0:k0 + dh] = 0
        for i in range(dh // 8):
            a = dist * sh.rope_theta ** (-2.0 * i / dh)
            wq[q0 + i, 0] = g
            wq[k0 + i, 0] = g * math.cos(a)
            wq[k0 + dh // 2 + i, 0] = g * math.sin(a)
    return dict(w, layers=[first] + w["layers"][1:])


def _delim_bitmap(v):
    bits = torch.zeros(v, dtype=torch.uint8)
    bits[DELIMS[0]:DELIMS[1] + 1] = 1
    bits = torch.nn.functional.pad(bits, (0, -v % 8)).view(-1, 8)
    return (bits * (2 ** torch.arange(8, dtype=torch.uint8))).sum(1).to(torch.uint8).to(DEV)


def _lengths(c):
    """Prompt and generation lengths of a batch: ragged."""
    return [c["prompt"] + 3 * b for b in range(c["batch"])], [c["gen"] - 5 * b for b in range(c["batch"])]


def _passes(c):
    """(rows, keys, masked rows) per sequence of every pass of the case."""
    p, g = _lengths(c)
    if c["kind"] == "pass":
        first = c["pend"] == c["prompt"]
        n = g if first else [max(1, c["left"] - 5 * b) if c["left"] > 5 * c["batch"] else c["left"] for b in range(c["batch"])]
        q = p if first else [c["pend"]] * c["batch"]
        keys = [p[b] + g[b] for b in range(c["batch"])]
        return [[(q[b] + n[b], keys[b], n[b]) for b in range(c["batch"])]]
    block = 32 if c["topology"] else BLOCK
    out = []
    for k in range(math.ceil(c["gen"] / block)):
        step = []
        for b in range(c["batch"]):
            n = int(g[b] - k * block)
            if n > 0:
                rows = (p[b] if k == 0 else 0) + g[b] if c["topology"] else (p[b] if k == 0 else int(block)) + n
                step.append((rows, p[b] + g[b], n))
        out.append(step)
    return out


# ---- the contract ----------------------------------------------------------------------------------------------
def prepare(case, seed):
    c = SimpleNamespace(**case)
    sh, w = _model(c.model)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    bm = _delim_bitmap(sh.vocab)
    if c.kind == "head":
        off = [0]
        for b in range(c.batch):
            off.append(off[-1] + max(1, c.rows - (7 * b if c.rows < 1024 else 0)))
        dec = LSPDecoder(sh, w, SchedCfg(tau=0.9, delim_bitmap=bm), c.batch, max(2, c.rows), device=DEV)
        hidden = torch.empty(off[-1], sh.d_model, dtype=torch.bfloat16, device=DEV).normal_(0.0, 1.0, generator=gen)
        return SimpleNamespace(c=c, dec=dec, hidden=hidden, off=off, bm=bm)
    p, g = _lengths(case)
    n_max = max(a + b for a, b in zip(p, g))
    scattered = c.kind == "decode" and c.topology == 1
    sched = SchedCfg(mode=2, fixed_k=32, topology=1, delim_bitmap=bm) if scattered else SchedCfg(tau=0.9, delim_bitmap=bm)
    dec = LSPDecoder(sh, _copy_heads(sh, w, c.gen), sched, c.batch, n_max, device=DEV)
    # text: 12 % delimiters, other ids uniform (the last id is [MASK])
    text = torch.randint(DELIMS[1] + 1, sh.vocab - 1, (c.batch, n_max), generator=gen, device=DEV, dtype=torch.int32)
    delim = torch.randint(DELIMS[0], DELIMS[1] + 1, text.shape, generator=gen, device=DEV, dtype=torch.int32)
    text = torch.where(torch.rand(text.shape, generator=gen, device=DEV) < 0.12, delim, text).contiguous()
    if c.kind == "decode":
        dec.set_option(3, c.inplace)
        dec.set_option(4, c.lagged)
        host = text.cpu().pin_memory()
        return SimpleNamespace(c=c, dec=dec, tokens=text, host=host, out=torch.empty_like(host).pin_memory(), p=p, g=g, bm=bm)
    dec.begin(text, p, g)
    if c.pend != c.prompt:           # walk the decode to the state: everything but the last pend + left positions, then pend
        left = [n for _, _, n in _passes(case)[0]]
        dec.denoise_step()
        dec.commit([g[b] - left[b] - c.pend for b in range(c.batch)])
        dec.denoise_step()
        dec.commit([c.pend] * c.batch)
    return SimpleNamespace(c=c, dec=dec, tokens=text, bm=bm)


def run(s):
    if s.c.kind == "head":
        r = s.dec.head_scan(s.hidden, s.off)
        y, p, m = s.dec.scores()
        return dict(run=r["L_run"], commit=r["L_commit"], flags=r["flags"].astype("int64"), yhat=y, pmax=p, margin=m)
    if s.c.kind == "pass":
        recs = s.dec.denoise_step()
        y, p, m = s.dec.scores()
        return dict(rec=torch.tensor([[r["n_before"], r["rows"], r["L_run"], r["L_commit"], r["flags"]] for r in recs]), yhat=y, pmax=p, margin=m)
    n, _ = s.dec.generate_host(s.tokens, s.host, s.out, s.p, s.g)
    return dict(tokens=s.out, steps=n, kv=s.dec.kv_view())


def work(case):
    L, d, hq, hkv, dh, f, v, _, dt = SHAPES[case["model"]]
    e = 4 if dt == "fp32" else 2
    if case["kind"] == "head":
        rows = sum(max(1, case["rows"] - (7 * b if case["rows"] < 1024 else 0)) for b in range(case["batch"]))
        return dict(bytes=(v * d + rows * d) * e + 12 * rows, flops=2.0 * rows * d * v)
    weights = L * ((hq + 2 * hkv) * dh * d + d * hq * dh + 3 * d * f)
    total = dict(bytes=0.0, flops=0.0)
    for seqs in _passes(case):
        rows, masked = sum(r for r, _, _ in seqs), sum(n for _, _, n in seqs)
        kv = sum(k for _, k, _ in seqs) * L * 2 * hkv * dh      # every key and value once
        total["bytes"] += (weights + v * d + kv + rows * d) * e + 12 * masked
        total["flops"] += 2.0 * rows * weights + 2.0 * masked * d * v + sum(4.0 * r * k * hq * dh * L for r, k, _ in seqs)
    return total


def tolerance(case):
    # Four times what the decoder shows against itself with other kernels (CUDA-core GEMMs, mma.sync attention), whose sums
    # run in another order: scores of a pass 1.4e-3 (largest 3.4e-3), the K/V rows of a whole bf16 decode 1.1e-2 (0.13), the
    # head alone 2e-5 (1e-4).  Whole values (tokens, argmax ids, block lengths) may differ where two logits tie.
    if case["kind"] == "head":
        return {"rel": 1e-4, "max": 5e-4, "differ": 1e-3}
    if SHAPES[case["model"]][-1] == "fp32":
        return {"rel": 2e-5, "max": 5e-4, "differ": 1e-3}
    if case["kind"] == "decode":
        return {"rel": 0.03, "max": 0.5, "differ": 5e-3}
    return {"rel": 6e-3, "max": 0.02, "differ": 5e-3}
