"""The measured work of this framework: what a user's decoding program has it do, through the public
entry points of `paper_2511_13587_b200.binding`.

A case is a dict of plain values; `kind` names the call:

  verify    one verified step of the decoding loop: `vvs_verify` on a block of drafts (a chain, or a candidate
            tree), then the feature cache takes the committed rows; with `fetch` the skip-masked images of
            the batch also get their cached features back, as a batched server does between steps
  epilogue  `vvs_epilogue`: LM head, guidance, softmax and decisions on features the caller holds
  decide    `vvs_decide` / `vvs_decide_noalloc`: the decisions alone, on probabilities the caller holds
  skip      one verification-free step: `vvs_skip_decide`, `vvs_select_unverified`,
            `vvs_feature_cache_fetch`

Inputs are drawn on the device from the seed.  Weights are N(0, 0.02^2) with the two matrices that write to
the residual stream scaled by 1 / sqrt(2 n_layers), as decoders are initialised; token embeddings and
cached keys / values are N(0, 1).

What is compared.  In bf16 the features, the cache with its appended rows and, where the caller asks for
them, the target probabilities.  The decisions of a bf16 step are not: an index drawn from 16384 nearly
equally likely codes moves when a logit moves by a rounding, so two correct implementations draw
different ones.  They are compared, as whole numbers, wherever the inputs fix them: on given
probabilities, on given features, and in float32.
"""
from __future__ import annotations

import math
import random
from dataclasses import replace

import torch

from paper_2511_13587_b200 import binding as vb
from vvs_synth.configs import B7, DTYPE_BF16, MODE_RELAXED, MODE_STRICT, ROPE_1D, TINY, XL, ModelShape

# A decoder between the two benchmark shapes, for drawn cases only.
MID = ModelShape("mid", 24, 2048, 16, 128, 5504, 12000, s_max=1152, rope_mode=ROPE_1D, n_prefix=1)
SHAPES = {"tiny": TINY, "xl": XL, "mid": MID, "7b": B7}


# ---------------------------------------------------------------------------------------------
# the cases


def _verify(name, model, n_images, n_cfg, n_forced, n_draft, fill_lo, fill_hi, fixed_order, relaxed_k=0, tree=False,
            probs=False, ragged=False, fetch=False, cfg_scale=2.0, temperature=1.0):
    c = dict(kind="verify", model=model, n_images=n_images, n_cfg=n_cfg, n_forced=n_forced, n_draft=n_draft,
             fill_lo=fill_lo, fill_hi=fill_hi, fixed_order=fixed_order, relaxed_k=relaxed_k, tree=tree, probs=probs,
             ragged=ragged, fetch=fetch, cfg_scale=cfg_scale, temperature=temperature)
    return dict(c, name=name) if name else c


def _epilogue(name, d, vocab, n_images, n_cfg, n_draft, relaxed_k=0, temperature=1.0, noise=1.0):
    c = dict(kind="epilogue", d=d, vocab=vocab, n_images=n_images, n_cfg=n_cfg, n_draft=n_draft, relaxed_k=relaxed_k,
             temperature=temperature, noise=noise)
    return dict(c, name=name) if name else c


def _decide(name, vocab, n_images, n_draft, relaxed_k=0, tree=False, noalloc=False):
    c = dict(kind="decide", vocab=vocab, n_images=n_images, n_draft=n_draft, relaxed_k=relaxed_k, tree=tree,
             noalloc=noalloc)
    return dict(c, name=name) if name else c


def _skip(name, n_images, n_paths, depth, vocab, dim, d, cap):
    c = dict(kind="skip", n_images=n_images, n_paths=n_paths, depth=depth, vocab=vocab, dim=dim, d=d, cap=cap)
    return dict(c, name=name) if name else c


def listed():
    return [
        # A verification-free step of a 16-image server (every second step of the fixed-interval schedule with
        # i = 2): similarity of 24 candidate paths per image, the selector, the features for the drafter.
        _skip("skip_step_b16", 16, 24, 5, 16384, 8, 1280, 16),
        # The tiny float32 step: the smallest model a user brings up and checks a port of their own with.
        _verify("tiny_fp32", "tiny", 1, 1, 1, 4, 64, 64, True, probs=True, cfg_scale=1.0),
        # Decisions of a batch on probabilities another engine computed (relaxed acceptance, k = 64).
        _decide("decide_b16_relaxed", 16384, 16, 8, 64),
        # The step of one image, guidance on, eight drafts: the headline workload.  Arrival-order sums
        # (what `bench.py` times), then a context as the binding makes it by default (repeatable sums).
        _verify("xl_b1", "xl", 1, 2, 1, 8, 300, 300, False),
        _verify("xl_b1_fixed", "xl", 1, 2, 1, 8, 300, 300, True),
        # The step after a skipped one: five unverified tokens ride along as forced rows (post verification).
        _verify("xl_b1_post", "xl", 1, 2, 6, 8, 451, 451, True, ragged=True),
        # A candidate tree of 26 nodes, as EAGLE-style drafters propose; tree calls return the probabilities.
        _verify("xl_tree26", "xl", 1, 2, 1, 26, 200, 200, False, tree=True, probs=True),
        # A batch of 16 images at their own fill levels, relaxed acceptance, feature cache reset / store / fetch.
        _verify("xl_b16_relaxed", "xl", 16, 2, 1, 8, 1, 575, False, relaxed_k=64, fetch=True),
        # The 7B-class model, one image: the weight stream of a large model.
        _verify("7b_b1", "7b", 1, 2, 1, 8, 1500, 1500, False),
        # Decisions on features from elsewhere: one image; a middle-sized batch; the largest batch and codebook.
        _epilogue("epilogue_b1", 1280, 16384, 1, 2, 8),
        _epilogue("epilogue_b32_relaxed", 4096, 16384, 32, 2, 8, relaxed_k=64, temperature=1.2),
        _epilogue("epilogue_b64", 4096, 65536, 64, 2, 16, noise=0.5),
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_verify(rng):
    model = rng.choice(["xl", "xl", "xl", "xl", "mid", "7b"])
    ms = SHAPES[model]
    n_cfg = rng.choice([1, 2, 2])
    n_forced = rng.choice([1, 1, 1, 2, 3, 4, 5, 6])
    tree = rng.random() < 0.2
    n_draft = rng.randint(8, 26) if tree else _log_int(rng, 1, 16)
    t_len = n_forced + n_draft
    most = {"xl": 288, "mid": 128, "7b": 32}[model]                 # block rows of the whole call
    top = max(1, most // (n_cfg * t_len))
    n_images = 1 if rng.random() < 0.35 else _log_int(rng, 1, min(16, top))
    hi = {"xl": 575, "mid": 1024, "7b": 1500}[model]
    hi = min(hi, ms.s_max - t_len)
    if n_images == 1:
        fill_lo = fill_hi = rng.randint(1, hi)
    else:
        fill_lo, fill_hi = 1, hi
    relaxed = rng.random() < 0.35
    return _verify(None, model, n_images, n_cfg, n_forced, n_draft, fill_lo, fill_hi, rng.random() < 0.5,
                   relaxed_k=rng.choice([16, 64, 256]) if relaxed else 0, tree=tree, probs=tree or rng.random() < 0.2,
                   ragged=not tree and rng.random() < 0.3, fetch=rng.random() < 0.3,
                   cfg_scale=round(rng.uniform(1.5, 4.0), 2) if n_cfg == 2 else 1.0,
                   temperature=rng.choice([1.0, 1.0, 0.8, 1.2]))


def _draw_epilogue(rng):
    d = rng.choice([1280, 2048, 4096])
    vocab = _log_int(rng, 4096, 65536)
    n_images = _log_int(rng, 1, 64)
    relaxed_k = rng.choice([0, 0, 1, 64, 1000]) if vocab <= 20000 else rng.choice([0, 0, 64])
    return _epilogue(None, d, vocab, n_images, rng.choice([1, 2]), rng.randint(2, 16), relaxed_k,
                     round(rng.uniform(0.5, 1.5), 2), round(rng.uniform(0.2, 2.0), 2))


def _draw_decide(rng):
    tree = rng.random() < 0.3
    n_images = _log_int(rng, 1, 16 if tree else 64)
    return _decide(None, _log_int(rng, 4096, 32768 if tree else 65536), n_images, rng.randint(4, 26) if tree
                   else rng.randint(1, 16), rng.choice([0, 16, 64]), tree, not tree and rng.random() < 0.4)


def _draw_skip(rng):
    depth = rng.randint(1, 8)
    return _skip(None, _log_int(rng, 1, 64), rng.randint(2, 60), depth, _log_int(rng, 1024, 65536),
                 rng.choice([8, 8, 16, 32, 256]), rng.choice([1280, 4096]), rng.randint(depth, 16))


def _draw_tiny(rng):
    n_images, n_cfg = rng.randint(1, 6), rng.choice([1, 2])
    n_forced, n_draft = rng.choice([1, 1, 2, 3]), rng.randint(1, 12)
    fill = rng.randint(1, TINY.s_max - n_forced - n_draft)
    return _verify(None, "tiny", n_images, n_cfg, n_forced, n_draft, 1 if n_images > 1 else fill, fill, True,
                   relaxed_k=rng.choice([0, 16]), probs=rng.random() < 0.5, ragged=rng.random() < 0.3,
                   cfg_scale=2.0 if n_cfg == 2 else 1.0)


def _cost(case):
    w = work(case)
    return max(w["bytes"] / 6.5e12, w["flops"] / 1.6e15)


def draw(rng: random.Random):
    most = max(_cost(c) for c in listed())
    while True:
        x = rng.random()
        c = (_draw_verify if x < 0.5 else _draw_epilogue if x < 0.72 else _draw_decide if x < 0.82 else
             _draw_skip if x < 0.91 else _draw_tiny)(rng)
        if _cost(c) <= most:
            return c


# ---------------------------------------------------------------------------------------------
# inputs


class State:
    """What a program holds between steps: a context, its buffers, and the keyword arguments of its calls."""

    ctx = None

    def __del__(self):
        if self.ctx is not None:
            vb.vvs_destroy(self.ctx)
            self.ctx = None


class _Rand:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)

    def normal(self, shape, std=1.0, mean=0.0, dtype=torch.float32):
        x = torch.randn(shape, generator=self.g, device="cuda", dtype=dtype)
        if std != 1.0:
            x.mul_(std)
        if mean != 0.0:
            x.add_(mean)
        return x

    def ints(self, lo, hi, shape):
        """int32 in [lo, hi)."""
        return torch.randint(lo, hi, shape, generator=self.g, device="cuda", dtype=torch.int32)

    def unit(self, shape):
        """float32 in (0, 1)."""
        return torch.rand(shape, generator=self.g, device="cuda").clamp_(2.0 ** -25, 1.0 - 2.0 ** -24)

    def pick(self, probs):
        """One index per row of probs [..., V], drawn from it."""
        v = probs.shape[-1]
        return torch.multinomial(probs.reshape(-1, v), 1, generator=self.g).view(probs.shape[:-1]).to(torch.int32)


def _weights(r, ms, dtype):
    d, ff = ms.d_model, ms.d_ff
    out_std = 0.02 / math.sqrt(2.0 * ms.n_layers)

    def layer():
        return dict(w_qkv=r.normal((3 * d, d), 0.02, dtype=dtype), w_o=r.normal((d, d), out_std, dtype=dtype),
                    w_gate=r.normal((ff, d), 0.02, dtype=dtype), w_up=r.normal((ff, d), 0.02, dtype=dtype),
                    w_down=r.normal((d, ff), out_std, dtype=dtype), norm1=r.normal((d,), 0.1, 1.0, dtype=dtype),
                    norm2=r.normal((d,), 0.1, 1.0, dtype=dtype))

    return dict(tok_emb=r.normal((ms.tok_rows, d), dtype=dtype), norm_f=r.normal((d,), 0.1, 1.0, dtype=dtype),
                w_lm=r.normal((ms.lm_rows, d), 0.02, dtype=dtype), layers=[layer() for _ in range(ms.n_layers)])


def _neighbours(r, vocab, k):
    """CSR of the k nearest codes of an 8-dimensional codebook, the code itself first."""
    e = r.normal((vocab, 8))
    col = torch.empty((vocab, k), dtype=torch.int32, device="cuda")
    for s in range(0, vocab, 4096):
        t = min(vocab, s + 4096)
        dist = torch.cdist(e[s:t], e, compute_mode="donot_use_mm_for_euclid_dist")
        dist[torch.arange(t - s, device="cuda"), torch.arange(s, t, device="cuda")] = -1.0
        col[s:t] = torch.topk(dist, k, dim=1, largest=False, sorted=True).indices.to(torch.int32)
    return torch.arange(0, (vocab + 1) * k, k, dtype=torch.int32, device="cuda"), col.view(-1)


def _tree(seed, n_images, n_forced, n_draft):
    """Parent block row of every block row: a chain of forced rows, then nodes below random earlier ones, most
    of them below the last two levels, as drafters grow their trees."""
    rng = random.Random(seed)
    rows = []
    for _ in range(n_images):
        par = [-1] + list(range(n_forced - 1))
        for t in range(n_forced, n_forced + n_draft):
            par.append(rng.randint(max(n_forced - 1, t - 6), t - 1))
        rows.append(par)
    return rows


def _chain_drafts(r, n_images, n_draft, vocab, std=1.0):
    """Drafter rows that know nothing of the target, and the drafts sampled from them."""
    q = torch.softmax(r.normal((n_images, n_draft, vocab), std), dim=-1)
    return q, r.pick(q)


def _tree_drafts(r, parents, n_forced, n_draft, vocab, std=1.0):
    """The children of a node are draws from that node's drafter row."""
    par = torch.tensor(parents, device="cuda")[:, n_forced:]
    n_images = par.shape[0]
    rows = torch.softmax(r.normal((n_images, n_draft + 1, vocab), std), dim=-1)
    q = torch.gather(rows, 1, (par - (n_forced - 1)).unsqueeze(-1).expand(-1, -1, vocab)).contiguous()
    return q, r.pick(q)


def _ints(n):
    return torch.zeros(n, dtype=torch.int32, device="cuda")


def _prepare_verify(s, case, r, seed):
    ms = SHAPES[case["model"]]
    dtype = torch.bfloat16 if ms.dtype == DTYPE_BF16 else torch.float32
    b, n_cfg, f, k = case["n_images"], case["n_cfg"], case["n_forced"], case["n_draft"]
    rows, t_len, nbr_k = b * n_cfg, f + k, case["relaxed_k"]
    w = _weights(r, ms, dtype)
    kv_shape = (ms.n_layers, rows, ms.n_heads, ms.s_max, ms.head_dim)
    s.kv_k, s.kv_v = r.normal(kv_shape, dtype=dtype), r.normal(kv_shape, dtype=dtype)
    s.ctx = vb.vvs_create(vb.make_desc(ms, rows, t_len, max(1, nbr_k), deterministic=case["fixed_order"]))
    vb.vvs_bind_weights(s.ctx, w)
    if nbr_k > 1:
        vb.vvs_bind_neighbors(s.ctx, *_neighbours(r, ms.vocab, nbr_k))
    fills = r.ints(case["fill_lo"], case["fill_hi"] + 1, (b,))
    parents = _tree(seed, b, f, k) if case["tree"] else None
    q, drafts = (_tree_drafts(r, parents, f, k, ms.vocab) if parents else
                 _chain_drafts(r, b, k, ms.vocab, 2.0 if case["model"] == "tiny" else 1.0))
    block = torch.cat([r.ints(0, ms.vocab, (b, f)), drafts], dim=1) + ms.vocab_offset
    n_draft = r.ints(max(1, k // 2), k + 1, (b,)) if case["ragged"] else None
    s.hidden = torch.zeros((rows, t_len, ms.d_model), dtype=dtype, device="cuda")
    s.probs = torch.zeros((b, t_len, ms.vocab), device="cuda") if case["probs"] else None
    s.whole = dict(accept_len=_ints(b), next_token=_ints(b), new_len=_ints(rows), n_commit=_ints(rows),
                   accept_mask=torch.zeros((b, k), dtype=torch.uint8, device="cuda"))
    s.cache_len, s.t_len, s.tree = fills.repeat(n_cfg).contiguous(), t_len, case["tree"]
    s.args = dict(n_images=b, n_cfg=n_cfg, n_forced=f, n_draft_max=k, block=block.contiguous(), n_draft=n_draft,
                  kv_k=s.kv_k, kv_v=s.kv_v, kv_rows=rows, cache_len=s.cache_len, draft_probs=q,
                  uniforms=r.unit((b, k + 1)), cfg_scale=case["cfg_scale"], temperature=case["temperature"],
                  mode=MODE_RELAXED if nbr_k else MODE_STRICT,
                  nbr_k=max(1, nbr_k), hidden=s.hidden, target_probs=s.probs, **s.whole)
    if parents:
        s.args["tree_parent"] = torch.tensor(parents, dtype=torch.int32, device="cuda")
    cap = t_len + 5
    s.feat = torch.zeros((rows, cap, ms.d_model), dtype=dtype, device="cuda")
    s.fpos = torch.zeros((rows, cap), dtype=torch.int32, device="cuda")
    s.newest = _ints(rows)
    s.fcache = vb.make_fcache(s.feat, s.fpos, s.newest)
    vb.vvs_feature_cache_reset(s.ctx, s.fcache)
    s.fetch = None
    if case["fetch"]:
        s.fetch = dict(skip_mask=(r.unit((b,)) < 0.5).to(torch.uint8), n_images=b,
                       gamma=torch.ones(rows, dtype=torch.int32, device="cuda"), gamma_max=5, staleness=0,
                       out=torch.zeros((rows, 5, ms.d_model), dtype=dtype, device="cuda"),
                       out_pos=torch.zeros((rows, 5), dtype=torch.int32, device="cuda"))
    s.exact = ms.dtype != DTYPE_BF16


def _prepare_epilogue(s, case, r):
    d, v, b, n_cfg, k = case["d"], case["vocab"], case["n_images"], case["n_cfg"], case["n_draft"]
    rows, nbr_k = k + 1, case["relaxed_k"]
    s.ctx = vb.vvs_create(vb.make_desc(ModelShape("head", 0, d, 0, 0, 0, v), b * n_cfg, rows, max(1, nbr_k)))
    w_lm = r.normal((v, d), 2.0 / math.sqrt(d), dtype=torch.bfloat16)
    vb.vvs_bind_weights(s.ctx, {"w_lm": w_lm, "layers": []})
    if nbr_k > 1:
        vb.vvs_bind_neighbors(s.ctx, *_neighbours(r, v, nbr_k))
    hidden = r.normal((b * n_cfg, rows, d), dtype=torch.bfloat16)
    # a drafter that follows the target: softmax(guided logits + noise * Gumbel), the drafts sampled from it
    logits = torch.matmul(hidden[:, :k].reshape(-1, d), w_lm.t()).float().view(n_cfg, b, k, v)
    guided = logits[1] + 2.0 * (logits[0] - logits[1]) if n_cfg == 2 else logits[0]
    guided = guided / case["temperature"]
    guided += case["noise"] * -torch.log(-torch.log(r.unit((b, k, v))))
    q = torch.softmax(guided, dim=-1)
    del logits, guided
    s.whole = dict(accept_len=_ints(b), next_token=_ints(b), accept_mask=torch.zeros((b, k), dtype=torch.uint8, device="cuda"))
    s.args = dict(hidden_in=hidden, n_rows_per_seq=rows, first_row=0, drafts=r.pick(q), n_images=b, n_cfg=n_cfg,
                  n_draft_max=k, draft_probs=q, uniforms=r.unit((b, k + 1)), cfg_scale=2.0 if n_cfg == 2 else 1.0,
                  temperature=case["temperature"], mode=MODE_RELAXED if nbr_k else MODE_STRICT, nbr_k=max(1, nbr_k), **s.whole)


def _prepare_decide(s, case, r, seed):
    v, b, k, nbr_k = case["vocab"], case["n_images"], case["n_draft"], case["relaxed_k"]
    parents = _tree(seed, b, 1, k) if case["tree"] else None
    q, drafts = _tree_drafts(r, parents, 1, k, v) if parents else _chain_drafts(r, b, k, v)
    # target rows as another engine would hand them over: related to the drafter's, not equal to them
    p = torch.softmax(r.normal((b, k + 1, v)), dim=-1)
    p[:, :k] = torch.softmax(torch.log(q) + 0.7 * r.normal((b, k, v)), dim=-1)
    nbr = _neighbours(r, v, nbr_k) if nbr_k > 1 else None
    s.whole = dict(accept_len=_ints(b), next_token=_ints(b), accept_mask=torch.zeros((b, k), dtype=torch.uint8, device="cuda"))
    s.args = dict(target_probs=p, n_rows_per_seq=k + 1, first_row=0, drafts=drafts, n_images=b, n_draft_max=k,
                  draft_probs=q, uniforms=r.unit((b, k + 1)), mode=MODE_RELAXED if nbr_k else MODE_STRICT, nbr_k=max(1, nbr_k),
                  **s.whole)
    if case["noalloc"]:
        s.args.update(vocab=v, vocab_offset=0)
        if nbr:
            s.args.update(nbr_row_ptr=nbr[0], nbr_col=nbr[1])
        return
    s.ctx = vb.vvs_create(vb.make_desc(ModelShape("rows", 0, 64, 0, 0, 0, v), b, k + 1, max(1, nbr_k)))
    if nbr:
        vb.vvs_bind_neighbors(s.ctx, *nbr)
    if parents:
        s.args["tree_parent"] = torch.tensor(parents, dtype=torch.int32, device="cuda")
        s.whole["accept_path"] = s.args["accept_path"] = torch.zeros((b, k), dtype=torch.int32, device="cuda")


def _prepare_skip(s, case, r):
    b, n, depth, v, d, cap = (case[x] for x in ("n_images", "n_paths", "depth", "vocab", "d", "cap"))
    rows = 2 * b                                                    # cond and uncond sequences
    s.ctx = vb.vvs_create(vb.make_desc(replace(XL, name="skip", n_layers=0, d_model=d), rows, 1))
    s.codebook = r.normal((v, case["dim"]))
    # candidate paths share a stem of random length with the first one
    s.paths = r.ints(0, v, (b, n, depth))
    stem = r.ints(0, depth + 1, (b, n, 1)) > torch.arange(depth, device="cuda")
    s.paths = torch.where(stem, s.paths[:, :1].expand(-1, n, -1), s.paths).contiguous()
    s.path_len = r.ints(max(1, depth - 2), depth + 1, (b, n))
    s.last_verified = torch.ones(b, dtype=torch.uint8, device="cuda")
    s.u = r.unit((b,))
    s.decision, s.similarity = torch.zeros(b, dtype=torch.uint8, device="cuda"), torch.zeros(b, device="cuda")
    s.path, s.n_kept, s.tokens = _ints(b), _ints(b), torch.zeros((b, depth), dtype=torch.int32, device="cuda")
    newest = r.ints(cap, 500, (b,)).repeat(2)
    ring = torch.arange(cap, device="cuda", dtype=torch.int32)
    fpos = newest[:, None] - torch.remainder(newest[:, None] - ring[None, :], cap)
    s.fcache = vb.make_fcache(r.normal((rows, cap, d), dtype=torch.bfloat16), fpos.to(torch.int32).contiguous(),
                              newest.contiguous())
    s.gamma = r.ints(1, min(depth, cap) + 1, (b,)).repeat(2).contiguous()
    s.gamma_max = depth
    s.feat = torch.zeros((rows, depth, d), dtype=torch.bfloat16, device="cuda")
    s.feat_pos = torch.zeros((rows, depth), dtype=torch.int32, device="cuda")


def prepare(case, seed):
    s = State()
    s.kind = case["kind"]
    r = _Rand(seed)
    if s.kind == "verify":
        _prepare_verify(s, case, r, seed)
    elif s.kind == "epilogue":
        _prepare_epilogue(s, case, r)
    elif s.kind == "decide":
        _prepare_decide(s, case, r, seed)
    else:
        _prepare_skip(s, case, r)
    return s


# ---------------------------------------------------------------------------------------------
# one pass


def run(s):
    if s.kind == "verify":
        vb.vvs_verify(s.ctx, **s.args)
        if s.fetch:                                                 # images of a batch start from an empty ring
            vb.vvs_feature_cache_reset(s.ctx, s.fcache)
        vb.vvs_feature_cache_store(s.ctx, s.fcache, s.hidden, s.t_len, s.cache_len, s.whole["n_commit"])
        if s.fetch:
            vb.vvs_feature_cache_fetch(s.ctx, s.fcache, **s.fetch)
        out = {"hidden": s.hidden}
        if s.probs is not None:
            out["probs"] = s.probs
        if not s.tree:                 # after a tree call the cache rows of the accepted nodes have moved
            out["kv_k"], out["kv_v"] = s.kv_k, s.kv_v
        if s.exact:
            out.update(s.whole, feat=s.feat, fpos=s.fpos, newest=s.newest)
        return out
    if s.kind == "epilogue":
        vb.vvs_epilogue(s.ctx, **s.args)
        return s.whole
    if s.kind == "decide":
        if s.ctx is None:
            vb.vvs_decide_noalloc(**s.args)
        else:
            vb.vvs_decide(s.ctx, **s.args)
        return s.whole
    vb.vvs_skip_decide(s.ctx, s.paths, s.path_len, s.codebook, s.last_verified, 2, 0.8, 0.65, s.decision, s.similarity)
    vb.vvs_select_unverified(s.ctx, s.paths, s.path_len, s.u, s.path, s.n_kept, s.tokens)
    vb.vvs_feature_cache_fetch(s.ctx, s.fcache, s.decision, s.decision.numel(), s.gamma, s.gamma_max, 0, s.feat, s.feat_pos)
    return dict(decision=s.decision, similarity=s.similarity, path=s.path, n_kept=s.n_kept, tokens=s.tokens, feat=s.feat,
                feat_pos=s.feat_pos)


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without, and how close two correct ones come


def work(case):
    if case["kind"] == "verify":
        ms = SHAPES[case["model"]]
        b, n_cfg, k = case["n_images"], case["n_cfg"], case["n_draft"]
        es = 2 if ms.dtype == DTYPE_BF16 else 4
        t_len = case["n_forced"] + k
        rows = b * n_cfg
        m, fill = rows * t_len, (case["fill_lo"] + case["fill_hi"]) / 2
        n_bytes = ms.streamed_params * es                                           # every weight once
        n_bytes += rows * (fill + 2 * t_len) * ms.n_layers * 2 * ms.d_model * es      # K / V read, and appended
        n_bytes += m * ms.d_model * es * 2 + b * ms.vocab * 4                         # embeddings, features, one drafter row
        if case["probs"]:
            n_bytes += b * t_len * ms.vocab * 4
        flops = 2.0 * m * ms.streamed_params + 4.0 * m * (fill + t_len / 2) * ms.d_model * ms.n_layers
        return {"bytes": n_bytes, "flops": flops}
    if case["kind"] == "epilogue":
        d, v, b, k = case["d"], case["vocab"], case["n_images"], case["n_draft"]
        m = b * case["n_cfg"] * (k + 1)
        return {"bytes": d * v * 2 + m * d * 2 + b * v * 4 + b * k * max(1, case["relaxed_k"]) * 4, "flops": 2.0 * m * d * v}
    if case["kind"] == "decide":
        v, b, k = case["vocab"], case["n_images"], case["n_draft"]
        # the sampled row of each distribution, the looked-at entries of the others
        return {"bytes": 2 * b * v * 4 + b * k * (8 + 8 * max(1, case["relaxed_k"])), "flops": 4.0 * b * v}
    b, n, depth, dim, d = (case[x] for x in ("n_images", "n_paths", "depth", "dim", "d"))
    kept = (n + 1) // 2
    return {"bytes": b * n * depth * 4 + b * kept * depth * dim * 4 + 2 * b * (1 + depth) / 2 * d * 2 * 2,
            "flops": b * kept * kept * depth * dim}


def tolerance(case):
    if case["kind"] == "verify":
        if SHAPES[case["model"]].dtype == DTYPE_BF16:
            return {"rel": 1e-2, "max": 0.1}
        return {"rel": 1e-5, "max": 1e-3}
    if case["kind"] == "epilogue":
        return {"rel": 0.0, "differ": 0.01}     # a sample point or a threshold within an fp32 rounding of an edge
    if case["kind"] == "decide":
        return "exact"
    return {"rel": 1e-6}
