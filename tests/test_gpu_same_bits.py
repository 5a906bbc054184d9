"""Results that stay what they were, bit for bit.  Deep models answer any change in the order or place of a rounding with guided
probabilities that move by more than a caller may see, so heads of 128 keep the arithmetic of their attention, and a projection whose
weights do not stay in L2 gives the same bits whichever of its two kernels runs it.  Inputs are small multiples of powers of two: the same everywhere."""
import hashlib
from dataclasses import replace

import pytest

from vvs_synth.configs import ROPE_1D, ModelShape

pytestmark = pytest.mark.gpu


def _ints(shape, span, scale, seed, base=0.0):
    import torch
    g = torch.Generator().manual_seed(seed)
    return (torch.randint(-span, span + 1, shape, generator=g).float() / scale + base).to(torch.bfloat16).cuda()


def _weights(ms, seed):
    d, ff = ms.d_model, ms.d_ff
    layers = []
    for l in range(ms.n_layers):
        s = seed + 100 * l
        layers.append(dict(w_qkv=_ints((3 * d, d), 127, 4096, s), w_o=_ints((d, d), 127, 8192, s + 1), w_gate=_ints((ff, d), 127, 4096, s + 2),
                           w_up=_ints((ff, d), 127, 4096, s + 3), w_down=_ints((d, ff), 127, 8192, s + 4),
                           norm1=_ints((d,), 16, 64, s + 5, 1.0), norm2=_ints((d,), 16, 64, s + 6, 1.0)))
    return dict(tok_emb=_ints((ms.tok_rows, d), 96, 32, seed + 7), norm_f=_ints((d,), 16, 64, seed + 8, 1.0),
                w_lm=_ints((ms.lm_rows, d), 127, 4096, seed + 9), layers=layers)


def _step(ms, w, n_images, n_cfg, n_forced, k, fills, seed):
    """Features and appended cache rows of one step, as integers."""
    import torch

    from paper_2511_13587_b200 import binding as vb
    rows, t_len = n_images * n_cfg, n_forced + k
    ctx = vb.vvs_create(vb.make_desc(ms, rows, t_len, 1))
    vb.vvs_bind_weights(ctx, w)
    kv = [_ints((ms.n_layers, rows, ms.n_heads, ms.s_max, ms.head_dim), 96, 32, seed + i) for i in range(2)]
    g = torch.Generator().manual_seed(seed)
    block = torch.randint(0, ms.vocab, (n_images, t_len), generator=g, dtype=torch.int32).cuda()
    zeros = lambda *shape: torch.zeros(shape, dtype=torch.int32, device="cuda")  # noqa: E731
    hidden = torch.zeros((rows, t_len, ms.d_model), dtype=torch.bfloat16, device="cuda")
    vb.vvs_verify(ctx, n_images=n_images, n_cfg=n_cfg, n_forced=n_forced, n_draft_max=k, block=block, kv_k=kv[0], kv_v=kv[1], kv_rows=rows,
                  cache_len=torch.tensor(fills * n_cfg, dtype=torch.int32, device="cuda"),
                  draft_probs=torch.full((n_images, k, ms.vocab), 1.0 / ms.vocab, device="cuda"),
                  uniforms=torch.full((n_images, k + 1), 0.5, device="cuda"), cfg_scale=2.0 if n_cfg == 2 else 1.0, temperature=1.0, mode=0,
                  nbr_k=1, hidden=hidden, accept_len=zeros(n_images), next_token=zeros(n_images), new_len=zeros(rows),
                  accept_mask=torch.zeros((n_images, k), dtype=torch.uint8, device="cuda"))
    assert vb.vvs_device_status(ctx) == 0
    vb.vvs_destroy(ctx)
    return [x.view(torch.int16).cpu() for x in (hidden, *kv)]


# (d_ff is no multiple of 64: one projection kernel for all token counts)
HEADS128 = ModelShape("heads128", 3, 1024, 8, 128, 328, 512, s_max=600, rope_mode=ROPE_1D, n_prefix=1)


@pytest.mark.parametrize("n_images,n_cfg,n_forced,k,fills,want", [
    (1, 2, 1, 8, [431], "0be59193331eacf8"),                                   # 16 items, two CTAs each
    (2, 2, 6, 24, [17, 540], "2b2fc140dd9bddb1"),                              # 32, two row groups
    (20, 1, 1, 8, [0, 7, 8, 15, 16, 17, 31, 32, 33, 150, 591, 47, 48, 63, 64, 20, 1, 2, 100, 90], "beef943aed6caffe"),       # 160: eight warps each
    (21, 2, 1, 3, [0, 12, 13, 28, 29, 300, 5, 60, 61, 99, 250, 596, 400, 31, 32, 33, 80, 81, 500, 3, 1], "4a4e6b2465bf05c8")])   # 336: four
def test_attention_of_heads_of_128(n_images, n_cfg, n_forced, k, fills, want):
    """Recorded before its kernel was rewritten for fewer instructions (CUDA 12.9)."""
    out = _step(HEADS128, _weights(HEADS128, 7100), n_images, n_cfg, n_forced, k, fills, 7200 + k)
    assert hashlib.sha256(b"".join(x.numpy().tobytes() for x in out)).hexdigest()[:16] == want


# Partial sums kept apart: QKV two slices in each of two CTAs, gate/up four in one, down projection two in each of four; one, two (and the
# output projection two in each of four); QKV unsplit, two in one CTA.
MID = ModelShape("mid", 2, 2048, 16, 128, 5504, 512, s_max=600, rope_mode=ROPE_1D, n_prefix=1)
WIDE = replace(MID, name="wide", d_model=4096, n_heads=32, d_ff=11008)
UNSPLIT = replace(MID, name="unsplit", n_layers=1, d_model=5120, n_heads=40, d_ff=13824)
EIGHT = replace(MID, name="eight", d_model=1536, n_heads=12, d_ff=4096)          # gate/up: eight in one CTA


@pytest.mark.parametrize("ms,n_images,n_cfg,n_forced,k,fills", [
    (MID, 1, 1, 1, 1, [300]), (MID, 1, 2, 1, 8, [20]), (MID, 1, 2, 1, 24, [570]), (MID, 1, 2, 6, 24, [99]), (MID, 4, 2, 1, 8, [0, 9, 333, 80]),
    (WIDE, 1, 1, 1, 8, [40]), (WIDE, 1, 2, 1, 8, [512]), (WIDE, 1, 2, 2, 14, [7]), (WIDE, 3, 2, 1, 7, [0, 9, 333]), (WIDE, 5, 2, 1, 7, [1, 2, 3, 4, 5]),
    (UNSPLIT, 1, 2, 1, 8, [60]), (UNSPLIT, 3, 2, 1, 8, [0, 9, 333]), (EIGHT, 1, 2, 1, 8, [60]), (EIGHT, 2, 2, 1, 14, [5, 200])])
def test_either_projection_kernel_gives_the_same_bits(ms, n_images, n_cfg, n_forced, k, fills):
    """d_ff less eight is no multiple of 64 (one kernel for everything), has the same plans, and with eight rows and columns of zeros
    is the same model again."""
    import torch
    w = _weights(replace(ms, d_ff=ms.d_ff - 8), 7300)
    want = _step(replace(ms, d_ff=ms.d_ff - 8), w, n_images, n_cfg, n_forced, k, fills, 7400 + k)
    for layer in w["layers"]:
        for name in ("w_gate", "w_up", "w_down"):
            pad = (0, 8) if name == "w_down" else (0, 0, 0, 8)
            layer[name] = torch.nn.functional.pad(layer[name], pad).contiguous()
    got = _step(ms, w, n_images, n_cfg, n_forced, k, fills, 7400 + k)
    for a, b in zip(want, got):
        assert torch.equal(a, b)
