"""Gate/up of many tokens on CTA pairs (gateup_pair.cu) gives the bits of proj_tc.cu.  A d_ff that is no multiple of 64 takes that kernel;
with eight rows and columns of zeros it is the same model again, in the same plans."""
from dataclasses import replace

import pytest

from test_gpu_same_bits import _step, _weights
from vvs_synth.configs import XL

pytestmark = pytest.mark.gpu

XL2 = replace(XL, name="xl2", n_layers=2, vocab=512, lm_rows=0, tok_rows=0, s_max=208)             # 54 CTAs of 64 outputs
ODD19 = replace(XL2, name="odd19", d_model=1216, n_heads=19, d_ff=2752)                          # the same with 19 k-blocks: passes of up to 128
ODD = replace(XL2, name="odd", d_model=1088, n_heads=17, d_ff=2752)                               # 43 of them, the last pair's second idle; 17 k-blocks


CASES = [
    (XL2, 97, 1, 0, False),                                  # 97 tokens: passes of 64, the last of 33
    (XL2, 7, 2, 8, True), (XL2, 16, 1, 15, False),           # 126, 256
    (ODD, 97, 1, 0, False), (ODD, 10, 1, 10, True),          # 110
    (ODD, 6, 2, 15, False), (ODD, 13, 2, 8, False),          # 192, 234
    (XL2, 16, 2, 8, True), (XL2, 20, 1, 15, False),          # 288, 320: passes of 160
    (ODD, 9, 2, 15, False), (ODD, 24, 1, 15, True),          # 288, 384
    (ODD19, 97, 1, 0, False), (ODD19, 11, 1, 9, True), (ODD19, 6, 2, 15, False), (ODD19, 13, 2, 8, True),
    (ODD19, 9, 2, 15, False), (ODD19, 24, 1, 15, True)]
# (what stays with proj_tc.cu: 17 k-blocks take passes of up to 64 tokens only)
NOT_TAKEN = {("odd", 234), ("odd", 288), ("odd", 384)}


@pytest.mark.parametrize("ms,n_images,n_cfg,k,up_first", CASES)
def test_pairs_give_the_same_bits(ms, n_images, n_cfg, k, up_first):
    import torch
    fills = [(37 * i) % (ms.s_max - k - 1) for i in range(n_images)]
    w = _weights(replace(ms, d_ff=ms.d_ff - 8), 8400)
    want = _step(replace(ms, d_ff=ms.d_ff - 8), w, n_images, n_cfg, 1, k, fills, 8500 + k)
    for layer in w["layers"]:
        layer["w_down"] = torch.nn.functional.pad(layer["w_down"], (0, 8)).contiguous()
        gate, up = (torch.nn.functional.pad(layer[n], (0, 0, 0, 8)) for n in ("w_gate", "w_up"))
        both = torch.stack([up, gate] if up_first else [gate, up])
        layer["w_gate"], layer["w_up"] = both[int(up_first)], both[1 - int(up_first)]
    got = _step(ms, w, n_images, n_cfg, 1, k, fills, 8500 + k)
    for a, b in zip(want, got):
        assert torch.equal(a, b)


# where proj_few.cu refuses gate/up (its 160 CTAs would not all fit at once) and takes the other projections
FEW = replace(XL2, name="few", d_model=1024, n_heads=16, d_ff=4800)
FEW_CASES = [(FEW, 5, 1, 7), (FEW, 4, 2, 7), (FEW, 5, 2, 8), (FEW, 6, 2, 7)]         # 40, 64, 90, 96 tokens: one pass of 64 and 96


@pytest.mark.parametrize("ms,n_images,n_cfg,k", FEW_CASES)
def test_few_tokens_give_the_same_bits(ms, n_images, n_cfg, k):
    """One matrix as both gate and up takes proj_tc.cu, two copies of it take the pairs."""
    fills = [(37 * i) % (ms.s_max - k - 1) for i in range(n_images)]
    w = _weights(ms, 8450)
    for layer in w["layers"]:
        layer["w_up"] = layer["w_gate"]
    want = _step(ms, w, n_images, n_cfg, 1, k, fills, 8550 + k)
    for layer in w["layers"]:
        layer["w_up"] = layer["w_gate"].clone()
    got = _step(ms, w, n_images, n_cfg, 1, k, fills, 8550 + k)
    for a, b in zip(want, got):
        assert (a == b).all()
