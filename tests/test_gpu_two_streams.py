"""Two contexts on two streams at once: kernels of both share the SMs, clusters and CTA pairs among them, each with a share of an SM's shared
memory as large as its share of tensor memory.  Every step gives the bits that it gives alone."""
from dataclasses import replace

import pytest

from test_gpu_same_bits import _ints, _weights
from vvs_synth.configs import XL

pytestmark = pytest.mark.gpu

SHAPE = replace(XL, name="streams", n_layers=6, d_model=1024, n_heads=16, d_ff=2752, vocab=512, lm_rows=0, tok_rows=0, s_max=300)


class _Program:
    """A context with inputs of its own and one step on them."""

    def __init__(self, w, n_images, n_cfg, k, seed):
        import torch

        from paper_2511_13587_b200 import binding as vb
        ms, rows, t_len = SHAPE, n_images * n_cfg, 1 + k
        self.vb, self.ctx = vb, vb.vvs_create(vb.make_desc(ms, rows, t_len, 1))
        vb.vvs_bind_weights(self.ctx, w)
        self.kv = [_ints((ms.n_layers, rows, ms.n_heads, ms.s_max, ms.head_dim), 96, 32, seed + i) for i in range(2)]
        zeros = lambda *shape: torch.zeros(shape, dtype=torch.int32, device="cuda")  # noqa: E731
        g = torch.Generator().manual_seed(seed)
        self.hidden = torch.zeros((rows, t_len, ms.d_model), dtype=torch.bfloat16, device="cuda")
        fills = [(53 * i) % (ms.s_max - t_len) for i in range(n_images)]
        self.args = dict(n_images=n_images, n_cfg=n_cfg, n_forced=1, n_draft_max=k, kv_k=self.kv[0], kv_v=self.kv[1], kv_rows=rows,
                         block=torch.randint(0, ms.vocab, (n_images, t_len), generator=g, dtype=torch.int32).cuda(),
                         cache_len=torch.tensor(fills * n_cfg, dtype=torch.int32, device="cuda"),
                         draft_probs=torch.full((n_images, k, ms.vocab), 1.0 / ms.vocab, device="cuda"),
                         uniforms=torch.full((n_images, k + 1), 0.5, device="cuda"), cfg_scale=2.0, temperature=1.0, mode=0, nbr_k=1,
                         hidden=self.hidden, accept_len=zeros(n_images), next_token=zeros(n_images), new_len=zeros(rows),
                         n_commit=zeros(rows), accept_mask=torch.zeros((n_images, k), dtype=torch.uint8, device="cuda"))

    def step(self, stream):
        self.vb.vvs_verify(self.ctx, stream=stream.cuda_stream, **self.args)

    def result(self):
        assert self.vb.vvs_device_status(self.ctx) == 0
        return [x.clone() for x in (self.hidden, *self.kv, self.args["accept_len"], self.args["next_token"])]


# (images, drafts) with guidance: QKV and attention as one kernel; split projections in clusters; gate and up on CTA pairs
@pytest.mark.parametrize("one,other", [((1, 8), (1, 13)), ((1, 8), (6, 8)), ((4, 8), (8, 8)), ((1, 26), (12, 8))])
def test_steps_of_two_streams(one, other):
    import torch
    w = _weights(SHAPE, 8800)
    programs = [_Program(w, *n, k, 8900 + i) for i, (*n, k) in enumerate([(one[0], 2, one[1]), (other[0], 2, other[1])])]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    alone = []
    for p, s in zip(programs, streams):
        p.step(s)
        torch.cuda.synchronize()
        alone.append(p.result())
        p.hidden.zero_()
    torch.cuda.synchronize()
    for _ in range(12):
        for p, s in zip(programs, streams):
            p.step(s)
    torch.cuda.synchronize()
    for p, want in zip(programs, alone):
        for a, b in zip(p.result(), want):
            assert torch.equal(a, b)
        p.vb.vvs_destroy(p.ctx)
