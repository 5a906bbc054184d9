"""The tree walk where the number of images decides how many CTAs an image gets: clusters of eight, four, two and one."""
import pytest

import test_gpu_decide as D
from vvs_synth.configs import MODE_RELAXED, MODE_STRICT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,nbr_k,delta,adjusted", [(MODE_STRICT, 1, float("inf"), False), (MODE_RELAXED, 16, 0.2, True)])
@pytest.mark.parametrize("v,n_images", [(16400, 15), (16400, 17), (8200, 35), (8200, 76)])
def test_tree_walk_batches(v, n_images, mode, nbr_k, delta, adjusted):
    D.test_tree_walk_is_exact_on_random_trees(v, n_images, 12, 2, 1.0, 1.5, 0, mode, nbr_k, delta, adjusted)


@pytest.mark.parametrize("v", [4096, 8192, 8195, 16384, 16397])
def test_sample_in_one_code_and_in_none(v):
    """All of the mass on one code, at the edges of the parts four and eight CTAs take; a row without mass draws no token and
    sets the status bit."""
    import torch
    from paper_2511_13587_b200 import binding as vb
    from vvs_synth.configs import ModelShape
    codes = [0, v // 8 - 1, v // 8, v // 4, v // 2 - 1, v // 2, v - v // 8, v - 1]
    n = len(codes) + 1
    p = torch.zeros((n, 3, v), device="cuda")
    for b, c in enumerate(codes):
        p[b, :, c] = 1.0
    q = torch.full((n, 2, v), 1.0 / v, device="cuda")
    # two siblings below the root, both rejected (uniforms close to one): the residual has mass on the one code only
    drafts = torch.tensor([[2, 5]], dtype=torch.int32, device="cuda").repeat(n, 1).contiguous()
    u = torch.full((n, 3), 0.999, device="cuda")
    u[:, 2] = torch.linspace(1e-6, 1.0 - 2.0 ** -24, n, device="cuda")
    parent = torch.tensor([[-1, 0, 0]], dtype=torch.int32, device="cuda").repeat(n, 1).contiguous()
    ctx = vb.vvs_create(vb.make_desc(ModelShape("rows", 0, 64, 0, 0, 0, v), n, 3, 1))
    o = dict(accept_len=torch.full((n,), -7, dtype=torch.int32, device="cuda"),
             next_token=torch.full((n,), -7, dtype=torch.int32, device="cuda"))
    vb.vvs_decide(ctx, target_probs=p, n_rows_per_seq=3, first_row=0, drafts=drafts, n_images=n, n_draft_max=2, draft_probs=q,
                  uniforms=u, tree_parent=parent, **o)
    assert vb.vvs_device_status(ctx) == vb.VVS_DEV_BAD_ARG
    assert o["accept_len"].tolist() == [0] * n
    assert o["next_token"].tolist() == codes + [-1]
    vb.vvs_destroy(ctx)
