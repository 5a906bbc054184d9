"""The one-kernel decision at the edges of its split: codebooks around the sizes where an image gets another CTA
(4096, 8192, 16384 codes), smaller than a warp's share, no multiple of anything; no draft and 32 drafts."""
import pytest

from test_gpu_decide import compare_exact, decide_case, gpu_decide, oracle_decide
from vvs_synth.configs import MODE_RELAXED, MODE_STRICT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("v,k,rows", [(2, 3, 4), (33, 4, 5), (4095, 5, 6), (4096, 5, 6), (8193, 32, 32), (16383, 1, 2),
                                      (16385, 8, 9)])
def test_decide_around_the_cluster_sizes(v, k, rows):
    from paper_2511_13587_b200 import binding as vb
    for mode, nbr_k, n_images in ((MODE_STRICT, 1, 5), (MODE_RELAXED, min(v, 40), 3)):
        c = decide_case(31 * v + k, v, n_images, k, rows, 0, mode, nbr_k, 0.3, 1.0, 0.6)
        ctx = vb.vvs_create(vb.make_desc(c["ms"], n_images, rows, nbr_k))

        def call(d, o):
            if "row_ptr" in d:
                vb.vvs_bind_neighbors(ctx, d["row_ptr"], d["col"])
            vb.vvs_decide(ctx, target_probs=d["target_probs"], n_rows_per_seq=rows, first_row=0, drafts=d["drafts"],
                          n_images=n_images, n_draft_max=k, n_draft=d["n_draft"], draft_probs=d["draft_probs"],
                          uniforms=d["uniforms"], mode=mode, nbr_k=nbr_k, delta=0.3, **o)
        got = gpu_decide(c, call)
        assert vb.vvs_device_status(ctx) == 0
        compare_exact(c, got, oracle_decide(c))
        vb.vvs_destroy(ctx)
