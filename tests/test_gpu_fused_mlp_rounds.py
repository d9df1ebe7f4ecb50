"""The fused MLP block where a CTA pair works several 256-row tiles in turn: the ring of hidden units, the output's staging area and the
accumulators are carried on from tile to tile.  Every logit has the bits of the same placement with each GEMM as its own launch."""
import pytest
import torch

from paper_2511_00603_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def mods():
    from paper_2511_00603_b200 import build
    build.build()
    from paper_2511_00603_b200 import epara, server
    return epara, server


def _logits(E, server, impl, models):
    srv = server.Server(workspace_bytes=4 << 30, gemm_impl=impl)
    tickets = []
    for p, imgs in models:
        m = srv.add_model(p, max_batch=len(imgs))
        tickets += [srv.submit(m, E.CAT_FS, x=x) for x in imgs]
    info = srv.step()
    torch.cuda.synchronize()
    out = [srv.collect(t) for t in tickets]
    assert all(s == E.OK for s, _, _ in out)
    srv.close()
    return info, [logits.clone() for _, logits, _ in out]


# (d, hidden width, images) of the step's models; 197 rows an image, 74 pairs, 2 * hidden / 128 units a tile in a ring of three
@pytest.mark.parametrize("shapes", [
    [(128, 256, 146)],                  # 113 tiles: a second one for 39 pairs; four units a tile
    [(128, 640, 256)],                  # 197 tiles: a third one for 49; ten units
    [(384, 1280, 192)],                 # 148 tiles: two each; twenty units, two MMAs a k step
    [(384, 1536, 146)],                 # 113 tiles; twenty-four units, the ring starts each tile anew
    [(128, 256, 75), (384, 640, 75)],   # 58 + 58 tiles: the second tile belongs to another model
], ids=str)
def test_tiles_after_a_pairs_first_have_the_bits_of_the_unfused_kernels(mods, shapes):
    E, server = mods
    models = [(synth.make_vit(d=d, n_layers=2, n_heads=d // 64, mlp=mlp, n_cls=40, seed=980 + i, device=DEV, std=0.05, perturb=0.2),
               synth.make_images(n, seed=990 + i, device=DEV)) for i, (d, mlp, n) in enumerate(shapes)]
    fused_info, fused = _logits(E, server, E.GEMM_TCGEN05, models)
    plain_info, plain = _logits(E, server, E.GEMM_TCGEN05_UNFUSED, models)
    assert fused_info.launches < plain_info.launches
    for a, b in zip(fused, plain):
        assert torch.equal(a, b)
