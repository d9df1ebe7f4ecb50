"""The tile-pair GEMM's last round in finer tiles (K of 2048 and more): a request's bits do not depend on whether its rows or columns fall into it."""
import numpy as np
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


def _answers(E, srv, tickets):
    srv.step()
    torch.cuda.synchronize()
    out = [srv.collect(t) for t in tickets]
    assert all(s == E.OK for s, _, _ in out)
    return [(logits.clone(), int(a.item())) for _, logits, a in out]


# FC2 (K 2048, fp32 residual) on 74 pairs, 256-wide tiles
@pytest.mark.parametrize("n", [
    50,     # 1.05 rounds: two row tiles 64 wide, the second half empty
    56,     # 1.19 rounds: seven row tiles, 64 wide
    64,     # 1.35 rounds: thirteen row tiles, 128 wide
])
def test_encoder_answers_do_not_depend_on_the_last_round(mods, n):
    E, server = mods
    p = synth.make_vit(d=512, n_layers=2, n_heads=8, mlp=2048, n_cls=40, seed=960, device=DEV, std=0.05, perturb=0.2)
    x = synth.make_images(n, seed=961, device=DEV)
    srv = server.Server(workspace_bytes=1 << 30)
    m = srv.add_model(p, max_batch=n)
    whole = _answers(E, srv, [srv.submit(m, E.CAT_FS, x=x[i]) for i in range(n)])
    for a in range(0, n, 8):                                   # at most 8 images: one round
        part = _answers(E, srv, [srv.submit(m, E.CAT_FS, x=x[i]) for i in range(a, min(n, a + 8))])
        for (u, iu), (v, iv) in zip(part, whole[a:a + 8]):
            assert torch.equal(u, v) and iu == iv
    srv.close()


@pytest.mark.parametrize("ffn,lens", [
    (2880, (1700, 1601)),    # QKV 13 x 6 tiles: the last row tile; gate and up 13 x 22.5: the last column, half empty; down 1.41 rounds: 128 wide
    (768, (1700, 1601)),     # gate and up 13 x 6 tiles: the last row tile
])
def test_prompts_do_not_depend_on_the_last_round(mods, ffn, lens):
    E, server = mods
    p = synth.make_decoder(d=2048, n_layers=2, n_q_heads=16, n_kv_heads=4, head_dim=64, ffn=ffn, vocab=300, seed=970, device=DEV, std=0.03,
                           perturb=0.2)
    rng = np.random.default_rng(971)
    pages = [-(-n // synth.PAGE) for n in lens]
    order = rng.permutation(sum(pages)).astype(np.int32)
    tabs = [torch.as_tensor(order[sum(pages[:i]):sum(pages[:i + 1])], device=DEV) for i in range(len(lens))]
    toks = [[int(t) for t in rng.integers(0, 300, n)] for n in lens]
    pool = synth.make_kv_pool(2, sum(pages), 4, 64, seed=972, device=DEV)
    pool0 = pool.clone()
    srv = server.Server(workspace_bytes=1 << 30)
    m = srv.add_model(p, kv_pool=pool, max_kv_len=max(lens), max_batch=sum(lens))

    def submit(i):
        return srv.submit(m, E.CAT_FS, tokens=toks[i], kv_len=0, table=tabs[i])

    whole = _answers(E, srv, [submit(i) for i in range(len(lens))])
    pool_whole = pool.clone()
    pool.copy_(pool0)
    for i in range(len(lens)):
        part = _answers(E, srv, [submit(i)])[0]
        assert torch.equal(part[0], whole[i][0]) and part[1] == whole[i][1]
    assert torch.equal(pool, pool_whole)
    srv.close()


# d 2048 on 74 pairs, 256-wide tiles, K 2048: the last columns of tiles, with a bias
@pytest.mark.parametrize("mlp,n", [
    (2080, 23),     # FC1: one column, 64 wide, of which 32 exist
    (4096, 20),     # QKV: one column in tiles 64 wide
    (2176, 15),     # FC1: three columns in tiles 128 wide
])
def test_encoder_answers_do_not_depend_on_columns_of_the_last_round(mods, mlp, n):
    E, server = mods
    p = synth.make_vit(d=2048, n_layers=1, n_heads=32, mlp=mlp, n_cls=40, seed=962, device=DEV, std=0.03, perturb=0.2)
    x = synth.make_images(n, seed=963, device=DEV)
    srv = server.Server(workspace_bytes=1 << 30)
    m = srv.add_model(p, max_batch=n)
    whole = _answers(E, srv, [srv.submit(m, E.CAT_FS, x=x[i]) for i in range(n)])
    for a in range(0, n, 3):                                   # three images: one round
        part = _answers(E, srv, [srv.submit(m, E.CAT_FS, x=x[i]) for i in range(a, min(n, a + 3))])
        for (u, iu), (v, iv) in zip(part, whole[a:a + 3]):
            assert torch.equal(u, v) and iu == iv
    srv.close()


def test_a_last_round_of_several_models(mods):
    """Two encoders of one shape in one launch, 50 and 14 images: the rows that are cut finer are those of the one with more tiles,
    whichever it is."""
    E, server = mods
    srv = server.Server(workspace_bytes=1 << 30)
    models = []
    for k in range(2):
        p = synth.make_vit(d=512, n_layers=2, n_heads=8, mlp=2048, n_cls=40, seed=964 + k, device=DEV, std=0.05, perturb=0.2)
        models.append((srv.add_model(p, max_batch=50), synth.make_images(50, seed=966 + k, device=DEV)))

    def submit(k, a, b):
        m, x = models[k]
        return [srv.submit(m, E.CAT_FS, x=x[i]) for i in range(a, b)]

    alone = [[r for a in range(0, 50, 8) for r in _answers(E, srv, submit(k, a, min(50, a + 8)))] for k in range(2)]
    for n0, n1 in ((50, 14), (14, 50)):
        both = _answers(E, srv, submit(0, 0, n0) + submit(1, 0, n1))
        for (u, iu), (v, iv) in zip(both, alone[0][:n0] + alone[1][:n1]):
            assert torch.equal(u, v) and iu == iv
    srv.close()
