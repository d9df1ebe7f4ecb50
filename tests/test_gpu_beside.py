"""Launches of one step that run side by side: the attention launches of a layer (prompt chunks, encoders, decode requests) and the
GEMM launches of a wave.  What runs beside what must not show in a single bit."""
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


@pytest.mark.parametrize("hd,chunk,dec_lens", [
    (64, 400, [300, 17]),                        # few decode blocks: one query tile per item of the chunk's attention
    (64, 400, [4200] * 8 + [16, 1, 255]),        # more than the SMs it leaves take: two tiles per item
    (64, 130, [600, 31, 5]),
    (128, 257, [513, 256, 16]),
])
def test_chunk_beside_decode_requests_has_the_bits_of_separate_steps(mods, hd, chunk, dec_lens):
    E, server = mods
    Hq, Hkv, layers = 32, 8, 2
    p = synth.make_decoder(d=256, n_layers=layers, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=hd, ffn=512, vocab=300, seed=910, device=DEV,
                           std=0.05, perturb=0.2)
    rng = np.random.default_rng(911)
    prefix = 33
    pages = [-(-(n + 1) // synth.PAGE) for n in dec_lens] + [-(-(prefix + chunk) // synth.PAGE)]
    order = rng.permutation(sum(pages)).astype(np.int32)
    tabs, at = [], 0
    for n in pages:
        tabs.append(torch.as_tensor(order[at:at + n], device=DEV))
        at += n
    pool = synth.make_kv_pool(layers, sum(pages), Hkv, hd, seed=912, device=DEV)
    pool0 = pool.clone()
    toks = [int(t) for t in rng.integers(0, 300, chunk)]
    dec = [int(t) for t in rng.integers(0, 300, len(dec_lens))]
    srv = server.Server(workspace_bytes=512 << 20)
    m = srv.add_model(p, kv_pool=pool, max_kv_len=4300, max_batch=chunk + len(dec_lens))

    def decode():
        return [srv.submit(m, E.CAT_FS, token=dec[i], kv_len=n, table=tabs[i]) for i, n in enumerate(dec_lens)]

    def finish(tickets):
        torch.cuda.synchronize()
        out = [srv.collect(t) for t in tickets]
        assert all(s == E.OK for s, _, _ in out)
        return [(l.clone(), int(a.item())) for _, l, a in out]

    t = decode()
    srv.step()
    apart = finish(t)
    t = [srv.submit(m, E.CAT_FS, tokens=toks, kv_len=prefix, table=tabs[-1])]
    srv.step()
    apart += finish(t)
    pool_apart = pool.clone()
    for _ in range(3):
        pool.copy_(pool0)
        t = decode() + [srv.submit(m, E.CAT_FS, tokens=toks, kv_len=prefix, table=tabs[-1])]
        srv.step()
        for (a, ia), (b, ib) in zip(apart, finish(t)):
            assert torch.equal(a, b) and ia == ib
        assert torch.equal(pool, pool_apart)
    srv.close()


def test_models_of_one_step_have_the_bits_of_steps_of_their_own(mods):
    """Two MLPs, two encoders (one with a nearly empty last round of the fused MLP launch) and two decoders: weight streaming,
    swapped operands, tile pairs, fused blocks, encoder and decode attention share the waves of one step."""
    E, server = mods
    srv = server.Server(workspace_bytes=2 << 30)
    reqs = []
    for n, dims, cap in ((12, [256, 512, 72], 12), (200, [1024, 2048, 520], 200)):
        p = synth.make_mlp(dims, seed=920 + n, device=DEV, std=0.06, perturb=0.2)
        x = synth.make_mlp_inputs(n, dims[0], seed=921 + n, device=DEV)
        reqs.append((srv.add_model(p, max_batch=cap), [dict(x=x[i]) for i in range(n)]))
    for n, d, heads in ((97, 384, 6), (3, 128, 2)):
        p = synth.make_vit(d=d, n_layers=2, n_heads=heads, mlp=4 * d, n_cls=50, seed=930 + n, device=DEV, std=0.05, perturb=0.2)
        x = synth.make_images(n, seed=931 + n, device=DEV)
        reqs.append((srv.add_model(p, max_batch=n), [dict(x=x[i]) for i in range(n)]))
    rng = np.random.default_rng(940)
    pools = []
    for n in (4, 150):
        p = synth.make_decoder(d=512, n_layers=2, n_q_heads=8, n_kv_heads=4, head_dim=64, ffn=1024, vocab=600, seed=941 + n, device=DEV,
                               std=0.05, perturb=0.2)
        lens = [int(v) for v in rng.integers(1, 900, n)]
        pages = [-(-(v + 1) // synth.PAGE) for v in lens]
        order = rng.permutation(sum(pages)).astype(np.int32)
        pool = synth.make_kv_pool(2, sum(pages), 4, 64, seed=942 + n, device=DEV)
        m = srv.add_model(p, kv_pool=pool, max_kv_len=900, max_batch=n)
        one, at = [], 0
        for v, k in zip(lens, pages):
            one.append(dict(token=int(rng.integers(0, 600)), kv_len=v, table=torch.as_tensor(order[at:at + k], device=DEV)))
            at += k
        reqs.append((m, one))
        pools.append(pool)

    def run(groups):
        t = [srv.submit(m, E.CAT_FS, **kw) for m, one in groups for kw in one]
        srv.step()
        torch.cuda.synchronize()
        out = [srv.collect(x) for x in t]
        assert all(s == E.OK for s, _, _ in out)
        return [(l.clone(), int(a.item())) for _, l, a in out]

    alone = [r for g in reqs for r in run([g])]
    after = [p.clone() for p in pools]
    for _ in range(3):
        for (a, ia), (b, ib) in zip(alone, run(reqs)):
            assert torch.equal(a, b) and ia == ib
        assert all(torch.equal(p, q) for p, q in zip(pools, after))
    srv.close()


def test_attention_launches_of_six_kinds_side_by_side(mods):
    """One layer's attention as prompt chunks of both head sizes, encoders, and decode requests of three shapes (tensor cores with head
    sizes 64 and 128 and a merge kernel behind each, CUDA cores with 32): every answer and cache has the bits of steps of one model."""
    E, server = mods
    srv = server.Server(workspace_bytes=2 << 30)
    rng = np.random.default_rng(950)
    reqs, pools = [], []
    # (the encoder's second attention falls into the same sweep as the decoders' second)
    v = synth.make_vit(d=128, n_layers=2, n_heads=2, mlp=256, n_cls=50, seed=951, device=DEV, std=0.05, perturb=0.2)
    x = synth.make_images(7, seed=952, device=DEV)
    reqs.append((srv.add_model(v, max_batch=7), [dict(x=x[i]) for i in range(7)]))
    for k, (hd, Hq, Hkv, chunk, lens) in enumerate(((64, 16, 4, 200, [900, 17, 300]), (128, 8, 4, 130, [520, 33]), (64, 8, 8, 0, [1500, 256, 5]),
                                                    (32, 8, 4, 0, [700, 40]))):
        p = synth.make_decoder(d=256, n_layers=2, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=hd, ffn=512, vocab=300, seed=953 + k, device=DEV,
                               std=0.05, perturb=0.2)
        new, old = [1] * len(lens) + [chunk] * (chunk > 0), lens + [45] * (chunk > 0)
        pages = [-(-(a + b) // synth.PAGE) for a, b in zip(old, new)]
        order = rng.permutation(sum(pages)).astype(np.int32)
        pool = synth.make_kv_pool(2, sum(pages), Hkv, hd, seed=960 + k, device=DEV)
        m = srv.add_model(p, kv_pool=pool, max_kv_len=1500, max_batch=sum(new))
        one, at = [], 0
        for n, length, k_pages in zip(new, old, pages):
            toks = [int(t) for t in rng.integers(0, 300, n)]
            one.append(dict(kv_len=length, table=torch.as_tensor(order[at:at + k_pages], device=DEV), **(dict(tokens=toks) if n > 1 else dict(token=toks[0]))))
            at += k_pages
        reqs.append((m, one))
        pools.append((pool, pool.clone()))

    def run(groups):
        t = [srv.submit(m, E.CAT_FS, **kw) for m, one in groups for kw in one]
        srv.step()
        torch.cuda.synchronize()
        out = [srv.collect(i) for i in t]
        assert all(s == E.OK for s, _, _ in out)
        return [(l.clone(), int(a.item())) for _, l, a in out]

    alone = [r for g in reqs for r in run([g])]
    after = [pool.clone() for pool, _ in pools]
    for _ in range(3):
        for pool, before in pools:
            pool.copy_(before)
        for (a, ia), (b, ib) in zip(alone, run(reqs)):
            assert torch.equal(a, b) and ia == ib
        assert all(torch.equal(pool, q) for (pool, _), q in zip(pools, after))
    srv.close()
