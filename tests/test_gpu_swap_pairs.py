"""The swapped-operand GEMM on pairs of CTAs (256 output columns a tile, up to 384 batch rows, one or two k ranges)."""
import numpy as np
import pytest
import torch

from tests.parity import assert_close
from tests.test_gpu_gemm_choice import _plan
from tests.test_gpu_kernels import E, _run_gemm  # noqa: F401  (E: the module's fixture)

pytestmark = pytest.mark.gpu

# row tile, k ranges, (M, N, K, epilogue)
CASES = [
    (64, 2, (129, 264, 768, ("bias", "gelu"))),         # last columns in the first CTA of a pair only, last row tile of one row
    (64, 2, (161, 2100, 2048, ("bias",))),              # N not a multiple of 8, stage ring used several times over
    (64, 2, (289, 1032, 3080, ())),                     # K not a multiple of a k-block, ranges of 25 and 24
    (64, 2, (385, 520, 1000, ("resid",))),              # fp32 residual
    (128, 2, (330, 2100, 3080, ("gelu", "bias"))),
    (160, 2, (385, 2100, 3080, ("swiglu",))),
    (64, 1, (300, 2100, 1000, ("bias", "resid"))),
    (192, 1, (330, 9000, 3080, ("bias",))),
    (224, 2, (199, 7000, 4104, ("bias",))),
    (224, 1, (406, 6152, 8200, ("resid",))),
    (288, 1, (280, 16384, 2048, ("swiglu",))),          # two MMAs, of 160 and 128 rows
    (288, 2, (1100, 2048, 8192, ("resid",))),           # ... in both k ranges, last row tile of 236 rows
    (320, 1, (577, 9000, 2048, ("swiglu",))),           # two MMAs of 160, last row tile ragged
    (352, 1, (641, 7000, 3080, ("bias", "gelu"))),      # of 192 and 160
    (384, 1, (705, 8200, 4104, ())),                    # two of 192: accumulator and exchange buffer fill tensor memory and ring
    (384, 1, (3000, 2048, 8192, ("resid",))),           # last row tile of 312 rows
    (256, 2, (1000, 2048, 8192, ("resid", "bias"))),
]


@pytest.mark.parametrize("nb,ranges,case", CASES)
def test_swapped_operands_on_pairs_match_the_oracle_alone_and_beside_others(E, nb, ranges, case):  # noqa: F811
    """Against the oracle, and the same bits beside problems of the other kernels (one launch per kernel and k ranges)."""
    assert _plan(E, case) == ("swapped pairs", nb, ranges)
    others = [(200, 768, 768, ("bias",)), (129, 136, 4096, ()), (9, 512, 512, ("bias",)), (700, 3072, 256, ("bias",))]
    assert [_plan(E, c)[0] for c in others] == ["swapped pairs", "swapped", "stream", "tile pairs"]
    probs, refs = _run_gemm(E, E.GEMM_TCGEN05, [case], seed=21)
    ref = refs[0]
    assert_close(probs[0]["C"][:ref.shape[0], :ref.shape[1]], ref, what=f"pair-swapped gemm {case}")
    # (the second run leaves the oracle's product of the large problem out)
    among, _ = _run_gemm(E, E.GEMM_TCGEN05, [case] + others, seed=21, oracle=False)
    assert torch.equal(among[0]["C"][:, :ref.shape[1]], probs[0]["C"][:, :ref.shape[1]])


def test_rows_past_the_live_ones_stay_untouched(E):  # noqa: F811
    """Fewer live rows than a tile holds: what lies behind them in C keeps its bits."""
    M, N, K = 300, 2100, 1000
    g = torch.Generator(device="cuda").manual_seed(22)
    A = torch.randn((M + 84, K), generator=g, device="cuda").to(torch.bfloat16)
    W = (torch.randn((N, K), generator=g, device="cuda") * 0.05).to(torch.bfloat16)
    C = torch.full((M + 84, 2104), 1e30, device="cuda", dtype=torch.bfloat16)
    untouched = C[M:].clone()
    p = [{"A": A, "W": W, "C": C, "M": M, "N": N, "K": K}]
    scratch = torch.empty(E.epara_gemm_scratch_bytes_for(p), dtype=torch.uint8, device="cuda")
    E.epara_grouped_gemm(p, torch.cuda.current_stream().cuda_stream, scratch)
    torch.cuda.synchronize()
    assert int(scratch[:4].view(torch.int32).item()) == 0
    assert torch.equal(C[M:], untouched)
    assert_close(C[:M, :N], A[:M].double().cpu().numpy() @ W.double().cpu().numpy().T, what="live rows")


@pytest.mark.parametrize("capacity,lens,down", [
    (1100, (90, 700, 200), ("swapped pairs", 288, 2)),
    (3000, (90, 1500, 1200), ("swapped pairs", 384, 1)),
])
def test_a_placement_for_many_rows_carries_few(E, capacity, lens, down):  # noqa: F811
    """A decoder layer placed for 1100 or 3000 token rows: a prompt of 90 tokens on its own, with the rows behind it left over from the
    step before, has the bits that it had among the others."""
    from paper_2511_00603_b200 import server, synth
    assert E.epara_gemm_plan(capacity, 2048, 8192, E.EPI_RESID_F32) == down
    p = synth.make_decoder(d=2048, n_layers=1, n_q_heads=32, n_kv_heads=8, head_dim=64, ffn=8192, vocab=300, seed=40, device="cuda", std=0.03,
                           perturb=0.2)
    rng = np.random.default_rng(41)
    pages = [-(-n // synth.PAGE) for n in lens]
    order = rng.permutation(sum(pages)).astype(np.int32)
    tabs = [torch.as_tensor(order[sum(pages[:i]):sum(pages[:i + 1])], device="cuda") for i in range(len(lens))]
    toks = [[int(t) for t in rng.integers(0, 300, n)] for n in lens]
    pool = synth.make_kv_pool(1, sum(pages), 8, 64, seed=42, device="cuda")
    srv = server.Server(workspace_bytes=1 << 30)
    m = srv.add_model(p, kv_pool=pool, max_kv_len=max(lens), max_batch=capacity)

    def answers(which):
        t = [srv.submit(m, E.CAT_FS, tokens=toks[i], kv_len=0, table=tabs[i]) for i in which]
        srv.step()
        torch.cuda.synchronize()
        out = [srv.collect(x) for x in t]
        assert all(s == E.OK for s, _, _ in out)
        return [(logits.clone(), int(a.item())) for _, logits, a in out], pool.clone()

    whole, cache = answers((0, 1, 2))
    for i in (0, 2, 1):
        part, after = answers((i,))
        assert torch.equal(part[0][0], whole[i][0]) and part[0][1] == whole[i][1] and torch.equal(after, cache)
    srv.close()
