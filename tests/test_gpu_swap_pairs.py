"""The swapped-operand GEMM on pairs of CTAs (256 output columns a tile, up to 384 batch rows, one or two k ranges)."""
import pytest
import torch

from tests.parity import assert_close
from tests.test_gpu_kernels import E, _run_gemm  # noqa: F401  (E: the module's fixture)

pytestmark = pytest.mark.gpu

# M, N, K, epilogue: row tile and k ranges it gets
CASES = [
    (129, 264, 768, ("bias", "gelu")),         # 64, two: last columns in the first CTA of a pair only, last row tile of one row
    (161, 2100, 2048, ("bias",)),              # 64, two: N not a multiple of 8, stage ring used several times over
    (289, 1032, 3080, ()),                     # 64, two: K not a multiple of a k-block, ranges of 25 and 24
    (385, 520, 1000, ("resid",)),              # 64, two: fp32 residual
    (330, 2100, 3080, ("gelu", "bias")),       # 128, two
    (385, 2100, 3080, ("swiglu",)),            # 160, two
    (300, 2100, 1000, ("bias", "resid")),      # 64, one
    (330, 9000, 3080, ("bias",)),              # 192, one
    (280, 16384, 2048, ("swiglu",)),           # 288, one: two MMAs, of 160 and 128 rows
    (577, 9000, 2048, ("swiglu",)),            # 320, one: two MMAs of 160, last row tile ragged
    (1000, 2048, 8192, ("resid", "bias")),     # 256, two
]


@pytest.mark.parametrize("case", CASES)
def test_swapped_operands_on_pairs_match_the_oracle_alone_and_beside_others(E, case):  # noqa: F811
    """Against the oracle, and the same bits beside problems of the other kernels (one launch per kernel and k ranges)."""
    probs, refs = _run_gemm(E, E.GEMM_TCGEN05, [case], seed=21)
    ref = refs[0]
    assert_close(probs[0]["C"][:ref.shape[0], :ref.shape[1]], ref, what=f"pair-swapped gemm {case}")
    among, _ = _run_gemm(E, E.GEMM_TCGEN05, [case, (200, 768, 768, ("bias",)), (300, 520, 3080, ()), (9, 512, 512, ("bias",)), (700, 3072, 256, ("bias",))], seed=21)
    assert torch.equal(among[0]["C"][:, :ref.shape[1]], probs[0]["C"][:, :ref.shape[1]])


def test_rows_past_the_live_ones_stay_untouched(E):  # noqa: F811
    """Fewer live rows than a tile holds: what lies behind them in C keeps its bits."""
    M, N, K = 300, 2100, 1000
    g = torch.Generator(device="cuda").manual_seed(22)
    A = torch.randn((M + 84, K), generator=g, device="cuda").to(torch.bfloat16)
    W = (torch.randn((N, K), generator=g, device="cuda") * 0.05).to(torch.bfloat16)
    C = torch.full((M + 84, 2104), 7.0, device="cuda", dtype=torch.bfloat16)
    p = [{"A": A, "W": W, "C": C, "M": M, "N": N, "K": K}]
    scratch = torch.empty(E.epara_gemm_scratch_bytes_for(p), dtype=torch.uint8, device="cuda")
    E.epara_grouped_gemm(p, torch.cuda.current_stream().cuda_stream, scratch)
    torch.cuda.synchronize()
    assert int(scratch[:4].view(torch.int32).item()) == 0
    assert torch.all(C[M:] == 7.0) and not torch.any(C[:M, :N] == 7.0)
