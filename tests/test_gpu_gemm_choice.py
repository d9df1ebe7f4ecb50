"""The GEMM kernels for more than 128 rows on problems that the plan gives to each of them (asserted: the choice rests on estimates, and a
problem that moves to another kernel leaves its test empty)."""
import pytest
import torch

from tests.parity import assert_close
from tests.test_gpu_kernels import E, _run_gemm  # noqa: F401  (E: the module's fixture)

pytestmark = pytest.mark.gpu


def _plan(E, case):  # noqa: F811
    M, N, K, fl = case
    flags = {"bias": E.EPI_BIAS, "gelu": E.EPI_GELU, "swiglu": E.EPI_SWIGLU, "resid": E.EPI_RESID_F32}
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return E.epara_gemm_plan(M, N, K, sum(flags[f] for f in fl), sms)


def _check(E, cases, plans, seed):  # noqa: F811
    """All in one call against the oracle; the first one alone has the same bits."""
    assert [_plan(E, c) for c in cases] == plans
    probs, refs = _run_gemm(E, E.GEMM_TCGEN05, cases, seed=seed)
    for p, ref, case in zip(probs, refs, cases):
        assert_close(p["C"][:ref.shape[0], :ref.shape[1]], ref, what=f"gemm {case}")
    alone, _ = _run_gemm(E, E.GEMM_TCGEN05, cases[:1], seed=seed)
    n = refs[0].shape[1]
    assert torch.equal(alone[0]["C"][:, :n], probs[0]["C"][:, :n])


# (last column: K beyond the ring of six stages)
PAIRS = [
    (129, 10, 256, ("bias",)),                # one row in the second half, N below one tile
    (200, 264, 264, ("bias", "gelu")),        # N = 264: eight columns in a third tile
    (256, 2048, 264, ("resid",)),             # K no multiple of a k-block
    (241, 9000, 4104, ("bias",)),             # ... and far beyond the ring
    (256, 9000, 2056, ("swiglu",)),
    (700, 264, 264, ("bias", "gelu")),        # last row tile with rows in its first half only
    (515, 768, 264, ("resid",)),
    (1500, 264, 1544, ("bias", "resid")),
    (1300, 1032, 3080, ("gelu", "bias")),
]


def test_tile_pairs_of_129_rows_and_more(E):  # noqa: F811
    _check(E, PAIRS, [("tile pairs", 128, 1)] * len(PAIRS), seed=31)


# rows of a tile, k ranges, problem: every tile height from 144 to 256 and every number of ranges, N and K with tails
ONE_CTA = [
    (144, 1, (129, 9604, 1032, ("bias",))), (160, 1, (150, 10000, 1544, ("swiglu",))),
    (144, 2, (257, 3072, 2056, ())), (160, 2, (300, 3072, 2056, ("resid",))), (176, 2, (330, 3072, 3080, ("gelu", "bias"))),
    (208, 2, (400, 3072, 3080, ("bias",))),
    (144, 4, (129, 3072, 1544, ("bias", "gelu"))), (160, 4, (150, 3072, 1544, ("swiglu",))), (176, 4, (520, 776, 2056, ("resid", "bias"))),
    (192, 4, (177, 3072, 4104, ())), (208, 4, (193, 3072, 2056, ("resid",))), (224, 4, (1100, 392, 2056, ("bias",))),
    (256, 4, (1000, 392, 8200, ("resid",))), (256, 4, (2000, 264, 3080, ("bias",))),
    (144, 8, (129, 10, 3080, ("bias",))), (160, 8, (150, 10, 4104, ("resid",))), (176, 8, (330, 10, 4104, ("gelu", "bias"))),
    (192, 8, (177, 10, 8200, ())), (208, 8, (193, 10, 8200, ("resid", "bias"))), (224, 8, (220, 10, 8200, ("swiglu",))),
    (240, 8, (690, 10, 8200, ("bias",))), (256, 8, (241, 10, 8200, ("resid",))),
]


@pytest.mark.parametrize("ranges", [1, 2, 4, 8])
def test_swapped_operands_on_one_cta_of_129_rows_and_more(E, ranges):  # noqa: F811
    chosen = [(nb, c) for nb, s, c in ONE_CTA if s == ranges]
    _check(E, [c for _, c in chosen], [("swapped", nb, ranges) for nb, _ in chosen], seed=32 + ranges)
