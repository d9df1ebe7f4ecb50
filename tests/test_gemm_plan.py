"""Which kernel, tile and K split a GEMM gets (host only; 148 SMs)."""
import pytest


@pytest.fixture(scope="module")
def E():
    from paper_2511_00603_b200 import build
    build.build()
    from paper_2511_00603_b200 import epara
    return epara


def test_plan_names_the_kernel_by_rows(E):
    """The 1B decoder's down projection from one row to thousands."""
    kinds = [E.epara_gemm_plan(m, 2048, 8192, E.EPI_RESID_F32)[0] for m in (1, 16, 17, 128, 1100, 8192)]
    assert kinds == ["stream", "stream", "swapped", "swapped", "swapped pairs", "tile pairs"]
    assert E.epara_gemm_plan(100, 1024, 1024) == ("stream", 16, 1)        # a matrix of 2^20 elements


@pytest.mark.parametrize("bad", [(0, 8, 8), (8, 0, 8), (8, 8, 0)])
def test_plan_refuses_empty_problems(E, bad):
    with pytest.raises(E.EparaError):
        E.epara_gemm_plan(*bad)
    assert E.lib.epara_gemm_plan(8, 8, 8, 0, 148, None, None) == E.E_INVALID


# rows, N, K, epilogue flags, kernel and tile that measured faster
MEASURED = [
    (336, 2048, 8192, 8, "swapped", 176), (400, 2048, 8192, 8, "swapped", 208), (512, 2048, 8192, 8, "swapped pairs", 128),
    (192, 4096, 14336, 8, "swapped", 192), (224, 4096, 14336, 8, "swapped", 224), (256, 4096, 14336, 8, "swapped pairs", 128),
    (129, 4096, 4096, 8, "swapped", 144), (208, 4096, 4096, 8, "swapped pairs", 128), (256, 6144, 4096, 0, "swapped pairs", 96),
    (1100, 2048, 8192, 8, "swapped pairs", 288), (3000, 2048, 8192, 8, "swapped pairs", 384), (8192, 2048, 8192, 8, "tile pairs", 256),
]


@pytest.mark.parametrize("rows,N,K,epi,kernel,tile", MEASURED)
def test_plan_takes_the_kernel_that_measured_faster(E, rows, N, K, epi, kernel, tile):
    assert E.epara_gemm_plan(rows, N, K, epi)[:2] == (kernel, tile)


def test_gpu_problems_get_the_kernels_they_are_written_for(E):
    """The GPU tests of a kernel assert its plan before they run; the same here, where a changed estimate shows without a GPU."""
    from tests import test_gpu_gemm_choice as choice, test_gpu_swap_pairs as pairs
    flags = {"bias": E.EPI_BIAS, "gelu": E.EPI_GELU, "swiglu": E.EPI_SWIGLU, "resid": E.EPI_RESID_F32}
    for want, (M, N, K, fl) in ([(("tile pairs", 128, 1), c) for c in choice.PAIRS] + [(("swapped", nb, s), c) for nb, s, c in choice.ONE_CTA] +
                                [(("swapped pairs", nb, s), c) for nb, s, c in pairs.CASES]):
        assert E.epara_gemm_plan(M, N, K, sum(flags[f] for f in fl)) == want, (M, N, K, fl)
