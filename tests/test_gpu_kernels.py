"""GPU parity of the single kernels against the fp64 oracle, through the C ABI."""
import numpy as np
import pytest
import torch

from oracle import epara_oracle as O
from paper_2511_00603_b200 import synth
from tests.parity import assert_close, to_f64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    from paper_2511_00603_b200 import build
    build.build()
    from paper_2511_00603_b200 import epara
    return epara


def _stream():
    return torch.cuda.current_stream().cuda_stream


GEMM_CASES = [
    # M, N, K, epilogue flags (names)
    (8, 512, 512, ("bias", "gelu")),
    (32, 1024, 256, ("bias",)),
    (197, 2304, 768, ("bias",)),
    (1, 3072, 2048, ()),
    (130, 10, 512, ("bias",)),          # N below one tile, not a multiple of 8
    (300, 1000, 768, ("bias",)),        # ragged M and N
    (33, 512, 256, ("swiglu",)),
    (77, 768, 3072, ("bias", "resid")),
    (0, 64, 64, ()),                    # empty group
    (257, 136, 64, ("gelu", "bias")),   # single k-block, N tail of 8
    (40, 1024, 1024, ("swiglu",)),      # the largest matrix of the weight-streaming kernel at more than 16 rows
    (256, 2048, 4096, ("resid",)),      # long K, split over a cluster of four
    (64, 512, 8192, ("bias", "resid")), # few tiles, very long K: split over a cluster of eight
    (20, 768, 4096, ("gelu", "bias")),  # split along K, bf16 output
    # at most 16 rows: the weight-streaming kernel (16 W rows per block, k-blocks of 32 dealt to 16 warps)
    (9, 256, 5120, ("swiglu",)),        # long K, SwiGLU
    (16, 1000, 776, ("bias",)),         # ragged N, K not a multiple of 32
    (3, 10, 512, ("bias",)),            # N below one block
    (5, 64, 8, ()),                     # a single 16-byte piece of K
    (12, 2048, 8192, ("resid",)),       # long K, fp32 residual
    (2, 512, 2048, ("swiglu",)),
    (1, 32000, 2048, ()),               # LM head of one request
]


def _run_gemm(E, impl, cases, seed=0, oracle=True):
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(seed)
    probs, refs = [], []
    for (M, N, K, fl) in cases:
        A = torch.randn((max(M, 1), K), generator=g, device=dev).to(torch.bfloat16)
        W = (torch.randn((N, K), generator=g, device=dev) * 0.05).to(torch.bfloat16)
        bias = (torch.randn((N,), generator=g, device=dev) * 0.5).to(torch.bfloat16) if "bias" in fl else None
        epi = (E.EPI_BIAS if "bias" in fl else 0) | (E.EPI_GELU if "gelu" in fl else 0) | \
              (E.EPI_SWIGLU if "swiglu" in fl else 0) | (E.EPI_RESID_F32 if "resid" in fl else 0)
        ldc = ((N // 2 if "swiglu" in fl else N) + 7) // 8 * 8
        if "resid" in fl:
            Cc = torch.randn((max(M, 1), ldc), generator=g, device=dev, dtype=torch.float32)
        else:
            Cc = torch.full((max(M, 1), ldc), float("nan"), device=dev, dtype=torch.bfloat16)
        C0 = Cc.clone()
        probs.append({"A": A, "W": W, "C": Cc, "bias": bias, "M": M, "N": N, "K": K, "epilogue": epi})
        if not oracle:
            continue
        y = O.linear(O.bf16_to_f64(synth.to_bits(A))[:M], O.bf16_to_f64(synth.to_bits(W)),
                     O.bf16_to_f64(synth.to_bits(bias)) if bias is not None else None)
        if "gelu" in fl:
            y = O.gelu(y)
        if "swiglu" in fl:
            y = O.silu(y[:, 0::2]) * y[:, 1::2]
        if "resid" in fl:
            y = C0[:M, :N].double().cpu().numpy() + y
        refs.append(y)
    scratch = torch.empty(E.epara_gemm_scratch_bytes_for(probs), dtype=torch.uint8, device=dev)
    E.epara_grouped_gemm(probs, _stream(), scratch, impl=impl)
    torch.cuda.synchronize()
    status = int(scratch[:4].view(torch.int32).item())
    assert status == 0, f"device status {status}"
    return probs, refs


@pytest.mark.parametrize("impl", ["simt", "tcgen05"])
def test_grouped_gemm_matches_oracle(E, impl):
    probs, refs = _run_gemm(E, E.GEMM_SIMT if impl == "simt" else E.GEMM_TCGEN05, GEMM_CASES)
    for p, ref, case in zip(probs, refs, GEMM_CASES):
        M, ncols = ref.shape
        if M == 0:
            continue
        assert_close(p["C"][:M, :ncols], ref, what=f"{impl} gemm {case}")
        if impl == "simt" and p["C"].dtype == torch.bfloat16 and p["C"].shape[1] > ncols:
            # (the tensor-core kernel stores through TMA in 16-byte units and may fill the pad
            # columns up to the next multiple of 8, which the C ABI allows)
            assert torch.isnan(p["C"][:M, ncols:].float()).all(), "wrote beyond N"


def test_grouped_gemm_many_tiles_and_group_independence(E):
    """More tiles than SMs, several k-blocks beyond the stage ring, and the same problem alone vs
    among others gives bit-identical output (no dependence on co-resident groups)."""
    big = [(1576, 768, 768, ("bias",)), (640, 3072, 768, ("bias", "gelu")), (1000, 768, 3072, ("bias", "resid"))]
    probs, refs = _run_gemm(E, E.GEMM_TCGEN05, big, seed=3)
    for p, ref, case in zip(probs, refs, big):
        assert_close(p["C"][:ref.shape[0], :ref.shape[1]], ref, what=f"gemm {case}")
    alone, _ = _run_gemm(E, E.GEMM_TCGEN05, big[:1], seed=3)
    assert torch.equal(alone[0]["C"], probs[0]["C"])


@pytest.mark.parametrize("M", [17, 32, 33, 65, 127, 128])
def test_grouped_gemm_small_matrices_in_tiles_of_32_rows(E, M):
    """Matrices of up to a million elements with 17 to 128 rows run in the weight-streaming kernel in tiles of 32 rows:
    row counts at the edges of a tile, N below one block and not a multiple of it, one 16-byte piece of K, K that is no
    multiple of a k-block, every epilogue, the largest matrix; a group of few rows in the same launch and the problem
    alone give the same bits."""
    cases = [(M, 10, 512, ("bias",)), (M, 1000, 776, ("bias", "gelu")), (M, 24, 8, ()), (M, 512, 2048, ("resid",)),
             (M, 512, 256, ("swiglu",)), (3, 520, 512, ("bias",))]
    probs, refs = _run_gemm(E, E.GEMM_TCGEN05, cases, seed=M)
    for p, ref, case in zip(probs, refs, cases):
        assert_close(p["C"][:ref.shape[0], :ref.shape[1]], ref, what=f"small gemm {case}")
    alone, _ = _run_gemm(E, E.GEMM_TCGEN05, cases[:1], seed=M)
    assert torch.equal(alone[0]["C"][:, :10], probs[0]["C"][:, :10])     # (the columns that pad the rows stay NaN)


def test_grouped_gemm_tile_pairs(E):
    """Problems of more than 128 rows.  256-row tiles on CTA pairs 128 columns wide (wider ones: test_grouped_gemm_wide_tile_pairs;
    129 to 256 rows, N below one tile, a K beyond the stage ring: tests/test_gpu_gemm_choice.py): ragged last pair (one CTA with no valid
    row), N tails, SwiGLU, one k-block, more pairs than SM pairs, fp32-residual outputs.  (700, 264, 1536), (384, 256, 4096),
    (515, 768, 1536), (200, 512, 512), (256, 2048, 2048) and (129, 10, 512) go to the swapped operands on CTA pairs, in the same call."""
    cases = [(1000, 1152, 384, ("bias",)), (513, 2048, 256, ("swiglu",)), (700, 264, 1536, ("bias", "gelu")),
             (257, 392, 64, ()), (20000, 512, 128, ("bias",)), (384, 256, 4096, ("gelu", "bias")),
             (900, 384, 384, ("bias", "resid")), (515, 768, 1536, ("resid",)), (1300, 576, 192, ("bias", "resid")),
             (200, 512, 512, ("bias", "gelu")), (256, 2048, 2048, ("resid",)), (129, 10, 512, ("bias",))]
    probs, refs = _run_gemm(E, E.GEMM_TCGEN05, cases, seed=9)
    for p, ref, case in zip(probs, refs, cases):
        assert_close(p["C"][:ref.shape[0], :ref.shape[1]], ref, what=f"pair gemm {case}")
    alone, _ = _run_gemm(E, E.GEMM_TCGEN05, cases[:1], seed=9)
    assert torch.equal(alone[0]["C"], probs[0]["C"])


def test_grouped_gemm_swapped_operands_17_to_128_rows(E):
    """Problems of 17 to 128 rows with matrices of more than a million elements run with W as the tensor core's 128-row
    operand and the batch as its N, a cluster of 1, 2, 4 or 8 CTAs per tile of 128 output columns splitting K (reduced
    through distributed shared memory in rank order): the decode shapes of the 1B decoder, batch sizes on both sides of
    the multiples of 16, beside smaller matrices, which go to the weight-streaming kernel in the same call (tails of N and K:
    test_grouped_gemm_swapped_operands_tails).  The same problem alone and among others gives the same bits."""
    cases = [(17, 10, 512, ("bias",)), (128, 3072, 2048, ()), (100, 1000, 776, ("bias",)), (48, 2048, 8192, ("resid",)),
             (33, 512, 256, ("swiglu",)), (64, 2048, 2048, ("resid", "bias")), (127, 16384, 2048, ("swiglu",)),
             (32, 1024, 256, ("bias", "gelu")), (96, 136, 64, ("gelu", "bias")), (20, 768, 4096, ("gelu", "bias")),
             (128, 32000, 2048, ()), (31, 264, 1536, ("bias", "resid")), (80, 4096, 4096, ("swiglu",))]
    probs, refs = _run_gemm(E, E.GEMM_TCGEN05, cases, seed=11)
    for p, ref, case in zip(probs, refs, cases):
        assert_close(p["C"][:ref.shape[0], :ref.shape[1]], ref, what=f"swapped gemm {case}")
    alone, _ = _run_gemm(E, E.GEMM_TCGEN05, cases[:2], seed=11)
    assert torch.equal(alone[1]["C"], probs[1]["C"])
    # fewer live rows than the capacity the tile was sized for leave the other rows' outputs untouched
    M, N, K = 128, 512, 512
    g = torch.Generator(device="cuda").manual_seed(12)
    A = torch.randn((M, K), generator=g, device="cuda").to(torch.bfloat16)
    W = (torch.randn((N, K), generator=g, device="cuda") * 0.05).to(torch.bfloat16)
    full = torch.zeros((M, N), device="cuda", dtype=torch.bfloat16)
    part = torch.full((M, N), 7.0, device="cuda", dtype=torch.bfloat16)
    for C_, rows in ((full, M), (part, 40)):
        pr = [{"A": A, "W": W, "C": C_, "bias": None, "M": rows, "N": N, "K": K, "epilogue": 0}]
        sc = torch.empty(E.epara_gemm_scratch_bytes_for(pr), dtype=torch.uint8, device="cuda")
        E.epara_grouped_gemm(pr, _stream(), sc)
    torch.cuda.synchronize()
    assert bool((part[40:] == 7.0).all())
    assert_close(part[:40], to_f64(full[:40]), what="first 40 rows", tol=1e-6)


def test_grouped_gemm_swapped_operands_tails(E):
    """17 to 128 rows and matrices of more than a million elements (smaller ones go to the weight-streaming kernel): N no
    multiple of a tile, of a vector store or of two, K no multiple of a k-block, clusters of 1, 2, 4 and 8, every epilogue,
    row counts on both sides of the multiples of 16.  Alone and among others: the same bits.  Rows past the live ones, in
    a matrix that has more, keep what they hold."""
    cases = [(17, 1000, 1544, ("bias",)), (33, 4100, 264, ("gelu", "bias")), (64, 4102, 520, ("swiglu",)), (100, 8200, 2056, ()),
             (128, 1030, 4104, ("resid",)), (96, 264, 8200, ("bias", "resid")), (50, 32001, 72, ("bias",)), (40, 1034, 1160, ("swiglu",))]
    probs, refs = _run_gemm(E, E.GEMM_TCGEN05, cases, seed=21)
    for p, ref, case in zip(probs, refs, cases):
        assert_close(p["C"][:ref.shape[0], :ref.shape[1]], ref, what=f"swapped gemm {case}")
    alone, _ = _run_gemm(E, E.GEMM_TCGEN05, cases[:2], seed=21)
    assert torch.equal(alone[1]["C"][:, :4100], probs[1]["C"][:, :4100])
    M, N, K = 128, 1032, 4104
    g = torch.Generator(device="cuda").manual_seed(22)
    A = torch.randn((M, K), generator=g, device="cuda").to(torch.bfloat16)
    W = (torch.randn((N, K), generator=g, device="cuda") * 0.05).to(torch.bfloat16)
    for rows in (40, 17, 113):
        full = torch.full((M, N), 7.0, device="cuda", dtype=torch.bfloat16)
        part = full.clone()
        for C_, n in ((full, M), (part, rows)):
            pr = [{"A": A, "W": W, "C": C_, "bias": None, "M": n, "N": N, "K": K, "epilogue": 0}]
            sc = torch.empty(E.epara_gemm_scratch_bytes_for(pr), dtype=torch.uint8, device="cuda")
            E.epara_grouped_gemm(pr, _stream(), sc)
        torch.cuda.synchronize()
        assert bool((part[rows:] == 7.0).all()) and torch.equal(part[:rows], full[:rows])


def test_grouped_gemm_wide_tile_pairs(E):
    """Tile pairs 256 and 192 columns wide: N tails in either half of the W rows, ragged last rows, more tiles than pairs (a
    pair's second tile uses the other accumulator), K no multiple of a k-block, every epilogue."""
    cases = [(900, 8200, 520, ("bias", "gelu")), (1537, 4200, 1096, ("swiglu",)), (1025, 6000, 1160, ("bias", "resid")),
             (1500, 3264, 1160, ("resid",)), (900, 5184, 712, ("bias", "resid"))]
    probs, refs = _run_gemm(E, E.GEMM_TCGEN05, cases, seed=23)
    for p, ref, case in zip(probs, refs, cases):
        assert_close(p["C"][:ref.shape[0], :ref.shape[1]], ref, what=f"wide pair gemm {case}")
    alone, _ = _run_gemm(E, E.GEMM_TCGEN05, cases[:1], seed=23)
    assert torch.equal(alone[0]["C"], probs[0]["C"])


def test_grouped_gemm_rejects_bad_arguments(E):
    dev = torch.device("cuda")
    A = torch.zeros((8, 64), device=dev, dtype=torch.bfloat16)
    W = torch.zeros((8, 64), device=dev, dtype=torch.bfloat16)
    Cc = torch.zeros((8, 8), device=dev, dtype=torch.bfloat16)
    scratch = torch.empty(4096, dtype=torch.uint8, device=dev)
    bad = {"A": A[:, 1:], "W": W, "C": Cc, "M": 8, "N": 8, "K": 63, "epilogue": 0}
    with pytest.raises(E.EparaError) as ei:
        E.epara_grouped_gemm([bad], _stream(), scratch)
    assert ei.value.status == E.E_INVALID
    small = torch.empty(256, dtype=torch.uint8, device=dev)
    ok = {"A": A, "W": W, "C": Cc, "M": 8, "N": 8, "K": 64, "epilogue": 0}
    with pytest.raises(E.EparaError) as ei:
        E.epara_grouped_gemm([ok], _stream(), small)
    assert ei.value.status == E.E_RESOURCE


@pytest.mark.parametrize("Hq,Hkv,hd", [(8, 2, 64), (8, 2, 128), (4, 4, 64), (4, 2, 16)])
def test_decode_attention_matches_oracle(E, Hq, Hkv, hd):
    dev = torch.device("cuda")
    lens = np.array([1, 16, 17, 255, 256, 257, 700, 1023], dtype=np.int32)
    B = len(lens)
    need = [(int(L) + 15) // 16 for L in lens]
    npages = sum(need) + 3
    rng = np.random.default_rng(5)
    perm = rng.permutation(npages).astype(np.int32)
    stride = max(need)
    tables = np.zeros((B, stride), dtype=np.int32)
    o = 0
    for b, n in enumerate(need):
        tables[b, :n] = perm[o:o + n]
        o += n
    pool = synth.make_kv_pool(1, npages, Hkv, hd, seed=6, device=dev)[0]
    # poison the slots past each request's length: they must never be read
    pool_ref = synth.to_bits(pool)
    for b, L in enumerate(lens):
        if L % 16:
            pool[int(tables[b, need[b] - 1]), :, :, L % 16:, :] = float("nan")
    q = torch.randn((B, Hq * hd), generator=torch.Generator(device=dev).manual_seed(7), device=dev).to(torch.bfloat16)
    out = torch.empty((B, Hq * hd), device=dev, dtype=torch.bfloat16)
    max_len = int(lens.max())
    scratch = torch.empty(E.lib.epara_decode_attention_scratch_bytes(B, Hq, hd, max_len), dtype=torch.uint8, device=dev)
    E.epara_decode_attention(q, pool, torch.as_tensor(lens, device=dev), torch.as_tensor(tables, device=dev), out,
                             Hq, Hkv, hd, max_len, scratch, _stream())
    torch.cuda.synchronize()
    qf = O.bf16_to_f64(synth.to_bits(q)).reshape(B, Hq, hd)
    for b, L in enumerate(lens):
        K, V = O.gather_kv(lambda l, pg: pool_ref[pg], 0, tables[b], int(L))
        ref = np.stack([O.attention(qf[b, h], K[h // (Hq // Hkv)], V[h // (Hq // Hkv)]) for h in range(Hq)])
        assert_close(out[b].reshape(Hq, hd), ref, what=f"decode attention b={b} L={L}")


@pytest.mark.parametrize("rows", [16, 100, 200, 1024])
def test_gelu_epilogue_sweep_through_identity_gemm(E, rows):
    """The device GELU over its whole range: x swept over [-8, 8] (every bf16 value of a fine grid) goes through a
    GEMM with the identity as weights, so the accumulator holds x exactly and the epilogue alone decides the
    output.  Bound: the fitted form's 2.6e-5, the hardware tanh's relative error 2^-11 scaled by 0.5 |x|
    (2.5e-4 |x|), and the rounding of the bf16 store (half an ulp: at most 2^-8 of the result).  The row counts select the
    weight-streaming kernel (16 rows and 100) and the tile-pair kernel; the swapped operands have a sweep of their own."""
    dev = torch.device("cuda")
    K = N = 256
    x = torch.linspace(-8.0, 8.0, rows * K, device=dev).reshape(rows, K)
    x = x[:, torch.randperm(K, generator=torch.Generator(device=dev).manual_seed(rows), device=dev)].to(torch.bfloat16)
    W = torch.eye(N, K, device=dev).to(torch.bfloat16)
    C = torch.full((rows, N), float("nan"), device=dev, dtype=torch.bfloat16)
    prob = [{"A": x, "W": W, "C": C, "bias": None, "M": rows, "N": N, "K": K, "epilogue": E.EPI_GELU}]
    scratch = torch.empty(E.epara_gemm_scratch_bytes_for(prob), dtype=torch.uint8, device=dev)
    E.epara_grouped_gemm(prob, _stream(), scratch, impl=E.GEMM_TCGEN05)
    torch.cuda.synchronize()
    assert int(scratch[:4].view(torch.int32).item()) == 0
    xs = O.bf16_to_f64(synth.to_bits(x))
    ref = O.gelu(xs)
    got = to_f64(C)
    bound = 2.6e-5 + 2.5e-4 * np.abs(xs) + 2.0 ** -8 * np.abs(ref) + 1e-7
    bad = np.abs(got - ref) > bound
    assert not bad.any(), f"{int(bad.sum())} of {bad.size} outside the bound; worst excess " \
                          f"{float(np.max(np.abs(got - ref) - bound)):.3e} at x = {float(xs[np.unravel_index(np.argmax(np.abs(got - ref) - bound), xs.shape)])}"


def test_gelu_epilogue_sweep_through_the_swapped_operands(E):
    """The sweep of the test above through the swapped-operand kernel, which takes identities of more than a million elements at
    100 rows."""
    dev = torch.device("cuda")
    rows, K = 100, 1032
    x = torch.linspace(-8.0, 8.0, rows * K, device=dev).reshape(rows, K)
    x = x[:, torch.randperm(K, generator=torch.Generator(device=dev).manual_seed(rows), device=dev)].to(torch.bfloat16)
    C = torch.full((rows, K), float("nan"), device=dev, dtype=torch.bfloat16)
    prob = [{"A": x, "W": torch.eye(K, device=dev).to(torch.bfloat16), "C": C, "bias": None, "M": rows, "N": K, "K": K, "epilogue": E.EPI_GELU}]
    scratch = torch.empty(E.epara_gemm_scratch_bytes_for(prob), dtype=torch.uint8, device=dev)
    E.epara_grouped_gemm(prob, _stream(), scratch)
    torch.cuda.synchronize()
    xs = O.bf16_to_f64(synth.to_bits(x))
    ref = O.gelu(xs)
    assert not (np.abs(to_f64(C) - ref) > 2.6e-5 + 2.5e-4 * np.abs(xs) + 2.0 ** -8 * np.abs(ref) + 1e-7).any()


@pytest.mark.parametrize("rows", [129, 197, 256, 257, 509, 1024])
def test_grouped_gemm_between_one_tile_and_a_full_chip(E, rows):
    """Problems of 129 to about a thousand rows, on whichever of the kernels the plan gives them: swapped operands on CTA pairs, on one CTA
    with K split over 2, 4 or 8 (each by itself: tests/test_gpu_swap_pairs.py, tests/test_gpu_gemm_choice.py), or tile pairs.  N below and
    not a multiple of a tile, K not a multiple of a k-block."""
    cases = [(rows, 768, 3072, ("bias", "resid")), (rows, 2048, 8192, ("resid",)), (rows, 136, 4096, ("bias", "gelu")),
             (rows, 264, 2056, ("swiglu",)), (rows, 1000, 1544, ("bias",)), (rows, 3072, 512, ()), (rows, 4096, 1024, ("swiglu",))]
    probs, refs = _run_gemm(E, E.GEMM_TCGEN05, cases, seed=rows)
    for p, ref, case in zip(probs, refs, cases):
        assert_close(p["C"][:ref.shape[0], :ref.shape[1]], ref, what=f"gemm {case}")
    alone, _ = _run_gemm(E, E.GEMM_TCGEN05, cases[:2], seed=rows)
    assert torch.equal(alone[1]["C"], probs[1]["C"])


@pytest.mark.parametrize("hd,Hq,Hkv", [(16, 4, 2), (64, 8, 2), (128, 4, 4)])
@pytest.mark.parametrize("B", [5, 100, 420])
def test_decode_attention_writes_out_at_any_bf16_boundary(E, hd, Hq, Hkv, B):
    """`out` one element past an aligned address: requests of one chunk and of several, merged by the second kernel and (100
    requests, head sizes up to 64) by the last block to arrive.  The same bits as in an aligned tensor, and nothing beside it."""
    dev = torch.device("cuda")
    lens = np.resize(np.array([700, 1, 256, 257, 530], dtype=np.int32), B)
    tables = torch.arange(44, dtype=torch.int32, device=dev).repeat(B, 1)
    pool = synth.make_kv_pool(1, 44, Hkv, hd, seed=31, device=dev)[0]
    q = torch.randn((B, Hq * hd), generator=torch.Generator(device=dev).manual_seed(32), device=dev).to(torch.bfloat16)
    scratch = torch.empty(E.lib.epara_decode_attention_scratch_bytes(B, Hq, hd, 700), dtype=torch.uint8, device=dev)
    buf = torch.full((B * Hq * hd + 2,), 9.0, device=dev, dtype=torch.bfloat16)
    ref, odd = torch.empty_like(q), buf[1:-1].view(B, Hq * hd)
    for out in (ref, odd):
        E.epara_decode_attention(q, pool, torch.as_tensor(lens, device=dev), tables, out, Hq, Hkv, hd, 700, scratch, _stream())
    torch.cuda.synchronize()
    assert torch.equal(ref, odd) and float(buf[0]) == 9.0 and float(buf[-1]) == 9.0
    for _ in range(2):                                  # (the second call finds the counters as the first left them)
        odd.zero_()
        E.epara_decode_attention_static(q, pool, torch.as_tensor(lens, device=dev), tables, odd, Hq, Hkv, hd, 700, _stream())
        torch.cuda.synchronize()
        assert torch.equal(ref, odd) and float(buf[0]) == 9.0 and float(buf[-1]) == 9.0


@pytest.mark.parametrize("M,N,K,fl,ldc", [(5, 100, 512, ("bias",), 101), (100, 250, 264, ("gelu", "bias"), 253), (64, 2048, 2048, ("resid",), 2052),
                                          (100, 1030, 1544, (), 1036), (33, 4096, 512, ("swiglu",), 2050), (300, 264, 512, ("resid",), 268)])
def test_grouped_gemm_takes_row_strides_of_c_that_its_kernels_can_store(E, M, N, K, fl, ldc):
    """Strides of C that are no multiple of 8: any for the weight-streaming kernel, four (SwiGLU: two) elements for the
    swapped operands up to 128 rows, 16 bytes above."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(M)
    A = torch.randn((M, K), generator=g, device=dev).to(torch.bfloat16)
    W = (torch.randn((N, K), generator=g, device=dev) * 0.05).to(torch.bfloat16)
    bias = torch.randn((N,), generator=g, device=dev).to(torch.bfloat16) if "bias" in fl else None
    epi = sum({"bias": E.EPI_BIAS, "gelu": E.EPI_GELU, "swiglu": E.EPI_SWIGLU, "resid": E.EPI_RESID_F32}[f] for f in fl)
    n_out = N // 2 if "swiglu" in fl else N
    C0 = torch.randn((M, ldc), generator=g, device=dev) if "resid" in fl else torch.zeros((M, ldc), device=dev, dtype=torch.bfloat16)
    wide = torch.zeros((M, (ldc + 7) // 8 * 8), device=dev, dtype=C0.dtype)
    wide[:, :ldc] = C0
    C = C0.clone()
    for out in (C, wide):
        prob = [{"A": A, "W": W, "C": out, "bias": bias, "M": M, "N": N, "K": K, "epilogue": epi}]
        scratch = torch.empty(E.epara_gemm_scratch_bytes_for(prob), dtype=torch.uint8, device=dev)
        E.epara_grouped_gemm(prob, _stream(), scratch)
    torch.cuda.synchronize()
    assert torch.equal(C[:, :n_out], wide[:, :n_out]) and bool((C[:, :n_out] != C0[:, :n_out]).any())
    pad = n_out + (-n_out) % (4 if "resid" in fl else 8)              # columns up to there may be overwritten
    assert torch.equal(C[:, pad:], C0[:, pad:])


@pytest.mark.parametrize("hd,Hq,Hkv", [(64, 8, 2), (128, 4, 4), (32, 4, 1)])
def test_decode_attention_merges_any_number_of_chunks(E, hd, Hq, Hkv):
    """16, 17, 32, 33 and 41 chunks of 256 tokens, whose partials are merged 16 at a time, and few: against the oracle, and with
    the same bits among more requests.  The keys of the later chunks are larger, so that the maximum of a later group of
    chunks is the larger one."""
    dev = torch.device("cuda")
    lens = np.array([4096, 4097, 8192, 8193, 10300, 700, 30], dtype=np.int32)
    B, n_pages = len(lens), (10300 + 15) // 16
    table = np.random.default_rng(41).permutation(n_pages).astype(np.int32)
    pool = synth.make_kv_pool(1, n_pages, Hkv, hd, seed=42, device=dev)[0]
    for i, pg in enumerate(table):
        pool[int(pg), 0] *= 0.5 + 2.0 * i / n_pages
    outs = []
    for times in (1, 40):
        n = B * times
        q = torch.randn((B, Hq * hd), generator=torch.Generator(device=dev).manual_seed(43), device=dev).to(torch.bfloat16).repeat(times, 1)
        out = torch.empty_like(q)
        scratch = torch.empty(E.lib.epara_decode_attention_scratch_bytes(n, Hq, hd, 10300), dtype=torch.uint8, device=dev)
        E.epara_decode_attention(q, pool, torch.as_tensor(np.tile(lens, times), device=dev), torch.as_tensor(table, device=dev).repeat(n, 1), out,
                                 Hq, Hkv, hd, 10300, scratch, _stream())
        torch.cuda.synchronize()
        outs.append((q, out))
    q, out = outs[0]
    assert torch.equal(outs[1][1], out.repeat(40, 1))
    pool_bits, qf = synth.to_bits(pool), O.bf16_to_f64(synth.to_bits(q)).reshape(B, Hq, hd)
    for b, L in enumerate(lens):
        K, V = O.gather_kv(lambda l, pg: pool_bits[pg], 0, table, int(L))
        ref = np.stack([O.attention(qf[b, h], K[h // (Hq // Hkv)], V[h // (Hq // Hkv)]) for h in range(Hq)])
        assert_close(out[b].reshape(Hq, hd), ref, what=f"decode attention of {L} tokens")


@pytest.mark.parametrize("hd,Hq,Hkv", [(16, 4, 2), (64, 8, 2), (64, 8, 1), (128, 4, 4)])
def test_decode_attention_merge_in_the_kernel_and_after_it_give_the_same_bits(E, hd, Hq, Hkv):
    """Requests of up to four chunks: few and very many of them are merged by the second kernel, some hundred blocks (three
    to ten per SM) at head sizes up to 64 by the block that arrives last.  A request has the same bits in all of them."""
    dev = torch.device("cuda")
    lens = np.array([1000, 1, 256, 257, 530, 1024, 700, 40], dtype=np.int32)
    tables = torch.arange(64, dtype=torch.int32, device=dev)
    pool = synth.make_kv_pool(1, 64, Hkv, hd, seed=51, device=dev)[0]
    q = torch.randn((8, Hq * hd), generator=torch.Generator(device=dev).manual_seed(52), device=dev).to(torch.bfloat16)
    outs = []
    for n in (1, -(-3 * 148 // (8 * 4 * Hkv)), 10 * 148 // (8 * 4 * Hkv), 10 * 148 // (8 * 4 * Hkv) + 1):
        out = torch.empty((8 * n, Hq * hd), device=dev, dtype=torch.bfloat16)
        scratch = torch.empty(E.lib.epara_decode_attention_scratch_bytes(8 * n, Hq, hd, 1024), dtype=torch.uint8, device=dev)
        E.epara_decode_attention(q.repeat(n, 1), pool, torch.as_tensor(np.tile(lens, n), device=dev), tables.repeat(8 * n, 1), out, Hq, Hkv, hd,
                                 1024, scratch, _stream())
        torch.cuda.synchronize()
        assert torch.equal(out, out[:8].repeat(n, 1))
        outs.append(out[:8])
    assert all(torch.equal(o, outs[0]) for o in outs)
