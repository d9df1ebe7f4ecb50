"""CPU tests: the library loads, exports what the header declares, and its host policy
(admission, Eq. 4, Eq. 5) agrees with the oracle.  No GPU compute is called."""
import ctypes
import os
import re
import shutil
import subprocess
import sys
import sysconfig
import threading
import time
import types

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def E():
    from paper_2511_00603_b200 import build
    build.build()
    from paper_2511_00603_b200 import epara
    return epara


def test_library_exports_every_declared_symbol(E):
    hdr = open(os.path.join(ROOT, "include", "epara.h")).read()
    hdr = re.sub(r"/\*.*?\*/", "", hdr, flags=re.S)
    declared = set(re.findall(r"\b(epara_[a-z_0-9]+)\s*\(", hdr))
    assert {"epara_register_model", "epara_submit", "epara_step", "epara_collect"} <= declared
    for name in declared:
        assert hasattr(E.lib, name), name
    assert declared == set(E.EXPORTS)


def test_strerror_and_null_arguments(E):
    assert E.lib.epara_strerror(E.E_TIMEOUT) == b"timeout"
    assert E.lib.epara_strerror(E.E_RESOURCE) == b"resource insufficiency"
    assert E.lib.epara_init(None, None) == E.E_INVALID
    assert E.lib.epara_submit(None, 0, 0, None, None) == E.E_INVALID
    assert E.lib.epara_step(None, None, 0, None) == E.E_INVALID
    assert E.lib.epara_collect(None, 1, None) == E.E_INVALID
    assert E.lib.epara_destroy(None) == E.E_INVALID


def test_decode_attention_refuses_an_output_between_two_bf16_elements(E):
    """(nothing is launched, so any aligned number stands in for a device pointer)"""
    for out, ok in ((4097, False), (4098, True)):
        args = (4096, 512, 4096, 8, 4096, 4096, 4, out)
        r = [E.lib.epara_decode_attention(0, None, *args, 0, 8, 2, 64, 64, 4096, 1 << 20), E.lib.epara_decode_attention_static(0, None, *args, 0, 8, 2, 64, 64)]
        assert r == [E.OK if ok else E.E_INVALID] * 2


@pytest.mark.parametrize("M,N,K,epi,ldc", [(129, 768, 3072, "RESID", 770), (509, 2048, 8192, "RESID", 2050), (300, 1000, 768, "BIAS", 1004),
                                           (512, 136, 4096, "BIAS", 140), (200, 4096, 1024, "SWIGLU", 2052), (64, 32000, 2048, "BIAS", 32002),
                                           (17, 2048, 8192, "RESID", 2050), (100, 16384, 2048, "SWIGLU", 8193)])
def test_grouped_gemm_refuses_an_ldc_its_vector_stores_cannot_take(E, M, N, K, epi, ldc):
    """A bad row stride of C is refused before anything is built or launched (aligned numbers stand in for pointers), whichever
    tensor-core kernel the sizes select, on its own and behind a good problem."""
    flag = {"RESID": E.EPI_RESID_F32, "BIAS": E.EPI_BIAS, "SWIGLU": E.EPI_SWIGLU}[epi]
    bad = E.GemmProblem(4096, 4096, 4096, 4096, M, N, K, K, K, ldc, flag)
    good = E.GemmProblem(4096, 4096, 4096, 4096, 300, 512, 512, 512, 512, 512, E.EPI_BIAS)
    for arr in ((E.GemmProblem * 1)(bad), (E.GemmProblem * 2)(good, bad)):
        assert E.lib.epara_grouped_gemm(0, None, E.GEMM_TCGEN05, arr, len(arr), 4096, 1 << 20) == E.E_INVALID


def test_eq4_eq5_match_oracle(E):
    from oracle import epara_oracle as O
    for req, grp in [(97, 49), (98, 49), (99, 49), (60, 60), (1, 100), (120.5, 30)]:
        assert E.epara_dp_group_count(req, grp) == O.dp_group_count(req, grp)
    for bs in [0, 1, 4, 7, 256, 512]:
        for mf in [1, 2, 3, 8, 300]:
            assert E.epara_inter_request_count(bs, mf) == O.inter_request_count(bs, mf)
    assert E.epara_inter_request_count(4, 0) == E.E_INVALID
    assert E.epara_dp_group_count(10, 0) == E.E_INVALID


def test_admission_matches_oracle_on_random_queues(E):
    from oracle import epara_oracle as O
    rng = np.random.default_rng(0)
    for trial in range(300):
        n = int(rng.integers(0, 40))
        now = int(rng.integers(0, 1000))
        q = [{"ticket": 100 + i, "deadline_ns": int(rng.choice([0, 0, rng.integers(1, 1000)])),
              "stream": int(rng.integers(0, 6))} for i in range(n)]
        cap = int(rng.integers(0, 20))
        mf = int(rng.choice([0, 0, 1, 2, 3, 5, 30]))
        exp = O.admit(q, now, cap, mf)
        got = E.epara_admit_queue([r["ticket"] for r in q], [r["deadline_ns"] for r in q],
                                  [r["stream"] for r in q], now, cap, mf)
        assert (list(exp[0]), list(exp[1])) == got, (trial, q, now, cap, mf)


def test_binding_refuses_to_import_without_the_library(E, tmp_path):
    """The product path has no fallback: a missing libepara.so is an ImportError."""
    code = ("import importlib.util, sys, os\n"
            "spec = importlib.util.spec_from_file_location('epara_copy', sys.argv[1])\n"
            "m = importlib.util.module_from_spec(spec)\n"
            "try:\n    spec.loader.exec_module(m)\nexcept ImportError as e:\n    print('IMPORTERROR'); sys.exit(0)\n"
            "sys.exit(1)\n")
    src = open(os.path.join(ROOT, "paper_2511_00603_b200", "epara.py")).read()
    p = tmp_path / "epara_copy.py"
    p.write_text(src)
    r = subprocess.run([sys.executable, "-c", code, str(p)], capture_output=True, text=True)
    assert r.returncode == 0 and "IMPORTERROR" in r.stdout


def test_product_path_does_not_import_the_oracle():
    pkg = os.path.join(ROOT, "paper_2511_00603_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                txt = open(os.path.join(dirpath, f)).read()
                assert not re.search(r"^\s*(from|import)\s+oracle|epara_oracle|oracle[/.]", txt, flags=re.M), f
    otxt = open(os.path.join(ROOT, "oracle", "epara_oracle.py")).read()
    assert "paper_2511_00603_b200" not in otxt and "ctypes" not in otxt


def test_collect_method_without_ctypes_takes_what_the_general_one_takes(E):
    """The binding's compiled epara_collect: positional, by keyword, ticket as a ctypes integer, wrong types; on a context without a
    handle every form answers INVALID.  (Where it can be built it is the one in use.)"""
    if os.path.exists(os.path.join(sysconfig.get_paths()["include"], "Python.h")) and shutil.which(os.environ.get("CXX", "g++")):
        assert not isinstance(E.Context.__dict__["epara_collect"], types.FunctionType)
    class NoContext(E.Context):
        def __init__(self):
            self.h, self._handle = E.C.c_void_p(), 0
    c = NoContext()
    for s, out in (c.epara_collect(7), c.epara_collect(ticket=7), c.epara_collect(E.C.c_uint64(7)), c.epara_collect(2**64 - 1), c.epara_collect(-1),
                   E.Context.epara_collect(c, 7)):
        assert s == E.E_INVALID and isinstance(out, E.Output)
    with pytest.raises(Exception):
        c.epara_collect("7")
    with pytest.raises(TypeError):
        c.epara_collect()


def test_collect_method_lets_other_threads_run(E):
    """The compiled method asks for an answer that is not there yet without the interpreter lock.  The C library's usleep stands in for
    epara_collect: it takes its microseconds where the context's address goes."""
    _fastcall = pytest.importorskip("paper_2511_00603_b200._fastcall")

    class Sleeper:
        _handle = 300_000
    usleep = ctypes.cast(ctypes.CDLL(None).usleep, ctypes.c_void_p).value
    not_there = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_uint64, ctypes.c_void_p)(lambda ctx, ticket, out: E.PENDING)
    Sleeper.collect = _fastcall.collect_method(usleep, ctypes.cast(not_there, ctypes.c_void_p).value, E.PENDING, E.Output, None, "_handle")
    inside = threading.Event()

    def call():
        inside.set()
        Sleeper().collect(1)
    t = threading.Thread(target=call)
    t.start()
    inside.wait()
    turns = 0
    while t.is_alive():
        time.sleep(0.002)
        turns += 1
    t.join()
    assert turns > 10


@pytest.mark.parametrize("cxx", ["/nowhere/c++", "false"])
def test_build_goes_on_without_the_compiled_collect_method(monkeypatch, tmp_path, capfd, cxx):
    """A compiler that is missing or fails leaves the extension out, one of an older source included, and the build goes on."""
    from paper_2511_00603_b200 import build
    old = tmp_path / os.path.basename(build.FAST_LIB)
    old.write_bytes(b"of an older source")
    monkeypatch.setattr(build, "FAST_LIB", str(old))
    monkeypatch.setattr(build, "_stale", lambda: False)
    os.utime(old, (0, 0))
    monkeypatch.setenv("CXX", cxx)
    assert build.build() == build.LIB
    assert not old.exists() and "ctypes" in capfd.readouterr().err


def test_collect_extension_is_named_for_this_interpreter(E, monkeypatch, tmp_path):
    """The extension is made for one interpreter's ABI: its file carries the tag, one without a tag is removed, nothing partial is left."""
    from paper_2511_00603_b200 import build
    _fastcall = pytest.importorskip("paper_2511_00603_b200._fastcall")
    suffix = sysconfig.get_config_var("EXT_SUFFIX")
    assert suffix != ".so" and os.path.basename(_fastcall.__file__) == "_fastcall" + suffix
    untagged, tagged = tmp_path / "_fastcall.so", tmp_path / os.path.basename(build.FAST_LIB)
    untagged.write_bytes(b"of some other interpreter")
    monkeypatch.setattr(build, "FAST_LIB", str(tagged))
    build.build_fastcall()
    assert os.listdir(tmp_path) == [tagged.name]


def test_bench_gives_dram_traffic_only_for_the_profiled_step():
    """The profile's figure belongs to a step of that many launches; other kernels, another number, no figure."""
    import bench
    n = bench.GEMM_TC_LAUNCHES_MIXED
    assert bench.gemm_traffic(False, n) == bench.GEMM_TC_TRAFFIC_MIXED / n
    assert bench.gemm_traffic(False, n - 14) is None and bench.gemm_traffic(True, n) is None


def test_collect_method_asks_once_for_an_answer_that_is_there(E):
    _fastcall = pytest.importorskip("paper_2511_00603_b200._fastcall")
    calls = []
    proto = ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_uint64, ctypes.c_void_p)
    fns = [proto(lambda ctx, ticket, out, k=k: calls.append((k, ctx, ticket)) or (E.PENDING if k == "ready" and ticket == 1 else E.E_TIMEOUT))
           for k in ("collect", "ready")]

    class Ctx:
        _handle = 4096
    Ctx.collect = _fastcall.collect_method(*(ctypes.cast(f, ctypes.c_void_p).value for f in fns), E.PENDING, E.Output, None, "_handle")
    assert Ctx().collect(2)[0] == E.E_TIMEOUT and calls == [("ready", 4096, 2)]
    assert Ctx().collect(1)[0] == E.E_TIMEOUT and calls[1:] == [("ready", 4096, 1), ("collect", 4096, 1)]
    assert E.lib.epara_collect_ready(None, 1, None) == E.E_INVALID
