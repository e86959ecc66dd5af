"""The C-ABI library loads and exports every entry point include/bmu.h declares,
and its host-side argument checks answer without touching a GPU."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2609_05138_b200 import build, binding
    build.build_library()
    return binding.load()


def declared_functions():
    text = open(os.path.join(ROOT, "include", "bmu.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"BMU_API\s+[\w\s\*]+?\b(bmu_\w+)\s*\(", text)))


def test_header_and_binding_agree(lib):
    from paper_2609_05138_b200 import binding
    names = declared_functions()
    assert len(names) >= 10
    assert sorted(binding.EXPORTS) == names
    for n in names:
        assert getattr(lib, n) is not None           # dlsym succeeds


def test_only_the_api_is_exported():
    import subprocess
    from paper_2609_05138_b200 import binding
    out = subprocess.check_output(["nm", "-D", "--defined-only", binding.LIB_PATH], text=True)
    syms = [l.split()[-1] for l in out.splitlines() if " T " in l]
    assert sorted(syms) == declared_functions()


def test_status_strings_and_version(lib):
    assert lib.bmu_status_string(0) == b"ok"
    assert b"workspace" in lib.bmu_status_string(3)
    assert lib.bmu_version() >= 100


def test_workspace_size_is_monotone(lib):
    f = lib.bmu_search_workspace_bytes
    a = f(4096, 1024, 10_000, 640_000, None)
    b = f(16384, 262144, 2_000_000, 160_000_000, None)
    assert 0 < a < b
    assert a % 256 == 0 and b >= 262144 * 4 + 2_000_000 * 8


def test_a_workspace_for_more_documents_serves_fewer(lib):
    """The size queries never fall when documents or listings are added: a workspace allocated once for the
    largest batch serves every smaller one, whichever kernel that takes."""
    import random
    from paper_2609_05138_b200 import Opts
    rng = random.Random(7)
    chunk, one, never = Opts(), Opts(), Opts()
    chunk.chunk_neurons = 512
    one.two_stage = 1
    never.two_stage = 2

    def log_int(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    def size(which, D, M, N, nnz, o):
        o = ctypes.byref(o) if o else None
        if which == "plan":
            return lib.bmu_plan_workspace_bytes(N, nnz, D, M, o)
        return getattr(lib, "bmu_search_%sworkspace_bytes" % which)(D, M, N, nnz, o)

    for trial in range(1500):
        which = rng.choice(["", "top2_", "f16_", "plan"])
        o = rng.choice([None, None, None, chunk, one, never])
        D = rng.choice([1, 300, 4096, 16384, log_int(100, 65000)])
        M = rng.choice([1024, 4096, 16384, 127 * 127, log_int(8, 300_000)])
        M = max(256, M // 256 * 256) if which == "f16_" else M
        N = log_int(1, 2_000_000)
        nnz = int(N * rng.choice([0.0, 1.0, 30.0, 80.0, 80.0, 80.0, 400.0, 2000.0]))
        need = size(which, D, M, N, nnz, o)
        for _ in range(6):
            n = rng.choice([N - 1, int(N * rng.uniform(0.9, 1.0)), int(N * rng.random()), rng.randint(0, min(N, 1500)), N])
            n = max(0, n)
            e = rng.choice([nnz, int(nnz * rng.random()), int(nnz * (n / N))])
            assert size(which, D, M, n, e, o) <= need, (which, D, M, (N, nnz), (n, e))


def test_the_two_stage_form_reserves_one_copy_of_the_ids(lib):
    """Its sweep walks 16-bit id lists by tile; the row lists of the other kernels are no part of it."""
    from paper_2609_05138_b200 import Opts
    o = Opts()
    o.two_stage = 1
    f = lambda nnz: lib.bmu_search_workspace_bytes(16384, 4096, 1_000_000, nnz, ctypes.byref(o))
    o.kernel = 6                                      # (kernel 0 makes room for the other kernels too)
    assert f(160_000_000) - f(80_000_000) <= 80_000_000 * 2 + 4096


def test_argument_checks_need_no_gpu(lib):
    # sizes are checked before any CUDA call is made
    assert lib.bmu_codebook_norms(None, -1, 4, None, None) == 1
    assert lib.bmu_search(None, 4, 1 << 30, None, None, 1, None, None, None) == 2
    assert b"limits" in lib.bmu_last_error()
    assert lib.bmu_search_ws(None, 4, 4, None, None, None, 0, 0, None, None, None, None, 0,
                             None) == 0           # N == 0: nothing to do
    assert lib.bmu_search_ws(None, 4, 4, None, None, None, 3, 0, None, None, None, None, 0,
                             None) == 1           # null pointers
    from paper_2609_05138_b200 import Opts
    o = Opts()
    o.vec = 3
    assert lib.bmu_search_ws(None, 4, 4, None, None, None, 3, 0, None, None,
                             ctypes.byref(o), None, 0, None) == 1


def test_an_empty_map_is_refused_before_any_launch(lib):
    """Documents have no unit on a map without units: refused like a search against an empty codebook."""
    p = ctypes.c_void_p(256)                          # never looked at
    assert lib.bmu_update_scatter(p, p, 5, 10, p, 16, 0, p, p, None) == 1
    assert b"empty map" in lib.bmu_last_error()
    assert lib.bmu_update_scatter(p, p, 0, 0, p, 16, 0, p, p, None) == 0       # no documents: nothing to do


def test_describe_search_needs_no_gpu_and_names_the_kernel(lib):
    """bmu_describe_search is host logic: the benchmark shapes route as documented (large
    sweeps take the tensor-core sweep, the small one the planned kernel) and the launch count
    follows from the chunk."""
    from paper_2609_05138_b200 import Opts, SearchDesc
    d = SearchDesc()
    shapes = {"cfg1": (4096, 1024, 10_000, 640_000), "cfg2": (16384, 4096, 1_000_000, 80_000_000),
              "cfg4": (16384, 262144, 2_000_000, 160_000_000)}
    for name, (D, M, N, nnz) in shapes.items():
        assert lib.bmu_describe_search(D, M, N, nnz, None, ctypes.byref(d)) == 0
        assert d.kernel == (3 if name == "cfg1" else 6)
        assert d.head_rows == (0 if name == "cfg1" else 640)
        assert d.docs_per_block == (16 if name == "cfg1" else 128)
        assert d.chunk_neurons % d.slab == 0 and d.ragged_neurons == 0
        assert d.sweep_launches == -(-M // d.chunk_neurons)
    o = Opts()
    o.kernel, o.chunk_neurons = 6, 2048
    assert lib.bmu_describe_search(16384, 262144 + 36, 1000, 80_000, ctypes.byref(o), ctypes.byref(d)) == 0
    assert (d.kernel, d.chunk_neurons, d.sweep_launches, d.ragged_neurons, d.repack) == (6, 2048, 128, 36, 1)
    o.kernel = 6
    assert lib.bmu_describe_search(32, 1024, 10, 100, ctypes.byref(o), ctypes.byref(d)) == 2   # D < head
    assert lib.bmu_describe_search(32, 1024, 10, 100, None, None) == 1


@pytest.mark.parametrize("D,M,N,length,two_stage", [
    (4096, 1024, 48, 64, 0), (16384, 16384, 256, 79, 0), (16384, 65536, 1000, 80, 0), (4096, 1024, 1000, 80, 0),
    (4096, 127 * 127, 1000, 400, 1), (4096, 127 * 127, 1000, 80, 1), (16384, 65536, 1000, 400, 1),
    (16384, 262144, 1000, 400, 1)])
def test_few_documents_take_the_faster_way(lib, D, M, N, length, two_stage):
    """The few-documents kernel where it is faster, not wherever the documents are few: long lists and large
    maps are screened (or, with that ruled out, swept on the tensor cores)."""
    from paper_2609_05138_b200 import Opts, SearchDesc
    d, o = SearchDesc(), Opts()
    assert lib.bmu_describe_search(D, M, N, N * length, None, ctypes.byref(d)) == 0
    assert (d.kernel, d.two_stage > 0) == ((6, True) if two_stage else (1, False))
    o.two_stage = 2
    assert lib.bmu_describe_search(D, M, N, N * length, ctypes.byref(o), ctypes.byref(d)) == 0
    large = N * length * M >= 2e10 and M % 4 == 0
    assert (d.kernel, d.two_stage) == ((6 if large else 1), 0)


def test_status_words_map_to_errors_without_a_gpu(lib):
    """The host entry points that read a search's status word back (bmu_search_host,
    bmu_search_batches_host, bmu_plan_create, bmu_last_status) turn it into an error through
    this mapping: a clean word is no error, a failed size check of the tiling pass is a
    workspace error, a wait that ran out a timeout."""
    assert lib.bmu_status_of_word(0) == 0
    assert lib.bmu_status_of_word(64) == 3 and b"tiling pass" in lib.bmu_last_error()
    assert lib.bmu_status_of_word(64 | 8) == 3
    for word in (1, 2, 4, 8, 16, 32):
        assert lib.bmu_status_of_word(word) == 5
        assert b"wait ran out" in lib.bmu_last_error() and str(word).encode() in lib.bmu_last_error()
    assert lib.bmu_status_of_word(128) == 5
