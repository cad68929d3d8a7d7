"""The C-ABI library builds for sm_103a, loads, and exports every function that
include/*.h declares (no compute calls: this runs without a GPU)."""
import ctypes
import glob
import os
import re

import paper_2608_03199_gb300 as sieve

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    names = set()
    for h in glob.glob(os.path.join(ROOT, "include", "*.h")):
        text = open(h).read()
        text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
        for m in re.finditer(r"^[A-Za-z_][\w \*]*?\b(sieve_\w+)\s*\(", text, flags=re.M):
            names.add(m.group(1))
    return names


def test_header_declares_the_boundary():
    names = declared_functions()
    for required in ("sieve_rank_partitions", "sieve_search", "sieve_search_host",
                     "sieve_build_layout", "sieve_search_workspace_size", "sieve_status_str"):
        assert required in names


def test_library_exports_every_declared_symbol():
    path = sieve.build()
    lib = ctypes.CDLL(path)
    missing = [n for n in declared_functions() if not hasattr(lib, n)]
    assert not missing, missing
    assert set(declared_functions()) <= set(sieve._SIGNATURES), "binding lacks a declared call"


def test_host_only_calls_without_gpu():
    lib = sieve.lib()
    assert lib.sieve_version().startswith(b"libsieve")
    assert lib.sieve_status_str(-1) == b"invalid argument"
    n = ctypes.c_size_t()
    assert lib.sieve_layout_workspace_size(1000, 16, ctypes.byref(n)) == 0 and n.value > 0
    assert lib.sieve_layout_workspace_size(-1, 16, ctypes.byref(n)) == -1
    v = sieve.IndexViewC(n=1000, nlist=16, d=64, vectors=16, ids=16, list_offsets=16, centroids=16)
    p = sieve._params(0.9, 10, 8, 4, True, 0, 0)
    assert lib.sieve_search_workspace_size(ctypes.byref(v), 100, ctypes.byref(p), 0,
                                           ctypes.byref(n)) == 0
    small = n.value
    assert lib.sieve_search_workspace_size(ctypes.byref(v), 100, ctypes.byref(p), 1,
                                           ctypes.byref(n)) == 0 and n.value > small
    for bad in (sieve._params(0.9, 0, 8, 4, True, 0, 0), sieve._params(0.9, 65, 8, 4, True, 0, 0),
                sieve._params(0.9, 10, 17, 4, True, 0, 0), sieve._params(0.9, 10, 8, 0, True, 0, 0),
                sieve._params(float("nan"), 10, 8, 4, True, 0, 0)):
        assert lib.sieve_search_workspace_size(ctypes.byref(v), 100, ctypes.byref(bad), 0,
                                               ctypes.byref(n)) == -1
    v.d = 62
    assert lib.sieve_search_workspace_size(ctypes.byref(v), 100, ctypes.byref(p), 0,
                                           ctypes.byref(n)) == -1
    # the status query rejects a missing or misaligned workspace before any copy
    st = ctypes.c_int32(5)
    assert lib.sieve_search_status(None, 1 << 20, ctypes.byref(st), None) == -1
    assert lib.sieve_search_status(ctypes.c_void_p(16), 1 << 20, ctypes.byref(st), None) == -1
    assert lib.sieve_search_status(ctypes.c_void_p(256), 1 << 20, None, None) == -1
    assert st.value == 5


def test_scan_path_values_without_gpu():
    """scan_path 0..3 (automatic, FP32 FMA, three fp16 products, the screen)
    are accepted; anything else is SIEVE_EINVAL before any device work."""
    lib = sieve.lib()
    n = ctypes.c_size_t()
    v = sieve.IndexViewC(n=1000, nlist=16, d=64, vectors=16, ids=16, list_offsets=16, centroids=16)
    for path in ("auto", "simt", "tensor", "screen", 0, 1, 2, 3):
        p = sieve._params(0.9, 10, 8, 4, True, 0, 0, scan_path=path)
        assert lib.sieve_search_workspace_size(ctypes.byref(v), 100, ctypes.byref(p), 0,
                                               ctypes.byref(n)) == 0
    for serial in (0, 1):
        p = sieve._params(0.9, 10, 8, 4, True, 0, 0, serial=serial)
        assert lib.sieve_search_workspace_size(ctypes.byref(v), 100, ctypes.byref(p), 0,
                                               ctypes.byref(n)) == 0
    p = sieve._params(0.9, 10, 8, 4, True, 0, 0)
    p.serial = 2
    assert lib.sieve_search_workspace_size(ctypes.byref(v), 100, ctypes.byref(p), 0,
                                           ctypes.byref(n)) == -1
    p.serial, p.wait_limit = 0, -1
    assert lib.sieve_search_workspace_size(ctypes.byref(v), 100, ctypes.byref(p), 0,
                                           ctypes.byref(n)) == -1
    for path in (-1, 4):
        p = sieve._params(0.9, 10, 8, 4, True, 0, 0, scan_path=path)
        assert lib.sieve_search_workspace_size(ctypes.byref(v), 100, ctypes.byref(p), 0,
                                               ctypes.byref(n)) == -1


def test_screen_scores_rejects_bad_arguments_without_gpu():
    """sieve_screen_scores checks its arguments on the host before any device
    work: it needs the centroids' tensor layout and d <= 256, and its output
    rows must hold every centroid at a 32-float stride (SIEVE_EINVAL)."""
    lib = sieve.lib()
    ok = dict(n=1000, nlist=100, d=64, vectors=16, ids=16, list_offsets=16, centroids=16,
              tc_centroids=16)
    q, out = ctypes.c_void_p(256), ctypes.c_void_p(512)
    v = sieve.IndexViewC(**{**ok, "tc_centroids": None})
    assert lib.sieve_screen_scores(ctypes.byref(v), q, 10, out, 128, None) == -1   # no layout
    v = sieve.IndexViewC(**{**ok, "d": 260})
    assert lib.sieve_screen_scores(ctypes.byref(v), q, 10, out, 128, None) == -1   # d > 256
    v = sieve.IndexViewC(**ok)
    assert lib.sieve_screen_scores(ctypes.byref(v), q, 10, out, 96, None) == -1    # ld < nlist
    assert lib.sieve_screen_scores(ctypes.byref(v), q, 10, out, 112, None) == -1   # ld % 32
    assert lib.sieve_screen_scores(ctypes.byref(v), q, -1, out, 128, None) == -1   # nq < 0
    assert lib.sieve_screen_scores(ctypes.byref(v), ctypes.c_void_p(260), 10, out, 128, None) == -1
    assert lib.sieve_screen_scores(ctypes.byref(v), q, 10, None, 128, None) == -1


def test_workspace_has_prefix_lists_only_where_a_search_uses_them_without_gpu():
    """A search's workspace is that of the FP32 path plus the full ranking's
    scratch, unless the call ranks a prefix of each order (a layout of the
    centroids, a window of up to 24, and 2,048 centroids or 4,096 queries)."""
    lib = sieve.lib()

    def size(nlist, d, nq, nprobe, W, path="auto", layout=True):
        v = sieve.IndexViewC(n=1000, nlist=nlist, d=d, vectors=16, ids=16, list_offsets=16, centroids=16)
        if layout:
            v.tc_rows = v.tc_row_blocks = v.tc_centroids = 256
        p = sieve._params(0.9, 10, nprobe, W, True, 0, 0, 0, path)
        total, rank = ctypes.c_size_t(), ctypes.c_size_t()
        assert lib.sieve_search_workspace_size(ctypes.byref(v), nq, ctypes.byref(p), 0, ctypes.byref(total)) == 0
        assert lib.sieve_rank_workspace_size(ctypes.byref(v), nq, nprobe, ctypes.byref(rank)) == 0
        return total.value, rank.value

    for nlist, d, nq, nprobe, W, layout in ((1024, 256, 2_000, 64, 8, True), (149, 100, 4_000, 24, 4, True),
                                            (1024, 256, 20_000, 64, 64, True), (8192, 96, 20_000, 128, 8, False),
                                            (8192, 516, 200, 128, 8, False)):
        total, rank = size(nlist, d, nq, nprobe, W, layout=layout)
        assert total <= size(nlist, d, nq, nprobe, W, "simt", layout)[0] + rank + 512, (nlist, d, nq, nprobe, W)
    # where it is used, the lists and the extension's buffers come on top
    total, rank = size(8192, 96, 2_000, 128, 8)
    assert total > size(8192, 96, 2_000, 128, 8, "simt")[0] + rank + 512
