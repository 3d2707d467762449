"""CPU-only: the C-ABI library builds, loads and exports every symbol the header declares."""
import ctypes
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "gptq2d.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(gptq2d_[a-z0-9_]+)\s*\(", text)))


def test_library_builds_and_exports_header_symbols():
    from paper_2607_27042_b200 import build
    lib_path = build.build()
    lib = ctypes.CDLL(lib_path)
    syms = _declared_symbols()
    assert "gptq2d_round" in syms and "gptq2d_factor" in syms and "gptq2d_objective" in syms
    for s in syms:
        assert hasattr(lib, s), s
    from paper_2607_27042_b200 import gptq2d
    assert sorted(gptq2d.EXPORTS) == [s for s in syms]
    for s in syms:
        if s != "gptq2d_status_string":
            assert callable(getattr(gptq2d, s)), "binding lacks " + s


def test_workspace_queries_and_status_strings_need_no_gpu():
    from paper_2607_27042_b200 import gptq2d
    assert gptq2d.status_string(0) == "ok"
    assert "positive definite" in gptq2d.status_string(5)
    assert gptq2d.gptq2d_round_workspace_bytes(0, 5) == 0
    w = gptq2d.gptq2d_round_workspace_bytes(8192, 8192)
    assert 2 * 8192 * 8192 * 8 <= w < 2 * 8192 * 8192 * 8 + (1 << 20)
    assert gptq2d.gptq2d_round_workspace_bytes(100, 130) >= 2 * 128 * 256 * 8
    assert gptq2d.gptq2d_round_host_workspace_bytes(64, 64) > gptq2d.gptq2d_round_workspace_bytes(64, 64)
    assert gptq2d.gptq2d_factor_workspace_bytes(64, 256) >= 3 * 256 * 256 * 8
    assert gptq2d.gptq2d_objective_workspace_bytes(64, 256) >= 2 * 64 * 256 * 8


def test_product_package_does_not_import_the_oracle():
    pkg = os.path.join(ROOT, "paper_2607_27042_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                src = open(os.path.join(dirpath, f)).read()
                assert "import oracle" not in src and "from oracle" not in src, f


def test_batched_entry_argument_checks_need_no_gpu():
    """Host-side validation of the batched call: made-up (never dereferenced) device addresses."""
    import ctypes as c
    from paper_2607_27042_b200 import gptq2d as g
    lib = g._lib

    def probs(shapes):
        arr = (g.Problem * len(shapes))()
        for b, (m, n) in enumerate(shapes):
            arr[b] = g.Problem(m, n, 0x1000, n, 0x2000, m, 0x3000, n, 0x4000, n, None, 0)
        return arr

    shapes = [(64, 64), (200, 330), (1, 9)]
    arr = probs(shapes)
    total = lib.gptq2d_round_batched_workspace_bytes(3, c.cast(arr, c.c_void_p))
    # at least the padded E and C buffers of every matrix; no more than that plus bookkeeping
    bufs = sum(2 * 8 * (-(-m // 128) * 128) * (-(-n // 128) * 128) for m, n in shapes)
    assert bufs <= total < bufs + (1 << 16)
    one = [lib.gptq2d_round_batched_workspace_bytes(1, c.cast(probs([s]), c.c_void_p)) for s in shapes]
    assert total <= sum(one)
    assert lib.gptq2d_round_batched_workspace_bytes(0, c.cast(arr, c.c_void_p)) == 0
    # invalid descriptors are rejected before any CUDA call
    ws = c.c_void_p(0x100000)
    assert lib.gptq2d_round_batched(0, c.cast(arr, c.c_void_p), None, ws, 1 << 40, None, None) == 1
    assert lib.gptq2d_round_batched(3, None, None, ws, 1 << 40, None, None) == 1
    bad = probs(shapes)
    bad[1].ldx = 100                                   # leading dimension below n
    assert lib.gptq2d_round_batched(3, c.cast(bad, c.c_void_p), None, ws, 1 << 40, None, None) == 1
    bad = probs(shapes)
    bad[2].Z = None
    assert lib.gptq2d_round_batched(3, c.cast(bad, c.c_void_p), None, ws, 1 << 40, None, None) == 1
    big = probs([(g.BATCH_MAX_DIM + 1, 8)])
    assert lib.gptq2d_round_batched(1, c.cast(big, c.c_void_p), None, ws, 1 << 40, None, None) == 9
    many = probs([(8, 8)] * (g.BATCH_MAX_COUNT + 1))
    assert lib.gptq2d_round_batched(len(many), c.cast(many, c.c_void_p), None, ws, 1 << 40, None, None) == 9
    # workspace too small / missing
    assert lib.gptq2d_round_batched(3, c.cast(arr, c.c_void_p), None, ws, total - 1, None, None) == 2
    assert lib.gptq2d_round_batched(3, c.cast(arr, c.c_void_p), None, None, total, None, None) == 2


def test_batched_setup_argument_checks_need_no_gpu():
    """Host-side validation of gptq2d_factor_batched: made-up (never dereferenced) device addresses."""
    import ctypes as c
    from paper_2607_27042_b200 import gptq2d as g
    lib = g._lib

    def probs(shapes, a=0x1000):
        arr = (g.FactorProblem * len(shapes))()
        for b, (m, n) in enumerate(shapes):
            arr[b] = g.FactorProblem(m, n, a, m, 0x2000, n, 0x3000, m, 0x4000, n, None, None)
        return arr

    small = probs([(64, 64), (1, 128), (100, 7)])
    table = lib.gptq2d_factor_batched_workspace_bytes(3, c.cast(small, c.c_void_p))
    assert 0 < table <= 4096                                    # descriptors only: no blocked route needed
    mixed = probs([(64, 64), (300, 90)])
    total = lib.gptq2d_factor_batched_workspace_bytes(2, c.cast(mixed, c.c_void_p))
    assert total >= g.gptq2d_factor_workspace_bytes(300, 90)    # the blocked route's own workspace on top
    assert lib.gptq2d_factor_batched_workspace_bytes(0, c.cast(small, c.c_void_p)) == 0
    assert lib.gptq2d_factor_batched(0, c.cast(small, c.c_void_p), None, 0, None, None) == 1      # INVALID_ARG
    bad = probs([(64, 64)])
    bad[0].ldl = 10                                             # leading dimension below m
    assert lib.gptq2d_factor_batched(1, c.cast(bad, c.c_void_p), None, 0, None, None) == 1
    assert lib.gptq2d_factor_batched(3, c.cast(small, c.c_void_p), None, 0, None, None) == 2      # WORKSPACE


def test_long_matrices_are_not_swept_in_blocks():
    """A block's tile indices have 8 bits (32 768 rows or columns); a matrix with a longer block is swept whole.  The workspace
    query shows which: the bookkeeping of a sweep in blocks comes on top of that of the whole sweep."""
    from paper_2607_27042_b200 import gptq2d as g

    def in_blocks(m, n):
        got = g.gptq2d_round_workspace_bytes(m, n)
        g.gptq2d_internal_test_hook(7, 1 << 30)
        try:
            return got > g.gptq2d_round_workspace_bytes(m, n)
        finally:
            g.gptq2d_internal_test_hook(7, 0)

    assert in_blocks(5632, 5632) and not in_blocks(5631, 70000)
    for m, n in ((5632, 65536), (65536, 5632), (65409, 65409)):
        assert in_blocks(m, n), (m, n)
    for m, n in ((5632, 65537), (65537, 5632), (5632, 65664), (65664, 65664), (6000, 130000)):
        assert not in_blocks(m, n), (m, n)


def test_blocks_begin_at_32_rows_and_columns_of_tiles():
    from paper_2607_27042_b200 import gptq2d as g

    def extra(m, n):
        got = g.gptq2d_round_workspace_bytes(m, n)
        g.gptq2d_internal_test_hook(7, 1 << 30)
        try:
            return got - g.gptq2d_round_workspace_bytes(m, n)
        finally:
            g.gptq2d_internal_test_hook(7, 0)

    for m, n in ((3969, 3969), (3969, 65536), (65536, 3969), (4096, 4096)):
        assert extra(m, n) > 0, (m, n)
    for m, n in ((3968, 3968), (3968, 3969), (3968, 65536), (65536, 3968)):
        assert extra(m, n) == 0, (m, n)


def test_long_matrices_are_swept_in_blocks_whatever_k_has_to_be_cut_into():
    """Whether a resident sweep runs in blocks, and in how many products: at least four, and as few more as their planes need."""
    from paper_2607_27042_b200 import gptq2d as g

    def products(m, n, less=0):
        return g.gptq2d_internal_round_products(m, n, g.gptq2d_round_workspace_bytes(m, n) - less)

    assert products(4096, 4096) == 4 and products(8192, 8192) == 8                 # 134 MB of planes; 537 MB in 268 MB of free rows
    assert products(3968, 3968) == 0 and products(5632, 65537) == 0
    # planes of (2048 + k / 2) x k / 2 entries, 16 bytes each, in free rows of 2048 x k values of 8 bytes: two pieces of 2048 rows and one for
    # every 2048 k / (4096 + k) of the longer side
    for n in (16384, 30000, 48000, 58000, 65536):
        half = -(-n // 256) * 128
        want = 2 * 2 + 2 * -(-16 * (2048 + half) * half // (2048 * 2 * half * 8))
        for m, k in ((4000, n), (n, 4000)):
            assert want <= products(m, k) <= want + 2, (m, k, products(m, k), want)
    assert products(65409, 65409) >= 8


def test_blocks_need_little_more_room_than_the_whole_sweep():
    """The planes' own room only serves speed: with the bookkeeping alone they lie in rows of the workspace that are free at the time."""
    from paper_2607_27042_b200 import gptq2d as g

    for m, n in ((3969, 3969), (4096, 4096), (4609, 4700), (5003, 4100), (8192, 8192), (4000, 65536)):
        g.gptq2d_internal_test_hook(7, 1 << 30)
        whole = g.gptq2d_round_workspace_bytes(m, n)
        g.gptq2d_internal_test_hook(7, 0)
        full = g.gptq2d_round_workspace_bytes(m, n)
        lo, hi = whole, full
        while hi - lo > 1:
            mid = (lo + hi) // 2
            lo, hi = (lo, mid) if g.gptq2d_internal_round_products(m, n, mid) else (mid, hi)
        # four counters a tile, two a cell of 32 x 32 a byte each, a table of far parts, three rings; below 37 tiles a scale, a top and the bits of
        # half of the rows and columns
        tiles = -(-m // 128) * -(-n // 128)
        most = 60 * tiles + (1 << 17) + (16 * (m + n) if min(m, n) < 4609 else 0)
        assert g.gptq2d_internal_round_products(m, n, whole) == 0 and hi - whole <= most, (m, n, hi - whole)
        assert g.gptq2d_internal_round_products(m, n, hi) >= g.gptq2d_internal_round_products(m, n, full) >= 4
