"""The planner's choice of work lists (costa_debug_dispatch), on the CPU: for
each line of the rule the kinds that run on patches on both of its sides, and
that every kind has a list that covers it."""
import os
import subprocess
import sys

import numpy as np
import pytest

from workloads import layouts as L

costa = pytest.importorskip("paper_2106_06601_gb300")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FAKE = 1 << 40
ES = {"f32": 4, "f64": 8, "c64": 8, "c128": 16}
REAL = {"copy", "scale", "axpby", "axpby2"}
OF = {"f32": REAL, "f64": REAL, "c64": REAL | {"cplx", "cscale"}, "c128": REAL | {"cplx", "cscale", "cplxr"}}


def _layout(spec, dtype):
    ptrs = FAKE + spec.buf.astype(np.int64) * (1 << 34) + spec.off * ES[dtype]
    return costa.costa_layout_from_spec(spec, dtype, ptrs)


def _pair(dtype, op, mb, ma, m, n, pads=(0, 0), grid=2):
    B = L.block_cyclic(*((m, n) if op == "N" else (n, m)), mb, mb, grid, grid, ld_pad=pads[0], name="B")
    A = L.block_cyclic(m, n, ma, ma, grid, grid, grid_order="C", ld_pad=pads[1], name="A")
    return A, B


def dispatch(dtype, *problems, host=-1):
    """costa_debug_dispatch of (A, B, op) specs, the kinds those of the type."""
    As, Bs = [_layout(A, dtype) for A, _, _ in problems], [_layout(B, dtype) for _, B, _ in problems]
    try:
        d = costa.costa_debug_dispatch(As, Bs, [op for _, _, op in problems], host)
    finally:
        for x in As + Bs:
            x.destroy()
    for key in ("patch_kinds", "tma_kinds", "tma_halves_kinds"):
        d[key] &= OF[dtype]
    # every kind has a list: patches, or tiles that are not only other problems'
    assert d["patches"] > 0 if d["patch_kinds"] else d["patches"] == 0
    tiles = d["tiles"] + d["misaligned"] + d["pieces"]
    assert tiles > 0 or d["patch_kinds"] == OF[dtype] or all(A.numel() == 0 for A, _, _ in problems)
    if not d["tiles_are_rest"]:
        assert d["patch_kinds"] and tiles > 0
        # no TMA lists for kinds that do not run on these tiles
        assert not (d["tma_kinds"] | d["tma_halves_kinds"]) & d["patch_kinds"]
    return d


def kinds(dtype, op, mb, ma, m, n=None, pads=(0, 0), grid=2, host=-1):
    A, B = _pair(dtype, op, mb, ma, m, n or m, pads, grid)
    return dispatch(dtype, (A, B, op), host=host)["patch_kinds"]


ALL, NONE = REAL, set()


@pytest.mark.parametrize("dtype, op, mb, ma, m, n, pads, want", [
    # small, partial or misaligned tiles, whatever the size
    ("f64", "T", 50, 75, 150, 171, (0, 0), ALL),
    ("f64", "T", 24, 100, 1200, 1200, (0, 0), ALL),
    ("f32", "T", 24, 100, 1200, 1200, (0, 0), NONE),  # 4-byte partial tiles stay
    ("f64", "T", 64, 128, 2048, 2048, (1, 0), ALL),
    ("f32", "T", 64, 128, 2048, 2048, (0, 1), ALL),
    ("f32", "T", 64, 128, 2048, 2048, (1, 0), NONE),  # only the source misaligned: windows
    ("f64", "T", 64, 64, 7001, 6003, (0, 0), ALL),    # a twentieth misaligned
    # in large lists, tiles along A's runs from 16 x 16 on are not poor
    ("f64", "N", 24, 24, 1200, 1200, (0, 0), ALL),
    ("f64", "N", 24, 24, 3072, 3072, (0, 0), NONE),
    # power-of-two cells of doubles keep the kinds that read A on tiles in lists of middle size
    ("f64", "T", 8, 8, 1544, 1544, (0, 0), ALL),
    ("f64", "T", 8, 8, 1552, 1552, (0, 0), {"copy", "scale"}),
    ("f64", "T", 8, 8, 4464, 4464, (0, 0), {"copy", "scale"}),
    ("f64", "T", 8, 8, 4480, 4480, (0, 0), {"copy", "scale", "axpby2"}),
    ("f64", "T", 8, 8, 7064, 7064, (0, 0), {"copy", "scale", "axpby2"}),
    ("f64", "T", 8, 8, 7072, 7072, (0, 0), ALL),
    ("c64", "T", 8, 8, 2048, 2048, (0, 0), OF["c64"]),
    # ... a lower line where lines of B are shared
    ("f64", "N", 64, 8, 2816, 2816, (0, 0), {"copy", "scale"}),
    ("f64", "N", 64, 8, 2832, 2832, (0, 0), ALL),
    # ... and alpha b with blocks of different sizes
    ("f64", "T", 8, 64, 3136, 3136, (0, 0), {"copy", "scale"}),
    ("f64", "T", 8, 64, 3200, 3200, (0, 0), {"copy"}),
    ("f64", "T", 64, 8, 4416, 4416, (0, 0), {"copy"}),
    ("f64", "T", 64, 8, 4480, 4480, (0, 0), {"copy", "scale", "axpby2"}),
    # 8-byte copies of partial tiles stay up to 1.75 times the L2
    ("f64", "T", 48, 48, 2832, 2832, (0, 0), {"scale"}),
    ("f64", "T", 48, 48, 3840, 3840, (0, 0), {"copy", "scale"}),
    # f32 cells of 16 x 16 and more, block ratio no power of two
    ("f32", "T", 16, 48, 8064, 8064, (0, 0), {"axpby", "axpby2"}),
    ("f32", "T", 48, 16, 8064, 8064, (0, 0), NONE),
    ("f32", "T", 16, 32, 8064, 8064, (0, 0), ALL),
])
def test_lists_of_poor_tiles(dtype, op, mb, ma, m, n, pads, want):
    assert kinds(dtype, op, mb, ma, m, n, pads) == want


@pytest.mark.parametrize("dtype, op, mb, ma, m, want", [
    ("f64", "T", 64, 128, 3712, NONE),  # 1.75 times the L2
    ("f64", "T", 64, 128, 3840, {"copy", "axpby2"}),
    ("f64", "N", 64, 128, 3840, {"copy", "axpby2"}),
    ("c64", "T", 64, 128, 3840, OF["c64"]),
    ("c128", "T", 64, 128, 6016, NONE),
    ("f32", "T", 64, 128, 5632, NONE),  # twice the L2
    ("f32", "T", 64, 128, 5760, {"copy", "scale"}),
    ("f32", "N", 64, 128, 5760, NONE),
    ("f32", "T", 64, 128, 6848, {"copy", "scale"}),
    ("f32", "N", 64, 128, 6848, NONE),
    ("f32", "T", 64, 128, 6912, ALL),
    ("f32", "N", 64, 128, 6912, ALL),
    ("f64", "T", 40, 40, 8000, {"copy", "axpby", "axpby2"}),  # TMA could stage too few tiles
    ("f32", "T", 24, 100, 8000, NONE),  # ragged cells
    ("f32", "T", 48, 96, 8064, {"axpby", "axpby2"}),  # cells meet inside most patches
    ("f32", "N", 48, 96, 8064, ALL),
    ("f32", "T", 96, 48, 6144, NONE),  # ... A's blocks the smaller ones
    ("f32", "T", 96, 48, 7104, {"axpby", "axpby2"}),
    ("f32", "T", 96, 96, 6144, ALL),  # whole tiles, but blocks of no power of two
    ("f32", "T", 64, 128, 6148, {"copy", "scale"}),
    ("f32", "T", 64, 128, 6145, ALL),  # ragged
    ("f32", "N", 64, 128, 6145, ALL),
])
def test_lists_of_full_tiles(dtype, op, mb, ma, m, want):
    assert kinds(dtype, op, mb, ma, m) == want


@pytest.mark.parametrize("mb, ma, off, want", [(16, 32, 4, ALL), (16, 32, 0, ALL), (16, 48, 16, {"axpby", "axpby2"}),
                                               (16, 48, 32, {"axpby", "axpby2"})])
def test_block_sizes_of_submatrices(mb, ma, off, want):
    """A submatrix starts with a part of a block: the rule compares the block
    sizes, not these parts (12 against 28 for BC16 -> BC32 from element 4 on, 16
    against 32 or 16 for BC16 -> BC48 from 16 or 32 on)."""
    n = 8064
    full = off + n
    lld = [f[2] for f in L.scalapack_full(full, full, ma, ma, 0, 0, 2, 2, "C", ld_pad=0)]
    A = L.scalapack_sub(full, full, ma, ma, 0, 0, 2, 2, "C", off + 1, off + 1, n, n, [v + -v % 4 for v in lld])
    lld = [f[2] for f in L.scalapack_full(full, full, mb, mb, 0, 0, 2, 2, "R", ld_pad=0)]
    B = L.scalapack_sub(full, full, mb, mb, 0, 0, 2, 2, "R", off + 1, off + 1, n, n, [v + -v % 4 for v in lld])
    assert dispatch("f32", (A, B, "T"))["patch_kinds"] == want


def test_tma_lists_only_for_kinds_on_tiles():
    """The general beta of doubles is staged by TMA where it runs on tiles, and
    has no TMA lists to build on its first call where it runs on patches."""
    for mb, m, want in ((64, 3840, {"axpby"}), (40, 8000, set())):
        A, B = _pair("f64", "T", mb, 2 * mb if mb == 64 else mb, m, m)
        d = dispatch("f64", (A, B, "T"))
        assert not d["tiles_are_rest"] and d["tma_kinds"] == want and not d["tma_halves_kinds"]


def test_tma_for_every_kind_keeps_patches_off():
    """COSTA_TMA=1 (read once per process) stages every kind's tiles by TMA, so
    nothing runs on patches."""
    script = """
from tests.test_dispatch import REAL, _pair, dispatch
for args in (("f64", "T", 40, 40, 600, 640), ("f64", "T", 24, 100, 1200, 1200), ("f64", "T", 64, 128, 3840, 3840),
             ("c128", "N", 8, 8, 300, 300), ("f32", "T", 50, 75, 300, 300)):
    A, B = _pair(*args)
    d = dispatch(args[0], (A, B, args[1]))
    assert not d["patch_kinds"], args
    assert not d["tiles"] or d["tma_kinds"] >= REAL, args
"""
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, env=dict(os.environ, COSTA_TMA="1"),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]


@pytest.mark.parametrize("op, m, n, grid, want", [
    ("T", 8192, 8192, 1, {"axpby", "axpby2"}), ("N", 8192, 8192, 1, ALL), ("T", 8192, 8192, 2, ALL),
    ("T", 16384, 16384, 2, {"axpby", "axpby2"}), ("N", 16384, 16384, 2, ALL), ("T", 8192, 8064, 1, ALL)])
def test_f32_columns_a_multiple_of_32_kb_apart(op, m, n, grid, want):
    """Only transposed copies stay on tiles for it (the leading dimension of a
    rank's source is its rows: n / grid transposed, m / grid otherwise)."""
    assert kinds("f32", op, 64, 128, m, n, (0, 0), grid) == want


def test_f32_columns_32_kb_apart_count_by_their_share():
    """One problem of a batch, or an empty first block, does not decide for the
    whole list."""
    wide, plain = _pair("f32", "T", 64, 128, 8192, 8192, grid=1), _pair("f32", "T", 64, 128, 8192, 8064, grid=1)
    assert dispatch("f32", (*wide, "T"), (*plain, "T"), (*plain, "T"))["patch_kinds"] == ALL
    assert dispatch("f32", (*plain, "T"), (*wide, "T"), (*wide, "T"))["patch_kinds"] == {"axpby", "axpby2"}
    A = L.packed_blocks(np.arange(0, 8193, 128), np.arange(0, 8193, 128), np.zeros((64, 64)), 1)
    B = L.packed_blocks([0, 0, 8192], [0, 8192], np.zeros((2, 1)), 1)  # ld 1 of the empty block
    assert dispatch("f32", (A, B, "T"))["patch_kinds"] == {"axpby", "axpby2"}


@pytest.mark.parametrize("dtype, op, mb, ma, m, pads, device, a_host, b_host, both", [
    ("c128", "T", 8, 8, 600, (0, 0), True, True, False, False),
    ("c128", "N", 50, 75, 600, (0, 0), True, False, False, False),
    ("f32", "T", 8, 8, 1000, (0, 0), True, True, True, True),
    ("f32", "N", 8, 8, 1000, (0, 0), True, True, False, True),
    ("f32", "T", 50, 75, 1000, (0, 0), True, True, False, True),
    ("f32", "N", 50, 75, 1000, (0, 0), True, True, False, True),
    ("f32", "N", 64, 128, 1024, (1, 1), True, True, False, True),
    ("f32", "T", 64, 128, 8064, (0, 0), True, True, True, True),
    ("f32", "N", 64, 128, 8064, (0, 0), True, True, False, False),
    ("f64", "T", 50, 75, 1000, (0, 0), True, True, {"copy", "scale"}, True),
    ("f64", "N", 50, 75, 1000, (0, 0), True, True, True, True),
    ("c64", "T", 50, 75, 1000, (0, 0), True, True, {"copy", "scale", "cscale"}, True),
    ("f64", "T", 64, 128, 3840, (0, 0), {"copy", "axpby2"}, {"copy", "axpby2"}, {"copy", "axpby2"}, {"copy", "axpby2"}),
])
def test_storage_in_host_memory(dtype, op, mb, ma, m, pads, device, a_host, b_host, both):
    """Where B's storage is in host memory, lists whose patches would read it in
    shorter pieces than tiles do stay on tiles."""
    for host, want in enumerate((device, a_host, b_host, both)):
        want = OF[dtype] if want is True else want or NONE
        assert kinds(dtype, op, mb, ma, m, pads=pads, host=host) == want, host


@pytest.mark.parametrize("op", ["N", "T"])
def test_f32_lists_that_are_a_quarter_misaligned(op):
    """One rank row in four with an odd leading dimension: every kind moves, at
    sizes where whole aligned tiles of some kinds stay."""
    assert kinds("f32", op, 64, 128, 6145, grid=4) == ALL


def test_targets_of_whole_runs_stay_on_tiles():
    """16-row panels: every target tile is one contiguous run."""
    m, n = 16384, 4096
    A = L.block_cyclic(m, n, 16, n, m // 16, 1, name="A")
    B = L.block_cyclic(n, m, 64, 64, m // 16, 1, name="B")
    assert dispatch("f64", (A, B, "T"))["patch_kinds"] == NONE


def _stored_by_block(n, mb, nb, mode):
    """n x n in mb x nb blocks, each stored on its own: owners at random, or 4 x 4
    block-cyclic (a rank's blocks of one block row follow each other)."""
    R, S = np.append(np.arange(0, n, mb), n), np.append(np.arange(0, n, nb), n)
    i, j = np.meshgrid(np.arange(len(R) - 1), np.arange(len(S) - 1), indexing="ij")
    own = (i * 7919 + j * 104729 + i * j) % 16 if mode == "rand" else i % 4 * 4 + j % 4
    return L.packed_blocks(R, S, own, 16)


@pytest.mark.parametrize("dtype, n, block, mode, want", [
    ("f64", 256, (8, 8), "rand", True), ("f64", 704, (8, 8), "rand", False), ("f64", 3072, (8, 8), "rand", False),
    ("f32", 704, (16, 16), "rand", True), ("f32", 3072, (16, 16), "rand", False),
    ("f64", 1536, (8, 8), "cyc", True), ("f64", 3072, (8, 8), "cyc", False), ("f32", 3072, (4, 4), "cyc", True),
    ("f32", 3072, (6, 6), "cyc", True), ("c128", 560, (4, 4), "rand", True), ("c128", 1000, (4, 4), "rand", False),
    ("c128", 1536, (8, 8), "rand", True), ("c128", 2048, (8, 8), "rand", False), ("c128", 2048, (10, 10), "rand", True),
])
def test_blocks_stored_apart(dtype, n, block, mode, want):
    """Patches end where a rank's blocks do not continue each other in storage:
    lists of many small ones stay on tiles."""
    A = _stored_by_block(n, *block, mode)
    B = L.block_cyclic(n, n, 64, 64, 4, 4, name="B")
    got = dispatch(dtype, (A, B, "T"))["patch_kinds"]
    if want and dtype == "f64" and mode == "cyc":
        got = got | {"axpby", "axpby2"}  # power-of-two cells may keep these
    assert got == (OF[dtype] if want else NONE)


@pytest.mark.parametrize("dtype, block, mode, want", [
    ("f64", 48, "rand", NONE), ("f64", 100, "rand", {"copy", "axpby2"}), ("f64", 48, "cyc", {"copy", "axpby2"}),
    ("f32", 100, "rand", NONE), ("f32", 48, "cyc", NONE), ("f32", 96, "rand", ALL), ("c64", 48, "rand", NONE),
    ("c64", 96, "rand", OF["c64"])])
def test_full_tiles_of_blocks_stored_apart(dtype, block, mode, want):
    """Lists of full tiles move to patches only where these are nearly whole."""
    n = 7680
    A = _stored_by_block(n, block, block, mode)
    B = L.block_cyclic(n, n, 64, 64, 4, 4, name="B")
    got = dispatch(dtype, (A, B, "N"))["patch_kinds"]
    assert got - {"axpby"} == want - {"axpby"}  # (TMA may take the general beta)


def test_mixed_element_orders_stay_on_tiles():
    """Layouts that mix element orders have no patches; in a batch the other
    problems move to patches, and every kind runs on both lists."""
    B = L.block_cyclic(70, 90, 5, 7, 2, 2, name="B")
    order = np.zeros((2, 3), np.int32)
    order[0, 1] = 1
    mixed = L.packed_blocks([0, 33, 90], [0, 20, 41, 70], np.arange(6).reshape(2, 3) % 4, 4, order=order)
    plain = L.block_cyclic(90, 70, 3, 11, 2, 2, name="A")
    d = dispatch("f64", (mixed, B, "T"))
    assert d["patch_kinds"] == NONE and d["tiles"] + d["misaligned"] + d["pieces"] > 0
    d = dispatch("f64", (plain, B, "T"))
    assert d["patch_kinds"] == ALL and d["tiles"] + d["misaligned"] + d["pieces"] == 0
    d = dispatch("f64", (mixed, B, "T"), (plain, B, "T"))
    assert d["patch_kinds"] == ALL and d["tiles_are_rest"] and d["tiles"] + d["misaligned"] + d["pieces"] > 0


@pytest.mark.parametrize("dtype", ["f64", "c128", "f32"])
def test_empty_problems_in_a_batch(dtype):
    """A problem without elements neither has patches nor keeps the others from
    theirs."""
    A, B = _pair(dtype, "T", 5, 7, 70, 90)
    empty = L.packed_blocks([0], [0, 5], np.zeros((0, 1), np.int32), 4)
    empty_b = L.packed_blocks([0, 5], [0], np.zeros((1, 0), np.int32), 4)
    assert dispatch(dtype, (empty, empty_b, "T"), (A, B, "T"))["patch_kinds"] == OF[dtype]
    assert dispatch(dtype, (empty, empty_b, "T"))["patch_kinds"] == NONE
