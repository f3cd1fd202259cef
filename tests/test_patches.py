"""CPU check of the patch kernel's work list: patches, expanded element by
element with the kernel's own index arithmetic, move exactly the elements
that the tile list moves (the general path), each from the same source
address to the same target address, within the kernel's limits."""
import numpy as np
import pytest

from workloads import configs as C
from workloads import layouts as L

costa = pytest.importorskip("paper_2106_06601_gb300")

FAKE = 1 << 40
ES = {"f32": 4, "f64": 8, "c64": 8, "c128": 16}


def _layout(spec, dtype, shift=0):
    ptrs = FAKE + spec.buf.astype(np.int64) * (1 << 32) + (spec.off + shift) * ES[dtype]
    return costa.costa_layout_from_spec(spec, dtype, ptrs)


def _tile_moves(tiles, es):
    out = []
    for t in tiles:
        x, y = np.meshgrid(np.arange(t["nx"], dtype=np.int64), np.arange(t["ny"], dtype=np.int64))
        d = int(t["dst"]) + (x + y * int(t["dld"])) * es
        s = int(t["src"]) + ((x * int(t["sld"]) + y) if t["flags"] & 1 else (x + y * int(t["sld"]))) * es
        out.append(np.stack([d.ravel(), s.ravel()]))
    return np.concatenate(out, axis=1) if out else np.zeros((2, 0), np.int64)


def _patch_moves(patches, cells, es):
    ext = 16 if es == 16 else 32
    out = []
    for p in patches:
        nx, ny, lm, rm = int(p["nx"]), int(p["ny"]), int(p["lmask"]), int(p["rmask"])
        assert 1 <= nx <= ext and 1 <= ny <= ext
        tr = bool(p["flags"] & 1)
        nl, nr = (ny, nx) if tr else (nx, ny)
        assert lm & 1 and rm & 1 and lm < 1 << nl and rm < 1 << nr
        nls, nrs = bin(lm).count("1"), bin(rm).count("1")
        assert nls <= 8 and nrs <= 8
        seg = lambda m, i: bin(m & ((2 << i) - 1)).count("1") - 1
        ls = np.array([seg(lm, i) for i in range(nl)])
        rs = np.array([seg(rm, i) for i in range(nr)])
        c = cells[int(p["cell0"]):int(p["cell0"]) + nls * nrs]
        assert len(c) == nls * nrs
        r, l = np.meshgrid(np.arange(nr), np.arange(nl), indexing="ij")
        k = rs[r] * nls + ls[l]
        # biased addresses wrap modulo 2^64
        s = (c["src"][k] + ((r * c["sld"].astype(np.int64)[k] + l) * es).astype(np.uint64)).astype(np.int64)
        if p["flags"] & 2:  # staged by whole aligned 16-byte chunks
            q = s.reshape(nr, nl // 4, 4)
            assert es == 4 and nx > 16 and np.all(q[..., 0] % 16 == 0) and np.all(np.diff(q, axis=2) == 4)
        x, y = (r, l) if tr else (l, r)
        d = int(p["dst"]) + (x + y * int(p["dld"])) * es
        out.append(np.stack([d.ravel(), s.ravel()]))
    return np.concatenate(out, axis=1) if out else np.zeros((2, 0), np.int64)


def _same(a, b):
    a, b = (m[:, np.lexsort((m[1], m[0]))] for m in (a, b))
    return np.array_equal(a, b)


def check(p, shift=0):
    """True when the pair has patches (and they were checked)."""
    LA, LB = _layout(p.A, p.dtype, shift), _layout(p.B, p.dtype, shift)
    try:
        patches, cells = costa.costa_debug_patches(LA, LB, p.op)
        tiles = costa.costa_debug_tiles(LA, LB, p.op)
    finally:
        LA.destroy()
        LB.destroy()
    one = lambda s: len(set(s.order[i, j] for i in range(s.nbr) for j in range(s.nbc)
                            if s.rsplit[i + 1] > s.rsplit[i] and s.csplit[j + 1] > s.csplit[j])) <= 1
    if not one(p.A) or not one(p.B):
        assert len(patches) == 0
        return False
    es = ES[p.dtype]
    got = _patch_moves(patches, cells, es)
    assert got.shape[1] == p.A.m * p.A.n
    assert _same(got, _tile_moves(tiles, es))
    conj = p.op == "C"
    assert np.all(((patches["flags"] & 4) != 0) == conj)
    return len(patches) > 0


def test_fuzz_and_small_blocks():
    seen = sum(check(C.fuzz_problem(k, max_dim=90)) for k in range(160))
    assert seen > 10  # both sides block-cyclic (one element order each): about one in nine
    assert all(check(C.small_block_problem(k)) for k in range(96))


@pytest.mark.parametrize("dtype", ["f32", "f64", "c128"])
@pytest.mark.parametrize("op", ["N", "T", "C"])
@pytest.mark.parametrize("storage", ["CC", "CR", "RC", "RR"])
def test_block_cyclic_forms(dtype, op, storage):
    """Grids from 1 x 1 (where the blocks of both sides join) to 2 x 3, block
    sizes that divide each other and that do not, odd leading dimensions and
    base addresses, both storage orders."""
    m, n = 83, 101
    for (mb, nb), (ma, na), (pr, pc), pad, shift in (((5, 7), (3, 4), (1, 1), 0, 0), ((50, 50), (75, 75), (2, 2), 1, 1),
                                                     ((1, 1), (2, 3), (2, 3), 3, 0), ((8, 8), (4, 16), (3, 2), 0, 1),
                                                     ((33, 65), (32, 32), (2, 1), 2, 0)):
        bm, bn = (m, n) if op == "N" else (n, m)
        B = L.block_cyclic(bm, bn, mb, nb, pr, pc, storage=storage[1], ld_pad=pad, name="B")
        A = L.block_cyclic(m, n, ma, na, pr, pc, grid_order="C", storage=storage[0], ld_pad=1 - pad % 2, name="A")
        assert check(C.Problem("patch", dtype, op, 1.0, 0.0, A, B), shift)


def test_joined_blocks_make_few_cells():
    """On 1 x 1 grids every block continues its neighbours in storage, so a
    whole patch is one cell whatever the block sizes."""
    B = L.block_cyclic(1280, 960, 5, 7, 1, 1, name="B")
    A = L.block_cyclic(960, 1280, 3, 4, 1, 1, name="A")
    LA, LB = _layout(A, "f64"), _layout(B, "f64")
    patches, cells = costa.costa_debug_patches(LA, LB, "T")
    assert len(patches) == 30 * 40 and len(cells) == len(patches)
    assert np.all(patches["nx"] == 32) and np.all(patches["ny"] == 32)


@pytest.mark.parametrize("dtype", ["f32", "f64", "c128"])
@pytest.mark.parametrize("m, n", [(590, 590), (850, 850), (1101, 1103)])
def test_extents_by_size(dtype, m, n):
    """Patch extents follow the matrix size: every size class covers A once."""
    for op in "NT":
        B = L.block_cyclic(*((m, n) if op == "N" else (n, m)), 50, 37, 2, 2, ld_pad=1, name="B")
        A = L.block_cyclic(m, n, 75, 24, 2, 2, name="A")
        assert check(C.Problem("patch", dtype, op, 1.0, 0.0, A, B))


@pytest.mark.parametrize("op", ["N", "T"])
@pytest.mark.parametrize("mb, ma, pad, chunks", [(8, 16, 0, True), (64, 128, 0, True), (8, 12, 4, True), (64, 64, 1, False),
                                                 (6, 16, 0, False)])
def test_chunks_of_aligned_f32_runs(op, mb, ma, pad, chunks):
    """f32 patches are staged by 16-byte chunks exactly where their source
    runs allow it (checked patch by patch in _patch_moves)."""
    m, n = 1100, 1108
    B = L.block_cyclic(*((m, n) if op == "N" else (n, m)), mb, mb, 2, 2, ld_pad=pad, name="B")
    A = L.block_cyclic(m, n, ma, ma, 2, 2, ld_pad=1, name="A")
    p = C.Problem("patch", "f32", op, 1.0, 0.0, A, B)
    assert check(p)
    LA, LB = _layout(A, "f32"), _layout(B, "f32")
    patches, _ = costa.costa_debug_patches(LA, LB, op)
    share = np.mean((patches["flags"] & 2) != 0)
    assert share > 0.5 if chunks else share < 0.25


@pytest.mark.parametrize("ld_pad", [0, 8])
def test_order_with_an_empty_first_block(ld_pad):
    """The order of the patches follows the leading dimension of the source's
    blocks, not that of an empty first one: the same patches with and without
    one, mixed by rows of the chains only where the columns lie off a multiple
    of 1 KB."""
    m = n = 1024
    A = L.block_cyclic(m, n, 8, 8, 2, 2, name="A")
    B = L.block_cyclic(n, m, 64, 64, 2, 2, ld_pad=ld_pad, name="B")
    R = np.concatenate([[0], B.rsplit])
    grow = lambda a: np.concatenate([a[:1], a])
    E = L.LayoutSpec(n, m, R, B.csplit, grow(B.owner), B.nranks, grow(B.buf), grow(B.off), grow(B.ld), grow(B.order),
                     B.bufsize, name="B")
    LA, L1, L2 = _layout(A, "f32"), _layout(B, "f32"), _layout(E, "f32")
    one, two = costa.costa_debug_patches(LA, L1, "T"), costa.costa_debug_patches(LA, L2, "T")
    assert np.array_equal(one[0], two[0]) and np.array_equal(one[1], two[1])
    step = np.diff(one[0]["dst"].astype(np.int64)) >> 32  # changes of the rank's buffer of A
    assert (np.count_nonzero(step) == 3) == (ld_pad == 0)


def test_planning_time_of_one_long_chain_beside_many_short_ones():
    """The order that mixes the chains' rows takes one step per row of
    patches: a target of one wide block beside 60,000 single columns, over
    16 single-row blocks (1.9 million patches), is planned in about a second,
    not in the product of the three numbers of chains (3e10 steps)."""
    import time

    rows, wide, single = 16, 60000 * 32, 60000
    cols = np.concatenate([[0, wide], wide + 1 + np.arange(single)])
    nbc = single + 1
    at = np.arange(rows * nbc, dtype=np.int64).reshape(rows, nbc)
    one = np.ones((rows, nbc), np.int32)
    LA = costa.costa_layout_create("f64", 1, np.arange(rows + 1), cols, 0 * one, FAKE + at * (1 << 26), one, 0 * one)
    n = wide + single
    LB = costa.costa_layout_create("f64", 1, np.array([0, rows]), np.array([0, n]), np.zeros((1, 1), np.int32),
                                   np.array([[FAKE << 8]]), np.array([[rows + 1]]), np.zeros((1, 1), np.int32))
    try:
        t0 = time.perf_counter()
        patches, cells = costa.costa_debug_patches(LA, LB, "N")
        took = time.perf_counter() - t0
    finally:
        LA.destroy()
        LB.destroy()
    assert len(patches) == rows * (wide // 32 + single) == len(cells)
    # mixed: two patches of the wide block's first row, then single columns
    assert list(patches["ny"][:4]) == [32, 32, 32, 32] and patches["ny"][2 * rows] == 1
    assert took < 12, took  # two calls of the planner; 0.9 s on an idle host
