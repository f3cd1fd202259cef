"""The patch kernel against the oracle at the edges of its patches: extents
of one element, one less and one more than a patch and its segments, blocks
that do not divide each other, joined blocks (1 x 1 grids), odd leading
dimensions, every combine kind, element type, op and storage order."""
import pytest

from tests.test_gpu_parity import check_problem
from workloads import configs as C
from workloads import layouts as L

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

KINDS = {"copy": (1.0, 0.0), "scale": (-0.7, 0.0), "axpby": (-0.3, 0.7), "axpby2": (2.0, -0.5)}
CPLX_KINDS = {"cplx": (complex(1.0, 0.5), complex(0.5, -0.25)), "cplxr": (-1.5, complex(0.3, 0.7)), "cscale": (complex(0.3, -0.4), 0.0)}
#         m, n      source      target      grids   pads
SHAPES = (((1, 97), (5, 7), (3, 11), (1, 2), (0, 1)), ((97, 1), (5, 7), (3, 11), (2, 1), (1, 0)),
          ((33, 31), (50, 50), (75, 75), (1, 1), (1, 1)), ((17, 31), (50, 50), (75, 75), (1, 1), (1, 1)), ((65, 130), (1, 2), (3, 1), (2, 2), (0, 0)),
          ((131, 94), (17, 33), (16, 9), (2, 3), (3, 1)), ((160, 96), (8, 8), (4, 16), (2, 2), (0, 0)))


@pytest.fixture(scope="module")
def dev():
    d = torch.device("cuda:0")
    torch.cuda.set_device(d)
    return d


@pytest.mark.parametrize("dtype", ["f32", "f64", "c64", "c128"])
@pytest.mark.parametrize("op", ["N", "T", "C"])
def test_edges_of_patches(dtype, op, dev):
    kinds = {**KINDS, **(CPLX_KINDS if dtype[0] == "c" else {})}
    for i, ((m, n), (mb, nb), (ma, na), (pr, pc), (pb, pa)) in enumerate(SHAPES):
        for k, (alpha, beta) in enumerate(kinds.values()):
            sb, sa = ("C", "R")[(i + k) % 2], ("C", "R")[k // 2 % 2]
            bm, bn = (m, n) if op == "N" else (n, m)
            B = L.block_cyclic(bm, bn, mb, nb, pr, pc, storage=sb, ld_pad=pb)
            A = L.block_cyclic(m, n, ma, na, pr, pc, grid_order="C", storage=sa, ld_pad=pa)
            p = C.Problem(f"patch{i}", dtype, op, alpha, beta, A, B, "uniform", "nan" if beta == 0 else "uniform",
                          C.SEED0 + 11)
            # one aligned, nearly full tile stays on tiles (33 x 31; not in f32, and
            # not where the guards leave it misaligned)
            check_problem(p, dev, guard=2, lists=None if (m, n) == (33, 31) else {"patches"})


@pytest.mark.parametrize("dtype", ["f32", "f64", "c64", "c128"])
@pytest.mark.parametrize("m, n", [(590, 601), (850, 870), (1101, 1107)])
def test_extents_by_size(dtype, m, n, dev):
    """The patch extents of each size class, with and without A."""
    for op, (alpha, beta) in (("T", (1.0, 0.0)), ("N", (-0.3, 0.7)), ("C", (2.0, 0.5))):
        B = L.block_cyclic(*((m, n) if op == "N" else (n, m)), 50, 37, 2, 2, ld_pad=1)
        A = L.block_cyclic(m, n, 75, 24, 2, 2)
        check_problem(C.Problem("patch", dtype, op, alpha, beta, A, B, "uniform", "nan" if beta == 0 else "uniform",
                                C.SEED0 + 13), dev, lists={"patches"})


@pytest.mark.parametrize("op", ["N", "T"])
@pytest.mark.parametrize("mb, ma, pads", [(8, 16, (0, 0)), (8, 12, (4, 1)), (16, 5, (0, 0)), (24, 8, (8, 3))])
def test_chunks_of_aligned_f32_runs(mb, ma, pads, op, dev):
    """f32 patches that are staged by 16-byte chunks, beside ragged ones that
    are not, for every kind."""
    m, n = 1100, 1108
    for alpha, beta in KINDS.values():
        B = L.block_cyclic(*((m, n) if op == "N" else (n, m)), mb, mb, 2, 2, ld_pad=pads[0])
        A = L.block_cyclic(m, n, ma, ma, 2, 2, ld_pad=pads[1])
        check_problem(C.Problem("patch", "f32", op, alpha, beta, A, B, "uniform", "nan" if beta == 0 else "uniform",
                                C.SEED0 + 14), dev, lists={"patches"})


@pytest.mark.parametrize("dtype", ["f32", "f64", "c64", "c128"])
@pytest.mark.parametrize("m, n", [(32, 64), (68, 36), (128, 128), (600, 404), (800, 768)])
def test_lists_of_few_tiles(dtype, m, n, dev):
    """Short lists of aligned tiles, which are cut into halves and quarters
    by rows: one tile, ragged tiles, and lists about the limit."""
    for op, (alpha, beta) in zip("TNCT", KINDS.values()):
        B = L.block_cyclic(*((m, n) if op == "N" else (n, m)), 64, 32, 1, 2)
        A = L.block_cyclic(m, n, 32, 128, 2, 1)
        check_problem(C.Problem("few", dtype, op, alpha, beta, A, B, "uniform", "nan" if beta == 0 else "uniform",
                                C.SEED0 + 15), dev, guard=4, lists={"tiles"})


def _special_doubles(n, rng):
    """Random doubles with all exponents, exact halfway products, zeros,
    subnormals, infinities and NaNs among runs of ordinary values."""
    import numpy as np

    v = rng.standard_normal(n)
    k = n // 4  # ordinary runs stay: whole warps without a special value
    at = k + rng.permutation(n - k)[:k]
    bits = rng.integers(0, 1 << 63, k, dtype=np.uint64) | (rng.integers(0, 2, k, dtype=np.uint64) << np.uint64(63))
    v[at] = bits.view(np.float64)
    few = at[:k // 2]
    v[few] = np.ldexp(np.round(np.ldexp(rng.random(len(few)), 20)), rng.integers(-1070, 1000, len(few)))  # few bits: exact
    v[at[:64]] = np.resize([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -2.2e-308, 1.7e308], 64)
    return v


@pytest.mark.parametrize("factor", [0.7, -3.0, 1.0 + 2.0 ** -52, 1.5e-300, 7e250, 5e-324])
@pytest.mark.parametrize("scale", [True, False])
def test_products_of_doubles_are_rounded_once(factor, scale, dev):
    """beta * a (with a zero B) and alpha * b equal numpy's products bit for
    bit, whichever pipe forms them."""
    import numpy as np

    from tests._gpu import OnDevice, block_mask
    from tests._util import global_matrix
    from workloads.materialize import HostMatrix

    B = L.block_cyclic(300, 210, 50, 50, 2, 2, name="B")
    A = L.block_cyclic(210, 300, 75, 75, 2, 2, name="A")
    alpha, beta = (factor, 0.0) if scale else (1.0, factor)
    p = C.Problem("rn", "f64", "T", alpha, beta, A, B)
    rng = np.random.default_rng(7)
    hb, ha = HostMatrix(B, "f64"), HostMatrix(A, "f64")
    (hb if scale else ha).arena[...] = _special_doubles((hb if scale else ha).arena.size, rng)
    g = OnDevice(p, dev, B_host=hb, A_host=ha)
    g.run()
    got = g.Ad.download()
    g.close()
    with np.errstate(all="ignore"):
        want = factor * global_matrix(B, hb.buffers()).real.T if scale else factor * global_matrix(A, ha.buffers()).real + 0.0
    G = global_matrix(A, got.buffers()).real
    same = (G.view(np.int64) == np.ascontiguousarray(want).view(np.int64)) | (np.isnan(G) & np.isnan(want))
    assert np.all(same), np.argwhere(~same)[:3]
    mask = block_mask(A, ha)
    assert np.array_equal(got.arena[~mask], ha.arena[~mask], equal_nan=True)


def test_batch_of_tiles_and_patches(dev):
    """One batch whose problems differ in kind, op and work list: layouts with
    mixed element orders stay with the tile kernels."""
    import numpy as np

    import paper_2106_06601_gb300 as costa
    from tests._gpu import OnDevice, compare

    problems = []
    for k, (alpha, beta) in enumerate(KINDS.values()):
        B = L.block_cyclic(70, 90, 5, 7, 2, 2, ld_pad=1)
        order = np.zeros((2, 3), np.int32)
        order[0, 1] = k % 2
        am, an = (70, 90) if k % 2 else (90, 70)
        A = L.packed_blocks([0, 33, am], [0, 20, 41, an], np.arange(6).reshape(2, 3) % 4, 4, order=order)
        problems.append(C.Problem("batch", "f64", "NT"[1 - k % 2], alpha, beta, A, B, "uniform",
                                  "nan" if beta == 0 else "uniform", C.SEED0 + 12, index=k))
    runs = [OnDevice(p, dev, guard=2) for p in problems]
    d = costa.costa_debug_dispatch([g.LA for g in runs], [g.LB for g in runs], [p.op for p in problems])
    assert d["patches"] > 0 and d["tiles_are_rest"] and d["tiles"] + d["misaligned"] + d["pieces"] > 0
    stream = torch.cuda.current_stream(dev).cuda_stream
    costa.costa_transform_batched([g.LA for g in runs], [g.LB for g in runs], [p.op for p in problems],
                                  [p.alpha for p in problems], [p.beta for p in problems], stream=stream)
    torch.cuda.synchronize(dev)
    for p, g in zip(problems, runs):
        compare(p, g.Ad.download(), g.oracle_result(), g.Ah, g.Bh)
        g.close()


@pytest.mark.parametrize("m, n, mb, ma, on_tiles", [(1024, 768, 8, 8, {"axpby", "axpby2"}), (1920, 1952, 64, 128, {"axpby", "scale"})])
def test_batch_whose_kinds_differ_in_list(m, n, mb, ma, on_tiles, dev):
    """One batch of four kinds over the same layouts, some of which run on
    patches and some on the tiles of the same problems: each launch moves its
    own kind's problems and no others."""
    import numpy as np

    import paper_2106_06601_gb300 as costa
    from tests._gpu import OnDevice, compare, kind_name

    problems = []
    for k, (alpha, beta) in enumerate(KINDS.values()):
        B = L.block_cyclic(n, m, mb, mb, 2, 2)
        A = L.block_cyclic(m, n, ma, ma, 2, 2, grid_order="C")
        problems.append(C.Problem("kinds", "f64", "T", alpha, beta, A, B, "uniform", "nan" if beta == 0 else "uniform",
                                  C.SEED0 + 16, index=k))
    runs = [OnDevice(p, dev) for p in problems]
    d = costa.costa_debug_dispatch([g.LA for g in runs], [g.LB for g in runs], [p.op for p in problems])
    assert not d["tiles_are_rest"] and {kind_name(p.dtype, p.alpha, p.beta) for p in problems} - d["patch_kinds"] == on_tiles
    want = [g.oracle_result() for g in runs]
    n0 = costa.costa_kernel_launch_count()
    costa.costa_transform_batched([g.LA for g in runs], [g.LB for g in runs], [p.op for p in problems],
                                  [p.alpha for p in problems], [p.beta for p in problems],
                                  stream=torch.cuda.current_stream(dev).cuda_stream)
    torch.cuda.synchronize(dev)
    assert costa.costa_kernel_launch_count() > n0
    for p, g, w in zip(problems, runs, want):
        compare(p, g.Ad.download(), w, g.Ah, g.Bh)
        assert np.array_equal(g.Bd.download().arena, g.Bh.arena)
        g.close()


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("dtype, m, n, blocks", [("f64", 333, 257, (8, 5)), ("f32", 1100, 900, (50, 75)), ("c128", 200, 333, (6, 9)),
                                                 ("f64", 640, 512, (64, 128))])
def test_chain_of_calls_each_reading_what_the_last_wrote(dtype, m, n, blocks, graph, dev):
    """Kernels start before the one ahead of them has ended: in a chain of
    calls each reads as B what the call before it wrote as A (and adds it to
    what that call read), on patches, tiles and in message mode by turns,
    without a wait between them."""
    import numpy as np

    import oracle
    import paper_2106_06601_gb300 as costa
    from workloads.materialize import DeviceMatrix, HostMatrix

    spec = [L.block_cyclic(m, n, blocks[0], blocks[0], 2, 2), L.block_cyclic(n, m, blocks[1], blocks[1], 2, 2, grid_order="C")]
    host = [HostMatrix(s, dtype).fill("uniform", C.SEED0 + 17 + k, lambda r: r) for k, s in enumerate(spec)]
    mats = [DeviceMatrix(s, dtype, dev).upload(h) for s, h in zip(spec, host)]
    lay = [costa.costa_layout_from_spec(s, dtype, d.block_ptrs()) for s, d in zip(spec, mats)]
    on = costa.costa_debug_dispatch([lay[1]], [lay[0]], ["T"])["patch_kinds"]
    assert ("axpby2" in on) == (blocks != (64, 128))
    stream = torch.cuda.Stream(dev)
    calls = 30

    def chain():
        for k in range(calls):
            src, dst = k % 2, 1 - k % 2
            costa.costa_transform(lay[dst], lay[src], "T", 0.5, -0.5, stream=stream.cuda_stream,
                                  mode="message" if k % 5 == 4 else "direct")

    want = [h.copy() for h in host]
    for k in range(calls):
        src, dst = k % 2, 1 - k % 2
        oracle.transform(dtype, "T", 0.5, -0.5, spec[dst], want[dst].buffers(), spec[src], want[src].buffers())
    torch.cuda.synchronize(dev)
    if graph:
        for mode in ("direct", "message"):  # the plans, outside the capture
            for src in (0, 1):
                costa.costa_transform(lay[1 - src], lay[src], "T", 1.0, 0.0, stream=stream.cuda_stream, mode=mode)
        torch.cuda.synchronize(dev)
        for d, h in zip(mats, host):
            d.upload(h)
        torch.cuda.synchronize(dev)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            chain()
        with torch.cuda.stream(stream):
            g.replay()
    else:
        chain()
    torch.cuda.synchronize(dev)
    for d, w in zip(mats, want):
        assert np.array_equal(d.download().arena, w.arena)
    for x in lay:
        x.destroy()
