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
CPLX_KINDS = {"cplx": (complex(1.0, 0.5), complex(0.5, -0.25)), "cscale": (complex(0.3, -0.4), 0.0)}
#         m, n      source      target      grids   pads
SHAPES = (((1, 97), (5, 7), (3, 11), (1, 2), (0, 1)), ((97, 1), (5, 7), (3, 11), (2, 1), (1, 0)),
          ((33, 31), (50, 50), (75, 75), (1, 1), (1, 1)), ((65, 130), (1, 2), (3, 1), (2, 2), (0, 0)),
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
            check_problem(p, dev, guard=2)


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
    stream = torch.cuda.current_stream(dev).cuda_stream
    costa.costa_transform_batched([g.LA for g in runs], [g.LB for g in runs], [p.op for p in problems],
                                  [p.alpha for p in problems], [p.beta for p in problems], stream=stream)
    torch.cuda.synchronize(dev)
    for p, g in zip(problems, runs):
        compare(p, g.Ad.download(), g.oracle_result(), g.Ah, g.Bh)
        g.close()
