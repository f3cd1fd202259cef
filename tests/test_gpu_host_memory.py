"""Storage in host memory.  Blocks may live in host memory allocated or
registered with CUDA (pinned); the kernels then read and write it directly
over the host link, and the results equal the oracle's exactly as for device
storage.  Pageable host memory is rejected when the plan is built, before any
kernel touches a block (the check runs through costa_plan_stats_get, whose
only kernel, the volume count, reads layout tables and no block)."""
import numpy as np
import pytest

import paper_2106_06601_gb300 as costa
from tests._gpu import compare
from workloads import configs as C
from workloads.materialize import HostMatrix, block_element_offsets

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def dev():
    d = torch.device("cuda:0")
    torch.cuda.set_device(d)
    return d


def _pinned(host: HostMatrix):
    t = torch.from_numpy(host.arena).pin_memory()
    assert t.is_pinned()
    return t


def _ptrs(spec, host: HostMatrix, arena_tensor):
    off = block_element_offsets(spec, host.starts)
    return (arena_tensor.data_ptr() + off * arena_tensor.element_size()).astype(np.uint64)


@pytest.mark.parametrize("case", [3, 9, 21, 40, 55, 77])
@pytest.mark.parametrize("mode", ["direct", "message"])
def test_pinned_host_storage_matches_oracle(case, mode, dev):
    p = C.fuzz_problem(case)
    Bh = HostMatrix(p.B, p.dtype).fill(p.b_kind, p.seed, p.src_stream)
    Ah = HostMatrix(p.A, p.dtype).fill(p.a_kind, p.seed, p.tgt_stream)
    Bt, At = _pinned(Bh), _pinned(Ah)
    LA = costa.costa_layout_from_spec(p.A, p.dtype, _ptrs(p.A, Ah, At))
    LB = costa.costa_layout_from_spec(p.B, p.dtype, _ptrs(p.B, Bh, Bt))
    try:
        stream = torch.cuda.current_stream(dev).cuda_stream
        costa.costa_transform(LA, LB, p.op, p.alpha, p.beta, relabel=True, stream=stream, mode=mode)
        torch.cuda.synchronize(dev)
        got = HostMatrix.__new__(HostMatrix)
        got.spec, got.dtype, got.guard, got.starts = p.A, p.dtype, 0, Ah.starts
        got.arena = At.numpy().copy()
        want = Ah.copy()
        import oracle
        oracle.transform(p.dtype, p.op, p.alpha, p.beta, p.A, want.buffers(), p.B, Bh.buffers())
        compare(p, got, want, Ah, Bh)
        assert np.array_equal(Bt.numpy(), Bh.arena, equal_nan=True)  # B is read-only
    finally:
        LA.destroy()
        LB.destroy()


@pytest.mark.parametrize("dtype, op, mb, ma", [("c128", "T", 8, 8), ("c128", "N", 50, 75), ("f32", "N", 8, 8), ("f32", "T", 50, 75),
                                               ("f64", "T", 50, 75), ("c64", "N", 8, 16)])
@pytest.mark.parametrize("a_host, b_host", [(True, True), (True, False), (False, True)])
def test_work_lists_follow_where_the_storage_lies(dtype, op, mb, ma, a_host, b_host, dev):
    """The planner sees which side is in host memory and chooses the work lists
    for it; the results equal the oracle's on either, as they do on the device."""
    import oracle
    from workloads import layouts as L
    from workloads.materialize import DeviceMatrix
    m, n = 150, 203
    B = L.block_cyclic(*((m, n) if op == "N" else (n, m)), mb, mb, 2, 2, name="B")
    A = L.block_cyclic(m, n, ma, ma, 2, 2, grid_order="C", name="A")
    for alpha, beta in ((1.0, 0.0), (2.0, 0.5)):
        hb = HostMatrix(B, dtype).fill("uniform", C.SEED0 + 19, lambda r: r)
        ha = HostMatrix(A, dtype).fill("uniform", C.SEED0 + 20, lambda r: r)
        want = ha.copy()
        oracle.transform(dtype, op, alpha, beta, A, want.buffers(), B, hb.buffers())
        place = []
        for spec, h, on_host in ((A, ha, a_host), (B, hb, b_host)):
            t = _pinned(h) if on_host else DeviceMatrix(spec, dtype, dev).upload(h)
            ptrs = _ptrs(spec, h, t) if on_host else t.block_ptrs()
            place.append((t, costa.costa_layout_from_spec(spec, dtype, ptrs)))
        (At, LA), (_, LB) = place
        before = costa.costa_debug_dispatch([LA], [LB], [op])
        costa.costa_transform(LA, LB, op, alpha, beta, stream=torch.cuda.current_stream(dev).cuda_stream)
        torch.cuda.synchronize(dev)
        got = At.numpy() if a_host else At.download().arena
        assert np.array_equal(got, want.arena)
        assert before == costa.costa_debug_dispatch([LA], [LB], [op], host=0)  # not looked at yet
        lists = costa.costa_debug_dispatch([LA], [LB], [op], host=(1 if a_host else 0) | (2 if b_host else 0))
        assert costa.costa_debug_dispatch([LA], [LB], [op]) == lists
        if dtype == "c128" and b_host:
            assert not lists["patch_kinds"] and before["patch_kinds"]
        LA.destroy()
        LB.destroy()


def test_pageable_host_storage_is_rejected(dev):
    from workloads.materialize import DeviceMatrix
    p = C.fuzz_problem(3)
    Bh = HostMatrix(p.B, p.dtype).fill(p.b_kind, p.seed, p.src_stream)
    Ad = DeviceMatrix(p.A, p.dtype, dev)
    LA = costa.costa_layout_from_spec(p.A, p.dtype, Ad.block_ptrs())
    # B's blocks point into a plain numpy array: pageable memory
    LB = costa.costa_layout_from_spec(p.B, p.dtype, _ptrs(p.B, Bh, torch.from_numpy(Bh.arena)))
    try:
        with pytest.raises(costa.CostaError) as e:
            costa.costa_plan_stats_get(LA, LB, p.op, relabel=True,
                                       stream=torch.cuda.current_stream(dev).cuda_stream)
        assert e.value.status == 2 and "pageable" in str(e.value)
    finally:
        LA.destroy()
        LB.destroy()
