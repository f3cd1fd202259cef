"""GPU-side helpers for the parity tests: put a Problem on the device, run the
library through its C ABI, and compare with the CPU oracle."""
from __future__ import annotations

import numpy as np

import oracle
from tests._util import assert_close, exact_case, global_matrix, op_apply, scatter_global
from workloads.materialize import DeviceMatrix, HostMatrix, host_problem

SENTINEL = {"f32": -77.25, "f64": -77.25, "c64": complex(-77.25, 3.5), "c128": complex(-77.25, 3.5)}


def kind_name(dtype, alpha, beta) -> str:
    """The combine kind of a problem's scalars, by its name in
    costa_debug_dispatch."""
    al, be = oracle.scalar(dtype, alpha), oracle.scalar(dtype, beta)
    if al.imag or be.imag:
        if be == 0:
            return "cscale"
        return "cplxr" if dtype == "c128" and al.imag == 0 else "cplx"
    if be != 0:
        return "axpby2" if np.frexp(abs(be.real))[0] == 0.5 else "axpby"
    return "copy" if al == 1 else "scale"


class OnDevice:
    def __init__(self, prob, device, guard: int = 0, B_host=None, A_host=None):
        import paper_2106_06601_gb300 as costa
        self.p = prob
        self.device = device
        sentinel = SENTINEL[prob.dtype] if guard else None
        if B_host is None:
            B_host = HostMatrix(prob.B, prob.dtype, guard, sentinel).fill(
                prob.b_kind, prob.seed, prob.src_stream)
            A_host = HostMatrix(prob.A, prob.dtype, guard, sentinel).fill(
                prob.a_kind, prob.seed, prob.tgt_stream)
        self.Bh, self.Ah = B_host, A_host
        self.Bd = DeviceMatrix(prob.B, prob.dtype, device, guard).upload(self.Bh)
        self.Ad = DeviceMatrix(prob.A, prob.dtype, device, guard).upload(self.Ah)
        self.LA = costa.costa_layout_from_spec(prob.A, prob.dtype, self.Ad.block_ptrs())
        self.LB = costa.costa_layout_from_spec(prob.B, prob.dtype, self.Bd.block_ptrs())

    def run(self, relabel=True, mode="direct"):
        import torch
        import paper_2106_06601_gb300 as costa
        stream = torch.cuda.current_stream(self.device).cuda_stream
        sigma = costa.costa_transform(self.LA, self.LB, self.p.op, self.p.alpha, self.p.beta,
                                      relabel=relabel, stream=stream, mode=mode)
        torch.cuda.synchronize(self.device)
        return sigma

    def lists(self) -> set:
        """The work lists that a direct call of this problem runs (the planner's
        own choice)."""
        import paper_2106_06601_gb300 as costa
        d = costa.costa_debug_dispatch([self.LA], [self.LB], [self.p.op])
        patches = kind_name(self.p.dtype, self.p.alpha, self.p.beta) in d["patch_kinds"]
        tiles = {k for k in ("tiles", "misaligned", "pieces") if d[k]}
        return ({"patches"} if patches else set()) | (tiles if d["tiles_are_rest"] or not patches else set())

    def reset_A(self):
        self.Ad.upload(self.Ah)

    def oracle_result(self) -> HostMatrix:
        want = self.Ah.copy()
        oracle.transform(self.p.dtype, self.p.op, self.p.alpha, self.p.beta, self.p.A,
                         want.buffers(), self.p.B, self.Bh.buffers())
        return want

    def close(self):
        self.LA.destroy()
        self.LB.destroy()


def block_mask(spec, host: HostMatrix) -> np.ndarray:
    """Boolean arena mask of the elements that belong to some block."""
    mk = HostMatrix.__new__(HostMatrix)
    mk.spec, mk.dtype, mk.guard, mk.starts = spec, "f64", host.guard, host.starts
    mk.arena = np.zeros(host.arena.size, np.float64)
    scatter_global(spec, mk.buffers(), np.ones((spec.m, spec.n)))
    return mk.arena != 0


def compare(p, got: HostMatrix, want: HostMatrix, A_in: HostMatrix, B_in: HostMatrix):
    """Whole-arena comparison: block elements bit-exact or within the derived
    tolerance; every other element (padding, guards) unchanged."""
    al, be = oracle.scalar(p.dtype, p.alpha), oracle.scalar(p.dtype, p.beta)
    if exact_case(p.dtype, al, be):
        ok = (got.arena == want.arena) | (np.isnan(got.arena) & np.isnan(want.arena))
        if not np.all(ok):
            bad = np.flatnonzero(~ok)
            raise AssertionError(f"{p.name}: {bad.size} elements differ; first {bad[:5]} "
                                 f"got {got.arena[bad[:5]]} want {want.arena[bad[:5]]}")
        return
    mask = block_mask(p.A, A_in)
    assert np.array_equal(got.arena[~mask], A_in.arena[~mask], equal_nan=True)
    G = global_matrix(p.A, got.buffers())
    W = global_matrix(p.A, want.buffers())
    X = op_apply(p.op, global_matrix(p.B, B_in.buffers()))
    A0 = global_matrix(p.A, A_in.buffers())
    assert_close(p.dtype, G, W, al, be, X if p.dtype in ("c64", "c128") else X.real, A0,
                 exact=False)
