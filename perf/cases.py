"""The work that is timed: reshuffles A = alpha * op(B) + beta * A through the
library's public entry points, as a program that holds its matrices on the GPU
calls them.

The layouts, matrices and expected results are built here in plain torch; the
package is used for the calls themselves (layouts, plans, transforms).  A
state holds what such a program keeps between calls: the two matrices, their
layouts, the plan of the pair (costa_plan_stats_get builds it, as a program
would before capturing or timing), and for the exchange its buffers.
"""
import math
import random

import numpy as np
import torch

import paper_2106_06601_gb300 as costa

DEV = "cuda"
TYPES = {"f32": torch.float32, "f64": torch.float64, "c64": torch.complex64, "c128": torch.complex128}
SIZE = {"f32": 4, "f64": 8, "c64": 8, "c128": 16}

# Every key of a case, with the value that an ordinary call has.
#   api      transform | batched | scalapack | exchange
#   m, n     A's extent (the submatrix's with api = scalapack)
#   b_*, a_* source and target: block size mb x nb on a pr x pc process grid;
#            pad: elements that each rank's leading dimension has beyond its rows
#   perm     the target's ranks are a fixed permutation of the grid's
#   target   cyclic | irregular (an 8 x 8 grid of unequal blocks) | panels (row panels, one per rank)
#   count    pairs in a batch; their block sizes are drawn from 16 .. 128, N and T in turn
#   bi, ai   first row = first column of the submatrix in the source and in the target (1-based)
#   gpus     processes that share the ranks of an exchange (this one is process 0)
DEFAULT = dict(api="transform", dtype="f64", op="N", m=1024, n=1024, b_mb=64, b_nb=64, b_pr=4, b_pc=4, b_pad=0,
               a_mb=64, a_nb=64, a_pr=4, a_pc=4, a_pad=0, perm=False, target="cyclic", alpha_re=1.0, alpha_im=0.0,
               beta_re=0.0, beta_im=0.0, relabel=False, count=1, bi=1, ai=1, gpus=1)


def _blocks(side, mb, nb, pr, pc, pad=0):
    return {side + "_mb": mb, side + "_nb": nb, side + "_pr": pr, side + "_pc": pc, side + "_pad": pad}


def _scalars(alpha, beta):
    a, b = complex(alpha), complex(beta)
    return dict(alpha_re=a.real, alpha_im=a.imag, beta_re=b.real, beta_im=b.imag)


def _case(name, b, a, scalars=(1.0, 0.0), **more):
    return {**DEFAULT, **_blocks("b", *b), **_blocks("a", *a), **_scalars(*scalars), **more, "name": name}


def listed():
    return [
        # One small redistribution between two solver steps: latency of a call.
        _case("small_copy", (16, 16, 2, 2), (32, 32, 2, 2), dtype="f64", m=256, n=256, relabel=True),
        # A panel-sized accumulate on a ragged matrix: a few microseconds of data.
        _case("panel_add", (32, 32, 2, 2), (64, 64, 2, 2), (1.0, 1.0), dtype="f64", op="T", m=1000, n=1500),
        # ScaLAPACK-style redistribute-and-transpose to larger blocks with an update of the target.
        _case("square_t", (64, 64, 4, 4), (128, 128, 4, 4), (2.0, 0.5), dtype="f64", op="T", m=8192, n=8192,
              perm=True),
        # Conjugate transpose of a complex matrix into an application's own unequal blocks.
        _case("irregular_c", (32, 32, 8, 8), (32, 32, 8, 8), dtype="c128", op="C", m=16384, n=16384,
              target="irregular"),
        # Many independent matrices of one round of communication in one call.
        _case("batch", (64, 64, 4, 4), (64, 64, 4, 4), api="batched", dtype="f32", m=2048, n=3072, count=64),
        # Tall-skinny RPA matrix, block-cyclic to one row panel per rank, accumulated; the largest.
        _case("tall_skinny", (32, 32, 16, 16), (16, 16, 16, 16), (1.0, 1.0), dtype="f64", op="T", m=4096, n=131072,
              target="panels"),
        # Small blocks on both sides (fine load balance of a factorisation).
        _case("small_blocks", (8, 8, 4, 4), (8, 8, 4, 4), (2.0, 0.5), dtype="f64", op="T", m=8192, n=8192, perm=True),
        # Block sizes that are no power of two, on both sides: every run starts anywhere.
        _case("odd_blocks", (50, 50, 4, 4), (75, 75, 4, 4), dtype="f64", op="T", m=8192, n=8192),
        # Single precision into local matrices with an odd leading dimension.
        _case("odd_ld", (64, 64, 4, 4), (128, 128, 4, 4, 1), dtype="f32", op="T", m=8192, n=8192),
        # A complex update of a complex matrix: arithmetic beside the traffic.
        _case("complex_add", (64, 64, 4, 4), (128, 128, 4, 4), (1.0, 0.5 + 0.25j), dtype="c128", op="T", m=4096,
              n=4096, perm=True),
        # pdtran on a submatrix of a ragged matrix, other grids on the two sides, general scalars.
        _case("pdtran_sub", (64, 64, 4, 4), (64, 64, 2, 8), (-0.3, 0.7), api="scalapack", dtype="f64", op="T",
              m=6001, n=4999, bi=34, ai=66),
        # One process's share of a reshuffle over four GPUs: pack, local part, unpack.
        _case("exchange", (64, 64, 4, 4), (128, 128, 4, 4), (2.0, 0.5), api="exchange", dtype="f64", op="T", m=8192,
              n=8192, perm=True, gpus=4),
    ]


GRIDS = ((1, 1), (2, 2), (2, 4), (4, 2), (4, 4), (2, 8), (8, 8))


def draw(rng):
    """One more call of the same kinds: any element type, op, scalars and entry point, extents over their whole
    range (half of them ragged), usual, odd and small block sizes."""
    api = rng.choices(("transform", "scalapack", "batched", "exchange"), (62, 20, 8, 10))[0]
    dtype = rng.choices(("f64", "f32", "c128", "c64"), (40, 25, 18, 17))[0]
    es = SIZE[dtype]
    elems = 2.0 ** rng.uniform(14, 27 if es < 16 else 26.5)
    aspect = 2.0 ** rng.uniform(-2, 2)
    m, n = max(40, int(math.sqrt(elems * aspect))), max(40, int(math.sqrt(elems / aspect)))
    if rng.random() < 0.5:
        m, n = max(64, m // 64 * 64), max(64, n // 64 * 64)
    sizes = []
    for _ in range(2):
        kind = rng.choices(("usual", "odd", "small"), (60, 25, 15))[0]
        pick = {"usual": (16, 32, 64, 128, 256), "odd": (10, 24, 37, 48, 50, 75, 100), "small": (4, 6, 8, 12)}[kind]
        mb = rng.choice(pick)
        sizes.append((mb, mb if rng.random() < 0.7 else rng.choice(pick)))
    # a program with a million blocks or more would not choose them this small
    sizes = [(max(b, math.ceil(x / 1024)), max(c, math.ceil(y / 1024)))
             for (b, c), (x, y) in zip(sizes, ((min(m, n), min(m, n)), (m, n)))]
    g = [rng.choice(GRIDS), rng.choice(GRIDS)]
    if g[0][0] * g[0][1] != g[1][0] * g[1][1]:
        g[1] = g[0][::-1]
    kinds = [((1.0, 0.0), 45), ((2.0, 0.5), 12), ((1.0, 1.0), 13), ((-0.3, 0.7), 15), ((1.5, 0.0), 8)]
    if dtype[0] == "c":
        kinds += [((0.3 - 0.4j, 0.0), 8), ((1.0, 0.5 + 0.25j), 10)]
    scalars = rng.choices([k for k, _ in kinds], [w for _, w in kinds])[0]
    pads = [rng.choice((0, 0, 0, 1, 3, 8)) for _ in range(2)]
    op = rng.choice("NT" if dtype[0] == "f" else "NTC")
    case = {**DEFAULT, **_blocks("b", *sizes[0], *g[0], pads[0]), **_blocks("a", *sizes[1], *g[1], pads[1]),
            **_scalars(*scalars), "api": api, "dtype": dtype, "op": op, "m": m, "n": n,
            "perm": rng.random() < 0.5, "relabel": rng.random() < 0.3}
    if api == "scalapack":
        case.update(bi=rng.choice((1, 1, 33, 34, 130)), ai=rng.choice((1, 1, 66, 65, 7)), perm=False, relabel=False)
        if op == "N":  # pxgemr2d copies
            case.update(_scalars(1.0, 0.0))
    elif api == "batched":
        count = rng.choice((2, 3, 8, 24))
        case.update(count=count, m=max(40, m // 4), n=max(40, n // 4), perm=False)
    elif api == "exchange":
        ranks = g[0][0] * g[0][1]
        case.update(gpus=rng.choice([k for k in (2, 4) if ranks % k == 0] or [1]), relabel=False)
        if case["gpus"] == 1:
            case["api"] = "transform"
    elif rng.random() < 0.15:
        case.update(target="irregular", a_pr=8, a_pc=8, b_pr=8, b_pc=8, a_pad=0, m=max(64, m), n=max(64, n))
    return case


# ---- layouts in plain arrays ----

def _cyclic_index(extent, b, p, first=0):
    """For each process of one axis, the global indices it holds, in local order (blocks b, p processes)."""
    g = np.arange(extent)
    return [g[(g // b + first) % p == k] for k in range(p)]


class _Layout:
    """Where each rank's local matrices lie in one arena: parts (owner, rows, columns, offset, ld), each a
    column-major local matrix with the global rows and columns that it holds."""

    def __init__(self, m, n):
        self.m, self.n, self.parts, self.size, self.make = m, n, [], 0, None

    def add(self, owner, rows, cols, ld, es):
        align = 256 // es
        self.parts.append((owner, rows, cols, self.size, ld))
        self.size += -(-max(1, ld * len(cols)) // align) * align

    def put(self, arena, matrix, owners=None):
        """Writes a global matrix into the arena (only the blocks of `owners`, if given)."""
        for owner, rows, cols, off, ld in self.parts:
            if owners is not None and owner not in owners or len(rows) == 0 or len(cols) == 0:
                continue
            out = torch.as_strided(arena, (len(rows), len(cols)), (1, ld), off)
            if isinstance(rows, _Span):
                out.copy_(matrix[rows.lo:rows.hi, cols.lo:cols.hi])
            else:
                out.copy_(matrix[torch.as_tensor(rows, device=DEV)][:, torch.as_tensor(cols, device=DEV)])
        return arena


class _Span:
    """The indices lo .. hi - 1, taken as a slice."""

    def __init__(self, lo, hi):
        self.lo, self.hi = int(lo), int(hi)

    def __len__(self):
        return self.hi - self.lo


def _permutation(p):
    order = list(range(p))
    random.Random(p).shuffle(order)
    return order


def _cyclic(m, n, mb, nb, pr, pc, pad, perm, dtype):
    lay, es = _Layout(m, n), SIZE[dtype]
    owners = _permutation(pr * pc) if perm else list(range(pr * pc))
    rows, cols = _cyclic_index(m, mb, pr), _cyclic_index(n, nb, pc)
    for r in range(pr * pc):
        i, j = r // pc, r % pc
        lay.add(owners[r], rows[i], cols[j], max(1, len(rows[i])) + pad, es)
    place = {part[0]: part for part in lay.parts}
    ld = [place[o][4] for o in range(pr * pc)]

    def make(arena):
        ptrs = [arena.data_ptr() + place[o][3] * es for o in range(pr * pc)]
        return costa.costa_layout_create_block_cyclic(dtype, m, n, mb, nb, pr, pc, "R", owners, ptrs, ld)

    lay.make, lay.owners = make, owners
    lay.row_proc, lay.col_proc = (np.arange(m) // mb) % pr, (np.arange(n) // nb) % pc
    return lay


def _blocked(row_cuts, col_cuts, owners, ranks, dtype):
    """Blocks of a grid of cuts, each dense and column-major."""
    lay, es = _Layout(row_cuts[-1], col_cuts[-1]), SIZE[dtype]
    for i in range(len(row_cuts) - 1):
        for j in range(len(col_cuts) - 1):
            h = row_cuts[i + 1] - row_cuts[i]
            lay.add(owners[i][j], _Span(row_cuts[i], row_cuts[i + 1]), _Span(col_cuts[j], col_cuts[j + 1]),
                    h, es)

    def make(arena):
        ptrs = [arena.data_ptr() + p[3] * es for p in lay.parts]
        return costa.costa_layout_create(dtype, ranks, row_cuts, col_cuts, owners, ptrs, [p[4] for p in lay.parts],
                                         [0] * len(lay.parts))

    lay.make = make
    return lay


def _unequal_cuts(extent, blocks):
    r = random.Random(extent)
    weights = [r.uniform(0.5, 1.7) for _ in range(blocks)]
    return [round(extent * sum(weights[:k]) / sum(weights)) for k in range(blocks + 1)]


def _pair(case):
    """(target, source) layouts of one pair."""
    m, n, dt = case["m"], case["n"], case["dtype"]
    bm, bn = (m, n) if case["op"] == "N" else (n, m)
    src = _cyclic(bm, bn, case["b_mb"], case["b_nb"], case["b_pr"], case["b_pc"], case["b_pad"], False, dt)
    ranks = case["a_pr"] * case["a_pc"]
    if case["target"] == "irregular":
        order = _permutation(64)
        tgt = _blocked(_unequal_cuts(m, 8), _unequal_cuts(n, 8), [order[8 * i:8 * i + 8] for i in range(8)], 64, dt)
    elif case["target"] == "panels":
        tgt = _blocked([m * k // ranks for k in range(ranks + 1)], [0, n], [[k] for k in range(ranks)], ranks, dt)
    else:
        tgt = _cyclic(m, n, case["a_mb"], case["a_nb"], case["a_pr"], case["a_pc"], case["a_pad"], case["perm"], dt)
    return tgt, src


def _batch(case):
    """The pairs of a batch, each a case of its own."""
    r, sizes = random.Random(4), (16, 32, 64, 128)
    pairs = []
    for k in range(case["count"]):
        bs = [r.choice(sizes) for _ in range(4)]
        op = "N" if k % 2 == 0 else "T"
        m, n = (case["m"], case["n"]) if op == "N" else (case["n"], case["m"])
        pairs.append({**case, "op": op, "m": m, "n": n, "b_mb": bs[0], "b_nb": bs[1], "a_mb": bs[2], "a_nb": bs[3]})
    return pairs


def _alpha_beta(case):
    a, b = complex(case["alpha_re"], case["alpha_im"]), complex(case["beta_re"], case["beta_im"])
    return (a, b) if case["dtype"][0] == "c" else (a.real, b.real)


def _values(shape, dtype, seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * seed + stream)
    return torch.randn(shape, generator=g, device=DEV, dtype=TYPES[dtype])


def _inputs(case, tgt, src, seed, k=0):
    """Global (A, B); A is None when it is not read (its storage is then zero)."""
    A = _values((tgt.m, tgt.n), case["dtype"], seed, 2 * k) if _alpha_beta(case)[1] != 0 else None
    return A, _values((src.m, src.n), case["dtype"], seed, 2 * k + 1)


def _arenas(case, tgt, src, A, B):
    a = torch.zeros(tgt.size, dtype=TYPES[case["dtype"]], device=DEV)
    b = torch.zeros(src.size, dtype=TYPES[case["dtype"]], device=DEV)
    if A is not None:
        tgt.put(a, A)
    return a, src.put(b, B)


# ---- ScaLAPACK submatrices ----

def _sl_side(m, n, mb, nb, pr, pc, pad, first, dtype):
    """The whole matrix that holds an m x n submatrix at (first, first), some more rows and columns behind it."""
    return _cyclic(m + first + 17, n + first + 17, mb, nb, pr, pc, pad, False, dtype)


def _sl_pair(case):
    m, n = case["m"], case["n"]
    bm, bn = (m, n) if case["op"] == "N" else (n, m)
    dt = case["dtype"]
    src = _sl_side(bm, bn, case["b_mb"], case["b_nb"], case["b_pr"], case["b_pc"], case["b_pad"], case["bi"], dt)
    tgt = _sl_side(m, n, case["a_mb"], case["a_nb"], case["a_pr"], case["a_pc"], case["a_pad"], case["ai"], dt)
    return tgt, src, bm, bn


# ---- the interface ----

def prepare(case, seed):
    case = {**DEFAULT, **case}
    alpha, beta = _alpha_beta(case)
    state = {"case": case, "alpha": alpha, "beta": beta}
    if case["api"] == "batched":
        state.update(LA=[], LB=[], ops=[], a=[], b=[])
        pairs = _batch(case)
        for k, c in enumerate(pairs):
            tgt, src = _pair(c)
            a, b = _arenas(c, tgt, src, *_inputs(c, tgt, src, seed, k))
            state["a"].append(a)
            state["b"].append(b)
            state["LA"].append(tgt.make(a))
            state["LB"].append(src.make(b))
            state["ops"].append(c["op"])
        state["alphas"], state["betas"] = [alpha] * len(pairs), [beta] * len(pairs)
        costa.costa_plan_stats_get(state["LA"], state["LB"], state["ops"], case["relabel"],
                                   torch.cuda.current_stream().cuda_stream)
        state["out"] = state["a"]
        return state
    if case["api"] == "scalapack":
        tgt, src, bm, bn = _sl_pair(case)
        a, b = _arenas(case, tgt, src, *_inputs(case, tgt, src, seed))
        for side, lay, arena in (("a", tgt, a), ("b", src, b)):
            pr, pc = case[side + "_pr"], case[side + "_pc"]
            es = SIZE[case["dtype"]]
            state["grid_" + side] = costa.BlacsGrid(pr, pc, "R", [arena.data_ptr() + p[3] * es for p in lay.parts],
                                                    [p[4] for p in lay.parts])
            state["desc_" + side] = [1, 0, lay.m, lay.n, case[side + "_mb"], case[side + "_nb"], 0, 0,
                                     max(p[4] for p in lay.parts)]
        state.update(a=a, b=b, out=a)
        return state
    tgt, src = _pair(case)
    a, b = _arenas(case, tgt, src, *_inputs(case, tgt, src, seed))
    state.update(a=a, b=b, LA=tgt.make(a), LB=src.make(b), out=a)
    stream = torch.cuda.current_stream().cuda_stream
    if case["api"] == "transform":
        costa.costa_plan_stats_get(state["LA"], state["LB"], case["op"], case["relabel"], stream)
        return state
    # exchange: what the other processes send to process 0 arrives in its receive buffer beforehand
    G, ranks = case["gpus"], case["a_pr"] * case["a_pc"]
    place = [r * G // ranks for r in range(ranks)]
    byte = lambda size: torch.zeros(max(16, int(size)), dtype=torch.uint8, device=DEV)  # noqa: E731
    LA, LB, op = state["LA"], state["LB"], case["op"]
    sb, rb = costa.costa_exchange_sizes(LA, LB, op, G, place, 0)
    send, recv = byte(sb.sum()), byte(rb.sum())
    for g in range(1, G):
        s, r = costa.costa_exchange_sizes(LA, LB, op, G, place, g)
        buf, other = byte(s.sum()), byte(r.sum())
        x = costa.Exchange(LA, LB, op, G, place, g, buf.data_ptr(), other.data_ptr())
        x.pack(stream)
        at = int(rb[:g].sum())
        recv[at:at + int(s[0])].copy_(buf[:int(s[0])])
        torch.cuda.synchronize()
        x.destroy()
    state.update(send=send, recv=recv, place=place,
                 exchange=costa.Exchange(LA, LB, op, G, place, 0, send.data_ptr(), recv.data_ptr()))
    real = torch.float32 if case["dtype"] in ("f32", "c64") else torch.float64
    state["out"] = {"A": a, "send": send.view(real)}
    return state


def run(state):
    case, stream = state["case"], torch.cuda.current_stream().cuda_stream
    alpha, beta, api = state["alpha"], state["beta"], case["api"]
    if api == "transform":
        costa.costa_transform(state["LA"], state["LB"], case["op"], alpha, beta, relabel=case["relabel"],
                              stream=stream)
    elif api == "batched":
        costa.costa_transform_batched(state["LA"], state["LB"], state["ops"], state["alphas"], state["betas"],
                                      relabel=case["relabel"], stream=stream)
    elif api == "exchange":
        x = state["exchange"]
        x.pack(stream)
        x.local(alpha, beta, stream)
        x.unpack(alpha, beta, stream)
    elif case["op"] == "N":
        costa.costa_pxgemr2d(case["dtype"], case["m"], case["n"], state["grid_b"], case["bi"], case["bi"],
                             state["desc_b"], state["grid_a"], case["ai"], case["ai"], state["desc_a"], stream)
    else:
        costa.costa_pxtran(case["dtype"], case["m"], case["n"], alpha, state["grid_b"], case["bi"], case["bi"],
                           state["desc_b"], beta, state["grid_a"], case["ai"], case["ai"], state["desc_a"],
                           conjugate=case["op"] == "C", stream=stream)
    return state["out"]


def _shares(case):
    """Elements of process 0's exchange: (sent, kept, received)."""
    tgt, src = _pair(case)
    G, ranks = case["gpus"], case["a_pr"] * case["a_pc"]
    rows_b, cols_b = (src.row_proc, src.col_proc) if case["op"] == "N" else (src.col_proc, src.row_proc)
    pr, pc = case["b_pr"], case["b_pc"]
    # rows and columns of A by (target process, source process) of their axis
    nr = np.zeros((case["a_pr"], max(pr, pc)), np.int64)
    nc = np.zeros((case["a_pc"], max(pr, pc)), np.int64)
    np.add.at(nr, (tgt.row_proc, rows_b), 1)
    np.add.at(nc, (tgt.col_proc, cols_b), 1)
    sent = kept = received = 0
    for ai in range(case["a_pr"]):
        for aj in range(case["a_pc"]):
            to = tgt.owners[ai * case["a_pc"] + aj] * G // ranks
            for i in range(pr):
                for j in range(pc):
                    x, y = (i, j) if case["op"] == "N" else (j, i)
                    v = int(nr[ai, x] * nc[aj, y])
                    frm = src.owners[i * pc + j] * G // ranks
                    sent += v if frm == 0 and to != 0 else 0
                    kept += v if frm == 0 and to == 0 else 0
                    received += v if frm != 0 and to == 0 else 0
    return sent, kept, received


def work(case):
    case = {**DEFAULT, **case}
    alpha, beta = _alpha_beta(case)
    es, streams = SIZE[case["dtype"]], 2 if beta == 0 else 3  # B read, A written, and read when beta != 0
    if case["api"] == "exchange":
        sent, kept, received = _shares(case)
        moved, used = es * (2 * sent + streams * (kept + received)), kept + received
    else:
        used = case["count"] * case["m"] * case["n"]
        moved = es * streams * used
    cplx = case["dtype"][0] == "c"
    flops = 0
    if beta != 0 or alpha != 1:
        per = (0 if alpha == 1 else 1) + (0 if beta == 0 else 2)
        if cplx:
            per = 2 * per if alpha == complex(alpha).real and beta == complex(beta).real else 6 + (0 if beta == 0 else 8)
        flops = per * used
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    case = {**DEFAULT, **case}
    alpha, beta = _alpha_beta(case)
    if alpha == 1 and beta == 0:
        return "exact"  # a copy
    # products and a sum per element, each rounded to the type: 5e-17 (double) and 3e-8 (single) off the 64-bit
    # result as measured
    return {"rel": 1.2e-7 if case["dtype"] in ("f32", "c64") else 2.4e-16}


def exact(case, seed):
    case = {**DEFAULT, **case}
    alpha, beta = _alpha_beta(case)
    wide = "c128" if case["dtype"][0] == "c" else "f64"

    def op(x, name):
        return x if name == "N" else x.T if name == "T" else x.T.conj()

    def combine(c, A, B):
        out = (op(B, c["op"]) * alpha) if alpha != 1 else op(B, c["op"])
        return out if A is None else out + beta * A

    def one(c, tgt, src, k=0):
        A, B = (x if x is None else x.to(TYPES[wide]) for x in _inputs(c, tgt, src, seed, k))
        arena = torch.zeros(tgt.size, dtype=TYPES[wide], device=DEV)
        if c["api"] == "exchange":
            if A is not None:
                tgt.put(arena, A)
            G, ranks = c["gpus"], c["a_pr"] * c["a_pc"]
            mine = [r for r in range(ranks) if r * G // ranks == 0]
            return {"A": tgt.put(arena, combine(c, A, B), mine), "send": None}
        return tgt.put(arena, combine(c, A, B))

    if case["api"] == "batched":
        return [one(c, *_pair(c), k) for k, c in enumerate(_batch(case))]
    if case["api"] == "scalapack":
        tgt, src, bm, bn = _sl_pair(case)
        A, B = (x if x is None else x.to(TYPES[wide]) for x in _inputs(case, tgt, src, seed))
        i, j, m, n = case["ai"] - 1, case["bi"] - 1, case["m"], case["n"]
        full = torch.zeros((tgt.m, tgt.n), dtype=TYPES[wide], device=DEV) if A is None else A.clone()
        full[i:i + m, i:i + n] = combine(case, None if A is None else A[i:i + m, i:i + n], B[j:j + bm, j:j + bn])
        return tgt.put(torch.zeros(tgt.size, dtype=TYPES[wide], device=DEV), full)
    return one(case, *_pair(case))
