// Patches: the work list of the patch kernel, for problems whose grid-overlay
// cells are small or whose runs start off 16-byte boundaries.  Host code only.
//
// A tile lies inside one cell of the grid overlay (Sec. 5), so small blocks
// or two block sizes that do not divide each other cut the tiles small.  But
// the blocks of one rank are usually neighbours in its local matrix (a
// block-cyclic rank stores block rows i, i + pr, i + 2 pr, ... one below the
// other), so a window of A's *storage* covers many cells.  A patch is such a
// window of at most patch_x x patch_y elements: affine in A, and
// in B a product of segments (at most kPatchSegs per axis), each segment
// pair one cell with its own source address and stride.
#include <climits>
#include <unordered_map>

#include "tiles.h"

namespace costa {

namespace {

// Chains of one axis of a layout: blocks that continue each other in storage
// for every block of the other axis, so that an index into the chain is
// affine in storage.  chain[b]: id; pos[b]: the block's start in its chain.
struct AxisMap {
    std::vector<int32_t> chain;
    std::vector<int64_t> pos;
};

AxisMap axis_map(const costa_layout_s *L, int axis) {
    const int n = axis == 0 ? L->nbr : L->nbc, other = axis == 0 ? L->nbc : L->nbr;
    const std::vector<int64_t> &S = axis == 0 ? L->R : L->C, &O = axis == 0 ? L->C : L->R;
    const int64_t es = esize_of(L->dt);
    auto blk = [&](int i, int k) -> const DevBlock & {
        return L->blocks[axis == 0 ? static_cast<size_t>(i) * L->nbc + k : static_cast<size_t>(k) * L->nbc + i];
    };
    auto step = [&](const DevBlock &b) -> int64_t {
        return (b.order == COSTA_COL_MAJOR) == (axis == 0) ? 1 : b.ld;
    };
    auto follows = [&](const DevBlock &a, const DevBlock &b, int64_t len) {
        return b.ptr == a.ptr + static_cast<uint64_t>(len * step(a) * es) && b.ld == a.ld && b.order == a.order;
    };
    AxisMap m;
    m.chain.assign(static_cast<size_t>(n), -1);
    m.pos.assign(static_cast<size_t>(n), 0);
    int k0 = 0;
    while (k0 < other && O[k0 + 1] == O[k0]) ++k0;
    if (k0 == other) return m;
    std::unordered_map<uint64_t, int> at;
    at.reserve(static_cast<size_t>(n) * 2);
    for (int i = 0; i < n; ++i)
        if (S[i + 1] > S[i]) at.emplace(blk(i, k0).ptr, i);
    std::vector<int> next(static_cast<size_t>(n), -1);
    for (int i = 0; i < n; ++i) {
        if (S[i + 1] == S[i]) continue;
        const DevBlock &b = blk(i, k0);
        auto it = at.find(b.ptr + static_cast<uint64_t>((S[i + 1] - S[i]) * step(b) * es));
        if (it != at.end() && it->second != i && follows(b, blk(it->second, k0), S[i + 1] - S[i])) next[i] = it->second;
    }
    // the neighbours must continue each other for every block of the other axis
    if (axis == 0) {
        for (int i = 0; i < n; ++i)
            for (int k = 0; k < other && next[i] >= 0; ++k)
                if (O[k + 1] > O[k] && !follows(blk(i, k), blk(next[i], k), S[i + 1] - S[i])) next[i] = -1;
    } else {
        for (int k = 0; k < other; ++k) {
            if (O[k + 1] == O[k]) continue;
            for (int i = 0; i < n; ++i)
                if (next[i] >= 0 && !follows(blk(i, k), blk(next[i], k), S[i + 1] - S[i])) next[i] = -1;
        }
    }
    std::vector<char> has_prev(static_cast<size_t>(n), 0);
    for (int i = 0; i < n; ++i)
        if (next[i] >= 0) {
            if (has_prev[next[i]]) next[i] = -1;  // not expected: two blocks at one address
            else has_prev[next[i]] = 1;
        }
    int id = 0;
    for (int i = 0; i < n; ++i) {
        if (S[i + 1] == S[i] || has_prev[i]) continue;
        int64_t p = 0;
        for (int j = i; j >= 0; j = next[j]) {
            m.chain[j] = id;
            m.pos[j] = p;
            p += S[j + 1] - S[j];
        }
        ++id;
    }
    return m;
}

struct Seg {  // a run of one axis that is affine in A's and in op(B)'s storage
    int32_t a_chain, b_chain;
    int64_t a_pos, b_pos, len;
    int32_t a_blk, b_blk;
    int64_t a_off, b_off;
};

struct PatchSeg {  // one segment of a patch along one axis
    int32_t b_blk;
    int32_t start;  // within the patch
    int64_t b_off;
};

struct AxisPatch {
    int32_t a_blk;
    int64_t a_off;
    int32_t len, nseg;
    uint32_t mask;
    size_t seg0;
};

struct AxisPatches {
    std::vector<AxisPatch> patches;
    std::vector<PatchSeg> segs;
    std::vector<size_t> chain0;     // first patch of each chain of A, then the number of patches
    std::vector<int64_t> nseg_sum;  // prefix sums of nseg
    int64_t shared = 0;             // ends of segments whose neighbour in B's storage is in another chain of A
    int64_t extent = 0;
};

// Cuts one axis of A's storage into patches of at most `ext` elements and
// kPatchSegs segments, ends preferably at multiples of `unit` (elements)
// from address phase `phase[chain]`.
AxisPatches cut_patches(const costa_layout_s *A, const costa_layout_s *B, costa_op op, int axis, int ext, int unit) {
    const bool tr = op != COSTA_OP_N;
    const AxisMap ma = axis_map(A, axis), mb = axis_map(B, tr ? 1 - axis : axis);
    const std::vector<int64_t> &SA = axis == 0 ? A->R : A->C;
    const std::vector<int64_t> &SB = (axis == 0) != tr ? B->R : B->C;
    const AxisCut cut = cut_axis(SA, SB, axis == 0 ? A->m : A->n, INT_MAX, 1, true);
    std::vector<Seg> segs;
    segs.reserve(cut.tiles.size());
    bool sorted = true;
    for (const AxisTile &t : cut.tiles) {
        Seg s;
        s.a_blk = t.a_blk;
        s.b_blk = t.b_blk;
        s.a_off = t.a_off;
        s.b_off = t.b_off;
        s.len = t.len;
        s.a_chain = ma.chain[t.a_blk];
        s.b_chain = mb.chain[t.b_blk];
        s.a_pos = ma.pos[t.a_blk] + t.a_off;
        s.b_pos = mb.pos[t.b_blk] + t.b_off;
        segs.push_back(s);
    }
    auto before = [](const Seg &x, const Seg &y) {
        return x.a_chain != y.a_chain ? x.a_chain < y.a_chain : x.a_pos < y.a_pos;
    };
    for (size_t i = 1; i < segs.size() && sorted; ++i) sorted = before(segs[i - 1], segs[i]);
    if (!sorted) std::sort(segs.begin(), segs.end(), before);
    // neighbours in A that are neighbours in B too are one segment
    size_t w = 0;
    for (size_t i = 0; i < segs.size(); ++i) {
        if (w > 0) {
            Seg &p = segs[w - 1];
            const Seg &s = segs[i];
            if (p.a_chain == s.a_chain && p.b_chain == s.b_chain && p.a_pos + p.len == s.a_pos &&
                p.b_pos + p.len == s.b_pos) {
                p.len += s.len;
                continue;
            }
        }
        segs[w++] = segs[i];
    }
    segs.resize(w);
    const int es = esize_of(A->dt);
    AxisPatches out;
    out.extent = axis == 0 ? A->m : A->n;
    {
        // B's line (128 bytes) at such an end is read by patches of two chains
        std::vector<uint32_t> by_b(segs.size());
        for (size_t k = 0; k < segs.size(); ++k) by_b[k] = static_cast<uint32_t>(k);
        std::sort(by_b.begin(), by_b.end(), [&](uint32_t x, uint32_t y) {
            return segs[x].b_chain != segs[y].b_chain ? segs[x].b_chain < segs[y].b_chain : segs[x].b_pos < segs[y].b_pos;
        });
        const bool b_rows = (axis == 0) != tr;
        for (size_t k = 1; k < by_b.size(); ++k) {
            const Seg &p = segs[by_b[k - 1]], &s = segs[by_b[k]];
            if (p.b_chain != s.b_chain || p.a_chain == s.a_chain) continue;
            const DevBlock &b = b_rows ? B->blocks[static_cast<size_t>(s.b_blk) * B->nbc] : B->blocks[static_cast<size_t>(s.b_blk)];
            if (((b.ptr + static_cast<uint64_t>(s.b_off) * es) | (static_cast<uint64_t>(b.ld) * es)) % 128) ++out.shared;
        }
    }
    size_t i = 0;
    while (i < segs.size()) {
        const int32_t chain = segs[i].a_chain;
        out.chain0.push_back(out.patches.size());
        const DevBlock &first = axis == 0 ? A->blocks[static_cast<size_t>(segs[i].a_blk) * A->nbc]
                                          : A->blocks[static_cast<size_t>(segs[i].a_blk)];
        int64_t pos = 0, used = 0;  // position in the chain; elements of segs[i] already taken
        const int64_t phase = static_cast<int64_t>(first.ptr / static_cast<uint64_t>(es) % static_cast<uint64_t>(unit));
        while (i < segs.size() && segs[i].a_chain == chain) {
            AxisPatch p;
            p.a_blk = segs[i].a_blk;
            p.a_off = segs[i].a_off + used;
            p.seg0 = out.segs.size();
            p.len = 0;
            p.nseg = 0;
            p.mask = 0;
            const int want = ext - static_cast<int>((pos + phase) % unit);
            while (p.len < want && p.nseg < kPatchSegs && i < segs.size() && segs[i].a_chain == chain) {
                const int64_t take = std::min<int64_t>(want - p.len, segs[i].len - used);
                out.segs.push_back({segs[i].b_blk, p.len, segs[i].b_off + used});
                p.mask |= 1u << p.len;
                ++p.nseg;
                p.len += static_cast<int32_t>(take);
                used += take;
                if (used == segs[i].len) {
                    ++i;
                    used = 0;
                }
            }
            pos += p.len;
            out.patches.push_back(p);
        }
    }
    out.chain0.push_back(out.patches.size());
    out.nseg_sum.assign(out.patches.size() + 1, 0);
    for (size_t k = 0; k < out.patches.size(); ++k) out.nseg_sum[k + 1] = out.nseg_sum[k] + out.patches[k].nseg;
    return out;
}

// Whether every nonempty block of a layout has one element order.
bool one_order(const costa_layout_s *L, int &order) {
    bool any = false;
    for (int i = 0; i < L->nbr; ++i) {
        if (L->R[i + 1] == L->R[i]) continue;
        for (int j = 0; j < L->nbc; ++j) {
            if (L->C[j + 1] == L->C[j]) continue;
            const int o = L->blocks[static_cast<size_t>(i) * L->nbc + j].order;
            if (any && o != order) return false;
            order = o;
            any = true;
        }
    }
    return any;
}

// Whether at least half of a layout's elements lie in blocks whose leading
// dimension is a multiple of `step`.
bool mostly_ld_multiple(const costa_layout_s *L, int step) {
    int64_t sum = 0;
    for (int i = 0; i < L->nbr; ++i)
        for (int j = 0; j < L->nbc; ++j)
            if (L->blocks[static_cast<size_t>(i) * L->nbc + j].ld % step == 0)
                sum += (L->R[i + 1] - L->R[i]) * (L->C[j + 1] - L->C[j]);
    return 2 * sum >= L->m * L->n;
}

}  // namespace

bool append_patches(const ProblemHost &ph, int prob, int64_t total, int64_t most, PatchList &out) {
    const costa_layout_s *A = ph.A, *B = ph.B;
    int oa = 0, ob = 0;
    if (!one_order(A, oa) || !one_order(B, ob)) return false;
    const int es = esize_of(A->dt);
    const bool op_tr = ph.op != COSTA_OP_N;
    const bool a_col = oa == COSTA_COL_MAJOR, b_col = ob == COSTA_COL_MAJOR;
    const bool transpose = a_col != (op_tr ? !b_col : b_col);
    int ex = patch_x(es), ey = patch_y(es);
    // Few patches: smaller ones, with fewer passes along the run axis (and, for
    // very few 8-byte ones, shorter runs), so that more warps share the work.
    // us per call on GB300, whole / half / quarter patches:
    //   f64 BC8 T beta = 0.5    512^2 5.2 / 3.7 / 3.5, 768^2 5.3 / 4.1 / 4.3,
    //                           1024^2 5.8 / 5.2 / 6.7, 1536^2 12.3 / 13.2
    //   f32 BC8 T beta = 0.5    512^2 3.1 / 2.8 / 3.1, 768^2 3.2 / 3.0 / 3.8,
    //                           1024^2 3.6 / 3.8
    //   c128 BC8 T beta = 0.5   256^2 3.6 / 3.0, 512^2 4.0 / 3.9, 768^2 5.4 / 6.1
    int &run_ext = transpose ? ex : ey;
    const int64_t half_below = es == 16 ? 300000 : es == 8 ? 1200000 : 700000;
    if (total < half_below) run_ext /= 2;
    if (es == 8 && total < 350000) (transpose ? ey : ex) /= 2;
    const int unit = std::max(1, std::min(ex, 128 / es));
    const AxisPatches rows = cut_patches(A, B, ph.op, 0, a_col ? ex : ey, a_col ? unit : 1);
    const AxisPatches cols = cut_patches(A, B, ph.op, 1, a_col ? ey : ex, a_col ? 1 : unit);
    const AxisPatches &X = a_col ? rows : cols, &Y = a_col ? cols : rows;
    const int64_t ncells = rows.nseg_sum.back() * cols.nseg_sum.back();
    const int64_t npatches = static_cast<int64_t>(X.patches.size()) * static_cast<int64_t>(Y.patches.size());
    if (npatches > most || static_cast<int64_t>(out.cells.size()) + ncells >= (int64_t(1) << 32)) return false;
    // Order: per pair of chains (a rank's local matrix) A's storage order, x
    // fastest, so that the patches in flight together form long runs of A.
    struct Row {
        size_t x0, x1, y;
        int64_t patch0, cell0;
    };
    std::vector<Row> work;
    int64_t patch0 = static_cast<int64_t>(out.patches.size()), cell0 = static_cast<int64_t>(out.cells.size());
    // Unless the source's runs are cut often by blocks of A of different
    // chains: then two rows of patches of every chain follow each other, so
    // that a line of B that patches of two chains read in part is read from
    // DRAM once (BC50 -> BC75 f64 T copy: 754 -> 551 MB read for 537 MB of B).
    // The line lies at one such end per 350 bytes (transposed) or 1 KB (op's
    // runs along A's).  us per call on GB300, 8192^2, in order / mixed:
    //   f64 T  BC50 -> BC75 (300 B per end) 225 / 175, odd lds (512 B) 191 /
    //          188 (beta = 0.5: 267 / 269), B's ld odd 197 / 201
    //   f64 N  BC50 -> BC75 193 / 172, odd lds 183 / 170, BC64 -> BC8 255 /
    //          168, BC37 -> BC128 216 / 169
    //   f32    BC50 -> BC75 T 123 / 108, N 111 / 107, odd lds T 110 / 117, N
    //          114 / 108, BC64 -> BC8 N 197 / 100
    //   c128   BC50 -> BC75 T 190 / 196, N 194 / 188
    // and not for a transposed source whose columns lie (mostly) a multiple of 1 KB
    // apart, where fewer rows in flight crowd the same channels: f32 T BC64 ->
    // BC8 131 / 198, BC8 -> BC64 106 / 130, BC16 -> BC48 beta = 0.5 153 / 172.
    const AxisPatches &lane_axis = transpose ? Y : X;
    size_t longest = 0;
    for (size_t cy = 0; cy + 1 < Y.chain0.size(); ++cy) longest = std::max(longest, Y.chain0[cy + 1] - Y.chain0[cy]);
    const bool mix = lane_axis.shared * (transpose ? 350 : 1024) > lane_axis.extent * es &&
                     !(transpose && mostly_ld_multiple(B, 1024 / es));
    const size_t chunk = mix ? 2 : longest;
    std::vector<size_t> live(Y.chain0.size() - 1);  // the chains with rows left, so that the work is one step per row
    for (size_t cy = 0; cy < live.size(); ++cy) live[cy] = cy;
    for (size_t k0 = 0; !live.empty(); k0 += chunk) {
        size_t left = 0;
        for (const size_t cy : live) {
            const size_t y0 = Y.chain0[cy] + k0, y1 = std::min(y0 + chunk, Y.chain0[cy + 1]);
            for (size_t cx = 0; cx + 1 < X.chain0.size(); ++cx)
                for (size_t y = y0; y < y1; ++y) {
                    const size_t x0 = X.chain0[cx], x1 = X.chain0[cx + 1];
                    work.push_back({x0, x1, y, patch0, cell0});
                    patch0 += static_cast<int64_t>(x1 - x0);
                    cell0 += (X.nseg_sum[x1] - X.nseg_sum[x0]) * Y.patches[y].nseg;
                }
            if (y1 < Y.chain0[cy + 1]) live[left++] = cy;
        }
        live.resize(left);
    }
    out.patches.resize(out.patches.size() + static_cast<size_t>(npatches));
    out.cells.resize(out.cells.size() + static_cast<size_t>(ncells));
    const int64_t per_row = std::max<int64_t>(1, (npatches + ncells) / std::max<int64_t>(1, static_cast<int64_t>(work.size())));
    parallel_for(static_cast<int64_t>(work.size()), std::max<int64_t>(1, (1 << 14) / per_row), [&](int64_t w0, int64_t w1) {
        for (int64_t w = w0; w < w1; ++w) {
            const Row &row = work[static_cast<size_t>(w)];
            const AxisPatch &py = Y.patches[row.y];
            int64_t cell = row.cell0;
            for (size_t x = row.x0; x < row.x1; ++x) {
                const AxisPatch &px = X.patches[x];
                const AxisPatch &pr = a_col ? px : py, &pc = a_col ? py : px;  // rows and columns of A
                const DevBlock &da = A->blocks[static_cast<size_t>(pr.a_blk) * A->nbc + pc.a_blk];
                PatchDesc d;
                d.dst = da.ptr + static_cast<uint64_t>((px.a_off + py.a_off * da.ld) * es);
                d.dld = da.ld;
                d.cell0 = static_cast<uint32_t>(cell);
                d.lmask = transpose ? py.mask : px.mask;
                d.rmask = transpose ? px.mask : py.mask;
                d.nx = static_cast<uint8_t>(px.len);
                d.ny = static_cast<uint8_t>(py.len);
                d.prob = static_cast<uint16_t>(prob);
                d.flags = static_cast<uint16_t>((transpose ? TF_TRANSPOSE : 0) | (ph.op == COSTA_OP_C ? TF_CONJ : 0));
                d.pad = 0;
                const AxisPatch &run = transpose ? px : py, &lane = transpose ? py : px;
                // 4-byte elements: source runs of whole aligned 16-byte chunks, and
                // one row of A per pass
                bool chunks = es == 4 && d.nx > 16 && lane.len % 4 == 0 && (lane.mask & 0xEEEEEEEEu) == 0;
                const std::vector<PatchSeg> &rs = transpose ? X.segs : Y.segs, &ls = transpose ? Y.segs : X.segs;
                for (int r = 0; r < run.nseg; ++r)
                    for (int l = 0; l < lane.nseg; ++l) {
                        const PatchSeg &sr = rs[run.seg0 + r], &sl = ls[lane.seg0 + l];
                        const PatchSeg &sx = transpose ? sr : sl, &sy = transpose ? sl : sr;
                        const PatchSeg &row_seg = a_col ? sx : sy, &col_seg = a_col ? sy : sx;
                        // op(B)'s rows are B's columns when op transposes
                        const PatchSeg &br = op_tr ? col_seg : row_seg, &bc = op_tr ? row_seg : col_seg;
                        const DevBlock &db = B->blocks[static_cast<size_t>(br.b_blk) * B->nbc + bc.b_blk];
                        const int64_t off = b_col ? br.b_off + bc.b_off * db.ld : br.b_off * db.ld + bc.b_off;
                        PatchCell c;
                        // biased, so that element (r, l) of the patch is at src + r * sld + l
                        c.src = db.ptr + static_cast<uint64_t>((off - sr.start * static_cast<int64_t>(db.ld) - sl.start) * es);
                        c.sld = db.ld;
                        c.pad = 0;
                        chunks = chunks && c.src % 16 == 0 && db.ld % 4 == 0;
                        out.cells[static_cast<size_t>(cell++)] = c;
                    }
                if (chunks) d.flags = static_cast<uint16_t>(d.flags | TF_FAST);
                out.patches[static_cast<size_t>(row.patch0) + (x - row.x0)] = d;
            }
        }
    });
    return true;
}

}  // namespace costa
