// The patch kernel of the reshuffle (combine kinds, staging and launch idiom
// as in remap_impl.cuh): it moves pairs whose grid-overlay cells are mostly
// small or whose runs start off 16-byte boundaries, and large lists of 4- and
// 8-byte elements (take_patches in costa.cpp has the rule).
//
// What bounds the tile kernel there: a tile lies in one overlay cell, so
// small or odd cells leave lanes idle, bytes out of flight and a descriptor
// per few hundred bytes.  A patch (patches.cpp) is a window of A's storage
// instead, over as many cells as it takes: 32 x 32 elements (16 x 16 of 16
// bytes; a half or a quarter of that in small problems; less at the ends of a
// rank's local matrix and where more than 8 segments meet along an axis), its
// writes whole runs of A whatever the blocks.  One warp moves one patch:
//   1. the patch's cells (source address and stride of each segment pair,
//      loaded one patch ahead) go to shared memory;
//   2. the source is copied one element per lane (cp.async at the element's
//      own alignment, so any phase is the same case), lanes along the
//      source's contiguous axis, one run per step of the other axis; a lane
//      reads its cell's address when a segment starts and adds the stride
//      after that (4-byte runs of whole aligned 16-byte chunks: by chunks);
//   3. the warp writes A one run per step, one element per lane, reading the
//      staged rows across (transposed) or along; an odd row pitch keeps both
//      free of bank conflicts and the addresses free of swizzles.
// Kinds that read A load two groups of G passes of A's elements before the
// wait and the next group after each one is used.
//
// Element-wide copies in flight occupy L1 lines (only 16-byte cp.async
// bypasses L1), so the launch leaves the L1 its share of the SM's 256 KB: with
// shared memory sized for the most blocks that fit, f64 BC8 T copy runs at
// 190 us, with 3 blocks and 124 KB of L1 at 161 (8192^2; 6660 GB/s).
#pragma once

#include "remap_impl.cuh"
#include "rnmul.h"

namespace costa {
namespace remap {

// Launch shape: 4 warps per block, the resident blocks per SM (also the
// shared memory that is carved out), one buffer per warp (a second one lost
// 1-20% on every case: its bytes come off the L1).  us per call on GB300,
// 8192^2 (c128 6016^2) T, by blocks per SM:
//              2     3     4     5     6
//   f64 copy  175   161   171   167   190   (BC8)
//   f64 b=0.5 327   262   242   243   393   (BC8)
//   f64 scale  -    211   206   218    -    (BC50 -> BC75)
//   f32 copy   -     -     89    84    91   (BC8)
//   f32 b=0.5 177   149   130   197    -    (BC8)
//   c128 copy 248   200   179   178   192   (BC8)
//   c128 b=.5 400   307   267   269   470   (BC8)
#ifndef COSTA_PW
#define COSTA_PW 4
#endif
#ifndef COSTA_PB_4
#define COSTA_PB_4 5
#endif
#ifndef COSTA_PB_4A
#define COSTA_PB_4A 4
#endif
#ifndef COSTA_PB_8
#define COSTA_PB_8 3
#endif
#ifndef COSTA_PB_8S
#define COSTA_PB_8S 4
#endif
#ifndef COSTA_PB_8A
#define COSTA_PB_8A 4
#endif
// complex scalars on double complex data
#ifndef COSTA_PB_16C
#define COSTA_PB_16C 4
#endif
#ifndef COSTA_PGR
#define COSTA_PGR 2
#endif
#ifndef COSTA_PB_16
#define COSTA_PB_16 4
#endif

constexpr int patch_blocks(int es, bool cplx, int kind) {
    const bool reads_a = kind_reads_a(kind);
    if (es == 4) return reads_a ? COSTA_PB_4A : COSTA_PB_4;
    if (es == 16) return kind_cplx(kind) || kind == K_CSCALE ? COSTA_PB_16C : COSTA_PB_16;
    return reads_a ? COSTA_PB_8A : kind == K_SCALE && !cplx ? COSTA_PB_8S : COSTA_PB_8;
}

template <typename T, int KIND> struct PCfg {
    static constexpr int ES = static_cast<int>(sizeof(T));
    static constexpr int EX = patch_x(ES), EY = patch_y(ES);
    // staged rows, one run of the source each: an odd pitch, so that lanes
    // reading one position of consecutive rows hit distinct banks
    static constexpr int PITCH_T = EY + 1, PITCH_N = ES == 4 ? EX + 4 : EX + 1;
    static constexpr int WARPS = COSTA_PW;
    static constexpr bool READS_A = kind_reads_a(KIND);
    // real doubles: part of the products beta * a and alpha * b are formed on
    // the integer pipes (mul_group)
    static constexpr bool INT_MUL = sizeof(T) == 8 && !ET<T>::CPLX;
    static constexpr int MINB = patch_blocks(ES, ET<T>::CPLX != 0, KIND);
    // 4-byte elements: patches with TF_FAST stage whole 16-byte chunks (N: the
    // pitch is whole chunks; T: rows of 128 bytes, chunk_slot)
    static constexpr bool CHUNKED = ES == 4;
    static constexpr int ELEMS = EX * PITCH_T > EY * PITCH_N ? EX * PITCH_T : EY * PITCH_N;
    static constexpr int BUF = (ELEMS * ES + 15) / 16 * 16;
    static constexpr int CELLS = kPatchCells * 16;
    // complex scalars on double complex data: two passes together, rolled (the
    // fixed-point sums are long; BC50 -> BC75, 4096^2, complex beta, one, two,
    // four passes: 306, 276, 322 us)
    static constexpr bool ROLLED = ES == 16 && (kind_cplx(KIND) || KIND == K_CSCALE);
    // passes whose elements of A are loaded together: the whole patch in two
    // groups, a quarter for 8-byte elements (registers)
    static constexpr int G = ROLLED ? COSTA_PGR : ES == 4 ? 16 : ES == 8 ? 8 : 4;
};

// Index of the segment that holds element i of an axis (mask: bit k set
// where a segment starts at element k; bit 0 always).
__device__ __forceinline__ int seg_of(uint32_t mask, int i) { return __popc(mask & ((2u << i) - 1u)) - 1; }

struct PatchRaw {
    uint4 lo, hi;
};
__device__ __forceinline__ PatchDesc unpack_patch(const PatchRaw &r) {
    PatchDesc d;
    d.dst = (static_cast<uint64_t>(r.lo.y) << 32) | r.lo.x;
    d.dld = static_cast<int32_t>(r.lo.z);
    d.cell0 = r.lo.w;
    d.lmask = r.hi.x;
    d.rmask = r.hi.y;
    d.nx = static_cast<uint8_t>(r.hi.z & 0xFFu);
    d.ny = static_cast<uint8_t>((r.hi.z >> 8) & 0xFFu);
    d.prob = static_cast<uint16_t>(r.hi.z >> 16);
    d.flags = static_cast<uint16_t>(r.hi.w & 0xFFFFu);
    d.pad = 0;
    return d;
}
// Patch t, the same for every lane (one broadcast load per half).
__device__ __forceinline__ PatchRaw load_patch(const PatchLaunch &a, int64_t t) {
    PatchRaw r;
    const uint4 *p = reinterpret_cast<const uint4 *>(a.patches + t);
    r.lo = __ldg(p);
    r.hi = __ldg(p + 1);
    return r;
}

// The cells of a patch, two per lane.
struct CellRegs {
    uint4 a, b;
};
__device__ __forceinline__ CellRegs load_cells(const PatchLaunch &a, const PatchDesc &d, int lane) {
    CellRegs c;
    const int n = min(__popc(d.lmask) * __popc(d.rmask), kPatchCells);
    const uint4 *p = reinterpret_cast<const uint4 *>(a.cells + d.cell0);
    c.a = make_uint4(0, 0, 0, 0);
    c.b = make_uint4(0, 0, 0, 0);
    if (lane < n) c.a = __ldg(p + lane);
    if (lane + 32 < n) c.b = __ldg(p + lane + 32);
    return c;
}
__device__ __forceinline__ void put_cells(const CellRegs &c, uint4 *sm, int lane) {
    sm[lane] = c.a;
    sm[lane + 32] = c.b;
}

// Byte offset of chunk c of row r of a transposed patch that is staged by
// 16-byte chunks: lanes that read chunk c of consecutive rows hit distinct banks.
__device__ __forceinline__ int chunk_slot(int r, int c) { return r * 128 + ((c ^ (r & 7)) << 4); }

// Copies a patch's source into `buf`, one run of the source per row.  4-byte
// patches more than 16 elements wide whose source runs are whole aligned
// 16-byte chunks (TF_FAST) copy those: they bypass the L1 and take a quarter of the instructions.  GB300,
// 8192^2 f32 T, us per call, elements -> chunks: copy BC8 101 -> 83, A's ld odd
// 108 -> 90; beta = 0.5 BC8 138 -> 126, A's ld odd 149 -> 134.
template <typename T, int KIND>
__device__ __forceinline__ void patch_stage(const PatchDesc &d, const uint4 *cells, unsigned char *buf, int lane) {
    using P = PCfg<T, KIND>;
    constexpr int ES = P::ES;
    const bool tr = (d.flags & TF_TRANSPOSE) != 0;
    const int nr = tr ? d.nx : d.ny, nl = tr ? d.ny : d.nx;
    const int nls = __popc(d.lmask);
    if (P::CHUNKED && (d.flags & TF_FAST)) {
        const LaneMap m = lane_map(nl / 4, lane);
        if (m.c >= nl / 4) return;
        const uint4 *cl = cells + seg_of(d.lmask, m.c * 4);
#pragma unroll 4
        for (int r = m.r0; r < nr; r += m.rpp) {
            const uint4 c = cl[seg_of(d.rmask, r) * nls];
            const char *p = reinterpret_cast<const char *>((static_cast<uint64_t>(c.y) << 32) | c.x) + m.c * 16 +
                            static_cast<int64_t>(r) * (static_cast<int64_t>(static_cast<int32_t>(c.z)) * 4);
            cp_async16(buf + (tr ? chunk_slot(r, m.c) : r * (P::PITCH_N * 4) + m.c * 16), p);
        }
        return;
    }
    const LaneMap m = lane_map(nl, lane);
    if (m.c >= nl) return;
    const uint4 *cl = cells + seg_of(d.lmask, m.c);
    const int pitch = tr ? P::PITCH_T : P::PITCH_N;
    unsigned char *sp = buf + (m.r0 * pitch + m.c) * ES;
    const int sstep = m.rpp * (pitch * ES);
    if (m.rpp == 1) {  // r is the same for every lane: walk the run segments
        uint32_t rest = d.rmask;
        int r = 0;
        do {
            rest &= rest - 1u;  // starts of the later segments
            const int end = min(rest ? __ffs(rest) - 1 : nr, nr);
            const uint4 c = *cl;
            cl += nls;
            const int64_t sb = static_cast<int64_t>(static_cast<int32_t>(c.z)) * ES;
            const char *p = reinterpret_cast<const char *>((static_cast<uint64_t>(c.y) << 32) | c.x) + m.c * ES + r * sb;
#pragma unroll 8
            for (; r < end; ++r, p += sb, sp += sstep) cp_async_elem<ES>(sp, p);
        } while (rest);
    } else {
#pragma unroll 4
        for (int r = m.r0; r < nr; r += m.rpp, sp += sstep) {
            const uint4 c = cl[seg_of(d.rmask, r) * nls];
            const char *p = reinterpret_cast<const char *>((static_cast<uint64_t>(c.y) << 32) | c.x) + m.c * ES +
                            static_cast<int64_t>(r) * (static_cast<int64_t>(static_cast<int32_t>(c.z)) * ES);
            cp_async_elem<ES>(sp, p);
        }
    }
}

// Multiplies the doubles of a group by c, each product rounded to nearest:
// every other one on the integer pipes (rnmul.h), the others on the FP64
// pipe; all of them there when some lane of the warp holds a value that the
// integer form does not admit (one vote, so that no predicated-off FP64
// instruction is issued).  GB300, 8192^2, none / every fourth / every other /
// all of them on the integer pipes, us per call: f64 T beta = 0.7 BC50 -> BC75
// 293 / 294 / 287 / 294, odd lds 295 / 295 / 287 / 288, T alpha = 1.5 BC50 ->
// BC75 206 / 187 / 192 / 240.  One share serves both kinds: every other, the
// best for beta; alpha alone would be 2.6% faster there with every fourth.  c128
// (half the values per row) loses 5%.
template <typename T, int N>
__device__ __forceinline__ void mul_group(Chunk<T> (&v)[N], double c, unsigned mask) {
    double *d = reinterpret_cast<double *>(v);
    const rn::Factor f = rn::factor(c);
    bool bad = false;
#pragma unroll
    for (int k = 1; k < 2 * N; k += 2) bad |= !rn::admits(f, d[k]);
    const bool all_fp64 = __any_sync(mask, bad);
#pragma unroll
    for (int k = 0; k < 2 * N; k += 2) d[k] = __dmul_rn(c, d[k]);
    if (all_fp64) {
#pragma unroll
        for (int k = 1; k < 2 * N; k += 2) d[k] = __dmul_rn(c, d[k]);
    } else {
#pragma unroll
        for (int k = 1; k < 2 * N; k += 2) d[k] = rn::mul(f, d[k]);
    }
}

// Writes a staged patch to A in A's contiguous order, one element per lane
// (CHUNKS: a transposed patch that is staged by 16-byte chunks).
template <typename T, int KIND, bool CHUNKS>
__device__ __forceinline__ void patch_write(const PatchLaunch &a, const PatchDesc &d, Sc &s, int &cached,
                                            const unsigned char *buf, int lane) {
    using P = PCfg<T, KIND>;
    constexpr int V = ET<T>::VEC, G = P::G, NC = (G + V - 1) / V, ES = P::ES;
    if (a.per_problem && d.prob != cached) {
        make_sc(a.per_problem[d.prob], s);
        cached = d.prob;
    }
    s.conj_mask = ET<T>::CPLX && (d.flags & TF_CONJ) ? 0x80000000u : 0u;
    const bool tr = CHUNKS || (d.flags & TF_TRANSPOSE) != 0;
    const LaneMap m = lane_map(d.nx, lane);
    const bool on = m.c < d.nx;
    const unsigned mask = __ballot_sync(0xffffffffu, on);
    // passes of this lane
    const int cnt = d.ny > m.r0 ? (d.ny - m.r0 + m.rpp - 1) / m.rpp : 0;
    const int npass = (d.ny + m.rpp - 1) / m.rpp;
    T *dst = reinterpret_cast<T *>(d.dst) + m.c + static_cast<int64_t>(m.r0) * d.dld;
    const int64_t step = static_cast<int64_t>(m.rpp) * d.dld;
    const unsigned char *sp = buf + (tr ? m.c * P::PITCH_T + m.r0 : m.r0 * P::PITCH_N + m.c) * ES;
    const int sstep = m.rpp * (tr ? ES : P::PITCH_N * ES);
    // CHUNKS: the staged elements of rows p .. p + 3 (a pass is one row; p a
    // multiple of 4)
    auto staged4 = [&](int p) {
        Chunk<T> b;
        b.raw = *reinterpret_cast<const uint4 *>(buf + chunk_slot(m.c, p / 4));
        return b;
    };
    Chunk<T> av[2][NC];
    const T *q = dst;
    auto load = [&](Chunk<T> (&v)[NC], int p0) {  // A's elements of passes p0 .. p0 + G - 1
#pragma unroll
        for (int k = 0; k < G; ++k) {
            T e = T();
            if (p0 + k < cnt) e = *q;
            v[k / V].e[k % V] = e;
            q += step;
        }
    };
    auto write = [&](Chunk<T> (&v)[NC], int p0) {
        if (KIND == K_AXPBY2) prescale<T>(v, NC, s, mask);
        if constexpr (KIND == K_AXPBY && P::INT_MUL) mul_group<T>(v, s.br, mask);  // beta * a, then as K_AXPBY2
        if constexpr (CHUNKS) {
#pragma unroll
            for (int c = 0; c < G; c += 4) {
                if (p0 + c >= npass) break;  // uniform across the warp
                const Chunk<T> b = staged4(p0 + c);
#pragma unroll
                for (int k = c; k < c + 4; ++k) {
                    if (p0 + k < cnt) *dst = combine<KIND>(b.e[(k - c) % V], v[k / V].e[k % V], s);
                    dst += step;
                }
            }
        } else {
#pragma unroll
            for (int k = 0; k < G; ++k) {
                if (p0 + k < cnt) {
                    const T b = *reinterpret_cast<const T *>(sp);
                    *dst = combine<KIND == K_AXPBY && P::INT_MUL ? K_AXPBY2 : KIND>(b, v[k / V].e[k % V], s);
                }
                dst += step;
                sp += sstep;
            }
        }
    };
    if (P::READS_A && on) {
        load(av[0], 0);
        load(av[1], G);
    }
    cp_async_wait<0>();
    __syncwarp();
    if (on) {
        if constexpr (P::READS_A) {
#pragma unroll 1
            for (int p0 = 0; p0 < npass; p0 += 2 * G) {
                write(av[0], p0);
                if (p0 + 2 * G < npass) load(av[0], p0 + 2 * G);
                if (p0 + G < npass) {
                    write(av[1], p0 + G);
                    if (p0 + 3 * G < npass) load(av[1], p0 + 3 * G);
                }
            }
        } else if constexpr (KIND == K_SCALE && P::INT_MUL) {
#pragma unroll 1
            for (int p0 = 0; p0 < npass; p0 += G) {  // uniform across the lanes in `mask`
                Chunk<T> (&v)[NC] = av[0];
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    T e = T();
                    if (p0 + k < cnt) e = *reinterpret_cast<const T *>(sp);
                    v[k / V].e[k % V] = e;
                    sp += sstep;
                }
                mul_group<T>(v, s.ar, mask);
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    if (p0 + k < cnt) *dst = combine<K_COPY>(v[k / V].e[k % V], T(), s);
                    dst += step;
                }
            }
        } else if constexpr (CHUNKS) {
#pragma unroll 2
            for (int p = 0; p < npass; p += 4) {
                const Chunk<T> b = staged4(p);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (p + k < cnt) *dst = combine<KIND>(b.e[k % V], T(), s);
                    dst += step;
                }
            }
        } else {
            constexpr int U = P::ROLLED ? COSTA_PGR : 8;
#pragma unroll U
            for (int p = 0; p < cnt; ++p) {
                *dst = combine<KIND>(*reinterpret_cast<const T *>(sp), T(), s);
                dst += step;
                sp += sstep;
            }
        }
    }
    __syncwarp();  // the buffer and the cells are free again
}

template <typename T, int KIND>
__global__ void __launch_bounds__(PCfg<T, KIND>::WARPS * 32, PCfg<T, KIND>::MINB)
    remap_patch_kernel(const PatchLaunch args) {
    using P = PCfg<T, KIND>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *buf = smem_raw + warp * (P::BUF + P::CELLS);
    uint4 *cells = reinterpret_cast<uint4 *>(buf + P::BUF);
    const int64_t stride = static_cast<int64_t>(gridDim.x) * P::WARPS;
    int64_t t = static_cast<int64_t>(blockIdx.x) * P::WARPS + warp;  // the patch in `raw`
    Sc s;
    int cached = -1;
    if (!args.per_problem) make_sc(args.s, s);
    // descriptors are loaded two patches ahead of the patch that is staged,
    // its cells one ahead
    PatchRaw raw;
    bool have_raw = t < args.n;
    if (have_raw) raw = load_patch(args, t);
    PatchDesc next;
    bool more = false;
    CellRegs cr;
    auto advance = [&]() {  // next = the warp's next patch of this kind
        for (;;) {
            more = have_raw;
            if (!more) return;
            next = unpack_patch(raw);
            t += stride;
            have_raw = t < args.n;
            if (have_raw) raw = load_patch(args, t);
            if (args.per_problem && kind_of(args.per_problem[next.prob].flags) != KIND) continue;
            cr = load_cells(args, next, lane);
            return;
        }
    };
    if (args.per_problem) pdl_wait();  // advance reads the batch's scalars
    advance();
    pdl_wait();
    while (more) {
        const PatchDesc d = next;
        put_cells(cr, cells, lane);
        __syncwarp();
        advance();
        patch_stage<T, KIND>(d, cells, buf, lane);
        cp_async_commit();
        if constexpr (P::CHUNKED) {
            if ((d.flags & (TF_TRANSPOSE | TF_FAST)) == (TF_TRANSPOSE | TF_FAST)) {
                patch_write<T, KIND, true>(args, d, s, cached, buf, lane);
                continue;
            }
        }
        patch_write<T, KIND, false>(args, d, s, cached, buf, lane);
    }
}

template <typename T, int KIND>
cudaError_t launch_patch(const PatchLaunch &a, cudaStream_t st) {
    using P = PCfg<T, KIND>;
    auto kern = remap_patch_kernel<T, KIND>;
    const size_t smem = static_cast<size_t>(P::WARPS) * (P::BUF + P::CELLS);
    static int per_sm = 0;
    if (per_sm == 0) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(smem));
        if (e != cudaSuccess) return e;
        // no more shared memory than MINB blocks need: the rest of the SM's
        // 256 KB is the L1 cache that element-wide copies in flight occupy
        const int pct = static_cast<int>((P::MINB * (smem + 1024) * 100 + 228 * 1024 - 1) / (228 * 1024));
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, pct < 100 ? pct : 100);
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, P::WARPS * 32, smem);
        if (e != cudaSuccess) return e;
        if (per_sm > P::MINB) per_sm = P::MINB;
        if (per_sm < 1) per_sm = 1;
    }
    const int64_t want = (a.n + P::WARPS - 1) / P::WARPS;
    const int64_t cap = static_cast<int64_t>(sm_count()) * per_sm;
    const int blocks = static_cast<int>(want < cap ? want : cap);
    if (blocks <= 0) return cudaSuccess;
    const cudaError_t e = pdl_launch(kern, blocks, P::WARPS * 32, smem, st, a);
    if (e == cudaSuccess) count_launch();
    return e;
}

template <typename T>
cudaError_t launch_patch_t(const PatchLaunch &a, int kind, cudaStream_t st) {
    switch (kind) {
    case K_COPY: return launch_patch<T, K_COPY>(a, st);
    case K_SCALE: return launch_patch<T, K_SCALE>(a, st);
    case K_AXPBY: return launch_patch<T, K_AXPBY>(a, st);
    case K_AXPBY2: return launch_patch<T, K_AXPBY2>(a, st);
    case K_CPLX:
        if constexpr (ET<T>::CPLX) return launch_patch<T, K_CPLX>(a, st);
        return cudaErrorInvalidValue;
    case K_CPLXR:
        if constexpr (sizeof(T) == 16) return launch_patch<T, K_CPLXR>(a, st);
        return cudaErrorInvalidValue;
    case K_CSCALE:
        if constexpr (ET<T>::CPLX) return launch_patch<T, K_CSCALE>(a, st);
        return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace remap
}  // namespace costa
