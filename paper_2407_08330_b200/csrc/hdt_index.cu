// Device-side index builder: (level, parent, cu_seqlens) -> staged family ranges, row blocks,
// work queues.  Integer work only; every array must equal the sequential definition bit for bit.
//
// Two launches, whatever the number of stages (four for batches of many blocks, see many_blocks):
//   k_seq     one CTA per sequence, its arrays in shared memory: validation, child counts, family
//             ranges, compaction to the next stage, greedy packing of row blocks, block records - for
//             all stages of the sequence, in sequence-relative numbers, beside the counts of the stage
//   k_finish  adds the sequences' offsets (sums over the sequences before it), ranks the blocks of a
//             stage by cost (longest first), and sends the header to the host
//             (many blocks: with the offsets from k_offsets, the ranks from the runs that k_sort has sorted)
// Per stage (array of n elements in document order):
//   counts    cnt[p] = children of p, and whether one of them has children
//   ranges    a node whose children are all childless heads a family; head and children get
//             their key range; children of heads (and PAD) are removed for the next stage
//   compact   tok / par of the kept elements in the next stage's array
//   walk      greedy packing of row blocks
// What bounds it: latency (about 40 bytes a token move; a chain of barriers and shared-memory round
// trips per stage).  The stages of a sequence only meet the other sequences' in their offsets, so the
// grid-wide steps (formerly nine launches for three stages and a hundred for twenty, each a launch
// latency behind the one before) are one kernel boundary.  Device time from the first kernel's start to the second's end: 57
// tokens 18 us, 8 x 2048 19, 4 x 8192 tokens 26, 16 documents of 131 000 tokens 43, 2 x 32768 43, 200 trees of 20 stages 58.  Of
// whole passes their first form made, with all else as it was then: 81 -> 57 us (57 tokens, fp32, build and
// forward), 76 -> 56 (8 x 2048, build and forward), 1100 -> 807 (200 trees, build, forward and backward).
#include <cstdio>
#include <climits>
#include <cstring>
#include <atomic>
#include <mutex>
#include <type_traits>
#include <vector>

#include "hdt_internal.cuh"

namespace hdt {

// What k_seq leaves about one sequence for k_finish.
struct SeqInfo {
    int stages;                // stages this sequence's own hierarchy needs (at least 1)
    int res;                   // elements it still has in any later stage of the batch: its root, or nothing
    int err, err_pos;          // structure error, 0 = none
    int more, real;            // elements were left after the last allowed stage; tokens that are not PAD
    long long nnz, nnz_upper, visited;
};

// Sums over the sequences of a batch of many (k_offsets).
struct BatchSums {
    int stages, first_err, more;         // stages of the batch; first sequence with an error, or NO_SEQ; SeqInfo::more of any
    long long nnz, visited, nnz_upper, real;
    int count[HDT_MAX_STAGES][4];        // of each stage: elements, blocks, SELF non-EMPTY blocks, EMPTY blocks
};
static constexpr int NO_SEQ = 0x7fffffff;

struct Layout {
    size_t header, info, sums, offs, counts, rank, recs, el, upl, glob, keys, before, stage0, stage_stride;
    size_t s_tok, s_par, s_rng, s_up, s_scu, s_blocks, s_queue, s_queue2;  // offsets inside a stage
    size_t total;
    int capnb;
};

static size_t al(size_t x) { return (x + 255) & ~size_t(255); }

static constexpr int NGLOB = 11;      // element arrays of the sequences that do not fit in shared memory

static Layout make_layout(int B, int T, int bm, int max_stages) {   // bm: the smaller of the two block sizes
    Layout L;
    L.capnb = 2 * (T / bm + 1) + 4 * B + 2;
    size_t o = 0;
    L.header = o; o += al(sizeof(DevHeader));
    L.info = o; o += al(sizeof(SeqInfo) * (size_t)B);
    L.sums = o; o += al(sizeof(BatchSums));
    L.offs = o; o += al(sizeof(int) * 2 * (size_t)max_stages * B);
    L.counts = o; o += al(sizeof(int) * 4 * (size_t)max_stages * B);
    L.rank = o; o += al(sizeof(int) * (size_t)T);
    L.recs = o; o += al(sizeof(int4) * (size_t)max_stages * L.capnb);
    L.keys = o; o += al(sizeof(long long) * (size_t)max_stages * L.capnb);
    L.before = o; o += al(sizeof(int) * (size_t)max_stages * L.capnb);
    L.el = o; o += al(sizeof(int4) * (size_t)(max_stages - 1) * T);
    L.upl = o; o += al(sizeof(int) * (size_t)(max_stages - 1) * T);
    L.glob = o; o += NGLOB * al(sizeof(int) * (size_t)T);
    L.stage0 = o;
    size_t s = 0;
    L.s_tok = s; s += al(sizeof(int) * (size_t)T);
    L.s_par = s; s += al(sizeof(int) * (size_t)T);
    L.s_rng = s; s += al(sizeof(int) * 2 * (size_t)T);
    L.s_up = s; s += al(sizeof(int) * (size_t)T);
    L.s_scu = s; s += al(sizeof(int) * (size_t)(B + 1));
    L.s_blocks = s; s += al(sizeof(int) * 5 * (size_t)L.capnb);
    L.s_queue = s; s += al(sizeof(int) * (size_t)L.capnb);
    L.s_queue2 = s; s += al(sizeof(int) * (size_t)L.capnb);
    L.stage_stride = s;
    L.total = o + s * (size_t)max_stages;
    return L;
}

// First block slot of a sequence that starts at token c: a walk packs two consecutive blocks into
// more than bm elements, so a sequence of n elements has at most 2 ceil(n / bm) + 1 blocks.
__device__ __forceinline__ int block_slot(int c, int b, int bm) { return 2 * (c / bm) + 4 * b; }

// Keys of row e with range [lo, hi) that the direction bits keep.  A row whose range starts at or
// after itself is the head of its family (the keys after it are its children); otherwise lo is
// the row's parent and the remaining keys are its siblings.  dirs: 1 = child -> parent,
// 2 = sibling <-> sibling, 4 = parent -> child; the diagonal always stays.
__device__ __forceinline__ int row_pairs(int e, int lo, int hi, int dirs) {
    if (hi <= lo) return 0;
    if (lo >= e) return (lo == e ? 1 : 0) + ((dirs & 4) ? hi - e - 1 : 0);
    return 1 + ((dirs & 1) ? 1 : 0) + ((dirs & 2) ? hi - lo - 2 : 0);
}

// Element numbers and child counts of a stage: 16 bits in shared memory, 32 bits in the workspace
// for sequences too long for it.  The top bit of a count says that a child has children itself.
template <class I> struct Elem;
template <> struct Elem<uint16_t> {
    static constexpr unsigned NONE = 0xffffu, FLAG = 0x8000u, MASK = 0x7fffu;
    static __device__ __forceinline__ unsigned *word(uint16_t *c, int &sh) {
        sh = ((uintptr_t)c & 2) * 8;
        return reinterpret_cast<unsigned *>((uintptr_t)c & ~(uintptr_t)3);
    }
    static __device__ __forceinline__ void add(uint16_t *c, unsigned v) { int sh; unsigned *q = word(c, sh); atomicAdd(q, v << sh); }
    static __device__ __forceinline__ void flag(uint16_t *c) { int sh; unsigned *q = word(c, sh); atomicOr(q, FLAG << sh); }
};
template <> struct Elem<uint32_t> {
    static constexpr unsigned NONE = 0xffffffffu, FLAG = 0x80000000u, MASK = 0x7fffffffu;
    static __device__ __forceinline__ void add(uint32_t *c, unsigned v) { atomicAdd(c, v); }
    static __device__ __forceinline__ void flag(uint32_t *c) { atomicOr(c, FLAG); }
};

// Arrays of a sequence.  Flat: in one piece.  Sliced: 2^sl elements in the shared memory of each CTA of the
// sequence's cluster; another CTA's slice is read and added to over distributed shared memory (parents
// of anchors, rows of a block that straddles two slices: a few percent of the accesses).
template <class T> struct Flat {
    using I = T;
    I *base;
    __device__ __forceinline__ I *ptr(unsigned e) const { return base + e; }
    __device__ __forceinline__ unsigned get(unsigned e) const { return base[e]; }
};
template <class T>
__device__ __forceinline__ T *map_rank(T *p, unsigned rank) {
    uint64_t r;
    asm("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"(p), "r"(rank));
    return reinterpret_cast<T *>(r);
}
struct Sliced {
    using I = uint16_t;
    I *loc;
    unsigned sl, rank;
    __device__ __forceinline__ I *ptr(unsigned e) const {
        I *p = loc + (e & ((1u << sl) - 1u));
        const unsigned r = e >> sl;
        return r == rank ? p : map_rank(p, r);
    }
    __device__ __forceinline__ unsigned get(unsigned e) const {
        const unsigned r = e >> sl;
        return r == rank ? loc[e & ((1u << sl) - 1u)] : *ptr(e);
    }
};

// Child counts of 32 consecutive elements (one per lane, NONE beyond the end): siblings follow one another,
// so a run of equal parents is one addition (thirty additions to one word are thirty turns of the
// shared-memory atomic unit).
template <class A>
__device__ __forceinline__ void count_children(const A &cnt, unsigned p, int lane) {
    using E = Elem<typename A::I>;
    const unsigned before = __shfl_up_sync(0xffffffffu, p, 1);
    const bool first = lane == 0 || p != before;
    const unsigned m = __ballot_sync(0xffffffffu, first);
    if (first && p != E::NONE) {
        const unsigned rest = lane == 31 ? 0u : m >> (lane + 1);
        E::add(cnt.ptr(p), rest ? (unsigned)__ffs(rest) : 32u - (unsigned)lane);
    }
}

static constexpr int SEQ_CAP_MAX = 32768;   // tokens of a sequence held in shared memory (15-bit counts)
static constexpr int UC_MAX = 4096;         // elements of an upper stage held there
static constexpr int SB0 = 1024, SBU = 256, SBA = 1024; // block starts of stage 0 / an upper stage / all upper stages held there
static constexpr int SEQ_CLUSTER = 8;       // CTAs of a long sequence

struct SeqArgs {
    const int8_t *level;
    const int32_t *parent, *cu;
    int B, T, ms, bm, bmu, bmin, dirs;
    int cap, uc, pool;         // tokens of stage 0 / elements of an upper stage that fit in shared memory; bytes for the upper stages
    int *tok, *par, *rng, *up, *scu;     // stage 0 (final, but for `up`: relative to the sequence)
    int *rank;
    SeqInfo *info;
    int *counts;               // [4][ms][B]: elements, blocks, SELF non-EMPTY blocks, EMPTY blocks
    int4 *recs;                // [ms][capnb]: r0, a, b, rows | flags << 8, relative to the sequence
    int capnb;
    int *ticket;               // (see HostHeader::done) cleared here for k_finish
    int4 *el;                  // [ms - 1][T]: tok, par, lo, hi of the upper stages, relative to the sequence
    int *upl;                  // [ms - 1][T]: index in the next stage, -1 = removed
    uint32_t *glob;            // NGLOB arrays of glob_stride elements
    size_t glob_stride;
};

struct SeqShared {
    int bst0[SB0], bst[SBU];
    int wtot[32], wtotu[32], ctot[SEQ_CLUSTER];
    int err, err_pos, real, flag0, flag, nb, nf, ne;
    int ns[HDT_MAX_STAGES], nbs[HDT_MAX_STAGES], bso[HDT_MAX_STAGES], nfs[HDT_MAX_STAGES], nes[HDT_MAX_STAGES], bsu[SBA], bsu_n;     // (seq_upper_all)
    uint32_t seg[2][4][128], slice[2][128], slices[SEQ_CLUSTER][128];     // (walk_slice)
    int bstf[SB0];                         // block starts of the first slice
    int own[2], own_end[2], base;          // blocks of this slice and of the first one, ends of their last ones; blocks before this slice
    unsigned long long nnz, nnz_upper, vis;
};

__device__ __forceinline__ void seq_fail(SeqShared *sh, int pos) {
    if (atomicCAS(&sh->err, 0, HDT_ERR_BAD_HIERARCHY) == 0) sh->err_pos = pos;
}

// Barrier of the warps that build the upper stages (with one CTA per sequence its last warp meanwhile walks stage 0's blocks).
__device__ __forceinline__ void bar_upper(int n) { asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory"); }
__device__ __forceinline__ void cluster_arrive() { __syncwarp(); asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { __syncwarp(); asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void seq_sync(unsigned cs) {
    if (cs > 1) { cluster_arrive(); cluster_wait(); }
    else __syncthreads();
}

// Range and fate of element e with parent p; y, yp: count words of the two.  lone_root: stage 0's root without children,
// a family of its own there.  Returns whether a family holds the element as a child.
template <class E>
__device__ __forceinline__ bool elem_range(unsigned e, unsigned p, unsigned y, unsigned yp, bool lone_root, unsigned &lo, unsigned &hi) {
    const unsigned c = y & E::MASK, cp = yp & E::MASK;
    lo = hi = 0;
    if ((c > 0 && !(y & E::FLAG)) || (lone_root && c == 0)) {
        lo = (p == E::NONE) ? e : e + 1;
        hi = e + 1 + c;
    } else if (p != E::NONE && cp > 0 && !(yp & E::FLAG)) {
        lo = p;
        hi = p + 1 + cp;
        return true;
    }
    return false;
}

// Greedy packing of row blocks (one thread): a cut that would split a family which starts inside the
// block moves to the family's head.  fpos[e]: distance of e from the head of the family that holds it as
// a child (0 = none, capped at 255 >= bm): one dependent load per block.
__device__ __forceinline__ int walk_blocks(const uint8_t *fpos, int n, int bm, int *bst, int nbst, int4 *rec) {
    int pos = 0, nb = 0;
    while (pos < n) {
        int end = min(pos + bm, n);
        if (end < n) {
            const int f = fpos[end];
            if (f < end - pos) end -= f;
        }
        if (nb < nbst) bst[nb] = pos; else rec[nb].x = pos;
        ++nb;
        pos = end;
    }
    return nb;
}

// Rows of block i of a stage with nb blocks and n elements: its first nbst starts are in bst, the others in the records.
__device__ __forceinline__ void block_rows(const int *bst, int nbst, const int4 *rec, int i, int nb, int n, int &r0, int &r1) {
    r0 = i < nbst ? bst[i] : rec[i].x;
    r1 = i + 1 < nb ? (i + 1 < nbst ? bst[i + 1] : rec[i + 1].x) : n;
}

// Records of the blocks i0, i0 + di, ... < i1, one warp per block.  rows(i, r0, r1) gives the rows of a block,
// get(e, lo, hi) the range of an element and returns whether it lives on.  (The loops stay rolled: nearly
// every instruction of this kernel is executed once or twice by a warp, and fetching it costs more than that.)
template <class Get, class Rows>
__device__ __forceinline__ void make_records(Get get, Rows rows, int4 *rec, int i0, int i1, int di, int lane, int *nf, int *ne,
                                             unsigned long long *vis_out) {
    long long vis = 0;
    int mf = 0, me = 0;
#pragma unroll 1
    for (int i = i0; i < i1; i += di) {
        int r0, r1;
        rows(i, r0, r1);
        // a block is dense where all its rows have one range
        int a = INT_MAX, bb = INT_MIN, a2 = INT_MIN, bb2 = INT_MAX;
        bool carry = false, none = false;
#pragma unroll 1
        for (int e = r0 + lane; e < r1; e += 32) {
            int lo, hi;
            carry |= get(e, lo, hi);
            if (hi > lo) { a = min(a, lo); bb = max(bb, hi); a2 = max(a2, lo); bb2 = min(bb2, hi); }
            else none = true;
        }
        __syncwarp();
        a = __reduce_min_sync(0xffffffffu, a);
        bb = __reduce_max_sync(0xffffffffu, bb);
        a2 = __reduce_max_sync(0xffffffffu, a2);
        bb2 = __reduce_min_sync(0xffffffffu, bb2);
        carry = __any_sync(0xffffffffu, carry);
        none = __any_sync(0xffffffffu, none);
        const bool any = bb > a;
        const bool dense = any && !none && a == a2 && bb == bb2;
        if (!any) { a = r0; bb = r0; }
        if (lane == 0) {
            int fl = 0;
            if (a >= r0 && bb <= r1) fl |= HDT_BLK_SELF;
            if (dense) fl |= HDT_BLK_DENSE;
            if (carry) fl |= HDT_BLK_CARRY;
            if (!any) fl |= HDT_BLK_EMPTY;
            rec[i] = make_int4(r0, a, bb, (r1 - r0) | (fl << 8));
            vis += (long long)(r1 - r0) * (bb - a);
            mf += (fl & HDT_BLK_SELF) && any;
            me += !any;
        }
    }
    if (lane == 0) {
        if (mf) atomicAdd(nf, mf);
        if (me) atomicAdd(ne, me);
        if (vis) atomicAdd(vis_out, (unsigned long long)vis);
    }
}

// log2 of the contiguous elements each of nw warps takes of n (at least one 32-element step).
__device__ __forceinline__ int seg_shift(int n, int nw) {
    int k = 5;
    while (((long long)nw << k) < n) ++k;
    return k;
}
// Exclusive offsets of the warps (lane w holds that of warp w) and the total.
__device__ __forceinline__ int warp_offsets(const int *wtot, int nw, int lane, int &total) {
    const int v0 = lane < nw ? wtot[lane] : 0;
    int v = v0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += x;
    }
    total = __shfl_sync(0xffffffffu, v, 31);
    return v - v0;
}

// The part of a sequence one CTA holds in stage 0.
struct Slice {
    unsigned rank, cs, sl;     // CTA in the cluster, its size, log2 of the slice length
    int s0, L, e0, ne;         // sequence start and length; first element of the slice and their number
};

// The walk of a sequence whose slices lie in the CTAs of a cluster.  A walk enters a stretch of the array at one of bm
// offsets, and where it leaves the stretch depends on nothing else: so a thread per offset walks each quarter of a
// slice (seg: offset behind it | blocks << 8), the quarters are composed, then the slices, and four threads
// repeat the walk that was the right one.  One thread for the whole sequence took 120 cycles a block: 11 000 cycles of the
// build of 8192 tokens, 37 000 of 32768.  fpos(e): see walk_blocks.
template <class F>
__device__ __forceinline__ int next_block(F fpos, int pos, int bm, int n) {
    int end = min(pos + bm, n);
    if (end < n) {
        const int f = fpos(end);
        if (f < end - pos) end -= f;
    }
    return end;
}
template <class F>
__device__ __forceinline__ void walk_slice(F fpos, int bm, SeqShared &sh, const Slice &c, unsigned rank, int at) {
    const int t = threadIdx.x, g = t >> 7, o = t & 127, len = 1 << (c.sl - 2);
    const int a = (int)(rank << c.sl) + g * len, b = a + len;
    int pos = a + o, k = 0;
    while (pos < min(b, c.L)) { pos = next_block(fpos, pos, bm, c.L); ++k; }
    sh.seg[at][g][o] = (uint32_t)min(max(pos - b, 0), 127) | (uint32_t)k << 8;
    __syncthreads();
    if (t < 128) {
        unsigned x = t, n = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) { const uint32_t v = sh.seg[at][i][x]; x = v & 255u; n += v >> 8; }
        sh.slice[at][t] = x | n << 8;
    }
}
// Behind a cluster barrier, in every CTA but the first: the block starts of its slice (bst0) and of the first one (bstf),
// the first SB0 of each (the others' in the records).  nb: the number of all.
template <class F>
__device__ __forceinline__ void walk_starts(F fpos, int bm, SeqShared &sh, const Slice &c, int4 *rec, int *nb) {
    const int t = threadIdx.x;
    for (int i = t; i < (int)c.cs * 128; i += blockDim.x) {
        const int r = i >> 7, k = i & 127;
        sh.slices[r][k] = *map_rank(&sh.slice[r ? 0 : 1][k], r ? r : 1);
    }
    __syncthreads();
    const int f = t >> 5, q = t & 31;          // warp 0: this slice, warp 1: the first one; a lane per quarter
    if (f < 2 && q < 4) {
        unsigned x = 0, n = 0;
        for (unsigned r = 0; r < (f ? 0u : c.rank); ++r) { const uint32_t v = sh.slices[r][x]; x = v & 255u; n += v >> 8; }
        const SeqShared *shs = f ? map_rank(&sh, 1) : &sh;
        unsigned m = 0;
        for (int i = 0; i < q; ++i) { const uint32_t v = shs->seg[f][i][x]; x = v & 255u; m += v >> 8; }
        const int len = 1 << (c.sl - 2), a = (f ? 0 : (int)(c.rank << c.sl)) + q * len, b = min(a + len, c.L);
        int *bst = f ? sh.bstf : sh.bst0;
        int pos = a + (int)x;
        for (; pos < b; ++m) {
            if (m < SB0) bst[m] = pos; else rec[n + m].x = pos;
            pos = next_block(fpos, pos, bm, c.L);
        }
        if (q == 3) {
            sh.own[f] = (int)m;
            sh.own_end[f] = min(max(pos, a), c.L);
            if (!f) sh.base = (int)n;
            if (!f && c.rank + 1 == c.cs) *nb = (int)(n + m);
        }
    }
    __syncthreads();
}

// Stage 0 of one slice up to the keep flags: X parents, Y counts, Z levels and then the number of kept
// elements before each kept one, relative to the slice.  sh: this CTA's, sh0: the first CTA's shared state.
template <class A>
__device__ __forceinline__ void seq_stage0(const SeqArgs &a, SeqShared &sh, SeqShared *sh0, const A &X, const A &Y, const A &Z, const Slice &c,
                                           uint8_t *fpos, bool &root_real) {
    using I = typename A::I;
    using E = Elem<I>;
    const int t = threadIdx.x, nt = blockDim.x, lane = t & 31, w = t >> 5, nw = nt >> 5;
    I *x = X.ptr(c.e0), *y = Y.ptr(c.e0), *z = Z.ptr(c.e0);
    int bad = -1;
    for (int i0 = 0; i0 < c.ne; i0 += 8 * nt) {          // (eight loads in flight per thread)
        int p8[8], l8[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int i = i0 + k * nt + t;
            if (i < c.ne) { p8[k] = a.parent[c.s0 + c.e0 + i]; l8[k] = a.level[c.s0 + c.e0 + i]; }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int i = i0 + k * nt + t, e = c.e0 + i;
            if (i >= c.ne) break;
            const int p = p8[k], l = l8[k];
            bool ok = true;
            unsigned q = E::NONE;
            if (l < 0) ok = (l == -1 && p == -1);
            else if (e == 0) ok = (l == 0 && p == -1);
            else if (l > HDT_MAX_STAGES * 8 || p < 0 || p >= e) ok = false;
            else q = (unsigned)p;
            x[i] = (I)q;
            z[i] = (I)(uint8_t)l;
            y[i] = 0;
            if (!ok) bad = e;
        }
    }
    seq_sync(c.cs);
    if (bad >= 0) seq_fail(sh0, c.s0 + bad);
    root_real = c.L > 0 && (int8_t)(uint8_t)Z.get(0) >= 0;
    for (int i0 = 32 * w; i0 < c.ne; i0 += nt) {
        const int i = i0 + lane, e = c.e0 + i;
        unsigned p = E::NONE;
        if (i < c.ne) {
            p = x[i];
            const int l = (int8_t)(uint8_t)z[i];
            if (l >= 0 && e > 0) {
                if (p != E::NONE && (int)(int8_t)(uint8_t)Z.get(p) != l - 1) seq_fail(sh0, c.s0 + e);
                if ((int8_t)(uint8_t)Z.get(e - 1) < 0) seq_fail(sh0, c.s0 + e);     // PAD only as a suffix
            }
        }
        count_children(Y, p, lane);
    }
    seq_sync(c.cs);
    for (int i = t; i < c.ne; i += nt) {
        const unsigned p = x[i];
        if ((y[i] & E::MASK) > 0 && p != E::NONE) E::flag(Y.ptr(p));
    }
    seq_sync(c.cs);
    const int k = seg_shift(c.ne, nw);
    int run = 0, next = 0, nreal = 0;
    long long deg = 0;
    for (int i0 = w << k; i0 < min((w + 1) << k, c.ne); i0 += 32) {
        const int i = i0 + lane, e = c.e0 + i, g = c.s0 + e;
        bool kp = false;
        if (i < c.ne) {
            const bool real = (int8_t)(uint8_t)z[i] >= 0;
            const unsigned p = x[i];
            unsigned lo, hi;
            const bool child = elem_range<E>(e, p, y[i], p != E::NONE ? Y.get(p) : 0u, e == 0 && root_real, lo, hi);
            if (child && !((int)p < e && e < (int)hi)) seq_fail(sh0, g);
            kp = real && !child;
            nreal += real;
            fpos[i] = child ? (uint8_t)min(e - (int)p, 255) : 0;
            deg += row_pairs(e, (int)lo, (int)hi, a.dirs);
            if (kp && p != E::NONE) next = 1;
        }
        const unsigned m = __ballot_sync(0xffffffffu, kp);
        if (i < c.ne) z[i] = (I)(kp ? (unsigned)(run + __popc(m & ((1u << lane) - 1u))) : E::NONE);
        run += __popc(m);
    }
    for (int o = 16; o; o >>= 1) deg += __shfl_xor_sync(0xffffffffu, deg, o);
    next = __any_sync(0xffffffffu, next);
    nreal = __reduce_add_sync(0xffffffffu, nreal);
    if (lane == 0) {
        sh.wtot[w] = run;
        if (nreal) atomicAdd(&sh0->real, nreal);
        if (deg) atomicAdd(&sh0->nnz, (unsigned long long)deg);
        if (next) sh0->flag0 = 1;
    }
    __syncthreads();
    int total;
    const int mine = __shfl_sync(0xffffffffu, warp_offsets(sh.wtot, nw, lane, total), w);
    if (mine)
        for (int i = (w << k) + lane; i < min((w + 1) << k, c.ne); i += 32)
            if (z[i] != E::NONE) z[i] = (I)(z[i] + mine);
    if (t < (int)c.cs) (c.cs > 1 ? map_rank(&sh, t) : &sh)->ctot[c.rank] = total;      // to every CTA of the cluster
}

// Stage 0 -> stage 1: the kept elements' parents and tokens.
template <class A, class J>
__device__ __forceinline__ void seq_compact0(const SeqArgs &a, const A &X, const A &Z, const int *coff, J *par2, J *tok2, const Slice &c) {
    using I = typename A::I;
    using E = Elem<I>;
    const I *x = X.ptr(c.e0), *z = Z.ptr(c.e0);
    for (int i = threadIdx.x; i < c.ne; i += blockDim.x) {
        const unsigned v = z[i];
        if (v != E::NONE) {
            const int u = (int)v + coff[c.rank];
            const unsigned p = x[i];
            unsigned q = E::NONE;
            if (p != E::NONE) q = Z.get(p);
            par2[u] = (J)(q != E::NONE ? q + (unsigned)coff[p >> c.sl] : Elem<J>::NONE);
            tok2[u] = (J)(c.e0 + i);
        }
    }
}

// All stages above 0 of one sequence, by the first nw warps of its first CTA.
template <class J>
__device__ __forceinline__ void seq_upper(const SeqArgs &a, SeqShared &sh, J *par, J *tok, J *par2, J *tok2, J *cnt, J *pre, uint8_t *fpos, int b,
                                          int s0, int slot, int n, int nw, int &stages, int &res, int &more) {
    using E = Elem<J>;
    const int t = threadIdx.x, tu = nw * 32, lane = t & 31, w = t >> 5;
    const Flat<J> C{cnt};
    int s = 1;
    while (true) {
        if (s == a.ms) { more = 1; break; }          // elements left that no stage may take
        int4 *rec = a.recs + (size_t)s * a.capnb + slot;
        int4 *el = a.el + (size_t)(s - 1) * a.T + s0;
        int *upl = a.upl + (size_t)(s - 1) * a.T + s0;
        for (int e = t; e < n; e += tu) cnt[e] = 0;
        if (t == 0) { sh.flag = 0; sh.nf = 0; sh.ne = 0; }
        bar_upper(tu);
        for (int e0 = 32 * w; e0 < n; e0 += tu) count_children(C, e0 + lane < n ? (unsigned)par[e0 + lane] : E::NONE, lane);
        bar_upper(tu);
        for (int e = t; e < n; e += tu) {
            const unsigned p = par[e];
            if (p != E::NONE && (cnt[e] & E::MASK) > 0) E::flag(cnt + p);
        }
        bar_upper(tu);
        const int k = seg_shift(n, nw);
        int run = 0, next = 0;
        long long deg = 0;
        for (int i0 = w << k; i0 < min((w + 1) << k, n); i0 += 32) {
            const int e = i0 + lane;
            bool kp = false;
            if (e < n) {
                const unsigned p = par[e];
                unsigned lo, hi;
                const bool child = elem_range<E>(e, p, cnt[e], p != E::NONE ? cnt[p] : 0u, false, lo, hi);
                const int tk = tok[e];
                if (child) {
                    if (!((int)p < e && e < (int)hi)) seq_fail(&sh, s0 + tk);
                    a.rank[s0 + tk] = e - (int)p;
                }
                kp = !child;
                el[e] = make_int4(tk, (p == E::NONE) ? -1 : (int)p, (int)lo, (int)hi);
                fpos[e] = child ? (uint8_t)min(e - (int)p, 255) : 0;
                deg += row_pairs(e, (int)lo, (int)hi, a.dirs);
                if (kp && p != E::NONE) next = 1;
            }
            const unsigned m = __ballot_sync(0xffffffffu, kp);
            if (e < n) pre[e] = (J)(kp ? (unsigned)(run + __popc(m & ((1u << lane) - 1u))) : E::NONE);
            run += __popc(m);
        }
        for (int o = 16; o; o >>= 1) deg += __shfl_xor_sync(0xffffffffu, deg, o);
        next = __any_sync(0xffffffffu, next);
        if (lane == 0) {
            sh.wtotu[w] = run;
            if (deg) atomicAdd(&sh.nnz_upper, (unsigned long long)deg);
            if (next) sh.flag = 1;
        }
        bar_upper(tu);
        const bool go_on = sh.flag != 0;
        if (t == tu - 1) sh.nb = walk_blocks(fpos, n, a.bmu, sh.bst, SBU, rec);
        __syncwarp();
        int total;
        const int wo = warp_offsets(sh.wtotu, nw, lane, total);
        for (int i0 = w << k; i0 < min((w + 1) << k, n); i0 += 32) {
            const int e = i0 + lane;
            const unsigned z = e < n ? pre[e] : E::NONE;
            unsigned p = E::NONE, q = E::NONE;
            if (z != E::NONE) { p = par[e]; if (p != E::NONE) q = pre[p]; }
            const int wp = __shfl_sync(0xffffffffu, wo, q != E::NONE ? (int)(p >> k) : 0);
            const int mine = __shfl_sync(0xffffffffu, wo, w);
            const int u = z != E::NONE ? (int)z + mine : -1;
            if (e < n) upl[e] = u;
            if (u >= 0 && go_on) {
                par2[u] = (J)(q != E::NONE ? q + (unsigned)wp : E::NONE);
                tok2[u] = tok[e];
            }
        }
        bar_upper(tu);
        make_records([&](int e, int &lo, int &hi) {
                         const unsigned p = par[e];
                         unsigned l, h;
                         const bool child = elem_range<E>(e, p, cnt[e], p != E::NONE ? cnt[p] : 0u, false, l, h);
                         lo = (int)l; hi = (int)h;
                         return !child;
                     },
                     [&](int i, int &r0, int &r1) { block_rows(sh.bst, SBU, rec, i, sh.nb, n, r0, r1); }, rec, w, sh.nb, nw, lane, &sh.nf, &sh.ne, &sh.vis);
        bar_upper(tu);
        if (t == 0) {
            int *c = a.counts + (size_t)s * a.B + b;
            const size_t q = (size_t)a.ms * a.B;
            c[0] = n; c[q] = sh.nb; c[2 * q] = sh.nf; c[3 * q] = sh.ne;
        }
        ++s;
        res = total;
        if (!go_on) break;
        n = total;
        J *x = par; par = par2; par2 = x;
        x = tok; tok = tok2; tok2 = x;
    }
    stages = s;
}

// The same for all stages at once, where the maps fit in the pool.  With g(e) the height of e in stage 1's
// tree, e lives in the stages 1 .. g(parent of e) and heads its family in stage g(e): every stage's elements and
// ranges follow from the heights, and the stages need not follow one another (twenty stages of a
// 500-token tree: 50 us one by one, each a chain of six barriers).  Returns whether they fitted.
__device__ __forceinline__ bool seq_upper_all(const SeqArgs &a, SeqShared &sh, const uint16_t *par, const uint16_t *tok, uint32_t *pool, size_t pool_bytes,
                                              int b, int s0, int slot, int n, int nw, int &stages, int &res, int &more) {
    using E = Elem<uint16_t>;
    const int t = threadIdx.x, tu = nw * 32, lane = t & 31, w = t >> 5;
    uint32_t *g = pool;
    uint16_t *cn = reinterpret_cast<uint16_t *>(g + n);
    const int n2 = (n + 1) & ~1;
    for (int e = t; e < n2; e += tu) { if (e < n) g[e] = 0; cn[e] = 0; }
    bar_upper(tu);
    for (int e0 = 32 * w; e0 < n; e0 += tu) count_children(Flat<uint16_t>{cn}, e0 + lane < n ? (unsigned)par[e0 + lane] : E::NONE, lane);
    bar_upper(tu);
    for (int e = t; e < n; e += tu) {
        if (cn[e] != 0) continue;
        unsigned p = par[e];
        for (unsigned k = 1; p != E::NONE; ++k) {          // climb while this leaf is the deepest seen
            if (atomicMax(&g[p], k) >= k) break;
            p = par[p];
        }
    }
    bar_upper(tu);
    const int S = min(1 + (int)g[0], a.ms);
    uint16_t *map = cn + n2 - 2 * (size_t)n2;              // (used from stage 2 on)
    uint8_t *fp = reinterpret_cast<uint8_t *>(cn + n2 + (size_t)max(S - 2, 0) * n2) - n2;      // (from stage 1 on)
    const int nch = (n + 31) / 32;
    uint16_t *coff = reinterpret_cast<uint16_t *>(fp + (size_t)max(S, 1) * n2) - 2 * nch;    // (from stage 2 on)
    if (reinterpret_cast<uint8_t *>(pool) + pool_bytes < reinterpret_cast<uint8_t *>(coff + S * nch)) return false;
    more = 1 + (int)g[0] > a.ms;
    stages = S;
    res = 1;
    // tasks of 32 elements of one stage, dealt to the warps
    for (int i = w; i < nch * (S - 2); i += nw) {
        const int s = 2 + i / nch, ch = i % nch, e = 32 * ch + lane;
        bool in = false;
        if (e < n) { const unsigned p = par[e]; in = p == E::NONE || (int)g[p] >= s; }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (e < n) map[s * (size_t)n2 + e] = in ? (uint16_t)__popc(m & ((1u << lane) - 1u)) : (uint16_t)E::NONE;
        if (lane == 0) coff[s * nch + ch] = (uint16_t)__popc(m);
    }
    bar_upper(tu);
    for (int s = 2 + w; s < S; s += nw) {
        int run = 0;
        for (int c0 = 0; c0 < nch; c0 += 32) {
            const int c = c0 + lane, v0 = c < nch ? coff[s * nch + c] : 0;
            int v = v0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += x;
            }
            if (c < nch) coff[s * nch + c] = (uint16_t)(run + v - v0);
            run += __shfl_sync(0xffffffffu, v, 31);
        }
        if (lane == 0) sh.ns[s] = run;
    }
    if (t == 0) { sh.ns[1] = n; sh.bsu_n = 0; }
    bar_upper(tu);
    long long deg = 0;
    for (int i = w; i < nch * (S - 1); i += nw) {
        const int s = 1 + i / nch, ch = i % nch, e = 32 * ch + lane;
        if (e >= n) continue;
        const uint16_t *ms = map + s * (size_t)n2, *mn = ms + n2;
        const unsigned p = par[e];
        const int tk = tok[e], ge = (int)g[e], ce = cn[e];
        int pos = e, pp = -1, gp = INT_MAX, cp = 0;
        if (p != E::NONE) { gp = (int)g[p]; cp = cn[p]; }
        if (gp < s) continue;                               // not in this stage
        if (s > 1) pos = ms[e] + coff[s * nch + ch];
        if (p != E::NONE) pp = s > 1 ? (int)ms[p] + coff[s * nch + (p >> 5)] : (int)p;
        const bool child = gp == s;
        int lo = 0, hi = 0;
        if (ge == s) {
            lo = p == E::NONE ? pos : pos + 1;
            hi = pos + 1 + ce;
        } else if (child) {
            lo = pp;
            hi = pp + 1 + cp;
            if (!(pp < pos && pos < hi)) seq_fail(&sh, s0 + tk);
            a.rank[s0 + tk] = pos - pp;
        }
        const size_t o = (size_t)(s - 1) * a.T + s0 + pos;
        a.el[o] = make_int4(tk, pp, lo, hi);
        a.upl[o] = child ? -1 : (s + 1 < S ? (int)mn[e] + coff[(s + 1) * nch + ch] : 0);
        fp[s * (size_t)n2 + pos] = child ? (uint8_t)min(pos - pp, 255) : 0;
        deg += row_pairs(pos, lo, hi, a.dirs);
    }
    for (int o = 16; o; o >>= 1) deg += __shfl_xor_sync(0xffffffffu, deg, o);
    if (lane == 0 && deg) atomicAdd(&sh.nnz_upper, (unsigned long long)deg);
    bar_upper(tu);
    for (int s = 1 + w; s < S; s += nw) {          // a warp per stage: where its blocks start
        if (lane == 0) {
            const int o = atomicAdd(&sh.bsu_n, 2 * (sh.ns[s] / a.bmu) + 2);
            sh.bso[s] = o;
            sh.nbs[s] = walk_blocks(fp + s * (size_t)n2, sh.ns[s], a.bmu, sh.bsu + min(o, SBA), max(SBA - o, 0), a.recs + (size_t)s * a.capnb + slot);
            sh.nfs[s] = 0; sh.nes[s] = 0;
        }
    }
    bar_upper(tu);
    const int split = max(nw / max(S - 1, 1), 1);     // warps that share a stage
#pragma unroll 1
    for (int s = 1 + w / split; s < S; s += nw / split) {
        const int4 *el = a.el + (size_t)(s - 1) * a.T + s0;
        const int *upl = a.upl + (size_t)(s - 1) * a.T + s0;
        int4 *rec = a.recs + (size_t)s * a.capnb + slot;
        const int nb = sh.nbs[s], ns = sh.ns[s], o = sh.bso[s], held = max(SBA - o, 0);
        const int *bst = sh.bsu + min(o, SBA);
        make_records([&](int e, int &lo, int &hi) {
            const int4 x = el[e];
            lo = x.z; hi = x.w;
            return upl[e] >= 0;
        }, [&](int i, int &r0, int &r1) { block_rows(bst, held, rec, i, nb, ns, r0, r1); }, rec, w % split, nb, split, lane, &sh.nfs[s], &sh.nes[s],
           &sh.vis);
    }
    bar_upper(tu);
    for (int s = 1 + t; s < S; s += tu) {
        int *c = a.counts + (size_t)s * a.B + b;
        const size_t q = (size_t)a.ms * a.B;
        c[0] = sh.ns[s]; c[q] = sh.nbs[s]; c[2 * q] = sh.nfs[s]; c[3 * q] = sh.nes[s];
    }
    return true;
}

// A sequence's stages, by one CTA or, for long sequences, a cluster of SEQ_CLUSTER CTAs: stage 0 a slice per CTA
// (one SM issues about 1500 instructions per 32 tokens of it: 25 us of an 8192-token sequence on one CTA), then
// the stages above it on the first CTA beside the records of stage 0's blocks on the others, each by the CTA that
// holds its first row.
// Shared memory: 7 bytes per token of the slice (parents, counts, prefix sums, places in the family), `pool` for the
// upper stages.
__global__ void __launch_bounds__(512) k_seq(const SeqArgs a) {
    pdl_wait();
    pdl_launch_dependents();
    extern __shared__ __align__(16) uint16_t s_dyn[];
    __shared__ SeqShared sh;
    Slice c;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(c.rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(c.cs));
    const int b = blockIdx.x / c.cs, t = threadIdx.x, lane = t & 31, w = t >> 5, nw = blockDim.x >> 5;
    const int c0 = a.cu[b], c1 = a.cu[b + 1];
    c.s0 = min(max(c0, 0), a.T);
    c.L = min(max(c1, c.s0), a.T) - c.s0;
    c.sl = 5;
    while (((long long)c.cs << c.sl) < c.L) ++c.sl;
    c.e0 = min((int)(c.rank << c.sl), c.L);
    c.ne = min(1 << c.sl, c.L - c.e0);
    const bool first = c.rank == 0;
    if (t == 0) {
        sh.err = 0; sh.err_pos = 0; sh.real = 0; sh.flag0 = 0; sh.nnz = 0; sh.nnz_upper = 0; sh.vis = 0;
        if (first) {
            if (c1 < c0 || c0 < 0 || c1 > a.T || (b == 0 && c0 != 0) || (b == a.B - 1 && c1 != a.T)) seq_fail(&sh, b);
            int *p = a.counts + b;          // stage 0's sums over the CTAs: cleared behind two barriers, added to at the end
            const size_t q = (size_t)a.ms * a.B;
            p[2 * q] = 0; p[3 * q] = 0;
            a.info[b].visited = 0;
            a.scu[b] = c0;
            if (b == a.B - 1) { a.scu[a.B] = c1; *a.ticket = 0; }
        }
    }
    SeqShared *sh0 = c.cs > 1 ? map_rank(&sh, 0) : &sh;
    const int slot = block_slot(c.s0, b, a.bmin);
    const int piece = a.cap / c.cs;
    uint16_t *U = s_dyn + 3 * piece;
    uint8_t *fu = reinterpret_cast<uint8_t *>(U + 6 * a.uc), *f0 = reinterpret_cast<uint8_t *>(U) + a.pool;
    const bool in_smem = c.L <= a.cap;
    const Sliced X{s_dyn, c.sl, c.rank}, Y{s_dyn + piece, c.sl, c.rank}, Z{s_dyn + 2 * piece, c.sl, c.rank};
    uint32_t *G[NGLOB];
    for (int i = 0; i < NGLOB; ++i) G[i] = a.glob + a.glob_stride * i + c.s0;
    if (!in_smem) f0 = reinterpret_cast<uint8_t *>(a.glob + a.glob_stride * 9) + c.s0;
    uint8_t *fw = in_smem ? f0 : f0 + c.e0;
    const Flat<uint32_t> GX{G[0]}, GY{G[1]}, GZ{G[2]};
    bool root_real = false;
    if (in_smem) seq_stage0(a, sh, sh0, X, Y, Z, c, fw, root_real);
    else seq_stage0(a, sh, sh0, GX, GY, GZ, c, fw, root_real);
    seq_sync(c.cs);
    int n1;
    const int coff_ = warp_offsets(sh.ctot, c.cs, lane, n1);
    __syncthreads();
    if (w == 0 && lane < (int)c.cs) sh.ctot[lane] = coff_;          // (now the slices' offsets)
    __syncthreads();
    const bool next = sh0->flag0 != 0;
    const bool up_smem = n1 <= a.uc && c.L < 65535;
    uint16_t *P0 = c.cs > 1 ? map_rank(U, 0) : U, *T0 = P0 + a.uc;
    if (!next) {}
    else if (in_smem && up_smem) seq_compact0(a, X, Z, sh.ctot, P0, T0, c);
    else if (in_smem) seq_compact0(a, X, Z, sh.ctot, G[3], G[4], c);
    else if (up_smem) seq_compact0(a, GX, GZ, sh.ctot, P0, T0, c);
    else seq_compact0(a, GX, GZ, sh.ctot, G[3], G[4], c);
    auto fpos = [&](int e) -> int {
        if (!in_smem) return f0[e];
        const unsigned r = (unsigned)e >> c.sl;
        uint8_t *p = f0 + ((unsigned)e & ((1u << c.sl) - 1u));
        return r == c.rank ? *p : *map_rank(p, r);
    };
    seq_sync(c.cs);
    int stages = 1, res = n1, more = 0;
    const int nwu = c.cs > 1 ? nw : nw - 1;
    int4 *rec = a.recs + slot;
    int *cnt0 = a.counts + b;
    const size_t q = (size_t)a.ms * a.B;
    // In a cluster the first CTA builds the stages above 0; the others meanwhile walk stage 0 and make its records, the
    // first slice's too (of which the second CTA makes the walk's table).  The first one only arrives at their
    // barrier, and waits for it when it is done.
    if (c.cs > 1) {
        if (!first) {
#pragma unroll 1
            for (int at = 0; at < (c.rank == 1 ? 2 : 1); ++at) walk_slice(fpos, a.bm, sh, c, at ? 0u : c.rank, at);
        }
        cluster_arrive();
        if (!first) {
            cluster_wait();
            walk_starts(fpos, a.bm, sh, c, rec, cnt0 + q);
        }
    }
    if (c.cs == 1 && w == nw - 1) {
        if (lane == 0) {
            cnt0[q] = sh.own[0] = walk_blocks(f0, c.L, a.bm, sh.bst0, SB0, rec);
            sh.own_end[0] = c.L;
            sh.base = 0;
        }
    } else if (first && next) {
        const bool done = up_smem && seq_upper_all(a, sh, U, U + a.uc, reinterpret_cast<uint32_t *>(U + 2 * a.uc), a.pool - 4 * (size_t)a.uc, b, c.s0, slot, n1,
                                                   nwu, stages, res, more);
        if (done) {}
        else if (up_smem) seq_upper<uint16_t>(a, sh, U, U + a.uc, U + 2 * a.uc, U + 3 * a.uc, U + 4 * a.uc, U + 5 * a.uc, fu, b, c.s0, slot, n1, nwu, stages, res, more);
        else seq_upper<uint32_t>(a, sh, G[3], G[4], G[5], G[6], G[7], G[8], reinterpret_cast<uint8_t *>(a.glob + a.glob_stride * 10) + c.s0, b, c.s0, slot, n1, nwu, stages, res, more);
    }
    if (c.cs == 1) __syncthreads();
    else if (first) cluster_wait();
    // (the elements' arrays are written here, not where they are first known: a cluster barrier waits for the
    // CTA's outstanding stores, and the blocks cover every token)
    auto records = [&](const auto &par, const auto &cnt, const auto &pre, int f, int i0, int di) {
        const int base = f ? 0 : sh.base, nb = sh.own[f], end = sh.own_end[f];
        const int *bst = f ? sh.bstf : sh.bst0;
        using E = Elem<typename std::remove_reference_t<decltype(par)>::I>;
        make_records([&](int e, int &lo, int &hi) {
            const unsigned p = par.get(e);
            const bool root = e == 0 && root_real;
            unsigned l, h;
            const bool child = elem_range<E>(e, p, cnt.get(e), p != E::NONE ? cnt.get(p) : 0u, root, l, h);
            const bool kept = !child && (p != E::NONE || root);
            lo = (int)l; hi = (int)h;
            const bool has = h > l;
            const int g = c.s0 + e;
            reinterpret_cast<int2 *>(a.rng)[g] = make_int2(has ? c.s0 + lo : 0, has ? c.s0 + hi : 0);
            a.tok[g] = g;
            a.par[g] = p == E::NONE ? -1 : c.s0 + (int)p;
            a.up[g] = kept ? (int)pre.get(e) + sh.ctot[e >> c.sl] : -1;
            if (child) a.rank[g] = e - (int)p;       // the token's number among its siblings (hierarchical positions)
            return kept;
        }, [&](int i, int &r0, int &r1) { block_rows(bst, SB0, rec + base, i - base, nb, end, r0, r1); }, rec, base + i0, base + nb, di, lane,
           cnt0 + 2 * q, cnt0 + 3 * q, reinterpret_cast<unsigned long long *>(&a.info[b].visited));
    };
    if (c.cs == 1 || !first) {
#pragma unroll 1
        for (int f = 0; f < (c.cs > 1 ? 2 : 1); ++f) {
            // (the first slice's: to the warps that have none of their own, one CTA after the other)
            const int i0 = f ? (nw - 1 - w) * (int)(c.cs - 1) + (int)c.rank - 1 : w, di = f ? (int)(c.cs - 1) * nw : nw;
            if (in_smem) records(X, Y, Z, f, i0, di);
            else records(GX, GY, GZ, f, i0, di);
        }
    }
    if (first && t == 0) {
        int *p = cnt0;
        p[0] = c.L;
        for (int s = stages; s < a.ms; ++s) {          // beyond its own stages: its root in a block of its own
            p = a.counts + (size_t)s * a.B + b;
            p[0] = res; p[q] = res; p[2 * q] = 0; p[3 * q] = res;
        }
        SeqInfo &f = a.info[b];
        f.stages = stages; f.res = res; f.err = sh.err; f.err_pos = sh.err_pos; f.more = more; f.real = sh.real;
        f.nnz = (long long)(sh.nnz + sh.nnz_upper); f.nnz_upper = (long long)sh.nnz_upper;
        if (sh.vis) atomicAdd(reinterpret_cast<unsigned long long *>(&f.visited), sh.vis);
    }
    // (nothing passes between the CTAs here: the others' shared memory has been read.  A barrier with release
    // semantics would wait for the outstanding stores of all of them, 3000 cycles)
    __syncwarp();
    if (c.cs > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

struct FinishArgs {
    StagePtrs st[HDT_MAX_STAGES];
    const int32_t *cu;             // the index's own copy (scu of stage 0): the caller's arrays are not read behind k_seq
    int B, T, ms, bm, bmu, bmin, capnb, gy, r0, r1;   // gy: CTAs of a sequence; r0 / r1: CTAs that rank the blocks of stage 0 / of another stage
    const SeqInfo *info;
    const int *counts;
    const BatchSums *sums;         // set: k_offsets has run, and offs[2][ms][B] holds the elements and blocks before each sequence
    const int *offs;
    const int4 *recs, *el;
    const int *upl;
    long long *keys;
    int *before;
    DevHeader *hdr;
    HostHeader *host;              // pinned landing buffer
    int tell;                      // 1: HostHeader::done is sent
};

static constexpr int FT = 256;     // threads of k_finish
static constexpr int FKEYS = 4096; // blocks of a stage whose sort keys fit in shared memory

__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums over sequences [0, m) of rows row(i), i = w, w + nw, ...: four rows of a warp at a time, so that the
// loads of one pass are in flight together.  put(i, sum) runs on lane 0.
template <class Row, class Put>
__device__ __forceinline__ void row_sums(int rows, int m, int w, int nw, int lane, Row row, Put put) {
    for (int i0 = w; i0 < rows; i0 += 4 * nw) {
        int v[4] = {0, 0, 0, 0};
        for (int b = lane; b < m; b += 32)
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (i0 + k * nw < rows) v[k] += row(i0 + k * nw)[b];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int x = __reduce_add_sync(0xffffffffu, v[k]);
            if (lane == 0 && i0 + k * nw < rows) put(i0 + k * nw, x);
        }
    }
}

// Totals over the sequences by nt threads, added to sum[4] and merged into *err (the first sequence with one) and *more in
// shared memory.
__device__ __forceinline__ void seq_sums(const SeqInfo *info, int B, int t, int nt, long long *sum, int *err, int *more) {
    long long v[4] = {0, 0, 0, 0};
    for (int b = t; b < B; b += nt) {
        const SeqInfo &x = info[b];
        v[0] += x.nnz; v[1] += x.visited; v[2] += x.nnz_upper; v[3] += x.real;
        if (x.err) atomicMin(err, b);
        if (x.more) *more = 1;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[i] = warp_sum(v[i]);
        if ((t & 31) == 0) atomicAdd((unsigned long long *)&sum[i], (unsigned long long)v[i]);
    }
}

// Batches of many sequences (see hdt_build_index), between the two others: CTA i the sums and, of elements and blocks, the
// offsets of count row i; the last CTA what is summed over SeqInfo.
static constexpr int OT = 512;
__global__ void __launch_bounds__(OT) k_offsets(const SeqInfo *info, const int *counts, int B, int ms, BatchSums *sums, int *offs) {
    pdl_wait();
    pdl_launch_dependents();
    __shared__ int s_w[OT / 32], s_err, s_more, s_stages;
    __shared__ long long s_sum[4];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if ((int)blockIdx.x == 4 * ms) {
        if (t == 0) { s_err = NO_SEQ; s_more = 0; s_stages = 1; s_sum[0] = s_sum[1] = s_sum[2] = s_sum[3] = 0; }
        __syncthreads();
        seq_sums(info, B, t, OT, s_sum, &s_err, &s_more);
        int m = 1;
        for (int b = t; b < B; b += OT) m = max(m, info[b].stages);
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) atomicMax(&s_stages, m);
        __syncthreads();
        if (t == 0) {
            sums->stages = s_stages; sums->first_err = s_err; sums->more = s_more;
            sums->nnz = s_sum[0]; sums->visited = s_sum[1]; sums->nnz_upper = s_sum[2]; sums->real = s_sum[3];
        }
        return;
    }
    const int c = blockIdx.x & 3, s = blockIdx.x >> 2;
    const int *row = counts + (size_t)c * ms * B + (size_t)s * B;
    int *out = c < 2 ? offs + ((size_t)c * ms + s) * B : nullptr;
    int run = 0;
    for (int b0 = 0; b0 < B; b0 += OT) {
        const int x = b0 + t < B ? row[b0 + t] : 0;
        int v = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += y; }
        if (lane == 31) s_w[w] = v;
        __syncthreads();
        int all;
        const int before = __shfl_sync(0xffffffffu, warp_offsets(s_w, OT / 32, lane, all), w);
        if (out != nullptr && b0 + t < B) out[b0 + t] = run + before + v - x;
        run += all;
        __syncthreads();
    }
    if (t == 0) sums->count[s][c] = run;
}

// Header: totals over the sequences.  The words go to the workspace (kernels read them there) and to the host.
__device__ void finish_header(const FinishArgs &f, int S) {
    volatile HostHeader *host = f.host;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    __shared__ int s_err, s_more;
    __shared__ long long s_sum[4];
    if (t == 0) { s_err = NO_SEQ; s_more = 0; s_sum[0] = s_sum[1] = s_sum[2] = s_sum[3] = 0; }
    __syncthreads();
    const size_t q = (size_t)f.ms * f.B;
    auto put_count = [&](int i, int v) {
        StageDesc &d = f.hdr->st[i >> 2];
        const int c = i & 3;
        int *pd = c == 0 ? &d.n : c == 1 ? &d.nb : c == 2 ? &d.n_fused : &d.n_empty;
        *pd = v;
        host->st[i >> 2][c] = v;
    };
    if (f.sums != nullptr) {
        if (t < 4 * S) put_count(t, f.sums->count[t >> 2][t & 3]);
        if (t == 0) {
            s_err = f.sums->first_err; s_more = f.sums->more;
            s_sum[0] = f.sums->nnz; s_sum[1] = f.sums->visited; s_sum[2] = f.sums->nnz_upper; s_sum[3] = f.sums->real;
        }
    } else {
        row_sums(4 * S, f.B, w, FT / 32, lane, [&](int i) { return f.counts + (i & 3) * q + (size_t)(i >> 2) * f.B; }, put_count);
        seq_sums(f.info, f.B, t, FT, s_sum, &s_err, &s_more);
    }
    __syncthreads();
    if (t <= HDT_MAX_STAGES) {
        const int more = (t + 1 < S) || (t + 1 == S && s_more);
        f.hdr->st[t].has_next = more;
        if (t < f.ms) host->st[t][4] = more;
        if (t >= S) {
            StageDesc &d = f.hdr->st[t];
            d.n = d.nb = d.n_fused = d.n_empty = 0;
            if (t < f.ms) for (int c = 0; c < 4; ++c) host->st[t][c] = 0;
        }
    }
    if (t == 0) {
        int err = 0, pos = 0;
        if (f.B == 0) { f.st[0].scu[0] = f.cu[0]; if (f.cu[0] != 0 || f.T != 0) err = HDT_ERR_BAD_HIERARCHY; }
        else if (s_err != NO_SEQ) { err = f.info[s_err].err; pos = f.info[s_err].err_pos; }
        f.hdr->status = err; f.hdr->err_pos = pos; f.hdr->nnz = s_sum[0]; f.hdr->visited = s_sum[1]; f.hdr->nnz_upper = s_sum[2]; f.hdr->real = s_sum[3];
        host->status = err; host->err_pos = pos;
        for (int i = 0; i < HostHeader::TOTALS; ++i)
            for (int k = 0; k < 3; ++k) host->total[i][k] = (int)((s_sum[i] >> (30 * k)) & 0x3fffffff);
    }
}

// cost << 1 | SELF non-EMPTY
__device__ __forceinline__ long long block_key(const int4 &r) {
    const int fl = r.w >> 8;
    return ((long long)(r.w & 255) * (r.z - r.y)) * 2 + ((fl & HDT_BLK_SELF) && !(fl & HDT_BLK_EMPTY) ? 1 : 0);
}

// Large batches (see hdt_build_index): the blocks of a stage in runs of SORT_RUN, each sorted by one CTA.  keys: descending cost,
// then id, as one ascending number (SORT_COST - cost) << 12 | place in the run << 1 | SELF non-EMPTY; before: how
// many of the last kind come before an entry in its run.
static constexpr int SORT_RUN = 1024, ST = 512;
static constexpr long long SORT_COST = (1LL << 40) - 1;     // (128 rows x 2^31 keys at most)
__global__ void __launch_bounds__(ST) k_sort(const FinishArgs f) {
    pdl_wait();
    pdl_launch_dependents();
    __shared__ long long s_key[SORT_RUN];
    __shared__ int s_w[ST / 32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, s = blockIdx.y, j0 = blockIdx.x * SORT_RUN;
    const int nb = f.sums->count[s][1], n = min(SORT_RUN, nb - j0);
    if (f.sums->first_err != NO_SEQ || s >= f.sums->stages || n <= 0) return;
    const int *offs = f.offs + ((size_t)f.ms + s) * f.B;
    for (int i = t; i < SORT_RUN; i += ST) {
        long long k = LLONG_MAX;
        if (i < n) {
            int lo = 0, hi = f.B;        // its sequence is the last one that starts at or before it
            while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (offs[mid] <= j0 + i) lo = mid; else hi = mid; }
            k = 0;                       // (beyond its own stages a sequence has its root alone, in a block without keys: cost 0)
            if (s < f.info[lo].stages)
                k = block_key(f.recs[(size_t)s * f.capnb + block_slot(min(max(f.cu[lo], 0), f.T), lo, f.bmin) + (j0 + i - offs[lo])]);
            k = (SORT_COST - (k >> 1)) << 12 | (long long)i << 1 | (k & 1);
        }
        s_key[i] = k;
    }
    __syncthreads();
    for (int len = 2; len <= SORT_RUN; len *= 2)
        for (int d = len / 2; d > 0; d /= 2) {
            for (int i = t; i < SORT_RUN / 2; i += ST) {
                const int a = 2 * i - (i & (d - 1)), b = a + d;
                const long long x = s_key[a], y = s_key[b];
                if ((x > y) == ((a & len) == 0)) { s_key[a] = y; s_key[b] = x; }
            }
            __syncthreads();
        }
    constexpr int PER = SORT_RUN / ST;
    int c = 0;
    for (int i = 0; i < PER; ++i) if (PER * t + i < n) c += (int)(s_key[PER * t + i] & 1);
    int v = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += y; }
    if (lane == 31) s_w[w] = v;
    __syncthreads();
    int all;
    int run = __shfl_sync(0xffffffffu, warp_offsets(s_w, ST / 32, lane, all), w) + v - c;
    const size_t base = (size_t)s * f.capnb + j0;
    for (int i = PER * t; i < min(PER * t + PER, n); ++i) {
        f.before[base + i] = run;
        run += (int)(s_key[i] & 1);
    }
    for (int i = t; i < n; i += ST) f.keys[base + i] = s_key[i];
}

// The ranks from the sorted runs, eight lanes a block: its place in its own run and, by bisection, in the others.
__device__ void finish_merge(const FinishArgs &f, int s, int part, int parts) {
    const int t = threadIdx.x, sub = t & 7, nb = f.sums->count[s][1], n_fused = f.sums->count[s][2];
    const int runs = (nb + SORT_RUN - 1) / SORT_RUN;
    const long long *keys = f.keys + (size_t)s * f.capnb;
    const int *before = f.before + (size_t)s * f.capnb;
    for (int g0 = part * (FT / 8); g0 < nb; g0 += parts * (FT / 8)) {
        const int g = g0 + (t >> 3), u = g / SORT_RUN;
        int rank = 0, fused = 0;
        long long key = 0;
        if (g < nb) {
            key = keys[g];
            for (int r = sub; r < runs; r += 8) {
                const int r0 = r * SORT_RUN, r1 = min(r0 + SORT_RUN, nb);
                int p = g;
                if (r != u) {        // entries of run r before this one: larger cost, or the same in an earlier run
                    const long long bound = ((key >> 12) + (r < u ? 1 : 0)) << 12;
                    int lo = r0, hi = r1;
                    while (lo < hi) { const int mid = (lo + hi) >> 1; if (keys[mid] < bound) lo = mid + 1; else hi = mid; }
                    p = lo;
                }
                rank += p - r0;
                fused += p < r1 ? before[p] : before[r1 - 1] + (int)(keys[r1 - 1] & 1);
            }
        }
#pragma unroll
        for (int o = 1; o < 8; o *= 2) {
            rank += __shfl_xor_sync(0xffffffffu, rank, o);
            fused += __shfl_xor_sync(0xffffffffu, fused, o);
        }
        if (g < nb && sub == 0) {
            const int id = u * SORT_RUN + (int)((key >> 1) & (SORT_RUN - 1));
            f.st[s].queue[rank] = id;
            f.st[s].queue_split[(key & 1) ? fused : n_fused + rank - fused] = id;
        }
    }
}

// Rank sort of a stage's blocks: queue[rank] = block id, cost descending, id ascending.  queue_split:
// the same order inside two groups, blocks that are SELF and not EMPTY first, then the others.
// Every CTA gathers all keys (cost << 1 | SELF non-EMPTY), a warp ranks a block at a time.
__device__ void finish_rank(const FinishArgs &f, int s, int part, int parts, long long *s_keys) {
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, nw = FT / 32;
    __shared__ int s_base[FT], s_slot[FT], s_w[FT / 32];
    const int *cb = f.counts + (size_t)f.ms * f.B + (size_t)s * f.B;
    int nb = 0;
    for (int b = t; b < f.B; b += FT) nb += cb[b];
    nb = __reduce_add_sync(0xffffffffu, nb);
    if (lane == 0) s_w[w] = nb;
    __syncthreads();
    nb = 0;
    for (int i = 0; i < nw; ++i) nb += s_w[i];
    __syncthreads();
    long long *keys = nb <= FKEYS ? s_keys : f.keys + (size_t)s * f.capnb;    // (every CTA of the stage writes the same values)
    int run = 0;
    for (int b0 = 0; b0 < f.B; b0 += FT) {
        const int b = b0 + t, c = b < f.B ? cb[b] : 0;
        int v = c;
        for (int o = 1; o < 32; o <<= 1) { const int x = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += x; }
        if (lane == 31) s_w[w] = v;
        // (beyond its own stages a sequence has its root alone, in a block without keys: cost 0)
        s_slot[t] = (b < f.B && s < f.info[b].stages) ? block_slot(min(max(f.cu[b], 0), f.T), b, f.bmin) : -1;
        __syncthreads();
        int off = run, all = 0;
        for (int i = 0; i < nw; ++i) { if (i < w) off += s_w[i]; all += s_w[i]; }
        s_base[t] = off + v - c;
        __syncthreads();
        // a thread per block; its sequence is the last one that starts at or before it (an empty one has the base of its successor)
        for (int j = run + t; j < run + all; j += FT) {
            int lo = 0, hi = FT;
            while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (s_base[mid] <= j) lo = mid; else hi = mid; }
            keys[j] = s_slot[lo] >= 0 ? block_key(f.recs[(size_t)s * f.capnb + s_slot[lo] + (j - s_base[lo])]) : 0;
        }
        run += all;
        __syncthreads();
    }
    for (int i = part * nw + w; i < nb; i += nw * parts) {
        const long long ki = keys[i];
        int rank = 0, rank2 = 0;
        for (int j = lane; j < nb; j += 32) {
            const long long kj = keys[j];
            const int before = ((kj >> 1) > (ki >> 1)) || ((kj >> 1) == (ki >> 1) && j < i);
            rank += before;
            rank2 += ((kj & 1) > (ki & 1)) || ((kj & 1) == (ki & 1) && before);
        }
        rank = __reduce_add_sync(0xffffffffu, rank);
        rank2 = __reduce_add_sync(0xffffffffu, rank2);
        if (lane == 0) {
            f.st[s].queue[rank] = i;
            f.st[s].queue_split[rank2] = i;
        }
    }
}

// CTA 0: header; then r0 CTAs rank stage 0's blocks and r1 each those of the other stages; then gy
// CTAs per sequence move its elements and block records to their place in the batch's arrays.
__device__ __forceinline__ void finish_part(const FinishArgs &f) {
    __shared__ long long s_keys[FKEYS];
    __shared__ int s_stages, s_bad;
    __shared__ int s_n[HDT_MAX_STAGES], s_b[HDT_MAX_STAGES], s_cn[HDT_MAX_STAGES], s_cb[HDT_MAX_STAGES];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, nw = FT / 32;
    const int first_seq = 1 + f.r0 + f.r1 * (f.ms - 1);
    const bool seq = (int)blockIdx.x >= first_seq;
    const int b = seq ? ((int)blockIdx.x - first_seq) / f.gy : 0, y = seq ? ((int)blockIdx.x - first_seq) % f.gy : 0;
    const size_t q = (size_t)f.ms * f.B;
    if (t == 0) { s_stages = 1; s_bad = 0; }
    __syncthreads();
    int s0 = 0, L = 0;
    pdl_wait();
    // One round of loads: the stages of the batch and its errors; in a sequence's CTA also the sums over the
    // sequences before it (elements and blocks of every stage) and its own numbers.
    int m = 1, bad = 0;
    SeqInfo info{};
    if (seq) {
        s0 = f.cu[b];
        L = f.cu[b + 1] - s0;
        info = f.info[b];
        if (t < f.ms) {
            s_cn[t] = f.counts[(size_t)t * f.B + b];
            s_cb[t] = f.counts[q + (size_t)t * f.B + b];
        }
    }
    if (f.sums != nullptr) {
        m = f.sums->stages;
        bad = f.sums->first_err != NO_SEQ;
        if (seq && t < f.ms) {
            s_n[t] = f.offs[(size_t)t * f.B + b];
            s_b[t] = f.offs[q + (size_t)t * f.B + b];
        }
    } else {
        for (int i = t; i < f.B; i += FT) { m = max(m, f.info[i].stages); bad |= f.info[i].err; }
    }
    if (seq && f.sums == nullptr)
        row_sums(2 * f.ms, b, w, nw, lane, [&](int i) { return f.counts + ((i & 1) ? q : 0) + (size_t)(i >> 1) * f.B; },
                 [&](int i, int v) {
                     if (i & 1) s_b[i >> 1] = v;
                     else s_n[i >> 1] = v;
                 });
    m = __reduce_max_sync(0xffffffffu, m);
    bad = __any_sync(0xffffffffu, bad);
    if (lane == 0) { atomicMax(&s_stages, m); if (bad) s_bad = 1; }
    __syncthreads();
    const int S = s_stages;
    int id = blockIdx.x;
    if (id == 0) { finish_header(f, S); return; }
    if (s_bad) return;               // (offsets of a broken hierarchy mean nothing)
    id -= 1;
    if (!seq) {
        const int s = id < f.r0 ? 0 : (id - f.r0) / f.r1 + 1, parts = s ? f.r1 : f.r0, part = s ? (id - f.r0) % f.r1 : id;
        if (s >= S) return;
        if (f.sums != nullptr) finish_merge(f, s, part, parts);
        else finish_rank(f, s, part, parts, s_keys);
        return;
    }
    const int step = FT * f.gy, me = y * FT + t;
    const int slot = block_slot(s0, b, f.bmin);
    {
        int *up = f.st[0].up;
        const int off = S > 1 ? s_n[1] : 0;
        for (int e = me; e < L; e += 4 * step) {
            int v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = e + k * step < L ? up[s0 + e + k * step] : -1;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (v[k] >= 0) up[s0 + e + k * step] = S > 1 ? v[k] + off : -1;
        }
    }
    // stage 0's records by all threads, then a stage per warp (deep trees have twenty small ones)
    auto put_records = [&](int s, int i0, int di) {
        const StagePtrs &P = f.st[s];
        const int off = s ? s_n[s] : s0, boff = s_b[s];
        const int4 *rec = f.recs + (size_t)s * f.capnb + slot;
        for (int i = i0; i < s_cb[s]; i += di) {
            const int4 r = rec[i];
            int fl = r.w >> 8;
            if (s + 1 == S) fl &= ~HDT_BLK_CARRY;
            int *o = P.blocks + 5 * (size_t)(boff + i);
            o[0] = off + r.x; o[1] = off + r.x + (r.w & 255); o[2] = off + r.y; o[3] = off + r.z; o[4] = fl;
        }
    };
    put_records(0, me, step);
    const int split = S > 4 ? 1 : nw / max(S - 1, 1);      // warps that share a stage of a hierarchy of few
    for (int s = 1 + w / split; s < S; s += nw / split) {
        const StagePtrs &P = f.st[s];
        const int off = s_n[s], n = s_cn[s];
        const bool last = s + 1 == S;
        const int noff = last ? 0 : s_n[s + 1];
        const int i0 = (y * split + w % split) * 32 + lane, di = f.gy * split * 32;
        if (i0 == 0) {
            P.scu[b] = off;
            if (b == f.B - 1) P.scu[f.B] = off + n;
        }
        if (s < info.stages) {
            const int4 *el = f.el + (size_t)(s - 1) * f.T + s0;
            const int *upl = f.upl + (size_t)(s - 1) * f.T + s0;
            for (int e = i0; e < n; e += di) {
                const int4 x = el[e];
                const int u = upl[e];
                const bool has = x.w > x.z;
                P.tok[off + e] = s0 + x.x;
                P.par[off + e] = x.y < 0 ? -1 : off + x.y;
                reinterpret_cast<int2 *>(P.rng)[off + e] = make_int2(has ? off + x.z : 0, has ? off + x.w : 0);
                P.up[off + e] = (u < 0 || last) ? -1 : u + noff;
            }
            put_records(s, i0, di);
        } else if (info.res && i0 == 0) {       // (res is 0 or 1 here)
            P.tok[off] = s0;
            P.par[off] = -1;
            reinterpret_cast<int2 *>(P.rng)[off] = make_int2(0, 0);
            P.up[off] = last ? -1 : noff;
            int *o = P.blocks + 5 * (size_t)s_b[s];
            o[0] = off; o[1] = off + 1; o[2] = off; o[3] = off;
            o[4] = HDT_BLK_SELF | HDT_BLK_EMPTY | (last ? 0 : HDT_BLK_CARRY);
        }
    }
}

// The header's words go straight to the host's pinned buffer, which the host watches, so no copy has to be queued behind
// the build.  A build that is waited for also says when it has ended (`tell`): every CTA's fence and ticket stand behind
// its writes, so the word of the CTA that is last stands behind all of them.  That makes the kernel 2 us longer, which
// the host's way to the next call hides there, but not where the attention is queued behind it already (deferred builds).
__global__ void __launch_bounds__(FT) k_finish(const FinishArgs f) {
    pdl_launch_dependents();
    finish_part(f);
    if (!f.tell) return;
    __syncthreads();
    if (threadIdx.x != 0) return;
    __threadfence();
    if (gridDim.x > 1 && atomicAdd(&f.hdr->ticket, 1) != (int)gridDim.x - 1) return;      // (alone: no sequences, no k_seq that cleared the ticket)
    __threadfence_system();
    *(volatile int *)&f.host->done = 1;
}

}  // namespace hdt

using namespace hdt;

static int norm_dirs(const hdt_index_params_t *p) { return p ? (~p->mask_off) & 7 : 7; }

static void norm_params(const hdt_index_params_t *p, int &bm, int &ms, int &bmu) {
    bm = (p && p->block_m) ? p->block_m : 128;
    ms = (p && p->max_stages) ? p->max_stages : 4;
    bmu = (p && p->block_m_upper) ? p->block_m_upper : 128;
}

extern "C" size_t hdt_index_workspace_bytes(int32_t batch, int32_t total_tokens,
                                            const hdt_index_params_t *params) {
    int bm, ms, bmu;
    norm_params(params, bm, ms, bmu);
    if (batch < 0 || total_tokens < 0 || bm < 1 || bm > 128 || bmu < 1 || bmu > 128 || ms < 1 || ms > HDT_MAX_STAGES)
        return 0;
    return make_layout(batch, total_tokens, min(bm, bmu), ms).total;
}

// Pinned landing buffers for index headers: a small pool shared by all host threads (an index keeps
// its buffer until the header has been read).
static std::mutex g_pinned_mu;
static std::vector<HostHeader *> g_pinned_free;
static HostHeader *pinned_acquire() {
    {
        std::lock_guard<std::mutex> lk(g_pinned_mu);
        if (!g_pinned_free.empty()) {
            HostHeader *p = g_pinned_free.back();
            g_pinned_free.pop_back();
            return p;
        }
    }
    HostHeader *p = nullptr;
    if (cudaHostAlloc((void **)&p, sizeof(HostHeader), cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
        (void)cudaGetLastError();
        return nullptr;
    }
    return p;
}
static void pinned_release(HostHeader *p) {
    if (!p) return;
    std::lock_guard<std::mutex> lk(g_pinned_mu);
    g_pinned_free.push_back(p);
}

// Waits for all that is on the stream, also where another stream of this thread is being captured.  A stream that is being
// captured itself takes no wait, and needs none: what is captured on it runs behind what it holds.
static cudaError_t stream_passed(cudaStream_t st) {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaError_t e = cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) return e;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing(st, &cap);
    if (e == cudaSuccess && cap == cudaStreamCaptureStatusNone) e = cudaStreamSynchronize(st);
    const cudaError_t back = cudaThreadExchangeStreamCaptureMode(&mode);
    return e != cudaSuccess ? e : back;
}

// The counts that attention calls need, from the header.
static void index_counts(hdt_index *ix, const HostHeader &h) {
    ix->failed = h.status;
    ix->err_pos = h.err_pos;
    if (h.status != 0) return;
    int ns = 1;
    while (ns < ix->max_stages && h.st[ns][0] > 0) ++ns;
    if (h.st[ns - 1][4] && ns == ix->max_stages) {
        ix->failed = HDT_ERR_BAD_HIERARCHY;
        ix->err_pos = -1;
        return;
    }
    ix->n_stages = ns;
    auto total = [&](int i) { return (int64_t)h.total[i][0] | (int64_t)h.total[i][1] << 30 | (int64_t)h.total[i][2] << 60; };
    ix->nnz = total(0);
    ix->visited = total(1);
    ix->nnz_upper = total(2);
    ix->real = total(3);
    for (int s = 0; s <= HDT_MAX_STAGES; ++s) {
        StageDesc &d = ix->desc[s];
        d = StageDesc{};
        if (s >= ix->max_stages) continue;
        d.n = h.st[s][0]; d.nb = h.st[s][1]; d.n_fused = h.st[s][2]; d.n_empty = h.st[s][3]; d.has_next = h.st[s][4];
    }
}

// Batches whose offsets and ranks take two kernels more.  In k_finish alone every CTA of a sequence sums the counts of all
// sequences before it and every block is compared with every other: work that grows with their squares.  The line is in
// blocks (T / bm + B is about their number) and lies between the sizes timed, us without and with the two kernels: trees of
// 370 tokens 200 (780) 49.8 and 57.0, 300 (1170) 81.6 and 59.7, 6400 14100 and 664; 8192 tokens 16 (1040) 43.1 and 48.2, 24
// (1560) 57.7 and 49.0, 256 3540 and 289; 1024 tokens 64 (576) 40.4 and 45.5, 128 (1152) 81.3 and 72.3; 128 tokens 512 (1024)
// 34.1 and 42.0, 768 (1540) 53.0 and 56.5, 1024 (2050) 71.2 and 66.5.
static bool many_blocks(int B, int T, int bm) { return B > 0 && (long long)T / bm + B > 1100; }

extern "C" int hdt_build_index(const int8_t *level, const int32_t *parent, const int32_t *cu_seqlens,
                               int32_t batch, int32_t total_tokens, const hdt_index_params_t *params,
                               void *workspace, size_t workspace_bytes, void *stream, hdt_index_t **out) {
    if (out) *out = nullptr;
    int bm, ms, bmu;
    norm_params(params, bm, ms, bmu);
    const int dirs = norm_dirs(params);
    if (!out || !cu_seqlens || !workspace || batch < 0 || total_tokens < 0 ||
        (total_tokens > 0 && (!level || !parent)))
        return set_error(HDT_ERR_INVALID_ARG, "hdt_build_index: null pointer or negative size");
    if (bm < 1 || bm > 128 || bmu < 1 || bmu > 128 || ms < 1 || ms > HDT_MAX_STAGES)
        return set_error(HDT_ERR_INVALID_ARG, "hdt_build_index: block_m, block_m_upper must be 1..128, max_stages 1..%d",
                         HDT_MAX_STAGES);
    if (params && (params->mask_off & ~7))
        return set_error(HDT_ERR_INVALID_ARG, "hdt_build_index: mask_off has bits outside 0..7");
    if (((uintptr_t)workspace & 255) != 0)
        return set_error(HDT_ERR_INVALID_ARG, "hdt_build_index: workspace must be 256-byte aligned");
    const int B = batch, T = total_tokens;
    const int bmin = min(bm, bmu);
    const Layout L = make_layout(B, T, bmin, ms);
    if (workspace_bytes < L.total)
        return set_error(HDT_ERR_WORKSPACE, "hdt_build_index: workspace %zu < required %zu", workspace_bytes,
                         L.total);
    cudaStream_t st = (cudaStream_t)stream;
    char *ws = (char *)workspace;

    // Shared memory of k_seq.  The host knows the mean length, not the longest: room for four times the
    // mean (documents of one batch differ that much; a longer one works in the workspace), in powers of
    // two up to SEQ_CAP_MAX.  Upper stages: as many elements as tokens up to UC_MAX (deep trees keep most of
    // their tokens above stage 0, documents a few percent).  One CTA where a mean sequence is an element
    // or two per thread of it, else a cluster.
    const long long mean = B > 0 ? ((long long)T + B - 1) / B : 0;
    const long long want = B == 1 ? T : 4 * mean;
    int cap = 1024;
    while (cap < want && cap < SEQ_CAP_MAX) cap *= 2;
    const int cs = mean > 768 ? SEQ_CLUSTER : 1, threads = 512;
    SeqArgs a{};
    a.cap = cap;
    a.uc = min(cap, UC_MAX);
    a.pool = (cap <= 2048 ? 32 : 16) * a.uc;       // (13 at least, for the stages one by one)
    const size_t smem = 7 * (size_t)(cap / cs) + a.pool;
    static constexpr size_t kSmemMax = 7 * 4096 + 16 * UC_MAX;
    static DevOnce attr_done;
    if (!attr_done.done()) {
        HDT_CUDA_CHECK(cudaFuncSetAttribute(k_seq, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
        attr_done.set();
    }
    HostHeader *hp = pinned_acquire();
    if (!hp) return set_error(HDT_ERR_CUDA, "hdt_build_index: no pinned host memory for the index header");
    hp->done = HostHeader::UNSET;
    for (int i = 0; i < HostHeader::words(ms); ++i) (&hp->status)[i] = HostHeader::UNSET;

    hdt_index *ix = new hdt_index();
    ix->batch = B; ix->total_tokens = T; ix->block_m = bm; ix->block_m_upper = bmu; ix->n_stages = 0;
    ix->directions = dirs;
    ix->workspace = workspace; ix->workspace_bytes = workspace_bytes;
    ix->rank = (const int *)(ws + L.rank);
    for (int s = 0; s < ms; ++s) {
        char *base = ws + L.stage0 + L.stage_stride * (size_t)s;
        ix->st[s] = StagePtrs{(int *)(base + L.s_tok), (int *)(base + L.s_par), (int *)(base + L.s_rng),
                              (int *)(base + L.s_up), (int *)(base + L.s_scu), (int *)(base + L.s_blocks),
                              (int *)(base + L.s_queue), (int *)(base + L.s_queue2)};
    }
    ix->h_pinned = hp;
    ix->hdr_dev = (const DevHeader *)(ws + L.header);
    ix->stream = st;
    ix->max_stages = ms;
    const bool deferred = params && params->deferred;
    ix->tells = !deferred || st == cudaStreamPerThread;
    ix->state.store(INDEX_QUEUED, std::memory_order_relaxed);

    a.level = level; a.parent = parent; a.cu = cu_seqlens;
    a.B = B; a.T = T; a.ms = ms; a.bm = bm; a.bmu = bmu; a.bmin = bmin; a.dirs = dirs;
    a.tok = ix->st[0].tok; a.par = ix->st[0].par; a.rng = ix->st[0].rng; a.up = ix->st[0].up; a.scu = ix->st[0].scu;
    a.rank = (int *)(ws + L.rank);
    a.info = (SeqInfo *)(ws + L.info);
    a.counts = (int *)(ws + L.counts);
    a.recs = (int4 *)(ws + L.recs);
    a.capnb = L.capnb;
    a.ticket = &((DevHeader *)(ws + L.header))->ticket;
    a.el = (int4 *)(ws + L.el);
    a.upl = (int *)(ws + L.upl);
    a.glob = (uint32_t *)(ws + L.glob);
    a.glob_stride = al(sizeof(int) * (size_t)T) / sizeof(int);
    FinishArgs f{};
    for (int s = 0; s < ms; ++s) f.st[s] = ix->st[s];
    f.cu = B > 0 ? ix->st[0].scu : cu_seqlens; f.B = B; f.T = T; f.ms = ms; f.bm = bm; f.bmu = bmu; f.bmin = bmin; f.capnb = L.capnb;
    f.gy = (int)min(16LL, max(1LL, mean / 2048));
    f.r0 = max(1, min(64, L.capnb / 16));
    f.r1 = ms > 4 ? max(1, min(8, L.capnb / 128)) : max(1, min(16, L.capnb / 64));
    if (many_blocks(B, T, bmin)) {
        f.sums = (const BatchSums *)(ws + L.sums);
        f.offs = (const int *)(ws + L.offs);
        f.r0 = max(f.r0, min(512, L.capnb / 64));
        f.r1 = max(f.r1, min(ms > 4 ? 32 : 128, L.capnb / 512));
    }
    f.info = a.info; f.counts = a.counts; f.recs = a.recs; f.el = a.el; f.upl = a.upl;
    f.keys = (long long *)(ws + L.keys);
    f.before = (int *)(ws + L.before);
    f.hdr = (DevHeader *)(ws + L.header);
    f.host = hp;
    f.tell = ix->tells;
    cudaError_t e = cudaSuccess;
    {
        ProfScope ps(PROF_INDEX, st);
        if (B > 0) {
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3((unsigned)(B * cs));
            cfg.blockDim = dim3(threads);
            cfg.dynamicSmemBytes = smem;
            cfg.stream = st;
            cudaLaunchAttribute at[2];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = cs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
            at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            at[1].val.programmaticStreamSerializationAllowed = g_no_pdl ? 0 : 1;
            cfg.attrs = at;
            cfg.numAttrs = 2;
            e = cudaLaunchKernelEx(&cfg, k_seq, a);
            count_launch();
        }
        if (e == cudaSuccess && f.sums != nullptr)
            e = launch_dependent(k_offsets, true, dim3(4 * ms + 1), OT, 0, st, a.info, a.counts, B, ms, (BatchSums *)(ws + L.sums), (int *)(ws + L.offs));
        if (e == cudaSuccess && f.sums != nullptr)
            e = launch_dependent(k_sort, true, dim3((L.capnb + SORT_RUN - 1) / SORT_RUN, ms), ST, 0, st, f);
        if (e == cudaSuccess) {
            // a programmatic dependent: its CTAs are scheduled while k_seq runs and wait for its end
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3(B > 0 ? (unsigned)(1 + f.r0 + f.r1 * (ms - 1) + (size_t)B * f.gy) : 1u);
            cfg.blockDim = dim3(FT);
            cfg.stream = st;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            at[0].val.programmaticStreamSerializationAllowed = g_no_pdl ? 0 : 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            e = cudaLaunchKernelEx(&cfg, k_finish, f);
            count_launch();
        }
    }
    if (e != cudaSuccess) {
        pinned_release(hp);
        delete ix;
        return set_error(HDT_ERR_CUDA, "hdt_build_index: launch failed: %s", cudaGetErrorString(e));
    }
    if (!deferred) {
        const int rc = index_wait(ix, INDEX_COUNTED);
        if (rc) {
            (void)hdt_index_destroy(ix);
            return rc;
        }
    }
    *out = ix;
    return HDT_OK;
}

namespace hdt {
// (the per-thread default stream has one handle and is another stream in every thread)
bool index_on_stream(const hdt_index *ix, cudaStream_t st) { return st == ix->stream && st != cudaStreamPerThread; }

int index_wait(const hdt_index *cix, IndexState want) {
    hdt_index *ix = const_cast<hdt_index *>(cix);
    if (ix->state.load(std::memory_order_acquire) < want) {
        std::lock_guard<std::mutex> lk(ix->mu);
        HostHeader *hp = ix->h_pinned;
        // The host watches words of the pinned header.  After a bounded number of looks it waits for the stream instead.
        auto watch = [&](int *first, int n) {
            const volatile int *words = first;
            int got = 0;
            auto look = [&]() {
                while (got < n && words[got] != HostHeader::UNSET) ++got;
                return got == n;
            };
            for (long long spin = 0; spin < 20000000LL && !look(); ++spin) {}
            cudaError_t e = cudaSuccess;
            if (!look()) {
                e = cudaStreamSynchronize(ix->stream);
                if (e == cudaSuccess && !look()) e = cudaErrorUnknown;
            }
            std::atomic_thread_fence(std::memory_order_acquire);
            return e;
        };
        cudaError_t e = cudaSuccess;
        int state = ix->state.load(std::memory_order_relaxed);
        if (state == INDEX_QUEUED) {
            e = watch(&hp->status, HostHeader::words(ix->max_stages));
            if (e == cudaSuccess) index_counts(ix, *hp);
            state = INDEX_COUNTED;
        }
        if (e == cudaSuccess && state == INDEX_COUNTED && want == INDEX_COMPLETE) {
            if (ix->tells) e = watch(&hp->done, 1);
            else e = stream_passed(ix->stream);
            state = INDEX_COMPLETE;
        }
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            ix->failed = HDT_ERR_CUDA;
            state = INDEX_COMPLETE;
        }
        if (hp != nullptr && (state == INDEX_COMPLETE || !ix->tells)) {      // nothing more comes
            ix->h_pinned = nullptr;
            pinned_release(hp);
        }
        ix->state.store(state, std::memory_order_release);
        if (e != cudaSuccess) return set_error(HDT_ERR_CUDA, "waiting for the index build failed: %s", cudaGetErrorString(e));
    }
    if (ix->failed == 0) return HDT_OK;
    if (ix->failed == HDT_ERR_BAD_HIERARCHY && ix->err_pos < 0)
        return set_error(HDT_ERR_BAD_HIERARCHY, "hdt_build_index: hierarchy needs more than max_stages = %d stages",
                         ix->max_stages);
    return set_error(ix->failed, "hdt_build_index: structure arrays violate a precondition near element %d", ix->err_pos);
}
}  // namespace hdt

extern "C" int hdt_index_info(const hdt_index_t *ix, int32_t *n_stages, int64_t *nnz, int64_t *visited) {
    if (!ix) return set_error(HDT_ERR_INVALID_ARG, "hdt_index_info: null index");
    if (const int rc = index_wait(ix, INDEX_COUNTED)) return rc;
    if (n_stages) *n_stages = ix->n_stages;
    if (nnz) *nnz = ix->nnz;
    if (visited) *visited = ix->visited;
    return HDT_OK;
}

extern "C" int hdt_index_export(const hdt_index_t *ix, int32_t stage, hdt_stage_view_t *v) {
    if (!ix || !v) return set_error(HDT_ERR_INVALID_ARG, "hdt_index_export: null argument");
    if (const int rc = index_ready(ix)) return rc;
    if (stage < 0 || stage >= ix->n_stages)
        return set_error(HDT_ERR_INVALID_ARG, "hdt_index_export: stage %d outside [0,%d)", stage, ix->n_stages);
    const StagePtrs &P = ix->st[stage];
    v->n = ix->desc[stage].n;
    v->n_blocks = ix->desc[stage].nb;
    v->tok = P.tok; v->par = P.par; v->rng = P.rng; v->up = P.up; v->scu = P.scu;
    v->blocks = P.blocks; v->queue = P.queue;
    v->queue_split = P.queue_split;
    v->n_fused = ix->desc[stage].n_fused;
    return HDT_OK;
}

extern "C" int hdt_index_destroy(hdt_index_t *ix) {
    // The header must not land in a recycled buffer; the workspace is the caller's again (of a deferred build: behind its stream).
    if (ix) (void)index_wait(ix, ix->tells ? INDEX_COMPLETE : INDEX_COUNTED);
    delete ix;
    return HDT_OK;
}
