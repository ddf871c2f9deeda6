// Device-side index builder: (level, parent, cu_seqlens) -> staged family ranges, row blocks,
// work queues.  Integer work only; every array must equal the sequential definition bit for bit.
//
// Two launches, whatever the number of stages:
//   k_seq     one CTA per sequence, its arrays in shared memory: validation, child counts, family
//             ranges, compaction to the next stage, greedy packing of row blocks, block records - for
//             all stages of the sequence, in sequence-relative numbers, beside the counts of the stage
//   k_finish  adds the sequences' offsets (sums over the sequences before it), ranks the blocks of a
//             stage by cost (longest first), and sends the header to the host
// Per stage (array of n elements in document order):
//   counts    cnt[p] = children of p, and whether one of them has children
//   ranges    a node whose children are all childless heads a family; head and children get
//             their key range; children of heads (and PAD) are removed for the next stage
//   compact   tok / par of the kept elements in the next stage's array
//   walk      greedy packing of row blocks
// What bounds it: latency (about 40 bytes a token move; a chain of barriers and shared-memory round
// trips per stage).  The stages of a sequence only meet the other sequences' in their offsets, so the
// grid-wide steps (formerly nine launches for three stages and a hundred for twenty, each a launch
// latency behind the one before) are one kernel boundary.
#include <cstdio>
#include <cstring>
#include <atomic>
#include <mutex>
#include <vector>

#include "hdt_internal.cuh"

namespace hdt {

// What k_seq leaves about one sequence for k_finish.
struct SeqInfo {
    int stages;                // stages this sequence's own hierarchy needs (at least 1)
    int res;                   // elements it still has in any later stage of the batch: its root, or nothing
    int err, err_pos;          // structure error, 0 = none
    int more, pad;             // elements were left after the last allowed stage
    long long nnz, visited;
};

struct Layout {
    size_t header, info, counts, rank, recs, el, upl, glob, keys, stage0, stage_stride;
    size_t s_tok, s_par, s_rng, s_up, s_scu, s_blocks, s_queue, s_queue2;  // offsets inside a stage
    size_t total;
    int capnb;
};

static size_t al(size_t x) { return (x + 255) & ~size_t(255); }

static constexpr int NGLOB = 9;      // element arrays of the sequences that do not fit in shared memory

static Layout make_layout(int B, int T, int bm, int max_stages) {   // bm: the smaller of the two block sizes
    Layout L;
    L.capnb = 2 * (T / bm + 1) + 4 * B + 2;
    size_t o = 0;
    L.header = o; o += al(sizeof(DevHeader));
    L.info = o; o += al(sizeof(SeqInfo) * (size_t)B);
    L.counts = o; o += al(sizeof(int) * 4 * (size_t)max_stages * B);
    L.rank = o; o += al(sizeof(int) * (size_t)T);
    L.recs = o; o += al(sizeof(int4) * (size_t)max_stages * L.capnb);
    L.keys = o; o += al(sizeof(long long) * (size_t)max_stages * L.capnb);
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
    static __device__ __forceinline__ void add(uint16_t *c, unsigned i) {
        atomicAdd(reinterpret_cast<unsigned *>(c) + (i >> 1), 1u << ((i & 1) * 16));
    }
    static __device__ __forceinline__ void flag(uint16_t *c, unsigned i) {
        atomicOr(reinterpret_cast<unsigned *>(c) + (i >> 1), FLAG << ((i & 1) * 16));
    }
};
template <> struct Elem<uint32_t> {
    static constexpr unsigned NONE = 0xffffffffu, FLAG = 0x80000000u, MASK = 0x7fffffffu;
    static __device__ __forceinline__ void add(uint32_t *c, unsigned i) { atomicAdd(c + i, 1u); }
    static __device__ __forceinline__ void flag(uint32_t *c, unsigned i) { atomicOr(c + i, FLAG); }
};

static constexpr int SEQ_CAP_MAX = 32768;   // tokens of a sequence held in shared memory (15-bit counts)
static constexpr int SB0 = 1024, SBU = 256; // block starts of stage 0 / an upper stage held in shared memory

struct SeqArgs {
    const int8_t *level;
    const int32_t *parent, *cu;
    int B, T, ms, bm, bmu, bmin, dirs;
    int cap, uc;               // tokens of stage 0 / elements of an upper stage that fit in shared memory
    int overlay;               // the upper stages' arrays lie over stage 0's prefix sums
    int *tok, *par, *rng, *up, *scu;     // stage 0 (final, but for `up`: relative to the sequence)
    int *rank;
    SeqInfo *info;
    int *counts;               // [4][ms][B]: elements, blocks, SELF non-EMPTY blocks, EMPTY blocks
    int4 *recs;                // [ms][capnb]: r0, a, b, rows | flags << 8, relative to the sequence
    int capnb;
    int4 *el;                  // [ms - 1][T]: tok, par, lo, hi of the upper stages, relative to the sequence
    int *upl;                  // [ms - 1][T]: index in the next stage, -1 = removed
    uint32_t *glob;            // NGLOB arrays of glob_stride elements
    size_t glob_stride;
};

struct SeqShared {
    int bst0[SB0], bst[SBU];
    int wtot[32], wtotu[32];
    int err, err_pos, flag0, flag, nb0, nb, nf0, ne0, nf, ne;
    unsigned long long nnz, vis;
};

__device__ __forceinline__ void seq_fail(SeqShared &sh, int pos) {
    if (atomicCAS(&sh.err, 0, HDT_ERR_BAD_HIERARCHY) == 0) sh.err_pos = pos;
}

// Barrier of the warps that build the upper stages (the last warp meanwhile walks stage 0's blocks).
__device__ __forceinline__ void bar_upper(int n) { asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory"); }

// Range and fate of one element.  root_real (stage 0 only): the sequence's first token is a root, not
// PAD; a root without children is a family of its own there.  Returns whether a family holds it as a child.
template <class I>
__device__ __forceinline__ bool elem_range(const I *par, const I *cnt, int e, bool stage0, bool root_real, unsigned &p, unsigned &lo,
                                           unsigned &hi) {
    using E = Elem<I>;
    p = par[e];
    const unsigned y = cnt[e], c = y & E::MASK;
    lo = hi = 0;
    if ((c > 0 && !(y & E::FLAG)) || (stage0 && e == 0 && c == 0 && root_real)) {
        lo = (p == E::NONE) ? e : e + 1;
        hi = e + 1 + c;
    } else if (p != E::NONE) {
        const unsigned yp = cnt[p], cp = yp & E::MASK;
        if (cp > 0 && !(yp & E::FLAG)) {
            lo = p;
            hi = p + 1 + cp;
            return true;
        }
    }
    return false;
}

// Greedy packing of row blocks (one thread): a cut that would split a family which starts inside the
// block moves to the family's head.
template <class I>
__device__ __forceinline__ int walk_blocks(const I *par, const I *cnt, int n, int bm, int *bst, int nbst, int4 *rec) {
    using E = Elem<I>;
    int pos = 0, nb = 0;
    while (pos < n) {
        int end = min(pos + bm, n);
        if (end < n) {
            const unsigned p = par[end];
            if (p != E::NONE && (int)p > pos) {
                const unsigned yp = cnt[p];
                const unsigned y = cnt[end];
                const bool head = (y & E::MASK) > 0 && !(y & E::FLAG);
                if (!head && (yp & E::MASK) > 0 && !(yp & E::FLAG)) end = (int)p;
            }
        }
        if (nb < nbst) bst[nb] = pos; else rec[nb].x = pos;
        ++nb;
        pos = end;
    }
    return nb;
}

// Block records of one stage, one warp per block.
template <class I>
__device__ __forceinline__ void make_records(const I *par, const I *cnt, int n, bool stage0, bool root_real, int nb, const int *bst, int nbst,
                                             int4 *rec, int w, int nw, int lane, int *nf, int *ne, unsigned long long *vis_out) {
    using E = Elem<I>;
    long long vis = 0;
    int mf = 0, me = 0;
    for (int i = w; i < nb; i += nw) {
        const int r0 = i < nbst ? bst[i] : rec[i].x;
        const int r1 = (i + 1 < nb) ? (i + 1 < nbst ? bst[i + 1] : rec[i + 1].x) : n;
        int a = INT_MAX, bb = INT_MIN, carry = 0;
        unsigned lo[4], hi[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int e = r0 + lane + 32 * k;
            lo[k] = hi[k] = 0;
            if (e < r1) {
                unsigned p;
                const bool child = elem_range<I>(par, cnt, e, stage0, root_real, p, lo[k], hi[k]);
                if (hi[k] > lo[k]) { a = min(a, (int)lo[k]); bb = max(bb, (int)hi[k]); }
                const bool real = !stage0 || p != E::NONE || (e == 0 && root_real);
                if (real && !child) carry = 1;
            }
        }
        a = __reduce_min_sync(0xffffffffu, a);
        bb = __reduce_max_sync(0xffffffffu, bb);
        carry = __any_sync(0xffffffffu, carry);
        const bool any = bb > a;
        if (!any) { a = r0; bb = r0; }
        int dense = 1;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (r0 + lane + 32 * k < r1 && ((int)lo[k] != a || (int)hi[k] != bb)) dense = 0;
        dense = __all_sync(0xffffffffu, dense);
        if (lane == 0) {
            int fl = 0;
            if (a >= r0 && bb <= r1) fl |= HDT_BLK_SELF;
            if (dense && any) fl |= HDT_BLK_DENSE;
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

// Stage 0 of one sequence up to the compaction, by all threads of the CTA.  X: parents, Y: counts,
// Z: levels, then prefix sums of the keep flags.  Returns the number of kept elements.
template <class I>
__device__ __forceinline__ void seq_stage0(const SeqArgs &a, SeqShared &sh, I *X, I *Y, I *Z, int s0, int L, bool root_real) {
    using E = Elem<I>;
    const int t = threadIdx.x, nt = blockDim.x, lane = t & 31, w = t >> 5, nw = nt >> 5;
    for (int e = t; e < L; e += nt) {
        const int p = a.parent[s0 + e], l = a.level[s0 + e];
        bool ok = true;
        unsigned q = E::NONE;
        if (l < 0) ok = (l == -1 && p == -1);
        else if (e == 0) ok = (l == 0 && p == -1);
        else if (l > HDT_MAX_STAGES * 8 || p < 0 || p >= e) ok = false;
        else q = (unsigned)p;
        X[e] = (I)q;
        Z[e] = (I)(uint8_t)l;
        Y[e] = 0;
        if (!ok) seq_fail(sh, s0 + e);
    }
    __syncthreads();
    for (int e = t; e < L; e += nt) {
        const unsigned p = X[e];
        const int l = (int8_t)(uint8_t)Z[e];
        if (l >= 0 && e > 0) {
            if (p != E::NONE && (int)(int8_t)(uint8_t)Z[p] != l - 1) seq_fail(sh, s0 + e);
            if ((int8_t)(uint8_t)Z[e - 1] < 0) seq_fail(sh, s0 + e);     // PAD only as a suffix
        }
        if (p != E::NONE) E::add(Y, p);
    }
    __syncthreads();
    for (int e = t; e < L; e += nt) {
        const unsigned p = X[e];
        if (p != E::NONE && (Y[e] & E::MASK) > 0) E::flag(Y, p);
    }
    __syncthreads();
    const int k = seg_shift(L, nw);
    int run = 0, next = 0;
    long long deg = 0;
    for (int i = 0; i < (1 << (k - 5)); ++i) {
        const int base = (w << k) + 32 * i, e = base + lane;
        if (base >= L) break;
        bool kp = false;
        if (e < L) {
            const bool real = (int8_t)(uint8_t)Z[e] >= 0;
            unsigned p, lo, hi;
            const bool child = elem_range<I>(X, Y, e, true, root_real, p, lo, hi);
            if (child) {
                if (!((int)p < e && e < (int)hi)) seq_fail(sh, s0 + e);
                a.rank[s0 + e] = e - (int)p;        // the token's number among its siblings (hierarchical positions)
            }
            kp = real && !child;
            const bool has = hi > lo;
            reinterpret_cast<int2 *>(a.rng)[s0 + e] = make_int2(has ? s0 + (int)lo : 0, has ? s0 + (int)hi : 0);
            a.tok[s0 + e] = s0 + e;
            a.par[s0 + e] = (p == E::NONE) ? -1 : s0 + (int)p;
            deg += row_pairs(e, (int)lo, (int)hi, a.dirs);
            if (kp && p != E::NONE) next = 1;
        }
        const unsigned m = __ballot_sync(0xffffffffu, kp);
        if (e < L) Z[e] = (I)(kp ? (unsigned)(run + __popc(m & ((1u << lane) - 1u))) : E::NONE);
        run += __popc(m);
    }
    for (int o = 16; o; o >>= 1) deg += __shfl_xor_sync(0xffffffffu, deg, o);
    next = __any_sync(0xffffffffu, next);
    if (lane == 0) {
        sh.wtot[w] = run;
        if (deg) atomicAdd(&sh.nnz, (unsigned long long)deg);
        if (next) sh.flag0 = 1;
    }
}

// Stage 0 -> stage 1: the kept elements' parents and tokens (only when the sequence has a stage 1), `up`.
template <class I, class J>
__device__ __forceinline__ void seq_compact0(const SeqArgs &a, const SeqShared &sh, const I *X, const I *Z, J *par2, J *tok2, int s0, int L, bool next) {
    using E = Elem<I>;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, nw = blockDim.x >> 5;
    const int k = seg_shift(L, nw);
    int total;
    const int wo = warp_offsets(sh.wtot, nw, lane, total);
    const int mine = __shfl_sync(0xffffffffu, wo, w);
    for (int i = 0; i < (1 << (k - 5)); ++i) {
        const int base = (w << k) + 32 * i, e = base + lane;
        if (base >= L) break;
        const unsigned z = e < L ? Z[e] : E::NONE;
        unsigned p = E::NONE, q = E::NONE;
        if (z != E::NONE) { p = X[e]; if (p != E::NONE) q = Z[p]; }
        const int wp = __shfl_sync(0xffffffffu, wo, q != E::NONE ? (int)(p >> k) : 0);
        const int u = z != E::NONE ? (int)z + mine : -1;
        if (e < L) a.up[s0 + e] = u;
        if (u >= 0 && next) {
            par2[u] = (J)(q != E::NONE ? q + (unsigned)wp : Elem<J>::NONE);
            tok2[u] = (J)e;
        }
    }
}

// All stages above 0 of one sequence, by the first nw warps of the CTA (tu threads).
template <class J>
__device__ __forceinline__ void seq_upper(const SeqArgs &a, SeqShared &sh, J *par, J *tok, J *par2, J *tok2, J *cnt, J *pre, int b, int s0,
                                          int slot, int n, int &stages, int &res, int &more) {
    using E = Elem<J>;
    const int t = threadIdx.x, tu = blockDim.x - 32, lane = t & 31, w = t >> 5, nw = tu >> 5;
    int s = 1;
    while (true) {
        if (s == a.ms) { more = 1; break; }          // elements left that no stage may take
        int4 *rec = a.recs + (size_t)s * a.capnb + slot;
        int4 *el = a.el + (size_t)(s - 1) * a.T + s0;
        int *upl = a.upl + (size_t)(s - 1) * a.T + s0;
        for (int e = t; e < n; e += tu) cnt[e] = 0;
        if (t == 0) { sh.flag = 0; sh.nf = 0; sh.ne = 0; }
        bar_upper(tu);
        for (int e = t; e < n; e += tu) { const unsigned p = par[e]; if (p != E::NONE) E::add(cnt, p); }
        bar_upper(tu);
        for (int e = t; e < n; e += tu) {
            const unsigned p = par[e];
            if (p != E::NONE && (cnt[e] & E::MASK) > 0) E::flag(cnt, p);
        }
        bar_upper(tu);
        if (t == 0) sh.nb = walk_blocks<J>(par, cnt, n, a.bmu, sh.bst, SBU, rec);
        __syncwarp();
        const int k = seg_shift(n, nw);
        int run = 0, next = 0;
        long long deg = 0;
        for (int i = 0; i < (1 << (k - 5)); ++i) {
            const int base = (w << k) + 32 * i, e = base + lane;
            if (base >= n) break;
            bool kp = false;
            if (e < n) {
                unsigned p, lo, hi;
                const bool child = elem_range<J>(par, cnt, e, false, false, p, lo, hi);
                const int tk = tok[e];
                if (child) {
                    if (!((int)p < e && e < (int)hi)) seq_fail(sh, s0 + tk);
                    a.rank[s0 + tk] = e - (int)p;
                }
                kp = !child;
                el[e] = make_int4(tk, (p == E::NONE) ? -1 : (int)p, (int)lo, (int)hi);
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
            if (deg) atomicAdd(&sh.nnz, (unsigned long long)deg);
            if (next) sh.flag = 1;
        }
        bar_upper(tu);
        const bool go_on = sh.flag != 0;
        int total;
        const int wo = warp_offsets(sh.wtotu, nw, lane, total);
        const int mine = __shfl_sync(0xffffffffu, wo, w);
        for (int i = 0; i < (1 << (k - 5)); ++i) {
            const int base = (w << k) + 32 * i, e = base + lane;
            if (base >= n) break;
            const unsigned z = e < n ? pre[e] : E::NONE;
            unsigned p = E::NONE, q = E::NONE;
            if (z != E::NONE) { p = par[e]; if (p != E::NONE) q = pre[p]; }
            const int wp = __shfl_sync(0xffffffffu, wo, q != E::NONE ? (int)(p >> k) : 0);
            const int u = z != E::NONE ? (int)z + mine : -1;
            if (e < n) upl[e] = u;
            if (u >= 0 && go_on) {
                par2[u] = (J)(q != E::NONE ? q + (unsigned)wp : E::NONE);
                tok2[u] = tok[e];
            }
        }
        make_records<J>(par, cnt, n, false, false, sh.nb, sh.bst, SBU, rec, w, nw, lane, &sh.nf, &sh.ne, &sh.vis);
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

// A sequence's stages.  Shared memory per token of `cap`: 6 bytes (parents, counts, prefix sums) and,
// per upper element of `uc`, 12 (two sets of parents and tokens, counts, prefix sums), of which 8 may
// lie over stage 0's prefix sums, which are dead after its compaction.
__global__ void __launch_bounds__(1024) k_seq(const SeqArgs a) {
    pdl_launch_dependents();
    extern __shared__ __align__(16) uint16_t s_dyn[];
    __shared__ SeqShared sh;
    const int b = blockIdx.x, t = threadIdx.x, lane = t & 31, w = t >> 5, nw = blockDim.x >> 5;
    const int c0 = a.cu[b], c1 = a.cu[b + 1];
    const int s0 = min(max(c0, 0), a.T), L = min(max(c1, s0), a.T) - s0;
    if (t == 0) {
        sh.err = 0; sh.err_pos = 0; sh.flag0 = 0; sh.nf0 = 0; sh.ne0 = 0; sh.nnz = 0; sh.vis = 0;
        if (c1 < c0 || c0 < 0 || c1 > a.T || (b == 0 && c0 != 0) || (b == a.B - 1 && c1 != a.T)) seq_fail(sh, b);
        a.scu[b] = c0;
        if (b == a.B - 1) a.scu[a.B] = c1;
    }
    const bool root_real = L > 0 && a.level[s0] >= 0;
    const int slot = block_slot(s0, b, a.bmin);
    __syncthreads();
    const bool in_smem = L <= a.cap;
    uint16_t *X = s_dyn, *Y = X + a.cap, *Z = Y + a.cap, *U = Z + a.cap;
    uint32_t *G[NGLOB];
    for (int i = 0; i < NGLOB; ++i) G[i] = a.glob + a.glob_stride * i + s0;
    if (in_smem) seq_stage0<uint16_t>(a, sh, X, Y, Z, s0, L, root_real);
    else seq_stage0<uint32_t>(a, sh, G[0], G[1], G[2], s0, L, root_real);
    __syncthreads();
    int n1;
    (void)warp_offsets(sh.wtot, nw, lane, n1);
    const bool next = sh.flag0 != 0;
    const bool up_smem = n1 <= a.uc;
    // (the first parent / token set of the upper stages never lies over the prefix sums)
    uint16_t *P0 = U, *T0 = U + a.uc, *V = a.overlay ? Z : U + 2 * a.uc;
    if (in_smem && up_smem) seq_compact0<uint16_t, uint16_t>(a, sh, X, Z, P0, T0, s0, L, next);
    else if (in_smem) seq_compact0<uint16_t, uint32_t>(a, sh, X, Z, G[3], G[4], s0, L, next);
    else if (up_smem && L < 65535) seq_compact0<uint32_t, uint16_t>(a, sh, G[0], G[2], P0, T0, s0, L, next);
    else seq_compact0<uint32_t, uint32_t>(a, sh, G[0], G[2], G[3], G[4], s0, L, next);
    __syncthreads();
    int stages = 1, res = n1, more = 0;
    if (w == nw - 1) {
        if (lane == 0)
            sh.nb0 = in_smem ? walk_blocks<uint16_t>(X, Y, L, a.bm, sh.bst0, SB0, a.recs + slot)
                             : walk_blocks<uint32_t>(G[0], G[1], L, a.bm, sh.bst0, SB0, a.recs + slot);
    } else if (next) {
        if (up_smem && (in_smem || L < 65535)) seq_upper<uint16_t>(a, sh, P0, T0, V, V + a.uc, V + 2 * a.uc, V + 3 * a.uc, b, s0, slot, n1, stages, res, more);
        else seq_upper<uint32_t>(a, sh, G[3], G[4], G[5], G[6], G[7], G[8], b, s0, slot, n1, stages, res, more);
    }
    __syncthreads();
    if (in_smem) make_records<uint16_t>(X, Y, L, true, root_real, sh.nb0, sh.bst0, SB0, a.recs + slot, w, nw, lane, &sh.nf0, &sh.ne0, &sh.vis);
    else make_records<uint32_t>(G[0], G[1], L, true, root_real, sh.nb0, sh.bst0, SB0, a.recs + slot, w, nw, lane, &sh.nf0, &sh.ne0, &sh.vis);
    __syncthreads();
    if (t == 0) {
        const size_t q = (size_t)a.ms * a.B;
        int *c = a.counts + b;
        c[0] = L; c[q] = sh.nb0; c[2 * q] = sh.nf0; c[3 * q] = sh.ne0;
        for (int s = stages; s < a.ms; ++s) {          // beyond its own stages: its root in a block of its own
            c = a.counts + (size_t)s * a.B + b;
            c[0] = res; c[q] = res; c[2 * q] = 0; c[3 * q] = res;
        }
        SeqInfo f;
        f.stages = stages; f.res = res; f.err = sh.err; f.err_pos = sh.err_pos; f.more = more; f.pad = 0;
        f.nnz = (long long)sh.nnz; f.visited = (long long)sh.vis;
        a.info[b] = f;
    }
}

struct FinishArgs {
    StagePtrs st[HDT_MAX_STAGES];
    const int32_t *cu;
    int B, T, ms, bm, bmu, bmin, capnb, gy, r0;   // gy: CTAs of a sequence; r0: CTAs that rank stage 0's blocks
    const SeqInfo *info;
    const int *counts;
    const int4 *recs, *el;
    const int *upl;
    long long *keys;
    DevHeader *hdr, *host;         // host: pinned landing buffer (its words are not 0 at `tail` before)
};

static constexpr int FT = 256;     // threads of k_finish
static constexpr int FKEYS = 4096; // blocks of a stage whose sort keys fit in shared memory

__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Header: totals over the sequences.  The words go to the workspace (kernels read them there) and
// straight to the host's pinned buffer, the tail word last and behind a system-wide fence: the host
// watches for it, so no copy has to be queued behind the build.
__device__ void finish_header(const FinishArgs &f, int S) {
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    __shared__ int s_err, s_more;
    __shared__ long long s_sum[2];
    if (t == 0) { s_err = 0x7fffffff; s_more = 0; s_sum[0] = s_sum[1] = 0; }
    __syncthreads();
    const size_t q = (size_t)f.ms * f.B;
    for (int i = w; i < 4 * S; i += FT / 32) {
        const int s = i >> 2, c = i & 3;
        int v = 0;
        for (int b = lane; b < f.B; b += 32) v += f.counts[c * q + (size_t)s * f.B + b];
        v = __reduce_add_sync(0xffffffffu, v);
        if (lane == 0) {
            StageDesc &d = f.hdr->st[s], &h = f.host->st[s];
            int *pd = c == 0 ? &d.n : c == 1 ? &d.nb : c == 2 ? &d.n_fused : &d.n_empty;
            int *ph = c == 0 ? &h.n : c == 1 ? &h.nb : c == 2 ? &h.n_fused : &h.n_empty;
            *pd = v;
            *reinterpret_cast<volatile int *>(ph) = v;
        }
    }
    long long nnz = 0, vis = 0;
    for (int b = t; b < f.B; b += FT) {
        const SeqInfo &x = f.info[b];
        nnz += x.nnz; vis += x.visited;
        if (x.err) atomicMin(&s_err, b);
        if (x.more) s_more = 1;
    }
    nnz = warp_sum(nnz); vis = warp_sum(vis);
    if (lane == 0) { atomicAdd((unsigned long long *)&s_sum[0], (unsigned long long)nnz); atomicAdd((unsigned long long *)&s_sum[1], (unsigned long long)vis); }
    __syncthreads();
    if (t <= HDT_MAX_STAGES) {
        const int more = (t + 1 < S) || (t + 1 == S && s_more);
        f.hdr->st[t].has_next = more;
        *reinterpret_cast<volatile int *>(&f.host->st[t].has_next) = more;
        if (t >= S) {
            StageDesc &d = f.hdr->st[t];
            d.n = d.nb = d.n_fused = d.n_empty = 0;
            volatile StageDesc *h = &f.host->st[t];
            h->n = 0; h->nb = 0; h->n_fused = 0; h->n_empty = 0;
        }
    }
    if (t == 0) {
        int err = 0, pos = 0;
        if (f.B == 0) { f.st[0].scu[0] = f.cu[0]; if (f.cu[0] != 0 || f.T != 0) err = HDT_ERR_BAD_HIERARCHY; }
        else if (s_err != 0x7fffffff) { err = f.info[s_err].err; pos = f.info[s_err].err_pos; }
        volatile DevHeader *h = f.host;
        f.hdr->status = err; f.hdr->err_pos = pos; f.hdr->nnz = s_sum[0]; f.hdr->visited = s_sum[1]; f.hdr->tail = 0;
        h->status = err; h->err_pos = pos; h->nnz = s_sum[0]; h->visited = s_sum[1];
    }
    __threadfence_system();
    __syncthreads();
    if (t == 0) *reinterpret_cast<volatile int *>(&f.host->tail) = 0;
}

// Rank sort of a stage's blocks: queue[rank] = block id, cost descending, id ascending.  queue_split:
// the same order inside two groups, blocks that are SELF and not EMPTY first, then the others.
// Every CTA gathers all keys (cost << 1 | SELF non-EMPTY), a warp ranks a block at a time.
__device__ void finish_rank(const FinishArgs &f, int s, int part, int parts, long long *s_keys) {
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, nw = FT / 32;
    __shared__ int s_base[FT], s_cnt[FT], s_w[FT / 32];
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
        __syncthreads();
        int off = run, all = 0;
        for (int i = 0; i < nw; ++i) { if (i < w) off += s_w[i]; all += s_w[i]; }
        s_base[t] = off + v - c;
        s_cnt[t] = c;
        __syncthreads();
        const int nseq = min(FT, f.B - b0);
        for (int i = w; i < nseq; i += nw) {
            const int bb = b0 + i;
            const bool own = s < f.info[bb].stages;     // else its root alone, in a block without keys: cost 0
            const int4 *rec = f.recs + (size_t)s * f.capnb + block_slot(min(max(f.cu[bb], 0), f.T), bb, f.bmin);
            for (int j = lane; j < s_cnt[i]; j += 32) {
                long long k = 0;
                if (own) {
                    const int4 r = rec[j];
                    const int fl = r.w >> 8;
                    k = ((long long)(r.w & 255) * (r.z - r.y)) * 2 + ((fl & HDT_BLK_SELF) && !(fl & HDT_BLK_EMPTY) ? 1 : 0);
                }
                keys[s_base[i] + j] = k;
            }
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

// CTA 0: header; then r0 CTAs rank stage 0's blocks and one each those of the other stages; then gy
// CTAs per sequence move its elements and block records to their place in the batch's arrays.
__global__ void __launch_bounds__(FT) k_finish(const FinishArgs f) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ long long s_keys[FKEYS];
    __shared__ int s_stages, s_bad;
    __shared__ int s_n[HDT_MAX_STAGES + 1], s_b[HDT_MAX_STAGES + 1], s_tot[HDT_MAX_STAGES + 1];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, nw = FT / 32;
    if (t == 0) { s_stages = 1; s_bad = 0; }
    __syncthreads();
    {
        int m = 1, bad = 0;
        for (int b = t; b < f.B; b += FT) { m = max(m, f.info[b].stages); bad |= f.info[b].err; }
        m = __reduce_max_sync(0xffffffffu, m);
        bad = __any_sync(0xffffffffu, bad);
        if (lane == 0) { atomicMax(&s_stages, m); if (bad) s_bad = 1; }
    }
    __syncthreads();
    const int S = s_stages;
    int id = blockIdx.x;
    if (id == 0) { finish_header(f, S); return; }
    if (s_bad) return;               // (offsets of a broken hierarchy mean nothing)
    id -= 1;
    if (id < f.r0) { finish_rank(f, 0, id, f.r0, s_keys); return; }
    id -= f.r0;
    if (id < f.ms - 1) { if (id + 1 < S) finish_rank(f, id + 1, 0, 1, s_keys); return; }
    id -= f.ms - 1;
    const int b = id / f.gy, y = id % f.gy;
    // sums over the sequences before this one: elements and blocks of every stage
    const size_t q = (size_t)f.ms * f.B;
    for (int i = w; i < 2 * S; i += nw) {
        const int s = i >> 1;
        const int *c = f.counts + ((i & 1) ? q : 0) + (size_t)s * f.B;
        int v = 0;
        for (int j = lane; j < b; j += 32) v += c[j];
        v = __reduce_add_sync(0xffffffffu, v);
        if (lane == 0) {
            if (i & 1) s_b[s] = v;
            else { s_n[s] = v; s_tot[s] = v + c[b]; }      // (s_tot: the batch's elements where b is the last sequence)
        }
    }
    __syncthreads();
    const SeqInfo info = f.info[b];
    const int s0 = f.cu[b], L = f.cu[b + 1] - s0;
    const int step = FT * f.gy, me = y * FT + t;
    {
        int *up = f.st[0].up;
        const int off = S > 1 ? s_n[1] : 0;
        for (int e = me; e < L; e += step) {
            const int v = up[s0 + e];
            if (v >= 0) up[s0 + e] = S > 1 ? v + off : -1;
        }
    }
    const int slot = block_slot(s0, b, f.bmin);
    for (int s = 0; s < S; ++s) {
        const StagePtrs &P = f.st[s];
        const int off = s ? s_n[s] : s0, boff = s_b[s];
        const bool last = s + 1 == S;
        const int n = f.counts[(size_t)s * f.B + b], nb = f.counts[q + (size_t)s * f.B + b];
        if (s > 0 && me == 0) {
            P.scu[b] = off;
            if (b == f.B - 1) P.scu[f.B] = s_tot[s];
        }
        if (s < info.stages) {
            if (s > 0) {
                const int4 *el = f.el + (size_t)(s - 1) * f.T + s0;
                const int *upl = f.upl + (size_t)(s - 1) * f.T + s0;
                const int noff = last ? 0 : s_n[s + 1];
                for (int e = me; e < n; e += step) {
                    const int4 x = el[e];
                    const int u = upl[e];
                    const bool has = x.w > x.z;
                    P.tok[off + e] = s0 + x.x;
                    P.par[off + e] = x.y < 0 ? -1 : off + x.y;
                    reinterpret_cast<int2 *>(P.rng)[off + e] = make_int2(has ? off + x.z : 0, has ? off + x.w : 0);
                    P.up[off + e] = (u < 0 || last) ? -1 : u + noff;
                }
            }
            const int4 *rec = f.recs + (size_t)s * f.capnb + slot;
            for (int i = me; i < nb; i += step) {
                const int4 r = rec[i];
                int fl = r.w >> 8;
                if (last) fl &= ~HDT_BLK_CARRY;
                int *o = P.blocks + 5 * (size_t)(boff + i);
                o[0] = off + r.x; o[1] = off + r.x + (r.w & 255); o[2] = off + r.y; o[3] = off + r.z; o[4] = fl;
            }
        } else if (info.res && me == 0) {       // (res is 0 or 1 here)
            P.tok[off] = s0;
            P.par[off] = -1;
            reinterpret_cast<int2 *>(P.rng)[off] = make_int2(0, 0);
            P.up[off] = last ? -1 : s_n[s + 1];
            int *o = P.blocks + 5 * (size_t)boff;
            o[0] = off; o[1] = off + 1; o[2] = off; o[3] = off;
            o[4] = HDT_BLK_SELF | HDT_BLK_EMPTY | (last ? 0 : HDT_BLK_CARRY);
        }
    }
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
static const int kUnset = 0x7fffffff;
static std::mutex g_pinned_mu;
static std::vector<DevHeader *> g_pinned_free;
static DevHeader *pinned_acquire() {
    {
        std::lock_guard<std::mutex> lk(g_pinned_mu);
        if (!g_pinned_free.empty()) {
            DevHeader *p = g_pinned_free.back();
            g_pinned_free.pop_back();
            return p;
        }
    }
    DevHeader *p = nullptr;
    if (cudaHostAlloc((void **)&p, sizeof(DevHeader), cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
        (void)cudaGetLastError();
        return nullptr;
    }
    return p;
}
static void pinned_release(DevHeader *p) {
    if (!p) return;
    std::lock_guard<std::mutex> lk(g_pinned_mu);
    g_pinned_free.push_back(p);
}

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
    // two up to SEQ_CAP_MAX.  Up to 8192 tokens the upper stages' arrays have room of their own for as
    // many elements as tokens (deep trees keep most of them above stage 0); beyond, for 4096 elements
    // (documents keep a few percent), over stage 0's prefix sums.
    const long long mean = B > 0 ? ((long long)T + B - 1) / B : 0;
    const long long want = B == 1 ? T : 4 * mean;
    int cap = 1024;
    while (cap < want && cap < SEQ_CAP_MAX) cap *= 2;
    SeqArgs a{};
    a.cap = cap;
    a.uc = min(cap, 4096);
    a.overlay = cap > 8192 ? 1 : 0;
    const size_t smem = sizeof(uint16_t) * (3 * (size_t)cap + (a.overlay ? 2 : 6) * (size_t)a.uc);
    static constexpr size_t kSmemMax = sizeof(uint16_t) * (3 * (size_t)SEQ_CAP_MAX + 2 * 4096);
    static DevOnce attr_done;
    if (!attr_done.done()) {
        HDT_CUDA_CHECK(cudaFuncSetAttribute(k_seq, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
        attr_done.set();
    }
    DevHeader *hp = pinned_acquire();
    if (!hp) return set_error(HDT_ERR_CUDA, "hdt_build_index: no pinned host memory for the index header");
    hp->tail = kUnset;

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
    ix->pending = 1;

    a.level = level; a.parent = parent; a.cu = cu_seqlens;
    a.B = B; a.T = T; a.ms = ms; a.bm = bm; a.bmu = bmu; a.bmin = bmin; a.dirs = dirs;
    a.tok = ix->st[0].tok; a.par = ix->st[0].par; a.rng = ix->st[0].rng; a.up = ix->st[0].up; a.scu = ix->st[0].scu;
    a.rank = (int *)(ws + L.rank);
    a.info = (SeqInfo *)(ws + L.info);
    a.counts = (int *)(ws + L.counts);
    a.recs = (int4 *)(ws + L.recs);
    a.capnb = L.capnb;
    a.el = (int4 *)(ws + L.el);
    a.upl = (int *)(ws + L.upl);
    a.glob = (uint32_t *)(ws + L.glob);
    a.glob_stride = al(sizeof(int) * (size_t)T) / sizeof(int);
    FinishArgs f{};
    for (int s = 0; s < ms; ++s) f.st[s] = ix->st[s];
    f.cu = cu_seqlens; f.B = B; f.T = T; f.ms = ms; f.bm = bm; f.bmu = bmu; f.bmin = bmin; f.capnb = L.capnb;
    f.gy = (int)min(16LL, max(1LL, mean / 2048));
    f.r0 = max(1, min(32, L.capnb / 64));
    f.info = a.info; f.counts = a.counts; f.recs = a.recs; f.el = a.el; f.upl = a.upl;
    f.keys = (long long *)(ws + L.keys);
    f.hdr = (DevHeader *)(ws + L.header);
    f.host = hp;
    cudaError_t e = cudaSuccess;
    {
        ProfScope ps(PROF_INDEX, st);
        if (B > 0) {
            // a thread per element of short sequences: 8 warps (7 build the upper stages), else 32
            k_seq<<<B, mean <= 1024 ? 256 : 1024, smem, st>>>(a);
            count_launch();
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) {
            // a programmatic dependent: its CTAs are scheduled while k_seq runs and wait for its end
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3((unsigned)(1 + f.r0 + (ms - 1) + (size_t)B * f.gy));
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
    if (!(params && params->deferred)) {
        const int rc = index_ready(ix);
        if (rc) {
            delete ix;
            return rc;
        }
    }
    *out = ix;
    return HDT_OK;
}

namespace hdt {
int index_ready(const hdt_index *cix) {
    hdt_index *ix = const_cast<hdt_index *>(cix);
    if (ix->pending) {
        // The host watches the tail word of the pinned header, which the device writes last, behind a
        // system-wide fence.  After a bounded number of looks it waits for the stream instead.
        DevHeader *hp = ix->h_pinned;
        volatile int *p_tail = &hp->tail;
        for (long long spin = 0; spin < 20000000LL && *p_tail == kUnset; ++spin) {}
        cudaError_t e_ = cudaSuccess;
        if (*p_tail == kUnset) {
            e_ = cudaStreamSynchronize(ix->stream);
            if (e_ == cudaSuccess && *p_tail == kUnset) e_ = cudaErrorUnknown;
        }
        ix->pending = 0;
        ix->h_pinned = nullptr;
        if (e_ != cudaSuccess) {
            (void)cudaGetLastError();
            ix->failed = HDT_ERR_CUDA;
            pinned_release(hp);
            return set_error(HDT_ERR_CUDA, "waiting for the index build failed: %s", cudaGetErrorString(e_));
        }
        std::atomic_thread_fence(std::memory_order_acquire);
        const DevHeader h = *hp;
        pinned_release(hp);
        ix->failed = h.status;
        ix->err_pos = h.err_pos;
        if (h.status == 0) {
            int ns = 1;
            while (ns < ix->max_stages && h.st[ns].n > 0) ++ns;
            if (h.st[ns - 1].has_next && ns == ix->max_stages) {
                ix->failed = HDT_ERR_BAD_HIERARCHY;
                ix->err_pos = -1;
            } else {
                ix->n_stages = ns;
                ix->nnz = h.nnz;
                ix->visited = h.visited;
                for (int s = 0; s <= HDT_MAX_STAGES; ++s) ix->desc[s] = h.st[s];
            }
        }
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
    if (const int rc = index_ready(ix)) return rc;
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
    if (ix && ix->pending) (void)index_ready(ix);     // the header must not land in a recycled buffer
    delete ix;
    return HDT_OK;
}
