// Row-wise attention kernels: a row (element, head) is owned by a few lanes of a warp that walk its keys in
// every stage the element lives in and write its final result.  One launch does what takes a launch per
// stage and a merge on the tile kernels, so they serve
//   - the stages above 0, behind stage 0 (whose partial result they add), where their families are short:
//     documents keep about 3 % of their tokens above stage 0, with a few dozen keys each, and a tile kernel
//     there is a chain of gather, MMA, softmax, MMA and scatter with 128 rows for a dozen used ones;
//   - all stages of batches whose families are tiny throughout (expression trees: six keys a row).
// All arithmetic is fp32 (P and dS are not rounded).
//
// What bounds them: the latency of a row's chain of loads at the occupancy their registers leave, then instruction
// issue (200 trees: forward 56 us, 57 % of the issue slots and 40 % of the warps active; backward 125 us, 41 % and
// 20 %).  Of whole calls (build, forward and, with b, backward) the kernels' first form made, with all else as it was
// then: 200 trees 807 -> 260 us b, one tree 280 -> 82 b, 12 layers of 1 x 4096 tokens 389 -> 295,
// 2 x 220 tokens fp32 133 -> 46 b, 8 x 2048 padded 56 -> 51.
//
// Lanes: D / 8 lanes hold 8 dimensions each; a chunk of C keys is a C-fold load of 16 (bf16) or 32 (fp32)
// bytes per lane, all in flight together.  The C dot products are summed over the lanes by a reduce-scatter
// (C - 1 shuffles instead of 3 C or 4 C), which leaves one key's score per lane: one exponential per key
// and lane instead of one per key on every lane.  KP groups of lanes may share a row (each takes every
// KP-th chunk), for batches with too few rows to fill the SMs.
#include <climits>

#include <cuda_bf16.h>

#include "hdt_internal.cuh"
#include "hdt_rows.cuh"

namespace hdt {

// (small CTAs: one gives its place up when its longest row is done, and rows differ; 200 trees, forward and backward, 128 threads 244.8 us,
// 64 240.0, 32 242.6)
static constexpr int ROW_THREADS = 64;

// The keys of a row over the stages it lives in, a chunk at a time.  What the next stage needs first (range,
// next index) is loaded on entering a stage, and the tokens of a chunk while the one before it is worked
// on: the walk is a chain of dependent loads, and the kernels are bound by its length.
template <int C, int STEP>
struct RowCursor {
    const RowStage *st;
    int s, e, up, upn, j0;
    int2 r, rn;
    __device__ __forceinline__ void peek() {
        if (up >= 0) {
            rn = __ldg(reinterpret_cast<const int2 *>(st[s + 1].rng) + up);
            upn = __ldg(st[s + 1].up + up);
        }
    }
    __device__ __forceinline__ bool settle(int first) {      // to the next stage while this one is exhausted; false: no keys left
        while (j0 >= r.y) {
            if (up < 0) return false;
            e = up; r = rn; up = upn; ++s;
            j0 = r.x + first;
            peek();
        }
        return true;
    }
    __device__ __forceinline__ bool start(const RowStage *st_, int s_, int e_, int first) {
        st = st_; s = s_; e = e_;
        r = __ldg(reinterpret_cast<const int2 *>(st[s].rng) + e);
        up = __ldg(st[s].up + e);
        j0 = r.x + first;
        peek();
        return settle(first);
    }
    __device__ __forceinline__ bool next(int first) { j0 += STEP; return settle(first); }
    // token of this lane's key (keys past the end read the last one: in bounds, weight 0)
    __device__ __forceinline__ int token(int c) const {
        const int j = min(j0 + c, r.y - 1);
        return s ? __ldg(st[s].tok + j) : j;
    }
};

// ---------------------------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------------------------
// The keys of stages `first`, first + 1, ... of one row, read from global memory.
template <int D, bool BF16, int KP, int C, class Args>
__device__ __forceinline__ void fwd_walk(const Args &a, const Raw<BF16, D / 8> &q, RowSoftmax &S, int first, int e, int h, int g, int kp, int src, unsigned mask) {
    using R = Raw<BF16, D / 8>;
    RowCursor<C, KP * C> cur;
    bool more = cur.start(a.st, first, e, kp * C);
    int tm = more ? cur.token(g & (C - 1)) : 0;
    while (more) {
        const int jm = cur.j0 + (g & (C - 1)), tc = tm;
        const bool ok = jm < cur.r.y && (a.dirs == 7 || dir_ok(cur.e, jm, cur.r.x, a.dirs));
        R kr[C], vr[C];
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const unsigned r = (unsigned)__shfl_sync(mask, tc, src + i, 32) * a.H + h;
            kr[i].load(a.k, r, g);
            vr[i].load(a.v, r, g);
        }
        more = cur.next(kp * C);
        if (more) tm = cur.token(g & (C - 1));
        float sc[C];
        dots<C>(q, kr, sc);
        const float x = reduce_scatter<C, D / 8>(sc, g, mask) * a.scale_log2;
        const float p = S.add<C>(ok ? x : -INFINITY, mask);
        axpys<C>(S.acc, p, vr, mask, src);
    }
}

template <int D, bool BF16, int KP, int C>
__global__ void __launch_bounds__(ROW_THREADS, KP == 1 && C == 4 && BF16 ? 16 : 8) k_fwd_rows(const RowFwdArgs a) {
    constexpr int LPK = D / 8, G = LPK * KP;
    using R = Raw<BF16, LPK>;
    const int lane = threadIdx.x & 31, sub = lane % G, g = sub % LPK, kp = sub / LPK;
    const unsigned all = G == 32 ? 0xffffffffu : ((1u << G) - 1u) << (lane - sub);     // the lanes of the row
    const int src = lane - g;                                                             // and of the group that shares a key
    const unsigned mask = ((1u << LPK) - 1u) << src;
    const unsigned long long id = ((unsigned long long)blockIdx.x * ROW_THREADS + threadIdx.x) / G;
    pdl_launch_dependents();
    if (a.first == 0) pdl_wait();     // (else: only what stage 0 leaves is waited for, behind the walk)
    if (id >= (unsigned long long)a.n * a.H) return;
    const int e = (int)(id / a.H), h = (int)(id % a.H);     // (the rows of a warp are heads of an element: one range, no divergence)
    const int t = a.first ? a.st[a.first].tok[e] : e;
    const unsigned row = (unsigned)t * a.H + h;
    R q;
    q.load(a.q, row, g);
    RowSoftmax S;
    S.clear();
    fwd_walk<D, BF16, KP, C>(a, q, S, a.first, e, h, g, kp, src, mask);
    // l over the C lanes that hold different keys (lanes g and g + C of a 16-lane group hold the same ones)
#pragma unroll
    for (int o = 1; o < C; o *= 2) S.l += __shfl_xor_sync(mask, S.l, o);
#pragma unroll
    for (int o = LPK; o < G; o *= 2) {      // the groups that share the row
        f2 acc2[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) acc2[i] = __shfl_xor_sync(all, S.acc[i], o);
        const float m2 = __shfl_xor_sync(all, S.m, o), l2 = __shfl_xor_sync(all, S.l, o);
        S.merge(m2, l2, acc2);
    }
    if (kp != 0) return;
    if (a.first != 0) pdl_wait();
    if (a.base_o != nullptr) {              // stage 0's partial result, normalised, as one more key
        f2 o0[4];
        R::load_f32(a.base_o, (size_t)e * a.H + h, g, o0);
        S.merge(a.base_lse[(size_t)e * a.H + h] * 1.4426950408889634f, 1.f, o0);
    }
    const float lse = S.finish();
    R::store(a.o, row, g, S.acc);
    if (g == 0) a.lse[(size_t)h * a.T + t] = lse;
}

// ---------------------------------------------------------------------------------------------
// backward
// ---------------------------------------------------------------------------------------------
// The family ranges of a stage are symmetric: the keys of a row are also the queries that attend to it, so
// one walk gives the row's dQ (as a query), dK and dV (as a key), each complete: no atomics.
// DELTA: rowsum(dO . O) is given; else it is computed from O here (one more row per key to read).
template <bool BF16, int N> struct RowGrad {
    Raw<BF16, N> q, k, v, go;          // the row's own values stay as loaded: registers decide how many warps hide the loads' latency
    float lse, delta;                  // lse in log2 units
    f2 dq[4], dk[4], dv[4];
    template <bool DELTA, class Args>
    __device__ __forceinline__ void load(const Args &a, int t, int h, int g, unsigned mask) {
        const unsigned row = (unsigned)t * a.H + h;
        q.load(a.q, row, g); k.load(a.k, row, g); v.load(a.v, row, g); go.load(a.d_o, row, g);
        lse = __ldg(a.lse + (size_t)h * a.T + t) * 1.4426950408889634f;
        if constexpr (DELTA) delta = __ldg(a.delta + (size_t)h * a.T + t);
        else {
            Raw<BF16, N> o;
            o.load(a.o, row, g);
            delta = dot(go, o);
#pragma unroll
            for (int x = 1; x < N; x *= 2) delta += __shfl_xor_sync(mask, delta, x);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) dq[i] = dk[i] = dv[i] = 0ull;
    }
    // The row as a query: K rows x and V rows y of a chunk of its keys; ok: this lane's key counts.
    template <int C>
    __device__ __forceinline__ void as_query(const Raw<BF16, N> (&x)[C], const Raw<BF16, N> (&y)[C], bool ok, float scale_log2, int g, unsigned mask, int src) {
        float v1[C], v2[C];
        dots<C>(q, x, v1);
        dots<C>(go, y, v2);
        const float s = reduce_scatter<C, N>(v1, g, mask) * scale_log2, dp = reduce_scatter<C, N>(v2, g, mask);
        const float p = ok ? exp2f(s - lse) : 0.f;
        axpys<C>(dq, ok ? p * (dp - delta) : 0.f, x, mask, src);      // (a row that is none's query may hold anything in dO: see k_bwd_tile)
    }
    // The row as a key: Q rows x and dO rows y of queries that attend to it, with their LSE and delta.
    template <int C>
    __device__ __forceinline__ void as_key(const Raw<BF16, N> (&x)[C], const Raw<BF16, N> (&y)[C], bool ok, float lse_j, float delta_j, float scale_log2, int g,
                                           unsigned mask, int src) {
        float v1[C], v2[C];
        dots<C>(k, x, v1);
        dots<C>(v, y, v2);
        const float s = reduce_scatter<C, N>(v1, g, mask) * scale_log2, dp = reduce_scatter<C, N>(v2, g, mask);
        const float p = ok ? exp2f(s - lse_j) : 0.f;
        axpys<C>(dk, ok ? p * (dp - delta_j) : 0.f, x, mask, src);
        axpys<C>(dv, p, y, mask, src);
    }
    __device__ __forceinline__ void scale(float c) {
        const f2 c2 = pack2(c, c);
#pragma unroll
        for (int i = 0; i < 4; ++i) { dq[i] = mul2(dq[i], c2); dk[i] = mul2(dk[i], c2); }
    }
};

template <int D, bool BF16, int KP, int C, bool DELTA, class Args>
__device__ __forceinline__ void bwd_walk(const Args &a, RowGrad<BF16, D / 8> &S, int first, int e, int h, int g, int kp, int src, unsigned mask) {
    using R = Raw<BF16, D / 8>;
    RowCursor<C, KP * C> cur;
    bool more = cur.start(a.st, first, e, kp * C);
    int tm = more ? cur.token(g & (C - 1)) : 0;
    while (more) {
        const int jm = cur.j0 + (g & (C - 1)), tc = tm;
        const bool in = jm < cur.r.y;
        const bool ok_q = in && (a.dirs == 7 || dir_ok(cur.e, jm, cur.r.x, a.dirs));          // the row attends to it
        const bool ok_k = in && (a.dirs == 7 || dir_ok_key(cur.e, jm, cur.r.x, a.dirs));      // it attends to the row
        const float lse_j = __ldg(a.lse + (size_t)h * a.T + tc) * 1.4426950408889634f;
        float dl_j = 0.f;
        if constexpr (DELTA) dl_j = __ldg(a.delta + (size_t)h * a.T + tc);
        R x[C], y[C];
        unsigned at[C];
#pragma unroll
        for (int i = 0; i < C; ++i) {
            at[i] = (unsigned)__shfl_sync(mask, tc, src + i, 32) * a.H + h;
            x[i].load(a.k, at[i], g);
            y[i].load(a.v, at[i], g);
        }
        more = cur.next(kp * C);
        if (more) tm = cur.token(g & (C - 1));
        S.template as_query<C>(x, y, ok_q, a.scale_log2, g, mask, src);
#pragma unroll
        for (int i = 0; i < C; ++i) {
            x[i].load(a.q, at[i], g);
            y[i].load(a.d_o, at[i], g);
        }
        if constexpr (!DELTA) {
            float v3[C];
#pragma unroll
            for (int i = 0; i < C; ++i) {
                R o;
                o.load(a.o, at[i], g);
                v3[i] = dot(o, y[i]);
            }
            dl_j = reduce_scatter<C, D / 8>(v3, g, mask);
        }
        S.template as_key<C>(x, y, ok_k, lse_j, dl_j, a.scale_log2, g, mask, src);
    }
}

template <int D, bool BF16, int KP, bool DELTA>
__global__ void __launch_bounds__(ROW_THREADS, BF16 ? 8 : 6) k_bwd_rows(const RowBwdArgs a) {
    constexpr int LPK = D / 8, G = LPK * KP, C = 2;
    using R = Raw<BF16, LPK>;
    const int lane = threadIdx.x & 31, sub = lane % G, g = sub % LPK, kp = sub / LPK;
    const unsigned all = G == 32 ? 0xffffffffu : ((1u << G) - 1u) << (lane - sub);     // the lanes of the row
    const int src = lane - g;                                                             // and of the group that shares a key
    const unsigned mask = ((1u << LPK) - 1u) << src;
    const unsigned long long id = ((unsigned long long)blockIdx.x * ROW_THREADS + threadIdx.x) / G;
    pdl_launch_dependents();
    if (a.first == 0) pdl_wait();     // (else: only what stage 0 leaves is waited for, behind the walk)
    if (id >= (unsigned long long)a.n * a.H) return;
    const int e = (int)(id / a.H), h = (int)(id % a.H);     // (the rows of a warp are heads of an element: one range, no divergence)
    const int t = a.first ? a.st[a.first].tok[e] : e;
    RowGrad<BF16, LPK> S;
    S.template load<DELTA>(a, t, h, g, mask);
    bwd_walk<D, BF16, KP, C, DELTA>(a, S, a.first, e, h, g, kp, src, mask);
#pragma unroll
    for (int o = LPK; o < G; o *= 2) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            S.dq[i] = add2(S.dq[i], __shfl_xor_sync(all, S.dq[i], o));
            S.dk[i] = add2(S.dk[i], __shfl_xor_sync(all, S.dk[i], o));
            S.dv[i] = add2(S.dv[i], __shfl_xor_sync(all, S.dv[i], o));
        }
    }
    if (kp != 0) return;
    if (a.first != 0) pdl_wait();
    S.scale(a.scale);
    if (a.base[0] != nullptr) {         // stage 0's partial gradients
        f2 y[4];
        auto plus = [&](f2 (&x)[4], const float *b) {
            R::load_f32(b, (size_t)e * a.H + h, g, y);
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = add2(x[i], y[i]);
        };
        plus(S.dq, a.base[0]); plus(S.dk, a.base[1]); plus(S.dv, a.base[2]);
    }
    const unsigned row = (unsigned)t * a.H + h;
    R::store(a.dq, row, g, S.dq);
    R::store(a.dk, row, g, S.dk);
    R::store(a.dv, row, g, S.dv);
}

// ---------------------------------------------------------------------------------------------
// fp32, stage 0: the rows' keys staged in shared memory
// ---------------------------------------------------------------------------------------------
// A CTA takes 32 (head_dim 64) or 16 (128) rows of a block and the keys of their ranges, in pieces of KT; a
// row is owned by D / 8 lanes as above.  The elements that live on leave their partial result in stage 1's
// buffers.  What bounds it is the chain of a key chunk (loads, products, reduction, exponential, broadcast) at the
// six warps a scheduler holds: 2 x 2048 tokens, 12 x 64, 54 us forward and 138 backward (148 with loops that end row by row), against 100 and 191 for
// the kernels that give 16 dimensions to a lane and walk a whole block's span in step.  Measured and not kept: a row
// on 2 (forward) or 4 (backward) lanes (49 and 173 us: fewer warps, twice the registers), four and two rows to
// eight lanes, so that a key read from shared memory serves several (58 and 213), going on to the
// stages above 0 inside this kernel (70 and 185: one long row holds the CTA).
// The rows of a warp walk in step: one with no keys left reads its last key again, one that has none in the piece a row of
// zeros behind it (KT), at weight 0 both.  A key of another family there would carry an inf into a row that does not attend to it.
// Forward and backward in step and, in brackets, with loops that end row by row: 2 x 2048 tokens, 12 x 64, 213 us (220), 12 x 128 401 (409);
// where all CTAs fit at once and the longest walk is what counts, 1 x 3119, 12 x 64, 207 (203), 4 x 741 196 (192).
// (KT: with the zero rows two backward CTAs take 196 KB of an SM, the step below the largest; at one row more, 228 KB, 28 instead of 60 are
// left for L1, and 2 x 2048 tokens forward and backward take 219 us instead of 215, as much as without the zero rows.)
static constexpr int TILE_THREADS = 256;
template <int D> struct TileShape {
    static constexpr int LPK = D / 8, ROWS = TILE_THREADS / LPK, KT = D == 64 ? 95 : 47, PIECE = (KT + 1) * (D / 4);      // PIECE: float4s of a tensor's rows
};
// The keys [lo, hi) of a row in the piece of n from c0 on, counted from c0.
template <int KT>
__device__ __forceinline__ void piece_range(int2 r, int c0, int n, int &lo, int &hi) {
    lo = max(r.x - c0, 0);
    hi = min(r.y - c0, n);
    if (hi <= lo) lo = hi = KT + 1;
}
__device__ __forceinline__ void cp_async16(float4 *dst, const float4 *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory"); }

// The rows of CTA x of a block and the span of their ranges.
struct TileRows {
    int r0, n, a, b;
    template <class Args>
    __device__ __forceinline__ void find(const Args &p, int rows, int per_block, int *s_ab) {
        const int *rec = p.blocks + 5 * (size_t)p.queue[blockIdx.x / per_block];
        r0 = rec[0] + (blockIdx.x % per_block) * rows;
        n = min(rows, rec[1] - r0);
        if (threadIdx.x == 0) { s_ab[0] = INT_MAX; s_ab[1] = 0; }
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const int2 r = __ldg(reinterpret_cast<const int2 *>(p.rng) + r0 + i);
            if (r.y > r.x) { atomicMin(s_ab, r.x); atomicMax(s_ab + 1, r.y); }
        }
        __syncthreads();
        a = s_ab[0]; b = s_ab[1];
    }
};
template <int D>
__device__ __forceinline__ void tile_load(float4 *dst, const void *src, int c0, int n, int H, int h) {
    constexpr int U = D / 4;
    for (int i = threadIdx.x; i < n * U; i += TILE_THREADS)
        cp_async16(dst + i, reinterpret_cast<const float4 *>(src) + ((size_t)(c0 + i / U) * H + h) * U + i % U);
}

template <int D>
__global__ void __launch_bounds__(TILE_THREADS, 3) k_fwd_tile(const TileFwdArgs a) {
    constexpr int LPK = D / 8, ROWS = TileShape<D>::ROWS, KT = TileShape<D>::KT, C = 4, U = D / 4;
    using R = Raw<false, LPK>;
    pdl_wait();
    pdl_launch_dependents();
    extern __shared__ float4 s_tile[];
    __shared__ int s_ab[2];
    float4 *sK = s_tile, *sV = sK + TileShape<D>::PIECE;
    for (int i = threadIdx.x; i < 2 * U; i += TILE_THREADS) s_tile[i / U * TileShape<D>::PIECE + KT * U + i % U] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int h = blockIdx.y, lane = threadIdx.x & 31, g = lane % LPK, src = lane - g;
    constexpr unsigned mask = 0xffffffffu;       // (the rows of a warp walk in step: with a mask per row their shuffles issue one after the other)
    TileRows T;
    T.find(a, ROWS, (a.block_rows + ROWS - 1) / ROWS, s_ab);
    if (T.n <= 0) return;
    const int rl = threadIdx.x / LPK, row = T.r0 + rl;
    const bool inb = rl < T.n;
    int2 r = make_int2(0, 0);
    R q;
    RowSoftmax S;
    S.clear();
    if (inb) {
        r = __ldg(reinterpret_cast<const int2 *>(a.rng) + row);
        q.load(a.q, (unsigned)row * a.H + h, g);
    }
    for (int c0 = T.a; c0 < T.b; c0 += KT) {
        const int n = min(KT, T.b - c0);
        if (c0 != T.a) __syncthreads();
        tile_load<D>(sK, a.k, c0, n, a.H, h);
        tile_load<D>(sV, a.v, c0, n, a.H, h);
        cp_async_wait();
        __syncthreads();
        int lo, hi;
        piece_range<KT>(r, c0, n, lo, hi);
        const int steps = __reduce_max_sync(mask, (hi - lo + C - 1) / C);
        for (int it = 0, j0 = lo; it < steps; ++it, j0 += C) {
            float sc[C];
            f2 qf[4];
            q.get(qf);
#pragma unroll
            for (int i = 0; i < C; ++i) {
                R x;
                f2 k[4];
                x.load_smem(sK + min(j0 + i, hi - 1) * U, g);      // (keys past the end: the last one or zeros, weight 0)
                x.get(k);
                sc[i] = dot8(qf, k);
            }
            const int jm = j0 + (g & (C - 1));
            const bool ok = jm < hi && (a.dirs == 7 || dir_ok(row, c0 + jm, r.x, a.dirs));
            const float x = reduce_scatter<C, LPK>(sc, g, mask) * a.scale_log2;
            const float p = S.add<C>(ok ? x : -INFINITY, mask);
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const float w = __shfl_sync(mask, p, src + i, 32);
                const f2 w2 = pack2(w, w);
                R y;
                f2 v[4];
                y.load_smem(sV + min(j0 + i, hi - 1) * U, g);
                y.get(v);
#pragma unroll
                for (int u = 0; u < 4; ++u) S.acc[u] = fma2(w2, v[u], S.acc[u]);
            }
        }
    }
    // (l over the C lanes that hold different keys)
#pragma unroll
    for (int o = 1; o < C; o *= 2) S.l += __shfl_xor_sync(mask, S.l, o);
    if (!inb) return;
    const int up = a.up ? __ldg(a.up + row) : -1;
    const float lse = S.finish();
    if (up >= 0) {
        R::store(a.part_o, (unsigned)up * a.H + h, g, S.acc);
        if (g == 0) a.part_lse[(size_t)up * a.H + h] = lse;
    }
    R::store(a.o, (unsigned)row * a.H + h, g, S.acc);
    if (g == 0) a.lse[(size_t)h * a.T + row] = lse;
}

template <int D>
__global__ void __launch_bounds__(TILE_THREADS, 2) k_bwd_tile(const TileBwdArgs a) {
    constexpr int LPK = D / 8, ROWS = TileShape<D>::ROWS, KT = TileShape<D>::KT, C = 2, U = D / 4;
    using R = Raw<false, LPK>;
    pdl_wait();
    pdl_launch_dependents();
    extern __shared__ float4 s_tile[];
    __shared__ int s_ab[2];
    __shared__ float s_lse[KT + 1], s_delta[KT + 1];
    constexpr int PIECE = TileShape<D>::PIECE;
    float4 *sK = s_tile, *sV = sK + PIECE, *sQ = sV + PIECE, *sG = sQ + PIECE;
    for (int i = threadIdx.x; i < 4 * U; i += TILE_THREADS) s_tile[i / U * PIECE + KT * U + i % U] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (threadIdx.x == 0) s_lse[KT] = s_delta[KT] = 0.f;
    const int h = blockIdx.y, lane = threadIdx.x & 31, g = lane % LPK, src = lane - g;
    constexpr unsigned mask = 0xffffffffu;       // (the rows of a warp walk in step: with a mask per row their shuffles issue one after the other)
    TileRows T;
    T.find(a, ROWS, (a.block_rows + ROWS - 1) / ROWS, s_ab);
    if (T.n <= 0) return;
    const int rl = threadIdx.x / LPK, row = T.r0 + min(rl, T.n - 1);
    const bool inb = rl < T.n;
    int2 r = inb ? __ldg(reinterpret_cast<const int2 *>(a.rng) + row) : make_int2(0, 0);
    RowGrad<false, LPK> S;
    S.template load<false>(a, row, h, g, mask);
    for (int c0 = T.a; c0 < T.b; c0 += KT) {
        const int n = min(KT, T.b - c0);
        if (c0 != T.a) __syncthreads();
        tile_load<D>(sK, a.k, c0, n, a.H, h);
        tile_load<D>(sV, a.v, c0, n, a.H, h);
        tile_load<D>(sQ, a.q, c0, n, a.H, h);
        tile_load<D>(sG, a.d_o, c0, n, a.H, h);
        cp_async_wait();
        __syncthreads();
        for (int i0 = 0; i0 < n; i0 += ROWS) {         // rowsum(dO . O) of the tile's rows
            const int i = min(i0 + rl, n - 1);
            R o, y;
            o.load(a.o, (unsigned)(c0 + i) * a.H + h, g);
            y.load_smem(sG + i * U, g);
            float d = dot(o, y);
#pragma unroll
            for (int x = 1; x < LPK; x *= 2) d += __shfl_xor_sync(mask, d, x);
            if (g == 0) {
                s_delta[i] = d;
                s_lse[i] = __ldg(a.lse + (size_t)h * a.T + c0 + i) * 1.4426950408889634f;
            }
        }
        __syncthreads();
        int lo, hi;
        piece_range<KT>(r, c0, n, lo, hi);
        const int steps = __reduce_max_sync(mask, (hi - lo + C - 1) / C);
        for (int it = 0, j0 = lo; it < steps; ++it, j0 += C) {
            const int jm = j0 + (g & (C - 1)), jc = min(jm, hi - 1);
            const bool in = jm < hi;
            const bool ok_q = in && (a.dirs == 7 || dir_ok(row, c0 + jm, r.x, a.dirs));
            const bool ok_k = in && (a.dirs == 7 || dir_ok_key(row, c0 + jm, r.x, a.dirs));
            R x[C], y[C];
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const int o = min(j0 + i, hi - 1) * U;
                x[i].load_smem(sK + o, g);
                y[i].load_smem(sV + o, g);
            }
            S.template as_query<C>(x, y, ok_q, a.scale_log2, g, mask, src);
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const int o = min(j0 + i, hi - 1) * U;
                x[i].load_smem(sQ + o, g);
                y[i].load_smem(sG + o, g);
            }
            S.template as_key<C>(x, y, ok_k, s_lse[jc], s_delta[jc], a.scale_log2, g, mask, src);
        }
    }
    if (!inb) return;
    const int up = a.up ? __ldg(a.up + row) : -1;
    S.scale(a.scale);
    if (up >= 0) {
        const unsigned p = (unsigned)up * a.H + h;
        R::store(a.part[0], p, g, S.dq); R::store(a.part[1], p, g, S.dk); R::store(a.part[2], p, g, S.dv);
    }
    const unsigned p = (unsigned)row * a.H + h;
    R::store(a.dq, p, g, S.dq); R::store(a.dk, p, g, S.dk); R::store(a.dv, p, g, S.dv);
}

template <int D>
static int launch_fwd_tile_t(const TileFwdArgs &a, cudaStream_t st) {
    if (a.nb == 0) return HDT_OK;
    constexpr int smem = 2 * TileShape<D>::PIECE * 16;
    static DevOnce once;
    if (!once.done()) {
        HDT_CUDA_CHECK(cudaFuncSetAttribute(k_fwd_tile<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        once.set();
    }
    constexpr int ROWS = TileShape<D>::ROWS;
    HDT_CUDA_CHECK(launch_dependent(k_fwd_tile<D>, true, dim3(a.nb * ((a.block_rows + ROWS - 1) / ROWS), a.H), TILE_THREADS, smem, st, a));
    return HDT_OK;
}
template <int D>
static int launch_bwd_tile_t(const TileBwdArgs &a, cudaStream_t st) {
    if (a.nb == 0) return HDT_OK;
    constexpr int smem = 4 * TileShape<D>::PIECE * 16;
    static DevOnce once;
    if (!once.done()) {
        HDT_CUDA_CHECK(cudaFuncSetAttribute(k_bwd_tile<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        once.set();
    }
    constexpr int ROWS = TileShape<D>::ROWS;
    HDT_CUDA_CHECK(launch_dependent(k_bwd_tile<D>, true, dim3(a.nb * ((a.block_rows + ROWS - 1) / ROWS), a.H), TILE_THREADS, smem, st, a));
    return HDT_OK;
}
int launch_fwd_tile(const TileFwdArgs &a, int D, cudaStream_t st) {
    if (D == 64) return launch_fwd_tile_t<64>(a, st);
    if (D == 128) return launch_fwd_tile_t<128>(a, st);
    return set_error(HDT_ERR_UNSUPPORTED, "head_dim %d not supported (64 or 128)", D);
}
int launch_bwd_tile(const TileBwdArgs &a, int D, cudaStream_t st) {
    if (D == 64) return launch_bwd_tile_t<64>(a, st);
    if (D == 128) return launch_bwd_tile_t<128>(a, st);
    return set_error(HDT_ERR_UNSUPPORTED, "head_dim %d not supported (64 or 128)", D);
}

// Groups of lanes per row.  A row's time is its chain of chunks (about two round trips to L2 each), the launch's that
// chain times the number of times the rows fill the SMs: take the split with the smallest product.  keys: mean
// keys of a row, chunk: keys a group takes at a time, warps: warps resident on an SM.
static int row_groups(long long rows, int D, float keys, int chunk, int warps, int n_sm) {
    int best = 1;
    double least = 0;
    for (int kp = 1; kp <= 256 / D; kp *= 2) {
        const double lanes = (double)rows * kp * (D / 8), waves = lanes / (32.0 * n_sm * warps);
        const double t = (waves < 1 ? 1 : waves) * (keys / (chunk * kp) + 2.5 + (kp > 1 ? 0.5 : 0));
        if (kp == 1 || t < least) { best = kp; least = t; }
    }
    return best;
}
template <int D, bool BF16>
static int launch_fwd_rows_t(const RowFwdArgs &a, cudaStream_t st) {
    const long long rows = (long long)a.n * a.H;
    if (rows == 0) return HDT_OK;
    int n_sm = 0;
    if (const int rc = sm_count(&n_sm)) return rc;
    const int kp = row_groups(rows, D, a.keys, a.first ? 8 : 4, BF16 ? 16 : 12, n_sm);
    const unsigned grid = (unsigned)((rows * kp * (D / 8) + ROW_THREADS - 1) / ROW_THREADS);
    auto *kern = kp == 4 ? k_fwd_rows<D, BF16, D == 64 ? 4 : 1, 8> : kp == 2 ? k_fwd_rows<D, BF16, 2, 8> : a.first ? k_fwd_rows<D, BF16, 1, 8> : k_fwd_rows<D, BF16, 1, 4>;
    HDT_CUDA_CHECK(launch_dependent(kern, true, dim3(grid), ROW_THREADS, 0, st, a));
    return HDT_OK;
}
template <int D, bool BF16, bool DELTA>
static int launch_bwd_rows_t(const RowBwdArgs &a, cudaStream_t st) {
    const long long rows = (long long)a.n * a.H;
    if (rows == 0) return HDT_OK;
    int n_sm = 0;
    if (const int rc = sm_count(&n_sm)) return rc;
    const int kp = row_groups(rows, D, a.keys, 2, BF16 ? 16 : 12, n_sm);
    const unsigned grid = (unsigned)((rows * kp * (D / 8) + ROW_THREADS - 1) / ROW_THREADS);
    auto *kern = kp == 4 ? k_bwd_rows<D, BF16, D == 64 ? 4 : 1, DELTA> : kp == 2 ? k_bwd_rows<D, BF16, 2, DELTA> : k_bwd_rows<D, BF16, 1, DELTA>;
    HDT_CUDA_CHECK(launch_dependent(kern, true, dim3(grid), ROW_THREADS, 0, st, a));
    return HDT_OK;
}
int launch_fwd_rows(const RowFwdArgs &a, int D, int dtype, cudaStream_t st) {
    if (D == 64) return dtype == HDT_BF16 ? launch_fwd_rows_t<64, true>(a, st) : launch_fwd_rows_t<64, false>(a, st);
    if (D == 128) return dtype == HDT_BF16 ? launch_fwd_rows_t<128, true>(a, st) : launch_fwd_rows_t<128, false>(a, st);
    return set_error(HDT_ERR_UNSUPPORTED, "head_dim %d not supported (64 or 128)", D);
}
template <int D, bool BF16>
static int launch_bwd_rows_d(const RowBwdArgs &a, cudaStream_t st) {
    return a.delta ? launch_bwd_rows_t<D, BF16, true>(a, st) : launch_bwd_rows_t<D, BF16, false>(a, st);
}
int launch_bwd_rows(const RowBwdArgs &a, int D, int dtype, cudaStream_t st) {
    if (D == 64) return dtype == HDT_BF16 ? launch_bwd_rows_d<64, true>(a, st) : launch_bwd_rows_d<64, false>(a, st);
    if (D == 128) return dtype == HDT_BF16 ? launch_bwd_rows_d<128, true>(a, st) : launch_bwd_rows_d<128, false>(a, st);
    return set_error(HDT_ERR_UNSUPPORTED, "head_dim %d not supported (64 or 128)", D);
}

}  // namespace hdt
