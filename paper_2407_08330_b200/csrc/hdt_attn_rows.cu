// Row-wise attention kernels: a row (element, head) is owned by a few lanes of a warp that walk its keys in
// every stage the element lives in and write its final result.  One launch does what takes a launch per
// stage and a merge on the tile kernels, so they serve
//   - the stages above 0, behind stage 0 (whose partial result they add), where their families are short:
//     documents keep about 3 % of their tokens above stage 0, with a few dozen keys each, and a tile kernel
//     there is a chain of gather, MMA, softmax, MMA and scatter with 128 rows for a dozen used ones;
//   - all stages of batches whose families are tiny throughout (expression trees: six keys a row).
// All arithmetic is fp32 (P and dS are not rounded).
//
// Lanes: D / 8 lanes hold 8 dimensions each; a chunk of C keys is a C-fold load of 16 (bf16) or 32 (fp32)
// bytes per lane, all in flight together.  The C dot products are summed over the lanes by a reduce-scatter
// (C - 1 shuffles instead of 3 C or 4 C), which leaves one key's score per lane: one exponential per key
// and lane instead of one per key on every lane.  KP groups of lanes may share a row (each takes every
// KP-th chunk), for batches with too few rows to fill the SMs.
#include <cuda_bf16.h>

#include "hdt_internal.cuh"

namespace hdt {

using f2 = unsigned long long;      // two packed floats (Blackwell issues a packed fma as one instruction)
__device__ __forceinline__ f2 pack2(float a, float b) { f2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ void unpack2(f2 x, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x)); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { f2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { f2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ f2 add2(f2 a, f2 b) { f2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }

// Eight consecutive values of a row as loaded, and as four packed pairs.  Offsets count groups of eight values.
template <bool BF16> struct Raw;
template <> struct Raw<true> {
    uint4 u;
    __device__ __forceinline__ void load(const void *p, unsigned i) { u = __ldg(reinterpret_cast<const uint4 *>(p) + i); }
    __device__ __forceinline__ void zero() { u = make_uint4(0, 0, 0, 0); }
    static __device__ __forceinline__ f2 two(uint32_t x) { return pack2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u)); }
    __device__ __forceinline__ void get(f2 (&v)[4]) const { v[0] = two(u.x); v[1] = two(u.y); v[2] = two(u.z); v[3] = two(u.w); }
    static __device__ __forceinline__ void store(void *p, unsigned i, const f2 (&v)[4]) {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float a, b;
            unpack2(v[k], a, b);
            const __nv_bfloat162 x = __floats2bfloat162_rn(a, b);
            w[k] = *reinterpret_cast<const uint32_t *>(&x);
        }
        reinterpret_cast<uint4 *>(p)[i] = make_uint4(w[0], w[1], w[2], w[3]);
    }
};
template <> struct Raw<false> {
    float4 a, b;
    __device__ __forceinline__ void load(const void *p, unsigned i) {
        const float4 *q = reinterpret_cast<const float4 *>(p) + 2 * (size_t)i;
        a = __ldg(q); b = __ldg(q + 1);
    }
    __device__ __forceinline__ void zero() { a = b = make_float4(0.f, 0.f, 0.f, 0.f); }
    __device__ __forceinline__ void get(f2 (&v)[4]) const { v[0] = pack2(a.x, a.y); v[1] = pack2(a.z, a.w); v[2] = pack2(b.x, b.y); v[3] = pack2(b.z, b.w); }
    static __device__ __forceinline__ void store(void *p, unsigned i, const f2 (&v)[4]) {
        float4 x, y;
        unpack2(v[0], x.x, x.y); unpack2(v[1], x.z, x.w); unpack2(v[2], y.x, y.y); unpack2(v[3], y.z, y.w);
        float4 *q = reinterpret_cast<float4 *>(p) + 2 * (size_t)i;
        q[0] = x; q[1] = y;
    }
};
__device__ __forceinline__ float dot8(const f2 (&a)[4], const f2 (&b)[4]) {
    f2 s = mul2(a[0], b[0]);
    s = fma2(a[1], b[1], s);
    s = fma2(a[2], b[2], s);
    s = fma2(a[3], b[3], s);
    float x, y;
    unpack2(s, x, y);
    return x + y;
}

template <bool BF16>
__device__ __forceinline__ float dot(const Raw<BF16> &a, const Raw<BF16> &b) {
    f2 x[4], y[4];
    a.get(x); b.get(y);
    return dot8(x, y);
}
template <int C, bool BF16>
__device__ __forceinline__ void dots(const Raw<BF16> &a, const Raw<BF16> (&b)[C], float (&out)[C]) {
    f2 x[4];
    a.get(x);
#pragma unroll
    for (int i = 0; i < C; ++i) {
        f2 y[4];
        b[i].get(y);
        out[i] = dot8(x, y);
    }
}
// acc += sum over the chunk of w (one per lane) times its row
template <int C, bool BF16>
__device__ __forceinline__ void axpys(f2 (&acc)[4], float w, const Raw<BF16> (&x)[C], unsigned mask, int src) {
#pragma unroll
    for (int i = 0; i < C; ++i) {
        const float wi = __shfl_sync(mask, w, src + i, 32);
        const f2 w2 = pack2(wi, wi);
        f2 y[4];
        x[i].get(y);
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] = fma2(w2, y[u], acc[u]);
    }
}

// Sums of C values over the LPK lanes of a group; lane g keeps the total of value g % C.
template <int C, int LPK>
__device__ __forceinline__ float reduce_scatter(float (&v)[C], int g, unsigned mask) {
#pragma unroll
    for (int half = C / 2; half >= 1; half /= 2) {
        const bool upper = (g & half) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float send = upper ? v[i] : v[i + half], keep = upper ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(mask, send, half);
        }
    }
    float s = v[0];
#pragma unroll
    for (int o = C; o < LPK; o *= 2) s += __shfl_xor_sync(mask, s, o);
    return s;
}

static constexpr int ROW_THREADS = 128;

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
template <int D, bool BF16, int KP, int C>
__global__ void __launch_bounds__(ROW_THREADS) k_fwd_rows(const RowFwdArgs a) {
    constexpr int LPK = D / 8, G = LPK * KP;
    const float NEG = -INFINITY;
    const int lane = threadIdx.x & 31, sub = lane % G, g = sub % LPK, kp = sub / LPK;
    const unsigned all = G == 32 ? 0xffffffffu : ((1u << G) - 1u) << (lane - sub);     // the lanes of the row
    const int src = lane - g;                                                             // and of the group that shares a key
    const unsigned mask = ((1u << LPK) - 1u) << src;
    const unsigned long long id = ((unsigned long long)blockIdx.x * ROW_THREADS + threadIdx.x) / G;
    if (id >= (unsigned long long)a.n * a.H) return;
    const int e = (int)(id / a.H), h = (int)(id % a.H);
    const int t = a.first ? a.st[a.first].tok[e] : e;
    const unsigned row = ((unsigned)t * a.H + h) * LPK + g;
    f2 q[4], acc[4];
    {
        Raw<BF16> r;
        r.load(a.q, row);
        r.get(q);
        const f2 c = pack2(a.scale_log2, a.scale_log2);
#pragma unroll
        for (int i = 0; i < 4; ++i) { q[i] = mul2(q[i], c); acc[i] = 0ull; }
    }
    float m = NEG, l = 0.f;          // l: this lane's keys only
    RowCursor<C, KP * C> cur;
    bool more = cur.start(a.st, a.first, e, kp * C);
    int tm = more ? cur.token(g & (C - 1)) : 0;
    {
        while (more) {
            const int jm = cur.j0 + (g & (C - 1)), tc = tm;
            const bool ok = jm < cur.r.y && (a.dirs == 7 || dir_ok(cur.e, jm, cur.r.x, a.dirs));
            Raw<BF16> kr[C], vr[C];
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const unsigned at = ((unsigned)__shfl_sync(mask, tc, src + i, 32) * a.H + h) * LPK + g;
                kr[i].load(a.k, at);
                vr[i].load(a.v, at);
            }
            more = cur.next(kp * C);
            if (more) tm = cur.token(g & (C - 1));
            float sc[C];
#pragma unroll
            for (int i = 0; i < C; ++i) {
                f2 k[4];
                kr[i].get(k);
                sc[i] = dot8(q, k);
            }
            float x = reduce_scatter<C, LPK>(sc, g, mask);
            x = ok ? x : NEG;
            float mx = x;
#pragma unroll
            for (int o = 1; o < C; o *= 2) mx = fmaxf(mx, __shfl_xor_sync(mask, mx, o));
            mx = fmaxf(mx, m);
            const float ref = mx > NEG ? mx : 0.f;
            const float p = exp2f(x - ref), al = exp2f(m - ref);
            m = mx;
            l = l * al + p;
            const f2 al2 = pack2(al, al);
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = mul2(acc[i], al2);
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const float w = __shfl_sync(mask, p, src + i, 32);
                f2 v[4];
                vr[i].get(v);
                const f2 w2 = pack2(w, w);
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[u] = fma2(w2, v[u], acc[u]);
            }
        }
    }
    // l over the C lanes that hold different keys (lanes g and g + C of a 16-lane group hold the same ones)
#pragma unroll
    for (int o = 1; o < C; o *= 2) l += __shfl_xor_sync(mask, l, o);
#pragma unroll
    for (int o = LPK; o < G; o *= 2) {      // the groups that share the row
        const float m2 = __shfl_xor_sync(all, m, o), l2 = __shfl_xor_sync(all, l, o);
        const float mx = fmaxf(m, m2), ref = mx > NEG ? mx : 0.f;
        const float w1 = exp2f(m - ref), w2 = exp2f(m2 - ref);
        const f2 p1 = pack2(w1, w1), p2 = pack2(w2, w2);
        l = l * w1 + l2 * w2;
        m = mx;
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = fma2(p2, __shfl_xor_sync(all, acc[i], o), mul2(acc[i], p1));
    }
    if (a.base_o != nullptr) {              // stage 0's partial result, normalised, as one more key
        const size_t r1 = (size_t)e * a.H + h;
        const float s0 = a.base_lse[r1] * 1.4426950408889634f;
        const float4 *bo = reinterpret_cast<const float4 *>(a.base_o + r1 * D + 8 * g);
        const float4 x = bo[0], y = bo[1];
        const float mx = fmaxf(m, s0), ref = mx > NEG ? mx : 0.f;
        const float w1 = exp2f(m - ref), w0 = exp2f(s0 - ref);
        const f2 p1 = pack2(w1, w1), p0 = pack2(w0, w0);
        l = l * w1 + w0;
        m = mx;
        acc[0] = fma2(p0, pack2(x.x, x.y), mul2(acc[0], p1));
        acc[1] = fma2(p0, pack2(x.z, x.w), mul2(acc[1], p1));
        acc[2] = fma2(p0, pack2(y.x, y.y), mul2(acc[2], p1));
        acc[3] = fma2(p0, pack2(y.z, y.w), mul2(acc[3], p1));
    }
    if (kp == 0) {
        const float inv = l > 0.f ? 1.f / l : 0.f;
        const f2 i2 = pack2(inv, inv);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = mul2(acc[i], i2);
        Raw<BF16>::store(a.o, row, acc);
        if (g == 0) a.lse[(size_t)h * a.T + t] = l > 0.f ? (m + log2f(l)) * 0.6931471805599453f : NEG;
    }
}

// ---------------------------------------------------------------------------------------------
// backward
// ---------------------------------------------------------------------------------------------
// The family ranges of a stage are symmetric: the keys of a row are also the queries that attend to it, so
// one walk gives the row's dQ (as a query), dK and dV (as a key), each complete: no atomics.
// DELTA: rowsum(dO . O) is given; else it is computed from O here (one more row per key to read).
template <int D, bool BF16, int KP, bool DELTA>
__global__ void __launch_bounds__(ROW_THREADS, BF16 ? 4 : 3) k_bwd_rows(const RowBwdArgs a) {
    constexpr int LPK = D / 8, G = LPK * KP, C = BF16 ? 4 : 2;
    const int lane = threadIdx.x & 31, sub = lane % G, g = sub % LPK, kp = sub / LPK;
    const unsigned all = G == 32 ? 0xffffffffu : ((1u << G) - 1u) << (lane - sub);     // the lanes of the row
    const int src = lane - g;                                                             // and of the group that shares a key
    const unsigned mask = ((1u << LPK) - 1u) << src;
    const unsigned long long id = ((unsigned long long)blockIdx.x * ROW_THREADS + threadIdx.x) / G;
    if (id >= (unsigned long long)a.n * a.H) return;
    const int e = (int)(id / a.H), h = (int)(id % a.H);
    const int t = a.first ? a.st[a.first].tok[e] : e;
    const unsigned row = ((unsigned)t * a.H + h) * LPK + g;
    const float L2E = 1.4426950408889634f;
    // (the row's own values stay as loaded and are unpacked once per chunk: registers decide how many warps hide
    // the loads' latency here)
    Raw<BF16> q, k, v, go;
    f2 dq[4], dk[4], dv[4];
    q.load(a.q, row); k.load(a.k, row); v.load(a.v, row); go.load(a.d_o, row);
    const float lse_i = __ldg(a.lse + (size_t)h * a.T + t) * L2E;
    float dl_i;
    if constexpr (DELTA) dl_i = __ldg(a.delta + (size_t)h * a.T + t);
    else {
        Raw<BF16> ro;
        ro.load(a.o, row);
        dl_i = dot(go, ro);
#pragma unroll
        for (int x = 1; x < LPK; x *= 2) dl_i += __shfl_xor_sync(mask, dl_i, x);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) dq[i] = dk[i] = dv[i] = 0ull;
    RowCursor<C, KP * C> cur;
    bool more = cur.start(a.st, a.first, e, kp * C);
    int tm = more ? cur.token(g & (C - 1)) : 0;
    while (more) {
        const int jm = cur.j0 + (g & (C - 1)), tc = tm;
        const bool in = jm < cur.r.y;
        const bool ok_q = in && (a.dirs == 7 || dir_ok(cur.e, jm, cur.r.x, a.dirs));          // the row attends to it
        const bool ok_k = in && (a.dirs == 7 || dir_ok_key(cur.e, jm, cur.r.x, a.dirs));      // it attends to the row
        const float lse_j = __ldg(a.lse + (size_t)h * a.T + tc) * L2E;
        float dl_j = 0.f;
        if constexpr (DELTA) dl_j = __ldg(a.delta + (size_t)h * a.T + tc);
        Raw<BF16> x[C], y[C];
        unsigned at[C];
        float v1[C], v2[C];
        // the row as a query: K and V of its keys
#pragma unroll
        for (int i = 0; i < C; ++i) {
            at[i] = ((unsigned)__shfl_sync(mask, tc, src + i, 32) * a.H + h) * LPK + g;
            x[i].load(a.k, at[i]);
            y[i].load(a.v, at[i]);
        }
        more = cur.next(kp * C);
        if (more) tm = cur.token(g & (C - 1));
        dots<C>(q, x, v1);
        dots<C>(go, y, v2);
        {
            const float s_ij = reduce_scatter<C, LPK>(v1, g, mask) * a.scale_log2, dp_ij = reduce_scatter<C, LPK>(v2, g, mask);
            const float p_ij = ok_q ? exp2f(s_ij - lse_i) : 0.f;
            axpys<C>(dq, p_ij * (dp_ij - dl_i), x, mask, src);
        }
        // the row as a key: Q and dO of the queries that attend to it
#pragma unroll
        for (int i = 0; i < C; ++i) {
            x[i].load(a.q, at[i]);
            y[i].load(a.d_o, at[i]);
        }
        if constexpr (!DELTA) {
            float v3[C];
#pragma unroll
            for (int i = 0; i < C; ++i) {
                Raw<BF16> o;
                o.load(a.o, at[i]);
                v3[i] = dot(o, y[i]);
            }
            dl_j = reduce_scatter<C, LPK>(v3, g, mask);
        }
        dots<C>(k, x, v1);
        dots<C>(v, y, v2);
        const float s_ji = reduce_scatter<C, LPK>(v1, g, mask) * a.scale_log2, dp_ji = reduce_scatter<C, LPK>(v2, g, mask);
        const float p_ji = ok_k ? exp2f(s_ji - lse_j) : 0.f;
        axpys<C>(dk, p_ji * (dp_ji - dl_j), x, mask, src);
        axpys<C>(dv, p_ji, y, mask, src);
    }
#pragma unroll
    for (int o = LPK; o < G; o *= 2) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            dq[i] = add2(dq[i], __shfl_xor_sync(all, dq[i], o));
            dk[i] = add2(dk[i], __shfl_xor_sync(all, dk[i], o));
            dv[i] = add2(dv[i], __shfl_xor_sync(all, dv[i], o));
        }
    }
    if (kp == 0) {
        const f2 c = pack2(a.scale, a.scale);
#pragma unroll
        for (int i = 0; i < 4; ++i) { dq[i] = mul2(dq[i], c); dk[i] = mul2(dk[i], c); }
        if (a.base[0] != nullptr) {         // stage 0's partial gradients
            const size_t r1 = ((size_t)e * a.H + h) * D + 8 * g;
            auto plus = [&](f2 (&x)[4], const float *b) {
                const float4 y = *reinterpret_cast<const float4 *>(b + r1), z = *reinterpret_cast<const float4 *>(b + r1 + 4);
                x[0] = add2(x[0], pack2(y.x, y.y)); x[1] = add2(x[1], pack2(y.z, y.w));
                x[2] = add2(x[2], pack2(z.x, z.y)); x[3] = add2(x[3], pack2(z.z, z.w));
            };
            plus(dq, a.base[0]); plus(dk, a.base[1]); plus(dv, a.base[2]);
        }
        Raw<BF16>::store(a.dq, row, dq);
        Raw<BF16>::store(a.dk, row, dk);
        Raw<BF16>::store(a.dv, row, dv);
    }
}

// Lanes per row: while all rows fit on the SMs at once several groups of lanes share one, for latency; beyond, one
// group each (no final merge, fewer idle lanes in short families).
static int row_groups(long long rows, int D) {
    for (int kp = 256 / D; kp > 1; kp /= 2)
        if (rows * kp * (D / 8) <= 148LL * 20 * 32) return kp;
    return 1;
}
template <int D, bool BF16>
static int launch_fwd_rows_t(const RowFwdArgs &a, cudaStream_t st) {
    const long long rows = (long long)a.n * a.H;
    if (rows == 0) return HDT_OK;
    const int kp = row_groups(rows, D);
    const unsigned grid = (unsigned)((rows * kp * (D / 8) + ROW_THREADS - 1) / ROW_THREADS);
    if (kp == 4) k_fwd_rows<D, BF16, D == 64 ? 4 : 1, 8><<<grid, ROW_THREADS, 0, st>>>(a);
    else if (kp == 2) k_fwd_rows<D, BF16, 2, 8><<<grid, ROW_THREADS, 0, st>>>(a);
    else if (a.first) k_fwd_rows<D, BF16, 1, 8><<<grid, ROW_THREADS, 0, st>>>(a);
    else k_fwd_rows<D, BF16, 1, 4><<<grid, ROW_THREADS, 0, st>>>(a);
    count_launch();
    HDT_CUDA_CHECK(cudaGetLastError());
    return HDT_OK;
}
template <int D, bool BF16, bool DELTA>
static int launch_bwd_rows_t(const RowBwdArgs &a, cudaStream_t st) {
    const long long rows = (long long)a.n * a.H;
    if (rows == 0) return HDT_OK;
    const int kp = row_groups(2 * rows, D);
    const unsigned grid = (unsigned)((rows * kp * (D / 8) + ROW_THREADS - 1) / ROW_THREADS);
    if (kp == 4) k_bwd_rows<D, BF16, D == 64 ? 4 : 1, DELTA><<<grid, ROW_THREADS, 0, st>>>(a);
    else if (kp == 2) k_bwd_rows<D, BF16, 2, DELTA><<<grid, ROW_THREADS, 0, st>>>(a);
    else k_bwd_rows<D, BF16, 1, DELTA><<<grid, ROW_THREADS, 0, st>>>(a);
    count_launch();
    HDT_CUDA_CHECK(cudaGetLastError());
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
