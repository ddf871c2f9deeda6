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

// Eight consecutive values of a row as loaded, and as four packed pairs.
template <bool BF16> struct Raw;
template <> struct Raw<true> {
    uint4 u;
    __device__ __forceinline__ void load(const void *p, size_t i) { u = __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<const __nv_bfloat16 *>(p) + i)); }
    __device__ __forceinline__ void zero() { u = make_uint4(0, 0, 0, 0); }
    static __device__ __forceinline__ f2 two(uint32_t x) { return pack2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u)); }
    __device__ __forceinline__ void get(f2 (&v)[4]) const { v[0] = two(u.x); v[1] = two(u.y); v[2] = two(u.z); v[3] = two(u.w); }
    static __device__ __forceinline__ void store(void *p, size_t i, const f2 (&v)[4]) {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float a, b;
            unpack2(v[k], a, b);
            const __nv_bfloat162 x = __floats2bfloat162_rn(a, b);
            w[k] = *reinterpret_cast<const uint32_t *>(&x);
        }
        *reinterpret_cast<uint4 *>(reinterpret_cast<__nv_bfloat16 *>(p) + i) = make_uint4(w[0], w[1], w[2], w[3]);
    }
};
template <> struct Raw<false> {
    float4 a, b;
    __device__ __forceinline__ void load(const void *p, size_t i) {
        const float4 *q = reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(p) + i);
        a = __ldg(q); b = __ldg(q + 1);
    }
    __device__ __forceinline__ void zero() { a = b = make_float4(0.f, 0.f, 0.f, 0.f); }
    __device__ __forceinline__ void get(f2 (&v)[4]) const { v[0] = pack2(a.x, a.y); v[1] = pack2(a.z, a.w); v[2] = pack2(b.x, b.y); v[3] = pack2(b.z, b.w); }
    static __device__ __forceinline__ void store(void *p, size_t i, const f2 (&v)[4]) {
        float4 x, y;
        unpack2(v[0], x.x, x.y); unpack2(v[1], x.z, x.w); unpack2(v[2], y.x, y.y); unpack2(v[3], y.z, y.w);
        float4 *q = reinterpret_cast<float4 *>(reinterpret_cast<float *>(p) + i);
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

// ---------------------------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------------------------
template <int D, bool BF16, int KP>
__global__ void __launch_bounds__(ROW_THREADS) k_fwd_rows(const RowFwdArgs a) {
    constexpr int LPK = D / 8, G = LPK * KP, C = 8;
    const float NEG = -INFINITY;
    const int lane = threadIdx.x & 31, sub = lane % G, g = sub % LPK, kp = sub / LPK;
    const unsigned all = G == 32 ? 0xffffffffu : ((1u << G) - 1u) << (lane - sub);     // the lanes of the row
    const int src = lane - g;                                                             // and of the group that shares a key
    const unsigned mask = ((1u << LPK) - 1u) << src;
    const unsigned long long id = ((unsigned long long)blockIdx.x * ROW_THREADS + threadIdx.x) / G;
    if (id >= (unsigned long long)a.n * a.H) return;
    int e = (int)(id / a.H);
    const int h = (int)(id % a.H), e_first = e;
    const int t = a.first ? a.st[a.first].tok[e] : e;
    const size_t row = ((size_t)t * a.H + h) * D + 8 * g;
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
    for (int s = a.first; ; ++s) {
        const RowStage &S = a.st[s];
        const int2 r = __ldg(reinterpret_cast<const int2 *>(S.rng) + e);
        const int up = __ldg(S.up + e);
        for (int j0 = r.x + kp * C; j0 < r.y; j0 += KP * C) {
            const int jm = j0 + (g & (C - 1));
            const bool ok = jm < r.y && (a.dirs == 7 || dir_ok(e, jm, r.x, a.dirs));
            int tm = jm < r.y ? jm : r.y - 1;         // (keys past the end read the last one: in bounds, weight 0)
            if (s) tm = __ldg(S.tok + tm);
            Raw<BF16> kr[C], vr[C];
            size_t at[C];
#pragma unroll
            for (int i = 0; i < C; ++i) {
                at[i] = ((size_t)__shfl_sync(mask, tm, src + i, 32) * a.H + h) * D + 8 * g;
                kr[i].load(a.k, at[i]);
            }
#pragma unroll
            for (int i = 0; i < C; ++i) vr[i].load(a.v, at[i]);
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
        if (up < 0) break;
        e = up;
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
        const size_t r1 = (size_t)e_first * a.H + h;
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
__global__ void __launch_bounds__(ROW_THREADS) k_bwd_rows(const RowBwdArgs a) {
    constexpr int LPK = D / 8, G = LPK * KP, C = 4;
    const int lane = threadIdx.x & 31, sub = lane % G, g = sub % LPK, kp = sub / LPK;
    const unsigned all = G == 32 ? 0xffffffffu : ((1u << G) - 1u) << (lane - sub);     // the lanes of the row
    const int src = lane - g;                                                             // and of the group that shares a key
    const unsigned mask = ((1u << LPK) - 1u) << src;
    const unsigned long long id = ((unsigned long long)blockIdx.x * ROW_THREADS + threadIdx.x) / G;
    if (id >= (unsigned long long)a.n * a.H) return;
    int e = (int)(id / a.H);
    const int h = (int)(id % a.H), e_first = e;
    const int t = a.first ? a.st[a.first].tok[e] : e;
    const size_t row = ((size_t)t * a.H + h) * D + 8 * g;
    const float L2E = 1.4426950408889634f;
    f2 q[4], k[4], v[4], go[4], dq[4], dk[4], dv[4];
    float lse_i, dl_i;
    {
        Raw<BF16> rq, rk, rv, rg;
        rq.load(a.q, row); rk.load(a.k, row); rv.load(a.v, row); rg.load(a.d_o, row);
        lse_i = __ldg(a.lse + (size_t)h * a.T + t) * L2E;
        const f2 c = pack2(a.scale_log2, a.scale_log2);
        rq.get(q); rk.get(k); rv.get(v); rg.get(go);
        if constexpr (DELTA) dl_i = __ldg(a.delta + (size_t)h * a.T + t);
        else {
            Raw<BF16> ro;
            f2 o[4];
            ro.load(a.o, row);
            ro.get(o);
            dl_i = dot8(go, o);
#pragma unroll
            for (int x = 1; x < LPK; x *= 2) dl_i += __shfl_xor_sync(mask, dl_i, x);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) { q[i] = mul2(q[i], c); k[i] = mul2(k[i], c); dq[i] = dk[i] = dv[i] = 0ull; }
    }
    for (int s = a.first; ; ++s) {
        const RowStage &S = a.st[s];
        const int2 r = __ldg(reinterpret_cast<const int2 *>(S.rng) + e);
        const int up = __ldg(S.up + e);
        for (int j0 = r.x + kp * C; j0 < r.y; j0 += KP * C) {
            const int jm = j0 + (g & (C - 1));
            const bool in = jm < r.y;
            const bool ok_q = in && (a.dirs == 7 || dir_ok(e, jm, r.x, a.dirs));          // the row attends to it
            const bool ok_k = in && (a.dirs == 7 || dir_ok_key(e, jm, r.x, a.dirs));      // it attends to the row
            int tm = in ? jm : r.y - 1;
            if (s) tm = __ldg(S.tok + tm);
            const float lse_j = __ldg(a.lse + (size_t)h * a.T + tm) * L2E;
            float dl_j = 0.f;
            if constexpr (DELTA) dl_j = __ldg(a.delta + (size_t)h * a.T + tm);
            Raw<BF16> kr[C], qr[C], gr[C], xr[C];
            size_t at[C];
#pragma unroll
            for (int i = 0; i < C; ++i) {
                at[i] = ((size_t)__shfl_sync(mask, tm, src + i, 32) * a.H + h) * D + 8 * g;
                kr[i].load(a.k, at[i]);
                xr[i].load(a.v, at[i]);
            }
#pragma unroll
            for (int i = 0; i < C; ++i) { qr[i].load(a.q, at[i]); gr[i].load(a.d_o, at[i]); }
            float sc[C], x1[C], x2[C], x3[C];
#pragma unroll
            for (int i = 0; i < C; ++i) {
                f2 y[4];
                kr[i].get(y); sc[i] = dot8(q, y);
                xr[i].get(y); x1[i] = dot8(go, y);
                qr[i].get(y); x2[i] = dot8(k, y);
                gr[i].get(y); x3[i] = dot8(v, y);
            }
            if constexpr (!DELTA) {
                float x4[C];
#pragma unroll
                for (int i = 0; i < C; ++i) {
                    f2 y[4], z[4];
                    xr[i].load(a.o, at[i]);
                    xr[i].get(y); gr[i].get(z);
                    x4[i] = dot8(z, y);
                }
                dl_j = reduce_scatter<C, LPK>(x4, g, mask);
            }
            const float s_ij = reduce_scatter<C, LPK>(sc, g, mask), dp_ij = reduce_scatter<C, LPK>(x1, g, mask);
            const float s_ji = reduce_scatter<C, LPK>(x2, g, mask), dp_ji = reduce_scatter<C, LPK>(x3, g, mask);
            const float p_ij = ok_q ? exp2f(s_ij - lse_i) : 0.f, p_ji = ok_k ? exp2f(s_ji - lse_j) : 0.f;
            const float ds_ij = p_ij * (dp_ij - dl_i), ds_ji = p_ji * (dp_ji - dl_j);
#pragma unroll
            for (int i = 0; i < C; ++i) {
                const float w1 = __shfl_sync(mask, ds_ij, src + i, 32), w2 = __shfl_sync(mask, ds_ji, src + i, 32),
                            w3 = __shfl_sync(mask, p_ji, src + i, 32);
                const f2 c1 = pack2(w1, w1), c2 = pack2(w2, w2), c3 = pack2(w3, w3);
                f2 y[4];
                kr[i].get(y);
#pragma unroll
                for (int u = 0; u < 4; ++u) dq[u] = fma2(c1, y[u], dq[u]);
                qr[i].get(y);
#pragma unroll
                for (int u = 0; u < 4; ++u) dk[u] = fma2(c2, y[u], dk[u]);
                gr[i].get(y);
#pragma unroll
                for (int u = 0; u < 4; ++u) dv[u] = fma2(c3, y[u], dv[u]);
            }
        }
        if (up < 0) break;
        e = up;
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
            const size_t r1 = ((size_t)e_first * a.H + h) * D + 8 * g;
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

// Lanes per row: with few rows several groups of lanes share one, for latency; with many, one group each
// (no final merge, fewer idle lanes in short families).
template <int D, bool BF16>
static int launch_fwd_rows_t(const RowFwdArgs &a, cudaStream_t st) {
    const long long rows = (long long)a.n * a.H;
    if (rows == 0) return HDT_OK;
    const bool share = rows * (D / 8) < 148LL * 1024;
    const int g = share ? 32 : D / 8;
    const unsigned grid = (unsigned)((rows * g + ROW_THREADS - 1) / ROW_THREADS);
    if (share) k_fwd_rows<D, BF16, 256 / D><<<grid, ROW_THREADS, 0, st>>>(a);
    else k_fwd_rows<D, BF16, 1><<<grid, ROW_THREADS, 0, st>>>(a);
    count_launch();
    HDT_CUDA_CHECK(cudaGetLastError());
    return HDT_OK;
}
template <int D, bool BF16>
static int launch_bwd_rows_t(const RowBwdArgs &a, cudaStream_t st) {
    const long long rows = (long long)a.n * a.H;
    if (rows == 0) return HDT_OK;
    const bool share = rows * (D / 8) < 148LL * 1024;
    const int g = share ? 32 : D / 8;
    const unsigned grid = (unsigned)((rows * g + ROW_THREADS - 1) / ROW_THREADS);
    if (a.delta) {
        if (share) k_bwd_rows<D, BF16, 256 / D, true><<<grid, ROW_THREADS, 0, st>>>(a);
        else k_bwd_rows<D, BF16, 1, true><<<grid, ROW_THREADS, 0, st>>>(a);
    } else {
        if (share) k_bwd_rows<D, BF16, 256 / D, false><<<grid, ROW_THREADS, 0, st>>>(a);
        else k_bwd_rows<D, BF16, 1, false><<<grid, ROW_THREADS, 0, st>>>(a);
    }
    count_launch();
    HDT_CUDA_CHECK(cudaGetLastError());
    return HDT_OK;
}
int launch_fwd_rows(const RowFwdArgs &a, int D, int dtype, cudaStream_t st) {
    if (D == 64) return dtype == HDT_BF16 ? launch_fwd_rows_t<64, true>(a, st) : launch_fwd_rows_t<64, false>(a, st);
    if (D == 128) return dtype == HDT_BF16 ? launch_fwd_rows_t<128, true>(a, st) : launch_fwd_rows_t<128, false>(a, st);
    return set_error(HDT_ERR_UNSUPPORTED, "head_dim %d not supported (64 or 128)", D);
}
int launch_bwd_rows(const RowBwdArgs &a, int D, int dtype, cudaStream_t st) {
    if (D == 64) return dtype == HDT_BF16 ? launch_bwd_rows_t<64, true>(a, st) : launch_bwd_rows_t<64, false>(a, st);
    if (D == 128) return dtype == HDT_BF16 ? launch_bwd_rows_t<128, true>(a, st) : launch_bwd_rows_t<128, false>(a, st);
    return set_error(HDT_ERR_UNSUPPORTED, "head_dim %d not supported (64 or 128)", D);
}

}  // namespace hdt
