// Building blocks of the row-wise kernels: a row of head_dim values on head_dim / 8 lanes of a warp, dot products
// with a chunk of keys, their reduction, the online softmax.
#pragma once
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

namespace hdt {

using f2 = unsigned long long;      // two packed floats (Blackwell issues a packed fma as one instruction)
__device__ __forceinline__ f2 pack2(float a, float b) { f2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ void unpack2(f2 x, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x)); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { f2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { f2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ f2 add2(f2 a, f2 b) { f2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }

// Eight values of a row as loaded, and as four packed pairs.  Of a row of 8 N values lane g < N holds the values
// 8 g .. 8 g + 7 (bf16: one 16-byte load) or 4 g .. + 3 and 4 N + 4 g .. + 3 (fp32: two loads, each contiguous
// over the lanes).  r: row number (token * heads + head).
template <bool BF16, int N> struct Raw;
template <int N> struct Raw<true, N> {
    uint4 u;
    __device__ __forceinline__ void load(const void *p, unsigned r, int g) { u = __ldg(reinterpret_cast<const uint4 *>(p) + r * N + g); }
    static __device__ __forceinline__ f2 two(uint32_t x) { return pack2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u)); }
    __device__ __forceinline__ void get(f2 (&v)[4]) const { v[0] = two(u.x); v[1] = two(u.y); v[2] = two(u.z); v[3] = two(u.w); }
    static __device__ __forceinline__ void store(void *p, unsigned r, int g, const f2 (&v)[4]) {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float a, b;
            unpack2(v[k], a, b);
            const __nv_bfloat162 x = __floats2bfloat162_rn(a, b);
            w[k] = *reinterpret_cast<const uint32_t *>(&x);
        }
        reinterpret_cast<uint4 *>(p)[r * N + g] = make_uint4(w[0], w[1], w[2], w[3]);
    }
    // the same values of an fp32 row (partial results)
    static __device__ __forceinline__ void store_f32(float *p, size_t r, int g, const f2 (&v)[4]) {
        float4 x, y;
        unpack2(v[0], x.x, x.y); unpack2(v[1], x.z, x.w); unpack2(v[2], y.x, y.y); unpack2(v[3], y.z, y.w);
        float4 *q = reinterpret_cast<float4 *>(p) + (r * N + g) * 2;
        q[0] = x; q[1] = y;
    }
    static __device__ __forceinline__ void load_f32(const float *p, size_t r, int g, f2 (&v)[4]) {
        const float4 *q = reinterpret_cast<const float4 *>(p) + (r * N + g) * 2;
        const float4 x = q[0], y = q[1];
        v[0] = pack2(x.x, x.y); v[1] = pack2(x.z, x.w); v[2] = pack2(y.x, y.y); v[3] = pack2(y.z, y.w);
    }
};
template <int N> struct Raw<false, N> {
    float4 a, b;
    __device__ __forceinline__ void load(const void *p, unsigned r, int g) {
        const float4 *q = reinterpret_cast<const float4 *>(p) + (size_t)r * (2 * N) + g;
        a = __ldg(q); b = __ldg(q + N);
    }
    __device__ __forceinline__ void load_smem(const float4 *row, int g) { a = row[g]; b = row[N + g]; }
    __device__ __forceinline__ void get(f2 (&v)[4]) const { v[0] = pack2(a.x, a.y); v[1] = pack2(a.z, a.w); v[2] = pack2(b.x, b.y); v[3] = pack2(b.z, b.w); }
    static __device__ __forceinline__ void store(void *p, unsigned r, int g, const f2 (&v)[4]) {
        float4 x, y;
        unpack2(v[0], x.x, x.y); unpack2(v[1], x.z, x.w); unpack2(v[2], y.x, y.y); unpack2(v[3], y.z, y.w);
        float4 *q = reinterpret_cast<float4 *>(p) + (size_t)r * (2 * N) + g;
        q[0] = x; q[N] = y;
    }
    static __device__ __forceinline__ void store_f32(float *p, size_t r, int g, const f2 (&v)[4]) { store(p, (unsigned)r, g, v); }
    static __device__ __forceinline__ void load_f32(const float *p, size_t r, int g, f2 (&v)[4]) {
        const float4 *q = reinterpret_cast<const float4 *>(p) + r * (2 * N) + g;
        const float4 x = q[0], y = q[N];
        v[0] = pack2(x.x, x.y); v[1] = pack2(x.z, x.w); v[2] = pack2(y.x, y.y); v[3] = pack2(y.z, y.w);
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

template <class R>
__device__ __forceinline__ float dot(const R &a, const R &b) {
    f2 x[4], y[4];
    a.get(x); b.get(y);
    return dot8(x, y);
}
template <int C, class R>
__device__ __forceinline__ void dots(const R &a, const R (&b)[C], float (&out)[C]) {
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
template <int C, class R>
__device__ __forceinline__ void axpys(f2 (&acc)[4], float w, const R (&x)[C], unsigned mask, int src) {
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

// A row's online softmax: maximum (log2), sum (this lane's keys only) and accumulator.
struct RowSoftmax {
    float m, l;
    f2 acc[4];
    __device__ __forceinline__ void clear() {
        m = -INFINITY; l = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = 0ull;
    }
    // x: score of this lane's key (-inf: none).  Returns its weight.
    template <int C>
    __device__ __forceinline__ float add(float x, unsigned mask) {
        float mx = x;
#pragma unroll
        for (int o = 1; o < C; o *= 2) mx = fmaxf(mx, __shfl_xor_sync(mask, mx, o));
        mx = fmaxf(mx, m);
        const float ref = mx > -INFINITY ? mx : 0.f;
        const float p = exp2f(x - ref), al = exp2f(m - ref);
        m = mx;
        l = l * al + p;
        const f2 al2 = pack2(al, al);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = mul2(acc[i], al2);
        return p;
    }
    // another partial result: maximum, sum, accumulator
    __device__ __forceinline__ void merge(float m2, float l2, const f2 (&acc2)[4]) {
        const float mx = fmaxf(m, m2), ref = mx > -INFINITY ? mx : 0.f;
        const float w1 = exp2f(m - ref), w2 = exp2f(m2 - ref);
        const f2 p1 = pack2(w1, w1), p2 = pack2(w2, w2);
        l = l * w1 + l2 * w2;
        m = mx;
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = fma2(p2, acc2[i], mul2(acc[i], p1));
    }
    __device__ __forceinline__ float finish() {         // normalises; natural-log LSE
        const float inv = l > 0.f ? 1.f / l : 0.f;
        const f2 i2 = pack2(inv, inv);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = mul2(acc[i], i2);
        return l > 0.f ? (m + log2f(l)) * 0.6931471805599453f : -INFINITY;
    }
};

}  // namespace hdt
