// Decoder cross-attention to a level subset of the encoder tokens (paper, paragraph "Results on
// FacetSum (Encoder-Decoder Models)": the decoder attends only to [SEC] anchors, to [SEC] and
// [SENT] anchors, or to all tokens of the encoder output; decoder of the paragraph "Hierarchical
// Encoder and Decoder Stacks").  Within the chosen subset it is plain softmax attention between
// the decoder rows of a document and the chosen encoder rows of the same document.
//
// The chosen rows are never copied.
//   few decoder rows a document (a step of autoregressive decoding): k_cross_decode reads levels, K and V once, the
//         tokens of a document dealt to many CTAs, and k_cross_combine merges their partial results.  No index.
//   otherwise k_cross_index (of large batches behind a count and a scan) builds one element space for both sides: elements 0 .. Tq-1 are
//         the decoder rows (token map = identity, into Q / dO / O), elements Tq .. Tq+ns-1 the chosen
//         encoder tokens in order (token map = their index, into K / V); a decoder row's key range is its
//         document's slice of the second part, a chosen token's range the document's decoder rows.  The
//         attention kernels of the hierarchical path take any (row blocks, per-row range, token map)
//         description, so they serve as they are:
//   bf16  the gathering tcgen05 kernels (128-row blocks): forward over the decoder-row blocks;
//         backward in one launch over the decoder-row blocks (dQ) and the blocks of chosen
//         tokens (dK, dV); their epilogues round to bf16 and write each element's rows at its token in
//         the caller's tensors.  Long key lists are split over CTAs, whose fp32 partial results
//         k_cross_combine merges;
//   fp32  the SIMT kernels (32-row blocks), which write the caller's tensors directly.
// Encoder rows outside the subset get zero dK, dV from a kernel of their own beside the others.  Block slots are
// assigned without a scan: document b owns the slots from start / rows_per_block + b on, unused slots stay
// empty (r0 == r1).
#include <cuda_bf16.h>

#include "hdt_internal.cuh"
#include "hdt_rows.cuh"

namespace hdt {

constexpr int XC = 32;      // CTAs (contiguous chunks) per document in the index kernel
constexpr int DEC_LIST = 1024, DEC_ROWS = 8;     // decode kernel: tokens looked over at a time, rows of a document walked by one CTA

struct CrossLayout {
    size_t sel, used, tokx, rngx, blocks, queue, delta, part, part_lse, total;
    int nbq, nbk, xr;
};

static size_t al256c(size_t v) { return (v + 255) & ~size_t(255); }

// Decoding: few decoder rows a document on average (the host knows no more; k_cross_decode deals a document's rows beyond
// its first DEC_ROWS to CTAs of their own).  Every row reads its document's K and V again, while the other path's 128-row tile costs the
// same up to 128 rows.  us a forward call of 1, 4, 5 and 8 rows a document, bf16, here and (in brackets) on the tiles: 4 x 8192 tokens with
// 12 x 64 heads 19, 50, 58, 94 (85); 8 x 2048 14, 27, 31, 49 (53); 1 x 4096 with 16 x 128 14, 36, 43, 64 (35); 64 x 2048 75, 264, 326,
// 512 (262); 4 x 8192, anchors alone, 10, 15, 17, 23 (36).  All rows of a batch of 4 a document on one of 64 x 2048
// 186 (99), of 256 x 512 163 (72).  (fp32 tiles cost far more: 4 x 2048 at 8 rows 50 (722); the line stays where bf16 has it.)
static bool cross_decode(int B, int Tq) { return (long long)Tq <= 4LL * B; }
// Shape of a CTA of the decode kernel: heads side by side (lanes of 8 dimensions each), keys at a time.
struct DecodeShape {
    int HC, KS, threads, per_sm;           // per_sm: CTAs an SM's registers hold (64 a thread)
    DecodeShape(int H, int D) {
        const int lpk = D / 8;
        HC = min(H, 512 / lpk);
        KS = max(1, min(16, 384 / (HC * lpk)));
        threads = (HC * lpk * KS + 31) / 32 * 32;
        per_sm = 1024 / threads;
    }
};
// How the decode kernel deals a batch's tokens: in pieces of P of them, so that a long document has its share of the CTAs
// whatever the others are.  Up to DEC_DOCS documents, whose lengths a warp sees at once: ceil(n / P) for a document of n tokens, P the
// shortest of three (32 at least) of which there are no more than CTAs fit on the SMs at once: the shortest of which documents of one
// length have no more; the CTAs' mean share, half a CTA a document kept back; and with one a document kept back, which always fits.
// More documents: max(1, n / P) of even length, P the mean share, of which every document leaves half a piece.
// us a call of one row a document, bf16, 12 x 64 heads, and in brackets with the same number of pieces for every document: documents of
// one length, 4 x 8192 18.8 (18.4), 8 x 2048 13.5 (13.5), 64 x 2048 73.6 (72.2), 256 x 512 73.8 (71.0), with 16 x 128 8 x 1500 21.8 (21.3);
// one long one, 8192 + 15 x 512 13.6 (25.3), 8192 + 63 x 256 18 (106), 4096 + 200 x 128 21 (282); 16 from 200 to 16384 72 (104).  (A CTA
// begins with a chain of loads, so a second wave costs more than its shorter pieces save: 4 x 8192 at four CTAs an SM of which two fit 27.3, three
// 28.5, six 31.7, two 23.5, timed one behind the other with the form before.)
constexpr int DEC_DOCS = 31;         // (a lane each, and the end of the last)
struct DecodePieces {
    int piece[3], ctas, pieces, most, rows;   // pieces: CTAs for them; most: those of documents of several, at most; rows: decoder rows of a document that leave partial results there
    float inv[3];                    // 1 / piece
    int splits;                      // pieces of a document of more than DEC_ROWS decoder rows
    bool several;                    // whether a document may have several
    DecodePieces() = default;
    DecodePieces(int B, int T, int Tq, int H, int D) {
        const DecodeShape d(H, D);
        ctas = max(1, PLAN_SMS * d.per_sm / ((H + d.HC - 1) / d.HC));
        B = max(B, 1);
        const int mean = (int)(((long long)T + B - 1) / B), n = max(1, ctas / B);
        auto share = [&](int c) { return (int)(((long long)T + max(1, c) - 1) / max(1, c)); };
        piece[0] = max(32, B > DEC_DOCS ? T / ctas : (mean + n - 1) / n);
        piece[1] = max(piece[0], share(ctas - B / 2));
        piece[2] = max(piece[1], share(ctas - B));
        for (int i = 0; i < 3; ++i) inv[i] = 1.0f / (float)piece[i];
        most = B > DEC_DOCS ? T / piece[0] : min(T / piece[0] + B, max(ctas, B));      // (up to DEC_DOCS: no more than CTAs fit, or one each)
        pieces = B > DEC_DOCS ? most + B : most;
        several = B > DEC_DOCS ? most >= 2 : T > piece[0];
        rows = min(Tq, DEC_ROWS);
        splits = max(1, (int)min((mean + 31LL) / 32, (4LL * PLAN_SMS + B - 1) / B));
    }
    size_t part(int Tq) const { return (size_t)most * rows + (Tq > DEC_ROWS ? (size_t)splits * Tq : 0); }      // rows of partial results in all
};
// x / d for 0 <= x, 0 < d, shorter than the integer division.  Both conversions and the quotient are off by 2^-21 of it at most, so below 2^20
// the first guess is off by one at most.
__device__ __forceinline__ int quotient(int x, int d) {
    const int q = (int)__fdividef((float)x, (float)d);
    if (q >= 1 << 20) return x / d;
    const int r = x - q * d;
    return q + (r >= d) - (r < 0);
}
__device__ __forceinline__ int doc_pieces(int tokens, int piece) { return max(1, quotient(tokens, piece)); }
// Up to DEC_DOCS documents: P, and of lane b's document (k0, k1: its tokens) the pieces n and the number `base` of the first one.
// By a whole warp.  (The division as above: there are fewer than 2^20 pieces.)
__device__ __forceinline__ int choose_piece(const DecodePieces &p, int B, int tokens, int &n, int &base) {
    const int lane = threadIdx.x & 31;
    int n3[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int q = (int)((float)tokens * p.inv[i]), r = tokens - q * p.piece[i];
        n3[i] = lane < B ? max(1, q + (r > 0) + (r > p.piece[i]) - (r <= -p.piece[i])) : 0;
    }
    const bool fit0 = __reduce_add_sync(0xffffffffu, n3[0]) <= p.ctas, fit1 = __reduce_add_sync(0xffffffffu, n3[1]) <= p.ctas;
    n = fit0 ? n3[0] : fit1 ? n3[1] : n3[2];
    int end = n;
#pragma unroll
    for (int o = 1; o < 32; o *= 2)
        if (o < B) { const int v = __shfl_up_sync(0xffffffffu, end, o); if (lane >= o) end += v; }
    base = end - n;
    return fit0 ? p.piece[0] : fit1 ? p.piece[1] : p.piece[2];
}
// CTAs a row block's keys are dealt to in the tile kernels: enough to fill the SMs (`per_sm` CTAs each), pieces of
// four chunks at least.  level_mask < 0: every level (for the workspace size).  The host does not know how many tokens a level has:
// a subset with level 3 or a deeper one is taken for all tokens, any other for the anchors of a [DOC]/[SEC]/[SENT]/token document and
// put at a sixteenth of them (documents have a thirtieth; more pieces than needed cost a merge of mostly empty partial
// results).  Where the words are on level 2, a subset with them is split too little, at worst not at all, as every subset was
// before there were pieces: 1 x 4096 tokens, 64 decoder rows, forward 155 us and backward 137, with bit 3 set as well (a caller may: no
// token has it) 31 and 61; 4 x 8192, 256 rows 310 and 597, so 191 and 516.
static int tile_splits(int B, int T, int Tq, int H, int level_mask, int per_sm) {
    if (B <= 0 || Tq <= 0) return 1;
    const long long mean = (T + B - 1) / B, keys = (level_mask < 0 || (level_mask >> 3)) ? mean : mean / 16;
    const long long ctas = (long long)B * ((Tq + 128LL * B - 1) / (128LL * B)) * H;
    return (int)max(1LL, min((keys + 511) / 512, ((long long)PLAN_SMS * per_sm + ctas - 1) / ctas));
}

// tc: bf16 on the tensor-core kernels (128-row blocks)
static CrossLayout cross_layout(int B, int T, int Tq, int H, int D, bool tc, int bwd) {
    CrossLayout L{};
    L.xr = tc ? 128 : 32;
    L.nbq = Tq / L.xr + B + 1;
    L.nbk = T / L.xr + B + 1;
    const size_t n = (size_t)Tq + T;
    size_t o = 0;
    L.blocks = o; o += al256c(sizeof(int) * 5 * (size_t)(L.nbq + L.nbk));       // blocks of the decoder rows, then of the chosen tokens
    L.tokx = o; o += al256c(sizeof(int) * max(n, (size_t)1));
    L.rngx = o; o += al256c(sizeof(int) * 2 * max(n, (size_t)1));
    L.queue = o; o += al256c(sizeof(int) * (size_t)(L.nbq + L.nbk));
    L.sel = o; o += al256c(sizeof(int) * (size_t)(B + 1));
    L.used = o; o += 256;
    L.delta = o; if (bwd) o += al256c(sizeof(float) * (size_t)H * max(Tq, 1));
    // partial results: rows of [H, D] and, in the forward, their LSE
    const size_t rows = !bwd && cross_decode(B, Tq) ? DecodePieces(B, T, Tq, H, D).part(Tq) : (size_t)tile_splits(B, T, Tq, H, -1, bwd ? 8 : 2) * Tq;
    L.part = o; o += al256c(sizeof(float) * rows * H * D);
    L.part_lse = o; if (!bwd) o += al256c(sizeof(float) * rows * H);
    L.total = o + 256;
    return L;
}

__device__ __forceinline__ int chosen_level(int lv, int level_mask) { return (lv >= 0 && lv < 31 && ((level_mask >> lv) & 1)) ? 1 : 0; }
__device__ __forceinline__ int chosen(const int8_t *level, int i, int level_mask) { return chosen_level(level[i], level_mask); }

struct CrossIndexArgs {
    const int8_t *level;
    const int32_t *cu_k, *cu_q;
    int B, T, Tq, level_mask, xr, nbq, nbk;
    const int *sel;               // [B + 1] chosen tokens before each document and in all, or nullptr: counted by every CTA itself
    int *tokx, *rngx, *blocks, *queue, *used;      // used: slots of the chosen tokens' blocks from the first to the last one in use
};

// Which of 16 levels are chosen, one bit each.
__device__ __forceinline__ unsigned chosen_bits(const uint4 &x, int level_mask) {
    const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
    unsigned bits = 0;
#pragma unroll
    for (int j = 0; j < 16; ++j) bits |= (unsigned)chosen_level((int8_t)(xs[j >> 2] >> (8 * (j & 3))), level_mask) << j;
    return bits;
}
// This thread's share (t of 256) of the number of chosen tokens in [lo, hi).
__device__ __forceinline__ int count_chosen(const int8_t *level, int lo, int hi, int level_mask, int t) {
    int n = 0;
    const bool vec = ((uintptr_t)level & 15) == 0;
    const int u1 = vec ? hi / 16 : 0, body = min(hi, (lo + 15) / 16 * 16);      // whole units: [body / 16, u1)
    for (int u = body / 16 + t; u < u1; u += 256) n += __popc(chosen_bits(reinterpret_cast<const uint4 *>(level)[u], level_mask));
    const int rest = max(body, 16 * u1);
    for (int i = lo + t; i < body; i += 256) n += chosen(level, i, level_mask);
    for (int i = rest + t; i < hi; i += 256) n += chosen(level, i, level_mask);
    return n;
}

// Many tokens and documents (see cross_build): chosen tokens of each document, sel[b + 1], and their sums, sel[0] = 0.
__global__ void __launch_bounds__(256) k_cross_count(const int8_t *level, const int32_t *cu_k, int level_mask, int *sel) {
    pdl_wait();
    pdl_launch_dependents();
    __shared__ int s_n;
    const int b = blockIdx.x, t = threadIdx.x;
    if (t == 0) s_n = 0;
    __syncthreads();
    const int n = __reduce_add_sync(0xffffffffu, count_chosen(level, cu_k[b], cu_k[b + 1], level_mask, t));
    if ((t & 31) == 0) atomicAdd(&s_n, n);
    __syncthreads();
    if (t == 0) sel[b + 1] = s_n;
}
__global__ void __launch_bounds__(1024) k_cross_scan(int *sel, int B) {
    pdl_wait();
    pdl_launch_dependents();
    __shared__ int s_w[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int run = 0;
    if (t == 0) sel[0] = 0;
    for (int b0 = 0; b0 < B; b0 += 1024) {
        int v = b0 + t < B ? sel[b0 + t + 1] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int x = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += x; }
        if (lane == 31) s_w[w] = v;
        __syncthreads();
        int u = s_w[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int x = __shfl_up_sync(0xffffffffu, u, o); if (lane >= o) u += x; }
        const int before = w ? __shfl_sync(0xffffffffu, u, w - 1) : 0;
        if (b0 + t < B) sel[b0 + t + 1] = run + before + v;
        run += __shfl_sync(0xffffffffu, u, 31);
        __syncthreads();
    }
}

// Chunk y of document b: its part of the ordered list of chosen tokens (elements Tq + position, with their row
// ranges) and its share of the document's decoder rows and of the block records of both sides.  Where
// its part starts is counted over the levels of all tokens before it by the CTA itself while that costs less than the
// launches of a count and a scan kernel; beyond, over those of its document (see cross_build).
__global__ void __launch_bounds__(256) k_cross_index(const CrossIndexArgs a) {
    pdl_wait();
    pdl_launch_dependents();
    __shared__ int s_w[8], s_n[4];
    __shared__ int s_carry;
    const int b = blockIdx.x, y = blockIdx.y, t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int8_t *level = a.level;
    const int KO = a.Tq, xr = a.xr, mask = a.level_mask;
    const int k0 = a.cu_k[b], k1 = a.cu_k[b + 1], q0 = a.cu_q[b], q1 = a.cu_q[b + 1];
    const int cs = (k1 - k0 + XC - 1) / XC, c0 = min(k1, k0 + y * cs), c1 = min(k1, c0 + cs);
    if (t < 4) s_n[t] = 0;
    __syncthreads();
    if (a.sel != nullptr) {
        const int n = __reduce_add_sync(0xffffffffu, count_chosen(level, k0, c0, mask, t));
        if (lane == 0) atomicAdd(&s_n[1], n);
        if (t == 0) { s_n[0] = a.sel[b]; s_n[2] = a.sel[b + 1]; s_n[3] = a.sel[a.B]; atomicAdd(&s_n[1], a.sel[b]); }
    } else {   // chosen tokens below k0, c0, k1 and in all
        int n0 = 0, n1 = 0, n2 = 0, n3 = 0;
        const bool vec = ((uintptr_t)level & 15) == 0;
        const int units = vec ? a.T / 16 : 0;
        for (int u0 = t; u0 < units; u0 += 4 * 256) {
            uint4 x4[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) x4[k] = u0 + 256 * k < units ? reinterpret_cast<const uint4 *>(level)[u0 + 256 * k] : make_uint4(~0u, ~0u, ~0u, ~0u);
#pragma unroll 1
            for (int k = 0; k < 4; ++k) {
                const unsigned bits = chosen_bits(k == 0 ? x4[0] : k == 1 ? x4[1] : k == 2 ? x4[2] : x4[3], mask);
                const int i0 = 16 * (u0 + 256 * k);
                auto below = [&](int lim) { const int d = lim - i0; return d <= 0 ? 0 : __popc(d >= 16 ? bits : bits & ((1u << d) - 1u)); };
                n0 += below(k0); n1 += below(c0); n2 += below(k1); n3 += __popc(bits);
            }
        }
        for (int i = units * 16 + t; i < a.T; i += 256) {
            const int f = chosen(level, i, mask);
            n0 += f & (i < k0); n1 += f & (i < c0); n2 += f & (i < k1); n3 += f;
        }
        n0 = __reduce_add_sync(0xffffffffu, n0); n1 = __reduce_add_sync(0xffffffffu, n1);
        n2 = __reduce_add_sync(0xffffffffu, n2); n3 = __reduce_add_sync(0xffffffffu, n3);
        if (lane == 0) { atomicAdd(&s_n[0], n0); atomicAdd(&s_n[1], n1); atomicAdd(&s_n[2], n2); atomicAdd(&s_n[3], n3); }
    }
    __syncthreads();
    const int s0 = s_n[0], s1 = s_n[2], total = s_n[3];
    if (t == 0) s_carry = s_n[1];
    __syncthreads();
    for (int base = c0; base < c1; base += 256) {
        const int i = base + t;
        const int f = (i < c1) ? chosen(level, i, mask) : 0;
        const unsigned m = __ballot_sync(0xffffffffu, f);
        if (lane == 0) s_w[w] = __popc(m);
        __syncthreads();
        int before = s_carry;
        for (int j = 0; j < w; ++j) before += s_w[j];
        if (f) {
            const int e = KO + before + __popc(m & ((1u << lane) - 1u));
            a.tokx[e] = i;
            a.rngx[2 * e] = q0;
            a.rngx[2 * e + 1] = q1;
        }
        __syncthreads();
        if (t == 0) { int tot = 0; for (int j = 0; j < 8; ++j) tot += s_w[j]; s_carry += tot; }
        __syncthreads();
    }
    // decoder rows and block records: spread over the document's chunks
    const int nt = XC * 256, gt = y * 256 + t;
    for (int r = q0 + gt; r < q1; r += nt) { a.tokx[r] = r; a.rngx[2 * r] = KO + s0; a.rngx[2 * r + 1] = KO + s1; }
    const int live = (s1 > s0 && q1 > q0) ? 0 : HDT_BLK_EMPTY;
    const bool last = b == a.B - 1;
    auto put = [&](int slot, int next, int x0, int x1, int off, int ka, int kb) {      // slots [slot, next): this document's
        for (int j = gt; j < next - slot; j += nt) {
            int *rec = a.blocks + 5 * (size_t)(slot + j);
            const int r0 = min(x1, x0 + j * xr);
            rec[0] = off + r0; rec[1] = off + min(x1, r0 + xr); rec[2] = ka; rec[3] = kb; rec[4] = live;
        }
    };
    put(q0 / xr + b, last ? a.nbq : q1 / xr + b + 1, q0, q1, 0, KO + s0, KO + s1);
    put(a.nbq + s0 / xr + b, a.nbq + (last ? a.nbk : s1 / xr + b + 1), s0, s1, KO, q0, q1);
    // tiles of the gathering kernels reach past the elements in use: element 0 is a valid row of every tensor
    const int all = a.B * nt, ga = b * nt + gt;
    if (ga == 0) *a.used = total / xr + a.B;
    for (int e = KO + total + ga; e < KO + a.T; e += all) a.tokx[e] = 0;
    for (int i = ga; i < a.nbq + a.nbk; i += all) a.queue[i] = i;
}

// Zero dK, dV rows of the encoder tokens that no decoder row attends to.  n16: 16-byte pieces of a token's row.  A warp looks `per` tokens (up to 32)
// over at a time, a lane each, then writes row after row.  CTAs of 128 threads have few enough registers to run beside those of
// the tile kernel at head_dim 64 (which leaves 4096 an SM; at 128 it leaves none); see hdt_cross_attn_bwd.
__global__ void __launch_bounds__(128) k_cross_zero(const int8_t *__restrict__ level, const int32_t *__restrict__ cu_k, const int32_t *__restrict__ cu_q, int B,
                                                    int T, int level_mask, int per, int n16, uint4 *dk, uint4 *dv) {
    const int lane = threadIdx.x & 31, warps = gridDim.x * 4;
    for (int i0 = (blockIdx.x * 4 + (threadIdx.x >> 5)) * per; i0 < T; i0 += warps * per) {
        const int i = i0 + lane;
        bool zero = lane < per && i < T;
        if (zero && chosen(level, i, level_mask)) {
            int lo = 0, hi = B;          // its document: the last b with cu_k[b] <= i
            while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (cu_k[mid] <= i) lo = mid; else hi = mid; }
            zero = cu_q[lo + 1] <= cu_q[lo];
        }
        for (unsigned m = __ballot_sync(0xffffffffu, zero); m != 0u; m &= m - 1u) {
            const size_t row = (size_t)(i0 + __ffs(m) - 1) * n16;
            for (int j = lane; j < n16; j += 32) {
                dk[row + j] = make_uint4(0, 0, 0, 0);
                dv[row + j] = make_uint4(0, 0, 0, 0);
            }
        }
    }
}

// ---- decoding ------------------------------------------------------------------------------------
// CTA (x, y): a piece of a document's tokens (see DecodePieces) for its decoder rows in turn, heads y * HC ...  The CTAs behind those
// of the pieces take the documents of more than DEC_ROWS rows, DEC_ROWS of all rows and an even share of their document's
// tokens each.  (All along x, where a grid has no limit that
// matters; a document's CTAs follow one another, since some that lie a multiple of eight apart share a part of the
// chip: 8 rows on one of 8 documents of 2048 tokens 28 us, so 19.)
// Thread (slot, head, lane): D / 8 lanes per (key, head), the heads of a token next to one another, so that a
// CTA reads whole token rows.  The bound is reading K and V once (4 x 8192 tokens, 12 x 64: 101 MB, 15 us at the
// copy rate; 20 us as one wave of CTAs): four keys a thread in flight; the tile kernel took 352 us here, one CTA per
// document and head walking 64 chunks with one row of 128 in use.
struct DecodeArgs {
    const int8_t *level;
    const int32_t *cu_k, *cu_q;
    int B, level_mask, H, HC, KS, Tq;
    DecodePieces p;
    const void *q, *k, *v;
    float scale_log2;
    void *o;
    float *lse, *part_o, *part_lse;       // rows of partial results: [rows, most], then [splits, Tq]
};
// The last i of [0, n) with le(i); le holds for 0 and for no i behind one for which it does not.  By a whole warp.
template <class F>
__device__ __forceinline__ int warp_last(int n, F le) {
    const int lane = threadIdx.x & 31;
    int lo = 0;
    while (n > 1) {
        const int step = (n + 31) / 32, i = lane * step;
        const int k = max(0, __popc(__ballot_sync(0xffffffffu, i < n && le(lo + i))) - 1) * step;
        lo += k;
        n = min(step, n - k);
    }
    return lo;
}

// What a CTA of the decode kernel does: tokens [c0, c1), rows [row0, row1); row r leaves its partial result at part + r * step (step
// 0: its result, since these are all the tokens).
struct DecodeJob {
    int c0, c1, row0, row1;
    unsigned part, step;
};
// The same for more than DEC_DOCS documents, and for documents of more than DEC_ROWS rows.  By a whole warp.
__device__ __forceinline__ void decode_job(const DecodeArgs &a, int x, DecodeJob *out) {
    const int lane = threadIdx.x & 31;
    DecodeJob w{};
    int b = 0, j, n;
    if (x < a.p.pieces) {                            // document b's pieces from number cu[b] / piece + b on: some numbers are no piece's
        const int piece = a.p.piece[0];
        b = warp_last(a.B, [&](int i) { return quotient(a.cu_k[i], piece) + i <= x; });
        const int k0 = a.cu_k[b], q0 = a.cu_q[b], q1 = a.cu_q[b + 1], base = quotient(k0, piece);
        n = doc_pieces(a.cu_k[b + 1] - k0, piece);
        j = x - (base + b);
        w.row0 = q0;
        w.row1 = j >= 0 && j < n && q1 - q0 <= DEC_ROWS ? q1 : q0;
        if (n > 1) { w.step = a.p.most; w.part = base + j - q0 * w.step; }
    } else {                                         // DEC_ROWS of all rows hold those of two documents of more at most
        const int groups = (a.Tq + DEC_ROWS - 1) / DEC_ROWS, y = (x - a.p.pieces) / a.p.splits, second = y >= groups, group = y - second * groups, row = DEC_ROWS * group + lane;
        j = (x - a.p.pieces) % a.p.splits;
        n = a.p.splits;
        int hi = a.B;                                // its document: the last one that starts at or before the row
        while (hi - b > 1) { const int mid = (b + hi) >> 1; if (a.cu_q[mid] <= row) b = mid; else hi = mid; }
        const int q0 = a.cu_q[b], q1 = a.cu_q[b + 1];
        unsigned m = __ballot_sync(0xffffffffu, lane < DEC_ROWS && q1 - q0 > DEC_ROWS && row >= q0 && row < min(a.Tq, q1)), mine = 0;
        int f = 0, d = 0;
        for (int i = 0; i <= second; ++i) {
            f = m ? __ffs(m) - 1 : 0;
            d = __shfl_sync(0xffffffffu, b, f);
            mine = m & __ballot_sync(0xffffffffu, b == d);
            m &= ~mine;
        }
        b = d;
        w.row0 = DEC_ROWS * group + f;
        w.row1 = w.row0 + __popc(mine);
        if (n > 1) { w.step = 1; w.part = a.p.most * a.p.rows + j * a.Tq; }
    }
    const int k0 = a.cu_k[b], k1 = a.cu_k[b + 1], per = quotient(k1 - k0 + n - 1, n);
    w.c0 = min(k1, k0 + j * per);
    w.c1 = min(k1, w.c0 + per);
    if (lane == 0) *out = w;
    __syncwarp();
}

template <int D, bool BF16>
__global__ void __launch_bounds__(512, 2) k_cross_decode(const DecodeArgs a) {
    pdl_wait();
    pdl_launch_dependents();
    constexpr int LPK = D / 8, C = 4;
    using W = Raw<BF16, LPK>;
    extern __shared__ float s_red[];                 // [KS][HC][D + 2]
    __shared__ int s_list[DEC_LIST];
    __shared__ int s_n;
    __shared__ DecodeJob s_job;
    const int t = threadIdx.x, lane = t & 31, g = t % LPK, src = lane - g;
    const unsigned mask = ((1u << LPK) - 1u) << src;
    const int pair = t / LPK, hl = pair % a.HC, ks = pair / a.HC, h = blockIdx.y * a.HC + hl;
    const bool on = ks < a.KS && h < a.H;
    auto list = [&](int p0, int p1) {                // by warp 0: the chosen tokens of [p0, p1), in order
        int n = 0;
        for (int i0 = p0; i0 < p1; i0 += 128) {      // (four loads in flight: nothing of K and V is requested before the list is there)
            bool f[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) f[k] = i0 + 32 * k + lane < p1 && chosen(a.level, i0 + 32 * k + lane, a.level_mask);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const unsigned m = __ballot_sync(0xffffffffu, f[k]);
                if (f[k]) s_list[n + __popc(m & ((1u << lane) - 1u))] = i0 + 32 * k + lane;
                n += __popc(m);
            }
        }
        if (lane == 0) s_n = n;
    };
    if (t < 32) {                                    // what to do, by one warp: the others' registers are the keys'
        const int x = blockIdx.x;
        if (x < a.p.pieces && a.B <= DEC_DOCS) {     // one round of loads, the documents' pieces one behind the other
            const int i = min(lane, a.B - 1), k0 = a.cu_k[i], k1 = a.cu_k[i + 1], q0 = a.cu_q[i], q1 = a.cu_q[i + 1];
            int n, base;
            const int piece = choose_piece(a.p, a.B, k1 - k0, n, base), j = x - base;
            if (lane == 0) s_job.row0 = s_job.row1 = 0;      // (a number that is no piece's)
            __syncwarp();
            if (j >= 0 && j < n) {                   // (one lane)
                const int c0 = min(k1, k0 + j * piece);
                s_job = DecodeJob{c0, min(k1, c0 + piece), q0, q1 - q0 <= DEC_ROWS ? q1 : q0, n > 1 ? x - q0 * (unsigned)a.p.most : 0u, n > 1 ? (unsigned)a.p.most : 0u};
            }
            __syncwarp();
        } else decode_job(a, x, &s_job);
        if (s_job.row1 > s_job.row0) list(s_job.c0, min(s_job.c1, s_job.c0 + DEC_LIST));
    }
    __syncthreads();
    const int c0 = s_job.c0, c1 = s_job.c1, row0 = s_job.row0, row1 = s_job.row1;
    for (int row = row0; row < row1; ++row) {
        RowSoftmax S;
        S.clear();
        W q;
        if (on) q.load(a.q, (unsigned)row * a.H + h, g);
        for (int p0 = c0; p0 < c1; p0 += DEC_LIST) {
            if (c1 - c0 > DEC_LIST && (p0 != c0 || row != row0)) {
                __syncthreads();
                if (t < 32) list(p0, min(c1, p0 + DEC_LIST));
                __syncthreads();
            }
            const int n = s_n;
            if (!on) continue;
            for (int i0 = ks * C; i0 < n; i0 += a.KS * C) {
                W x[C], y[C];
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const unsigned r = (unsigned)s_list[min(i0 + c, n - 1)] * a.H + h;      // (past the end: the last key, weight 0)
                    x[c].load(a.k, r, g);
                    y[c].load(a.v, r, g);
                }
                float sc[C];
                dots<C>(q, x, sc);
                const float s = reduce_scatter<C, LPK>(sc, g, mask) * a.scale_log2;
                const float p = S.add<C>(i0 + (g & (C - 1)) < n ? s : -INFINITY, mask);
                axpys<C>(S.acc, p, y, mask, src);
            }
        }
        // the slots of a head: one after the other through shared memory
        if (on) {
#pragma unroll
            for (int o = 1; o < C; o *= 2) S.l += __shfl_xor_sync(mask, S.l, o);
            float *d = s_red + (size_t)(ks * a.HC + hl) * (D + 2);
            const float lse = S.finish();
#pragma unroll
            for (int u = 0; u < 4; ++u) unpack2(S.acc[u], d[8 * g + 2 * u], d[8 * g + 2 * u + 1]);
            if (g == 0) d[D] = lse;
        }
        __syncthreads();
        if (on && ks == 0) {
            RowSoftmax R;
            R.clear();
            for (int i = 0; i < a.KS; ++i) {
                const float *d = s_red + (size_t)(i * a.HC + hl) * (D + 2);
                f2 x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) x[u] = pack2(d[8 * g + 2 * u], d[8 * g + 2 * u + 1]);
                R.merge(d[D] * 1.4426950408889634f, d[D] > -INFINITY ? 1.f : 0.f, x);
            }
            const float lse = R.finish();
            if (s_job.step == 0) {
                W::store(a.o, (unsigned)row * a.H + h, g, R.acc);
                if (g == 0) a.lse[(size_t)h * a.Tq + row] = lse;
            } else {
                const size_t r = (size_t)(s_job.part + row * s_job.step) * a.H + h;
                W::store_f32(a.part_o, r, g, R.acc);
                if (g == 0) a.part_lse[r] = lse;
            }
        }
        __syncthreads();
    }
}

// Where the partial results of decoder rows are, if not at [splits, Tq]: cu_k == nullptr says that they are.
struct DecodeParts {
    const int32_t *cu_k, *cu_q;
    int B;
    DecodePieces p;
};
// Merge of partial results over `splits`, a CTA per (row, head) or for some heads of a row.  Forward (lse given): log-sum-exp merge of
// normalised rows; backward: sum.  Groups of D / 8 lanes take every G-th partial result, then meet: inside a warp by
// shuffles, the warps through shared memory (all groups one after the other there: 0.7 us more).  Bound by the round trips to
// L2: 256 threads where a row may have many partial results (decoding, 4 x 8192 tokens: 23.5 us a call with 128, 22.9 with 256).
template <int D, bool BF16, bool PACK>
__global__ void __launch_bounds__(256) k_cross_combine(int splits, int Tq, int H, const float *part, const float *part_lse, void *out, float *lse, const DecodeParts dp) {
    constexpr int LPK = D / 8;
    const int G = blockDim.x / LPK;
    using W = Raw<BF16, LPK>;
    __shared__ float s_red[8][D + 2];
    const int row = blockIdx.x, g = threadIdx.x % LPK, i = threadIdx.x / LPK, w = threadIdx.x >> 5;
    size_t first = row, step = Tq;
    if (dp.cu_k != nullptr) {         // (before the wait: the kernel in front writes neither array, and began behind what did)
        int r, rows, n, base;
        if (dp.B <= DEC_DOCS) {
            const int lane = threadIdx.x & 31, x = min(lane, dp.B - 1), q0 = dp.cu_q[x];
            choose_piece(dp.p, dp.B, dp.cu_k[x + 1] - dp.cu_k[x], n, base);
            const int b = max(0, __popc(__ballot_sync(0xffffffffu, lane < dp.B && q0 <= row)) - 1);
            r = row - __shfl_sync(0xffffffffu, q0, b);
            rows = __shfl_sync(0xffffffffu, dp.cu_q[x + 1] - q0, b);
            n = __shfl_sync(0xffffffffu, n, b);
            base = __shfl_sync(0xffffffffu, base, b);
        } else {
            const int b = warp_last(dp.B, [&](int x) { return dp.cu_q[x] <= row; }), k0 = dp.cu_k[b];
            r = row - dp.cu_q[b];
            rows = dp.cu_q[b + 1] - dp.cu_q[b];
            n = doc_pieces(dp.cu_k[b + 1] - k0, dp.p.piece[0]);
            base = quotient(k0, dp.p.piece[0]);
        }
        if (r < 0) splits = 1;                       // (no document's row)
        else if (rows <= DEC_ROWS) {
            splits = n;
            first = (size_t)r * dp.p.most + base;
            step = 1;
        } else first += (size_t)dp.p.most * dp.p.rows;
    }
    pdl_wait();
    pdl_launch_dependents();
    if (dp.cu_k != nullptr && splits == 1) return;      // written by the one CTA that walked the row
    // (PACK, several heads to a CTA: a warp for each where there are few partial results)
    const bool alone = PACK && splits <= 4 * (32 / LPK);
    const int s0 = alone ? (threadIdx.x & 31) / LPK : i, sG = alone ? 32 / LPK : G, hw = alone ? (int)blockDim.x / 32 : 1;
    for (int h = blockIdx.y + (alone ? w * gridDim.y : 0); h < H; h += gridDim.y * hw) {
        if (!alone && h != (int)blockIdx.y) __syncthreads();
        RowSoftmax R;
        R.clear();
        auto add = [&](float m, float l, const f2 (&x)[4]) {
            if (part_lse != nullptr) R.merge(m, l, x);
            else
#pragma unroll
                for (int u = 0; u < 4; ++u) R.acc[u] = add2(R.acc[u], x[u]);
        };
#pragma unroll 4
        for (int s = s0; s < splits; s += sG) {
            const size_t r = (first + s * step) * H + h;
            f2 x[4];
            W::load_f32(part, r, g, x);
            const float L = part_lse != nullptr ? part_lse[r] : 0.f;
            add(L * 1.4426950408889634f, L > -INFINITY ? 1.f : 0.f, x);
        }
#pragma unroll
        for (int o = LPK; o < 32; o *= 2) {
            f2 x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = __shfl_xor_sync(0xffffffffu, R.acc[u], o);
            const float m = __shfl_xor_sync(0xffffffffu, R.m, o), l = __shfl_xor_sync(0xffffffffu, R.l, o);
            add(m, l, x);
        }
        if (!alone && (threadIdx.x & 31) < LPK) {
#pragma unroll
            for (int u = 0; u < 4; ++u) unpack2(R.acc[u], s_red[w][8 * g + 2 * u], s_red[w][8 * g + 2 * u + 1]);
            if (g == 0) { s_red[w][D] = R.m; s_red[w][D + 1] = R.l; }
        }
        if (!alone) __syncthreads();
        if (alone ? (threadIdx.x & 31) >= LPK : i != 0) continue;
        for (int j = 1; !alone && j < (int)blockDim.x / 32; ++j) {
            f2 x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = pack2(s_red[j][8 * g + 2 * u], s_red[j][8 * g + 2 * u + 1]);
            add(s_red[j][D], s_red[j][D + 1], x);
        }
        if (part_lse != nullptr) {
            const float L = R.finish();
            if (g == 0) lse[(size_t)h * Tq + row] = L;
        }
        W::store(out, (unsigned)row * H + h, g, R.acc);
    }
}

static int launch_combine(int splits, int Tq, int H, int D, int dtype, const float *part, const float *part_lse, void *out, float *lse, cudaStream_t st,
                          const DecodeParts &dp = DecodeParts{}) {
    // (decoding: rows of documents of one piece have nothing to merge, so where there are many, few CTAs a row)
    const bool decode = dp.cu_k != nullptr;
    const dim3 grid(Tq, decode ? max(1, min(H, 8 * PLAN_SMS / Tq)) : H);
    const int threads = decode ? 256 : 128;
    const bool pack = (int)grid.y < H;
    auto launch = [&](auto kernel) { return launch_dependent(kernel, true, grid, threads, 0, st, splits, Tq, H, part, part_lse, out, lse, dp); };
    cudaError_t e;
    if (D == 64) e = dtype == HDT_BF16 ? launch(pack ? k_cross_combine<64, true, true> : k_cross_combine<64, true, false>)
                                       : launch(pack ? k_cross_combine<64, false, true> : k_cross_combine<64, false, false>);
    else e = dtype == HDT_BF16 ? launch(pack ? k_cross_combine<128, true, true> : k_cross_combine<128, true, false>)
                               : launch(pack ? k_cross_combine<128, false, true> : k_cross_combine<128, false, false>);
    if (e != cudaSuccess) return set_error(HDT_ERR_CUDA, "launch of the combining kernel failed: %s", cudaGetErrorString(e));
    return HDT_OK;
}

template <int D, bool BF16>
static int launch_decode_t(DecodeArgs a, int B, cudaStream_t st) {
    const DecodeShape d(a.H, D);
    a.HC = d.HC;
    a.KS = d.KS;
    a.B = B;
    const int threads = d.threads;
    const unsigned grid = a.p.pieces + (a.Tq > DEC_ROWS ? 2u * ((a.Tq + DEC_ROWS - 1) / DEC_ROWS) * a.p.splits : 0u);
    const size_t smem = sizeof(float) * (size_t)a.KS * a.HC * (D + 2);
    HDT_CUDA_CHECK(launch_dependent(k_cross_decode<D, BF16>, true, dim3(grid, (a.H + a.HC - 1) / a.HC), threads, smem, st, a));
    return HDT_OK;
}

// Index of both sides.  Counting in every CTA reads a batch's levels 32 times per document, a time that grows with documents
// times tokens; the count and scan kernels read them once more, for two launches.  The line lies between the
// sizes timed (forward, 8 rows a document, 2 x 64): 4 x 8192 tokens (131 000) 23.2 us without them, 24.4 with; 8 x 8192
// (524 000) 29.9 and 24.9; 256 x 1024 892 and 43; 1024 x 128 1806 and 138.
static constexpr long long COUNT_LINE = 200000;
static int cross_build(const CrossLayout &L, char *ws, const int8_t *level, const int32_t *cu_k, const int32_t *cu_q, int B, int T, int Tq, int level_mask,
                       cudaStream_t st) {
    if (B <= 0) return HDT_OK;
    CrossIndexArgs a{};
    a.level = level; a.cu_k = cu_k; a.cu_q = cu_q; a.B = B; a.T = T; a.Tq = Tq; a.level_mask = level_mask;
    a.xr = L.xr; a.nbq = L.nbq; a.nbk = L.nbk;
    a.tokx = (int *)(ws + L.tokx); a.rngx = (int *)(ws + L.rngx); a.blocks = (int *)(ws + L.blocks); a.queue = (int *)(ws + L.queue);
    a.used = (int *)(ws + L.used);
    if ((long long)B * T > COUNT_LINE) {
        int *sel = (int *)(ws + L.sel);
        a.sel = sel;
        HDT_CUDA_CHECK(launch_dependent(k_cross_count, true, dim3(B), 256, 0, st, level, cu_k, level_mask, sel));
        HDT_CUDA_CHECK(launch_dependent(k_cross_scan, true, dim3(1), 1024, 0, st, sel, B));
    }
    HDT_CUDA_CHECK(launch_dependent(k_cross_index, true, dim3(B, XC), 256, 0, st, a));
    return HDT_OK;
}

static int cross_check(const void *level, const void *cu_k, const void *cu_q, int B, int T, int Tq, int H, int D,
                       int dtype, int level_mask, const void *ws, size_t ws_bytes, size_t need, const char *who) {
    if (B < 0 || T < 0 || Tq < 0 || H < 1) return set_error(HDT_ERR_INVALID_ARG, "%s: negative size or no head", who);
    if (D != 64 && D != 128) return set_error(HDT_ERR_UNSUPPORTED, "%s: head_dim %d not supported (64 or 128)", who, D);
    if (dtype != HDT_F32 && dtype != HDT_BF16) return set_error(HDT_ERR_UNSUPPORTED, "%s: unknown dtype %d", who, dtype);
    if (level_mask < 0) return set_error(HDT_ERR_INVALID_ARG, "%s: level_mask must be a set of level bits 0..30", who);
    if (!cu_k || !cu_q || (T > 0 && !level)) return set_error(HDT_ERR_INVALID_ARG, "%s: null structure pointer", who);
    if (!ws || ws_bytes < need) return set_error(HDT_ERR_WORKSPACE, "%s: workspace %zu < required %zu", who, ws_bytes, need);
    if ((uintptr_t)ws & 255) return set_error(HDT_ERR_INVALID_ARG, "%s: workspace must be 256-byte aligned", who);
    return HDT_OK;
}

}  // namespace hdt

using namespace hdt;

static bool cross_tc(int dtype) { return dtype == HDT_BF16 && !g_force_simt; }

extern "C" size_t hdt_cross_workspace_bytes(int32_t batch, int32_t total_tokens, int32_t total_q, int32_t heads,
                                            int32_t head_dim, int32_t dtype, int32_t bwd) {
    if (batch < 0 || total_tokens < 0 || total_q < 0 || heads < 1 || (head_dim != 64 && head_dim != 128)) return 0;
    // for either path: the SIMT kernels' (fp32, option "force_simt") smaller blocks have more records
    return max(cross_layout(batch, total_tokens, total_q, heads, head_dim, false, bwd).total,
               cross_layout(batch, total_tokens, total_q, heads, head_dim, true, bwd).total);
}

extern "C" int hdt_cross_attn_fwd(const int8_t *level, const int32_t *cu_seqlens_k, const int32_t *cu_seqlens_q,
                                  int32_t batch, int32_t total_tokens, int32_t total_q, int32_t level_mask,
                                  const void *q, const void *k, const void *v, void *o, float *lse, int32_t heads,
                                  int32_t head_dim, int32_t dtype, float softmax_scale, void *workspace,
                                  size_t workspace_bytes, void *stream) {
    const size_t need = hdt_cross_workspace_bytes(batch, total_tokens, total_q, heads, head_dim, dtype, 0);
    int rc = cross_check(level, cu_seqlens_k, cu_seqlens_q, batch, total_tokens, total_q, heads, head_dim, dtype,
                         level_mask, workspace, workspace_bytes, need, "hdt_cross_attn_fwd");
    if (rc) return rc;
    if (total_q == 0) return HDT_OK;
    if (!q || !o || !lse || (total_tokens > 0 && (!k || !v)))
        return set_error(HDT_ERR_INVALID_ARG, "hdt_cross_attn_fwd: null tensor pointer");
    if (batch == 0) return HDT_OK;
    const bool tc = cross_tc(dtype);
    const CrossLayout L = cross_layout(batch, total_tokens, total_q, heads, head_dim, tc, 0);
    cudaStream_t st = (cudaStream_t)stream;
    char *ws = (char *)workspace;
    const float scale = softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)head_dim);
    float *part = (float *)(ws + L.part), *part_lse = (float *)(ws + L.part_lse);
    if (cross_decode(batch, total_q) && !g_force_simt) {
        DecodeArgs a{};
        a.level = level; a.cu_k = cu_seqlens_k; a.cu_q = cu_seqlens_q; a.level_mask = level_mask; a.H = heads; a.Tq = total_q;
        const DecodePieces p(batch, total_tokens, total_q, heads, head_dim);
        a.p = p;
        a.q = q; a.k = k; a.v = v; a.scale_log2 = scale * 1.4426950408889634f;
        a.o = o; a.lse = lse; a.part_o = part; a.part_lse = part_lse;
        if (head_dim == 64) rc = dtype == HDT_BF16 ? launch_decode_t<64, true>(a, batch, st) : launch_decode_t<64, false>(a, batch, st);
        else rc = dtype == HDT_BF16 ? launch_decode_t<128, true>(a, batch, st) : launch_decode_t<128, false>(a, batch, st);
        if (rc || (!p.several && (p.splits == 1 || total_q <= DEC_ROWS))) return rc;      // no document of several pieces
        return launch_combine(p.splits, total_q, heads, head_dim, dtype, part, part_lse, o, lse, st,
                              DecodeParts{cu_seqlens_k, cu_seqlens_q, batch, p});
    }
    rc = cross_build(L, ws, level, cu_seqlens_k, cu_seqlens_q, batch, total_tokens, total_q, level_mask, st);
    if (rc) return rc;
    FwdStageArgs a{};
    a.n = total_q + total_tokens; a.nb = L.nbq; a.H = heads; a.T = total_q;
    a.tok = (const int *)(ws + L.tokx);
    a.tok_rows = a.tok;
    a.rng = (const int *)(ws + L.rngx); a.blocks = (const int *)(ws + L.blocks);
    a.queue = (const int *)(ws + L.queue); a.queue_split = a.queue;
    a.q = q; a.k = k; a.v = v; a.o = o; a.lse = lse;
    a.scale_log2 = scale * 1.4426950408889634f;
    a.status = device_status_ptr();
    a.block_rows = L.xr; a.dirs = 7;
    if (!tc) return launch_fwd_simt(a, head_dim, dtype, st);
    a.splits = tile_splits(batch, total_tokens, total_q, heads, level_mask, head_dim == 64 ? 2 : 1);
    a.pdl = 1;
    if (a.splits == 1) {
        a.final_merge = 2;       // the kernel's epilogue writes the bf16 rows and the LSE of the decoder rows itself
        return launch_fwd_tc_upper(a, head_dim, st);
    }
    a.split_rows = total_q;
    a.own_o = part; a.own_lse = part_lse;
    rc = launch_fwd_tc_upper(a, head_dim, st);
    if (rc) return rc;
    return launch_combine(a.splits, total_q, heads, head_dim, dtype, part, part_lse, o, lse, st);
}

extern "C" int hdt_cross_attn_bwd(const int8_t *level, const int32_t *cu_seqlens_k, const int32_t *cu_seqlens_q,
                                  int32_t batch, int32_t total_tokens, int32_t total_q, int32_t level_mask,
                                  const void *q, const void *k, const void *v, const void *o, const float *lse,
                                  const void *d_o, void *dq, void *dk, void *dv, int32_t heads, int32_t head_dim,
                                  int32_t dtype, float softmax_scale, void *workspace, size_t workspace_bytes,
                                  void *stream) {
    const size_t need = hdt_cross_workspace_bytes(batch, total_tokens, total_q, heads, head_dim, dtype, 1);
    int rc = cross_check(level, cu_seqlens_k, cu_seqlens_q, batch, total_tokens, total_q, heads, head_dim, dtype,
                         level_mask, workspace, workspace_bytes, need, "hdt_cross_attn_bwd");
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t esz = dtype == HDT_BF16 ? 2 : 4;
    if (total_tokens > 0 && (!dk || !dv)) return set_error(HDT_ERR_INVALID_ARG, "hdt_cross_attn_bwd: null tensor pointer");
    if (total_q > 0 && (!q || !o || !lse || !d_o || !dq || (total_tokens > 0 && (!k || !v))))
        return set_error(HDT_ERR_INVALID_ARG, "hdt_cross_attn_bwd: null tensor pointer");
    // Encoder rows outside the subset (and of documents without decoder rows) get zero gradients: writes of
    // their own, beside the other kernels, from one small CTA an SM on the stream of the highest priority.  On another it starts
    // only when the last CTA of the tile kernel has (so a backward of 4 x 8192 tokens and 256 rows ended 8 us behind that
    // kernel); half as many CTAs, so that the tile kernel has more of HBM, cost 1 us more, a quarter as many 5.
    // At head_dim 128 an SM runs either kernel's CTA, and this grid is the better one too: 16 documents of 8192 tokens, 128 rows, 16 heads
    // 375 us, 404 with sixteen CTAs an SM, 375 on a stream of no priority; 4 x 8192 with 256 rows 162, 161, 182.
    Side *sd = nullptr;
    if (total_tokens > 0 && batch == 0) {
        HDT_CUDA_CHECK(cudaMemsetAsync(dk, 0, (size_t)total_tokens * heads * head_dim * esz, st));
        HDT_CUDA_CHECK(cudaMemsetAsync(dv, 0, (size_t)total_tokens * heads * head_dim * esz, st));
    } else if (total_tokens > 0) {
        cudaStream_t sz = st;
        if (total_q > 0 && !g_no_overlap) {
            rc = get_side(&sd);
            if (rc) return rc;
            HDT_CUDA_CHECK(cudaEventRecord(sd->fork, st));
            HDT_CUDA_CHECK(cudaStreamWaitEvent(sd->first, sd->fork, 0));
            sz = sd->first;
        }
        int n_sm = 0;
        if ((rc = sm_count(&n_sm))) return rc;
        // (few tokens: a share for every warp.  32 a warp left two warps to a backward of 300 tokens, 16 heads x 128, 16 rows: 17.0 -> 21.2 us)
        const int ctas = sd ? n_sm : 16 * n_sm, per = max(1, min(32, (total_tokens + 4 * ctas - 1) / (4 * ctas)));
        k_cross_zero<<<min((total_tokens + 4 * per - 1) / (4 * per), ctas), 128, 0, sz>>>(level, cu_seqlens_k, cu_seqlens_q, batch, total_tokens, level_mask, per,
                                                                        (int)(heads * head_dim * esz / 16), (uint4 *)dk, (uint4 *)dv);
        count_launch();
        HDT_CUDA_CHECK(cudaGetLastError());
        if (sd) HDT_CUDA_CHECK(cudaEventRecord(sd->join, sd->first));
    }
    if (total_q == 0 || batch == 0) return HDT_OK;
    auto attend = [&]() -> int {
        const bool tc = cross_tc(dtype);
        const CrossLayout L = cross_layout(batch, total_tokens, total_q, heads, head_dim, tc, 1);
        char *ws = (char *)workspace;
        int r = cross_build(L, ws, level, cu_seqlens_k, cu_seqlens_q, batch, total_tokens, total_q, level_mask, st);
        if (r) return r;
        const float scale = softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)head_dim);
        BwdStageArgs a{};
        a.n = total_q + total_tokens; a.H = heads; a.T = total_q;
        a.tok = (const int *)(ws + L.tokx); a.tok_rows = a.tok;
        a.rng = (const int *)(ws + L.rngx);
        a.queue = (const int *)(ws + L.queue); a.queue_split = a.queue;
        a.blocks = (const int *)(ws + L.blocks);
        a.q = q; a.k = k; a.v = v; a.d_o = d_o; a.o = o; a.lse = lse;
        a.scale = scale; a.scale_log2 = scale * 1.4426950408889634f;
        a.dq = dq; a.dk = dk; a.dv = dv;
        a.status = device_status_ptr();
        a.block_rows = L.xr; a.dirs = 7;
        if (!tc) {
            float *delta = (float *)(ws + L.delta);
            r = launch_delta(o, d_o, delta, total_q, heads, head_dim, dtype, st);
            if (r) return r;
            a.delta = delta;
            BwdStageArgs aq = a, ak = a;
            aq.nb = L.nbq; aq.phases = 1;                                            // decoder rows as queries: dQ
            ak.nb = L.nbk; ak.phases = 2; ak.blocks = a.blocks + 5 * (size_t)L.nbq;   // chosen tokens as keys: dK, dV
            r = launch_bwd_simt(aq, head_dim, dtype, st);
            return r ? r : launch_bwd_simt(ak, head_dim, dtype, st);
        }
        // One launch over the blocks of both sides: the decoder rows' leave dq, the chosen tokens' dk and dv, as
        // bf16 rows at the element's token (decoder rows: token = row).  dO . O comes from the rows as they are gathered.
        a.gather_end_q = total_q;                       // Q, dO have total_q rows
        a.gather_end_k = total_q + total_tokens;
        a.nb = L.nbq + L.nbk; a.phase_split = L.nbq;
        a.final_merge = 2;
        a.splits = tile_splits(batch, total_tokens, total_q, heads, level_mask, 8);
        a.split_rows = total_q;
        a.own_dq = (float *)(ws + L.part);
        a.pdl = 1;
        a.used_slots = (const int *)(ws + L.used);
        r = launch_bwd_tc_upper(a, head_dim, st);
        if (r || a.splits == 1) return r;
        return launch_combine(a.splits, total_q, heads, head_dim, dtype, a.own_dq, nullptr, dq, nullptr, st);
    };
    rc = attend();
    if (sd) HDT_CUDA_CHECK(cudaStreamWaitEvent(st, sd->join, 0));
    return rc;
}
