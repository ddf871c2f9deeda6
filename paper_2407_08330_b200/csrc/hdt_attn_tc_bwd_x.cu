// Warp-specialised looping backward for stage 0 in bf16 at D = 128: SELF, non-EMPTY blocks (both tiles of the pass are
// the block itself).
//
// One resident CTA per SM (its tiles take 224 KB of shared memory, its accumulators all of TMEM) walks the items
// blockIdx.x, + gridDim.x, ... of queue_split x heads.  Sixteen compute warps (thread: query row = TMEM lane tid % 128,
// quarter tid / 128 of the columns), and a warp each, one lane of it, for the tile loads, the MMAs and the stores; the
// roles meet at mbarriers.
//   MMA      S = Q K^T, dP = dO V^T
//   compute  P = exp2(S c - LSE), dS = P o (dP - delta) on the row's own range -> shared memory (bf16)
//   MMA      dV = P^T dO over S, dK = dS^T Q over dP, dQ = dS K
//   compute  each gradient as it is done: -> bf16 rows in shared memory -> TMA stores
// Every input tile is requested again as soon as its last MMA has read it: V behind dP, dO behind dV, Q behind dK, K
// behind dQ.  TMEM holds two pairs of 128-column regions, which items take in turns: S (then dV) and dP (then dK) of
// item i in pair i % 2, dQ of item i over the S region of the other pair, whose dV has left.  So dP of item
// i + 1 is computed before item i's dQ is read, and S behind it.
//
// What bounds it: HBM (16 documents of 512 to 16384 tokens, 16 heads: 630 us, 81 % of the measured copy rate on the 260 KB an
// item cannot do without; 75 % where nothing of the inputs is in L2 at the start; 4 x 8192 tokens, cold, 222 us for 1187 MB of DRAM traffic, 82 %, tensor
// pipe 21 %, issue slots 34 %).  The kernel before it did an item's phases one after the other with eight warps, no load
// or MMA beside another item's: 810 us.
#include <cuda_bf16.h>

#include "hdt_internal.cuh"
#include "hdt_sm100.cuh"
#include "hdt_tmap.cuh"

namespace hdt {
using namespace sm100;

namespace {
constexpr int SUB = 16384;
constexpr long long WAIT_CYCLES = 400000000LL;
constexpr int KID = 8;     // kernel id in the device status word
__device__ __forceinline__ uint32_t swz(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }
// Barrier `id` over `n` threads that also tells every thread whether ALL of them passed `pred`.
__device__ __forceinline__ bool group_all(bool pred, int id, int n) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.and.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)pred), "r"(id), "r"(n)
        : "memory");
    return r != 0;
}
constexpr int X_COMPUTE = 512, X_THREADS = X_COMPUTE + 96;      // sixteen compute warps, then the load, MMA and store warps
struct XItem { int valid, r0, r1, h; };
}  // namespace

// FD (fused delta): a.delta is not read; delta[row] = dO[row] . O[row] is computed here: the sixteen lanes that share a
// token row fetch 16 bytes each of its O and dO rows at the top of the item (past L1).
template <bool FD>
__global__ void __launch_bounds__(X_THREADS, 1) k_bwd_tc_x(const __grid_constant__ CUtensorMap tm_q,
                                                           const __grid_constant__ CUtensorMap tm_k,
                                                           const __grid_constant__ CUtensorMap tm_v,
                                                           const __grid_constant__ CUtensorMap tm_do,
                                                           const __grid_constant__ CUtensorMap tm_o,
                                                           const __grid_constant__ StoreMaps sm_out, const BwdStageArgs a) {
    constexpr int D = 128, NSUB = 2;
    constexpr uint32_t TM_COLS = 512;
    pdl_wait();                   // (a programmatic dependent: what it reads is complete from here on)
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *sQ = smem_raw, *sDO = sQ + 2 * SUB, *sK = sDO + 2 * SUB, *sV = sK + 2 * SUB;
    uint8_t *sP = sV + 2 * SUB, *sDS = sP + 2 * SUB;     // P, dS; later staging of dK, dQ
    uint8_t *sStg = sDS + 2 * SUB;                       // staging of dV
    uint64_t *bars = (uint64_t *)(sStg + 2 * SUB);
    uint64_t *bar_dov = bars, *bar_qk = bars + 1;                                // dO and V, Q and K have landed
    uint64_t *bar_a = bars + 2, *bar_p = bars + 3;                               // S and dP are there; P and dS are written
    uint64_t *bar_v = bars + 4, *bar_k = bars + 5, *bar_q = bars + 6;            // dV, dK, dQ are there
    uint64_t *bar_sv = bars + 7, *bar_sk = bars + 8, *bar_sq = bars + 9;         // ... are read and staged
    uint64_t *bar_free = bars + 10;                                              // the previous item's stores have read their tiles
    uint32_t *slot = (uint32_t *)(bars + 11);
    volatile int *abort_flag = (volatile int *)(slot + 1);
    int4 *ring = (int4 *)(bars + 12);     // [4] records of this CTA's items: valid, r0, r1, head
    float *s_delta = (float *)(ring + 4); // FD: dO . O of the item's 128 rows

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int H = a.H, G = gridDim.x, i0 = (int)blockIdx.x;
    const int n_items = a.n_fused * H;
    const float LOG2E = 1.4426950408889634f;

    if ((smem_u32(smem_raw) & 1023u) != 0u) {      // the swizzled tiles need 1024-byte alignment
        if (tid == 0) atomicCAS(a.status, 0, HDT_ERR_CUDA);
        return;
    }
    auto block_of = [&](int i) { return i < n_items ? a.queue_split[i / H] : -1; };
    auto fetch = [&](int i, int blk) {
        XItem x{0, 0, 0, 0};
        if (blk >= 0) {
            const int *rec = a.blocks + 5 * (size_t)blk;
            x.valid = 1; x.r0 = rec[0]; x.r1 = rec[1]; x.h = i % H;
        }
        return x;
    };
    if (tid == 0) {
        for (int i = 0; i < 11; ++i) mbar_init(bars + i, i == 3 || (i >= 7 && i <= 9) ? X_COMPUTE / 32 : 1);
        *abort_flag = (*a.status != 0);
        fence_mbar_init();
        for (int i = 0; i < 2; ++i) {
            const XItem d = fetch(i0 + i * G, block_of(i0 + i * G));
            ring[i] = make_int4(d.valid, d.r0, d.r1, d.h);
        }
    }
    if (warp == 1) tmem_alloc(slot, TM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_launch_dependents();      // (behind the TMEM allocation: a successor that becomes resident now takes none this CTA waits for)
    const uint32_t tmem = *slot;
    const bool dead = (*abort_flag != 0);
    bool ok = true;
    int fail_site = 0;
#define X_WAIT(bar, parity, site)                                                     \
    do {                                                                              \
        if (ok && !mbar_wait((bar), (uint32_t)(parity), abort_flag, WAIT_CYCLES)) {   \
            ok = false;                                                               \
            fail_site = (site);                                                       \
        }                                                                             \
    } while (0)

    if (dead || !ring[0].x) {
        // (an earlier failure, or nothing to do)
    } else if (warp == X_COMPUTE / 32) {
        // ================= load warp =================
        if (lane == 0) {
            auto load = [&](uint8_t *dst, const CUtensorMap *tm, const XItem &d, uint64_t *bar) {
#pragma unroll
                for (int s = 0; s < NSUB; ++s) tma_load_3d(dst + s * SUB, tm, 64 * s, d.h, d.r0, bar);
            };
            auto prefetch = [&](const CUtensorMap *tm, const XItem &d) {
#pragma unroll
                for (int s = 0; s < NSUB; ++s) tma_prefetch_3d(tm, 64 * s, d.h, d.r0);
            };
            const int4 q0 = ring[0], q1 = ring[1];
            XItem d1{q1.x, q1.y, q1.z, q1.w};
            int b2 = block_of(i0 + 2 * G);
            int n_dov = 1, n_qk = 1;          // tiles requested so far, pairs
            {
                const XItem d{q0.x, q0.y, q0.z, q0.w};
                mbar_expect_tx(bar_dov, 2u * NSUB * SUB);
                mbar_expect_tx(bar_qk, 2u * NSUB * SUB);
                load(sDO, &tm_do, d, bar_dov); load(sV, &tm_v, d, bar_dov);
                load(sQ, &tm_q, d, bar_qk); load(sK, &tm_k, d, bar_qk);
            }
            for (uint32_t ph = 0; d1.valid; ph ^= 1) {
                const XItem d2 = fetch(i0 + (n_dov + 1) * G, b2);
                b2 = block_of(i0 + (n_dov + 2) * G);
                // the next item's last tiles, and the rows that the compute warps read, start their way into L2 now
                prefetch(&tm_k, d1);
                prefetch(&tm_q, d1);
                if constexpr (FD) prefetch(&tm_o, d1);
                prefetch(&tm_do, d1);
                X_WAIT(bar_a, ph, 1);
                if (!ok) break;
                mbar_expect_tx(bar_dov, 2u * NSUB * SUB);
                load(sV, &tm_v, d1, bar_dov);
                ++n_dov;
                X_WAIT(bar_v, ph, 2);       // (the barrier's bytes are expected: dO is requested whether or not a wait has run out)
                load(sDO, &tm_do, d1, bar_dov);
                X_WAIT(bar_k, ph, 3);
                if (!ok) break;
                mbar_expect_tx(bar_qk, 2u * NSUB * SUB);
                load(sQ, &tm_q, d1, bar_qk);
                ++n_qk;
                X_WAIT(bar_q, ph, 4);
                load(sK, &tm_k, d1, bar_qk);
                if (!ok) break;
                d1 = d2;
            }
            if (*abort_flag) {        // a wait ran out: the tiles under way land before the CTA ends
                volatile int none = 0;
                (void)mbar_wait(bar_dov, (n_dov - 1) & 1, &none, WAIT_CYCLES);
                (void)mbar_wait(bar_qk, (n_qk - 1) & 1, &none, WAIT_CYCLES);
            }
        }
        __syncwarp();
    } else if (warp == X_COMPUTE / 32 + 1) {
        // ================= MMA warp =================
        if (lane == 0) {
            // base descriptors; an MMA adds (byte offset >> 4) to the low word.  K-major: sbo 1024; MN-major: lbo = SUB between 64-element groups
            const uint64_t dk_ = smem_desc(smem_u32(sQ), 0, 1024), dm_ = smem_desc(smem_u32(sQ), SUB, 1024);
            const uint32_t kl = (uint32_t)dk_, kh = (uint32_t)(dk_ >> 32), ml = (uint32_t)dm_, mh = (uint32_t)(dm_ >> 32);
            constexpr uint32_t S16 = SUB >> 4, Q_ = 0, DO_ = 2 * S16, K_ = 4 * S16, V_ = 6 * S16, P_ = 8 * S16, DS_ = 10 * S16;      // tiles in descriptor address units
            const uint32_t id_kv = idesc_bf16(D, true, true), id_q = idesc_bf16(D, false, true);
            auto scores = [&](uint32_t col, uint32_t A, uint32_t B, uint32_t id) {       // [128 x Nc] = A B^T over the head dimension
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    const uint32_t off = (kk / 4) * S16 + 2 * (kk % 4);
                    mma_ss_w(col, kl + A + off, kh, kl + B + off, kh, id, kk > 0);
                }
            };
            const int4 q0 = ring[0], q1 = ring[1];
            int n0 = (q0.z - q0.y + 15) & ~15;
            XItem d1{q1.x, q1.y, q1.z, q1.w};
            int b2 = block_of(i0 + 2 * G);
            X_WAIT(bar_dov, 0, 5);
            X_WAIT(bar_qk, 0, 6);
            if (ok) {
                tc_fence_after();
                scores(tmem + 128, DO_, V_, idesc_bf16(n0, false, false));
                scores(tmem, Q_, K_, idesc_bf16(n0, false, false));
                mma_commit(bar_a);
            }
            for (int it = 0; ok; ++it) {
                const uint32_t ph = it & 1, own = tmem + 256 * ph, other = tmem + 256 * (ph ^ 1);       // this item's pair of regions, the other one
                const int nk = n0 >> 4;
                const XItem d2 = fetch(i0 + (it + 2) * G, b2);
                b2 = block_of(i0 + (it + 3) * G);
                X_WAIT(bar_p, ph, 7);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)      // dV = P^T dO
                    if (kk < nk) mma_ss_w(own, ml + P_ + 128 * kk, mh, ml + DO_ + 128 * kk, mh, id_kv, kk > 0);
                mma_commit(bar_v);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)      // dK = dS^T Q
                    if (kk < nk) mma_ss_w(own + 128, ml + DS_ + 128 * kk, mh, ml + Q_ + 128 * kk, mh, id_kv, kk > 0);
                mma_commit(bar_k);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)      // dQ = dS K
                    if (kk < nk) mma_ss_w(other, kl + DS_ + (kk / 4) * S16 + 2 * (kk % 4), kh, ml + K_ + 128 * kk, mh, id_q, kk > 0);
                mma_commit(bar_q);
                if (!d1.valid) break;
                n0 = (d1.r1 - d1.r0 + 15) & ~15;
                const uint32_t id_s = idesc_bf16(n0, false, false);
                X_WAIT(bar_dov, ph ^ 1, 8);
                if (!ok) break;
                tc_fence_after();
                scores(other + 128, DO_, V_, id_s);      // (dK of the item before was read before this item's P was written)
                X_WAIT(bar_sq, ph, 9);                    // dQ has been read
                X_WAIT(bar_qk, ph ^ 1, 10);
                if (!ok) break;
                tc_fence_after();
                scores(other, Q_, K_, id_s);
                mma_commit(bar_a);
                d1 = d2;
            }
        }
        __syncwarp();
    } else if (warp == X_COMPUTE / 32 + 2) {
        // ================= store warp: rows [0, nrows) of a staged tile as at most two boxes of b rows, b the largest power
        // of two <= min(nrows, 64): [0, b) and [nrows - b, nrows); where the two overlap the same values are written
        // twice.  Lanes 0..3: (box, sub-tile) =================
        const int second = (lane >> 1) & 1, u = lane & 1;
        int b2 = lane == 0 ? block_of(i0 + 2 * G) : -1;
        for (int it = 0; ok; ++it) {
            const uint32_t ph = it & 1;
            if (lane == 0) {
                const XItem d2 = fetch(i0 + (it + 2) * G, b2);
                b2 = block_of(i0 + (it + 3) * G);
                ring[(it + 2) & 3] = make_int4(d2.valid, d2.r0, d2.r1, d2.h);
                mbar_arrive(bar_free);      // (all stores of the item before have read their tiles)
            }
            const int4 d = ring[it & 3];
            const int n = d.z - d.y, bx = max(__clz(n) - 25, 0), b = 64 >> bx;          // box of 64 >> bx rows: 64 for n >= 64
            const int off = second ? n - b : 0;
            const bool mine = lane < 4 && (!second || n > b);
            X_WAIT(bar_sv, ph, 11);
            if (ok && mine) tma_store_3d(&sm_out.m[2][bx], 64 * u, d.w, d.y + off, sStg + u * SUB + off * 128);
            X_WAIT(bar_sk, ph, 12);
            if (ok && mine) tma_store_3d(&sm_out.m[1][bx], 64 * u, d.w, d.y + off, sP + u * SUB + off * 128);
            X_WAIT(bar_sq, ph, 13);
            if (ok && mine) tma_store_3d(&sm_out.m[0][bx], 64 * u, d.w, d.y + off, sDS + u * SUB + off * 128);
            bulk_commit();
            bulk_wait_read();
            ok = __all_sync(0xffffffffu, ok);
            if (!ring[(it + 1) & 3].x) break;
        }
    } else if (warp < X_COMPUTE / 32) {
        // ================= compute warps =================
        const int rl = tid & 127, qt = tid >> 7, c0 = 32 * qt;
        const uint32_t lane_col = ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0;       // this thread's lane, its quarter of a region's columns
        auto arrive = [&](uint64_t *bar) {      // this warp's share of a barrier, behind what its lanes wrote
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar);
        };
        for (int it = 0;; ++it) {
            const uint32_t ph = it & 1;
            const uint32_t own = tmem + lane_col + 256 * ph, other = tmem + lane_col + 256 * (ph ^ 1);
            const int4 d = ring[it & 3];
            const int r0 = d.y, nrows = d.z - d.y, h = d.w;
            const int Nc = (nrows + 15) & ~15;
            uint4 xo[4], xg[4];      // FD: 16-byte chunk tid % 16 of rows tid / 16 + 32 k of O and dO
            if constexpr (FD) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int r = (tid >> 4) + 32 * k;
                    xo[k] = make_uint4(0u, 0u, 0u, 0u);
                    xg[k] = make_uint4(0u, 0u, 0u, 0u);
                    if (r < nrows) {
                        const size_t off = ((size_t)(r0 + r) * H + h) * D + (tid & 15) * 8;
                        xo[k] = ld_stream16(reinterpret_cast<const __nv_bfloat16 *>(a.o) + off);
                        xg[k] = ld_stream16(reinterpret_cast<const __nv_bfloat16 *>(a.d_o) + off);
                    }
                }
            }
            const int row = r0 + rl;
            const bool inq = rl < nrows;
            int2 rg = make_int2(0, 0);
            float lse2 = 0.f, dl = 0.f;
            if (inq) {
                rg = *reinterpret_cast<const int2 *>(a.rng + 2 * (size_t)row);
                lse2 = a.lse[(size_t)h * a.T + row] * LOG2E;
                if constexpr (!FD) dl = a.delta[(size_t)h * a.T + row];
            }
            if constexpr (FD) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t xs[4] = {xo[k].x, xo[k].y, xo[k].z, xo[k].w}, ys[4] = {xg[k].x, xg[k].y, xg[k].z, xg[k].w};
                    float acc = 0.f;
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        acc = fmaf(__uint_as_float(xs[w] << 16), __uint_as_float(ys[w] << 16), acc);
                        acc = fmaf(__uint_as_float(xs[w] & 0xffff0000u), __uint_as_float(ys[w] & 0xffff0000u), acc);
                    }
#pragma unroll
                    for (int m = 1; m < 16; m <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, m);
                    if ((tid & 15) == 0) s_delta[(tid >> 4) + 32 * k] = acc;
                }
            }
            X_WAIT(bar_free, ph, 14);
            if (!group_all(ok, 1, X_COMPUTE)) break;      // (a wait ran out: the compute warps leave together)
            if constexpr (FD) dl = s_delta[rl];
            const int jl = max(rg.x - r0, 0), jh = min(rg.y - r0, nrows);
            X_WAIT(bar_a, ph, 15);
            tc_fence_after();
            // ---- P and dS of this thread's 32 columns ----
            if (c0 < Nc) {                                 // same decision in the whole warp
                const uint32_t km = (inq && jh > jl) ? keep_mask<false>(c0, 32, jl, jh, 0, 0, false, false) : 0u;
                const uint32_t at = (uint32_t)(qt >> 1) * SUB;
                const int ch = (qt & 1) * 4;
                if (__any_sync(0xffffffffu, km != 0u)) {
                    uint32_t rs[32], rd[32];
                    tmem_ld32(own, rs);
                    tmem_ld32(own + 128, rd);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 4; ++c) {      // (eight columns at a time: what is finished leaves the registers)
                        uint32_t pp[4], pd[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int j = 8 * c + 2 * i;
                            float p0 = 0.f, p1 = 0.f, e0 = 0.f, e1 = 0.f;
                            if (km & (1u << j)) {
                                p0 = exp2f(fmaf(__uint_as_float(rs[j]), a.scale_log2, -lse2));
                                e0 = p0 * (__uint_as_float(rd[j]) - dl);
                            }
                            if (km & (2u << j)) {
                                p1 = exp2f(fmaf(__uint_as_float(rs[j + 1]), a.scale_log2, -lse2));
                                e1 = p1 * (__uint_as_float(rd[j + 1]) - dl);
                            }
                            pp[i] = pack_bf16(p0, p1);
                            pd[i] = pack_bf16(e0, e1);
                        }
                        const uint32_t o = at + swz(rl, ch + c);
                        *reinterpret_cast<uint4 *>(sP + o) = make_uint4(pp[0], pp[1], pp[2], pp[3]);
                        *reinterpret_cast<uint4 *>(sDS + o) = make_uint4(pd[0], pd[1], pd[2], pd[3]);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const uint32_t o = at + swz(rl, ch + c);
                        *reinterpret_cast<uint4 *>(sP + o) = make_uint4(0u, 0u, 0u, 0u);
                        *reinterpret_cast<uint4 *>(sDS + o) = make_uint4(0u, 0u, 0u, 0u);
                    }
                }
            }
            fence_proxy_async_smem();
            arrive(bar_p);
            const int up = (inq && a.part_dq != nullptr) ? a.up[row] : -1;
            // ---- drain: this thread's row, its quarter of the columns of each gradient ----
            auto drain = [&](uint32_t col, uint8_t *dst, float *parts, float sc) {
                float *part = up >= 0 ? parts + ((size_t)up * H + h) * D + c0 : nullptr;
                uint32_t r[32];
                tmem_ld32(col, r);
                tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    float x[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) x[i] = __uint_as_float(r[8 * c + i]) * sc;
                    if (part != nullptr) {
                        *reinterpret_cast<float4 *>(part + 8 * c) = make_float4(x[0], x[1], x[2], x[3]);
                        *reinterpret_cast<float4 *>(part + 8 * c + 4) = make_float4(x[4], x[5], x[6], x[7]);
                    }
                    *reinterpret_cast<uint4 *>(dst + (qt >> 1) * SUB + swz(rl, (qt & 1) * 4 + c)) =
                        make_uint4(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]), pack_bf16(x[4], x[5]), pack_bf16(x[6], x[7]));
                }
                fence_proxy_async_smem();
            };
            X_WAIT(bar_v, ph, 16);
            tc_fence_after();
            drain(own, sStg, a.part_dv, 1.f);
            arrive(bar_sv);
            X_WAIT(bar_k, ph, 17);
            tc_fence_after();
            drain(own + 128, sP, a.part_dk, a.scale);
            arrive(bar_sk);
            X_WAIT(bar_q, ph, 18);
            tc_fence_after();
            drain(other, sDS, a.part_dq, a.scale);
            arrive(bar_sq);
            if (!ring[(it + 1) & 3].x) break;
        }
    }
#undef X_WAIT
    if (!ok) {
        if (fail_site && a.status[1] == 0) a.status[1] = (KID << 8) | fail_site;
        atomicCAS(a.status, 0, HDT_ERR_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, TM_COLS);
}

int launch_bwd_tc_fused128(const BwdStageArgs &a, const CUtensorMap &tq, const CUtensorMap &tk, const CUtensorMap &tv,
                           const CUtensorMap &tdo, const StoreMaps &outs, cudaStream_t st) {
    constexpr int smem = 14 * SUB + 12 * 8 + 4 * 16 + 128 * 4;
    static DevOnce attr;
    int n_sm = 0;
    if (const int rc = sm_count(&n_sm)) return rc;
    if (!attr.done()) {
        HDT_CUDA_CHECK(cudaFuncSetAttribute(k_bwd_tc_x<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        HDT_CUDA_CHECK(cudaFuncSetAttribute(k_bwd_tc_x<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        attr.set();
    }
    const long long items = (long long)a.n_fused * a.H;
    if (items == 0) return HDT_OK;
    const bool fd = a.delta == nullptr;
    if (a.dirs != 7 || (fd && a.o == nullptr)) return set_error(HDT_ERR_INVALID_ARG, "launch_bwd_tc_fused128: needs the full rule, and o without delta");
    CUtensorMap to = tdo;         // O's tiles are only prefetched into L2
    if (fd) if (const int rc = make_tmap_bf16(&to, a.o, 128, a.H, a.T, 128)) return rc;
    HDT_CUDA_CHECK(launch_dependent(fd ? k_bwd_tc_x<true> : k_bwd_tc_x<false>, true, dim3((unsigned)(items < n_sm ? items : n_sm)), X_THREADS, smem, st,
                                    tq, tk, tv, tdo, to, outs, a));
    return HDT_OK;
}

}  // namespace hdt
