// Max-over-query relevance in one pass over the features (the scorer of
// reading R22): the token x query-row cosines on the
// 5th-generation tensor cores, and, from the same shared-memory tiles, each
// token's norm and the per-frame channel sums that the frame statistics
// (r_t, delta_t; Section 3.2.1, Eq. 7) need.
//
//   a_{t,n} = max_{j < Lq} <u_{t,n}, q_j / ||q_j||> / ||u_{t,n}||
//
// Token tiles of 128 rows (M; fewer at the end of a video or of the CTA's
// range) x K steps of 64 channels: A = the features, K-major with 128-byte
// swizzle; B = the unit query rows of the tile's video as bf16 hi rows then lo
// rows (query_rows_kernel), N = 2 Lqp <= 256.  A feature stage holds G
// consecutive K steps, a query-row stage as many as it has room for (gb(Lqp):
// 1, 2 or 4, at most G), each loaded by one 3D TMA box ({64, 128, G} and {64,
// 2 Lqp, gb}, one tensor map per Lqp): a token row arrives as G * 128
// contiguous bytes per load, not 128, which keeps HBM reads efficient.  The
// features and the query rows have rings of their own; the query rows (read
// from L2 for every tile) take about kXBFlight bytes and the rest of shared
// memory keeps feature reads in flight.  fp32 accumulators in tensor
// memory, two buffers, so the epilogue of a tile overlaps the main loop of the
// next.  CTA c covers the tokens [c L1, (c+1) L1) of the flattened [V*T*N]
// index, exactly as the relevance pass does, and writes its channel sums of
// every frame f it touches into partial slot c + f, where the frame statistics
// expect them.
//   warp 0       TMA producer of the features (one thread)
//   warp 1       TMEM allocation and the MMA issuer (one thread)
//   warps 2-9    channel sums and token norms: 4 channel pairs per warp, a
//                lane per channel pair and class of the tile's rows mod 8
//                (two warps per SM sub-partition; every element is read from
//                shared memory once); the classes combined by shuffles; the
//                squares of a row's channels kept per lane over the tile's K
//                steps and combined at the end of the tile; the sums of the
//                frame open at the start of a tile and of the frame that
//                starts inside it (frames have >= 128 tokens, so at most one
//                starts inside a tile) accumulate in shared memory and are
//                written to the frame's slot when the frame ends or the
//                CTA's range does.  After each tile warps 2-5 also form
//                a_{t,n} for the rows of their tensor-memory lane quadrant:
//                tcgen05.ld -> max over the query rows of hi + lo -> / ||u||
//   warp 10      TMA producer of the query rows (one thread)
// Every mbarrier wait is bounded; on a timeout the kernel records a status
// bit, drains what it issued, frees tensor memory and exits.
// HBM bound up to Lq = 64 (256 frames of 27 x 27 x 3584: 0.231 ms at Lq = 16,
// 0.238 at 64), then by the query rows' L2 reads (0.298 at 128).  On 8 videos of
// 64 frames of 13 x 13 x 3584 and 8 to 119 rows one pass takes 0.175 ms where
// the relevance pass and one GEMM launch per video took 0.38; frame ends fall
// inside most tiles there.  The channel sums work on the rows of the tile's box
// (a CTA's last tile is a short one), one K step per loop iteration: with all
// 128 rows and four K steps unrolled 0.243, 0.265, 0.309 and 0.185 ms.  Measured
// and not taken: 16 channel-sum warps (0.196), more query-row bytes in flight
// (0.19).
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <type_traits>
#include <cstring>

#include "wz_internal.cuh"
#include "wz_ptx.cuh"

namespace wz {

namespace {

constexpr int kXM = 128, kXK = 64;
constexpr int kXABytes = kXM * kXK * 2;             // 16 KB
constexpr int kXMaxStages = 8;
constexpr int kXGroups = 4;                         // K steps per feature stage (at most)
constexpr int kXMinStages = 2;
constexpr int kXRowMaps = kXM / 32;                 // feature boxes: 32, 64, 96, 128 rows
constexpr int kXMaps = WZ_MAX_LQ_MAXSIM / 16;       // query-row boxes: Lqp = 16, 32, ..
constexpr int kXThreads = 11 * 32;
constexpr int kXMaxBStages = 8;                     // query-row stages (their own ring)
constexpr int kXBFlight = 64 * 1024;                // query-row bytes to keep in flight (L2 latency)
constexpr int kXAccCols = 256;
constexpr uint64_t kXTimeoutNs = 2000000000ull;
constexpr int kXReaders = 8;                        // channel-sum warps reading each stage

struct XShared {
    uint64_t full[kXMaxStages];    // feature ring
    uint64_t empty[kXMaxStages];
    uint64_t bfull[kXMaxBStages];  // query-row ring
    uint64_t bempty[kXMaxBStages];
    uint64_t tfull[2], tempty[2];
    uint64_t csync[2];
    uint64_t drain;
    uint32_t tmem_base;
    int abort;
    float npart[2][kXReaders][kXM];   // per channel-sum warp: squares of its channels, per row
};

struct XMaps {
    CUtensorMap a[kXRowMaps];   // boxes of 32 (k + 1) token rows
    CUtensorMap b[kXMaps];      // boxes of 2 Lqp rows, Lqp = 16 (k + 1)
};

struct XArgs {
    int stages, stage_stride;             // feature ring: stages and bytes per stage (G A tiles)
    int bstages, b_off, b_stride;         // query-row ring: stages, byte offset, bytes per stage
    int acc_off;                // byte offset of the two channel-sum buffers (2 x D floats)
    int shared_off;             // byte offset of XShared
};

// K steps of 2 Lqp query rows in a stage of `bytes`, at most G.
__host__ __device__ __forceinline__ int xgb(int Lqp, int bytes, int G) {
    int gb = G;
    while (gb > 1 && gb * 2 * Lqp * kXK * 2 > bytes) gb >>= 1;
    return gb;
}

__device__ __forceinline__ void xfail(const Ctx &c, volatile int *abort_flag, int code) {
    *abort_flag = 1;
    atomicOr(c.status, code);
}

// The token tiles of this CTA in order: at most 128 rows, none across a video.
// A tile's feature boxes have its rows rounded up to 32; the rows past them in
// shared memory are stale, and nothing reads the results of rows >= nr.
struct XTile {
    int64_t base, end, vend;   // first token; end of the CTA's range and of the video
    int nr, v;                 // rows, video
    int Lq, Lqp, qrow;         // the video's query rows: valid, padded to 16, first row of qhl

    __device__ __forceinline__ int rows() const { return (nr + 31) & ~31; }
    __device__ __forceinline__ void query(const Ctx &c) {
        const VideoPar vp = c.vpar[v];
        Lq = vp.Lq;
        Lqp = (Lq + 15) & ~15;
        qrow = qhl_row(vp.q_row0, v) - c.qhl_row0;
    }
    // the first tile; false when the CTA has no tokens
    __device__ __forceinline__ bool first(const Ctx &c) {
        const int64_t per = (int64_t)c.T * c.N, total = per * c.V;
        base = (int64_t)blockIdx.x * c.L1;
        end = min(total, base + c.L1);
        if (base >= end) return false;
        v = (int)(base / per);
        vend = (v + 1) * per;
        nr = (int)min((int64_t)kXM, min(end, vend) - base);
        query(c);
        return true;
    }
    __device__ __forceinline__ bool next(const Ctx &c) {
        base += nr;
        if (base >= end) return false;
        if (base >= vend) {
            ++v;
            vend += (int64_t)c.T * c.N;
            query(c);
        }
        nr = (int)min((int64_t)kXM, min(end, vend) - base);
        return true;
    }
};

// The channel sums of this warp's 8 channels of every K step (acc), to the
// partial slot of frame f, then acc cleared: lane group lane / 8 takes every
// fourth K step.
__device__ __forceinline__ void xflush(const Ctx &c, float *acc, int64_t f, int ch_lo, int lane) {
    float *dst = c.part + ((size_t)blockIdx.x + (size_t)f) * c.D;
    for (int k0 = (lane >> 3) * kXK; k0 < c.D; k0 += 4 * kXK) {
        const int ch = k0 + ch_lo + (lane & 7);
        if (wz_in_range(c.status, (int64_t)blockIdx.x + f < (int64_t)c.G1 + (int64_t)c.V * c.T)) dst[ch] = acc[ch];
        acc[ch] = 0.f;
    }
}

}  // namespace

template <int G>   // K steps per feature stage
__global__ void __launch_bounds__(kXThreads, 1) maxsim_pass_kernel(const __grid_constant__ XMaps maps, Ctx c, XArgs p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const size_t ring_off = (size_t)(ring - smem_raw);
    float *acc_buf = reinterpret_cast<float *>(ring + p.acc_off);
    XShared *S = reinterpret_cast<XShared *>(ring + p.shared_off);
    volatile int *abort_flag = &S->abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            ptx::mbar_init(&S->full[s], 1);
            ptx::mbar_init(&S->empty[s], 1 + kXReaders);
        }
        for (int s = 0; s < p.bstages; ++s) {
            ptx::mbar_init(&S->bfull[s], 1);
            ptx::mbar_init(&S->bempty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(&S->tfull[b], 1);
            ptx::mbar_init(&S->tempty[b], 4);
            ptx::mbar_init(&S->csync[b], kXReaders);
        }
        ptx::mbar_init(&S->drain, 1);
        S->abort = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async_smem();
    }
    if (warp == 1) {
        ptx::tmem_alloc(&S->tmem_base, 2 * kXAccCols);
        ptx::tmem_relinquish();
    }
    if (warp == 0 && lane == 0) {
        ptx::prefetch_tmap(&maps.a[kXRowMaps - 1]);
    }
    // channel sums start at zero (shared memory only: before the wait)
    for (int k = threadIdx.x; k < 2 * c.D; k += blockDim.x) acc_buf[k] = 0.f;
    pdl_wait();   // the query rows come from the previous grid
    pdl_trigger();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = S->tmem_base;
    XTile t;
    const bool any = t.first(c);   // vpar is the previous grid's
    const int KS = c.D / kXK;

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer: features ----------------
        const uint64_t pol_a = ptx::policy_evict_first();
        int stage = 0;
        uint32_t phase = 0;
        int issued_parity[kXMaxStages];
        for (int s = 0; s < kXMaxStages; ++s) issued_parity[s] = -1;
        for (bool on = any; on && !*abort_flag; on = t.next(c)) {
            const CUtensorMap *map = &maps.a[(t.rows() >> 5) - 1];
            const uint32_t stage_bytes = (uint32_t)(G * t.rows() * kXK * 2);
            bool ok = true;
            for (int ks = 0; ks < KS; ks += G) {
                if (!ptx::mbar_wait(&S->empty[stage], phase ^ 1u, kXTimeoutNs)) {
                    xfail(c, abort_flag, 16);
                    ok = false;
                    break;
                }
                uint8_t *st = ring + (size_t)stage * p.stage_stride;
                ptx::mbar_arrive_expect_tx(&S->full[stage], stage_bytes);
                ptx::tma_load_3d(st, map, &S->full[stage], 0, (int)t.base, ks, pol_a);
                issued_parity[stage] = (int)phase;
                if (++stage == p.stages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            if (!ok) break;
        }
        for (int s = 0; s < p.stages; ++s)
            if (issued_parity[s] >= 0) ptx::mbar_wait(&S->full[s], (uint32_t)issued_parity[s], kXTimeoutNs);
    } else if (warp == 10 && lane == 0) {
        // ---------------- TMA producer: query rows (from L2), K step by K step ----------------
        const uint64_t pol_b = ptx::policy_evict_last();
        int stage = 0;
        uint32_t phase = 0;
        int issued_parity[kXMaxBStages];
        for (int s = 0; s < kXMaxBStages; ++s) issued_parity[s] = -1;
        for (bool on = any; on && !*abort_flag; on = t.next(c)) {
            const int gb = xgb(t.Lqp, p.b_stride, G);
            const uint32_t stage_bytes = (uint32_t)gb * 2u * (uint32_t)t.Lqp * kXK * 2u;
            const CUtensorMap *map = &maps.b[(t.Lqp >> 4) - 1];
            bool ok = true;
            for (int ks = 0; ks < KS; ks += gb) {
                if (!ptx::mbar_wait(&S->bempty[stage], phase ^ 1u, kXTimeoutNs)) {
                    xfail(c, abort_flag, 16);
                    ok = false;
                    break;
                }
                ptx::mbar_arrive_expect_tx(&S->bfull[stage], stage_bytes);
                ptx::tma_load_3d(ring + p.b_off + (size_t)stage * p.b_stride, map, &S->bfull[stage], 0, t.qrow, ks,
                                 pol_b);
                issued_parity[stage] = (int)phase;
                if (++stage == p.bstages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            if (!ok) break;
        }
        for (int s = 0; s < p.bstages; ++s)
            if (issued_parity[s] >= 0) ptx::mbar_wait(&S->bfull[s], (uint32_t)issued_parity[s], kXTimeoutNs);
    } else if (warp == 1 && lane == 0) {
        // ---------------- MMA issuer ----------------
        const uint32_t ring32 = ptx::smem_u32(ring);
        const uint64_t a_base = ptx::smem_desc(ring32, 16, 1024, 2);              // 128-B swizzle
        const uint64_t b_base = ptx::smem_desc(ring32 + (uint32_t)p.b_off, 16, 1024, 2);
        const uint64_t stage_desc = (uint64_t)(p.stage_stride >> 4), bstage_desc = (uint64_t)(p.b_stride >> 4);
        int stage = 0, bstage = 0;
        uint32_t phase = 0, bphase = 0;
        int it = 0;
        for (bool on = any; on && !*abort_flag; on = t.next(c), ++it) {
            const int b = it & 1;
            const uint32_t use = (uint32_t)(it >> 1);
            if (!ptx::mbar_wait(&S->tempty[b], (use & 1u) ^ 1u, kXTimeoutNs)) {
                xfail(c, abort_flag, 16);
                break;
            }
            ptx::tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(b * kXAccCols);
            const uint32_t idesc = ptx::idesc_bf16(kXM, 2 * t.Lqp, false, false);   // both K-major
            const uint64_t b_sub = (uint64_t)((2 * t.Lqp * kXK * 2) >> 4);          // one K step of B
            const uint64_t a_sub = (uint64_t)((t.rows() * kXK * 2) >> 4);            // and of A
            const int gb1 = xgb(t.Lqp, p.b_stride, G) - 1;
            bool ok = true;
            for (int ks = 0; ks < KS && ok; ks += G) {
                if (!ptx::mbar_wait(&S->full[stage], phase, kXTimeoutNs)) {
                    xfail(c, abort_flag, 16);
                    ok = false;
                    break;
                }
                const uint64_t so = (uint64_t)stage * stage_desc;
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    if ((g & gb1) == 0) {
                        if (!ptx::mbar_wait(&S->bfull[bstage], bphase, kXTimeoutNs)) {
                            xfail(c, abort_flag, 16);
                            ok = false;
                            break;
                        }
                        ptx::tc_fence_after();
                    }
                    const uint64_t ao = so + (uint64_t)g * a_sub;
                    const uint64_t bo = (uint64_t)bstage * bstage_desc + (uint64_t)(g & gb1) * b_sub;
#pragma unroll
                    for (int k = 0; k < kXK / 16; ++k)   // K = 16 per MMA: 32 bytes along the swizzled row
                        ptx::mma_bf16(d, a_base + ao + (uint64_t)(2 * k), b_base + bo + (uint64_t)(2 * k), idesc,
                                      (ks | g | k) ? 1u : 0u);
                    if ((g & gb1) == gb1) {
                        ptx::mma_commit(&S->bempty[bstage]);
                        if (++bstage == p.bstages) {
                            bstage = 0;
                            bphase ^= 1u;
                        }
                    }
                }
                if (!ok) break;
                ptx::mma_commit(&S->empty[stage]);
                if (++stage == p.stages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            if (!ok) break;
            ptx::mma_commit(&S->tfull[b]);
        }
        ptx::mma_commit(&S->drain);
        ptx::mbar_wait(&S->drain, 0, kXTimeoutNs);
    } else if (warp >= 2 && warp < 10) {
        // ---------------- channel sums and token norms (warps 2-9), a_{t,n} (warps 2-5) ----------------
        // lane: channel pair p4 of this warp's 8 channels of a K step, and the
        // rows r = 8 i + re (i < 16) of the tile it sums.  With the 128-byte
        // swizzle (16-byte chunk k of row r at r * 128 + ((k ^ (r & 7)) << 4))
        // every one of those rows has r & 7 = re, so the lane's words sit at
        // lane_off + 1024 i (the eight values of re put the 32 lanes on 32
        // banks).  Warps 2-5 then take the tile's a_{t,n} for the rows of
        // their tensor-memory lane quadrant.
        const int wsel = warp - 2;
        const bool epi = warp < 6;
        const int p4 = lane & 3, re = lane >> 2;
        const int cw = wsel * 8 + 2 * p4;               // channels cw, cw + 1 of the K step
        const uint32_t lane_off = (uint32_t)(re * 128) + ((uint32_t)(wsel ^ re) << 4) + (uint32_t)(4 * p4);
        float *acc_open = acc_buf, *acc_next = acc_buf + c.D;
        int64_t open_f = any ? t.base / c.N : 0;
        bool open_has = false;
        int stage = 0;
        uint32_t phase = 0;
        int it = 0;
        for (bool on = any; on && !*abort_flag; on = t.next(c), ++it) {
            const int64_t base = t.base;
            const int nr = t.nr;
            // a frame starts inside the tile at row rb (frames have >= 128 tokens)
            const int to_end = (int)((int64_t)c.N - base % c.N);
            const int rb = to_end < nr ? to_end : nr;
            float sq[16];                   // squares of this lane's two channels, row 8 i + re
#pragma unroll
            for (int i = 0; i < 16; ++i) sq[i] = 0.f;
            const int a_sub = t.rows() * kXK * 2;   // bytes of one K step
            const int rbl = rb - re, nrl = nr - re;   // row 8 i + re below rb, nr: 8 i < rbl, nrl
            bool ok = true;
            for (int ks = 0; ks < KS; ks += G) {
                if (!ptx::mbar_wait(&S->full[stage], phase, kXTimeoutNs)) {
                    xfail(c, abort_flag, 32);
                    ok = false;
                    break;
                }
                // (indexed from the shared array itself: shared-memory loads)
                const uint8_t *st0 = smem_raw + ring_off + (size_t)stage * p.stage_stride;
#pragma unroll 1
                for (int g = 0; g < G; ++g) {
                    const uint8_t *lb = st0 + g * a_sub + lane_off;
                    // s0 the open frame's rows, s1 the next's: NI rows per lane
                    // (the tile's box), those past the tile as zeros; without a
                    // frame end in the tile packed sums of even and odd rows,
                    // else predicated ones (in PTX: as branches they take 1.4
                    // times the kernel's time)
                    float s0x = 0.f, s0y = 0.f, s1x = 0.f, s1y = 0.f;
                    auto rows = [&](auto ni, auto split) {
                        constexpr int NI = decltype(ni)::value;
                        uint32_t w[NI];
#pragma unroll
                        for (int i = 0; i < NI; ++i) {
                            w[i] = *reinterpret_cast<const uint32_t *>(lb + 1024 * i);
                            if (i >= NI - 4) w[i] = 8 * i < nrl ? w[i] : 0u;
                        }
                        f2_t e = 0ull, o = 0ull;
#pragma unroll
                        for (int i = 0; i < NI; ++i) {
                            const float x = bf16_lo(w[i]), y = bf16_hi(w[i]);
                            sq[i] = fmaf(x, x, fmaf(y, y, sq[i]));
                            if constexpr (decltype(split)::value)
                                asm("{\n"
                                    ".reg .pred p;\n"
                                    "setp.lt.s32 p, %6, %7;\n"
                                    "@p add.f32 %0, %0, %4;\n"
                                    "@p add.f32 %1, %1, %5;\n"
                                    "@!p add.f32 %2, %2, %4;\n"
                                    "@!p add.f32 %3, %3, %5;\n"
                                    "}"
                                    : "+f"(s0x), "+f"(s0y), "+f"(s1x), "+f"(s1y)
                                    : "f"(x), "f"(y), "r"(8 * i), "r"(rbl));
                            else if (i & 1) o = add2(o, pack2(x, y));
                            else e = add2(e, pack2(x, y));
                        }
                        if constexpr (!decltype(split)::value) {
                            const float2 s = unpack2(add2(e, o));
                            s0x = s.x;
                            s0y = s.y;
                        }
                    };
                    using std::integral_constant;
                    if (rb == nr) {
                        if (nr > 96) rows(integral_constant<int, 16>(), std::false_type());
                        else if (nr > 64) rows(integral_constant<int, 12>(), std::false_type());
                        else if (nr > 32) rows(integral_constant<int, 8>(), std::false_type());
                        else rows(integral_constant<int, 4>(), std::false_type());
                    } else {
                        if (nr > 96) rows(integral_constant<int, 16>(), std::true_type());
                        else if (nr > 64) rows(integral_constant<int, 12>(), std::true_type());
                        else if (nr > 32) rows(integral_constant<int, 8>(), std::true_type());
                        else rows(integral_constant<int, 4>(), std::true_type());
                    }
                    if (g == G - 1) {   // the stage's last K step is in registers: hand the stage back
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive(&S->empty[stage]);
                    }
                    // the eight row classes (lane bits 2-4), in a fixed order:
                    // the values are split over the lanes on the way, so that
                    // lanes with bit 4 clear end with the open frame's sum and
                    // those with it set with the next's, of channel cw (bit 3
                    // clear) or cw + 1
                    const bool up = (lane & 16) != 0, odd = (lane & 8) != 0;
                    const float a = (up ? s1x : s0x) + __shfl_xor_sync(0xffffffffu, up ? s0x : s1x, 16);
                    const float b = (up ? s1y : s0y) + __shfl_xor_sync(0xffffffffu, up ? s0y : s1y, 16);
                    float r = (odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
                    r += __shfl_xor_sync(0xffffffffu, r, 4);
                    const int ch = (ks + g) * kXK + cw + (odd ? 1 : 0);
                    if ((lane & 4) == 0 && (!up || rb < nr)) {
                        float *dst = up ? acc_next : acc_open;
                        dst[ch] += r;
                    }
                }
                if (++stage == p.stages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            if (!ok) break;
            // token norms: this warp's squares summed over its 4 channel pairs,
            // one partial per warp and row
            const int b = it & 1;
            const uint32_t use = (uint32_t)(it >> 1);
            // the rows' partials of the tile before the last have been read
            // (tiles of few stages let some warps run two tiles ahead)
            if (!ptx::mbar_wait(&S->tempty[b], (use & 1u) ^ 1u, kXTimeoutNs)) {
                xfail(c, abort_flag, 32);
                break;
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                float v = sq[i];
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                if (p4 == 0) S->npart[b][wsel][8 * i + re] = v;
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&S->csync[b]);
            open_has = true;
            if (rb < nr) {   // the open frame ended inside the tile
                xflush(c, acc_open, open_f, wsel * 8, lane);
                float *other = acc_open;
                acc_open = acc_next;
                acc_next = other;
                ++open_f;
            }
            if ((base + nr) % c.N == 0) {   // and the frame open now ends with the tile
                __syncwarp();
                xflush(c, acc_open, open_f, wsel * 8, lane);
                ++open_f;
                open_has = false;
            }
            __syncwarp();
            if (epi) {
                // a_{t,n} of the rows of this warp's lane quadrant: the eight
                // warps' partial squares in a fixed order, then the max over
                // the query rows of hi + lo from tensor memory
                if (!ptx::mbar_wait(&S->csync[b], use & 1u, kXTimeoutNs) ||
                    !ptx::mbar_wait(&S->tfull[b], use & 1u, kXTimeoutNs)) {
                    xfail(c, abort_flag, 32);
                    break;
                }
                ptx::tc_fence_after();
                const int q = warp & 3;                  // TMEM lane quadrant: rows q*32 .. q*32+31
                const int row = q * 32 + lane;
                float t2 = 0.f;
#pragma unroll
                for (int w = 0; w < kXReaders; ++w) t2 += S->npart[b][w][row];
                const float nrm = sqrtf(t2);
                const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * kXAccCols);
                float best = -INFINITY;
                for (int c0 = 0; c0 < t.Lqp; c0 += 16) {
                    uint32_t hi[16], lo[16];
                    ptx::tmem_ld_32x32b_x16(tbase + (uint32_t)c0, hi);
                    ptx::tmem_ld_32x32b_x16(tbase + (uint32_t)(t.Lqp + c0), lo);
                    ptx::tmem_ld_wait();
                    ptx::reg_fence16(hi);
                    ptx::reg_fence16(lo);
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (c0 + j < t.Lq) best = fmaxf(best, __uint_as_float(hi[j]) + __uint_as_float(lo[j]));
                }
                if (row < nr && wz_in_range(c.status, base + row < (int64_t)c.V * c.T * c.N))
                    c.a[base + row] = nrm > 0.f ? best / nrm : 0.f;
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&S->tempty[b]);
            }
        }
        if (open_has && !*abort_flag) xflush(c, acc_open, open_f, wsel * 8, lane);   // the CTA's share of it
    }
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, 2 * kXAccCols);
    }
}

namespace {

// [rows][cols] bf16 as {64 channels, rows, cols / 64 K steps}: box {64,
// box_rows, G}, i.e. G consecutive K-step tiles of box_rows rows.
bool xencode(PFN_cuTensorMapEncodeTiled_v12000 enc, CUtensorMap *m, const void *base, int64_t rows, int cols,
             int box_rows, int G) {
    cuuint64_t dims[3] = {(cuuint64_t)kXK, (cuuint64_t)rows, (cuuint64_t)(cols / kXK)};
    cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)kXK * 2};
    cuuint32_t box[3] = {(cuuint32_t)kXK, (cuuint32_t)box_rows, (cuuint32_t)G};
    cuuint32_t es[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct XLayout {
    int stages, stride, G, bstages, b_off, b_stride, acc_off, shared_off;
    size_t smem;
};

// K steps per feature stage (G, at most kXGroups, dividing the D / 64 K
// steps), the longest reads first, such that kXMinStages feature stages fit
// beside two query-row stages of one K step of the longest query; then the
// query-row stages up to kXBFlight bytes (of gb K steps where two such stages
// fit), then the rest to feature stages.
XLayout xlayout(int D, int Lqp) {
    XLayout L{};
    const size_t fixed = 1024 + (size_t)2 * D * 4 + (sizeof(XShared) + 127) / 128 * 128;
    const int room = (int)((size_t)227 * 1024 - fixed);
    const int step = 2 * Lqp * kXK * 2;   // one K step of query rows: a multiple of 4 KB
    for (L.G = kXGroups; L.G >= 1; L.G >>= 1) {
        if ((D / kXK) % L.G != 0) continue;
        L.stride = L.G * kXABytes;
        const int left = room - kXMinStages * L.stride;   // for query rows
        if (left < 2 * step) continue;
        int gb = L.G;
        while (gb > 1 && 2 * gb * step > std::min(left, kXBFlight)) gb >>= 1;
        L.b_stride = gb * step;
        L.bstages = std::max(2, std::min(std::min(left, kXBFlight) / L.b_stride, kXMaxBStages));
        L.stages = std::min((room - L.bstages * L.b_stride) / L.stride, kXMaxStages);
        break;
    }
    L.b_off = L.stages * L.stride;
    L.acc_off = L.b_off + L.bstages * L.b_stride;
    L.shared_off = L.acc_off + 2 * D * 4;
    L.smem = 1024 + (size_t)L.shared_off + sizeof(XShared);
    return L;
}

}  // namespace

// The fused pass applies to frames of at least 128 tokens, D a multiple of 64
// up to 4096 and at most 128 query rows per video (Lqp <= 128: the longest
// query, padded to 16).
bool maxsim_pass_supported(const Ctx &c, int Lqp) {
    if (c.N < kXM || c.D % kXK != 0 || c.D > 4096 || c.dtype != WZ_DTYPE_BF16) return false;
    if ((int64_t)c.V * c.T * c.N > (int64_t)INT32_MAX) return false;   // token coordinates of the tensor map
    if (Lqp < 16 || Lqp > WZ_MAX_LQ_MAXSIM || Lqp % 16 != 0) return false;
    return xlayout(c.D, Lqp).stages >= kXMinStages;
}

// Lqp: the longest query's padded rows; c.qhl holds qrows rows in all.
cudaError_t launch_maxsim_pass(const Ctx &c, int Lqp, int64_t qrows, cudaStream_t s) {
    if (!maxsim_pass_supported(c, Lqp)) return cudaErrorInvalidValue;
    auto enc = tmap_encode_fn();
    if (!enc) return cudaErrorNotSupported;
    XMaps maps;
    memset(&maps, 0, sizeof(maps));
    const XLayout L = xlayout(c.D, Lqp);
    for (int k = 0; k < kXRowMaps; ++k)
        if (!xencode(enc, &maps.a[k], c.X, (int64_t)c.V * c.T * c.N, c.D, 32 * (k + 1), L.G)) return cudaErrorInvalidValue;
    for (int k = 0; k < Lqp / 16; ++k)
        if (!xencode(enc, &maps.b[k], c.qhl, qrows, c.D, 32 * (k + 1), xgb(16 * (k + 1), L.b_stride, L.G)))
            return cudaErrorInvalidValue;
    XArgs p{};
    p.stages = L.stages;
    p.stage_stride = L.stride;
    p.bstages = L.bstages;
    p.b_off = L.b_off;
    p.b_stride = L.b_stride;
    p.acc_off = L.acc_off;
    p.shared_off = L.shared_off;
    const void *fn = L.G == 4 ? (const void *)maxsim_pass_kernel<4>
                     : L.G == 2 ? (const void *)maxsim_pass_kernel<2>
                                : (const void *)maxsim_pass_kernel<1>;
    cudaError_t e = allow_smem(fn, L.smem);
    if (e != cudaSuccess) return e;
    void *args[] = {&maps, const_cast<Ctx *>(&c), &p};
    return launch_kernel(fn, dim3(c.G1), dim3(kXThreads), L.smem, s, args, c.pdl != 0);
}

}  // namespace wz
