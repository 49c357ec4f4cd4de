// Cross-Modal Scorer, similarity branch (Section 3.2.1), on the GPU.
//
//   query_pool      u_q = mean of the query rows (compensated fp32 -> fp64).
//   relevance_pass  one streaming read of the features: per token
//                   a_{t,n} = <u, u_q> / (||u|| ||u_q||) (the input of Eq. 6)
//                   and per-CTA column sums of every frame it touches (the
//                   average pool of Section 3.2.1 / Eq. 7), in fp32.
//   frame_stats     one block per frame sums the column partials of the frame
//                   in a fixed order and forms r_t and delta_t (Eq. 7) from
//                   <v_t,u_q>, <v_t,v_t>, <v_t,v_{t-1}>, <v_{t-1},v_{t-1}>
//                   and <u_q,u_q>, reduced in fp64.
//   query_rows      (max-over-query scorer) the norms of the query rows and
//                   the rows scaled to unit length, split into bf16 hi + lo
//                   halves: the B operand of the token x row cosine GEMM.
//
// With the max-over-query scorer the relevance pass stores ||u|| in place of
// a_{t,n}; the tensor-core GEMM that follows divides max_j <u, q_j/||q_j||>
// by it, and frame_stats takes r_t = max_j cos(v_bar_t, q_j) from the raw
// rows and their norms.
//
// The relevance pass is HBM bound: it reads T*H*W*D elements once, streamed
// by TMA bulk copies through a shared-memory ring; each CTA owns one
// contiguous range of the flattened token index so the grid is balanced.
#include <algorithm>
#include <cstring>

#include "wz_internal.cuh"
#include "wz_ptx.cuh"

namespace wz {

// The videos' parameters in the kernel arguments, in blocks of a few sizes: a
// launch copies its whole argument block (20 KB at WZ_MAX_VIDEOS).
template <int N>
struct VideoParBlock {
    VideoPar v[N];
};

// What every kernel after the first one reads of video v.
__device__ __forceinline__ void video_init(const Ctx &c, int v, const VideoPar &vp) {
    c.vpar[v] = vp;
    if (v == 0 && c.clear_status) *c.status = 0;   // (a wait that gives up does so seconds later)
    if (c.drange) {   // empty range of delta_t, filled by frame_stats
        c.drange[2 * v] = 0x7ff0000000000000ull;   // +inf
        c.drange[2 * v + 1] = 0ull;                // +0
    }
}

__device__ __forceinline__ float2 load_two(const __nv_bfloat16 *p) {
    const uint32_t v = *reinterpret_cast<const uint32_t *>(p);
    return make_float2(bf16_lo(v), bf16_hi(v));
}
__device__ __forceinline__ float2 load_two(const float *p) { return *reinterpret_cast<const float2 *>(p); }

// u_q = mean of the query rows: a block covers 64 channels, two per thread (a
// warp reads 128 bytes or more of a row), with 8 row slices; compensated fp32
// sums (TwoSum) per slice, combined in a fixed order, stored as fp64 and fp32.
// Latency bound; half the CTAs of one channel per thread also leave the SMs to
// the relevance pass sooner (whole calls: 128 frames of 16 x 16, 64 rows 103.4
// -> 101.3 us, 32 videos of 64 frames 739.9 -> 738.0; 16 slices of 512 threads
// 100.6 and 740.5).
template <typename T, int NPAR>
__global__ void __launch_bounds__(256) query_pool_kernel(Ctx c, VideoParBlock<NPAR> par) {
    __shared__ float2 ps[8][32], pe[8][32];
    pdl_wait();
    pdl_trigger();
    const int v = blockIdx.y;
    const VideoPar vp = par.v[v];
    if (blockIdx.x == 0 && threadIdx.x == 0) video_init(c, v, vp);
    const int cl = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const int d = (blockIdx.x * 32 + cl) * 2;   // (D is even)
    float2 s = make_float2(0.f, 0.f), e = s;
    auto add = [](float2 &s, float2 &e, const float2 &x) {
        float t, err;
        two_sum(s.x, x.x, t, err);
        s.x = t;
        e.x += err;
        two_sum(s.y, x.y, t, err);
        s.y = t;
        e.y += err;
    };
    if (d < c.D) {
        const T *Q = static_cast<const T *>(c.Q) + (size_t)vp.q_row0 * c.D + d;
        // rows slice, slice + 8, ...: loaded 8 at a time, then summed in order
        for (int j0 = slice; j0 < vp.Lq; j0 += 64) {
            float2 x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int j = j0 + 8 * k;
                x[k] = j < vp.Lq ? load_two(Q + (size_t)j * c.D) : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (j0 + 8 * k < vp.Lq) add(s, e, x[k]);
        }
    }
    ps[slice][cl] = s;
    pe[slice][cl] = e;
    __syncthreads();
    if (slice < 2 && d < c.D) {   // warp h: the threads' channel h
        const bool h = slice != 0;
        float S = 0.f, E = 0.f;
        for (int k = 0; k < 8; ++k) {
            const float2 s2 = ps[k][cl], e2 = pe[k][cl];
            float t, err;
            two_sum(S, h ? s2.y : s2.x, t, err);
            S = t;
            E += err + (h ? e2.y : e2.x);
        }
        const double m = ((double)S + (double)E) / (double)vp.Lq;
        c.qbar64[(size_t)v * c.D + d + slice] = m;
        c.qbar32[(size_t)v * c.D + d + slice] = (float)m;
    }
}

// Unit query rows for the max-over-query scorer, blockIdx.y = video v0 + y:
// block j < Lq writes ||q_j|| (fp64 sum of fp32 squares) to qnorm and q_j /
// ||q_j|| as bf16 hi (row j of the video's rows in qhl, see qhl_row) and lo =
// bf16(x - hi) (row Lqp + j); blocks Lq <= j < Lqp write zero rows, so the
// GEMM's padding columns are zero.  bf16 rows, D % 64 == 0, read as 16-byte
// vectors and kept in registers between the two passes (the first kQRowKeep
// per thread).  With init != 0 the kernel is the first of the call.
constexpr int kQRowKeep = 2;

template <int NPAR>
__global__ void __launch_bounds__(256) query_rows_kernel(Ctx c, VideoParBlock<NPAR> par, int v0, int init) {
    __shared__ double red[33];
    pdl_wait();
    pdl_trigger();
    const int v = v0 + (int)blockIdx.y, j = blockIdx.x;
    const VideoPar vp = par.v[blockIdx.y];
    if (init && j == 0 && threadIdx.x == 0) video_init(c, v, vp);
    const int Lqp = (vp.Lq + 15) & ~15;
    if (j >= Lqp) return;
    const int n8 = c.D / 8;
    uint4 *hi = reinterpret_cast<uint4 *>(c.qhl + (size_t)(qhl_row(vp.q_row0, v) - c.qhl_row0 + j) * c.D);
    uint4 *lo = hi + (size_t)Lqp * n8;
    if (j >= vp.Lq) {
        for (int i = threadIdx.x; i < n8; i += 256) hi[i] = lo[i] = make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    const uint4 *q = reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(c.Q) +
                                                     (size_t)(vp.q_row0 + j) * c.D);
    uint4 keep[kQRowKeep];
    float ss = 0.f;
    auto square = [&](const uint4 &w) {
        float x[8];
        unpack(w, x, (__nv_bfloat16 *)nullptr);
#pragma unroll
        for (int e = 0; e < 8; ++e) ss = fmaf(x[e], x[e], ss);
    };
#pragma unroll
    for (int k = 0; k < kQRowKeep; ++k) {
        const int i = (int)threadIdx.x + 256 * k;
        keep[k] = i < n8 ? q[i] : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int k = 0; k < kQRowKeep; ++k) square(keep[k]);
    for (int i = (int)threadIdx.x + 256 * kQRowKeep; i < n8; i += 256) square(q[i]);
    const double qn = sqrt(block_sum((double)ss, red));
    if (threadIdx.x == 0) c.qnorm[(size_t)v * WZ_MAX_LQ_MAXSIM + j] = (float)qn;
    const float inv = qn > 0.0 ? (float)(1.0 / qn) : 0.f;
    auto split = [&](int i, const uint4 &w) {
        float x[8];
        unpack(w, x, (__nv_bfloat16 *)nullptr);
        uint32_t h[4], l[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float x0 = x[2 * e] * inv, x1 = x[2 * e + 1] * inv;
            const __nv_bfloat162 hh = __floats2bfloat162_rn(x0, x1);
            const __nv_bfloat162 ll = __floats2bfloat162_rn(x0 - __low2float(hh), x1 - __high2float(hh));
            h[e] = *reinterpret_cast<const uint32_t *>(&hh);
            l[e] = *reinterpret_cast<const uint32_t *>(&ll);
        }
        hi[i] = make_uint4(h[0], h[1], h[2], h[3]);
        lo[i] = make_uint4(l[0], l[1], l[2], l[3]);
    };
#pragma unroll
    for (int k = 0; k < kQRowKeep; ++k) {
        const int i = (int)threadIdx.x + 256 * k;
        if (i < n8) split(i, keep[k]);
    }
    for (int i = (int)threadIdx.x + 256 * kQRowKeep; i < n8; i += 256) split(i, q[i]);
}

// Reduce the NV values held by every lane across the warp (NV a power of
// two <= 32).  Each of the first log2(NV) steps halves the values a lane
// keeps; the remaining steps are plain butterflies.  On return lane l holds
// the warp total of value l >> (5 - log2(NV)).
template <int NV>
__device__ __forceinline__ float transpose_reduce(float (&v)[NV]) {
    const int lane = threadIdx.x & 31;
    int half = NV / 2;
    int o = 16;
#pragma unroll
    for (; half >= 1; half >>= 1, o >>= 1) {
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float keep = upper ? v[i + half] : v[i];
            const float send = upper ? v[i] : v[i + half];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    float r = v[0];
#pragma unroll
    for (; o >= 1; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}

constexpr int kRelMaxStages = 16;
constexpr int kRelMaxWarps = 24;         // consumer warps of a CTA (all groups)
constexpr int kRelWindow = 128;          // tokens per cross-warp reduction
constexpr int kRelGroupTokens = 8;       // tokens per warp transpose-reduction
constexpr size_t kRelSmem = 224 * 1024;   // dynamic shared memory of a CTA (at most)
constexpr uint64_t kRelTimeoutNs = 2000000000ull;

// Launch shape of the relevance pass (relevance_config).
struct RelShape {
    int ch;        // tokens per chunk (a multiple of kRelGroupTokens unless the row is long)
    int stages;    // ring stages: a multiple of groups, so that a stage always serves the same
                   // group and that group's warps see every phase of its barrier
    int groups;    // consumer groups; chunk k of the CTA goes to group k mod groups
    int gthreads;  // threads of a group (a multiple of 32)
    int wpart_off, csum_off;   // byte offsets of the window and of the groups' column sums
};

// One CTA streams tokens [blockIdx.x*L1, +L1) of the flattened [V*T*N] index.
// The last warp copies chunks of consecutive tokens (contiguous in HBM, never
// across a frame) into a shared-memory ring with cp.async.bulk.  The other
// warps form `groups` groups, each wide enough for one token row (VPT 16-byte
// vectors per thread); a group takes every groups-th chunk, waits for it,
// hands it back, and keeps its own column sums of the open frame, so a row of
// few vectors still occupies 15 to 24 warps.  Per-token partial dots and norms
// go to a window that all consumers reduce together once per <= 128 tokens;
// the groups' column sums are added (in group order) when the frame ends.
template <typename T, int VPT, int MAXTHREADS>
__global__ void __launch_bounds__(MAXTHREADS, 1) relevance_pass_kernel(Ctx c, RelShape sh) {
    // The producer streams only the features, which the kernels before this
    // one do not write, so where the launches overlap (the condensation calls;
    // wz_relevance and wz_relevance_static launch one after the other) it starts
    // before the wait for the previous grid (the query pooling) and fills the
    // ring meanwhile; the consumers wait for it before they read u_q or write
    // anything.
    pdl_trigger();
    constexpr int VEC = VecOf<T>::kElems;
    // tokens per transpose-reduction: chunks of long rows hold no more (1 or 2
    // tokens with 8 vectors per thread, at most 4 with 4); with 8 for all, the
    // widest rows spilled and took 2 % longer
    constexpr int GROUP = VPT == 8 ? 1 : VPT == 4 ? 4 : kRelGroupTokens;
    constexpr int NV = 2 * GROUP;            // GROUP dots + GROUP squared norms
    constexpr int HOLD = 32 / NV;            // lanes that end with the same value
    extern __shared__ __align__(128) uint8_t rsm[];
    __shared__ float qsum[kRelMaxWarps];
    __shared__ uint64_t full[kRelMaxStages], empty[kRelMaxStages];
    __shared__ volatile int abort_flag;
    const int NC = blockDim.x - 32;          // consumer threads
    const int nwg = sh.gthreads >> 5;        // warps of a group
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_vec = c.D / VEC;
    const int N = c.N, CH = sh.ch;
    const bool maxsim = c.relevance_mode == WZ_RELEVANCE_MAXSIM;
    const uint32_t rowb = (uint32_t)c.D * (uint32_t)sizeof(T);
    const uint32_t stage_bytes = (uint32_t)CH * rowb;
    const int64_t total = (int64_t)c.V * c.T * N;
    const int64_t start = (int64_t)blockIdx.x * c.L1;
    const int len = start < total ? (int)min(c.L1, total - start) : 0;   // tokens of this CTA (grid <= 2048 CTAs)
    if (threadIdx.x == 0) {
        for (int s = 0; s < sh.stages; ++s) {
            ptx::mbar_init(&full[s], 1);
            ptx::mbar_init(&empty[s], (uint32_t)nwg);
        }
        abort_flag = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async_smem();
    }
    __syncthreads();
    if (len <= 0) return;
    const int64_t f0 = start / N;
    const int pos0 = (int)(start - f0 * N);   // token index within its frame

    if (threadIdx.x >= NC) {
        // ---------------- producer ----------------
        if (lane == 0) {
            const uint64_t pol = ptx::policy_evict_first();
            const char *src = static_cast<const char *>(c.X) + (size_t)start * rowb;
            int s = 0;
            uint32_t ph = 0;
            uint32_t issued = 0, par = 0;    // per stage: copied to, parity of the last copy
            for (int tok = 0, pos = pos0; tok < len && !abort_flag;) {
                const int n = min(min(CH, N - pos), len - tok);
                if (!ptx::mbar_wait(&empty[s], ph ^ 1u, kRelTimeoutNs)) {
                    atomicOr(c.status, 16);
                    abort_flag = 1;
                    break;
                }
                ptx::mbar_arrive_expect_tx(&full[s], (uint32_t)n * rowb);
                ptx::bulk_load(rsm + s * stage_bytes, src, (uint32_t)n * rowb, &full[s], pol);
                issued |= 1u << s;
                par = (par & ~(1u << s)) | (ph << s);
                src += (size_t)n * rowb;
                tok += n;
                pos += n;
                if (pos == N) pos = 0;
                if (++s == sh.stages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            for (int k = 0; k < sh.stages; ++k)
                if (issued >> k & 1u) ptx::mbar_wait(&full[k], par >> k & 1u, kRelTimeoutNs);
        }
        return;
    }

    // ---------------- consumers ----------------
    pdl_wait();
    auto consumer_sync = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(NC) : "memory"); };
    constexpr int NP = VEC / 2;                  // packed pairs per 16-byte vector
    const int grp = (int)threadIdx.x / sh.gthreads;
    const int gtid = (int)threadIdx.x - grp * sh.gthreads;
    const int gwarp = gtid >> 5;
    // window: [2 buffers][nwg][dot, norm][kRelWindow]
    float *const wpart = reinterpret_cast<float *>(rsm + sh.wpart_off);
    const int wbuf = nwg * 2 * kRelWindow;
    float *const csum = reinterpret_cast<float *>(rsm + sh.csum_off);   // [groups - 1][D]
    // one group: two sets of column sums by token parity (shorter dependent chains)
    constexpr int CSP = VPT == 1 && MAXTHREADS <= 544 ? 2 : 1;
    f2_t q[VPT][NP], cs[CSP][VPT][NP];
    float qn = 0.f;
    const uint32_t ring = ptx::smem_u32(rsm) + (uint32_t)gtid * 16u;
    bool dead = false;
    // chunk counter modulo the groups, and the stage and phase of the chunk
    int turn = 0, s = 0;
    uint32_t ph = 0;
    int buf = 0, wcount = 0, wbase = 0;
    bool csum_read = false;                  // group 0 may still be reading csum
    int64_t f = f0;
    int pos = pos0;
    int tf = (int)(f0 % c.T), v = (int)(f0 / c.T), cur_v = -1;
    bool frame_new = true;
    for (int tok = 0; tok < len;) {
        const int n = min(min(CH, N - pos), len - tok);
        if (frame_new) {
            frame_new = false;
            if (v != cur_v) {
                cur_v = v;
                float qq = 0.f;
#pragma unroll
                for (int vi = 0; vi < VPT; ++vi) {
                    const int vidx = gtid + vi * sh.gthreads;
#pragma unroll
                    for (int e = 0; e < NP; ++e) {
                        const float q0 = vidx < n_vec ? c.qbar32[(size_t)v * c.D + vidx * VEC + 2 * e] : 0.f;
                        const float q1 = vidx < n_vec ? c.qbar32[(size_t)v * c.D + vidx * VEC + 2 * e + 1] : 0.f;
                        q[vi][e] = pack2(q0, q1);
                        qq = fmaf(q0, q0, fmaf(q1, q1, qq));
                    }
                }
                for (int o = 16; o > 0; o >>= 1) qq += __shfl_xor_sync(0xffffffffu, qq, o);
                consumer_sync();
                if (lane == 0) qsum[warp] = qq;
                consumer_sync();
                qq = 0.f;
                for (int w = 0; w < nwg; ++w) qq += qsum[w];
                qn = sqrtf(qq);
            }
#pragma unroll
            for (int vi = 0; vi < VPT; ++vi)
#pragma unroll
                for (int e = 0; e < NP; ++e) cs[0][vi][e] = cs[CSP - 1][vi][e] = 0ull;
        }
        if (turn == grp) {
            // this warp waits for the chunk itself (bounded; one verdict per warp)
            if (!dead && !__all_sync(0xffffffffu, ptx::mbar_wait(&full[s], ph, kRelTimeoutNs))) {
                dead = true;
                if (lane == 0) {
                    abort_flag = 1;
                    atomicOr(c.status, 32);
                }
            }
            if (!dead) {
                float *const wp = wpart + buf * wbuf + gwarp * 2 * kRelWindow;
                uint32_t row = ring + (uint32_t)s * stage_bytes;
                for (int g0 = 0; g0 < n; g0 += GROUP) {
                    float acc[NV];
                    const int left = n - g0;
#pragma unroll
                    for (int k = 0; k < GROUP; ++k) {
                        f2_t dd = 0ull, nn = 0ull;
                        if (k < left) {
#pragma unroll
                            for (int vi = 0; vi < VPT; ++vi) {
                                if (gtid + vi * sh.gthreads < n_vec) {
                                    const uint4 raw = ptx::lds128(row + (uint32_t)(vi * sh.gthreads) * 16u);
                                    f2_t x[NP];
                                    unpack_pairs(raw, x, (T *)nullptr);
#pragma unroll
                                    for (int e = 0; e < NP; ++e) {
                                        cs[k & (CSP - 1)][vi][e] = add2(cs[k & (CSP - 1)][vi][e], x[e]);
                                        dd = fma2(x[e], q[vi][e], dd);
                                        nn = fma2(x[e], x[e], nn);
                                    }
                                }
                            }
                        }
                        row += rowb;
                        const float2 d2 = unpack2(dd), n2 = unpack2(nn);
                        acc[k] = d2.x + d2.y;
                        acc[k + GROUP] = n2.x + n2.y;
                    }
                    const float tot = transpose_reduce<NV>(acc);
                    const int kk = (lane / HOLD) & (GROUP - 1);   // lane l holds value l / HOLD: token kk, dot or norm
                    if (lane % HOLD == 0 && kk < left) wp[(lane >> 4) * kRelWindow + wcount + g0 + kk] = tot;
                }
            }
            // hand the stage back once this warp's reads are done
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&empty[s]);
        }
        if (++turn == sh.groups) turn = 0;
        if (++s == sh.stages) {
            s = 0;
            ph ^= 1u;
        }
        tok += n;
        pos += n;
        wcount += n;
        if (pos == N || tok >= len) {
            // column partial of frame f from this CTA: slot blockIdx.x + f
            if (CSP == 2)
#pragma unroll
                for (int vi = 0; vi < VPT; ++vi)
#pragma unroll
                    for (int e = 0; e < NP; ++e) cs[0][vi][e] = add2(cs[0][vi][e], cs[CSP - 1][vi][e]);
            if (sh.groups > 1) {
                if (csum_read) consumer_sync();
                if (grp > 0) {
#pragma unroll
                    for (int vi = 0; vi < VPT; ++vi) {
                        const int vidx = gtid + vi * sh.gthreads;
                        if (vidx < n_vec) {
                            float *dst = csum + (size_t)(grp - 1) * c.D + vidx * VEC;
#pragma unroll
                            for (int e = 0; e < NP; ++e) *reinterpret_cast<f2_t *>(dst + 2 * e) = cs[0][vi][e];
                        }
                    }
                }
                consumer_sync();
                csum_read = true;
            }
            if (grp == 0 && !dead &&
                wz_in_range(c.status, (int64_t)blockIdx.x + f < (int64_t)c.G1 + (int64_t)c.V * c.T)) {
                float *dst = c.part + ((size_t)blockIdx.x + (size_t)f) * c.D;
#pragma unroll
                for (int vi = 0; vi < VPT; ++vi) {
                    const int vidx = gtid + vi * sh.gthreads;
                    if (vidx < n_vec) {
                        for (int g = 0; g < sh.groups - 1; ++g) {
                            const float *src = csum + (size_t)g * c.D + vidx * VEC;
#pragma unroll
                            for (int e = 0; e < NP; ++e)
                                cs[0][vi][e] = add2(cs[0][vi][e], *reinterpret_cast<const f2_t *>(src + 2 * e));
                        }
#pragma unroll
                        for (int e = 0; e < NP; e += 2) {
                            const float2 a = unpack2(cs[0][vi][e]), b = unpack2(cs[0][vi][e + 1]);
                            *reinterpret_cast<float4 *>(dst + vidx * VEC + 2 * e) = make_float4(a.x, a.y, b.x, b.y);
                        }
                    }
                }
            }
        }
        if (pos == N) {
            pos = 0;
            ++f;
            frame_new = true;
            if (++tf == c.T) {
                tf = 0;
                ++v;
            }
        }
        // reduce the window across a group's warps: when it is full, at the end
        // of the range, and before a new video changes u_q
        if (tok >= len || wcount + CH > kRelWindow || v != cur_v) {
            consumer_sync();
            csum_read = false;   // group 0 arrived here after its reads
            if (!wz_in_range(c.status, start + wbase + wcount <= total)) wcount = 0;
            const float *w0 = wpart + buf * wbuf;
            for (int t = threadIdx.x; t < wcount && !dead; t += NC) {
                float dot = 0.f, nrm = 0.f;
                for (int w = 0; w < nwg; ++w) {
                    dot += w0[2 * w * kRelWindow + t];
                    nrm += w0[(2 * w + 1) * kRelWindow + t];
                }
                c.a[start + wbase + t] = maxsim ? sqrtf(nrm)   // ||u||, divided out by the row-max GEMM
                                         : (nrm > 0.f && qn > 0.f) ? dot / (sqrtf(nrm) * qn) : 0.f;
            }
            buf ^= 1;
            wbase = tok;
            wcount = 0;
        }
    }
}

// Gate of the WSM for frame f (Eq. 6, Eq. 12): the saliency map M = min-max
// normalised a_{t,n} over the frame, average-pooled to the subband grid of
// each DWT level (hp x wp for the first) and scaled by lambda.  Called by a
// whole CTA, or by a warp (M2 its own map), beside those that form the frame
// statistics, so that the two chains overlap.
template <bool WARP>
__device__ __forceinline__ void frame_gate(const Ctx &c, int64_t f, float *M2) {
    const int t0 = WARP ? threadIdx.x & 31 : threadIdx.x, nth = WARP ? 32 : blockDim.x;
    const int N = c.N, H = c.H, W = c.W;
    const float *a = (c.ext_a ? c.ext_a : c.a) + f * N;
    float lo = INFINITY, hi = -INFINITY;
    for (int k = t0; k < N; k += nth) {
        const float x = a[k];
        M2[k] = x;
        lo = fminf(lo, x);
        hi = fmaxf(hi, x);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if constexpr (!WARP) {
        __shared__ float red2[32];
        const int lane = t0 & 31, w = t0 >> 5, nw = nth >> 5;
        if (lane == 0) {
            red2[w] = lo;
            red2[16 + w] = hi;
        }
        __syncthreads();
        lo = INFINITY;
        hi = -INFINITY;
        for (int k = 0; k < nw; ++k) {
            lo = fminf(lo, red2[k]);
            hi = fmaxf(hi, red2[16 + k]);
        }
    }
    const float rng = hi - lo;
    for (int k = t0; k < N; k += nth) M2[k] = rng > 0.f ? (M2[k] - lo) / rng : 0.f;
    if constexpr (WARP) __syncwarp();
    else __syncthreads();
    for (int l = 1; l <= c.wsm_levels; ++l) {
        const int hp = c.lvl_h[l], wp = c.lvl_w[l];
        if (!wz_in_range(c.status, c.goff[l - 1] + hp * wp <= c.gate_stride)) break;
        float *G = c.gate + f * (int64_t)c.gate_stride + c.goff[l - 1];
        for (int k = t0; k < hp * wp; k += nth) {
            const int ai = k / wp, bj = k % wp;
            const int r0 = (ai * H) / hp, r1 = ((ai + 1) * H + hp - 1) / hp;
            const int c0 = (bj * W) / wp, c1 = ((bj + 1) * W + wp - 1) / wp;
            float s = 0.f;
            for (int y = r0; y < r1; ++y)
                for (int x = c0; x < c1; ++x) s += M2[y * W + x];
            G[k] = c.lambda * (s / (float)((r1 - r0) * (c1 - c0)));
        }
    }
}

// The gates of a batch of many frames: CTA b of its kernel's gate CTAs forms
// one, or, where a frame has at most kWarpGateTokens tokens (gate_warps), one
// per warp.
constexpr int kWarpGateTokens = 512;

__device__ __forceinline__ void frame_gates(const Ctx &c, int b, int gate_warps, float *map) {
    if (!gate_warps) {
        frame_gate<false>(c, b, map);
        return;
    }
    const int warp = threadIdx.x >> 5, f = b * (int)(blockDim.x >> 5) + warp;
    if (f < c.V * c.T) frame_gate<true>(c, f, map + warp * kWarpGateTokens);
}

// The column partials of frame f: slots [slot, slot + cnt) (CTA c of the
// relevance pass holds its tokens [c L1, (c+1) L1) of frame f in slot c + f).
__device__ __forceinline__ void frame_slots(const Ctx &c, int64_t f, int64_t &slot, int &cnt) {
    const int64_t n0 = f * c.N, n1 = n0 + c.N - 1;
    int64_t lo, hi;
    if (n1 <= (int64_t)UINT32_MAX && c.L1 <= (int64_t)UINT32_MAX) {   // 32-bit divisions
        lo = (uint32_t)n0 / (uint32_t)c.L1;
        hi = (uint32_t)n1 / (uint32_t)c.L1;
    } else {
        lo = n0 / c.L1;
        hi = n1 / c.L1;
    }
    slot = lo + f;
    cnt = (int)(min((int64_t)c.G1 - 1, hi) - lo) + 1;
}

// r_t and delta_t of frame f = (v, t) from r's and delta's cosines (lanes 0 and
// 1 of a warp hold them, so that the two inverse square roots run side by
// side).  The cosine num * rsqrt(den2) of equal frames may miss 1 by its own
// rounding (an ulp of rsqrt, a half each of the products: less than 2^-51), so
// up to that delta_t is 0: a still video's gamma_t, min-max normalised, would be
// 1 otherwise.  (The square root and the division, whose cosine of equal frames
// is exactly 1, take 0.8 us more on 64 frames.)
constexpr double kCosineRounding = 1.0 / (1ull << 51);

__device__ __forceinline__ void frame_result(const Ctx &c, int64_t f, int v, int t, int lane, double cosine) {
    if (lane == 0) {
        const double r = c.ext_r ? (double)c.ext_r[f] : cosine;   // an external scorer's r_t
        c.fr[4 * f + 0] = r;
        if (c.frame_scores) c.frame_scores[f] = (float)r;
    }
    if (lane == 1) {
        const double away = 1.0 - cosine;
        const double d = t > 0 && away > kCosineRounding ? fmin(2.0, away) : 0.0;   // (NaN: 0)
        c.fr[4 * f + 1] = d;
        if (c.drange) {   // non-negative doubles order like their bit patterns
            const unsigned long long bits = (unsigned long long)__double_as_longlong(d);
            atomicMin(&c.drange[2 * v], bits);
            atomicMax(&c.drange[2 * v + 1], bits);
        }
    }
}

// <a, b> over four channels as two sums (even and odd ones).  A thread adds one
// number per vector to its running sums, so that these are short chains.
__device__ __forceinline__ f2_t dot4(const float4 &a, const float4 &b) {
    return fma2(pack2(a.x, a.y), pack2(b.x, b.y), fma2(pack2(a.z, a.w), pack2(b.z, b.w), 0ull));
}
__device__ __forceinline__ float pair_sum(f2_t v) {
    const float2 s = unpack2(v);
    return s.x + s.y;
}

// The squares and products of a frame's sums are fp32 within kStatsParts parts
// of the channels (trees that stop there) and fp64 over the parts: delta_t of a
// quiet video is a small difference of them, and gamma_t magnifies it.  Its rms
// error there, in 1e-8: 1.3 to 1.4 at D = 3584 and 1.4 to 3.3 at 8192 to 32768
// in every kernel below; 2.0 to 2.7 and 4.7 to 14 with chains over all of a
// thread's channels and one part per warp.
constexpr int kStatsParts = 32;

// Sum of N parts at p, p + stride, .. in fp64, as a tree (N a power of two).
template <int N>
__device__ __forceinline__ double parts_sum(const float *p, int stride) {
    if constexpr (N == 1) return (double)*p;
    else return parts_sum<N / 2>(p, stride) + parts_sum<N / 2>(p + N / 2 * stride, stride);
}

// Channels 4 i .. 4 i + 3 of the sums of FPB + 1 frames: the first two partials
// of every frame in flight together, further ones (frames of more than two
// CTAs' tokens) after them, in slot order.
template <int FPB>
__device__ __forceinline__ void partial_sums(const float4 *P, int nv, int i, const int (&slot)[FPB + 1],
                                             const int (&cnt)[FPB + 1], float4 (&sf)[FPB + 1]) {
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 y[FPB + 1];
#pragma unroll
    for (int k = 0; k <= FPB; ++k) {
        sf[k] = cnt[k] > 0 ? P[(size_t)slot[k] * nv + i] : zero;
        y[k] = cnt[k] > 1 ? P[(size_t)(slot[k] + 1) * nv + i] : zero;
    }
#pragma unroll
    for (int k = 0; k <= FPB; ++k) {
        sf[k].x += y[k].x; sf[k].y += y[k].y; sf[k].z += y[k].z; sf[k].w += y[k].w;
#pragma unroll 1
        for (int q = 2; q < cnt[k]; q += 2) {
            const float4 x = P[(size_t)(slot[k] + q) * nv + i];
            const float4 z = q + 1 < cnt[k] ? P[(size_t)(slot[k] + q + 1) * nv + i] : zero;
            sf[k].x += x.x; sf[k].y += x.y; sf[k].z += x.z; sf[k].w += x.w;
            sf[k].x += z.x; sf[k].y += z.y; sf[k].z += z.z; sf[k].w += z.w;
        }
    }
}

// One CTA per frame: the frame sums (fixed list of CTA partials) for all
// channels, read as 16-byte vectors, up to four partials of the frame and four
// of the one before it in flight; fp32 products summed to kStatsParts parts,
// these in fp64; then r_t = cos(v_bar_t, u_q) and delta_t = 1 - cos(v_bar_t,
// v_bar_{t-1}) clamped to [0, 2] (Eq. 7) in fp64.  Another CTA per frame forms its gate
// (where there is one).  Bound by the latency of these steps: 64 frames of
// 13 x 13 x 3584 take 4.6 us (first CTA past its wait to the last one's end);
// 6.0 us with the slots' divisions after the wait,
// 8.2 us with the partials of the two frames read one after the other, two at
// a time, 64-bit divisions, and the gate in the other half of the CTA.
__global__ void __launch_bounds__(512, 2) frame_stats_kernel(Ctx c) {
    __shared__ float wsum[kStatsParts][5];
    __shared__ float gate_map[WZ_MAX_HW * WZ_MAX_HW];   // the frame's saliency map
    const int VT = c.V * c.T, f = (int)blockIdx.x;
    const int v = f / c.T, t = f - v * c.T;
    int64_t sf_at = 0, sp_at = 0;
    int nf = 0, np = 0;
    if (f < VT) frame_slots(c, f, sf_at, nf);
    if (f < VT && t > 0) frame_slots(c, f - 1, sp_at, np);
    pdl_wait();
    pdl_trigger();
    if (f >= VT) {
        frame_gate<false>(c, f - VT, gate_map);
        return;
    }
    const int nv = c.D / 4;
    const float4 *Pf = reinterpret_cast<const float4 *>(c.part) + (size_t)sf_at * nv;
    const float4 *Pp = reinterpret_cast<const float4 *>(c.part) + (size_t)sp_at * nv;
    const float4 *Qv = reinterpret_cast<const float4 *>(c.qbar32 + (size_t)v * c.D);
    f2_t s0 = 0ull, s1 = 0ull, s2 = 0ull, s3 = 0ull, s4 = 0ull;
    const int nmax = max(nf, np);
    for (int i = threadIdx.x; i < nv; i += blockDim.x) {
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 q = Qv[i];
        float4 sf = zero, sp = zero;
        for (int k0 = 0; k0 < nmax; k0 += 4) {
            float4 x[4], y[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                x[k] = k0 + k < nf ? Pf[(size_t)(k0 + k) * nv + i] : zero;
                y[k] = k0 + k < np ? Pp[(size_t)(k0 + k) * nv + i] : zero;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {   // in slot order
                if (k0 + k < nf) { sf.x += x[k].x; sf.y += x[k].y; sf.z += x[k].z; sf.w += x[k].w; }
                if (k0 + k < np) { sp.x += y[k].x; sp.y += y[k].y; sp.z += y[k].z; sp.w += y[k].w; }
            }
        }
        if (c.frame_mean) {   // caller's buffer: 4-byte alignment only
            float *fm = c.frame_mean + (size_t)f * c.D + 4 * i;
            fm[0] = sf.x / (float)c.N;
            fm[1] = sf.y / (float)c.N;
            fm[2] = sf.z / (float)c.N;
            fm[3] = sf.w / (float)c.N;
        }
        s0 = add2(s0, dot4(sf, q));
        s1 = add2(s1, dot4(sf, sf));
        s2 = add2(s2, dot4(sf, sp));
        s3 = add2(s3, dot4(q, q));
        s4 = add2(s4, dot4(sp, sp));
    }
    float p0 = pair_sum(s0), p1 = pair_sum(s1), p2 = pair_sum(s2), p3 = pair_sum(s3), p4 = pair_sum(s4);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    auto halve = [&](int o) {
        p0 += __shfl_xor_sync(0xffffffffu, p0, o);
        p1 += __shfl_xor_sync(0xffffffffu, p1, o);
        p2 += __shfl_xor_sync(0xffffffffu, p2, o);
        p3 += __shfl_xor_sync(0xffffffffu, p3, o);
        p4 += __shfl_xor_sync(0xffffffffu, p4, o);
    };
    halve(16);
    halve(8);
    halve(4);
    if (nw == 16) halve(2);
    const int parts = kStatsParts / nw;   // of a warp: 2 of 16 warps, 4 of 8
    if (lane < parts) {
        float *w = wsum[warp * parts + lane];
        w[0] = p0;
        w[1] = p1;
        w[2] = p2;
        w[3] = p3;
        w[4] = p4;
    }
    __syncthreads();
    if (warp == 0) {
        // lane 4 k + h (k < 5) sums quantity k over the parts h, h + 4, ..; the
        // four sums in a tree
        double acc = lane < 20 ? parts_sum<kStatsParts / 4>(&wsum[lane & 3][lane >> 2], 4 * 5) : 0.0;
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        const double vq = __shfl_sync(0xffffffffu, acc, 0), vv = __shfl_sync(0xffffffffu, acc, 4);
        const double vp = __shfl_sync(0xffffffffu, acc, 8), qq = __shfl_sync(0xffffffffu, acc, 12);
        const double pp = __shfl_sync(0xffffffffu, acc, 16);
        const double den2 = vv * (lane == 0 ? qq : pp), num = lane == 0 ? vq : vp;
        frame_result(c, f, v, t, lane, den2 > 0.0 ? num * rsqrt(den2) : 0.0);
    }
}

// The same for many frames: a CTA takes FPB consecutive frames of one video
// (ceil(T / FPB) CTAs per video), so that a frame's partials are read once
// instead of twice and the frames' loads are in flight together; the same sums
// in the same order.  The gates are formed by further CTAs, a warp each where
// a frame is small.  2048 frames of 13 x 13 x 3584 with gates: 20.5 us (cold),
// 31.1 with a CTA per frame and per gate (6.7 waves of them).
constexpr int kStatsThreads = 256;   // of the kernels with several frames per CTA
constexpr int kStatsFrames = 4;

template <int FPB>
__global__ void __launch_bounds__(kStatsThreads, 3) frame_stats_many_kernel(Ctx c, int gate_warps) {
    constexpr int NW = kStatsThreads / 32, NQ = 3 * FPB + 2;   // vq, vv, vp of each frame; qq, the first pp
    constexpr int PW = kStatsParts / NW;   // parts of a warp
    __shared__ float wsum[kStatsParts][NQ];
    __shared__ float gate_map[WZ_MAX_HW * WZ_MAX_HW];
    static_assert(NW * kWarpGateTokens <= WZ_MAX_HW * WZ_MAX_HW && FPB <= NW, "a map and a frame per warp");
    const int per_video = (c.T + FPB - 1) / FPB, nstat = c.V * per_video;
    const int v = (int)blockIdx.x / per_video, t0 = ((int)blockIdx.x - v * per_video) * FPB;
    const int nf = min(FPB, c.T - t0);
    const int64_t f0 = (int64_t)v * c.T + t0;
    // the column partials of frame f0 - 1 + k
    int slot[FPB + 1], cnt[FPB + 1];
#pragma unroll
    for (int k = 0; k <= FPB; ++k) {
        int64_t at = 0;
        cnt[k] = 0;
        if ((int)blockIdx.x < nstat && (k > 0 || t0 > 0) && k <= nf) frame_slots(c, f0 - 1 + k, at, cnt[k]);
        slot[k] = (int)at;   // < G1 + V T
    }
    pdl_wait();
    pdl_trigger();
    if ((int)blockIdx.x >= nstat) {
        frame_gates(c, (int)blockIdx.x - nstat, gate_warps, gate_map);
        return;
    }
    const int nv = c.D / 4;
    const float4 *P = reinterpret_cast<const float4 *>(c.part);
    const float4 *Qv = reinterpret_cast<const float4 *>(c.qbar32 + (size_t)v * c.D);
    float acc[NQ];
#pragma unroll
    for (int k = 0; k < NQ; ++k) acc[k] = 0.f;
#pragma unroll 1
    for (int i = threadIdx.x; i < nv; i += kStatsThreads) {
        const float4 q = Qv[i];
        float4 sf[FPB + 1];
        partial_sums<FPB>(P, nv, i, slot, cnt, sf);
#pragma unroll
        for (int k = 0; k < FPB; ++k) {
            if (c.frame_mean && k < nf) {   // caller's buffer: 4-byte alignment only
                float *fm = c.frame_mean + (size_t)(f0 + k) * c.D + 4 * i;
                fm[0] = sf[k + 1].x / (float)c.N;
                fm[1] = sf[k + 1].y / (float)c.N;
                fm[2] = sf[k + 1].z / (float)c.N;
                fm[3] = sf[k + 1].w / (float)c.N;
            }
            acc[3 * k] += pair_sum(dot4(sf[k + 1], q));
            acc[3 * k + 1] += pair_sum(dot4(sf[k + 1], sf[k + 1]));
            acc[3 * k + 2] += pair_sum(dot4(sf[k + 1], sf[k]));
        }
        acc[3 * FPB] += pair_sum(dot4(q, q));
        acc[3 * FPB + 1] += pair_sum(dot4(sf[0], sf[0]));
    }
    for (int o = 16; o >= PW; o >>= 1)
#pragma unroll
        for (int k = 0; k < NQ; ++k) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane < PW)
#pragma unroll
        for (int k = 0; k < NQ; ++k) wsum[warp * PW + lane][k] = acc[k];
    __syncthreads();
    if (warp < nf) {
        // warp k's frame: lane 4 m + h (m < 5) sums quantity m over the parts h, h + 4, ..
        const int m = lane >> 2;
        const int col = m < 3 ? 3 * warp + m : m == 3 ? 3 * FPB : warp == 0 ? 3 * FPB + 1 : 3 * (warp - 1) + 1;
        double s = lane < 20 ? parts_sum<kStatsParts / 4>(&wsum[lane & 3][col], 4 * NQ) : 0.0;
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        const double vq = __shfl_sync(0xffffffffu, s, 0), vv = __shfl_sync(0xffffffffu, s, 4);
        const double vp = __shfl_sync(0xffffffffu, s, 8), qq = __shfl_sync(0xffffffffu, s, 12);
        const double pp = __shfl_sync(0xffffffffu, s, 16);
        const double den2 = vv * (lane == 0 ? qq : pp), num = lane == 0 ? vq : vp;
        frame_result(c, f0 + warp, v, t0 + warp, lane, den2 > 0.0 ? num * rsqrt(den2) : 0.0);
    }
}

// The max-over-query scorer's frame statistics: a cluster of S CTAs takes
// eight consecutive frames of one video (ceil(T / 8) clusters per video), each
// CTA 1 / S of the channels: it forms the frames' sums there (shared
// memory, [9][channels] with the frame before), their squares and neighbour
// products (a warp per frame), and their dots with the video's query rows (a
// warp per kMxRows rows: lanes over the channels, one transpose-reduction over
// the 32 dots).  CTA k of the cluster then adds the parts of the dots of
// frames k, k + S, .. and takes r_t = max_j <v_t, q_j> / ||q_j|| / ||v_t||.  The gates are
// formed by further clusters beside them, a warp each where there are many
// small frames.  The query rows are read once per eight frames, 1 / S by
// each CTA: with CTAs of one to four whole frames their L2 reads bounded the
// kernel (events around it: 512 frames of 13 x 13 x 3584 and 8 to 119 rows 35
// us, 30 now; 128 rows 41 and 34; 128 frames of 16 x 16, 64 rows 18.0 and 16.4),
// now the latency of its steps.  Eight CTAs per cluster there: 33 us (1.7 waves).
constexpr int kMxFrames = 8;         // of a cluster
constexpr int kMxRows = 4;

template <int S>
__global__ void __launch_bounds__(kStatsThreads, 2) frame_stats_maxsim_kernel(Ctx c, int gate_warps) {
    __shared__ float part[kMxFrames][WZ_MAX_LQ_MAXSIM];   // <v_f, q_j> over this CTA's channels
    constexpr int PW = kStatsParts / S;   // parts of a warp
    __shared__ float wsum[kMxFrames][3][PW];              // vv, v.v_prev, v_prev.v_prev over them
    __shared__ double best[kMxFrames / S][4], tot[kMxFrames / S][3];
    __shared__ int slots[kMxFrames + 1], counts[kMxFrames + 1];
    __shared__ float gate_map[WZ_MAX_HW * WZ_MAX_HW];
    extern __shared__ float4 sfs[];   // [9][2 * per] frame sums: frame f0 - 1 + k of this CTA's channels
    static_assert(kStatsThreads == 32 * kMxFrames && WZ_MAX_LQ_MAXSIM == 128, "a warp per frame, four for the rows");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per_video = (c.T + kMxFrames - 1) / kMxFrames, nstat = c.V * per_video * S;
    const int group = (int)blockIdx.x / S, v = group / per_video, t0 = (group - v * per_video) * kMxFrames;
    const int nf = min(kMxFrames, c.T - t0);
    const int64_t f0 = (int64_t)v * c.T + t0;
    // the column partials of frame f0 - 1 + k
    if ((int)blockIdx.x < nstat && tid <= kMxFrames) {
        int64_t at = 0;
        int n = 0;
        if ((tid > 0 || t0 > 0) && tid <= nf) frame_slots(c, f0 - 1 + tid, at, n);
        slots[tid] = (int)at;   // < G1 + V T
        counts[tid] = n;
    }
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    if ((int)blockIdx.x >= nstat) {   // whole clusters
        const int b = (int)blockIdx.x - nstat;
        if (gate_warps || b < c.V * c.T) frame_gates(c, b, gate_warps, gate_map);
        return;
    }
    const int rank = (int)ptx::cluster_rank();
    const int Lq = c.vpar[v].Lq, q_row0 = c.vpar[v].q_row0;
    // this CTA's channels: 16-byte vectors v0 .. v0 + nvec - 1 of a row
    const int n8 = c.D / 8, per = (n8 + S - 1) / S, v0 = min(rank * per, n8), nvec = min(per, n8 - v0);
    const int nq = 2 * nvec;
    {
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 *P = reinterpret_cast<const float4 *>(c.part) + 2 * v0;
        const size_t nv = (size_t)c.D / 4;
#pragma unroll 4
        for (int idx = tid; idx < (kMxFrames + 1) * nq; idx += kStatsThreads) {
            const int k = idx / nq, i = idx - k * nq, n = counts[k];
            const float4 *src = P + (size_t)slots[k] * nv + i;
            float4 s = n > 0 ? src[0] : zero;
            const float4 y = n > 1 ? src[nv] : zero;
            s.x += y.x; s.y += y.y; s.z += y.z; s.w += y.w;
            for (int q = 2; q < n; ++q) {
                const float4 z = src[(size_t)q * nv];
                s.x += z.x; s.y += z.y; s.z += z.z; s.w += z.w;
            }
            sfs[k * 2 * per + i] = s;
        }
    }
    __syncthreads();
    {
        const float4 *cur = sfs + (warp + 1) * 2 * per, *prev = sfs + warp * 2 * per;
        f2_t sum[3][2] = {};   // by vector parity: a lane's chains are as short as those of 512 threads
        for (int i = lane; i < nq; i += 64)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (i + 32 * h < nq) {
                    const float4 s = cur[i + 32 * h], p = prev[i + 32 * h];
                    sum[0][h] = add2(sum[0][h], dot4(s, s));
                    sum[1][h] = add2(sum[1][h], dot4(s, p));
                    sum[2][h] = add2(sum[2][h], dot4(p, p));
                }
        float vv = pair_sum(add2(sum[0][0], sum[0][1])), vp = pair_sum(add2(sum[1][0], sum[1][1]));
        float pp = pair_sum(add2(sum[2][0], sum[2][1]));
        for (int o = 16; o >= PW; o >>= 1) {
            vv += __shfl_xor_sync(0xffffffffu, vv, o);
            vp += __shfl_xor_sync(0xffffffffu, vp, o);
            pp += __shfl_xor_sync(0xffffffffu, pp, o);
        }
        if (lane < PW) {
            wsum[warp][0][lane] = vv;
            wsum[warp][1][lane] = vp;
            wsum[warp][2][lane] = pp;
        }
    }
    const uint4 *Qr = reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(c.Q) + (size_t)q_row0 * c.D) + v0;
    for (int j0 = warp * kMxRows; j0 < Lq; j0 += kStatsThreads / 32 * kMxRows) {
        f2_t acc[kMxFrames][kMxRows];
#pragma unroll
        for (int k = 0; k < kMxFrames; ++k)
#pragma unroll
            for (int u = 0; u < kMxRows; ++u) acc[k][u] = 0ull;
#pragma unroll 1
        for (int i = lane; i < nvec; i += 32) {
            f2_t q[kMxRows][4];
#pragma unroll
            for (int u = 0; u < kMxRows; ++u) {
                const uint4 x = j0 + u < Lq ? __ldg(Qr + (size_t)(j0 + u) * n8 + i) : make_uint4(0u, 0u, 0u, 0u);
                unpack_pairs(x, q[u], (__nv_bfloat16 *)nullptr);
            }
#pragma unroll
            for (int k = 0; k < kMxFrames; ++k) {
                const ulonglong2 *sk = reinterpret_cast<const ulonglong2 *>(sfs + (k + 1) * 2 * per + 2 * i);
                const ulonglong2 a = sk[0], b = sk[1];
#pragma unroll
                for (int u = 0; u < kMxRows; ++u)
                    acc[k][u] = fma2(q[u][0], a.x, fma2(q[u][1], a.y, fma2(q[u][2], b.x, fma2(q[u][3], b.y, acc[k][u]))));
            }
        }
        float d[kMxFrames * kMxRows];
#pragma unroll
        for (int k = 0; k < kMxFrames; ++k)
#pragma unroll
            for (int u = 0; u < kMxRows; ++u) {
                const float2 x = unpack2(acc[k][u]);
                d[k * kMxRows + u] = x.x + x.y;
            }
        const float r = transpose_reduce<kMxFrames * kMxRows>(d);   // lane l holds value l
        part[lane / kMxRows][j0 + lane % kMxRows] = r;
    }
    __syncwarp();
    ptx::cluster_sync();   // every CTA's parts
    for (int m = 0, f = rank; f < nf; ++m, f += S) {
        if (warp < 4) {
            const int j = tid;
            double x = -INFINITY;
            if (j < Lq) {
                const double qn = (double)c.qnorm[(size_t)v * WZ_MAX_LQ_MAXSIM + j];
                float p[S];
#pragma unroll
                for (int r = 0; r < S; ++r) p[r] = ptx::ld_cluster(ptx::map_cluster(&part[f][j], (uint32_t)r));
#pragma unroll
                for (int o = 1; o < S; o <<= 1)
#pragma unroll
                    for (int r = 0; r < S; r += 2 * o) p[r] += p[r + o];
                x = qn > 0.0 ? (double)p[0] / qn : 0.0;
            }
            for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
            if (lane == 0) best[m][warp] = x;
        } else if (warp == 4) {   // lane S q + r: quantity q of CTA r
            double s = 0.0;
            if (lane < 3 * S) {
                const uint32_t at = ptx::map_cluster(wsum[f][lane / S], (uint32_t)(lane % S));
                float w[PW];
#pragma unroll
                for (int k = 0; k < PW; ++k) w[k] = ptx::ld_cluster(at + 4u * k);
                s = parts_sum<PW>(w, 1);
            }
            for (int o = 1; o < S; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane < 3 * S && lane % S == 0) tot[m][lane / S] = s;
        }
    }
    __syncwarp();
    ptx::cluster_sync();   // the parts have been read (and best, tot are written)
    const int f = rank + warp * S;   // a warp per frame
    if (warp < kMxFrames / S && f < nf) {
        const double m = fmax(fmax(best[warp][0], best[warp][1]), fmax(best[warp][2], best[warp][3]));
        const double den2 = lane == 0 ? tot[warp][0] : tot[warp][0] * tot[warp][2], num = lane == 0 ? m : tot[warp][1];
        frame_result(c, f0 + f, v, t0 + f, lane, den2 > 0.0 ? num * rsqrt(den2) : 0.0);
    }
}

namespace {

template <int N>
VideoParBlock<N> par_block(const VideoPar *hpar, int n) {
    VideoParBlock<N> blk;
    memset(&blk, 0, sizeof(blk));
    for (int v = 0; v < n; ++v) blk.v[v] = hpar[v];
    return blk;
}

template <int N>
cudaError_t query_pool_n(const Ctx &c, const VideoPar *hpar, cudaStream_t s) {
    VideoParBlock<N> blk = par_block<N>(hpar, c.V);   // copied into the launch parameters
    const dim3 grid((unsigned)((c.D + 63) / 64), (unsigned)c.V);
    void *args[] = {const_cast<Ctx *>(&c), &blk};
    const void *fn = c.dtype == WZ_DTYPE_BF16 ? (const void *)query_pool_kernel<__nv_bfloat16, N>
                                              : (const void *)query_pool_kernel<float, N>;
    return launch_kernel(fn, grid, dim3(256), 0, s, args, c.pdl != 0);
}

template <int N>
cudaError_t query_rows_n(const Ctx &c, const VideoPar *hpar, int v0, int nv, int Lqp, int init, cudaStream_t s) {
    VideoParBlock<N> blk = par_block<N>(hpar + v0, nv);
    void *args[] = {const_cast<Ctx *>(&c), &blk, &v0, &init};
    return launch_kernel((const void *)query_rows_kernel<N>, dim3((unsigned)Lqp, (unsigned)nv), dim3(256), 0, s, args,
                         c.pdl != 0);
}

}  // namespace

cudaError_t launch_query_pool(const Ctx &c, const VideoPar *hpar, cudaStream_t s) {
    return c.V == 1 ? query_pool_n<1>(c, hpar, s)
           : c.V <= 32 ? query_pool_n<32>(c, hpar, s) : query_pool_n<WZ_MAX_VIDEOS>(c, hpar, s);
}

// Videos v0 .. v0 + nv - 1; Lqp: the longest of their queries, padded to 16.
cudaError_t launch_query_rows(const Ctx &c, const VideoPar *hpar, int v0, int nv, int Lqp, bool init, cudaStream_t s) {
    return nv == 1 ? query_rows_n<1>(c, hpar, v0, nv, Lqp, init, s)
           : nv <= 32 ? query_rows_n<32>(c, hpar, v0, nv, Lqp, init, s)
                      : query_rows_n<WZ_MAX_VIDEOS>(c, hpar, v0, nv, Lqp, init, s);
}

namespace {

struct RelCfg {
    const void *fn = nullptr;
    int threads = 0;     // consumers + one producer warp
    RelShape sh{};
    size_t smem = 0;
};

// Shape for one CTA per SM.  A row of w warps gets the most groups that fit 16
// warps when those come to at least 15, else 24: too few warps leave the
// shared-memory and barrier latencies exposed, more than needed cost
// registers and barrier arrivals.  Whole wz_relevance calls on about 0.55 GB
// (16 x 16 maps), one group / 16 / 24 warps: D = 512: 181 / 119 / 120 us;
// 1152: 212 / 161 / 158; 2304: 146 / - / 122; 2816: 127 / - / 116; 3072 (12
// warps a row): 120.3 / - / 120.1.  A thread holds at most 8 elements of a row
// in groups of more than one.  Rows of one warp take four groups: their chunks
// are short work, and with more groups (or more than 8 tokens a chunk) the
// barriers and the merge of the groups' sums at every frame end cost more than
// they hide.  wz_relevance, one / four / sixteen groups (sixteen with chunks of 32
// tokens): 4096 frames of 16 x 16 x 128 147 / 144 / 278 us, of 6 x 6 x 256 56 / 54 /
// 91, 3000 of 7 x 7 x 64 fp32 40 / 42 / 91.  CTAs of fewer than 64 tokens (short clips) stay
// with one group: the groups' column sums cost more than they save there (16
// frames of 13 x 13 x 896: 27 us with one group, 30 us with three).
template <typename T, int VPT>
void relevance_config(const Ctx &c, RelCfg &r) {
    constexpr int VEC = VecOf<T>::kElems;
    constexpr bool kNarrow = VPT * VEC <= 8;
    const int n_vec = c.D / VEC;
    const size_t rowb = (size_t)c.D * sizeof(T);
    RelShape &sh = r.sh;
    sh.gthreads = std::max(32, ((n_vec + VPT - 1) / VPT + 31) / 32 * 32);
    const int w = sh.gthreads / 32;
    sh.groups = 1;
    if (kNarrow) sh.groups = w == 1 ? 4 : std::max(1, (16 / w) * w >= 15 ? 16 / w : kRelMaxWarps / w);
    const int64_t per_cta = ((int64_t)c.V * c.T * c.N + c.sms - 1) / c.sms;
    sh.groups = (int)std::min<int64_t>(sh.groups, std::max<int64_t>(1, per_cta / 32));
    const size_t wpart = (size_t)2 * w * 2 * kRelWindow * 4;
    size_t csum = 0, ring = 0;
    for (; sh.groups > 1; --sh.groups) {
        // chunks of 8 tokens, at least two stages per group
        csum = (size_t)(sh.groups - 1) * c.D * 4;
        ring = kRelSmem - wpart - csum;
        sh.ch = 8;
        sh.stages = (int)std::min<size_t>(kRelMaxStages, ring / (sh.ch * rowb)) / sh.groups * sh.groups;
        if (sh.stages >= 2 * sh.groups) break;
    }
    if (sh.groups == 1) {   // three stages of up to 8 tokens (32: short rows)
        csum = 0;
        ring = kRelSmem - wpart;
        sh.ch = (int)std::max<size_t>(1, std::min<size_t>(32, ring / 3 / rowb));
        if (sh.ch >= 8) sh.ch = sh.ch / 8 * 8;
        sh.stages = 3;
    }
    const int cons = sh.groups * sh.gthreads;
    r.threads = cons + 32;
    if constexpr (kNarrow)
        r.fn = cons <= 512 ? (const void *)relevance_pass_kernel<T, VPT, 512 + 32>
                           : (const void *)relevance_pass_kernel<T, VPT, kRelMaxWarps * 32 + 32>;
    else
        r.fn = (const void *)relevance_pass_kernel<T, VPT, 512 + 32>;
    sh.wpart_off = (int)(((size_t)sh.stages * sh.ch * rowb + 127) / 128 * 128);
    sh.csum_off = sh.wpart_off + (int)wpart;
    r.smem = (size_t)sh.csum_off + csum;
}

template <typename T>
bool pick(const Ctx &c, RelCfg &r) {
    constexpr int VEC = VecOf<T>::kElems;
    const int n_vec = c.D / VEC;
    if (n_vec <= 512) relevance_config<T, 1>(c, r);
    else if (n_vec <= 1024) relevance_config<T, 2>(c, r);
    else if (n_vec <= 2048) relevance_config<T, 4>(c, r);
    else if (n_vec <= 4096) relevance_config<T, 8>(c, r);
    else return false;
    return true;
}

bool pick_any(const Ctx &c, RelCfg &r) {
    return c.dtype == WZ_DTYPE_BF16 ? pick<__nv_bfloat16>(c, r) : pick<float>(c, r);
}

}  // namespace

int relevance_grid(const Ctx &c) {
    RelCfg r;
    if (c.sms < 1 || !pick_any(c, r)) return 0;
    int per_sm = 0;
    if (allow_smem(r.fn, r.smem) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, r.fn, r.threads, r.smem) != cudaSuccess) return 0;
    if (per_sm < 1) per_sm = 1;
    const int64_t total = (int64_t)c.V * c.T * c.N;
    int64_t g = (int64_t)c.sms * per_sm;
    const int64_t min_tokens = 16;
    g = std::min<int64_t>(g, (total + min_tokens - 1) / min_tokens);
    g = std::min<int64_t>(g, kG1Max);
    return (int)std::max<int64_t>(g, 1);
}

cudaError_t launch_relevance_pass(const Ctx &c, cudaStream_t s) {
    RelCfg r;
    if (!pick_any(c, r) || r.sh.stages % r.sh.groups != 0) return cudaErrorInvalidValue;   // (see RelShape)
    cudaError_t e = allow_smem(r.fn, r.smem);
    if (e != cudaSuccess) return e;
    void *args[] = {const_cast<Ctx *>(&c), &r.sh};
    return launch_kernel(r.fn, dim3(c.G1), dim3(r.threads), r.smem, s, args, c.pdl != 0);
}

cudaError_t launch_frame_stats(const Ctx &c, cudaStream_t s) {
    void *args[] = {const_cast<Ctx *>(&c)};
    const int sms = c.sms;
    const int64_t frames = (int64_t)c.V * c.T, gates = c.gate && c.spatial_mode == WZ_SPATIAL_WSM ? frames : 0;
    if (c.relevance_mode == WZ_RELEVANCE_MAXSIM) {
        int gate_warps = frames > sms && c.N <= kWarpGateTokens;
        const int64_t per = gate_warps ? kStatsThreads / 32 : 1, gate_ctas = (gates + per - 1) / per;
        // eight CTAs per eight frames, four where those and the gates are more
        // than one wave (256 frames of 27 x 27, 16 / 64 / 128 rows: 18.3 / 21.3 /
        // 26.4 us with eight, 16.2 / 20.1 / 26.2 with four)
        const int64_t octets = c.V * (int64_t)((c.T + kMxFrames - 1) / kMxFrames);
        const int S = 8 * octets + gate_ctas > 2 * (int64_t)sms && c.D <= 8192 ? 4 : 8;
        const void *fn = S == 4 ? (const void *)frame_stats_maxsim_kernel<4> : (const void *)frame_stats_maxsim_kernel<8>;
        const size_t smem = (size_t)(kMxFrames + 1) * 2 * ((c.D / 8 + S - 1) / S) * 16;
        const cudaError_t e = allow_smem(fn, smem);
        if (e != cudaSuccess) return e;
        void *margs[] = {const_cast<Ctx *>(&c), &gate_warps};
        return launch_kernel(fn, dim3((unsigned)((octets + (gate_ctas + S - 1) / S) * S)), dim3(kStatsThreads), smem, s,
                             margs, c.pdl != 0, (unsigned)S);
    }
    if (frames > 4 * (int64_t)sms && c.T >= kStatsFrames) {
        // more than two waves of a CTA per frame and gate
        int gate_warps = c.N <= kWarpGateTokens;
        const int64_t per = gate_warps ? kStatsThreads / 32 : 1;
        const int64_t ctas = c.V * (int64_t)((c.T + kStatsFrames - 1) / kStatsFrames) + (gates + per - 1) / per;
        void *margs[] = {const_cast<Ctx *>(&c), &gate_warps};
        return launch_kernel((const void *)frame_stats_many_kernel<kStatsFrames>, dim3((unsigned)ctas),
                             dim3(kStatsThreads), 0, s, margs, c.pdl != 0);
    }
    // a CTA per frame and one per gate; 256 threads (more CTAs in flight) once
    // 512 no longer fit in one wave
    const int64_t ctas = frames + gates;
    const int threads = ctas > 2 * (int64_t)sms ? 256 : 512;
    return launch_kernel((const void *)frame_stats_kernel, dim3((unsigned)ctas), dim3(threads), 0, s, args, c.pdl != 0);
}

}  // namespace wz
