// Condensed tokens Z_m = W_m X_m on CUDA cores in fp32 (Eq. 16, 18).
//
// Used for fp32 features (the tensor cores would need a split of X as well)
// and as an independent second path for bf16.  Persistent CTAs take tiles of
// TM output rows of a frame x TN channels from a static list (the prefix of
// the frames' row blocks in shared memory), K in steps of 32 tokens through a
// ring of kSimtStages cp.async stages; a thread forms RT rows x 4 CG columns,
// products in f32x2 (column pairs), every output one chain in ascending K.
// Bound by latency for few frames and by the FMA pipe (43 of 75 TFLOP/s) for
// many: 64 frames of 13 x 13 x 3584 57 us (96 with one unpipelined 16-token step
// at a time, 64 x 64 tiles and a grid over every possible tile), 64 of 27 x 27 x
// 2048 0.81 ms (1.07).
#include <algorithm>

#include "wz_ptx.cuh"
#include "wz_spatial.cuh"

namespace wz {

namespace {

constexpr int kSimtK = 32;            // tokens per step
constexpr int kSimtStages = 3;
constexpr int kSimtWRow = kSimtK + 4; // staged operator row: the rows of a warp's threads in different banks

template <typename Tin, int TM, int TN>
__host__ __device__ constexpr size_t simt_stage_bytes() {
    return (size_t)TM * kSimtWRow * 4 + (size_t)kSimtK * TN * sizeof(Tin);
}

__device__ __forceinline__ void cols4(const float *p, f2_t (&x)[2]) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    x[0] = pack2(v.x, v.y);
    x[1] = pack2(v.z, v.w);
}
__device__ __forceinline__ void cols4(const __nv_bfloat16 *p, f2_t (&x)[2]) {
    const uint2 v = *reinterpret_cast<const uint2 *>(p);
    x[0] = pack2(bf16_lo(v.x), bf16_hi(v.x));
    x[1] = pack2(bf16_lo(v.y), bf16_hi(v.y));
}
__device__ __forceinline__ void put4(float *p, float2 a, float2 b) {
    *reinterpret_cast<float4 *>(p) = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void put4(__nv_bfloat16 *p, float2 a, float2 b) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(a.x, a.y), hi = __floats2bfloat162_rn(b.x, b.y);
    *reinterpret_cast<uint2 *>(p) =
        make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
}

}  // namespace

// compact != 0 (at most kCompactFrames frames): the tiles that exist, through
// the prefix of the frames' row blocks; else every (frame, row block) pair.
template <typename Tin, int TM, int TN, int RT, int CG>   // a thread: RT rows x CG groups of 4 columns
__global__ void __launch_bounds__((TM / RT) * (TN / (4 * CG))) condense_simt_kernel(Ctx c, int compact) {
    constexpr int TX = TN / (4 * CG), TY = TM / RT, NT = TX * TY;
    extern __shared__ __align__(16) unsigned char ssm[];
    __shared__ int s_wsum[NT / 32];
    int *pre = reinterpret_cast<int *>(ssm + kSimtStages * simt_stage_bytes<Tin, TM, TN>());   // compact: [VT + 1]
    pdl_wait();
    pdl_trigger();
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    const int N = c.N, D = c.D, VT = c.V * c.T, KC = c.K_pad / kSimtK;
    if (compact) {
        frame_prefix<NT>(VT, pre, s_wsum, [&](int f) { return (max(c.n[f], 0) + TM - 1) / TM; });
        __syncthreads();
    }
    const int ncb = (D + TN - 1) / TN, nrb = (N + TM - 1) / TM;
    const int64_t items = (int64_t)(compact ? pre[VT] : (int64_t)VT * nrb) * ncb;
    for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const int64_t block = item / ncb;
        const int c0 = (int)(item - block * ncb) * TN;
        int f, rb;
        if (compact) {   // the last frame whose first row block is <= block
            int lo = 0, hi = VT - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (pre[mid] <= block) lo = mid;
                else hi = mid - 1;
            }
            f = lo;
            rb = (int)block - pre[f];
        } else {
            f = (int)(block / nrb);
            rb = (int)(block - (int64_t)f * nrb);
        }
        const int r0 = rb * TM, n = c.n[f] - r0;   // rows of the frame from r0
        if (n <= 0) continue;
        const int64_t orow = (int64_t)c.off[f] + r0;
        const float *Wr = static_cast<const float *>(c.Wop) + (size_t)orow * c.K_pad;
        const Tin *Xf = static_cast<const Tin *>(c.X) + (size_t)f * N * D + c0;
        __syncthreads();   // the previous tile's reads of the ring
        auto load = [&](int kc) {
            unsigned char *st = ssm + (kc % kSimtStages) * simt_stage_bytes<Tin, TM, TN>();
            float *ws = reinterpret_cast<float *>(st);
            Tin *xs = reinterpret_cast<Tin *>(st + (size_t)TM * kSimtWRow * 4);
            constexpr int WQ = kSimtK / 4;                 // 16-byte pieces of an operator row
            for (int k = tid; k < TM * WQ; k += NT) {
                const int r = k / WQ, q = (k % WQ) * 4;
                ptx::copy_async16(ws + r * kSimtWRow + q, Wr + (size_t)r * c.K_pad + kc * kSimtK + q, r < n);
            }
            constexpr int XE = 16 / (int)sizeof(Tin), XQ = TN / XE;   // pieces of a token row
            for (int k = tid; k < kSimtK * XQ; k += NT) {
                const int r = k / XQ, q = (k % XQ) * XE, tok = kc * kSimtK + r;
                ptx::copy_async16(xs + r * TN + q, Xf + (size_t)tok * D + q, tok < N && c0 + q < D);
            }
        };
        f2_t acc[RT][2 * CG];
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int j = 0; j < 2 * CG; ++j) acc[i][j] = 0ull;
#pragma unroll
        for (int s = 0; s < kSimtStages - 1; ++s) {
            if (s < KC) load(s);
            ptx::copy_async_commit();
        }
        for (int kc = 0; kc < KC; ++kc) {
            ptx::copy_async_wait<kSimtStages - 2>();
            __syncthreads();   // step kc has landed for every thread; step kc - 1 has been read
            if (kc + kSimtStages - 1 < KC) load(kc + kSimtStages - 1);
            ptx::copy_async_commit();
            const unsigned char *st = ssm + (kc % kSimtStages) * simt_stage_bytes<Tin, TM, TN>();
            const float *ws = reinterpret_cast<const float *>(st) + ty * kSimtWRow;
            const Tin *xs = reinterpret_cast<const Tin *>(st + (size_t)TM * kSimtWRow * 4) + tx * 4;
            const int klast = min(kSimtK, N - kc * kSimtK);   // the tokens past N are zeros
#pragma unroll 2
            for (int k4 = 0; k4 < klast; k4 += 4) {
                float4 w[RT];
#pragma unroll
                for (int i = 0; i < RT; ++i) w[i] = *reinterpret_cast<const float4 *>(ws + TY * i * kSimtWRow + k4);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    f2_t x[2 * CG];
#pragma unroll
                    for (int j = 0; j < CG; ++j) cols4(xs + (k4 + kk) * TN + 4 * TX * j, *reinterpret_cast<f2_t(*)[2]>(x + 2 * j));
#pragma unroll
                    for (int i = 0; i < RT; ++i) {
                        const float wv = kk == 0 ? w[i].x : kk == 1 ? w[i].y : kk == 2 ? w[i].z : w[i].w;
                        const f2_t wp = pack2(wv, wv);
#pragma unroll
                        for (int j = 0; j < 2 * CG; ++j) acc[i][j] = fma2(wp, x[j], acc[i][j]);
                    }
                }
            }
        }
        Tin *out = static_cast<Tin *>(c.out) + c0 + tx * 4;
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            const int r = ty + TY * i;
            if (r >= n || !wz_in_range(c.status, orow + r < c.rows_total)) continue;
#pragma unroll
            for (int j = 0; j < CG; ++j)
                if (c0 + tx * 4 + 4 * TX * j < D)   // D is a multiple of 8: no group straddles it
                    put4(out + (size_t)(orow + r) * D + 4 * TX * j, unpack2(acc[i][2 * j]), unpack2(acc[i][2 * j + 1]));
        }
    }
}

namespace {

template <typename Tin, int TM, int TN, int RT, int CG>
cudaError_t launch_simt(const Ctx &c, int sms, cudaStream_t s) {
    const void *fn = (const void *)condense_simt_kernel<Tin, TM, TN, RT, CG>;
    constexpr int threads = (TM / RT) * (TN / (4 * CG));
    const int64_t frames = (int64_t)c.V * c.T;
    int compact = frames <= kCompactFrames ? 1 : 0;
    const size_t smem = kSimtStages * simt_stage_bytes<Tin, TM, TN>() + (compact ? (size_t)(frames + 1) * 4 : 0);
    cudaError_t e = allow_smem(fn, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem)) != cudaSuccess) return e;
    // at most one partial row block per frame beside the full ones
    const int64_t all = frames * ((c.N + TM - 1) / TM);
    const int64_t blocks = compact ? std::min<int64_t>(all, c.rows_total / TM + frames) : all;
    const int64_t grid = std::min<int64_t>(blocks * ((c.D + TN - 1) / TN), (int64_t)sms * std::max(1, per_sm));
    void *args[] = {const_cast<Ctx *>(&c), &compact};
    return launch_kernel(fn, dim3((unsigned)grid), dim3(threads), smem, s, args, c.pdl != 0);
}

// Tile rows by the rows an average frame has (a frame's last tile is partly
// empty; about half of the frames have none, so the others have twice the
// average), tile columns by how many tiles there are.  Kernel times, 32 x 64 /
// 32 x 128 / 64 x 128 / 128 x 128 tiles: 64 frames of 13 x 13 x 3584, 17 rows:
// 57 / 61 / - / - us; 128 of 16 x 16 x 2048, 25 rows: - / 127 / 149 / 199; 32 of
// 27 x 27 x 3584, 73 rows: - / - / 354 / 411; 64 of 27 x 27 x 2048, 182 rows:
// - / - / 873 / 811 (43 TFLOP/s).  Up to 64 channels wider tiles are half empty:
// calls on 128 frames of 16 x 16 x 8, every token, 96 / 141 / 117 / 108.
template <typename Tin>
cudaError_t launch_simt_tiles(const Ctx &c, int sms, cudaStream_t s) {
    const int64_t rows = c.rows_total / ((int64_t)c.V * c.T), full = 2 * (int64_t)sms;
    auto tiles = [&](int tm, int tn) { return (c.rows_total + tm - 1) / tm * ((c.D + tn - 1) / tn); };
    if (c.D <= 64) return launch_simt<Tin, 32, 64, 4, 1>(c, sms, s);
    if (rows >= 128 && tiles(128, 128) >= full) return launch_simt<Tin, 128, 128, 8, 2>(c, sms, s);
    if (rows >= 48 && tiles(64, 128) >= full) return launch_simt<Tin, 64, 128, 8, 2>(c, sms, s);
    if (tiles(32, 128) >= 2 * full) return launch_simt<Tin, 32, 128, 4, 2>(c, sms, s);
    return launch_simt<Tin, 32, 64, 4, 1>(c, sms, s);
}

}  // namespace

cudaError_t launch_condense_simt(const Ctx &c, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    return c.dtype == WZ_DTYPE_BF16 ? launch_simt_tiles<__nv_bfloat16>(c, sms, s) : launch_simt_tiles<float>(c, sms, s);
}

}  // namespace wz
