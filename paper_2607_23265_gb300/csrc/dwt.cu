// Standalone single-level DWT / IDWT (Eq. 8, 10, 11, 14).
//
//   dwt1d   cA[i] = sum_j dec_lo[j] x^[2i+1-j], cD with dec_hi (x^ extended)
//   idwt1d  x[k]  = sum_i cA[i] rec_lo[k+F-2-2i] + cD[i] rec_hi[k+F-2-2i]
//   dwt2d   height axis then width axis per frame and channel; bands LL, LH,
//           HL, HH with the height filter first
//   idwt2d  width inverse then height inverse
//
// The 2D kernels take a frame's map for a chunk of CT channels through both
// separable passes, with the plane between them in shared memory.
#include <algorithm>
#include <initializer_list>

#include "wz_internal.cuh"
#include "wz_ptx.cuh"

namespace wz {

struct Taps {
    float lo[kMaxTaps], hi[kMaxTaps];
};

__global__ void dwt1d_kernel(const float *x, int rows, int L, int F, int mode, Taps t,
                             float *cA, float *cD) {
    const int Lo = (L + F - 1) / 2;
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (int64_t)rows * Lo) return;
    const int64_t r = id / Lo;
    const int i = (int)(id % Lo);
    const float *xr = x + r * L;
    float a = 0.f, d = 0.f;
    for (int j = 0; j < F; ++j) {
        const int s = ext_index(2 * i + 1 - j, L, mode);
        if (s < 0) continue;
        const float v = xr[s];
        a = fmaf(t.lo[j], v, a);
        d = fmaf(t.hi[j], v, d);
    }
    cA[id] = a;
    cD[id] = d;
}

__global__ void idwt1d_kernel(const float *cA, const float *cD, int rows, int L, int F, Taps t,
                              float *x) {
    const int Lo = (L + F - 1) / 2;
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (int64_t)rows * L) return;
    const int64_t r = id / L;
    const int k = (int)(id % L);
    float s = 0.f;
    const int ilo = max(0, (k - 1 + 1) / 2), ihi = min(Lo - 1, (k + F - 2) / 2);
    for (int i = ilo; i <= ihi; ++i) {
        const int tt = k + F - 2 - 2 * i;
        if (tt < 0 || tt >= F) continue;
        s = fmaf(t.lo[tt], cA[r * Lo + i], s);
        s = fmaf(t.hi[tt], cD[r * Lo + i], s);
    }
    x[id] = s;
}

// ---- 2D: one CTA per (frame, CT channels) ------------------------------------
//
// HBM bound: the forward reads the map once and writes four fp32 bands, the
// inverse the other way round.  Both passes slide a window of samples along
// one axis in registers, so every sample is read once per pass instead of once
// per tap; a thread owns a run along the axis for one channel pair (f32x2
// arithmetic), and the lanes of a warp take neighbouring channels.  The filter
// length is a template parameter: the window lives in registers at
// compile-time indices (F / 2 steps are unrolled and rotate it).  Forward and
// inverse of 32 frames of 27 x 27 x 3584 (bf16, db4; 1.56 GB, 230 us at the
// copy rate): 7.18 ms with one output per thread and every tap re-read from
// shared memory, 0.324 ms (4.8 TB/s) now, 0.160 + 0.163 ms; what is left is
// instruction issue in the forward (67 %) and the latency of the bands' loads
// in the inverse.  Measured and not taken: twice the channels per CTA with
// half the CTAs (354 us), smaller CTAs (427-448 us).

// One or two fp32 channels of a thread.
template <int VC> struct Lane;
template <> struct Lane<1> {
    typedef float V;
    static __device__ __forceinline__ V zero() { return 0.f; }
    static __device__ __forceinline__ V tap(float t) { return t; }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return fmaf(a, b, c); }
    static __device__ __forceinline__ V load(const float *p) { return *p; }
    static __device__ __forceinline__ V load(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void store(float *p, V v) { *p = v; }
};
template <> struct Lane<2> {
    typedef f2_t V;
    static __device__ __forceinline__ V zero() { return 0ull; }
    static __device__ __forceinline__ V tap(float t) { return pack2(t, t); }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return fma2(a, b, c); }
    static __device__ __forceinline__ V load(const float *p) {
        const float2 v = *reinterpret_cast<const float2 *>(p);
        return pack2(v.x, v.y);
    }
    static __device__ __forceinline__ V load(const __nv_bfloat16 *p) {
        const uint32_t w = *reinterpret_cast<const uint32_t *>(p);
        return pack2(bf16_lo(w), bf16_hi(w));
    }
    static __device__ __forceinline__ void store(float *p, V v) { *reinterpret_cast<float2 *>(p) = unpack2(v); }
};

// Offsets (in elements, `stride` per sample) of the samples that the extended
// positions 2 - F .. 2 nb - 1 of an axis copy, formed once per CTA; the zero
// extension copies sample n, which the caller keeps at zero.
__device__ __forceinline__ void extension_table(int *tab, int F, int n, int nb, int mode, int stride) {
    for (int k = threadIdx.x; k < 2 * nb + F - 2; k += blockDim.x) {
        const int s = ext_index(k + 2 - F, n, mode);
        tab[k] = (s < 0 ? n : s) * stride;
    }
}
constexpr int kExtMax = WZ_MAX_HW + 2 * kMaxTaps;   // >= 2 nb + F - 2 (nb <= (64 + F - 1) / 2)

// Analysis along one axis of n samples src[i * stride], extended through ext:
// r[q] = sum_j tap[q][j] x^[2b + 1 - j], j ascending, for NB filters, given to
// out for b = 0 .. nb - 1 in order.  Steps whose samples all lie inside the
// axis load them without the table.
template <int F, int VC, int NB, typename Tin, class Out>
__device__ __forceinline__ void analyse(const Tin *src, int stride, int n, const int *ext, int nb,
                                        const typename Lane<VC>::V (&tap)[NB][F], Out out) {
    typedef Lane<VC> L;
    typedef typename L::V V;
    // slot (-i) mod F holds x^[i]: step b overwrites the two oldest samples
    V win[F];
    auto step = [&](int u) {
        V r[NB];
#pragma unroll
        for (int q = 0; q < NB; ++q) r[q] = L::zero();
#pragma unroll
        for (int j = 0; j < F; ++j)
#pragma unroll
            for (int q = 0; q < NB; ++q)   // x^[2(b0 + u) + 1 - j]
                r[q] = L::fma(tap[q][j], win[(2 * F - 2 * u - 1 + j) % F], r[q]);
        out(r);
    };
#pragma unroll
    for (int k = 2; k < F; ++k) win[k - 1] = L::load(src + ext[F - 1 - k]);   // x^[1 - k]
    int b0 = 0;
    for (const Tin *p = src; 2 * b0 + F <= n; b0 += F / 2) {   // b0 + F/2 <= n/2 <= nb
#pragma unroll
        for (int u = 0; u < F / 2; ++u) {
            win[(2 * F - 2 * u) % F] = L::load(p);
            p += stride;
            win[(2 * F - 2 * u - 1) % F] = L::load(p);
            p += stride;
            step(u);
        }
    }
    for (; b0 < nb; b0 += F / 2)
#pragma unroll
        for (int u = 0; u < F / 2; ++u)
            if (b0 + u < nb) {
                win[(2 * F - 2 * u) % F] = L::load(src + ext[2 * (b0 + u) + F - 2]);
                win[(2 * F - 2 * u - 1) % F] = L::load(src + ext[2 * (b0 + u) + F - 1]);
                step(u);
            }
}

// Synthesis along one axis: x[k] = sum_i A[i] rec_lo[k + F - 2 - 2i] +
// D[i] rec_hi[k + F - 2 - 2i], i ascending, given to out for k = 0 .. n - 1 in
// order, from nb coefficients of each band at a[i * stride], d[i * stride].
// Samples 2m and 2m + 1 both take the coefficients m .. m + F/2 - 1, which
// slide through registers (all of them exist where sample 2m does: nb >=
// (n + F - 2) / 2).  The coefficients of G steps are loaded together.
template <int F, int VC, class Out>
__device__ __forceinline__ void synthesise(const float *a, const float *d, int64_t stride, int n, int nb, const Taps &t,
                                           Out out) {
    typedef Lane<VC> L;
    typedef typename L::V V;
    constexpr int G = F / 2;
    V tl[F], th[F];
#pragma unroll
    for (int j = 0; j < F; ++j) {
        tl[j] = L::tap(t.lo[j]);
        th[j] = L::tap(t.hi[j]);
    }
    V wa[G], wd[G];   // slot i mod G holds coefficient i
    auto next = [&](V &x, V &y) {
        x = L::load(a);
        y = L::load(d);
        a += stride;
        d += stride;
    };
    auto step = [&](int u, const V &ca, const V &cd, bool two) {
        wa[(u + G - 1) % G] = ca;
        wd[(u + G - 1) % G] = cd;
        V x0 = L::zero(), x1 = L::zero();
#pragma unroll
        for (int i = 0; i < G; ++i) {
            x0 = L::fma(tl[F - 2 - 2 * i], wa[(u + i) % G], x0);
            x0 = L::fma(th[F - 2 - 2 * i], wd[(u + i) % G], x0);
            x1 = L::fma(tl[F - 1 - 2 * i], wa[(u + i) % G], x1);
            x1 = L::fma(th[F - 1 - 2 * i], wd[(u + i) % G], x1);
        }
        out(x0);
        if (two) out(x1);
    };
#pragma unroll
    for (int i = 0; i < G - 1; ++i) next(wa[i], wd[i]);
    int k = 0;
    for (; k + F <= n; k += F) {
        V na[G], nd[G];
#pragma unroll
        for (int u = 0; u < G; ++u) next(na[u], nd[u]);
#pragma unroll
        for (int u = 0; u < G; ++u) step(u, na[u], nd[u], true);
    }
#pragma unroll
    for (int u = 0; u < G; ++u)
        if (k + 2 * u < n) {
            V ca, cd;
            next(ca, cd);
            step(u, ca, cd, k + 2 * u + 1 < n);
        }
}

constexpr int kDwtThreads = 256, kIdwtThreads = 320;

// CTAs per SM that the registers are held to (the taps and the window of a
// pair take 4F to 6F of them).
constexpr int dwt_ctas(int F) { return F <= 10 ? 3 : F <= 14 ? 2 : 1; }

// A row of at least `n` positions in shared memory: an odd number, so that the
// rows that a warp's lanes work on start in different banks (CT = 16).
__host__ __device__ __forceinline__ int dwt_row(int n) { return n | 1; }

// The CTA's map goes to shared memory in one go (every read in flight at
// once; cp.async where `vec` says that 16-byte pieces are aligned), then for
// the width-low and the width-high half: width pass of every row into the
// plane, height pass of every plane column into the two bands.  One half at a
// time keeps the plane small enough for several CTAs per SM.
template <typename Tin, int F, int VC>
__global__ void __launch_bounds__(kDwtThreads, dwt_ctas(F))
dwt2d_kernel(const Tin *X, int H, int W, int D, int CT, int mode, int vec, Taps t, float *LL, float *LH, float *HL,
             float *HH) {
    typedef Lane<VC> L;
    typedef typename L::V V;
    // plane [H + 1][row(wp)][CT], then the map [H][row(W + 1)][CT]; the extra
    // row and column are the zero extension's sample
    extern __shared__ __align__(16) float pl[];
    __shared__ int ext_w[kExtMax], ext_h[kExtMax];
    const int hp = (H + F - 1) / 2, wp = (W + F - 1) / 2;
    const int ws = dwt_row(W + 1), ps = dwt_row(wp);
    Tin *sx = reinterpret_cast<Tin *>(pl + (H + 1) * ps * CT);
    const int64_t fr = blockIdx.y;
    const int c0 = blockIdx.x * CT;
    const int nc = min(CT, D - c0);                 // channels of this CTA
    const int G = CT / VC;                          // channel groups
    const Tin *Xf = X + (size_t)fr * H * W * D + c0;
    if (vec) {
        const int nv = nc * (int)sizeof(Tin) / 16, ve = 16 / (int)sizeof(Tin);
        for (int k = threadIdx.x; k < H * W * nv; k += blockDim.x) {
            const int p = k / nv, q = (k - p * nv) * ve, i = p / W;
            ptx::copy_async16(sx + (i * ws + p - i * W) * CT + q, Xf + (size_t)p * D + q);
        }
        ptx::copy_async_wait_all();
    } else {
        for (int k = threadIdx.x; k < H * W * nc; k += blockDim.x) {
            const int p = k / nc, q = k - p * nc, i = p / W;
            sx[(i * ws + p - i * W) * CT + q] = Xf[(size_t)p * D + q];
        }
    }
    extension_table(ext_w, F, W, wp, mode, CT);
    extension_table(ext_h, F, H, hp, mode, ps * CT);
    if (mode == WZ_MODE_ZERO) {
        for (int k = threadIdx.x; k < wp * CT; k += blockDim.x) pl[H * ps * CT + k] = 0.f;
        for (int k = threadIdx.x; k < H * CT; k += blockDim.x)
            sx[(k / CT * ws + W) * CT + k % CT] = from_float<Tin>(0.f);
    }
    for (int v = 0; v < 2; ++v) {
        __syncthreads();   // the map and the tables; the plane's readers of the other half
        {
            V tap[1][F];
#pragma unroll
            for (int j = 0; j < F; ++j) tap[0][j] = L::tap(v ? t.hi[j] : t.lo[j]);
            for (int k = threadIdx.x; k < H * G; k += blockDim.x) {
                const int i = k / G, cc = (k - i * G) * VC;
                if (cc >= nc) continue;
                float *row = pl + i * ps * CT + cc;
                analyse<F, VC, 1>((const Tin *)(sx + i * ws * CT + cc), CT, W, ext_w, wp, tap, [&](V(&r)[1]) {
                    L::store(row, r[0]);
                    row += CT;
                });
            }
        }
        __syncthreads();
        V tap[2][F];
#pragma unroll
        for (int j = 0; j < F; ++j) {
            tap[0][j] = L::tap(t.lo[j]);
            tap[1][j] = L::tap(t.hi[j]);
        }
        float *Bl = v ? LH : LL, *Bh = v ? HH : HL;
        for (int k = threadIdx.x; k < wp * G; k += blockDim.x) {
            const int b = k / G, cc = (k - b * G) * VC;
            if (cc >= nc) continue;
            const size_t o = ((size_t)fr * hp * wp + b) * D + c0 + cc, line = (size_t)wp * D;
            float *pa = Bl + o, *pb = Bh + o;
            analyse<F, VC, 2>((const float *)(pl + b * CT + cc), ps * CT, H, ext_h, hp, tap, [&](V(&r)[2]) {
                L::store(pa, r[0]);
                L::store(pb, r[1]);
                pa += line;
                pb += line;
            });
        }
    }
}

// Height inverse of every band column into the plane (rows y of the width-low
// and width-high halves), then width inverse of every row into the output.
template <int F, int VC>
__global__ void __launch_bounds__(kIdwtThreads, dwt_ctas(F))
idwt2d_kernel(const float *LL, const float *LH, const float *HL, const float *HH, int H, int W, int D, int CT, Taps t,
              float *out) {
    typedef Lane<VC> L;
    typedef typename L::V V;
    extern __shared__ __align__(16) float sr[];   // [H][row(2 wp)][CT]: width-low, then width-high
    const int hp = (H + F - 1) / 2, wp = (W + F - 1) / 2, ps = dwt_row(2 * wp);
    const int64_t fr = blockIdx.y;
    const int c0 = blockIdx.x * CT;
    const int G = CT / VC;
    // every band sector of the CTA on its way to L2 at once: the sliding loads
    // below keep too few in flight per thread (332 -> 324 us for the pair)
    const int nc = min(CT, D - c0);
    for (int k = threadIdx.x; k < 4 * hp * wp; k += blockDim.x) {
        const float *band = k & 2 ? (k & 1 ? HH : HL) : (k & 1 ? LH : LL);
        const float *p = band + ((size_t)fr * hp * wp + (k >> 2)) * D + c0;
        for (int q = 0; q < nc; q += 8) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + q));
    }
    for (int k = threadIdx.x; k < 2 * wp * G; k += blockDim.x) {
        const int vb = k / G, cc = (k - vb * G) * VC;
        if (c0 + cc >= D) continue;
        const int v = vb >= wp ? 1 : 0, b = vb - v * wp;
        const size_t o = ((size_t)fr * hp * wp + b) * D + c0 + cc;
        float *col = sr + vb * CT + cc;
        synthesise<F, VC>((v ? LH : LL) + o, (v ? HH : HL) + o, (int64_t)wp * D, H, hp, t,
                          [&](V x) {
                              L::store(col, x);
                              col += ps * CT;
                          });
    }
    __syncthreads();
    for (int k = threadIdx.x; k < H * G; k += blockDim.x) {
        const int y = k / G, cc = (k - y * G) * VC;
        if (c0 + cc >= D) continue;
        const float *row = sr + y * ps * CT + cc;
        float *o = out + ((size_t)fr * H + y) * W * D + c0 + cc;
        synthesise<F, VC>(row, row + wp * CT, CT, W, wp, t, [&](V x) {
            L::store(o, x);
            o += D;
        });
    }
}

namespace {

Taps make_taps(const float *lo, const float *hi, int F) {
    Taps t{};
    for (int k = 0; k < F; ++k) {
        t.lo[k] = lo[k];
        t.hi[k] = hi[k];
    }
    return t;
}

// Launch shape of the 2D kernels: CT channels per CTA (the most of 64, 32, 16
// whose shared memory is at most 72 KB, so that three CTAs share an SM, whose
// longer pass is at most one round of the CTA's threads, and which D fills to more
// than a half; else 8, which fits at the largest map and filter), one thread per
// run of that pass.
struct DwtCfg {
    int ct, threads;
    size_t smem;
};

DwtCfg dwt_config(size_t bytes_per_channel, int runs_per_channel, int D, int vc, int max_threads) {
    int ct = 64;
    while (ct > 8 && 2 * D <= ct) ct >>= 1;
    while (ct > 8 && (bytes_per_channel * ct > 72 * 1024 || runs_per_channel * ct / vc > max_threads)) ct >>= 1;
    return {ct, std::min(max_threads, (runs_per_channel * ct / vc + 31) / 32 * 32), bytes_per_channel * ct};
}

// Channel pairs need an even D and rows aligned for two elements.
bool pair_ok(int D, std::initializer_list<const void *> fp32, const void *x, size_t esz) {
    for (const void *p : fp32)
        if ((uintptr_t)p % 8 != 0) return false;
    return D % 2 == 0 && (uintptr_t)x % (2 * esz) == 0;
}

template <typename Tin, int F>
const void *dwt2d_fn(int vc) {
    return vc == 2 ? (const void *)dwt2d_kernel<Tin, F, 2> : (const void *)dwt2d_kernel<Tin, F, 1>;
}
template <int F>
const void *idwt2d_fn(int vc) {
    return vc == 2 ? (const void *)idwt2d_kernel<F, 2> : (const void *)idwt2d_kernel<F, 1>;
}

#define WZ_BY_TAPS(F, X)      \
    switch (F) {              \
        case 2: X(2);         \
        case 4: X(4);         \
        case 6: X(6);         \
        case 8: X(8);         \
        case 10: X(10);       \
        case 12: X(12);       \
        case 14: X(14);       \
        case 16: X(16);       \
        case 18: X(18);       \
        case 20: X(20);       \
        default: return nullptr; \
    }

template <typename Tin>
const void *pick_dwt2d(int F, int vc) {
#define WZ_CASE(N) return dwt2d_fn<Tin, N>(vc)
    WZ_BY_TAPS(F, WZ_CASE)
#undef WZ_CASE
}
const void *pick_idwt2d(int F, int vc) {
#define WZ_CASE(N) return idwt2d_fn<N>(vc)
    WZ_BY_TAPS(F, WZ_CASE)
#undef WZ_CASE
}

}  // namespace

cudaError_t launch_dwt1d(const float *x, int rows, int L, int F, int mode, const float *dlo,
                         const float *dhi, float *cA, float *cD, cudaStream_t s) {
    const int64_t n = (int64_t)rows * ((L + F - 1) / 2);
    if (n == 0) return cudaSuccess;
    dwt1d_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(x, rows, L, F, mode, make_taps(dlo, dhi, F), cA, cD);
    return cudaGetLastError();
}

cudaError_t launch_idwt1d(const float *cA, const float *cD, int rows, int L, int F,
                          const float *rlo, const float *rhi, float *x, cudaStream_t s) {
    const int64_t n = (int64_t)rows * L;
    if (n == 0) return cudaSuccess;
    idwt1d_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(cA, cD, rows, L, F, make_taps(rlo, rhi, F), x);
    return cudaGetLastError();
}

cudaError_t launch_dwt2d(const void *X, int dtype, int T, int H, int W, int D, int F, int mode,
                         const float *dlo, const float *dhi, float *LL, float *LH, float *HL,
                         float *HH, cudaStream_t s) {
    const bool bf = dtype == WZ_DTYPE_BF16;
    const int vc = pair_ok(D, {LL, LH, HL, HH}, X, bf ? 2 : 4) ? 2 : 1;
    const int wp = (W + F - 1) / 2;
    const size_t esz = bf ? 2 : 4;
    const DwtCfg k = dwt_config((size_t)(H + 1) * dwt_row(wp) * 4 + (size_t)H * dwt_row(W + 1) * esz, std::max(H, wp), D, vc,
                                kDwtThreads);
    int vec = ((uintptr_t)X % 16 == 0 && (size_t)D * esz % 16 == 0) ? 1 : 0;
    const void *fn = bf ? pick_dwt2d<__nv_bfloat16>(F, vc) : pick_dwt2d<float>(F, vc);
    if (!fn) return cudaErrorInvalidValue;
    const cudaError_t e = allow_smem(fn, k.smem);
    if (e != cudaSuccess) return e;
    Taps t = make_taps(dlo, dhi, F);
    int ct = k.ct;
    void *args[] = {&X, &H, &W, &D, &ct, &mode, &vec, &t, &LL, &LH, &HL, &HH};
    return launch_kernel(fn, dim3((unsigned)((D + ct - 1) / ct), (unsigned)T), dim3(k.threads), k.smem, s, args, false);
}

cudaError_t launch_idwt2d(const float *LL, const float *LH, const float *HL, const float *HH,
                          int T, int H, int W, int D, int F, const float *rlo, const float *rhi,
                          float *out, cudaStream_t s) {
    const int vc = pair_ok(D, {LL, LH, HL, HH, out}, nullptr, 4) ? 2 : 1;
    const int wp = (W + F - 1) / 2;
    const DwtCfg k = dwt_config((size_t)H * dwt_row(2 * wp) * 4, std::max(H, 2 * wp), D, vc, kIdwtThreads);
    const void *fn = pick_idwt2d(F, vc);
    if (!fn) return cudaErrorInvalidValue;
    const cudaError_t e = allow_smem(fn, k.smem);
    if (e != cudaSuccess) return e;
    Taps t = make_taps(rlo, rhi, F);
    int ct = k.ct;
    void *args[] = {&LL, &LH, &HL, &HH, &H, &W, &D, &ct, &t, &out};
    return launch_kernel(fn, dim3((unsigned)((D + ct - 1) / ct), (unsigned)T), dim3(k.threads), k.smem, s, args, false);
}

}  // namespace wz
