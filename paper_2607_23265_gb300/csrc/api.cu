// C ABI of the WaveZip library: argument checks, workspace layout and the
// launch sequence of the condensation pass (Section 3.2).
//
//   query_pool -> relevance_pass -> frame_stats -> temporal -> spatial ->
//   condense (tensor cores or CUDA cores)
//
// All launches go to the caller's stream; nothing synchronises the host.
// A call with a caller-owned workspace and no profiling events is captured
// once into a CUDA graph, keyed by every argument, and replayed on later
// calls with the same arguments (the replay cache below).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <list>
#include <mutex>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "wz_spatial.cuh"

namespace wz {

size_t spatial_smem_bytes(const Ctx &c);
bool tensor_path_available();

namespace {

constexpr size_t kAlign = 256;

size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

bool aligned(const void *p, size_t a) { return ((uintptr_t)p % a) == 0; }

// NVTX range around a host-side launch (a no-op unless a profiler listens).
struct Nvtx {
    explicit Nvtx(const char *name) { nvtxRangePushA(name); }
    ~Nvtx() { nvtxRangePop(); }
};

// Sub-buffer offsets of one call's workspace.
struct Layout {
    size_t qbar32, qbar64, vpar, a, part, fr, list, n, off, woff, hw, prod,
        units, ucount, ustart, ustartB, stab, drange, gate, krange, qnorm, qhl, status, snext, Wop, total;
};

struct Shape {
    int V, T, H, W, D, N, dtype, F, hp, wp, K_pad, n_ct, max_units_v;
    int64_t rows_total, w_rows;
};

Layout make_layout(const Shape &s, bool with_a, bool with_operator) {
    Layout L{};
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o = align_up(o + bytes);
        return at;
    };
    const size_t VT = (size_t)s.V * s.T;
    L.qbar32 = take((size_t)s.V * s.D * 4);
    L.qbar64 = take((size_t)s.V * s.D * 8);
    L.vpar = take((size_t)s.V * sizeof(VideoPar));
    L.a = with_a ? take(VT * s.N * 4) : 0;
    L.part = take(((size_t)kG1Max + VT) * s.D * 4);
    L.fr = take(VT * 4 * 8);
    L.list = take(VT * 2 * 4);
    L.n = take(VT * 4);
    L.off = take(VT * 4);
    L.woff = take(VT * 4);
    L.hw = take(VT * 2 * 4);
    L.prod = take((size_t)s.V * 4);
    L.units = take((size_t)s.V * s.max_units_v * 16);
    L.ucount = take((size_t)s.V * 4);
    L.ustart = take(VT * 4);
    L.ustartB = take(VT * 4);
    L.stab = take(std::max(spatial_table_bytes(s.H, s.W, kMaxTaps),            // any wavelet,
                           ml_table_bytes(s.H, s.W, kMaxTaps, kMaxLevels)));   // any level count
    L.drange = take((size_t)s.V * 16);
    L.qnorm = take((size_t)s.V * WZ_MAX_LQ_MAXSIM * 4);
    L.qhl = take((size_t)2 * WZ_MAX_LQ_MAXSIM * s.D * 2);
    L.gate = with_operator ? take(VT * (size_t)gate_floats(s.H, s.W, kMaxTaps, kMaxLevels) * 4) : 0;
    L.krange = with_operator ? take(VT * (size_t)((s.N + kColBlock - 1) / kColBlock) * (s.K_pad / 32) * 2) : 0;
    L.status = take(16);
    L.snext = take(16);
    L.Wop = with_operator ? take((size_t)std::max<int64_t>(s.rows_total, s.w_rows) * s.K_pad * 4) : 0;
    L.total = o;
    return L;
}

bool valid_ratio(float r) { return std::isfinite(r) && r > 0.f && r <= 1.f; }

int64_t budget(int T, int N, float ratio) {
    const double x = (double)ratio * (double)T * (double)N;   // exact: 24 + 12 + 12 bits
    return (int64_t)std::floor(x + 0.5);
}

int check_sizes(int V, int T, int H, int W, int D, int dtype) {
    if (V < 1 || T < 1 || H < 1 || W < 1 || D < 1) return WZ_ERR_INVALID_ARG;
    if (dtype != WZ_DTYPE_BF16 && dtype != WZ_DTYPE_F32) return WZ_ERR_INVALID_ARG;
    if (D % 8 != 0) return WZ_ERR_UNSUPPORTED;
    if (V > WZ_MAX_VIDEOS || T > WZ_MAX_T || H > WZ_MAX_HW || W > WZ_MAX_HW || D > WZ_MAX_D)
        return WZ_ERR_UNSUPPORTED;
    if (dtype == WZ_DTYPE_F32 && D > WZ_MAX_D / 2) return WZ_ERR_UNSUPPORTED;
    return WZ_OK;
}

// Tensor-core operator rows reserved for one video: every frame's block
// starts on a multiple of 16, so round16(B) + 16 T rows always suffice.
int64_t video_w_rows(int64_t B, int T) { return (B + 15) / 16 * 16 + (int64_t)16 * T; }

Shape make_shape(int V, int T, int H, int W, int D, int dtype, int F, const int64_t *B) {
    Shape s{};
    s.V = V; s.T = T; s.H = H; s.W = W; s.D = D; s.N = H * W; s.dtype = dtype; s.F = F;
    s.hp = (H + F - 1) / 2;
    s.wp = (W + F - 1) / 2;
    s.K_pad = (s.N + 31) / 32 * 32;
    s.n_ct = (D + kTileC - 1) / kTileC;
    int64_t rows = 0, bmax = 0, wrows = 0;
    for (int v = 0; v < V; ++v) {
        const int64_t b = B ? B[v] : 0;
        rows += b;
        wrows += video_w_rows(b, T);
        bmax = std::max<int64_t>(bmax, b);
    }
    s.rows_total = rows;
    s.w_rows = wrows;
    s.max_units_v = (int)((T + (bmax + kColBlock - 1) / kColBlock) * s.n_ct);
    return s;
}

struct Common {
    float lambda, tau;
    int wta_wavelet, wsm_wavelet, mode, path, temporal_mode, spatial_mode;
    int relevance_mode = WZ_RELEVANCE_MEAN;
    int wta_levels = 1, wsm_levels = 1;
};

int check_common(const Common &m, int dtype) {
    if (!std::isfinite(m.lambda) || m.lambda < 0.f || !std::isfinite(m.tau)) return WZ_ERR_INVALID_ARG;
    if (wavelet_taps(m.wta_wavelet) == 0 || wavelet_taps(m.wsm_wavelet) == 0) return WZ_ERR_INVALID_ARG;
    if (m.mode < WZ_MODE_SYMMETRIC || m.mode > WZ_MODE_PERIODIC) return WZ_ERR_INVALID_ARG;
    if (m.path < WZ_PATH_AUTO || m.path > WZ_PATH_SIMT) return WZ_ERR_INVALID_ARG;
    if (m.path == WZ_PATH_TENSOR && dtype != WZ_DTYPE_BF16) return WZ_ERR_UNSUPPORTED;
    if (m.temporal_mode < WZ_TEMPORAL_WTA || m.temporal_mode > WZ_TEMPORAL_UNIFORM) return WZ_ERR_INVALID_ARG;
    if (m.spatial_mode < WZ_SPATIAL_WSM || m.spatial_mode > WZ_SPATIAL_NONE) return WZ_ERR_INVALID_ARG;
    if (m.wta_levels < 1 || m.wta_levels > kMaxLevels || m.wsm_levels < 1 || m.wsm_levels > kMaxLevels)
        return WZ_ERR_INVALID_ARG;
    return WZ_OK;
}

int resolve_path(int path, int dtype) {
    if (path != WZ_PATH_AUTO) return path;
    return (dtype == WZ_DTYPE_BF16 && tensor_path_available()) ? WZ_PATH_TENSOR : WZ_PATH_SIMT;
}

void set_filters(Ctx &c, int p) {
    double dl[kMaxTaps], dh[kMaxTaps], rl[kMaxTaps], rh[kMaxTaps];
    wavelet_bank(p, dl, dh, rl, rh);
    c.F = wavelet_taps(p);
    for (int k = 0; k < kMaxTaps; ++k) {
        c.dec_lo[k] = k < c.F ? (float)dl[k] : 0.f;
        c.dec_hi[k] = k < c.F ? (float)dh[k] : 0.f;
        c.rec_lo[k] = k < c.F ? (float)rl[k] : 0.f;
        c.rec_hi[k] = k < c.F ? (float)rh[k] : 0.f;
    }
}

void set_wta_filters(Ctx &c, int p) {
    double dl[kMaxTaps], dh[kMaxTaps], rl[kMaxTaps], rh[kMaxTaps];
    wavelet_bank(p, dl, dh, rl, rh);
    c.wta_F = wavelet_taps(p);
    for (int k = 0; k < kMaxTaps; ++k) {
        c.wta_dec_lo[k] = k < c.wta_F ? dl[k] : 0.0;
        c.wta_dec_hi[k] = k < c.wta_F ? dh[k] : 0.0;
        c.wta_rec_lo[k] = k < c.wta_F ? rl[k] : 0.0;
        c.wta_rec_hi[k] = k < c.wta_F ? rh[k] : 0.0;
    }
}

// Level counts and the WSM subband grids of every level (c.F set).
void set_levels(Ctx &c, int H, int W, int wta_levels, int wsm_levels) {
    c.wta_levels = wta_levels;
    c.wsm_levels = wsm_levels;
    int off = 0;
    for (int l = 0; l <= kMaxLevels; ++l) {
        c.lvl_h[l] = level_size(H, c.F, l);
        c.lvl_w[l] = level_size(W, c.F, l);
        if (l >= 1) {
            c.goff[l - 1] = off;
            if (l <= wsm_levels) off += c.lvl_h[l] * c.lvl_w[l];
        }
    }
    c.gate_stride = off;
}

void bind(Ctx &c, const Shape &s, const Layout &L, char *ws) {
    c.V = s.V; c.T = s.T; c.H = s.H; c.W = s.W; c.D = s.D; c.N = s.N; c.dtype = s.dtype;
    c.hp = s.hp; c.wp = s.wp; c.K_pad = s.K_pad; c.n_ct = s.n_ct;
    c.max_units_v = s.max_units_v; c.rows_total = s.rows_total; c.w_rows = s.w_rows;
    c.qbar32 = reinterpret_cast<float *>(ws + L.qbar32);
    c.qbar64 = reinterpret_cast<double *>(ws + L.qbar64);
    c.vpar = reinterpret_cast<VideoPar *>(ws + L.vpar);
    if (L.a) c.a = reinterpret_cast<float *>(ws + L.a);
    c.part = reinterpret_cast<float *>(ws + L.part);
    c.fr = reinterpret_cast<double *>(ws + L.fr);
    c.list = reinterpret_cast<int *>(ws + L.list);
    c.n = reinterpret_cast<int *>(ws + L.n);
    c.off = reinterpret_cast<int *>(ws + L.off);
    c.woff = reinterpret_cast<int *>(ws + L.woff);
    c.hw = reinterpret_cast<int *>(ws + L.hw);
    c.prod = reinterpret_cast<int *>(ws + L.prod);
    c.units = reinterpret_cast<int4 *>(ws + L.units);
    c.ucount = reinterpret_cast<int *>(ws + L.ucount);
    c.ustart = reinterpret_cast<int *>(ws + L.ustart);
    c.ustartB = reinterpret_cast<int *>(ws + L.ustartB);
    c.stab = reinterpret_cast<float *>(ws + L.stab);
    c.drange = reinterpret_cast<unsigned long long *>(ws + L.drange);
    c.qnorm = reinterpret_cast<float *>(ws + L.qnorm);
    c.qhl = reinterpret_cast<__nv_bfloat16 *>(ws + L.qhl);
    c.gate = L.gate ? reinterpret_cast<float *>(ws + L.gate) : nullptr;
    c.status = reinterpret_cast<int *>(ws + L.status);
    c.spatial_next = reinterpret_cast<int *>(ws + L.snext);
    if (L.Wop) c.Wop = ws + L.Wop;
    if (L.krange) {
        c.krange = reinterpret_cast<uint16_t *>(ws + L.krange);
        c.krange_nblk = (s.N + kColBlock - 1) / kColBlock;
    }
}

// Scratch either from the caller or from the stream-ordered allocator.
struct Scratch {
    char *ptr = nullptr;
    bool owned = false;
    cudaStream_t stream = nullptr;
    int acquire(void *given, size_t given_bytes, size_t need, cudaStream_t s) {
        stream = s;
        if (given) {
            if (!aligned(given, kAlign)) return WZ_ERR_INVALID_ARG;
            if (given_bytes < need) return WZ_ERR_WORKSPACE;
            ptr = static_cast<char *>(given);
            return WZ_OK;
        }
        void *p = nullptr;
        if (cudaMallocAsync(&p, need, s) != cudaSuccess) {
            cudaGetLastError();
            return WZ_ERR_NO_MEMORY;
        }
        ptr = static_cast<char *>(p);
        owned = true;
        return WZ_OK;
    }
    ~Scratch() {
        if (owned) cudaFreeAsync(ptr, stream);
    }
};

#define WZ_CUDA(call)                        \
    do {                                     \
        if ((call) != cudaSuccess) {         \
            cudaGetLastError();              \
            return WZ_ERR_CUDA;              \
        }                                    \
    } while (0)

struct CondenseRequest {
    int V, T, H, W, D, dtype;
    const void *features, *queries;
    std::vector<int> Lq;
    std::vector<float> ratio;
    Common m;
    const float *token_scores = nullptr, *frame_scores = nullptr;
    void *out_tokens;
    int32_t *out_index, *out_budgets, *out_count, *device_status;
    float *out_relevance;
    void *workspace;
    size_t workspace_bytes;
    void *const *events;
    cudaStream_t stream;
};

int validate(const CondenseRequest &r, std::vector<int64_t> &B, int64_t &rows) {
    int st = check_sizes(r.V, r.T, r.H, r.W, r.D, r.dtype);
    if (st != WZ_OK) return st;
    st = check_common(r.m, r.dtype);
    if (st != WZ_OK) return st;
    if (!r.features || !r.queries) return WZ_ERR_INVALID_ARG;
    if (!aligned(r.features, 16) || !aligned(r.queries, 16)) return WZ_ERR_INVALID_ARG;
    if (!aligned(r.token_scores, 4) || !aligned(r.frame_scores, 4)) return WZ_ERR_INVALID_ARG;
    if (r.m.relevance_mode != WZ_RELEVANCE_MEAN && r.m.relevance_mode != WZ_RELEVANCE_MAXSIM) return WZ_ERR_INVALID_ARG;
    if (r.m.wsm_levels > 1 && r.m.spatial_mode == WZ_SPATIAL_WSM &&
        spatial_ml_smem_bytes(r.H, r.W, wavelet_taps(r.m.wsm_wavelet), r.m.wsm_levels) == 0)
        return WZ_ERR_UNSUPPORTED;   // the multi-level tables of this map do not fit one CTA
    if (r.m.relevance_mode == WZ_RELEVANCE_MAXSIM) {
        if (r.dtype != WZ_DTYPE_BF16 || r.D % 64 != 0) return WZ_ERR_UNSUPPORTED;
        for (int v = 0; v < r.V; ++v)
            if (r.Lq[v] > WZ_MAX_LQ_MAXSIM) return WZ_ERR_UNSUPPORTED;
    }
    B.assign(r.V, 0);
    rows = 0;
    int64_t qrows = 0;
    for (int v = 0; v < r.V; ++v) {
        if (r.Lq[v] < 1 || !valid_ratio(r.ratio[v])) return WZ_ERR_INVALID_ARG;
        B[v] = budget(r.T, r.H * r.W, r.ratio[v]);
        rows += B[v];
        qrows += r.Lq[v];
    }
    if (rows + (int64_t)16 * r.V * r.T > (int64_t)INT32_MAX || qrows > (int64_t)INT32_MAX) return WZ_ERR_UNSUPPORTED;
    if (rows > 0) {
        if (!r.out_tokens || !r.out_index) return WZ_ERR_INVALID_ARG;
        if (!aligned(r.out_tokens, 16) || !aligned(r.out_index, 4)) return WZ_ERR_INVALID_ARG;
    }
    return WZ_OK;
}

// Where the unit query rows of a call with the max-over-query scorer go.  The
// one pass over the features (token norms, channel sums, token x query-row
// maxima) wants those of all videos at once: in their own buffer, in the partial
// slots past the ones in use, or in the operator's memory, which the spatial
// kernel writes later.  Without room, or where the pass does not apply, the
// scorer runs video by video through the own buffer.
enum class QueryRows { kByVideo, kOwn, kSlots, kOperator };

// Lqp: the longest query, padded to 16; qrows: the rows of all videos (qhl_row).
// *at: their offset in the workspace (kSlots, kOperator).
QueryRows place_query_rows(const Ctx &c, const Shape &s, const Layout &L, int Lqp, int64_t qrows, size_t *at) {
    if (!maxsim_pass_supported(c, Lqp)) return QueryRows::kByVideo;
    const size_t need = (size_t)qrows * s.D * 2;
    if (need <= (size_t)2 * WZ_MAX_LQ_MAXSIM * s.D * 2) return QueryRows::kOwn;
    *at = L.part + align_up(((size_t)c.G1 + (size_t)s.V * s.T) * s.D * 4);
    if (*at + need <= L.fr) return QueryRows::kSlots;
    *at = L.Wop;
    return *at + need <= L.total ? QueryRows::kOperator : QueryRows::kByVideo;
}

int run_condense(const CondenseRequest &r) {
    std::vector<int64_t> B;
    int64_t rows = 0;
    int st = validate(r, B, rows);
    if (st != WZ_OK) return st;
    Ctx c{};
    c.lambda = r.m.lambda;
    c.tau = r.m.tau;
    c.mode = r.m.mode;
    c.path = resolve_path(r.m.path, r.dtype);
    c.temporal_mode = r.m.temporal_mode;
    c.spatial_mode = r.m.spatial_mode;
    c.ext_a = r.token_scores;
    c.ext_r = r.frame_scores;
    c.relevance_mode = r.m.relevance_mode;
    c.pdl = r.events ? 0 : 1;      // an event between two kernels would break the overlap
    set_filters(c, r.m.wsm_wavelet);
    set_wta_filters(c, r.m.wta_wavelet);
    set_levels(c, r.H, r.W, r.m.wta_levels, r.m.spatial_mode == WZ_SPATIAL_WSM ? r.m.wsm_levels : 1);
    const Shape s = make_shape(r.V, r.T, r.H, r.W, r.D, r.dtype, c.F, B.data());
    const Layout L = make_layout(s, true, true);
    Scratch ws;
    st = ws.acquire(r.workspace, r.workspace_bytes, L.total, r.stream);
    if (st != WZ_OK) return st;
    bind(c, s, L, ws.ptr);
    c.X = r.features;
    c.Q = r.queries;
    c.out = r.out_tokens;
    c.out_index = r.out_index;
    c.out_budgets = r.out_budgets;
    c.out_count = r.out_count;
    c.out_rel = r.out_relevance;
    if (r.device_status) c.status = r.device_status;
    else c.clear_status = 1;
    c.sms = sm_count();
    c.G1 = relevance_grid(c);
    if (c.G1 < 1) {
        cudaGetLastError();
        return WZ_ERR_CUDA;
    }
    const int64_t total = (int64_t)s.V * s.T * s.N;
    c.L1 = (total + c.G1 - 1) / c.G1;
    std::vector<VideoPar> par(r.V);
    int qrow = 0;
    int64_t row0 = 0, wrow0 = 0;
    for (int v = 0; v < r.V; ++v) {
        par[v].q_row0 = qrow;
        par[v].Lq = r.Lq[v];
        par[v].B = (int)B[v];
        par[v].row0 = (int)row0;
        par[v].w_row0 = (int)wrow0;
        qrow += r.Lq[v];
        row0 += B[v];
        wrow0 += video_w_rows(B[v], r.T);
    }
    auto mark = [&](int k) -> cudaError_t {
        return r.events ? cudaEventRecord((cudaEvent_t)r.events[k], r.stream) : cudaSuccess;
    };
    Nvtx whole("wz::condense");
    const bool maxsim = c.relevance_mode == WZ_RELEVANCE_MAXSIM;
    const int Lq_max = *std::max_element(r.Lq.begin(), r.Lq.end()), Lqp_max = (Lq_max + 15) / 16 * 16;
    bool fused_maxsim = false;
    int64_t qrows = 0;   // unit query rows of all videos
    if (maxsim) {
        qrows = qhl_row(qrow, r.V);
        size_t at = 0;
        const QueryRows place = place_query_rows(c, s, L, Lqp_max, qrows, &at);
        fused_maxsim = place != QueryRows::kByVideo;
        if (place == QueryRows::kSlots || place == QueryRows::kOperator)
            c.qhl = reinterpret_cast<__nv_bfloat16 *>(ws.ptr + at);
    }
    WZ_CUDA(mark(2 * WZ_KERNEL_QUERY_POOL));
    if (fused_maxsim) {   // needs no pooled query
        Nvtx n_("wz::query_rows");
        WZ_CUDA(launch_query_rows(c, par.data(), 0, r.V, Lqp_max, true, r.stream));
    } else {
        Nvtx n_("wz::query_pool");
        WZ_CUDA(launch_query_pool(c, par.data(), r.stream));
    }
    WZ_CUDA(mark(2 * WZ_KERNEL_QUERY_POOL + 1));
    WZ_CUDA(mark(2 * WZ_KERNEL_RELEVANCE));
    if (fused_maxsim) {
        Nvtx n_("wz::maxsim_pass");
        WZ_CUDA(launch_maxsim_pass(c, Lqp_max, qrows, r.stream));
    } else {
        Nvtx n_("wz::relevance_pass");
        WZ_CUDA(launch_relevance_pass(c, r.stream));
    }
    WZ_CUDA(mark(2 * WZ_KERNEL_RELEVANCE + 1));
    if (maxsim && !fused_maxsim) {
        // the token x query-row cosines on the tensor cores, video by video
        // (the relevance pass left ||u|| in c.a)
        Nvtx n_("wz::maxsim");
        for (int v = 0; v < r.V; ++v) {
            const int Lq = r.Lq[v], Lqp = (Lq + 15) / 16 * 16;
            const int64_t tok = (int64_t)s.T * s.N;
            c.qhl_row0 = qhl_row(par[v].q_row0, v);
            WZ_CUDA(launch_query_rows(c, par.data(), v, 1, Lqp, false, r.stream));
            WZ_CUDA(launch_maxsim_gemm(static_cast<const char *>(r.features) + (size_t)v * tok * s.D * 2, (int)tok,
                                       s.D, c.qhl, Lq, Lqp, c.a + v * tok, c.status, c.pdl != 0, r.stream));
        }
    }
    WZ_CUDA(mark(2 * WZ_KERNEL_FRAME_STATS));
    {
        Nvtx n_("wz::frame_stats");
        WZ_CUDA(launch_frame_stats(c, r.stream));
    }
    WZ_CUDA(mark(2 * WZ_KERNEL_FRAME_STATS + 1));
    WZ_CUDA(mark(2 * WZ_KERNEL_TEMPORAL));
    {
        Nvtx n_("wz::temporal");
        WZ_CUDA(launch_temporal(c, r.stream));
    }
    WZ_CUDA(mark(2 * WZ_KERNEL_TEMPORAL + 1));
    WZ_CUDA(mark(2 * WZ_KERNEL_SPATIAL));
    {
        Nvtx n_("wz::spatial");
        WZ_CUDA(launch_spatial(c, r.stream));
    }
    WZ_CUDA(mark(2 * WZ_KERNEL_SPATIAL + 1));
    WZ_CUDA(mark(2 * WZ_KERNEL_CONDENSE));
    if (rows > 0) {
        Nvtx n_("wz::condense_tokens");
        if (c.path == WZ_PATH_TENSOR) WZ_CUDA(launch_condense_tc(c, r.stream));
        else WZ_CUDA(launch_condense_simt(c, r.stream));
    }
    WZ_CUDA(mark(2 * WZ_KERNEL_CONDENSE + 1));
    return WZ_OK;
}

// Replay cache.  The six launches of an argument set seen for the second time
// are captured on a private stream (nothing runs during a capture),
// instantiated once, and the executable graph is launched into the caller's
// stream on that call and every later one with the same arguments (the first
// sighting launches directly, so calls whose buffers move every time never pay
// for a capture).  The graph keeps the launches' programmatic-dependency
// edges; submitted as one unit, the sequence loses the gaps that separate
// launches leave between dependent kernels.  Every argument is in the key
// (pointers, sizes, options, the current device), so a hit replays exactly the
// launches a direct call would make; the inputs are read when the replay runs.
struct GraphEntry {
    std::string key;
    cudaGraphExec_t exec;
};
std::mutex g_graph_mu;
std::list<GraphEntry> g_graphs;          // most recently used first
std::list<std::string> g_seen;           // keys launched directly once
int g_graph_capacity = 8;
int64_t g_graph_replays = 0, g_graph_captures = 0;

void trim_graphs(int cap) {
    // an executable graph still in flight is freed when its launch completes
    while ((int)g_graphs.size() > cap) {
        cudaGraphExecDestroy(g_graphs.back().exec);
        g_graphs.pop_back();
    }
    while ((int)g_seen.size() > 2 * cap) g_seen.pop_back();
}

std::string request_key(const CondenseRequest &r, int dev) {
    std::string k;
    auto put = [&k](const void *p, size_t n) { k.append(static_cast<const char *>(p), n); };
    const int ints[] = {dev, r.V, r.T, r.H, r.W, r.D, r.dtype, r.m.wta_wavelet, r.m.wsm_wavelet, r.m.mode,
                        r.m.path, r.m.temporal_mode, r.m.spatial_mode, r.m.relevance_mode, r.m.wta_levels,
                        r.m.wsm_levels};
    const float reals[] = {r.m.lambda, r.m.tau};
    const void *ptrs[] = {r.features, r.queries, r.token_scores, r.frame_scores, r.out_tokens, r.out_index,
                          r.out_budgets, r.out_count, r.device_status, r.out_relevance, r.workspace};
    put(ints, sizeof ints);
    put(reals, sizeof reals);
    put(ptrs, sizeof ptrs);
    put(&r.workspace_bytes, sizeof r.workspace_bytes);
    put(r.Lq.data(), r.Lq.size() * sizeof(int));
    put(r.ratio.data(), r.ratio.size() * sizeof(float));
    return k;
}

int run_condense_cached(const CondenseRequest &r) {
    if (r.events || !r.workspace) return run_condense(r);
    // the argument checks of a direct call, before any CUDA call
    std::vector<int64_t> B;
    int64_t rows = 0;
    int st = validate(r, B, rows);
    if (st != WZ_OK) return st;
    if (!aligned(r.workspace, kAlign)) return WZ_ERR_INVALID_ARG;
    const Shape s = make_shape(r.V, r.T, r.H, r.W, r.D, r.dtype, wavelet_taps(r.m.wsm_wavelet), B.data());
    if (r.workspace_bytes < make_layout(s, true, true).total) return WZ_ERR_WORKSPACE;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    WZ_CUDA(cudaStreamIsCapturing(r.stream, &cs));
    if (cs != cudaStreamCaptureStatusNone) return run_condense(r);   // the caller is capturing it
    int dev = 0;
    WZ_CUDA(cudaGetDevice(&dev));
    const std::string key = request_key(r, dev);
    std::unique_lock<std::mutex> lock(g_graph_mu);
    if (g_graph_capacity <= 0) {
        lock.unlock();
        return run_condense(r);
    }
    for (auto it = g_graphs.begin(); it != g_graphs.end(); ++it) {
        if (it->key != key) continue;
        g_graphs.splice(g_graphs.begin(), g_graphs, it);
        WZ_CUDA(cudaGraphLaunch(g_graphs.front().exec, r.stream));
        ++g_graph_replays;
        return WZ_OK;
    }
    const auto seen = std::find(g_seen.begin(), g_seen.end(), key);
    if (seen == g_seen.end()) {
        g_seen.push_front(key);
        trim_graphs(g_graph_capacity);
        lock.unlock();   // direct launches need no cache state
        return run_condense(r);
    }
    g_seen.erase(seen);
    cudaStream_t cap = nullptr;
    WZ_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    if (cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        cudaGetLastError();
        cudaStreamDestroy(cap);
        return WZ_ERR_CUDA;
    }
    CondenseRequest rc = r;
    rc.stream = cap;
    st = run_condense(rc);
    cudaGraph_t g = nullptr;
    const cudaError_t e = cudaStreamEndCapture(cap, &g);
    cudaStreamDestroy(cap);
    if (st != WZ_OK || e != cudaSuccess || !g) {
        if (g) cudaGraphDestroy(g);
        cudaGetLastError();
        return st != WZ_OK ? st : WZ_ERR_CUDA;
    }
    cudaGraphExec_t exec = nullptr;
    const cudaError_t ei = cudaGraphInstantiate(&exec, g, 0);
    cudaGraphDestroy(g);
    if (ei != cudaSuccess) {
        cudaGetLastError();
        return WZ_ERR_CUDA;
    }
    if (cudaGraphLaunch(exec, r.stream) != cudaSuccess) {
        cudaGetLastError();
        cudaGraphExecDestroy(exec);
        return WZ_ERR_CUDA;
    }
    g_graphs.push_front(GraphEntry{key, exec});
    ++g_graph_captures;
    trim_graphs(g_graph_capacity);
    return WZ_OK;
}

size_t condense_ws(int V, int T, int H, int W, int D, int dtype, const float *ratio) {
    if (check_sizes(V, T, H, W, D, dtype) != WZ_OK || !ratio) return 0;
    std::vector<int64_t> B(V);
    for (int v = 0; v < V; ++v) {
        if (!valid_ratio(ratio[v])) return 0;
        B[v] = budget(T, H * W, ratio[v]);
    }
    const Shape s = make_shape(V, T, H, W, D, dtype, 2, B.data());
    return make_layout(s, true, true).total;
}

}  // namespace
}  // namespace wz

using namespace wz;

extern "C" {

int64_t wz_budget_size(int T, int H, int W, float ratio) {
    if (T < 1 || H < 1 || W < 1 || !valid_ratio(ratio)) return -1;
    return budget(T, H * W, ratio);
}

void wz_condense_args_init(wz_condense_args *a) {
    if (!a) return;
    std::memset(a, 0, sizeof(*a));
    a->dtype = WZ_DTYPE_BF16;
    a->lambda = 1.5f;
    a->tau = 0.f;
    a->wta_wavelet = WZ_WAVELET_HAAR;
    a->wsm_wavelet = WZ_WAVELET_DB4;
    a->mode = WZ_MODE_SYMMETRIC;
    a->path = WZ_PATH_AUTO;
    a->wta_levels = 1;
    a->wsm_levels = 1;
}

void wz_batch_args_init(wz_batch_args *a) {
    if (!a) return;
    std::memset(a, 0, sizeof(*a));
    a->dtype = WZ_DTYPE_BF16;
    a->lambda = 1.5f;
    a->tau = 0.f;
    a->wta_wavelet = WZ_WAVELET_HAAR;
    a->wsm_wavelet = WZ_WAVELET_DB4;
    a->mode = WZ_MODE_SYMMETRIC;
    a->path = WZ_PATH_AUTO;
    a->wta_levels = 1;
    a->wsm_levels = 1;
}

size_t wz_condense_workspace_size(int T, int H, int W, int D, int dtype, float ratio) {
    return condense_ws(1, T, H, W, D, dtype, &ratio);
}

int wz_condense_ex(const wz_condense_args *a) {
    if (!a) return WZ_ERR_INVALID_ARG;
    CondenseRequest r;
    r.V = 1; r.T = a->T; r.H = a->H; r.W = a->W; r.D = a->D; r.dtype = a->dtype;
    r.features = a->features;
    r.queries = a->query;
    r.Lq.assign(1, a->Lq);
    r.ratio.assign(1, a->ratio);
    r.m = Common{a->lambda, a->tau, a->wta_wavelet, a->wsm_wavelet, a->mode, a->path, a->temporal_mode,
                 a->spatial_mode};
    r.token_scores = a->token_scores;
    r.frame_scores = a->frame_scores;
    r.m.relevance_mode = a->relevance_mode;
    r.m.wta_levels = a->wta_levels;
    r.m.wsm_levels = a->wsm_levels;
    r.out_tokens = a->out_tokens;
    r.out_index = a->out_index;
    r.out_budgets = a->out_budgets;
    r.out_count = a->out_count;
    r.out_relevance = a->out_relevance;
    r.device_status = a->device_status;
    r.workspace = a->workspace;
    r.workspace_bytes = a->workspace_bytes;
    r.events = a->kernel_events;
    r.stream = (cudaStream_t)a->stream;
    return run_condense_cached(r);
}

int wz_condense_host(const wz_condense_args *a) {
    if (!a || !a->features || !a->query || !a->out_tokens || !a->out_index) return WZ_ERR_INVALID_ARG;
    if (a->token_scores || a->frame_scores || a->kernel_events) return WZ_ERR_INVALID_ARG;   // device-only inputs
    int st = check_sizes(1, a->T, a->H, a->W, a->D, a->dtype);
    if (st != WZ_OK) return st;
    if (a->Lq < 1 || !valid_ratio(a->ratio)) return WZ_ERR_INVALID_ARG;
    const int64_t B = budget(a->T, a->H * a->W, a->ratio);
    const size_t esz = a->dtype == WZ_DTYPE_BF16 ? 2 : 4;
    const size_t xb = (size_t)a->T * a->H * a->W * a->D * esz, qb = (size_t)a->Lq * a->D * esz;
    const size_t tb = (size_t)B * a->D * esz, ib = (size_t)B * 3 * 4, bb = (size_t)a->T * 4, rb = (size_t)a->T * 16;
    cudaStream_t s = (cudaStream_t)a->stream;
    // device staging: features, query, the outputs, count and status, one allocation
    size_t o = 0;
    auto take = [&](size_t n) {
        const size_t at = o;
        o = align_up(o + n);
        return at;
    };
    const size_t ox = take(xb), oq = take(qb), ot = take(tb), oi = take(ib), obu = take(bb), orl = take(rb),
                 oc = take(16);
    char *dev = nullptr;
    if (cudaMallocAsync(reinterpret_cast<void **>(&dev), o, s) != cudaSuccess) {
        cudaGetLastError();
        return WZ_ERR_NO_MEMORY;
    }
    wz_condense_args d = *a;
    d.features = dev + ox;
    d.query = dev + oq;
    d.out_tokens = dev + ot;
    d.out_index = reinterpret_cast<int32_t *>(dev + oi);
    d.out_budgets = a->out_budgets ? reinterpret_cast<int32_t *>(dev + obu) : nullptr;
    d.out_relevance = a->out_relevance ? reinterpret_cast<float *>(dev + orl) : nullptr;
    d.out_count = a->out_count ? reinterpret_cast<int32_t *>(dev + oc) : nullptr;
    d.device_status = nullptr;
    d.workspace = nullptr;   // staging and workspace both from the stream-ordered allocator
    d.workspace_bytes = 0;
    st = WZ_OK;
    if (cudaMemcpyAsync(dev + ox, a->features, xb, cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(dev + oq, a->query, qb, cudaMemcpyHostToDevice, s) != cudaSuccess)
        st = WZ_ERR_CUDA;
    if (st == WZ_OK) st = wz_condense_ex(&d);
    if (st == WZ_OK) {
        if (cudaMemcpyAsync(a->out_tokens, dev + ot, tb, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(a->out_index, dev + oi, ib, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            (a->out_budgets && cudaMemcpyAsync(a->out_budgets, dev + obu, bb, cudaMemcpyDeviceToHost, s) != cudaSuccess) ||
            (a->out_relevance &&
             cudaMemcpyAsync(a->out_relevance, dev + orl, rb, cudaMemcpyDeviceToHost, s) != cudaSuccess) ||
            (a->out_count && cudaMemcpyAsync(a->out_count, dev + oc, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess))
            st = WZ_ERR_CUDA;
    }
    if (cudaFreeAsync(dev, s) != cudaSuccess && st == WZ_OK) st = WZ_ERR_CUDA;
    if (st == WZ_ERR_CUDA) cudaGetLastError();
    return st;
}

int wz_condense(const void *features, int T, int H, int W, int D, const void *query, int Lq,
                float ratio, void *out_tokens, int32_t *out_index, wz_stream_t stream) {
    wz_condense_args a;
    wz_condense_args_init(&a);
    a.features = features;
    a.T = T; a.H = H; a.W = W; a.D = D;
    a.query = query;
    a.Lq = Lq;
    a.ratio = ratio;
    a.out_tokens = out_tokens;
    a.out_index = out_index;
    a.stream = stream;
    return wz_condense_ex(&a);
}

int64_t wz_batch_rows(int V, int T, int H, int W, const float *ratio, int64_t *row_offsets) {
    if (V < 1 || T < 1 || H < 1 || W < 1 || !ratio) return -1;
    int64_t rows = 0;
    for (int v = 0; v < V; ++v) {
        if (!valid_ratio(ratio[v])) return -1;
        if (row_offsets) row_offsets[v] = rows;
        rows += budget(T, H * W, ratio[v]);
    }
    if (row_offsets) row_offsets[V] = rows;
    return rows;
}

size_t wz_batch_workspace_size(int V, int T, int H, int W, int D, int dtype, const float *ratio) {
    return condense_ws(V, T, H, W, D, dtype, ratio);
}

int wz_condense_batch(const wz_batch_args *a) {
    if (!a || !a->Lq || !a->ratio) return WZ_ERR_INVALID_ARG;
    if (a->V < 1 || a->V > WZ_MAX_VIDEOS) return a->V < 1 ? WZ_ERR_INVALID_ARG : WZ_ERR_UNSUPPORTED;
    CondenseRequest r;
    r.V = a->V; r.T = a->T; r.H = a->H; r.W = a->W; r.D = a->D; r.dtype = a->dtype;
    r.features = a->features;
    r.queries = a->queries;
    r.Lq.assign(a->Lq, a->Lq + a->V);
    r.ratio.assign(a->ratio, a->ratio + a->V);
    r.m = Common{a->lambda, a->tau, a->wta_wavelet, a->wsm_wavelet, a->mode, a->path, a->temporal_mode,
                 a->spatial_mode};
    r.token_scores = a->token_scores;
    r.frame_scores = a->frame_scores;
    r.m.relevance_mode = a->relevance_mode;
    r.m.wta_levels = a->wta_levels;
    r.m.wsm_levels = a->wsm_levels;
    r.out_tokens = a->out_tokens;
    r.out_index = a->out_index;
    r.out_budgets = a->out_budgets;
    r.out_count = a->out_count;
    r.out_relevance = a->out_relevance;
    r.device_status = a->device_status;
    r.workspace = a->workspace;
    r.workspace_bytes = a->workspace_bytes;
    r.events = a->kernel_events;
    r.stream = (cudaStream_t)a->stream;
    if (a->row_offsets && wz_batch_rows(a->V, a->T, a->H, a->W, a->ratio, a->row_offsets) < 0)
        return WZ_ERR_INVALID_ARG;
    return run_condense_cached(r);
}

int wz_graph_cache(int capacity, int64_t *stats) {
    std::lock_guard<std::mutex> lock(g_graph_mu);
    const int prev = g_graph_capacity;
    if (capacity >= 0) {
        g_graph_capacity = capacity;
        trim_graphs(capacity);
    }
    if (stats) {
        stats[0] = (int64_t)g_graphs.size();
        stats[1] = g_graph_replays;
        stats[2] = g_graph_captures;
    }
    return prev;
}

size_t wz_relevance_workspace_size(int T, int H, int W, int D) {
    if (check_sizes(1, T, H, W, D, WZ_DTYPE_BF16) != WZ_OK) return 0;
    const Shape s = make_shape(1, T, H, W, D, WZ_DTYPE_BF16, 2, nullptr);
    return make_layout(s, false, false).total;
}


int wz_relevance(const void *features, int T, int H, int W, int D, int dtype, const void *query,
                 int Lq, float *token_scores, float *frame_scores, float *frame_mean,
                 void *workspace, size_t workspace_bytes, int32_t *device_status, wz_stream_t stream) {
    int st = check_sizes(1, T, H, W, D, dtype);
    if (st != WZ_OK) return st;
    if (!features || !query || !token_scores || !frame_scores || Lq < 1) return WZ_ERR_INVALID_ARG;
    if (!aligned(features, 16) || !aligned(query, 16) || !aligned(token_scores, 4) ||
        !aligned(frame_scores, 4) || (frame_mean && !aligned(frame_mean, 4)) || !aligned(device_status, 4))
        return WZ_ERR_INVALID_ARG;
    const Shape s = make_shape(1, T, H, W, D, dtype, 2, nullptr);
    const Layout L = make_layout(s, false, false);
    Scratch ws;
    st = ws.acquire(workspace, workspace_bytes, L.total, (cudaStream_t)stream);
    if (st != WZ_OK) return st;
    Ctx c{};
    bind(c, s, L, ws.ptr);
    c.X = features;
    c.Q = query;
    c.a = token_scores;
    c.frame_scores = frame_scores;
    c.frame_mean = frame_mean;
    c.sms = sm_count();
    c.G1 = relevance_grid(c);
    if (c.G1 < 1) {
        cudaGetLastError();
        return WZ_ERR_CUDA;
    }
    c.L1 = ((int64_t)T * s.N + c.G1 - 1) / c.G1;
    VideoPar par{0, Lq, 0, 0, 0};
    const cudaStream_t cs = (cudaStream_t)stream;
    // a bounded wait that gives up reports to the caller's status word, else
    // to the workspace's, which starts each call at zero
    if (device_status) c.status = device_status;
    else c.clear_status = 1;
    WZ_CUDA(launch_query_pool(c, &par, cs));
    WZ_CUDA(launch_relevance_pass(c, cs));
    WZ_CUDA(launch_frame_stats(c, cs));
    return WZ_OK;
}

size_t wz_project_workspace_size(int64_t B, int C) {
    if (B < 0 || C < 1) return 0;
    return align_up((size_t)B * (size_t)C * 2) + kAlign;   // hidden layer, then the status word
}

int wz_project(const wz_project_args *a) {
    if (!a) return WZ_ERR_INVALID_ARG;
    const auto dim_ok = [](int x) { return x >= 64 && x <= 65536 && x % 64 == 0; };
    if (a->B < 0 || a->B > (int64_t)INT32_MAX || !dim_ok(a->D) || !dim_ok(a->C) || !dim_ok(a->E))
        return WZ_ERR_INVALID_ARG;
    if (a->B == 0) return WZ_OK;
    if (!a->tokens || !a->w1 || !a->w2 || !a->out) return WZ_ERR_INVALID_ARG;
    if (!aligned(a->tokens, 16) || !aligned(a->w1, 16) || !aligned(a->w2, 16) || !aligned(a->out, 16) ||
        !aligned(a->b1, 16) || !aligned(a->b2, 16) || !aligned(a->device_status, 4))
        return WZ_ERR_INVALID_ARG;
    const cudaStream_t s = (cudaStream_t)a->stream;
    const size_t need = wz_project_workspace_size(a->B, a->C);
    Scratch ws;
    int st = ws.acquire(a->workspace, a->workspace_bytes, need, s);
    if (st != WZ_OK) return st;
    int *status = a->device_status;
    const bool own = !status;
    if (own) status = reinterpret_cast<int *>(ws.ptr + align_up((size_t)a->B * (size_t)a->C * 2));
    const int M = (int)a->B;
    WZ_CUDA(launch_project_gemm(a->tokens, M, a->D, a->w1, a->C, a->b1, ws.ptr, true, status, own, false, s));
    WZ_CUDA(launch_project_gemm(ws.ptr, M, a->C, a->w2, a->E, a->b2, a->out, false, status, false, true, s));
    return WZ_OK;
}

int wz_dwt_len(int n, int wavelet) {
    const int F = wavelet_taps(wavelet);
    if (n < 1 || F == 0) return -1;
    return (n + F - 1) / 2;
}

int wz_wavelet_filters(int wavelet, double *dec_lo, double *dec_hi, double *rec_lo, double *rec_hi) {
    if (wavelet_taps(wavelet) == 0) return WZ_ERR_INVALID_ARG;
    return wavelet_bank(wavelet, dec_lo, dec_hi, rec_lo, rec_hi) ? WZ_OK : WZ_ERR_INVALID_ARG;
}

static void float_taps(int p, float *dl, float *dh, float *rl, float *rh) {
    double a[kMaxTaps], b[kMaxTaps], c[kMaxTaps], d[kMaxTaps];
    wavelet_bank(p, a, b, c, d);
    for (int k = 0; k < wavelet_taps(p); ++k) {
        dl[k] = (float)a[k];
        dh[k] = (float)b[k];
        rl[k] = (float)c[k];
        rh[k] = (float)d[k];
    }
}

int wz_dwt1d(const float *x, int rows, int L, int wavelet, int mode, float *cA, float *cD,
             wz_stream_t stream) {
    if (rows < 0 || L < 1 || wavelet_taps(wavelet) == 0 || mode < 0 || mode > 2) return WZ_ERR_INVALID_ARG;
    if (rows > 0 && (!x || !cA || !cD)) return WZ_ERR_INVALID_ARG;
    float dl[kMaxTaps], dh[kMaxTaps], rl[kMaxTaps], rh[kMaxTaps];
    float_taps(wavelet, dl, dh, rl, rh);
    WZ_CUDA(launch_dwt1d(x, rows, L, wavelet_taps(wavelet), mode, dl, dh, cA, cD, (cudaStream_t)stream));
    return WZ_OK;
}

int wz_idwt1d(const float *cA, const float *cD, int rows, int L, int wavelet, float *x,
              wz_stream_t stream) {
    if (rows < 0 || L < 1 || wavelet_taps(wavelet) == 0) return WZ_ERR_INVALID_ARG;
    if (rows > 0 && (!x || !cA || !cD)) return WZ_ERR_INVALID_ARG;
    float dl[kMaxTaps], dh[kMaxTaps], rl[kMaxTaps], rh[kMaxTaps];
    float_taps(wavelet, dl, dh, rl, rh);
    WZ_CUDA(launch_idwt1d(cA, cD, rows, L, wavelet_taps(wavelet), rl, rh, x, (cudaStream_t)stream));
    return WZ_OK;
}

int wz_dwt2d(const void *features, int T, int H, int W, int D, int dtype, int wavelet, int mode,
             float *LL, float *LH, float *HL, float *HH, wz_stream_t stream) {
    if (T < 1 || H < 1 || W < 1 || D < 1 || wavelet_taps(wavelet) == 0 || mode < 0 || mode > 2)
        return WZ_ERR_INVALID_ARG;
    if (dtype != WZ_DTYPE_BF16 && dtype != WZ_DTYPE_F32) return WZ_ERR_INVALID_ARG;
    if (H > WZ_MAX_HW || W > WZ_MAX_HW || T > 65535) return WZ_ERR_UNSUPPORTED;
    if (!features || !LL || !LH || !HL || !HH) return WZ_ERR_INVALID_ARG;
    float dl[kMaxTaps], dh[kMaxTaps], rl[kMaxTaps], rh[kMaxTaps];
    float_taps(wavelet, dl, dh, rl, rh);
    WZ_CUDA(launch_dwt2d(features, dtype, T, H, W, D, wavelet_taps(wavelet), mode, dl, dh, LL, LH, HL, HH,
                         (cudaStream_t)stream));
    return WZ_OK;
}

int wz_idwt2d(const float *LL, const float *LH, const float *HL, const float *HH, int T, int H, int W,
              int D, int wavelet, float *out, wz_stream_t stream) {
    if (T < 1 || H < 1 || W < 1 || D < 1 || wavelet_taps(wavelet) == 0) return WZ_ERR_INVALID_ARG;
    if (H > WZ_MAX_HW || W > WZ_MAX_HW || T > 65535) return WZ_ERR_UNSUPPORTED;
    if (!out || !LL || !LH || !HL || !HH) return WZ_ERR_INVALID_ARG;
    float dl[kMaxTaps], dh[kMaxTaps], rl[kMaxTaps], rh[kMaxTaps];
    float_taps(wavelet, dl, dh, rl, rh);
    WZ_CUDA(launch_idwt2d(LL, LH, HL, HH, T, H, W, D, wavelet_taps(wavelet), rl, rh, out, (cudaStream_t)stream));
    return WZ_OK;
}

const char *wz_status_string(int status) {
    switch (status) {
        case WZ_OK: return "ok";
        case WZ_ERR_INVALID_ARG: return "invalid argument";
        case WZ_ERR_UNSUPPORTED: return "unsupported: beyond the library's limits";
        case WZ_ERR_CUDA: return "CUDA error";
        case WZ_ERR_NO_MEMORY: return "workspace allocation failed";
        case WZ_ERR_WORKSPACE: return "workspace too small";
        default: return "unknown status";
    }
}

int wz_version(void) { return 100; }

#ifdef WZ_CHECKED
// Test hook: the QueryRows of a bf16 batch with the max-over-query scorer on the
// current device, as an int; negative on an error.
__attribute__((visibility("default"))) int wz_check_query_rows(int V, int T, int H, int W, int D, const int32_t *Lq,
                                                               const float *ratio) {
    if (!Lq || !ratio || check_sizes(V, T, H, W, D, WZ_DTYPE_BF16) != WZ_OK) return -1;
    std::vector<int64_t> B(V);
    int rows = 0;
    for (int v = 0; v < V; ++v) {
        B[v] = budget(T, H * W, ratio[v]);
        rows += Lq[v];
    }
    const Shape s = make_shape(V, T, H, W, D, WZ_DTYPE_BF16, 2, B.data());
    const Layout L = make_layout(s, true, true);
    Ctx c{};
    bind(c, s, L, nullptr);
    c.relevance_mode = WZ_RELEVANCE_MAXSIM;
    c.sms = sm_count();
    c.G1 = relevance_grid(c);
    size_t at = 0;
    return c.G1 < 1 ? -1
                    : (int)place_query_rows(c, s, L, (*std::max_element(Lq, Lq + V) + 15) / 16 * 16, qhl_row(rows, V), &at);
}
#endif

}  // extern "C"
