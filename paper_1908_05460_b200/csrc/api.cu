// C-ABI entry points of libgaconv: argument validation, workspace planning, kernel dispatch and the
// approximation-schedule driver (paper Section 2.5).  Every step of the path runs in this library's
// kernels; there is no CPU or library fallback.
#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "gaconv_internal.h"

using namespace gaconv;

static std::atomic<uint64_t> g_launches{0};
void gaconv::note_launch(int count) { g_launches.fetch_add((uint64_t)count, std::memory_order_relaxed); }

namespace {

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

gaconv_status_t make_geom(const gaconv_conv_desc_t* d, Geom* g)
{
    if (d == nullptr) return GACONV_ERR_NULL_POINTER;
    if (d->struct_size != sizeof(gaconv_conv_desc_t)) return GACONV_ERR_BAD_DESC;
    if (d->n < 1 || d->c < 1 || d->h < 1 || d->w < 1 || d->k < 1 || d->r < 1 || d->s < 1) return GACONV_ERR_BAD_DESC;
    if (d->stride_h < 1 || d->stride_w < 1 || d->pad_h < 0 || d->pad_w < 0) return GACONV_ERR_BAD_DESC;
    if (d->h + 2 * d->pad_h < d->r || d->w + 2 * d->pad_w < d->s) return GACONV_ERR_BAD_DESC;
    if (d->in_dtype != GACONV_F32 && d->in_dtype != GACONV_BF16) return GACONV_ERR_BAD_DESC;
    if (d->x_layout != GACONV_X_NHWC && d->x_layout != GACONV_X_NCHW) return GACONV_ERR_BAD_DESC;
    if (d->dy_layout != GACONV_DY_NKPQ && d->dy_layout != GACONV_DY_NPQK) return GACONV_ERR_BAD_DESC;
    if (d->dw_layout != GACONV_DW_KRSC && d->dw_layout != GACONV_DW_KCRS && d->dw_layout != GACONV_DW_RSCK) return GACONV_ERR_BAD_DESC;
    if (d->math != GACONV_MATH_DEFAULT && d->math != GACONV_MATH_TF32) return GACONV_ERR_BAD_DESC;
    if (d->algo < GACONV_ALGO_AUTO || d->algo > GACONV_ALGO_TENSOR) return GACONV_ERR_BAD_DESC;
    g->n = d->n; g->c = d->c; g->h = d->h; g->w = d->w; g->k = d->k; g->r = d->r; g->s = d->s;
    g->stride_h = d->stride_h; g->stride_w = d->stride_w; g->pad_h = d->pad_h; g->pad_w = d->pad_w;
    g->p = (d->h + 2 * d->pad_h - d->r) / d->stride_h + 1;
    g->q = (d->w + 2 * d->pad_w - d->s) / d->stride_w + 1;
    if (g->p < 1 || g->q < 1) return GACONV_ERR_BAD_DESC;
    // element counts must fit comfortably in 63 bits and per-map sizes in 31
    if ((long long)g->p * g->q > (1ll << 30) || (long long)g->r * g->s * g->c > (1ll << 30)) return GACONV_ERR_UNSUPPORTED;
    if (d->x_layout == GACONV_X_NHWC) {
        g->xs_c = 1; g->xs_w = d->c; g->xs_h = (long long)d->w * d->c; g->xs_n = (long long)d->h * d->w * d->c;
    } else {
        g->xs_w = 1; g->xs_h = d->w; g->xs_c = (long long)d->h * d->w; g->xs_n = (long long)d->c * d->h * d->w;
    }
    if (d->dw_layout == GACONV_DW_KRSC) {
        g->ws_c = 1; g->ws_s = d->c; g->ws_r = (long long)d->s * d->c; g->ws_k = (long long)d->r * d->s * d->c;
    } else if (d->dw_layout == GACONV_DW_KCRS) {
        g->ws_s = 1; g->ws_r = d->s; g->ws_c = (long long)d->r * d->s; g->ws_k = (long long)d->c * d->r * d->s;
    } else {
        g->ws_k = 1; g->ws_c = d->k; g->ws_s = (long long)d->c * d->k; g->ws_r = (long long)d->s * d->c * d->k;
    }
    g->bf16 = d->in_dtype == GACONV_BF16;
    g->alpha = d->alpha;
    if (d->sm_budget < 0) return GACONV_ERR_BAD_DESC;
    g->sm_budget = d->sm_budget;
    return GACONV_OK;
}

// ---- plans are kept: the planners run once per (problem, device), not once per call --------------------------------
// A key is every field a plan depends on, plus the device (SM count and resident clusters differ between devices).
struct PlanKey {
    long long v[26];
    bool operator==(const PlanKey& o) const { return memcmp(v, o.v, sizeof(v)) == 0; }
};
PlanKey plan_key(const Geom& g, int a, int b)
{
    int dev = 0;
    cudaGetDevice(&dev);
    uint32_t alpha_bits;
    memcpy(&alpha_bits, &g.alpha, sizeof(alpha_bits));
    return PlanKey{{g.n, g.c, g.h, g.w, g.k, g.r, g.s, g.p, g.q, g.stride_h, g.stride_w, g.pad_h, g.pad_w, g.xs_n, g.xs_c, g.xs_h,
                    g.xs_w, g.ws_k, g.ws_c, g.ws_r, g.ws_s, g.bf16 ? 1 : 0, (long long)alpha_bits, g.sm_budget, ((long long)a << 32) | (uint32_t)b, dev}};
}
template <typename L>
class PlanCache {
public:
    template <typename Build>
    L get(const PlanKey& key, Build build)
    {
#ifndef GACONV_TUNING            // tuning builds read planner overrides from the environment on every call
        {
            std::lock_guard<std::mutex> lock(m_);
            for (size_t i = 0; i < e_.size(); ++i)
                if (e_[i].first == key) {
                    if (i != 0) std::swap(e_[i], e_[i - 1]);       // frequently used entries drift to the front
                    return e_[i != 0 ? i - 1 : 0].second;
                }
        }
#endif
        L made = build();
#ifndef GACONV_TUNING
        std::lock_guard<std::mutex> lock(m_);
        try {                          // (no host memory: the plan is used and not kept; nothing may throw through the C interface)
            if (e_.size() >= kMaxEntries) e_.pop_back();
            e_.emplace_back(key, made);
        } catch (const std::bad_alloc&) { }
#endif
        return made;
    }
private:
    static constexpr size_t kMaxEntries = 256;
    std::mutex m_;
    std::vector<std::pair<PlanKey, L>> e_;
};

// A large dW with short sums, split over CTAs, on a GPU of its own: the channels-last kernel writes as many partial blocks as it has
// CTAs and reads them again, the older kernel adds them inside clusters.  The line is at one pixel for every hundred elements, where
// the two meet (us, the older kernel first): 0.002 256->512 on 4x4, N = 128 18.6 / 21.9; 0.007 256->256 on 8x8, N = 64 14.5 / 15.1;
// 0.009 the same, N = 80 15.9 / 15.7, 384->256 on 8x8 23.1 / 23.4, 192->384 on 8x8, N = 96 17.3 / 19.0; 0.0104 256->256 on 8x8, N = 96
// 17.3 / 16.6; 0.0108 256->256 on 4x4, N = 400 21.0 / 20.8; 0.014 256->256 on 8x8, N = 128 20.0 / 18.0, 128->512 on 4x4, N = 512 25.6 / 24.0.
bool short_sums(const Geom& g, const ClPlan& plan)
{
    const double elements = (double)g.k * g.c * g.r * g.s;
    return g.sm_budget == 0 && plan.partial_bytes > 0 && elements > 4e5 && (double)g.n * g.p * g.q < 0.01 * elements;
}

// Small maps with many channels (up to 4x4 pixels from 128 channels, up to 8x8 from 256): the N*K patch accumulations (N*K*R*S*C FMAs on the FP32 pipes,
// the same number of bytes gathered from L2) cost more than the dense contraction on tensor cores, and with so few
// pixels per map the sparse tensor is not that sparse (1 - 1/(PQ), Section 2.3).  Then the method is run
// literally as the paper states it: build the sparse version of dY (one entry per map, the signed sum) and take
// its exact filter gradient with the tensor-core kernel.  (8x8 maps: the gather kernel is faster with 128 channels;
// with 256 the two tie alone and the dense route is cheaper among other layers, so it is taken from 256 channels on.)
bool top1_dense_route(const Geom& g, TcPlan* tp)
{
    return g.bf16 && ((g.p * g.q <= 16 && g.c >= 128) || (g.p * g.q <= 64 && g.c >= 256)) && plan_tc(g, tp);
}

struct Top1Layout { size_t idx_off, sum_off, partial_off, sparse_off, scratch_off, total; GatherPlan gp; TcPlan tp; ClPlan cp; bool dense, cl; };
Top1Layout build_top1_layout(const Geom& g, bool cl)
{
    Top1Layout L;
    L.gp = plan_gather(g);
    L.dense = top1_dense_route(g, &L.tp);
    // the contraction: by the channels-last kernel, which reads either form of the sparse tensor (256->256 on 8x8, N = 256:
    // 37 us with the other kernel, 32)
    L.cl = cl && L.dense && tensor_maps_available() && plan_cl(g, L.tp.reads_transposed_dy, kNoLimit, &L.cp) && !short_sums(g, L.cp);
    const size_t cl_scratch = L.cl ? L.cp.x_bytes[0] + L.cp.dy_bytes[0] : 0;
    const size_t maps = (size_t)g.n * g.k;
    L.idx_off = kWsDataOffset;
    L.sum_off = align_up(L.idx_off + maps * sizeof(int32_t), 256);
    L.partial_off = align_up(L.sum_off + maps * sizeof(float), 256);
    size_t partial = L.gp.partial_bytes;
    if (L.dense) partial = std::max(partial, L.cl ? L.cp.partial_bytes : L.tp.partial_bytes);
    L.sparse_off = align_up(L.partial_off + partial, 256);
    L.scratch_off = align_up(L.sparse_off + (L.dense ? maps * g.p * g.q * 2 : 0), 256);
    L.total = align_up(L.scratch_off + (L.dense ? L.tp.scratch_bytes + cl_scratch : 0), 256);
    return L;
}

// cl = false: without the channels-last kernel (workspaces that its packed operand does not fit)
Top1Layout top1_layout(const Geom& g, bool cl)
{
    static PlanCache<Top1Layout> cache;
    return cache.get(plan_key(g, cl, 0), [&] { return build_top1_layout(g, cl); });
}

// kernels other than the channels-last one; least: the scratch that the one taken cannot do without
enum class ExactKernel { tc, stem, mma, direct };
struct ExactLayout { size_t partial_off, scratch_off, total, least; DirectPlan dp; TcPlan tp; StemPlan sp; bool tc_ok, stem_ok, mma_ok; ExactKernel kernel; };
// fp32 inputs take the tcgen05 kernel (TF32 MMAs on split operands) where the layer is wide enough for the
// tensor cores to pay for the extra pass that splits the operands: 64 input channels, or 32 when the filter
// rows share one MMA (measured: 32->32@16x16 18.7 us against 19.9 us on the warp-level path; without the
// stacking 24 us); the one-pass TF32 mode needs no split
bool tc_f32_wanted(const Geom& g, int math, int algo) { return !g.bf16 && (math == GACONV_MATH_TF32 || algo == GACONV_ALGO_TENSOR || g.c >= 32); }

ExactLayout build_exact_layout(const Geom& g, int math, int algo)
{
    ExactLayout L;
    L.dp = plan_direct(g);
    L.tc_ok = g.bf16 ? plan_tc(g, &L.tp) : (tc_f32_wanted(g, math, algo) && plan_tc_f32(g, math == GACONV_MATH_TF32 ? 1 : 3, &L.tp));
    // (32 channels: only with stacked rows and operands small enough that writing and re-reading their split planes
    //  stays cheap -- 32->16@32x32 with 25 MB of inputs measured 36 us on this path)
    const size_t in_bytes = ((size_t)g.n * g.c * g.h * g.w + (size_t)g.n * g.k * g.p * g.q) * 4;
    if (L.tc_ok && !g.bf16 && g.c < 64 && (!L.tp.stacked_rows || in_bytes > ((size_t)12 << 20)) && math != GACONV_MATH_TF32 &&
        algo != GACONV_ALGO_TENSOR) L.tc_ok = false;
    L.partial_off = kWsDataOffset;
    size_t partial = L.dp.partial_bytes;
    if (L.tc_ok && L.tp.partial_bytes > partial) partial = L.tp.partial_bytes;
    L.stem_ok = plan_stem(g, &L.sp);
    if (L.stem_ok && L.sp.partial_bytes > partial) partial = L.sp.partial_bytes;
    L.scratch_off = align_up(L.partial_off + partial, 256);
    L.total = align_up(L.scratch_off + (L.tc_ok ? L.tp.scratch_bytes : 0), 256);
    L.mma_ok = direct_mma_supported(g, L.dp);
    const bool any = algo != GACONV_ALGO_DIRECT;
    L.kernel = L.tc_ok && any ? ExactKernel::tc : L.stem_ok && any && math == GACONV_MATH_DEFAULT ? ExactKernel::stem
             : L.mma_ok && (any || math == GACONV_MATH_TF32) ? ExactKernel::mma : ExactKernel::direct;
    L.least = L.kernel == ExactKernel::tc ? L.total
            : L.partial_off + (L.kernel == ExactKernel::stem ? L.sp.partial_bytes : L.kernel == ExactKernel::mma ? L.dp.partial_bytes : 0);
    return L;
}

ExactLayout exact_layout(const Geom& g, int math, int algo)
{
    static PlanCache<ExactLayout> cache;
    return cache.get(plan_key(g, math, algo), [&] { return build_exact_layout(g, math, algo); });
}

// Which problems the channels-last kernel takes: those the kernels above do not tile, and of the others those on which it
// measured faster (in microseconds, the older kernel first; N = 128 unless said).  `reordered`: X or dY comes in the other
// order than N x H x W x C / N x K x P x Q, which costs the older kernels a transposing pass and this one none or a cheaper one.
// ALGO_DIRECT, ALGO_TENSOR and the one-pass TF32 mode stay with the older kernels.
bool prefer_cl(const Geom& g, const ExactLayout& L, const ClPlan& plan, bool reordered)
{
    const double products = (double)g.n * g.p * g.q * g.k * g.c * g.r * g.s;
    const bool shared = g.sm_budget > 0;            // other layers run beside this one
    // (below 30 million products the order of the operands does not change the kernel, nor the result's last bits)
    reordered = reordered && products > 3e7;
    if (g.bf16) {
        if (L.tc_ok) {
            if (!reordered && short_sums(g, plan)) return false;
            // maps under 64 pixels: 512->512 on 4x4, N = 256 31.8 / 27.3, 128->16 on 4x8, N = 100 11.3 / 8.8; many input and few output
            // channels (partial blocks of mostly idle lanes) 192->16 on 4x8, N = 23 7.9 / 11.3, 256->16 on 4x4, N = 200 11.5 / 13.6
            if (L.tp.reads_transposed_dy) return products > 5e6 && (g.k > 32 || g.c <= 128);
            if (products < 3e7) return false;
            if (reordered) return true;                             // 128->128 on 16x16, dY channels last 28.4 / 17.8
            if (g.c <= 16 || (g.c < 64 && shared)) return false;    // 16->16 on 32x32 12.4 / 12.8; on 18 SMs 29 / 39
            // 64 channels on few SMs: the older kernel's M = 64 fits, this one's 128 lanes are half idle or its tiles shared, until the
            // main loop outweighs the rest (on 12 lanes beside copies of itself, us a layer: 64->64 on 8x8, N = 32 1.84 / 1.96,
            // N = 128 2.69 / 2.93, N = 256 3.90 / 3.96, N = 512 6.3 / 5.8; 64->40 on 16x16, N = 64 3.0 / 3.8; not with 16 outputs,
            // 64->16 on 16x16 3.8 / 3.4, nor at stride 2, 64->64 on 16x16 4.1 / 2.8; exact phase of a ResNet-20 step, N = 64, 128 and
            // 256, with the one and with the other: 55 / 60, 78 / 80, 106 / 113)
            if (shared && g.c <= 64 && g.k > 16 && g.k <= 64 && g.stride_h == 1 && products < 1e9) return false;
            // Filters of five and more rows: with few input channels this kernel stacks the rows or has its M side full of shifts
            // (5x5 on 16x16: 32->32 17.6 / 14.4, 40->64 25.0 / 18.1, 32->128 22.9 / 14.8, N = 32 32->64 18.1 / 10.4; 48->64 on 8x8 18.1 / 11.9;
            // 7x7 32->32 on 16x16 21.0 / 14.3; 24->24 13.9 / 14.3); with 64 and more it is for 5x5 as long as most of M = 128 outputs are in use
            // (on 16x16 64->88 17.1 / 19.0, 64->96 22.8 / 19.2, 128->128 36.5 / 28.9, on 8x8 256->256 49.0 / 35.7, N = 16 12.2 / 10.4, on 32x32
            // 64->128, N = 64 35.2 / 28.3; but 64->64 16.2 / 18.9), while wider ones are quicker on the older (7x7 64->128 31.2 / 32.4, 128->128
            // 47.7 / 66.3).  3x3 64->64 on 32x32 25.0 / 23.1
            return g.r < 5 || g.c < 64 || (g.r == 5 && g.s <= 5 && g.k >= 96);
        }
        // stems, those whose windows are gathered (on 32x32): beside others 3->64 3x3 N = 64 7.1 / 4.7, N = 256 16.7 / 13.4, 5x5 N = 16 4.2 / 2.5, but 3->16
        // N = 256 7.3 / 9.2; alone 3x3 3->64 N = 64 11.6 / 12.4, N = 128 15.5 / 15.1, N = 256 23.8 / 20.8, 3->16 N = 256 16.0 / 16.5, 5x5 3->64 N = 8
        // 9.4 / 11.8, N = 32 13.7 / 12.3, N = 128 26.5 / 15.4, 3->16 N = 64 11.0 / 13.2; 3x3 on 64x64 3->32 N = 84 21.5 / 22.9, on 96x96 1->16 N = 232
        // 39 / 54.  Not the plain form, which is left for strides: 5x5 3->40 on 64x64 at stride 2, N = 38, beside others 7.0 / 9.2, alone 1->128 on 96x96,
        // N = 50 23.3 / 34.2.  (Of 178 stems alone 3 are more than 5 % off the better kernel, 10 % at most.)
        if (L.stem_ok) return reordered || (plan.windows && (shared ? g.k > 32 && products > 5e7 : g.r * g.s * g.c > 32 ? products > 1.2e8 : g.k > 32 && products > 2e8));
    } else {
        // stems: 3x3 3->64 on 32x32 28.7 / 36.8; gathered windows of 5x5 filters of three channels 3->64 on 32x32, N = 116 44.0 / 37.2, N = 59 26.8 / 24.9,
        // N = 23 15.3 / 16.4, on 40x40, N = 61 36.5 / 36.2, 3->96 on 32x32, N = 58 34.5 / 28.9, but 3->48, N = 38 18.6 / 18.6, 3->40 on 64x64, N = 45 44.5 / 58.3;
        // fewer columns 4->128 3x3, N = 28 17.8 / 22.4, 2->96 5x5 on 48x48, N = 98 70 / 96; the plain form, at stride 2, 3->40 5x5 on 64x64, N = 170 60 / 138
        // (beside the second layer of the two-layer CNN, N = 200, the step takes 63 / 68)
        if (L.stem_ok) return !shared && plan.windows && g.r * g.s * g.c > 64 && g.k >= 64 && products > 1.2e8;
        // (the tensor core truncates as it adds, 1e-8 for each MMA of the other kernel's CTA: where that has more than 1,500 of them
        // its results are over 1.4e-5 away from this one's, and stay what they have been)
        if (L.tc_ok && L.tp.chain > 1500) return false;
        if (L.tc_ok)                                                // 128->128 on 16x16 89 / 53, 64->64 on 8x8 18.0 / 19.9, on 18 SMs 45 / 35
            return reordered || products > (g.c >= 128 ? 4e8 : shared ? 1e8 : g.c >= 64 ? 1e9 : 2e8);      // 32->32 on 16x16 19.3 / 17.7, on 18 SMs 43 / 36
        if (L.mma_ok)                                               // 16->16 on 32x32 20 / 24.5, 48->96 on 16x16 (N = 64) 31 / 25
            return (g.c >= 64 && products > 4e6) || (g.c >= 24 && g.stride_h == 1 && !shared && products > 3e8);       // (N = 16) 24->16 on 32x32 10 / 13.5
    }
    // FP32 pipes: their one or two launches are as quick while the work is small -- longer with 3x3 filters of fp32 layers, whose
    // operands must be packed (16->64 on 6x6, N = 30 launched one by one 10.3 / 12.3 us; 1x1 80->22 on 6x6, N = 105 25 / 12), and with three channels
    return products > (!g.bf16 && g.r * g.s >= 9 ? 2e7 : g.c <= 4 ? 1e7 : 4e6);
}
struct ClRoute {
    bool use;
    bool lean_first;        // without room for it: another plan of this kernel is quicker than the other kernels
    ClPlan plan;
    size_t partial_off, x_off, dy_off[2], total[2];       // [0] copies packed tightly, [1] on aligned rows
};
ClRoute build_cl_route(const gaconv_conv_desc_t* desc, const Geom& g, size_t limit)
{
    ClRoute R{};
    if (!tensor_maps_available() || limit < kWsDataOffset || !plan_cl(g, desc->dy_layout == GACONV_DY_NPQK, limit == kNoLimit ? limit : limit - kWsDataOffset, &R.plan)) return R;
    gaconv_conv_desc_t native = *desc;
    native.x_layout = GACONV_X_NHWC; native.dy_layout = GACONV_DY_NKPQ;
    Geom gn;
    if (make_geom(&native, &gn) != GACONV_OK) return R;
    const ExactLayout L = exact_layout(gn, GACONV_MATH_DEFAULT, GACONV_ALGO_AUTO);
    const bool reordered = (desc->x_layout == GACONV_X_NCHW && g.c > 1) || (desc->dy_layout == GACONV_DY_NPQK && g.k > 1);
    R.use = limit != kNoLimit || prefer_cl(gn, L, R.plan, reordered);
    R.lean_first = R.plan.windows && (!L.stem_ok || (g.bf16 && reordered));
#ifdef GACONV_TUNING
    if (const char* e = getenv("GACONV_CL")) R.use = atoi(e) != 0;
#endif
    R.partial_off = kWsDataOffset;
    R.x_off = align_up(R.partial_off + R.plan.partial_bytes, 256);
    for (int wide = 0; wide < 2; ++wide) {
        R.dy_off[wide] = R.x_off + R.plan.x_bytes[wide];
        R.total[wide] = R.dy_off[wide] + R.plan.dy_bytes[wide];
    }
    return R;
}
// limit (a multiple of 256 bytes, or kNoLimit): scratch that the route may use
ClRoute planned_route(const gaconv_conv_desc_t* desc, const Geom& g, size_t limit)
{
    static PlanCache<ClRoute> cache;
    return cache.get(plan_key(g, desc->dy_layout, limit == kNoLimit ? -1 : (int)(limit >> 8)), [&] { return build_cl_route(desc, g, limit); });
}
// The channels-last kernel takes a call given `given` bytes of scratch.  Where its plan does not fit, the other kernels come next, except for
// gathered stems whose other kernels first have to transpose an operand or are the FP32 pipes: the plain form, or fewer splits, needs less (7x7
// 2->48 on 34x31 maps, N = 30, by the estimate 1.4 times the cycles).
bool cl_route(const gaconv_conv_desc_t* desc, const Geom& g, size_t given, ClRoute* R)
{
    if (desc->math != GACONV_MATH_DEFAULT || desc->algo != GACONV_ALGO_AUTO) return false;
    *R = planned_route(desc, g, kNoLimit);
    if (!R->use || given >= R->total[0]) return R->use;
    if (!R->lean_first) return false;
    const double most = 3 * R->plan.cycles;
    *R = planned_route(desc, g, given & ~(size_t)255);
    return R->use && R->plan.cycles <= most;
}
// In place of an error, where no other kernel fits: fewer splits, or copies of fewer bytes
bool cl_last_route(const gaconv_conv_desc_t* desc, const Geom& g, size_t given, ClRoute* R)
{
    if (desc->math != GACONV_MATH_DEFAULT || desc->algo != GACONV_ALGO_AUTO) return false;
    *R = planned_route(desc, g, given & ~(size_t)255);
    return R->use;
}

// entries retained per map by the top-k method: desc->topk clamped to the map size; 0 = invalid
int topk_of(const gaconv_conv_desc_t* d, const Geom& g)
{
    if (d->topk < 1 || d->topk > GACONV_MAX_TOPK) return 0;
    const long long pq = (long long)g.p * g.q;
    return d->topk < pq ? d->topk : (int)pq;
}

struct TopkLayout { size_t idx_off, sum_off, partial_off, total; GatherPlan gp; };
TopkLayout topk_layout(const Geom& g, int topk)
{
    TopkLayout L;
    L.gp = plan_gather(g);
    const size_t maps = (size_t)g.n * g.k;
    L.idx_off = kWsDataOffset;
    L.sum_off = align_up(L.idx_off + maps * topk * sizeof(int32_t), 256);
    L.partial_off = align_up(L.sum_off + maps * sizeof(float), 256);
    L.total = align_up(L.partial_off + L.gp.partial_bytes, 256);
    return L;
}

gaconv_status_t check_ws(const gaconv_conv_desc_t* d, size_t need)
{
    if (d->workspace == nullptr) return GACONV_ERR_NULL_POINTER;
    if (!aligned16(d->workspace)) return GACONV_ERR_MISALIGNED;
    if (d->workspace_bytes < need) return GACONV_ERR_WORKSPACE_TOO_SMALL;
    return GACONV_OK;
}

uint64_t splitmix64(uint64_t x)
{
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// ---- operand layouts other than the kernels' own ---------------------------------------------------------------
// The fast kernels (tensor-core, stem, vectorised gather) read channels-last activations, and every kernel reads dY
// as N x K x P x Q.  An N x P x Q x K gradient (what a channels-last framework hands over) is always transposed into
// the tail of the workspace; an N x C x H x W input is transposed where a fast kernel serves the channels-last
// version of the problem, and read in place by the FP32-pipe and scalar-gather kernels otherwise (odd shapes,
// GACONV_ALGO_DIRECT).  The call then continues with an inner descriptor in the kernels' layouts whose workspace is
// the head of the caller's.
struct Relayout { size_t inner_bytes, inner_least; bool move_x, move_dy; gaconv_conv_desc_t inner; };
size_t x_bytes_of(const gaconv_conv_desc_t* d) { return (size_t)d->n * d->c * d->h * d->w * (d->in_dtype == GACONV_BF16 ? 2 : 4); }
size_t dy_bytes_of(const Geom& g) { return (size_t)g.n * g.k * g.p * g.q * (g.bf16 ? 2 : 4); }

// workspace of a call in the kernels' own dY layout (x in either layout); 0 with *ok = false when the descriptor is bad
// (cl: with the channels-last kernel in the dense route of top-1; the exact method's takes every layout and is not asked here)
size_t native_ws_bytes(const gaconv_conv_desc_t* desc, const Geom& g, int32_t method, bool cl, bool* ok)
{
    *ok = true;
    switch (method) {
        case GACONV_METHOD_EXACT: return exact_layout(g, desc->math, desc->algo).total;
        case GACONV_METHOD_TOP1: return top1_layout(g, cl).total;
        case GACONV_METHOD_TOPK: {
            const int t = topk_of(desc, g);
            if (t < 1) { *ok = false; return 0; }
            return topk_layout(g, t).total;
        }
        case GACONV_METHOD_ZERO:
        case GACONV_METHOD_RANDOM: return kWsDataOffset;
    }
    *ok = false;
    return 0;
}

// which operands move, and the inner call's workspace size; move_x == move_dy == false: the call runs as it is
Relayout plan_relayout(const gaconv_conv_desc_t* desc, int32_t method, bool cl)
{
    Relayout R{};
    R.inner = *desc;
    const bool reads_inputs = method == GACONV_METHOD_EXACT || method == GACONV_METHOD_TOP1 || method == GACONV_METHOD_TOPK;
    if (!reads_inputs) return R;
    R.move_dy = desc->dy_layout == GACONV_DY_NPQK && desc->k > 1;          // (one output channel: the two orders coincide)
    R.inner.dy_layout = GACONV_DY_NKPQ;
    if (desc->x_layout == GACONV_X_NCHW && desc->c >= 2 && desc->algo != GACONV_ALGO_DIRECT) {
        gaconv_conv_desc_t nhwc = R.inner;
        nhwc.x_layout = GACONV_X_NHWC;
        Geom gi;
        if (make_geom(&nhwc, &gi) == GACONV_OK) {
            if (method == GACONV_METHOD_EXACT) {
                const ExactLayout L = exact_layout(gi, desc->math, desc->algo);
                R.move_x = L.tc_ok || L.stem_ok || L.mma_ok;
            } else if (method == GACONV_METHOD_TOP1) {
                R.move_x = top1_layout(gi, cl).dense || (top1_fused_supported(gi) && gi.c % 4 == 0);
            } else {
                R.move_x = topk_of(desc, gi) >= 1 && top1_fused_supported(gi) && gi.c % 4 == 0;
            }
            if (R.move_x) R.inner = nhwc;
        }
    }
    if (R.move_x || R.move_dy) {
        Geom gi;
        bool ok = false;
        if (make_geom(&R.inner, &gi) == GACONV_OK) {
            R.inner_bytes = native_ws_bytes(&R.inner, gi, method, cl, &ok);
            R.inner_least = method == GACONV_METHOD_EXACT ? exact_layout(gi, R.inner.math, R.inner.algo).least : R.inner_bytes;
        }
        if (!ok) { R.move_x = R.move_dy = false; R.inner = *desc; R.inner_bytes = R.inner_least = 0; }
    }
    return R;
}

// the inner call's scratch, then the transposed copies
size_t copied_bytes(const gaconv_conv_desc_t* desc, const Geom& g, const Relayout& R)
{
    return (R.move_x ? align_up(x_bytes_of(desc), 256) : 0) + (R.move_dy ? dy_bytes_of(g) : 0);
}
size_t moved_ws_bytes(const gaconv_conv_desc_t* desc, const Geom& g, const Relayout& R) { return align_up(R.inner_bytes, 256) + copied_bytes(desc, g, R); }

// Transposes what has to move into the workspace tail and hands back the inner descriptor and operand pointers.
// *moved == false: nothing to do, the caller goes on with its own descriptor.
gaconv_status_t relayout_operands(const void* x, const void* dy, const gaconv_conv_desc_t* desc, int32_t method, cudaStream_t cs,
                                  gaconv_conv_desc_t* inner, const void** x_out, const void** dy_out, bool* moved)
{
    Relayout R = plan_relayout(desc, method, true);
    *moved = R.move_x || R.move_dy;
    if (!*moved) return GACONV_OK;
    Geom g;
    gaconv_status_t st = make_geom(desc, &g);
    if (st != GACONV_OK) return st;
    if (desc->workspace_bytes < moved_ws_bytes(desc, g, R)) R = plan_relayout(desc, method, false);
    const size_t x_tail = R.move_x ? align_up(x_bytes_of(desc), 256) : 0, copies = copied_bytes(desc, g, R);
    st = check_ws(desc, align_up(R.inner_least, 256) + copies);
    if (st != GACONV_OK) return st;
    const size_t head = std::min(align_up(R.inner_bytes, 256), (desc->workspace_bytes - copies) & ~(size_t)255);
    char* ws = static_cast<char*>(desc->workspace);
    *x_out = x; *dy_out = dy;
    if (R.move_x) {
        if (launch_transpose_batched(x, ws + head, g.c, g.h * g.w, g.n, g.bf16, cs) != cudaSuccess) return GACONV_ERR_CUDA;
        *x_out = ws + head;
    }
    if (R.move_dy) {
        if (launch_transpose_batched(dy, ws + head + x_tail, g.p * g.q, g.k, g.n, g.bf16, cs) != cudaSuccess) return GACONV_ERR_CUDA;
        *dy_out = ws + head + x_tail;
    }
    *inner = R.inner;
    inner->workspace_bytes = head;
    return GACONV_OK;
}

}  // namespace

struct gaconv_schedule {
    int32_t num_layers, kind, method;
    double fraction;
    uint64_t seed;
    bool* mask;   // SEEDED_FRACTION: layers in the approximated subset
    struct StepCache* steps = nullptr;      // repeated steps as CUDA graphs, created on first use
};

// scratch of a call, exact ones without the channels-last kernel
// (cl: the dense route of top-1 with it)
static gaconv_status_t other_workspace(const gaconv_conv_desc_t* desc, const Geom& g, int32_t method, bool cl, size_t given, size_t* bytes)
{
    const Relayout R = plan_relayout(desc, method, cl);
    if (R.move_x || R.move_dy) {
        *bytes = moved_ws_bytes(desc, g, R);
        if (*bytes > given) *bytes = align_up(R.inner_least, 256) + copied_bytes(desc, g, R);
        return GACONV_OK;
    }
    bool ok = false;
    const size_t need = native_ws_bytes(desc, g, method, cl, &ok);
    if (!ok) return GACONV_ERR_BAD_DESC;
    *bytes = need <= given || method != GACONV_METHOD_EXACT ? need : exact_layout(g, desc->math, desc->algo).least;
    return GACONV_OK;
}

gaconv_status_t gaconv::method_workspace(const gaconv_conv_desc_t* desc, int32_t method, size_t given, size_t* bytes)
{
    Geom g;
    gaconv_status_t st = make_geom(desc, &g);
    if (st != GACONV_OK) return st;
    const bool exact = method == GACONV_METHOD_EXACT;
    ClRoute C;
    if (exact && cl_route(desc, g, given, &C)) { *bytes = C.total[given >= C.total[1]]; return GACONV_OK; }
    st = other_workspace(desc, g, method, !exact, given, bytes);
    if (st != GACONV_OK || *bytes <= given) return st;
    if (!exact) return other_workspace(desc, g, method, false, given, bytes);
    if (cl_last_route(desc, g, given, &C)) *bytes = C.total[0];
    return GACONV_OK;
}

static gaconv_status_t run_cl(const void* x, const void* dy, float* dw, const gaconv_conv_desc_t* desc, const ClRoute& C, cudaStream_t stream)
{
    const gaconv_status_t st = check_ws(desc, C.total[0]);
    if (st != GACONV_OK) return st;
    const bool wide = desc->workspace_bytes >= C.total[1];
    char* ws = static_cast<char*>(desc->workspace);
    return launch_cl(x, dy, dw, reinterpret_cast<float*>(ws + C.partial_off), ws + C.x_off, ws + C.dy_off[wide],
                     reinterpret_cast<uint32_t*>(ws), C.plan, wide, stream) == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
}

// exact dW by the kernels other than the channels-last one
static gaconv_status_t run_others(const void* x, const void* dy, float* dw, const gaconv_conv_desc_t* desc, const Geom& g, cudaStream_t stream)
{
    gaconv_status_t st;
    if (desc->dy_layout == GACONV_DY_NPQK && g.k > 1 && desc->algo != GACONV_ALGO_DIRECT) {
        // Small maps: the tensor-core kernel's dY operand IS the channels-last order (its pre-pass would transpose an
        // N x K x P x Q gradient into it), so a channels-last gradient is read where it lies; only X may have to move.
        const Relayout R = plan_relayout(desc, GACONV_METHOD_EXACT, false);
        Geom gi;
        if (make_geom(&R.inner, &gi) == GACONV_OK) {
            const ExactLayout Li = exact_layout(gi, desc->math, desc->algo);
            if (Li.tc_ok && Li.tp.reads_transposed_dy) {
                const size_t head = align_up(Li.total, 256);
                st = check_ws(desc, head + (R.move_x ? x_bytes_of(desc) : 0));
                if (st != GACONV_OK) return st;
                char* ws = static_cast<char*>(desc->workspace);
                const void* xs = x;
                if (R.move_x) {
                    if (launch_transpose_batched(x, ws + head, g.c, g.h * g.w, g.n, g.bf16, stream) != cudaSuccess)
                        return GACONV_ERR_CUDA;
                    xs = ws + head;
                }
                cudaError_t e = launch_tc(xs, nullptr, dw, reinterpret_cast<float*>(ws + Li.partial_off), const_cast<void*>(dy),
                                          reinterpret_cast<uint32_t*>(ws + kWsCounterOffset), reinterpret_cast<uint32_t*>(ws), Li.tp,
                                          stream);
                return e == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
            }
        }
    }
    {
        gaconv_conv_desc_t inner;
        Geom gi;
        const void *xt = nullptr, *dyt = nullptr;
        bool moved = false;
        st = relayout_operands(x, dy, desc, GACONV_METHOD_EXACT, stream, &inner, &xt, &dyt, &moved);
        if (st != GACONV_OK) return st;
        if (moved) return make_geom(&inner, &gi) == GACONV_OK ? run_others(xt, dyt, dw, &inner, gi, stream) : GACONV_ERR_BAD_DESC;
    }
    const ExactLayout L = exact_layout(g, desc->math, desc->algo);
    if (desc->math == GACONV_MATH_TF32 && !L.mma_ok && !L.tc_ok) return GACONV_ERR_UNSUPPORTED;
    if (desc->algo == GACONV_ALGO_TENSOR && !L.tc_ok) return GACONV_ERR_UNSUPPORTED;
    st = check_ws(desc, L.least);
    if (st != GACONV_OK) return st;
    char* ws = static_cast<char*>(desc->workspace);
    if (L.kernel == ExactKernel::tc) {
        cudaError_t e = launch_tc(x, dy, dw, reinterpret_cast<float*>(ws + L.partial_off), ws + L.scratch_off,
                                  reinterpret_cast<uint32_t*>(ws + kWsCounterOffset), reinterpret_cast<uint32_t*>(ws), L.tp,
                                  stream);
        return e == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
    }
    if (L.kernel == ExactKernel::stem) {
        cudaError_t e = launch_stem(x, dy, dw, reinterpret_cast<float*>(ws + L.partial_off), reinterpret_cast<uint32_t*>(ws), L.sp,
                                    stream);
        return e == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
    }
    if (L.kernel == ExactKernel::mma) {
        cudaError_t e = launch_direct_mma(x, dy, dw, reinterpret_cast<float*>(ws + L.partial_off), reinterpret_cast<uint32_t*>(ws),
                                          g, L.dp, desc->math != GACONV_MATH_TF32, stream);
        return e == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
    }
    DirectPlan dp = L.dp;
    limit_direct(g, desc->workspace_bytes - L.partial_off, &dp);
    cudaError_t e = launch_direct(x, dy, dw, reinterpret_cast<float*>(ws + L.partial_off), reinterpret_cast<uint32_t*>(ws), g, dp, stream);
    return e == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
}

extern "C" {

const char* gaconv_status_string(gaconv_status_t s)
{
    switch (s) {
        case GACONV_OK: return "ok";
        case GACONV_ERR_NULL_POINTER: return "null pointer";
        case GACONV_ERR_BAD_DESC: return "bad descriptor";
        case GACONV_ERR_UNSUPPORTED: return "unsupported request";
        case GACONV_ERR_MISALIGNED: return "pointer not 16-byte aligned";
        case GACONV_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
        case GACONV_ERR_CUDA: return "CUDA error";
        case GACONV_ERR_TIMEOUT: return "device-side wait timed out";
    }
    return "unknown status";
}

uint64_t gaconv_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

gaconv_status_t gaconv_workspace_size(const gaconv_conv_desc_t* desc, int32_t method, size_t* bytes)
{
    if (bytes == nullptr) return GACONV_ERR_NULL_POINTER;
    return method_workspace(desc, method, kNoLimit, bytes);
}

gaconv_status_t gaconv_workspace_init(void* workspace, size_t bytes, void* stream)
{
    if (workspace == nullptr) return GACONV_ERR_NULL_POINTER;
    if (!aligned16(workspace)) return GACONV_ERR_MISALIGNED;
    if (bytes < kWsDataOffset) return GACONV_ERR_WORKSPACE_TOO_SMALL;
    if (cudaMemsetAsync(workspace, 0, kWsDataOffset, static_cast<cudaStream_t>(stream)) != cudaSuccess) return GACONV_ERR_CUDA;
    return GACONV_OK;
}

gaconv_status_t gaconv_dw_exact(const void* x, const void* dy, float* dw, const gaconv_conv_desc_t* desc, void* stream)
{
    Geom g;
    gaconv_status_t st = make_geom(desc, &g);
    if (st != GACONV_OK) return st;
    if (x == nullptr || dy == nullptr || dw == nullptr) return GACONV_ERR_NULL_POINTER;
    if (!aligned16(x) || !aligned16(dy) || !aligned16(dw)) return GACONV_ERR_MISALIGNED;
    if (desc->math == GACONV_MATH_TF32 && g.bf16) return GACONV_ERR_BAD_DESC;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    const size_t given = desc->workspace != nullptr ? desc->workspace_bytes : kNoLimit;
    ClRoute C;
    if (cl_route(desc, g, given, &C)) return run_cl(x, dy, dw, desc, C, cs);
    st = run_others(x, dy, dw, desc, g, cs);
    return st == GACONV_ERR_WORKSPACE_TOO_SMALL && cl_last_route(desc, g, given, &C) ? run_cl(x, dy, dw, desc, C, cs) : st;
}

gaconv_status_t gaconv_dw_approx(int32_t method, const void* x, const void* dy, float* dw,
                                 const gaconv_conv_desc_t* desc, uint64_t seed, void* stream)
{
    Geom g;
    gaconv_status_t st = make_geom(desc, &g);
    if (st != GACONV_OK) return st;
    if (dw == nullptr) return GACONV_ERR_NULL_POINTER;
    if (!aligned16(dw)) return GACONV_ERR_MISALIGNED;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    const size_t count = (size_t)g.k * g.c * g.r * g.s;
    if (method == GACONV_METHOD_ZERO) return launch_zero(dw, count, cs) == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
    if (method == GACONV_METHOD_RANDOM)
        return launch_random(dw, g, seed, desc->rand_std, cs) == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
    if (method != GACONV_METHOD_TOP1 && method != GACONV_METHOD_TOPK) return GACONV_ERR_BAD_DESC;
    if (x == nullptr || dy == nullptr) return GACONV_ERR_NULL_POINTER;
    if (!aligned16(x) || !aligned16(dy)) return GACONV_ERR_MISALIGNED;
    {
        gaconv_conv_desc_t inner;
        const void *xt = nullptr, *dyt = nullptr;
        bool moved = false;
        st = relayout_operands(x, dy, desc, method, cs, &inner, &xt, &dyt, &moved);
        if (st != GACONV_OK) return st;
        if (moved) return gaconv_dw_approx(method, xt, dyt, dw, &inner, seed, stream);
    }
    if (method == GACONV_METHOD_TOPK) {
        // selection of the topk largest magnitudes per map, then the patch accumulation over the retained entries
        const int t = topk_of(desc, g);
        if (t < 1) return GACONV_ERR_BAD_DESC;
        const TopkLayout L = topk_layout(g, t);
        st = check_ws(desc, L.total);
        if (st != GACONV_OK) return st;
        char* ws = static_cast<char*>(desc->workspace);
        int32_t* idx = reinterpret_cast<int32_t*>(ws + L.idx_off);
        float* sum = reinterpret_cast<float*>(ws + L.sum_off);
        if (launch_select_topk(dy, idx, sum, g, t, cs) != cudaSuccess) return GACONV_ERR_CUDA;
        // the one-launch kernel of the top-1 method, fed with the selected list (t records per image), where its
        // shared-memory block fits; else the ticketed gather kernel
        if (top1_fused_supported(g) && (size_t)g.n * t * 16 <= 48 * 1024 && desc->algo != GACONV_ALGO_DIRECT)   // (16 bytes per record)
            return launch_top1_fused(x, dy, dw, g, cs, idx, sum, t) == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
        if (launch_gather(x, idx, sum, dw, reinterpret_cast<float*>(ws + L.partial_off),
                          reinterpret_cast<uint32_t*>(ws + kWsCounterOffset), g, L.gp, t, cs) != cudaSuccess)
            return GACONV_ERR_CUDA;
        return GACONV_OK;
    }
    Top1Layout L = top1_layout(g, true);
    if (L.cl && desc->workspace_bytes < L.total) L = top1_layout(g, false);
    st = check_ws(desc, L.total);       // required by every route, so that behaviour does not depend on the kernel picked
    if (st != GACONV_OK) return st;
    char* ws = static_cast<char*>(desc->workspace);
    int32_t* idx = reinterpret_cast<int32_t*>(ws + L.idx_off);
    float* sum = reinterpret_cast<float*>(ws + L.sum_off);
    if (L.dense && desc->algo != GACONV_ALGO_DIRECT) {
        void* sparse = ws + L.sparse_off;
        if (L.tp.reads_transposed_dy) {       // the dense kernel's operand layout is written directly: no separate transpose
            if (launch_select_sparse_transposed(dy, ws + L.scratch_off, g, cs) != cudaSuccess) return GACONV_ERR_CUDA;
            sparse = nullptr;
        } else if (launch_select(dy, idx, sum, sparse, g, cs) != cudaSuccess) return GACONV_ERR_CUDA;
        if (L.cl) {
            char* packed = ws + L.scratch_off + L.tp.scratch_bytes;
            return launch_cl(x, sparse != nullptr ? sparse : ws + L.scratch_off, dw, reinterpret_cast<float*>(ws + L.partial_off), packed,
                             packed + L.cp.x_bytes[0], reinterpret_cast<uint32_t*>(ws), L.cp, false, cs) == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
        }
        return launch_tc(x, sparse, dw, reinterpret_cast<float*>(ws + L.partial_off), ws + L.scratch_off,
                         reinterpret_cast<uint32_t*>(ws + kWsCounterOffset), reinterpret_cast<uint32_t*>(ws), L.tp,
                         cs) == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
    }
    if (top1_fused_supported(g) && desc->algo != GACONV_ALGO_DIRECT)
        return launch_top1_fused(x, dy, dw, g, cs) == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
    if (launch_select(dy, idx, sum, nullptr, g, cs) != cudaSuccess) return GACONV_ERR_CUDA;
    if (launch_gather(x, idx, sum, dw, reinterpret_cast<float*>(ws + L.partial_off),
                      reinterpret_cast<uint32_t*>(ws + kWsCounterOffset), g, L.gp, 1, cs) != cudaSuccess)
        return GACONV_ERR_CUDA;
    return GACONV_OK;
}

gaconv_status_t gaconv_approx_select(const void* dy, int32_t* idx, float* sum, void* dy_sparse,
                                     const gaconv_conv_desc_t* desc, void* stream)
{
    Geom g;
    gaconv_status_t st = make_geom(desc, &g);
    if (st != GACONV_OK) return st;
    if (dy == nullptr || idx == nullptr || sum == nullptr) return GACONV_ERR_NULL_POINTER;
    if (desc->dy_layout == GACONV_DY_NPQK && g.k > 1) return GACONV_ERR_UNSUPPORTED;      // selection alone has no scratch to transpose into
    if (!aligned16(dy) || !aligned16(idx) || !aligned16(sum) || !aligned16(dy_sparse)) return GACONV_ERR_MISALIGNED;
    return launch_select(dy, idx, sum, dy_sparse, g, static_cast<cudaStream_t>(stream)) == cudaSuccess ? GACONV_OK
                                                                                                         : GACONV_ERR_CUDA;
}

gaconv_status_t gaconv_approx_select_topk(const void* dy, int32_t* idx, float* sum, const gaconv_conv_desc_t* desc, void* stream)
{
    Geom g;
    gaconv_status_t st = make_geom(desc, &g);
    if (st != GACONV_OK) return st;
    if (dy == nullptr || idx == nullptr || sum == nullptr) return GACONV_ERR_NULL_POINTER;
    if (desc->dy_layout == GACONV_DY_NPQK && g.k > 1) return GACONV_ERR_UNSUPPORTED;
    if (!aligned16(dy) || !aligned16(idx) || !aligned16(sum)) return GACONV_ERR_MISALIGNED;
    const int t = topk_of(desc, g);
    if (t < 1) return GACONV_ERR_BAD_DESC;
    return launch_select_topk(dy, idx, sum, g, t, static_cast<cudaStream_t>(stream)) == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
}

static gaconv_status_t dw_from_host(int32_t method, const void* x_host, const void* dy_host, float* dw_host,
                                    void* x_dev, void* dy_dev, float* dw_dev, const gaconv_conv_desc_t* desc,
                                    uint64_t seed, void* stream, bool wait)
{
    Geom g;
    gaconv_status_t st = make_geom(desc, &g);
    if (st != GACONV_OK) return st;
    if (dw_host == nullptr || dw_dev == nullptr) return GACONV_ERR_NULL_POINTER;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    const bool needs_inputs = method == GACONV_METHOD_EXACT || method == GACONV_METHOD_TOP1 || method == GACONV_METHOD_TOPK;
    // everything the compute call would reject is rejected here, before the first copy is enqueued
    if (method < GACONV_METHOD_EXACT || method > GACONV_METHOD_TOPK) return GACONV_ERR_BAD_DESC;
    if (!aligned16(dw_dev)) return GACONV_ERR_MISALIGNED;
    if (needs_inputs) {
        // both host inputs NULL: the staging buffers already hold this layer's inputs (an earlier call of the step copied them)
        if ((x_host == nullptr) != (dy_host == nullptr) || x_dev == nullptr || dy_dev == nullptr) return GACONV_ERR_NULL_POINTER;
        if (!aligned16(x_dev) || !aligned16(dy_dev)) return GACONV_ERR_MISALIGNED;
        if (method == GACONV_METHOD_EXACT && desc->math == GACONV_MATH_TF32 && g.bf16) return GACONV_ERR_BAD_DESC;
        size_t need = 0;
        st = method_workspace(desc, method, desc->workspace_bytes, &need);
        if (st != GACONV_OK) return st;
        st = check_ws(desc, need);
        if (st != GACONV_OK) return st;
        if (method == GACONV_METHOD_EXACT) {
            const ExactLayout L = exact_layout(g, desc->math, desc->algo);
            if (desc->math == GACONV_MATH_TF32 && !L.mma_ok && !L.tc_ok) return GACONV_ERR_UNSUPPORTED;
            if (desc->algo == GACONV_ALGO_TENSOR && !L.tc_ok) return GACONV_ERR_UNSUPPORTED;
        }
        const size_t eb = g.bf16 ? 2 : 4;
        if (x_host != nullptr &&
            (cudaMemcpyAsync(x_dev, x_host, (size_t)g.n * g.c * g.h * g.w * eb, cudaMemcpyHostToDevice, cs) != cudaSuccess ||
             cudaMemcpyAsync(dy_dev, dy_host, (size_t)g.n * g.k * g.p * g.q * eb, cudaMemcpyHostToDevice, cs) != cudaSuccess))
            return GACONV_ERR_CUDA;
    }
    st = method == GACONV_METHOD_EXACT ? gaconv_dw_exact(x_dev, dy_dev, dw_dev, desc, stream)
                                       : gaconv_dw_approx(method, x_dev, dy_dev, dw_dev, desc, seed, stream);
    if (st != GACONV_OK) return st;
    if (cudaMemcpyAsync(dw_host, dw_dev, (size_t)g.k * g.c * g.r * g.s * sizeof(float), cudaMemcpyDeviceToHost, cs) != cudaSuccess)
        return GACONV_ERR_CUDA;
    if (!wait) return GACONV_OK;
    return cudaStreamSynchronize(cs) == cudaSuccess ? GACONV_OK : GACONV_ERR_CUDA;
}

gaconv_status_t gaconv_dw_from_host(int32_t method, const void* x_host, const void* dy_host, float* dw_host,
                                    void* x_dev, void* dy_dev, float* dw_dev, const gaconv_conv_desc_t* desc,
                                    uint64_t seed, void* stream)
{
    return dw_from_host(method, x_host, dy_host, dw_host, x_dev, dy_dev, dw_dev, desc, seed, stream, true);
}

gaconv_status_t gaconv_dw_from_host_async(int32_t method, const void* x_host, const void* dy_host, float* dw_host,
                                          void* x_dev, void* dy_dev, float* dw_dev, const gaconv_conv_desc_t* desc,
                                          uint64_t seed, void* stream)
{
    return dw_from_host(method, x_host, dy_host, dw_host, x_dev, dy_dev, dw_dev, desc, seed, stream, false);
}

gaconv_status_t gaconv_poll_async_status(const gaconv_conv_desc_t* desc, void* stream)
{
    if (desc == nullptr || desc->workspace == nullptr) return GACONV_ERR_NULL_POINTER;
    if (desc->workspace_bytes < kWsDataOffset) return GACONV_ERR_WORKSPACE_TOO_SMALL;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    uint32_t word = 0;
    if (cudaMemcpyAsync(&word, desc->workspace, sizeof(word), cudaMemcpyDeviceToHost, cs) != cudaSuccess) return GACONV_ERR_CUDA;
    if (cudaStreamSynchronize(cs) != cudaSuccess) return GACONV_ERR_CUDA;
    if (word == 0) return GACONV_OK;
    if (cudaMemsetAsync(desc->workspace, 0, sizeof(word), cs) != cudaSuccess) return GACONV_ERR_CUDA;
    return GACONV_ERR_TIMEOUT;
}

// ---- approximation schedules ----------------------------------------------------------------

gaconv_status_t gaconv_schedule_create(gaconv_schedule_t** out, int32_t num_layers, int32_t kind, int32_t method,
                                       double fraction, uint64_t seed)
{
    if (out == nullptr) return GACONV_ERR_NULL_POINTER;
    *out = nullptr;
    if (num_layers < 1 || num_layers > (1 << 20)) return GACONV_ERR_BAD_DESC;
    if (kind < GACONV_SCHED_EVERY_4TH_LAYER || kind > GACONV_SCHED_SEEDED_FRACTION_ALT_BATCH) return GACONV_ERR_BAD_DESC;
    if (method != GACONV_METHOD_ZERO && method != GACONV_METHOD_RANDOM && method != GACONV_METHOD_TOP1 && method != GACONV_METHOD_TOPK)
        return GACONV_ERR_BAD_DESC;
    if (!(fraction >= 0.0 && fraction <= 1.0)) return GACONV_ERR_BAD_DESC;
    gaconv_schedule* s = new (std::nothrow) gaconv_schedule{num_layers, kind, method, fraction, seed, nullptr};
    if (s == nullptr) return GACONV_ERR_BAD_DESC;
    if (kind == GACONV_SCHED_SEEDED_FRACTION_ALT_BATCH) {
        s->mask = new (std::nothrow) bool[num_layers]();
        uint64_t* hash = new (std::nothrow) uint64_t[num_layers];
        if (s->mask == nullptr || hash == nullptr) { delete[] s->mask; delete[] hash; delete s; return GACONV_ERR_BAD_DESC; }
        for (int l = 0; l < num_layers; ++l) hash[l] = splitmix64(seed + (uint64_t)l);
        int m = (int)(fraction * num_layers + 0.5);
        if (m > num_layers) m = num_layers;
        // a layer is chosen when fewer than m layers precede it in (hash, index) order
        for (int l = 0; l < num_layers; ++l) {
            int before = 0;
            for (int o = 0; o < num_layers; ++o)
                if (hash[o] < hash[l] || (hash[o] == hash[l] && o < l)) ++before;
            s->mask[l] = before < m;
        }
        delete[] hash;
    }
    *out = s;
    return GACONV_OK;
}

int32_t gaconv_schedule_method(const gaconv_schedule_t* s, int32_t layer, int64_t step)
{
    if (s == nullptr || layer < 0 || layer >= s->num_layers || step < 0) return -2;
    const int one_based = layer + 1;
    bool approx = false;
    switch (s->kind) {
        case GACONV_SCHED_EVERY_4TH_LAYER: approx = one_based >= 2 && (one_based - 2) % 4 == 0; break;
        case GACONV_SCHED_ALT_LAYER_ALT_BATCH: approx = one_based % 2 == 0 && step % 2 == 1; break;
        case GACONV_SCHED_ALL_LAYERS_EVERY_4TH_BATCH: approx = step % 4 == 3; break;
        case GACONV_SCHED_LAYER2_ALT_BATCH: approx = one_based == 2 && step % 2 == 1; break;
        case GACONV_SCHED_SEEDED_FRACTION_ALT_BATCH: approx = step % 2 == 1 && s->mask[layer]; break;
    }
    return approx ? s->method : GACONV_METHOD_EXACT;
}

// seed of a random-gradient layer at a step
static uint64_t layer_seed(const gaconv_schedule_t* s, int64_t step, int32_t layer)
{
    return splitmix64(s->seed ^ splitmix64((uint64_t)step * 0x100000001B3ull + (uint64_t)layer));
}

gaconv_status_t gaconv_schedule_run_layer(const gaconv_schedule_t* s, int32_t layer, int64_t step, const void* x,
                                          const void* dy, float* dw, const gaconv_conv_desc_t* desc, void* stream)
{
    const int32_t m = gaconv_schedule_method(s, layer, step);
    if (m == -2) return GACONV_ERR_BAD_DESC;
    if (m == GACONV_METHOD_EXACT) return gaconv_dw_exact(x, dy, dw, desc, stream);
    return gaconv_dw_approx(m, x, dy, dw, desc, layer_seed(s, step, layer), stream);
}

// ---- lanes: side streams on which the layers of a step run next to one another ----------------------
namespace {

constexpr int kMaxLanes = 16, kMaxLaneDevices = 64;
struct LanePool {
    bool ready = false;
    int device = -1;
    cudaStream_t side[kMaxLanes - 1] = {};
    cudaStream_t record = nullptr;                  // lane 0 of a step that is being recorded as a graph
    cudaEvent_t fork = nullptr, join[kMaxLanes - 1] = {};
};
std::mutex g_lane_mutex;
LanePool g_lanes[kMaxLaneDevices];

// streams and events of the current device, created on first use (host objects; no device memory)
LanePool* lane_pool()
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxLaneDevices) return nullptr;
    LanePool& p = g_lanes[dev];
    if (!p.ready) {
        p.device = dev;
        if (cudaEventCreateWithFlags(&p.fork, cudaEventDisableTiming) != cudaSuccess ||
            cudaStreamCreateWithFlags(&p.record, cudaStreamNonBlocking) != cudaSuccess) return nullptr;
        for (int i = 0; i < kMaxLanes - 1; ++i)
            if (cudaStreamCreateWithFlags(&p.side[i], cudaStreamNonBlocking) != cudaSuccess ||
                cudaEventCreateWithFlags(&p.join[i], cudaEventDisableTiming) != cudaSuccess) return nullptr;
        p.ready = true;
    }
    return &p;
}

}  // namespace

// ---- repeated steps ------------------------------------------------------------------------------------------------
// A step of a ResNet-20 is some fifty launches and event operations, 120-190 us of host time where the kernels take 40-80 us
// at small batches.  A training program calls run_step with the same buffers, descriptors and methods over and over, so the
// second time a schedule sees a step it is recorded as a CUDA graph, and from then on one graph launch enqueues it.  What the
// graph does not fix are the seeds of random-gradient layers, which change every step: their nodes get new ones before each
// launch.  A schedule keeps the kMaxSteps most recently used graphs; they go with it.
constexpr int kMinGraphLayers = 6;
struct StepKey {
    std::vector<unsigned char> bytes;
    void put(const void* p, size_t n) { const unsigned char* b = static_cast<const unsigned char*>(p); bytes.insert(bytes.end(), b, b + n); }
};
struct RandomNode { cudaGraphNode_t node; int32_t layer; int key_arg; };
struct StepGraph {
    std::vector<unsigned char> key;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;        // nullptr: seen once
    bool refused = false;                  // could not be recorded
    int launches = 0;
    int64_t step = -1;                     // whose seeds the graph holds
    std::vector<RandomNode> random;
    uint64_t used = 0;
};
struct StepCache {
    static constexpr size_t kMaxSteps = 8;
    std::vector<StepGraph> e;
    uint64_t clock = 0;
    static void drop(StepGraph& g)
    {
        if (g.exec != nullptr) cudaGraphExecDestroy(g.exec);      // (a graph still running is freed when it completes)
        if (g.graph != nullptr) cudaGraphDestroy(g.graph);
    }
    ~StepCache() { for (StepGraph& g : e) drop(g); }
};

// enqueues the layers of a step on the lanes; with `random`, notes the graph nodes of random-gradient layers (while capturing)
static gaconv_status_t enqueue_step(const gaconv_schedule_t* s, int64_t step, int32_t num_layers, const void* const* x, const void* const* dy,
                                    float* const* dw, const gaconv_conv_desc_t* const* descs, int32_t lanes, cudaStream_t main_stream,
                                    LanePool* pool, std::vector<RandomNode>* random)
{
    const int used = lanes < num_layers ? lanes : num_layers;
    // fork: the side streams start after everything already enqueued on the caller's stream
    if (used > 1) {
        if (cudaEventRecord(pool->fork, main_stream) != cudaSuccess) return GACONV_ERR_CUDA;
        for (int i = 0; i < used - 1; ++i)
            if (cudaStreamWaitEvent(pool->side[i], pool->fork, 0) != cudaSuccess) return GACONV_ERR_CUDA;
    }
    gaconv_status_t result = GACONV_OK;
    for (int l = 0; l < num_layers && result == GACONV_OK; ++l) {
        const int lane = l % used;
        cudaStream_t st = lane == 0 ? main_stream : pool->side[lane - 1];
        result = gaconv_schedule_run_layer(s, l, step, x[l], dy[l], dw[l], descs[l], st);
        if (result == GACONV_OK && random != nullptr && gaconv_schedule_method(s, l, step) == GACONV_METHOD_RANDOM) {
            cudaStreamCaptureStatus status;
            const cudaGraphNode_t* deps = nullptr;
            const cudaGraphEdgeData* edges = nullptr;
            cudaGraph_t graph;
            size_t n = 0;
            Geom g;
            if (cudaStreamGetCaptureInfo_v3(st, &status, nullptr, &graph, &deps, &edges, &n) != cudaSuccess || n != 1 || make_geom(descs[l], &g) != GACONV_OK)
                result = GACONV_ERR_CUDA;
            else
                random->push_back(RandomNode{deps[0], l, random_key_arg(g)});
        }
    }
    // join (also after an error, so that the side streams never stay forked from a capturing stream)
    for (int i = 0; i < used - 1; ++i)
        if (cudaEventRecord(pool->join[i], pool->side[i]) != cudaSuccess || cudaStreamWaitEvent(main_stream, pool->join[i], 0) != cudaSuccess)
            return GACONV_ERR_CUDA;
    return result;
}

// gives the random-gradient layers of a recorded step the seeds of `step`
static bool set_seeds(const gaconv_schedule_t* s, StepGraph& g, int64_t step)
{
    for (const RandomNode& r : g.random) {
        cudaKernelNodeParams p;
        if (cudaGraphKernelNodeGetParams(r.node, &p) != cudaSuccess) return false;
        const uint64_t seed = layer_seed(s, step, r.layer);
        uint32_t key0 = (uint32_t)seed, key1 = (uint32_t)(seed >> 32);
        void* args[8];
        for (int i = 0; i < r.key_arg + 3; ++i) args[i] = p.kernelParams[i];      // (the keys are followed by one more argument)
        args[r.key_arg] = &key0; args[r.key_arg + 1] = &key1;
        p.kernelParams = args;
        if (cudaGraphExecKernelNodeSetParams(g.exec, r.node, &p) != cudaSuccess) return false;
    }
    g.step = step;
    return true;
}

gaconv_status_t gaconv_schedule_run_step(const gaconv_schedule_t* s, int64_t step, int32_t num_layers, const void* const* x,
                                         const void* const* dy, float* const* dw, const gaconv_conv_desc_t* const* descs,
                                         int32_t lanes, void* stream)
{
    if (s == nullptr || x == nullptr || dy == nullptr || dw == nullptr || descs == nullptr) return GACONV_ERR_NULL_POINTER;
    if (num_layers < 1 || num_layers > s->num_layers || step < 0 || lanes < 1 || lanes > kMaxLanes) return GACONV_ERR_BAD_DESC;
    for (int l = 0; l < num_layers; ++l) {
        if (descs[l] == nullptr) return GACONV_ERR_NULL_POINTER;
        // layers that run next to one another must not share scratch
        if (lanes > 1 && descs[l]->workspace != nullptr)
            for (int o = 0; o < l; ++o)
                if (descs[o]->workspace == descs[l]->workspace) return GACONV_ERR_BAD_DESC;
    }
    cudaStream_t main_stream = static_cast<cudaStream_t>(stream);
    std::lock_guard<std::mutex> lock(g_lane_mutex);          // one set of lanes per device: enqueueing is serialised
    LanePool* pool = lane_pool();
    if (pool == nullptr) return GACONV_ERR_CUDA;
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    // Few layers: their launches cost the host less (~6 us a layer) than a graph's start and end cost the GPU between two steps
    // (two layers of the two-layer CNN at N = 256: 49 us launched, 65 us as a graph).  A capture in progress records the
    // launches themselves.
    if (num_layers < kMinGraphLayers || cudaStreamIsCapturing(main_stream, &capturing) != cudaSuccess || capturing != cudaStreamCaptureStatusNone)
        return enqueue_step(s, step, num_layers, x, dy, dw, descs, lanes, main_stream, pool, nullptr);

    // everything the recorded launches depend on
    // (without host memory for it, or for the cache, a step is enqueued and not kept)
    StepKey key;
    if (s->steps == nullptr) const_cast<gaconv_schedule*>(s)->steps = new (std::nothrow) StepCache;
    StepCache* cache = s->steps;
    try {
        key.bytes.reserve((size_t)num_layers * (sizeof(gaconv_conv_desc_t) + 3 * sizeof(void*) + 4) + 64);
        const int32_t head[3] = {pool->device, lanes, num_layers};
        key.put(head, sizeof(head));
        for (int l = 0; l < num_layers; ++l) {
            const int32_t method = gaconv_schedule_method(s, l, step);
            const void* ptrs[3] = {x[l], dy[l], dw[l]};
            key.put(&method, sizeof(method)); key.put(ptrs, sizeof(ptrs)); key.put(descs[l], sizeof(*descs[l]));
        }
    } catch (const std::bad_alloc&) { cache = nullptr; }
    StepGraph* g = nullptr;
    if (cache != nullptr) {
        for (StepGraph& c : cache->e)
            if (c.key == key.bytes) { g = &c; break; }
        if (g != nullptr) g->used = ++cache->clock;
    }
    if (g == nullptr || g->refused) {
        const gaconv_status_t st = enqueue_step(s, step, num_layers, x, dy, dw, descs, lanes, main_stream, pool, nullptr);
        if (st == GACONV_OK && g == nullptr && cache != nullptr) {      // a step that may come again
            if (cache->e.size() >= StepCache::kMaxSteps) {
                size_t oldest = 0;
                for (size_t i = 1; i < cache->e.size(); ++i)
                    if (cache->e[i].used < cache->e[oldest].used) oldest = i;
                StepCache::drop(cache->e[oldest]);
                cache->e.erase(cache->e.begin() + oldest);
            }
            try {
                cache->e.emplace_back();
                cache->e.back().key = std::move(key.bytes);
                cache->e.back().used = ++cache->clock;
            } catch (const std::bad_alloc&) { }
        }
        return st;
    }
    if (g->exec == nullptr) {
        const uint64_t before = gaconv_launch_count();
        gaconv_status_t st = GACONV_ERR_CUDA;
        g->random.clear();
        try { g->random.reserve(num_layers); } catch (const std::bad_alloc&) {      // (nothing is allocated while the step is recorded)
            return enqueue_step(s, step, num_layers, x, dy, dw, descs, lanes, main_stream, pool, nullptr);
        }
        if (cudaStreamBeginCapture(pool->record, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
            st = enqueue_step(s, step, num_layers, x, dy, dw, descs, lanes, pool->record, pool, &g->random);
            if (cudaStreamEndCapture(pool->record, &g->graph) != cudaSuccess) st = GACONV_ERR_CUDA;
        }
        if (st == GACONV_OK && cudaGraphInstantiate(&g->exec, g->graph, 0) != cudaSuccess) { g->exec = nullptr; st = GACONV_ERR_CUDA; }
        g->launches = (int)(gaconv_launch_count() - before);
        note_launch(-g->launches);              // recorded, not launched
        g->step = step;
        if (st != GACONV_OK) {
            (void)cudaGetLastError();
            StepCache::drop(*g);
            g->graph = nullptr; g->exec = nullptr; g->refused = true;
            return enqueue_step(s, step, num_layers, x, dy, dw, descs, lanes, main_stream, pool, nullptr);
        }
    }
    if (g->step != step && !set_seeds(s, *g, step)) {
        (void)cudaGetLastError();
        g->refused = true;
        return enqueue_step(s, step, num_layers, x, dy, dw, descs, lanes, main_stream, pool, nullptr);
    }
    if (cudaGraphLaunch(g->exec, main_stream) != cudaSuccess) return GACONV_ERR_CUDA;
    note_launch(g->launches);
    return GACONV_OK;
}

void gaconv_schedule_destroy(gaconv_schedule_t* s)
{
    if (s == nullptr) return;
    delete s->steps;
    delete[] s->mask;
    delete s;
}

}  // extern "C"
