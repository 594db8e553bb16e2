// Exact filter gradient on tcgen05 for any map, channel count, stride and layout: an implicit GEMM whose two
// operands are channels-last bf16 tensors, X as [n][h][w][c] and dY as [n][p][q][k].
//
//   dW[k, r, s, c] = alpha * sum_{n,p,q} dY[n,p,q,k] * Xz[n, p*st+r-pad, q*st+s-pad, c]         (Section 2.4)
//
// Why channels last for both: a pixel is then one row of shared memory (up to 64 channels = 128 bytes), both MMA
// operands are MN-major, and the reduction index (pixels) walks over rows.  A filter shift is a descriptor offset of
// whole rows, whatever the map's width, so no map size is special; the copy engine's zero fill supplies the padding,
// the ragged edges and the channels past the end.  Operands that are not in that form are brought into it by one
// packing pass into the workspace (pack_kernel): N x C x H x W activations, N x K x P x Q gradients, channel counts
// that are no multiple of 8, and fp32 inputs, which become three bf16 planes x = x0 + x1 + x2 (8 + 8 + 8 bits).  The
// fp32 product is then the six plane products of weight 2^-16 and more; what is left out is below 2^-23 of it.
//
// Reduction order inside a chunk (a few image rows, or several whole images), in k-steps of 16 pixels:
//   flat    rows of pitch Wp = Q + halo columns, walked end to end; dY is loaded with the same pitch, its columns past
//           Q reading as zeros.  Works for every Q; wastes (Wp - Q) / Q of the k-steps.
//   paired  Q a multiple of 8: a k-step is 8 columns of two neighbouring rows (the stride between the two 8-pixel
//           groups of a descriptor is one row), so that the halo columns are never multiplied.
// pixels  dY as it lies, N x K x P x Q (K-major rows of 64 pixels, Q a multiple of 8): a k-step is 16 consecutive pixels of an
//           image, no halo columns and no packing of dY.  Its two groups of 8 X pixels lie 8 pixels apart, or a row's end further,
//           so the X descriptor's stride belongs to the k-step.
//   images  (small or odd maps, many images) rows ordered (pixel, image): tensor maps with permuted dimensions deliver, for every
//           pixel of a band, the rows of `ci` images.  A column shift is then ci rows; a k-step is 16 images of a pixel (ci = 8:
//           of two pixels), no halo column is ever multiplied, and filter rows that fall outside the map are skipped.  The k-side
//           form at stride 1 does not even load halo columns: at the edge of the map its MMAs take fewer column shifts.
// A table of the plan holds the offsets of the k-steps of every order.
//
// Which operand is the MMA's M side:
//   k-side  M = 128 output channels, N = consecutive column shifts x channels (up to 256).  Every MMA has the N that its shifts need: at
//           stride 2 a 3x3 filter takes two shifts of the even columns and one of the odd, 128 + 64 accumulator columns, where two
//           equal MMAs would overrun them (fp32 64->128 on 28x28, N = 64: bound by the operands' reads of c-side MMAs of N = 64 before,
//           30.9 -> 27.4 us).  Filters too wide for 64 channels a tile take 32 or 16 (c-side MMAs of N = 32 to 64 before, bound the same
//           way; bf16 5x5 72->200 on 15x15, N = 60 39 -> 29, fp32 216 -> 124, fp32 7x7 160->120 on 21x21, N = 20 466 -> 111).
//   c-side  (few output channels) M = 128 = shifts x channels of X, N = output channels; M = 64 MMAs would take as
//           long as M = 128 ones, so with K <= 64 this form is the faster one although one shift in four is unused.
//           Filters of one column have filter rows in place of the shifts (row_atoms): the X operand's atoms lie one map row apart.
//   stack   (at most 64 output channels, stride 1) M = 128 = filter rows x output channels: the reduction walks over rows of X, and
//           the channel atoms of the dY operand lie one map row apart, so that atom j is the gradient row that meets this X row
//           in filter row r_hi - j.  One MMA does the work of two to eight whose M would be mostly idle.
//           (Bound by the tensor core: fp32 5x5 64->64 on 16x16, N = 128 53 -> 42 us, bf16 5x5 144->16 on 63x63, N = 16 43 -> 21.)
// The MMAs of one k-step differ only in the X offset and the accumulator columns; the list of them is part of the plan.
//
// CTA = one tile of dW (k-tile x c-tile x filter rows) and a contiguous range of chunks.  Its accumulator block goes to
// the workspace as [column][128 lanes] and cl_reduce_kernel adds the splits in order, so results are the same from run to run.
// (Adding them over a thread-block cluster's shared memory instead costs more: reads from other SMs came to ~10 bytes a cycle,
// where the workspace takes 21, and clusters of six leave SMs idle: 256->256 on 8x8, N = 128 19.1 us against 18.8.)
//
// Values that are not finite.  An Inf has no planes to split into (x - x0 = Inf - Inf), and the zero dY rows that end a chunk meet
// real X rows, so that an Inf or NaN there reaches elements it has no part in.  But nothing is hidden: what has an infinite or
// NaN product among those it should have comes out of the tensor core not finite.  So the writers look at every element, and
// those that are not finite are summed anew, product by product from the operands as they were handed over (cl_repair).  The look costs
// nothing where a second kernel writes dW; where this one does, ~0.2 us (exact phase of a VGG-19 step 171.3 -> 173.5 us; eight chains of
// additions, three-operand maxima or the repair in line instead of a call came to the same).
// (What may be missing are products of the padding with an Inf or NaN in dY: the orders and forms that skip the padding skip them.)
//
// Every wait is bounded; on expiry the kernel raises the workspace status word, lets its copies land, frees its tensor
// memory and returns.
#include <cuda.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "gaconv_internal.h"
#include "tma.cuh"
#include "umma.cuh"

// tuning builds: per CTA of the last launch, SM cycles of {entry, dependency, first data, issue done, accumulators done, exit},
// and the cycles the issuer waited for data / the producer for a free stage
#ifdef GACONV_TUNING
__device__ long long gaconv_tuning_cl[512][8];
#define GACONV_STAMP(slot, cond) do { if (cond) gaconv_tuning_cl[(blockIdx.y * gridDim.x + blockIdx.x) & 511][slot] = clock64(); } while (0)
#define GACONV_TALLY(slot, v) do { gaconv_tuning_cl[(blockIdx.y * gridDim.x + blockIdx.x) & 511][slot] = (v); } while (0)
#define GACONV_CLOCK() clock64()
#else
#define GACONV_STAMP(slot, cond) do { } while (0)
#define GACONV_TALLY(slot, v) do { } while (0)
#define GACONV_CLOCK() 0
#endif

namespace gaconv {
namespace {

constexpr int kMaxCols = 192;                   // accumulator columns of a CTA
constexpr int kMaxGroups = kMaxCols / 16, kMaxKsteps = 128, kMaxStages = 8;

// order of the reduction inside a chunk, see above
enum { kFlat = 0, kPaired = 1, kPixels = 2, kImages = 3 };

struct ClGroup {            // one MMA of a k-step
    int x_off;              // offset of its X rows inside the X region of a stage, 16-byte units
    int r, s0, cnt, cbase;  // filter row, first column shift, atoms in use, first channel (relative to the c-tile)
    int col, n;             // its first accumulator column, and how many it has
    uint32_t idesc;         // n in the instruction descriptor's place
};

struct ClShape {
    int n, c, h, w, k, r, s, p, q, stride, pad_h, pad_w;
    long long ws_k, ws_c, ws_r, ws_s;
    int vc, vw, vpad;               // few channels (vc, else 0): the problem is one of s = 1, whose c channels are the vc channels of every column
                                    // of a window in turn; columns of X and padding as the caller has them
    float alpha;
    int tiles_k, tiles_c, tiles_r, splits, chunk_base, chunk_rem, chunks;
    int ci, bp, cpi;                // chunk = ci whole images, or bp output rows of one; chunks per image
    int kt, rc, ct;                 // output channels, filter rows and channels per tile
    int ka, katoms, ca, na;         // channels per atom (one shared-memory row) and atoms per tile, dY and X
    int planes, nprod;              // bf16: 1, 1; fp32: 3, 6
    int phases, row_tiles;          // X tiles per chunk and atom: column phases x filter rows (stride > 1), else 1 x 1
    int dy_box, dy_alloc, x_box, x_alloc;       // bytes one copy writes, and the distance to the next tile
    int x_region, x_plane, dy_plane, stage_bytes, stages;
    uint32_t tx_bytes;
    int order, ksteps, x_pitch, dy_pitch, x_img, dy_img;
    int dy_subs;                    // kPixels: 64-pixel boxes of dY per image of a chunk
    int px_rows;                    // kImages: rows of a pixel (images); else 1
    int x_pre;                      // bytes of zeros before an X tile (kImages without halo columns; else 0)
    int skip;                       // kImages, whole maps, one filter row a tile: k-steps per map row, to leave out rows opposite the padding
    int c_side;                     // 1: X is the M side
    int slack;                      // bytes behind the last stage that MMAs may read
    int row_atoms;                  // c-side, one column: the atoms of the X operand are filter rows, one map row apart
    int stack;                      // 1: filter rows x output channels are the M side; chunks are bands of X rows
    int s_inner;                    // 1: column shifts lie next to one another in dW (K x C x R x S): columns are written shift by shift
    int merged;                     // 1: the MN atoms of an X operand are channel atoms, 0: column shifts
    int ngroups, cols, tmem_cols;
    int mma_cols;                   // columns of all MMAs of a chunk and product
    int epoch;                      // chunks of one issuer between two readings of its accumulators
    uint32_t dy_hi, x_lbo, dy_lbo, idesc;
    ClGroup g[kMaxGroups];
};
struct ClParams : ClShape {
    // k-step -> offsets of its X and dY rows (16-byte units), upper word of its X descriptor, and, with one k-side MMA a k-step,
    // the first column of that MMA | its N in the instruction descriptor's place (0 << 17 in idesc)
    uint4 k_off[kMaxKsteps];
};

// fp32 operands: which planes of X and dY each of the six products of a k-step takes
__device__ constexpr uint32_t prod_x(int i) { return i == 1 ? 2u : (i == 2 || i == 4) ? 1u : 0u; }
__device__ constexpr uint32_t prod_dy(int i) { return i == 0 ? 2u : (i == 2 || i == 3) ? 1u : 0u; }

// The MMA that writes a column
__device__ __forceinline__ int group_of(const ClShape& P, int col)
{
    int g = 0;
    while (g + 1 < P.ngroups && col >= P.g[g + 1].col) ++g;
    return g;
}
// The e-th column of a k-side block in the order of dW: where the shifts of a channel are neighbours in memory, shift by shift,
// so that a store of 32 lanes touches 13 sectors instead of 32 (K x C x R x S, 512->512 on 2x2 maps: the stores were 12 of 24 us).
__device__ __forceinline__ int written_column(const ClShape& P, int e)
{
    if (P.c_side || !P.s_inner) return e;
    const ClGroup& g = P.g[group_of(P, e)];
    const int j = e - g.col, atoms = g.n / P.ca, c = j / atoms;
    return g.col + (j - c * atoms) * P.ca + c;
}
// Element (column, lane) of a block that goes to dW directly, in words: [column][128], the lanes of a column exchanged by a key, so that neither a column's
// lanes, nor a lane's columns, nor the shifts of a channel meet in one bank.
__device__ __forceinline__ int block_key(int col, int ca_log) { return (col + 11 * (col >> ca_log)) & 31; }
// offset of a channel in dW
__device__ __forceinline__ long long channel_offset(const ClShape& P, int c)
{
    if (P.vc == 0) return c * P.ws_c;
    const int s = c / P.vc;
    return (c - s * P.vc) * P.ws_c + s * P.ws_s;
}
// c-side: distance in dW from one atom of the M side to the next
__device__ __forceinline__ long long atom_step(const ClShape& P) { return P.row_atoms ? P.ws_r : P.stride * P.ws_s; }
// Column -> {offset in dW, atoms in use (0: not an element)}
// (stack: without the filter row, which belongs to the lane)
__device__ __forceinline__ int2 column_target(const ClShape& P, int col, int k0, int c0, int r0)
{
    const ClGroup& g = P.g[group_of(P, col)];
    const int j = col - g.col;
    const int a = P.c_side || P.merged ? 0 : j / P.ca, k = P.c_side ? k0 + j : 0;
    const int c = c0 + g.cbase + (P.c_side ? 0 : P.merged ? j : j - a * P.ca);
    const bool valid = r0 + g.r < P.r && (P.c_side ? k < P.k : c < P.c && a < g.cnt);
    return make_int2((int)(k * P.ws_k + channel_offset(P, c) + (P.stack ? 0 : r0 + g.r) * P.ws_r + (g.s0 + P.stride * a) * P.ws_s), valid ? g.cnt : 0);
}

// k-side: lane -> offset in dW, -1: not an element
__device__ __forceinline__ int lane_target(const ClShape& P, int l, int k0, int r0)
{
    if (!P.stack) return k0 + l < P.k ? (int)((k0 + l) * P.ws_k) : -1;
    const int j = l >> (31 - __clz(P.ka)), k = l & (P.ka - 1), r = r0 + P.rc - 1 - j;
    return j < P.rc && r < P.r && k < P.k ? (int)(k * P.ws_k + r * P.ws_r) : -1;
}

// The operands as the caller has them
struct ClSource { const void *x, *dy; int f32, x_last, dy_last; };        // *_last: channels last

__device__ __forceinline__ double cl_load(const void* p, size_t i, int f32)
{
    return f32 ? static_cast<const float*>(p)[i] : __bfloat162float(static_cast<const __nv_bfloat16*>(p)[i]);
}
// Element (column, lane) of a tile
struct ClElement { int k, c, r, s; bool valid; };
__device__ __forceinline__ ClElement cl_element(const ClShape& P, int tile, int col, int l)
{
    const int tr = tile / P.tiles_r, r0 = (tile - tr * P.tiles_r) * P.rc, tk = tr / P.tiles_c, k0 = tk * P.kt, c0 = (tr - tk * P.tiles_c) * P.ct;
    const ClGroup& g = P.g[group_of(P, col)];
    const int j = col - g.col, ca_log = 31 - __clz(P.ca), ka_log = 31 - __clz(P.ka);
    const int mn = P.c_side ? l : j, a = P.merged ? 0 : mn >> ca_log;
    ClElement e;
    e.c = c0 + g.cbase + (P.merged ? mn : mn & (P.ca - 1)); e.s = P.row_atoms ? 0 : g.s0 + P.stride * a;
    e.k = P.c_side ? k0 + j : P.stack ? l & (P.ka - 1) : k0 + l;
    e.r = r0 + (P.stack ? P.rc - 1 - (l >> ka_log) : P.row_atoms ? a : g.r);
    e.valid = e.k < P.k && e.c < P.c && a < g.cnt && e.r >= r0 && e.r < P.r;
    return e;
}
// A warp sums the elements of the lanes in `left` anew, one by one, its lanes the output pixels in turn.  The padding counts as
// zeros that are multiplied.  In double, so that finite sums do not depend on the order; a NaN ends the sum.
// Never called on finite data, so that its speed is no matter.
__device__ __noinline__ void cl_repair(const ClShape& P, const ClSource& S, float* dw, int tile, int col, int l, uint32_t left)
{
    const int lane = threadIdx.x & 31, px = P.p * P.q, all = P.n * px;
    const ClElement mine = cl_element(P, tile, col, l);
    while (left != 0) {
        const int owner = __ffs(left) - 1;
        left &= left - 1;
        const int k = __shfl_sync(0xffffffffu, mine.k, owner), c = __shfl_sync(0xffffffffu, mine.c, owner);
        const int r = __shfl_sync(0xffffffffu, mine.r, owner), s = __shfl_sync(0xffffffffu, mine.s, owner);
        const int vs = P.vc != 0 ? c / P.vc : 0, cx = c - vs * P.vc, chans = P.vc != 0 ? P.vc : P.c, cols = P.vc != 0 ? P.vw : P.w;
        double sum = 0;
        for (int base = 0; base < all; base += 32) {
            const int i = base + lane;
            if (i < all) {
                const int n = i / px, p = (i - n * px) / P.q, q = i - n * px - p * P.q;
                const int h = p * P.stride + r - P.pad_h, w = q * P.stride + s + vs - (P.vc != 0 ? P.vpad : P.pad_w);
                const bool in = h >= 0 && h < P.h && w >= 0 && w < cols;
                const size_t xi = S.x_last ? (((size_t)n * P.h + h) * cols + w) * chans + cx : (((size_t)n * chans + cx) * P.h + h) * cols + w;
                const size_t yi = S.dy_last ? (size_t)i * P.k + k : ((size_t)n * P.k + k) * px + (i - n * px);
                sum += (in ? cl_load(S.x, xi, S.f32) : 0.0) * cl_load(S.dy, yi, S.f32);
            }
            if (__any_sync(0xffffffffu, isnan(sum))) break;
        }
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) dw[k * P.ws_k + channel_offset(P, c) + r * P.ws_r + s * P.ws_s] = P.alpha * (float)sum;
    }
}

// Warps: 0 and 1 issue MMAs, 2 and 3 fill the stages, 4 to 11 hold the sums.
//
// The tensor core adds into its accumulators by truncation, so an accumulator's error grows with the number of additions
// (~2e-8 of it each).  After every `epoch` chunks an issuer hands its accumulator set to the eight summing warps, which add
// it to fp32 registers, and starts afresh: the error stays that of a short sum.  There are two sets and two issuers, which
// take alternate chunks: while one waits (for data, for its set to be read, or merely for its own instructions), the other
// keeps the tensor core busy.
constexpr int kThreads = 384;

template <int NG, bool F32, bool CSIDE>
__global__ void __launch_bounds__(kThreads, 1)
cl_kernel(const __grid_constant__ CUtensorMap map_dy, const __grid_constant__ CUtensorMap map_x, float* __restrict__ dw,
          float* __restrict__ partial, uint32_t* __restrict__ status, const __grid_constant__ ClParams P, const __grid_constant__ ClSource S)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[kMaxStages], bar_empty[kMaxStages], bar_acc[2], bar_free[2];
    __shared__ uint32_t s_tmem_base;
    __shared__ volatile int s_abort;
    __shared__ int2 s_col[kMaxCols];        // column_target of every column

    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tile = blockIdx.x, split = blockIdx.y;
    const int r0 = (tile % P.tiles_r) * P.rc, kc = tile / P.tiles_r;
    const int k0 = (kc / P.tiles_c) * P.kt, c0 = (kc % P.tiles_c) * P.ct;
    const int ch_begin = split * P.chunk_base + min(split, P.chunk_rem);
    const int nchunks = P.chunk_base + (split < P.chunk_rem ? 1 : 0);

    GACONV_STAMP(0, threadIdx.x == 0);
    pdl_release_next_grid();
    // Rows behind the copied boxes that MMAs may touch: zeros, written once (no copy ever reaches them).  A zero dY row
    // makes the reduction end where the chunk ends; the X rows opposite only have to be finite.
    {
        const int tiles_dy = P.planes * P.katoms, tiles_all = tiles_dy + P.planes * P.na * P.phases * P.row_tiles;
        for (int t = warp; t < P.stages * tiles_all; t += kThreads / 32) {
            const int st = t / tiles_all, i = t - st * tiles_all;
            const bool is_dy = i < tiles_dy;
            const int base = st * P.stage_bytes + (is_dy ? i * P.dy_alloc : P.x_region + (i - tiles_dy) * P.x_alloc);
            const int from = is_dy ? P.dy_box : P.x_pre + P.x_box, to = is_dy ? P.dy_alloc : P.x_alloc;
            auto zero = [&](int o) { asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(smem_base + base + o), "r"(0) : "memory"); };
            for (int o = from + lane * 16; o < to; o += 512) zero(o);
            if (!is_dy)
                for (int o = lane * 16; o < P.x_pre; o += 512) zero(o);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_dy) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_x) : "memory");
        for (int i = 0; i < P.stages; ++i) { mbar_init(smem_u32(&bar_full[i]), 1); mbar_init(smem_u32(&bar_empty[i]), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&bar_acc[i]), 1); mbar_init(smem_u32(&bar_free[i]), 8); }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (P.splits == 1)
        for (int col = threadIdx.x; col < P.cols; col += kThreads) s_col[col] = column_target(P, col, k0, c0, r0);
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "r"(P.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = s_tmem_base;
    float finite = 0.f;         // NaN as soon as this thread has written an element that is not finite
    pdl_wait_prior_grid();
    GACONV_STAMP(1, threadIdx.x == 0);

    if (warp == 2 || warp == 3) {
        // ------------------------------------------------------------------ TMA producers
        // Each fills every other chunk; lane b issues copy b.  Filling a stage (wait, byte count, copies) takes a warp ~600
        // cycles however large the copies are: one producer gave 33 bytes a cycle on 37 KB stages, two give 66.
        const bool whole = P.cpi == 0;
        constexpr int np = 2;
        const int first = warp - 2, c_first = ch_begin + first;
        int n0 = (whole ? c_first : c_first / P.cpi) * P.ci, p0 = whole ? 0 : (c_first % P.cpi) * P.bp;
        // this lane's copy of every chunk (a plan has at most 32): where it goes, and its coordinates relative to the chunk's
        const int x_tiles = P.na * P.phases * P.row_tiles, per_plane = P.katoms + x_tiles;
        const int pl = lane / per_plane, i = lane - pl * per_plane, j = i - P.katoms, jt = j / P.na, rl = jt / P.phases;
        const bool mine = lane < P.planes * per_plane, is_dy = i < P.katoms;
        const CUtensorMap* map = is_dy ? &map_dy : &map_x;
        const uint32_t dst = is_dy ? pl * P.dy_plane + i * P.dy_alloc : P.x_region + pl * P.x_plane + j * P.x_alloc + P.x_pre;
        const bool images = P.order == kImages, pixels = is_dy && P.order == kPixels;          // box i: 64 pixels of image i / dy_subs, K-major
        const int dy_img = pixels ? i / P.dy_subs : 0, dy_px = 64 * (i - dy_img * P.dy_subs);
        const int ch = is_dy ? k0 + P.ka * i : c0 + P.ca * (j - jt * P.na), col = is_dy || P.x_pre ? 0 : jt - rl * P.phases - P.pad_w;
        const int row_mul = is_dy ? 1 : P.stride;
        const int row_add = P.stack ? (is_dy ? P.pad_h - (r0 + P.rc - 1) : 0) : is_dy ? 0 : r0 + rl - P.pad_h;
        int st = first, ph = 0, it = first;
        while (st >= P.stages) { st -= P.stages; ph ^= 1; }
        for (; it < nchunks; it += np) {
            const uint32_t full = smem_u32(&bar_full[st]);
            if (it >= P.stages && !mbar_wait(smem_u32(&bar_empty[st]), ph ^ 1)) { s_abort = 1; atomicOr(status, 1u); }
            if (__any_sync(0xffffffffu, s_abort)) break;
            if (lane == 0) mbar_expect_tx(full, P.tx_bytes);
            __syncwarp();
            if (pixels) { if (mine) tma_load_3d(smem_base + st * P.stage_bytes + dst, map, full, p0 * P.q + dy_px, k0, n0 + dy_img); }
            else if (mine) {
                const int row = p0 * row_mul + row_add;
                tma_load_5d(smem_base + st * P.stage_bytes + dst, map, full, ch, images ? n0 : col, images ? col : row, images ? row : n0, pl);
            }
            if (whole) n0 += np * P.ci;
            else for (p0 += np * P.bp; p0 >= P.cpi * P.bp; p0 -= P.cpi * P.bp) n0 += P.ci;
            for (st += np; st >= P.stages; st -= P.stages) ph ^= 1;
        }
        if (lane == 0 && s_abort)      // let the copies already issued land (bounded)
            for (int i = it - np; i >= first && i > it - np - P.stages; i -= np) mbar_wait(smem_u32(&bar_full[i % P.stages]), (i / P.stages) & 1);
    } else if (warp < 2) {
        // ------------------------------------------------------------------ MMA issuers
        // The whole warp walks the chunks and one elected lane issues (elected rather than "lane 0": the compiler then knows
        // that a single thread is active and moves descriptors to uniform registers without a loop over lanes; the lane
        // test cost ~100 cycles per MMA).  An MMA holds its registers until the tensor core takes it, and a loop that
        // comes round to the same registers waits for that, ~200 cycles; predicates computed per MMA cost ~100 each.
        // Hence straight-line code of a dozen MMAs per iteration, entered in the middle for a remainder, the offsets of the
        // k-steps in the parameter bank, and the one MMA that starts an accumulator issued apart.
        constexpr int PER = NG * (F32 ? 6 : 1), U = PER >= 8 ? 1 : PER == 1 ? 12 : PER == 2 ? 6 : PER == 3 ? 4 : 2;
        const uint32_t x_plane = (uint32_t)P.x_plane >> 4, dy_plane = (uint32_t)P.dy_plane >> 4;
        const uint64_t dy_hi = (uint64_t)P.dy_hi << 32;
        const int ngroups = P.ngroups;
        int k_first = 0, ksteps = P.ksteps;
        if (P.skip) {       // output rows whose input row r0 lies inside the map
            const int lo = max(0, (P.pad_h - r0 + P.stride - 1) / P.stride), hi = min(P.p, (P.h - 1 + P.pad_h - r0) / P.stride + 1);
            if (lo < hi) { k_first = lo * P.skip; ksteps = hi * P.skip; }       // (none: multiply the zeros)
        }
        const uint32_t idesc = P.idesc;
        uint32_t off[NG];
#pragma unroll
        for (int g = 0; g < NG; ++g) off[g] = NG <= 9 || g < ngroups ? (uint32_t)P.g[g].x_off : 0u;
        const uint32_t acc = tmem_base + warp * P.cols;
        int st = warp, ph = 0, in_epoch = 0, free_ph = 0;       // (the number of stages is even: a stage is always the same issuer's)
        long long waited = 0;          // (tuning builds)
        for (int it = warp; it < nchunks; it += 2) {
            if (in_epoch == P.epoch) {
                if (elect_one()) umma_commit(smem_u32(&bar_acc[warp]));
                if (!mbar_wait(smem_u32(&bar_free[warp]), free_ph)) { s_abort = 1; atomicOr(status, 1u); break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                free_ph ^= 1; in_epoch = 0;
            }
            const long long t0 = GACONV_CLOCK();
            if (!mbar_wait(smem_u32(&bar_full[st]), ph)) { s_abort = 1; atomicOr(status, 1u); break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            waited += GACONV_CLOCK() - t0;
            GACONV_STAMP(2, it == 0);
            const bool fresh = in_epoch == 0;
            if (elect_one()) {
                const uint32_t sa = smem_base + st * P.stage_bytes;
                const uint32_t dy_lo = P.dy_lbo | ((sa >> 4) & 0x3fffu), x_lo = P.x_lbo | (((sa + P.x_region) >> 4) & 0x3fffu);
                auto step = [&](int k, bool starts) {
                    const uint4 o = P.k_off[k];
                    const uint64_t x_hi = (uint64_t)o.z << 32;
#pragma unroll
                    for (int pr = 0; pr < (F32 ? 6 : 1); ++pr) {
                        const uint64_t dyd = dy_hi | (dy_lo + o.y + (F32 ? prod_dy(pr) * dy_plane : 0u));
                        const uint64_t xd = x_hi | (x_lo + o.x + (F32 ? prod_x(pr) * x_plane : 0u));
#pragma unroll
                        for (int g = 0; g < NG; ++g)
                            if (NG <= 9 || g < ngroups) {          // (up to nine MMAs there is an instance for every count)
                                const uint64_t ad = CSIDE ? xd + off[g] : dyd, bd = CSIDE ? dyd : xd + off[g];
                                const uint32_t d = acc + (NG == 1 && !CSIDE ? o.w & 0xffffu : (uint32_t)P.g[g].col);
                                const uint32_t id = idesc | (NG == 1 && !CSIDE ? o.w & 0xffff0000u : P.g[g].idesc);
                                if (starts && pr == 0) umma_bf16(d, ad, bd, id, 0u);
                                else umma_bf16_acc(d, ad, bd, id);
                            }
                    }
                };
                int k = k_first;
                if (fresh) step(k++, true);
                switch ((ksteps - k) % U) {
                    case 11: step(k++, false); [[fallthrough]];
                    case 10: step(k++, false); [[fallthrough]];
                    case 9: step(k++, false); [[fallthrough]];
                    case 8: step(k++, false); [[fallthrough]];
                    case 7: step(k++, false); [[fallthrough]];
                    case 6: step(k++, false); [[fallthrough]];
                    case 5: step(k++, false); [[fallthrough]];
                    case 4: step(k++, false); [[fallthrough]];
                    case 3: step(k++, false); [[fallthrough]];
                    case 2: step(k++, false); [[fallthrough]];
                    case 1: step(k++, false);
                }
                for (; k < ksteps; k += U) {
#pragma unroll
                    for (int u = 0; u < U; ++u) step(k + u, false);
                }
                umma_commit(smem_u32(&bar_empty[st]));
            }
            __syncwarp();
            ++in_epoch;
            for (st += 2; st >= P.stages; st -= P.stages) ph ^= 1;
        }
        if (warp < nchunks && elect_one()) {
            umma_commit(smem_u32(&bar_acc[warp]));
            GACONV_STAMP(3, warp == 0);
            if (warp == 0) GACONV_TALLY(6, waited);
        }
        __syncwarp();
    } else if (warp >= 4) {
        // ------------------------------------------------------------------ summing warps
        // Warps w and w + 4 read the same 32 lanes of tensor memory and take alternate 16-column pieces.
        constexpr int NB = kMaxCols / 32;
        const int sp = warp & 3, half = (warp - 4) >> 2, l128 = 32 * sp + lane, blocks = P.cols >> 4;
        float sum[NB][16];
#pragma unroll
        for (int i = 0; i < NB; ++i)
#pragma unroll
            for (int e = 0; e < 16; ++e) sum[i][e] = 0.f;
        bool ok = true;
        for (int done = 0, ph = 0; done < nchunks && ok; done += 2 * P.epoch, ph ^= 1)
            for (int set = 0; set < 2 && done + set < nchunks && ok; ++set) {
                ok = mbar_wait(smem_u32(&bar_acc[set]), ph);
                if (!ok) { s_abort = 1; atomicOr(status, 1u); }
                ok = __all_sync(0xffffffffu, ok && !s_abort);        // warp-uniform: the tensor-memory loads are warp-wide
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (!ok) break;
                const uint32_t src = tmem_base + set * P.cols + 16 * half + ((uint32_t)(32 * sp) << 16);
#pragma unroll
                for (int i = 0; i < NB; i += 2) {                    // two pieces in flight
                    if (2 * i + half < blocks) {
                        float v[2][16];
                        const bool two = i + 1 < NB && 2 * (i + 1) + half < blocks;
                        tmem_ld16_nowait(src + 32 * i, v[0]);
                        if (two) tmem_ld16_nowait(src + 32 * (i + 1), v[1]);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int e = 0; e < 16; ++e) sum[i][e] += v[0][e];
                        if (i + 1 < NB && two) {
#pragma unroll
                            for (int e = 0; e < 16; ++e) sum[i + 1 < NB ? i + 1 : i][e] += v[1][e];
                        }
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar_free[set])) : "memory");
            }
        GACONV_STAMP(4, threadIdx.x == 128);
        // The only split of a tile, channels innermost in dW: from the registers, eight channels (a sector) a store.
        const bool sectors = !CSIDE && P.splits == 1 && P.ws_c == 1 && (P.c & 7) == 0 && (reinterpret_cast<uintptr_t>(dw) & 31) == 0;
        if (ok && sectors) {
            const int lane_off = lane_target(P, l128, k0, r0);
            float* d = dw + lane_off;
#pragma unroll
            for (int i = 0; i < NB; ++i)
                if (2 * i + half < blocks && lane_off >= 0) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int2 o = s_col[16 * (2 * i + half) + 8 * h];
                        const float* v = sum[i] + 8 * h;
                        const float a = P.alpha;
                        if (o.y > 0) {
#pragma unroll
                            for (int u = 0; u < 8; ++u) finite = fmaf(v[u], 0.f, finite);
                            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(d + o.x), "f"(a * v[0]), "f"(a * v[1]),
                                         "f"(a * v[2]), "f"(a * v[3]), "f"(a * v[4]), "f"(a * v[5]), "f"(a * v[6]), "f"(a * v[7]) : "memory");
                        }
                    }
                }
        } else if (ok) {        // the block (the stages are free: every copy has landed and every MMA has read)
            float* blk = reinterpret_cast<float*>(smem_raw + (smem_base - smem_u32(smem_raw)));
            const int ca_log = 31 - __clz(P.ca);
            const bool keyed = P.splits == 1;
#pragma unroll
            for (int i = 0; i < NB; ++i)
                if (2 * i + half < blocks) {
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const int col = 16 * (2 * i + half) + e;
                        if (keyed) blk[col * 128 + (l128 ^ block_key(col, ca_log))] = sum[i][e];
                        else blk[col * 128 + l128] = sum[i][e];
                    }
                }
            if (P.splits > 1) {      // to the workspace, one bulk store per 16 columns
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("bar.sync 1, 256;" ::: "memory");
                const int t = threadIdx.x - 128;
                if (t < blocks) {
                    float* out = partial + ((size_t)tile * P.splits + split) * P.cols * 128;
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(out + t * 2048), "r"(smem_base + t * 8192), "r"(8192) : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    GACONV_STAMP(7, threadIdx.x == 0);
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(P.tmem_cols) : "memory");
    }
    // ---------------------------------------------------------------------- the only split of a tile: all warps, block -> dW
    const bool sectors = !CSIDE && P.ws_c == 1 && (P.c & 7) == 0 && (reinterpret_cast<uintptr_t>(dw) & 31) == 0;        // (written already)
    if (P.splits == 1 && !sectors && !s_abort) {
        const float* blk = reinterpret_cast<const float*>(smem_raw + (smem_base - smem_u32(smem_raw)));
        const int cols = P.cols;
        const int ca_log = 31 - __clz(P.ca);
        if (CSIDE) {
            const int third = threadIdx.x >> 7;
            int l = threadIdx.x & 127;
            if (P.s_inner) l = ((l & ((1 << (7 - ca_log)) - 1)) << ca_log) + (l >> (7 - ca_log));
            const int a = P.merged ? 0 : l >> ca_log, cc = P.merged ? l : l & (P.ca - 1);          // this lane's atom and channel
            float* d = dw + a * atom_step(P) + channel_offset(P, cc);
            if (c0 + cc < P.c && (!P.row_atoms || r0 + a < P.r)) {
#pragma unroll 4
                for (int col = third; col < cols; col += 3) {
                    const int2 o = s_col[col];
                    const float v = blk[col * 128 + (l ^ block_key(col, ca_log))];
                    if (a < o.y) { d[o.x] = P.alpha * v; finite = fmaf(v, 0.f, finite); }
                }
            }
        } else if (P.ws_c == 1 && (P.c & 3) == 0) {
            // a warp takes four rows x 32 columns: four lines of 128 bytes a store
            const int cgs = (cols + 31) >> 5, cq = (lane & 7) << 2;
#pragma unroll 2
            for (int t = warp; t < 32 * cgs; t += kThreads / 32) {
                const int cg = t >> 5, l = ((t & 31) << 2) + (lane >> 3), col = (cg << 5) + cq;
                const int lane_off = lane_target(P, l, k0, r0);
                if (col < cols && lane_off >= 0) {
                    const int2 o = s_col[col];
                    float v[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] = P.alpha * blk[(col + i) * 128 + (l ^ block_key(col + i, ca_log))];
                    if (o.y > 0) {
                        *reinterpret_cast<float4*>(dw + lane_off + o.x) = make_float4(v[0], v[1], v[2], v[3]);
#pragma unroll
                        for (int i = 0; i < 4; ++i) finite = fmaf(v[i], 0.f, finite);
                    }
                }
            }
        } else {
            for (int cb = 0; cb < cols; cb += 64) {        // two columns a lane
                int off[2], pos[2], key[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int e = cb + lane + 32 * u, col = e < cols ? written_column(P, e) : 0;
                    const int2 o = s_col[col];
                    off[u] = e < cols && o.y > 0 ? o.x : -1;
                    pos[u] = col * 128; key[u] = block_key(col, ca_log);
                }
#pragma unroll 4
                for (int l = warp; l < 128; l += kThreads / 32) {
                    const int lane_off = lane_target(P, l, k0, r0);
                    if (lane_off < 0) continue;
                    float* d = dw + lane_off;
#pragma unroll
                    for (int u = 0; u < 2; ++u)
                        if (off[u] >= 0) {
                            const float v = blk[pos[u] + (l ^ key[u])];
                            d[off[u]] = P.alpha * v;
                            finite = fmaf(v, 0.f, finite);
                        }
                }
            }
        }
    }
    if (P.splits == 1 && __syncthreads_or(isnan(finite)) && !s_abort)
        for (int e = warp; e < 4 * P.cols; e += kThreads / 32) {
            const int col = e >> 2, l = 32 * (e & 3) + lane;
            const ClElement el = cl_element(P, tile, col, l);
            const uint32_t left = __ballot_sync(0xffffffffu, el.valid && !isfinite(__ldcg(dw + (el.k * P.ws_k + channel_offset(P, el.c) + el.r * P.ws_r + el.s * P.ws_s))));
            if (left != 0) cl_repair(P, S, dw, tile, col, l, left);
        }
    GACONV_STAMP(5, threadIdx.x == 0);
}

// lane of the e-th element that a block of cl_reduce_kernel writes, and its column relative to the block's first
__device__ __forceinline__ int2 reduced_element(const ClShape& P, int e, int log_cb)
{
    int l = P.c_side ? e & 127 : e >> log_cb;
    if (P.c_side && P.s_inner) { const int t_shift = 7 - (31 - __clz(P.ca)); l = ((l & ((1 << t_shift) - 1)) << (7 - t_shift)) + (l >> t_shift); }
    return make_int2(l, P.c_side ? e >> 7 : e & ((1 << log_cb) - 1));
}
// Every warp of cl_reduce_kernel repairs what it has written (a thread reads its own elements back).  Apart, so that the kernel keeps
// nothing in registers for the sake of it.
__device__ __noinline__ void cl_repair_written(const ClShape& P, const ClSource& S, float* dw, int log_cb)
{
    const int tile = blockIdx.y, col0 = blockIdx.x << log_cb;
    for (int e = threadIdx.x; e < 128 << log_cb; e += blockDim.x) {          // (whole warps: both are multiples of 32)
        const int2 lc = reduced_element(P, e, log_cb);
        const bool in = col0 + lc.y < P.cols;
        const int col = written_column(P, in ? col0 + lc.y : 0);
        const ClElement el = cl_element(P, tile, col, lc.x);
        const float* out = dw + (el.k * P.ws_k + channel_offset(P, el.c) + el.r * P.ws_r + el.s * P.ws_s);
        const uint32_t left = __ballot_sync(0xffffffffu, in && el.valid && !isfinite(__ldcg(out)));
        if (left != 0) cl_repair(P, S, dw, tile, col, lc.x, left);
    }
}

// What cl_reduce_kernel has to know of a column, worked out with the plan: its blocks start when those of cl_kernel end, so that nothing hides the
// divisions and look-ups before their first loads, nor the banks in which the sums of a warp's columns meet (us, whole call, before / now with
// this table and rows of 132 sums: bf16 256->256 on 8x8, N = 128 18.1 / 17.3, 128->128 on 16x16 18.1 / 17.4, 36->16 5x5 on 44x44, N = 30 17.1 / 16.3).
struct ClColumn { int off; uint32_t info; };       // offset in dW from the tile's; column | channel << 8 | atoms in use << 16 | filter row << 20 | output << 24
struct ClReduce { FastDiv by_r, by_c; int ws_c, atom_step; ClColumn col[kMaxCols]; };

// Sum of the splits of every (tile, column), in a fixed order: grid (column blocks, tiles), 32 * CB * G threads.  Warp (g, c)
// adds the 128 lanes (a float4 each) of column c over the splits g, g + G, ...; the G partial sums meet in shared memory.  G is
// chosen so that a warp's loads are all in flight at once (eight, then a second round), CB so that the grid covers the GPU;
// where consecutive columns are consecutive channels of dW a block writes CB of them in one piece.  Latency-bound: what an
// element is, and where it goes, is worked out before the wait for the sums.
// LEAN: 32 registers.  With 56 all eight loads of a thread are in flight (fp32 64->128 stride 2 on 28x28, N = 64, whole call:
// 32.7 -> 31.3 us), but only where the SMs hold all blocks at once (352->288 on 9x9, N = 65, 648 blocks of 512 threads: 34.2 -> 35.3)
// and nothing else wants room on them (step of ResNet-20 150 -> 154).
template <bool LEAN>
__global__ void __launch_bounds__(1024, LEAN ? 2 : 1)
cl_reduce_kernel(const float* __restrict__ partial, float* __restrict__ dw, const __grid_constant__ ClShape P, const __grid_constant__ ClSource S, const __grid_constant__ ClReduce T, int log_cb, int G)
{
    __shared__ float s_sum[32][132];        // (rows four banks apart: the columns that a warp writes lie in different ones)
    __shared__ int2 s_col[16];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, CB = 1 << log_cb;
    const int tile = blockIdx.y, col0 = blockIdx.x << log_cb;
    pdl_release_next_grid();
    const int tr = T.by_r.div(tile), r0 = (tile - tr * P.tiles_r) * P.rc, tk = T.by_c.div(tr);
    const int k0 = tk * P.kt, c0 = (tr - tk * P.tiles_c) * P.ct;
    const int ca_shift = 31 - __clz(P.ca), mn_mask = P.merged ? 127 : P.ca - 1;
    // {offset in dW, atoms in use (0: not an element)} of a column, in the order in which they are written
    auto target = [&](int e, uint32_t info) {
        const bool valid = e < P.cols && r0 + (int)(info >> 20 & 15) < P.r && (P.c_side ? k0 + (int)(info >> 24) < P.k : c0 + (int)(info >> 8 & 255) < P.c);
        return valid ? (int)(info >> 16 & 15) : 0;
    };
    const int cb = warp & (CB - 1), grp = warp >> log_cb, mine = min(col0 + cb, P.cols - 1);
    const uint32_t info = T.col[mine].info;
    const float4* src = reinterpret_cast<const float4*>(partial + ((size_t)tile * P.splits * P.cols + (info & 255)) * 128) + lane;
    const size_t step = (size_t)P.cols * 32;
    const bool live = target(col0 + cb, info) > 0;
    if ((int)threadIdx.x < CB) {
        const int e = col0 + threadIdx.x;
        const ClColumn o = T.col[min(e, P.cols - 1)];
        s_col[threadIdx.x] = make_int2((int)(o.off + (P.c_side ? k0 * P.ws_k : 0) + c0 * P.ws_c + (P.stack ? 0 : r0 * P.ws_r)), target(e, o.info));
    }
    pdl_wait_prior_grid();
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (live)
        for (int s = grp; s < P.splits; s += 8 * G) {
            float4 u[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) u[i] = s + i * G < P.splits ? __ldcg(src + (size_t)(s + i * G) * step) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 8; ++i) { acc.x += u[i].x; acc.y += u[i].y; acc.z += u[i].z; acc.w += u[i].w; }
        }
    *reinterpret_cast<float4*>(&s_sum[warp][4 * lane]) = acc;
    float finite = 0.f;         // NaN as soon as this thread has written an element that is not finite
    __syncthreads();
    for (int e = threadIdx.x; e < CB << 7; e += blockDim.x) {
        const int2 lc = reduced_element(P, e, log_cb);
        const int l = lc.x, c = lc.y;
        const int2 o = s_col[c];
        bool valid; long long off = o.x;
        if (P.c_side) {
            const int a = P.merged ? 0 : l >> ca_shift, ch = l & mn_mask;
            valid = a < o.y && c0 + ch < P.c && (!P.row_atoms || r0 + a < P.r);
            off += (P.vc == 0 ? ch * T.ws_c : (int)channel_offset(P, ch)) + a * T.atom_step;         // (offsets in dW have 32 bits)
        } else {
            const int lane_off = lane_target(P, l, k0, r0);
            valid = o.y > 0 && lane_off >= 0;
            off += lane_off;
        }
        if (!valid) continue;
        float t = s_sum[c][l];
        for (int w = 1; w < G; ++w) t += s_sum[(w << log_cb) + c][l];
        dw[off] = P.alpha * t;
        finite = fmaf(t, 0.f, finite);
    }
    if (__any_sync(0xffffffffu, isnan(finite))) cl_repair_written(P, S, dw, log_cb);
}

// ---- packing: one operand -> channels-last bf16 planes, channels padded to a multiple of 8 with zeros -------------------
struct PackOp {
    const void* src;
    __nv_bfloat16* dst;
    int ch, chp, px, n;         // source: n images of px pixels and ch channels; destination rows of chp channels,
    int pitch;                  // this many apart
    int channels_last;          // source order: 1 [n][px][ch], 0 [n][ch][px]
    int vc, vw, vpad, q, h;     // ClShape::vc and so on: the destination's channels are gathered from windows of the source; its rows and columns
    int px_tiles, ch_tiles;     // tiles of an image (channels-first sources): tile_px pixels x
    int ch_tile;                // at most 64 channels, a multiple of 8
    int tile_px;                // pixels of a tile
    int gather;                 // rows of pixels that do not lie on 16-byte boundaries, or few channels
    int slab;                   // images per block, where an image's channels of a block are taken as one piece (0: by rows of pixels)
    int blocks;                 // tiles in all
    size_t plane;               // elements of a destination plane
};

__device__ __forceinline__ uint32_t bf16_pair(float a, float b) {
    const __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&t);
}
// two fp32 values -> their planes, packed pairwise: x0 = the upper 16 bits of x (no rounding, so nothing overflows),
// x1 = bf16(x - x0), x2 = bf16(x - x0 - x1); both differences are exact
__device__ __forceinline__ void split2(float u, float v, uint32_t (&w)[3]) {
    const uint32_t a = __float_as_uint(u) & 0xffff0000u, b = __float_as_uint(v) & 0xffff0000u;
    w[0] = (a >> 16) | b;
    const float ru = u - __uint_as_float(a), rv = v - __uint_as_float(b);
    w[1] = bf16_pair(ru, rv);
    w[2] = bf16_pair(ru - __uint_as_float(w[1] << 16), rv - __uint_as_float(w[1] & 0xffff0000u));
}
// copies the first n <= 16 bytes of a 16-byte piece to shared memory without a stop in registers; zeros behind them
__device__ __forceinline__ void copy_async(uint32_t dst, const void* src, int n) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// Blocks [0, x.blocks) pack X, the others dY.  E: the element as a plain number of its size (float, or the 16 bits of a
// bf16).  A block turns a tile of 64 channels x 128 pixels (64 of fp32, whose three planes take the room) of a channels-first source: rows of pixels arrive in shared memory
// by asynchronous copies, ldmatrix.trans turns 8 x 8 blocks on the way out, and with its
// row addresses ordered (0 1 8 9 16 17 24 25), (2 3 10 11 ...) ... a lane receives eight consecutive channels of a pixel, one
// 16-byte store.  (Turning by single elements in registers was bound by instructions: 22 us on 13 MB of gradients and 8 MB of
// activations.)  The 16-byte chunks of a row are permuted by the same order, so that the eight rows of a block sit in
// different banks.
template <typename E> constexpr int kPackPx = sizeof(E) == 4 ? 64 : 128;

// eight channels of a pixel -> 16 bytes of every plane
template <typename E>
__device__ __forceinline__ void store8(const E (&v)[8], __nv_bfloat16* dst, size_t plane) {
    uint4* out = reinterpret_cast<uint4*>(dst);
    if constexpr (sizeof(E) == 4) {
        uint32_t w[4][3];
#pragma unroll
        for (int j = 0; j < 4; ++j) split2(v[2 * j], v[2 * j + 1], w[j]);
#pragma unroll
        for (int pl = 0; pl < 3; ++pl) out[pl * (plane / 8)] = make_uint4(w[0][pl], w[1][pl], w[2][pl], w[3][pl]);
    } else {
        *out = make_uint4(v[0] | (uint32_t)v[1] << 16, v[2] | (uint32_t)v[3] << 16, v[4] | (uint32_t)v[5] << 16, v[6] | (uint32_t)v[7] << 16);
    }
}

// WINDOWS: X is gathered from windows (PackOp::vc); apart, so that the other calls carry nothing for it.
template <typename E, bool WINDOWS>
__global__ void __launch_bounds__(256)
pack_kernel(const PackOp x, const PackOp dy)
{
    constexpr int NP = sizeof(E) == 4 ? 3 : 1, TPX = kPackPx<E>, ROW = 2 * TPX;       // planes; bytes of a tile row
    constexpr int kTile = 64 * ROW, kBytes = NP * kTile > 17664 ? NP * kTile : 17664;         // (slabs and gathered rows: at most 17,664)
    __shared__ __align__(128) unsigned char s_tile[kBytes];
    pdl_release_next_grid();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool is_x = (int)blockIdx.x < x.blocks;
    const PackOp& o = is_x ? x : dy;
    const int blk = is_x ? blockIdx.x : blockIdx.x - x.blocks;
    const E* src = static_cast<const E*>(o.src);
    if (WINDOWS && is_x) {
        // A pixel of the destination: the channels of the columns of a window, neighbours in a channels-last row
        const int g8 = o.chp >> 3, row_el = o.vw * o.vc;
        const unsigned items = (unsigned)o.n * o.px * g8;
        pdl_wait_prior_grid();
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const unsigned it = blk * 512u + i * 256 + threadIdx.x;
            if (it >= items) return;
            const unsigned row = it / (unsigned)g8, nh = row / (unsigned)o.q;
            const int j0 = (int)(it - row * g8) * 8, q = (int)(row - nh * o.q);
            alignas(16) E v[8];
            if (o.channels_last) {
                const int f0 = (q - o.vpad) * o.vc + j0;
                const E* p = src + (size_t)nh * row_el;
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = j0 + u < o.ch && f0 + u >= 0 && f0 + u < row_el ? __ldg(p + f0 + u) : E(0);
            } else {
                const unsigned n = nh / (unsigned)o.h;
                const size_t plane = (size_t)o.h * o.vw;
                int s = j0 / o.vc, c = j0 - s * o.vc;
                const E* p = src + ((size_t)n * o.vc * o.h + (nh - n * o.h)) * o.vw + c * plane;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int w = q + s - o.vpad;
                    v[u] = j0 + u < o.ch && w >= 0 && w < o.vw ? __ldg(p + w) : E(0);
                    p += plane;
                    if (++c == o.vc) { c = 0; ++s; p -= o.vc * plane; }
                }
            }
            store8(v, o.dst + (size_t)row * o.pitch + j0, o.plane);
        }
        return;
    }
    if (o.channels_last) {
        const int g8 = o.chp >> 3;
        const unsigned items = (unsigned)o.n * o.px * g8;            // (an operand has at most 2^31 elements)
        const bool vec = (o.ch & 7) == 0;
        pdl_wait_prior_grid();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned it = blk * 1024u + i * 256 + threadIdx.x;
            if (it >= items) return;
            const unsigned row = it / (unsigned)g8;
            const int c = (int)(it - row * g8) * 8;
            const E* p = src + (size_t)row * o.ch + c;
            alignas(16) E v[8];
            if (vec) {
                const uint4* q = reinterpret_cast<const uint4*>(p);
#pragma unroll
                for (int j = 0; j < (int)sizeof(E) / 2; ++j) reinterpret_cast<uint4*>(v)[j] = __ldg(q + j);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = c + j < o.ch ? __ldg(p + j) : E(0);
            }
            store8(v, o.dst + (size_t)row * o.pitch + c, o.plane);
        }
        return;
    }
    if (o.slab) {
        // Maps under 64 pixels: 64 channels of an image are one piece of memory, read as such (rows of pixels would be short and
        // mostly outside the tile) and picked apart on the way out; eight channels' pixels are followed by 16 bytes of padding.
        constexpr int V = 16 / sizeof(E);
        const int ng = blk / o.ch_tiles, c0 = (blk - ng * o.ch_tiles) * 64, n0 = ng * o.slab, imgs = min(o.slab, o.n - n0);
        const int rows = min(64, o.ch - c0), vecs = rows * o.px / V, grp = 8 * o.px / V, img_vecs = 8 * (grp + 1);
        float4* tile = reinterpret_cast<float4*>(s_tile);
        pdl_wait_prior_grid();
#pragma unroll 4
        for (int e = threadIdx.x; e < imgs * vecs; e += 256) {
            const int i = e / vecs, v = e - i * vecs;
            tile[i * img_vecs + v + v / grp] = __ldg(reinterpret_cast<const float4*>(src + ((size_t)(n0 + i) * o.ch + c0) * o.px) + v);
        }
        __syncthreads();
        const int q8 = min(8, (o.chp - c0) >> 3), items = imgs * o.px * q8;
        for (int e = threadIdx.x; e < items; e += 256) {
            const int ip = e / q8, q = e - ip * q8, i = ip / o.px, j = ip - i * o.px;
            const E* p = reinterpret_cast<const E*>(tile + i * img_vecs + q * (grp + 1)) + j;
            alignas(16) E v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = 8 * q + u < rows ? p[u * o.px] : E(0);
            store8(v, o.dst + ((size_t)(n0 + i) * o.px + j) * o.pitch + c0 + 8 * q, o.plane);
        }
        return;
    }
    const int per_img = o.px_tiles * o.ch_tiles, n = blk / per_img, rest = blk - n * per_img, ct = rest / o.px_tiles, c0 = ct * o.ch_tile;
    const int p0 = (rest - ct * o.px_tiles) * o.tile_px, rows = min(o.ch_tile, o.ch - c0), left = min(o.tile_px, o.px - p0);
    const E* base = src + ((size_t)n * o.ch + c0) * o.px + p0;
    const uint32_t tile = smem_u32(s_tile);
    if (o.gather) {
        // The 16-byte pieces that hold a row, each row with its own offset from the boundary; eight elements per store are then
        // picked from eight rows (16 bytes between groups of eight rows keep their banks apart).  (30 MB of 23x23 maps: copied by
        // words into the order that ldmatrix wants 39 us, this way 18; bound by the instructions that pick.)
        const int pitch = o.tile_px * (int)sizeof(E) + 16, row_bytes = o.px * (int)sizeof(E), bytes = left * (int)sizeof(E);
        const char* first = reinterpret_cast<const char*>(base);
        const char* end = reinterpret_cast<const char*>(src + (size_t)o.n * o.ch * o.px);
        const int first_off = (int)(reinterpret_cast<uintptr_t>(base) & 15);
        pdl_wait_prior_grid();
#pragma unroll 4
        for (int row = warp; row < rows; row += 8) {
            const int off = (first_off + row * row_bytes) & 15;
            const char* piece = first + (size_t)row * row_bytes - off;
            const uint32_t dst = tile + row * pitch + (row >> 3) * 16;
            for (int k = 16 * lane; k < bytes + off; k += 512) copy_async(dst + k, piece + k, (int)min((ptrdiff_t)16, end - (piece + k)));
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        // a thread keeps its eight rows and walks over pixels
        const int q8 = min(o.ch_tile, o.chp - c0) >> 3, log_q = 32 - __clz(q8 - 1), q = threadIdx.x & ((1 << log_q) - 1), r8 = 8 * q;
        if (q >= q8) return;
        const unsigned char* at[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) at[u] = s_tile + (r8 + u) * pitch + q * 16 + ((first_off + (r8 + u) * row_bytes) & 15);
        const int valid = rows - r8;
        __nv_bfloat16* d = o.dst + ((size_t)n * o.px + p0) * o.pitch + c0 + r8;
#pragma unroll 2
        for (int j = threadIdx.x >> log_q; j < left; j += 256 >> log_q) {
            alignas(16) E v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = *reinterpret_cast<const E*>(at[u] + j * sizeof(E));
            if (valid < 8) {
#pragma unroll
                for (int u = 0; u < 8; ++u) if (u >= valid) v[u] = E(0);
            }
            store8(v, d + (size_t)j * o.pitch, o.plane);
        }
        return;
    }
    auto at = [&](int row, int px) {          // byte offset of a pixel in its (permuted) row
        const int sw = (((row >> 3) & 3) << 1) | (row & 1);
        return row * ROW + ((((px >> 3) ^ sw) << 4) | ((px & 7) << 1));
    };
    pdl_wait_prior_grid();
    if constexpr (sizeof(E) == 2) {
        if ((o.px & 7) == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int e = (i * 256 + (int)threadIdx.x) * 8, row = e >> 7, px = e & 127;
                const bool in = row < rows && px < left;
                copy_async(tile + at(row, px), in ? base + (size_t)row * o.px + px : src, in ? 16 : 0);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int e = (i * 256 + (int)threadIdx.x) * 4, row = e >> 7, px = e & 127;
                const bool in = row < rows && px < left;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(tile + at(row, px)), "l"(in ? base + (size_t)row * o.px + px : src), "r"(in ? 8 : 0) : "memory");
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else {
#pragma unroll 4
        for (int i = 0; i < TPX / 16; ++i) {
            const int e = (i * 256 + (int)threadIdx.x) * 4, row = e / TPX, px = e % TPX;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row < rows && px < left) v = __ldg(reinterpret_cast<const float4*>(base + (size_t)row * o.px + px));
            uint32_t w0[3], w1[3];
            split2(v.x, v.y, w0); split2(v.z, v.w, w1);
#pragma unroll
            for (int pl = 0; pl < NP; ++pl) *reinterpret_cast<uint2*>(&s_tile[pl * kTile + at(row, px)]) = make_uint2(w0[pl], w1[pl]);
        }
    }
    __syncthreads();
    const int rho = lane & 7, m = lane >> 3, end = min(c0 + o.ch_tile, o.chp);
#pragma unroll
    for (int i = 0; i < TPX / 32; ++i) {
        const int blk8 = warp * (TPX / 64) + (i >> 1), h = i & 1;        // eight pixels, half of the channels
        const int row = h * 32 + 8 * (rho >> 1) + 2 * m + (rho & 1);
        const int px = 8 * blk8 + (lane >> 2), c = c0 + h * 32 + 8 * (lane & 3);
#pragma unroll
        for (int pl = 0; pl < NP; ++pl) {
            uint32_t r[4];
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                         : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(tile + pl * 64 * ROW + at(row, 8 * blk8)) : "memory");
            if (px < left && c < end)
                *reinterpret_cast<uint4*>(o.dst + pl * o.plane + ((size_t)n * o.px + p0 + px) * o.pitch + c) = make_uint4(r[0], r[1], r[2], r[3]);
        }
    }
}

// ---------------------------------------------------------------- host side: the plan
int round_up(int v, int m) { return (v + m - 1) / m * m; }
int ceil_div(int a, int b) { return (a + b - 1) / b; }

constexpr int kStageBudget = 216 * 1024;

// What a candidate costs, in SM cycles, from rates measured with kernels of one kind each: an MMA of N columns takes N / 2
// cycles; shared memory moves 128 bytes a cycle (147 of a mix), the MMAs' operands, (128 + N) / 4 cycles, and what the copies write; copies
// deliver ~80 bytes a cycle and one row (pixel) in no less than 1.4 cycles; a chunk costs its producer and its issuer ~1200
// cycles of instructions each (two of either work in turn); a CTA writes its block at ~21 bytes a cycle to the workspace and at
// ~18 to dW; start, first loads, drain and the second kernel come to a few thousand.
struct Cost { double cycles; int splits; };
Cost cost_of(const ClParams& P, int sms, double block_share, size_t room)     // room: bytes for partial blocks
{
    double ksteps = P.ksteps;
    if (P.skip) {       // the tile with the fewest rows left out decides
        int most = 0;
        for (int r = 0; r < P.r; ++r)
            most = std::max(most, std::min(P.p, (P.h - 1 + P.pad_h - r) / P.stride + 1) - std::max(0, (P.pad_h - r + P.stride - 1) / P.stride));
        ksteps = std::max(1, most) * P.skip;
    }
    const double mma = ksteps / P.ksteps * P.mma_cols * P.nprod / 2.0;
    const double shared = ksteps / P.ksteps * P.nprod * (P.mma_cols / 4.0 + P.ksteps * P.ngroups * (128 / 4.0 + 2)) + P.tx_bytes / 128.0;
    const double rows = (double)P.planes * (P.katoms * (P.dy_box / (P.order == kPixels ? 128 : P.ka * 2)) + P.na * P.phases * P.row_tiles * (P.x_box / (P.ca * 2)));
    const double load = std::max(P.tx_bytes / 80.0, rows * 1.4);
    const double chunk = std::max({mma * 1.03, shared * 0.87, load, 600.0}) * (P.stages > 2 ? 1.0 : 1.2) + 40;
    const int tiles = P.tiles_k * P.tiles_c * P.tiles_r;
    const double block_bytes = (double)P.cols * 512 * block_share;
    Cost best{1e30, 1};
    int most = std::max(1, (int)std::min<size_t>(std::min(P.chunks, sms / tiles), room / ((size_t)tiles * P.cols * 512)));
#ifdef GACONV_TUNING
    if (const char* e = getenv("GACONV_CL_SP")) most = std::min(most, atoi(e));
#endif
    for (int sp = most; sp >= 1; sp = sp > 8 ? sp * 7 / 8 : sp - 1) {
        const int waves = ceil_div(tiles * sp, sms), per = ceil_div(P.chunks, sp);
        const double main = waves * (4500 + load * std::min({per, P.stages, 4}) / 2 + per * chunk + block_bytes / (sp == 1 ? 18 : 21));
        const double red = sp == 1 ? 0.0 : 4000 + (double)tiles * sp * block_bytes / (25.0 * sms);
        if (main + red < best.cycles) best = Cost{main + red, sp};
    }
    return best;
}

// column shifts that one MMA covers (not merged)
int shifts_of(const ClParams& P)
{
    const int most = P.c_side ? 128 / P.ca : 256 / P.ca, shifts = ceil_div(P.s, P.stride);
    return P.c_side ? most : ceil_div(shifts, ceil_div(shifts, most));
}
// the last column shift that an MMA touches, in use or not
int far_shift(const ClParams& P)
{
    const int shifts = ceil_div(P.s, P.stride), atoms = P.c_side && !P.merged ? shifts_of(P) : 1;
    return ceil_div(shifts, atoms) * atoms - 1;
}

bool build_groups(ClParams& P)
{
    P.ngroups = 0;
    const int rows = P.stack || P.row_atoms ? 1 : P.rc, st = P.stride, wt = P.x_pitch;
    // atoms of one MMA on the X side: c-side exactly fills M = 128; k-side as many as N = 256 takes, the shifts of a column phase
    // shared out evenly over as few MMAs as hold them
    const int atoms = P.merged ? P.na : shifts_of(P);
    P.cols = 0;
    auto add = [&](int tile_i, int row_px, int r, int s0, int cnt, int cbase) {
        if (P.ngroups == kMaxGroups) return false;
        const int n = P.c_side ? P.kt : (P.merged ? P.na : cnt) * P.ca;
        P.g[P.ngroups++] = ClGroup{(tile_i * P.x_alloc + row_px * P.px_rows * P.ca * 2) >> 4, r, s0, cnt, cbase, P.cols, n, (uint32_t)(n >> 3) << 17};
        P.cols += n;
        return true;
    };
    for (int rl = 0; rl < rows; ++rl)
        for (int ph = 0; ph < P.phases; ++ph) {
            const int base_tile = st > 1 ? (rl * P.phases + ph) * P.na : 0, base_px = st > 1 ? 0 : rl * wt;
            const int shifts = (P.s - ph + st - 1) / st;
            if (P.merged) {
                for (int i = 0; i < shifts; ++i)
                    if (!add(base_tile, base_px + i, rl, ph + st * i, 1, 0)) return false;
            } else {
                for (int a = 0; a < P.na; ++a)
                    for (int i = 0; i < shifts; i += atoms)
                        if (!add(base_tile + a, base_px + i, rl, ph + st * i, P.row_atoms ? P.rc : std::min(atoms, shifts - i), a * P.ca)) return false;
            }
        }
    P.s_inner = !P.merged && P.s > 1 && P.ws_s < P.ws_c;
    if (P.cols > kMaxCols) return false;
    P.tmem_cols = 32;
    while (P.tmem_cols < 2 * P.cols) P.tmem_cols *= 2;
    return true;
}

// Fills the chunk-dependent fields; false when the candidate does not fit.  bare: kImages without halo columns.
bool shape_chunk(ClParams& P, int ci, int bp, int order, bool bare = false)
{
    const int st = P.stride;
    const int all_rows = P.stack ? P.h : P.p;
    const bool images = order == kImages, whole = images ? bp >= all_rows : ci > 1 || bp >= all_rows;
    if (order == kPaired) bp = round_up(bp, 2);
    if (order == kPixels && !whole && bp * P.q % 16 != 0) return false;         // k-steps do not cross chunks
    P.ci = ci; P.bp = bp; P.order = order;
    P.cpi = whole ? 0 : ceil_div(all_rows, bp);
    P.mma_cols = 0;
    P.chunks = whole ? ceil_div(P.n, ci) : ceil_div(P.n, ci) * P.cpi;
    P.px_rows = images ? ci : 1;
    P.skip = images && !bare && !P.stack && whole && P.rc == 1 && P.q * ci % 16 == 0 ? P.q * ci / 16 : 0;
    const int wp = bare ? P.w : P.q + ceil_div(P.s, st) - 1, above = P.stack ? P.rc - 1 : 0, halo = st == 1 && !P.stack ? P.rc - 1 : 0;
    const bool same = order == kFlat && ci > 1;          // (images of both operands at the same distance)
    const int x_rows = bp + halo + (same ? above : 0), dy_rows = bp + above + (same ? halo : 0), dy_w = order == kFlat ? wp : P.q;
    if ((wp - 1) * st + 1 > kMaxMapBox || (x_rows - 1) * st + 1 > kMaxMapBox || dy_rows > kMaxMapBox || ci > kMaxMapBox) return false;
    P.x_pitch = wp; P.dy_pitch = dy_w; P.x_img = x_rows * wp; P.dy_img = dy_rows * dy_w;
    const int steps_img = order == kPaired ? (bp / 2) * (P.q / 8) : ceil_div(bp * P.q, 16);
    P.ksteps = order == kFlat ? ceil_div(ci > 1 ? ci * dy_rows * dy_w : bp * dy_w, 16) : images ? ceil_div(bp * P.q * ci, 16) : ci * steps_img;
    if (P.ksteps > kMaxKsteps) return false;
    const int xb = P.ca * 2, db = P.ka * 2;
    P.x_box = ci * x_rows * wp * xb;
    if (order == kPixels) {          // one box per 64 pixels: rows of 128 bytes, one per output channel
        P.dy_subs = ceil_div(bp * P.q, 64);
        P.katoms = ci * P.dy_subs;
        P.dy_box = std::min(P.kt, P.k) * 128;
        P.dy_alloc = round_up(P.kt * 128, 1024);
    } else {
        P.dy_box = ci * dy_rows * dy_w * db;
        P.dy_alloc = round_up(std::max(P.dy_box, order == kPaired ? 0 : (P.ksteps * 16 + above * dy_w * P.px_rows) * db), 1024);
    }
    // last X row an MMA touches: last k-step, last row and column shift, unused shifts of the c-side form
    // (kImages: in whole pixels, one more where the last k-step is half a k-step)
    const int last = order == kFlat ? P.ksteps * 16 - 1 : ((images ? 1 : ci) - 1) * P.x_img + (bp - 1) * wp + P.q - 1 + (order == kPixels ? wp - P.q + 8 : 0) + (images && ci % 16 != 0 ? 1 : 0);
    const int zeros = P.stack && images && ci == 8 && bp * P.q % 2 != 0 ? P.x_img + 1 + far_shift(P) : 0;      // pixels, see below
    P.x_pre = bare ? round_up(std::max(P.pad_w, 1) * ci * xb, 1024) : 0;
    const int far = P.row_atoms ? last + (128 / P.ca - 1) * wp : last + halo * wp + (images ? far_shift(P) : ceil_div(P.s, st) - 1 + (P.c_side ? 128 / P.ca : 256 / P.ca));
    P.x_alloc = P.x_pre + round_up(bare ? P.x_box : std::max(P.x_box, std::max(far + 1, zeros) * P.px_rows * xb), 1024);
    const int x_tiles = P.na * P.phases * P.row_tiles;
    P.x_plane = x_tiles * P.x_alloc;
    P.dy_plane = P.katoms * P.dy_alloc;
    P.x_region = P.planes * P.dy_plane;
    P.stage_bytes = P.x_region + P.planes * P.x_plane;
    if (P.planes * (P.katoms + x_tiles) > 32) return false;        // one copy per lane of a producer
    // (stack: idle atoms of the last stage read on past their rows; what they read is multiplied into rows that nobody reads)
    const int reach = P.stack ? (P.planes - 1) * P.dy_plane + (P.ksteps * 16 + (ci - 1) * P.dy_img + 128 / P.ka * dy_w * P.px_rows + 2 * dy_w) * db : 0;
    P.slack = std::max(0, reach - P.stage_bytes);
    P.stages = std::min(kMaxStages, (kStageBudget - P.slack) / P.stage_bytes) & ~1;
    P.epoch = std::max(1, (P.nprod > 1 ? 16 : 64) / P.ksteps);
    if (P.stages < 2) return false;
    P.tx_bytes = (uint32_t)(P.planes * (P.katoms * P.dy_box + x_tiles * P.x_box));
    if (P.tx_bytes >= (1u << 20)) return false;
    const uint32_t x_swz = P.ca == 64 ? 2 : P.ca == 32 ? 4 : 6, dy_swz = order == kPixels || P.ka == 64 ? 2 : P.ka == 32 ? 4 : 6;
    const uint32_t dy_sbo = order == kPixels ? 8 * 128 : order == kPaired ? dy_w * db : 8 * db;
    P.dy_hi = (dy_sbo >> 4) | (1u << 14) | (dy_swz << 29);
    P.x_lbo = (uint32_t)((P.merged ? P.x_alloc : (P.row_atoms ? wp : 1) * P.px_rows * xb) >> 4) << 16;
    // (one atom: the upper half of M repeats the lower)
    P.dy_lbo = P.stack ? (uint32_t)(dy_w * P.px_rows * db >> 4) << 16 : order == kPixels ? 1u << 16 : (uint32_t)((P.katoms > 1 ? P.dy_alloc : 0) >> 4) << 16;
    for (int i = 0; i < P.ksteps; ++i) {
        int s_lo = 0, s_hi = 0;                                        // bare: column shifts of the k-step
        int x_row = 16 * i, dy_off = 16 * i * db, x_sbo = 8;          // X row, dY bytes, X rows between the two 8-pixel groups
        if (order == kPaired) {
            const int j = i % (P.q / 8), t = i / (P.q / 8), pr = t % (bp / 2), im = t / (bp / 2);
            x_row = im * P.x_img + 2 * pr * wp + 8 * j;
            dy_off = (im * P.dy_img + 2 * pr * dy_w + 8 * j) * db;
            x_sbo = wp;
        } else if (images) {
            const int px = 16 * i / ci, p = px / P.q, q = px % P.q;
            x_row = (p * wp + q) * ci + 16 * i % ci;
            // (the other half of a last half k-step: in the stack form dY has rows there, so X must read zeros, those behind the tile)
            if (P.stack && ci == 8 && px + 1 == bp * P.q) x_sbo = P.x_img * ci - x_row;
            if (bare) {
                // the shifts whose column lies in the map; pixel 0 takes all of them, those to the left from the zeros before the
                // tile, so that the MMA that starts an accumulator writes every column of it
                if (px > 0) { s_lo = std::max(0, P.pad_w - q); s_hi = std::min(P.s, P.w + P.pad_w - q); }
                x_row += (s_lo - P.pad_w) * ci + P.x_pre / xb;
            }
            if (ci == 8 && q + 1 == P.q && px + 1 < bp * P.q) x_sbo = 8 * (wp - P.q + 1);       // the second pixel starts the next row
        } else if (order == kPixels) {
            const int im = i / steps_img, j = 16 * (i % steps_img), p = j / P.q, q = j % P.q;
            x_row = im * P.x_img + p * wp + q;
            dy_off = (im * P.dy_subs + j / 64) * P.dy_alloc + (j % 64) * 2;
            x_sbo = q + 8 < P.q ? 8 : wp - P.q + 8;
        }
        P.k_off[i] = make_uint4((unsigned)(x_row * xb) >> 4, (unsigned)dy_off >> 4, (unsigned)(x_sbo * xb) >> 4 | (1u << 14) | (x_swz << 29),
                                (unsigned)(s_lo * P.ca) | (unsigned)((bare ? (s_hi - s_lo) * P.ca : 0) >> 3) << 17);
    }
    if (!build_groups(P)) return false;
    if (!P.c_side && P.ngroups == 1)
        for (int i = 0; i < P.ksteps; ++i) {
            if (!bare || P.k_off[i].w >> 17 == 0) P.k_off[i].w = P.g[0].idesc;
            P.mma_cols += (P.k_off[i].w >> 17) * 8;
        }
    else P.mma_cols = P.ksteps * P.cols;
    return true;
}

struct ClHost {             // what ClPlan::opaque holds
    ClParams p;
    bool pack_x, pack_dy, f32, x_nhwc, dy_npqk;
    int xch[2], dych[2];    // elements from one pixel of the operands to the next: packed tightly, and on aligned rows
    int log_cb, groups;     // second kernel: columns per block, split groups per column
    bool lean;              // second kernel: with few registers
    ClReduce reduce;
};
static_assert(sizeof(ClHost) <= sizeof(ClPlan::opaque), "ClPlan::opaque too small");

// Elements from one pixel of a packed operand to the next.  64-channel boxes are read a pixel, 128 bytes, at a time: where pixels lie 240
// bytes apart (120 channels) most reads take two lines.  So rows are spread to whole multiples of 128 bytes where that makes the operand
// no more than a third longer (bf16 72->120 on 28x20, N = 100: main loop 27,000 -> 22,500 cycles, whole call 36.2 -> 33.9 us; 24->100 on
// 28x28, N = 60 22.4 -> 22.0).  Not 72 channels (21,200 cycles on rows of 144 bytes against 22,500 on 256), nor the planes of fp32
// operands, whose six products hide the reads (40->40 on 28x28, N = 60 47.0 / 52.7).
int wide_pitch(int ch, int atom)
{
    const int tight = round_up(ch, 8), wide = round_up(ch, atom);
    return atom == 64 && 3 * wide <= 4 * tight ? wide : tight;
}

PackOp pack_op(const void* src, void* dst, int ch, int pitch, int px, int n, bool last, int tile_px)
{
    PackOp o{};
    o.src = src; o.dst = static_cast<__nv_bfloat16*>(dst);
    o.ch = ch; o.chp = round_up(ch, 8); o.pitch = pitch; o.px = px; o.n = n; o.channels_last = last ? 1 : 0; o.plane = (size_t)n * px * pitch;
    const int vec = tile_px == kPackPx<float> ? 4 : 8;
    o.ch_tiles = ceil_div(ch, 64);
    o.ch_tile = round_up(ceil_div(ch, o.ch_tiles), 8);
    o.ch_tiles = ceil_div(ch, o.ch_tile);
    o.gather = px % 4 != 0 || ch <= 16;
    o.tile_px = tile_px;
    if (o.gather)                      // (few channels: more pixels, the same number of bytes)
        for (int c = o.ch_tile; c <= 32; c *= 2) o.tile_px *= 2;
    o.px_tiles = ceil_div(px, o.tile_px);
    // a slab: 16-byte pieces, up to 64 pixels of 64 channels; images enough for every thread to have work, blocks enough for every SM
    if (!last && px < 64 && (long long)ch * px % vec == 0) {
        o.ch_tile = 64; o.ch_tiles = ceil_div(ch, 64);
        o.slab = std::max(1, std::min(64 / px, n * o.ch_tiles / 296));
        o.blocks = ceil_div(n, o.slab) * o.ch_tiles;
        return o;
    }
    o.blocks = last ? (int)(((size_t)n * px * (o.chp / 8) + 1023) / 1024) : n * o.px_tiles * o.ch_tiles;
    return o;
}

typedef void (*ClKernel)(const CUtensorMap, const CUtensorMap, float*, float*, uint32_t*, const ClParams, const ClSource);
ClKernel kernel_for(int ng, bool f32, bool c_side)
{
#define GACONV_CL_PICK(N) if (ng <= N) return f32 ? (c_side ? cl_kernel<N, true, true> : cl_kernel<N, true, false>) : (c_side ? cl_kernel<N, false, true> : cl_kernel<N, false, false>);
    GACONV_CL_PICK(1) GACONV_CL_PICK(2) GACONV_CL_PICK(3) GACONV_CL_PICK(4) GACONV_CL_PICK(5) GACONV_CL_PICK(6) GACONV_CL_PICK(7) GACONV_CL_PICK(8)
    GACONV_CL_PICK(9) GACONV_CL_PICK(kMaxGroups)
#undef GACONV_CL_PICK
    return nullptr;
}

}  // namespace

namespace {
bool plan_problem(const Geom& g, bool dy_npqk, int vc, int vw, int vpad, size_t limit, ClPlan* out)
{
    if (g.stride_h != g.stride_w || g.stride_h > kMaxMapStep || g.r > 16 || g.s > 16 || !dw_offsets_fit(g)) return false;
    const bool nhwc = g.xs_c == 1 || (vc != 0 ? vc : g.c) == 1;
    ClHost H{};
    H.f32 = !g.bf16;
    H.x_nhwc = nhwc; H.dy_npqk = dy_npqk || g.k == 1;
    H.pack_x = H.f32 || !nhwc || g.c % 8 != 0 || vc != 0;
    H.pack_dy = H.f32 || !H.dy_npqk || g.k % 8 != 0;
    const size_t x_px = (size_t)g.n * g.h * g.w, dy_px = (size_t)g.n * g.p * g.q, x_el = x_px * round_up(g.c, 8), dy_el = dy_px * round_up(g.k, 8);
    if (x_el > ((size_t)1 << 31) || dy_el > ((size_t)1 << 31)) return false;

    ClParams B{};
    B.n = g.n; B.c = g.c; B.h = g.h; B.w = g.w; B.k = g.k; B.r = g.r; B.s = g.s; B.p = g.p; B.q = g.q;
    B.stride = g.stride_h; B.pad_h = g.pad_h; B.pad_w = g.pad_w; B.alpha = g.alpha;
    B.ws_k = g.ws_k; B.ws_c = g.ws_c; B.ws_r = g.ws_r; B.ws_s = g.ws_s;
    B.vc = vc; B.vw = vw; B.vpad = vpad;
    B.planes = H.f32 ? 3 : 1; B.nprod = H.f32 ? 6 : 1;
    B.phases = std::min(g.stride_h, g.s);
    B.ca = g.c > 32 ? 64 : g.c > 16 ? 32 : 16;
    const int sms = g.sm_budget > 0 ? std::min(g.sm_budget, device_sms()) : device_sms();

    ClParams best{};
    double best_cycles = 1e30;
    // a packing pass of dY: its launch, and its bytes twice
    const size_t x_copy = H.pack_x ? align_up(x_el * 2 * B.planes, 256) : 0, dy_copy = H.pack_dy ? align_up(dy_el * 2 * B.planes, 256) : 0;
    const double dy_pass = H.pack_dy ? 3500 + (double)dy_el * 2 * (1 + B.planes) / (16.0 * sms) : 0.0;
    for (int form = 0; form < 4; ++form) {           // k-side, c-side, stack, c-side with filter rows
        if (form == 3 && (g.s != 1 || g.r == 1 || g.stride_h != 1 || B.ca > 32)) break;
        if (form == 2 && (g.k > 64 || g.r == 1 || g.stride_h != 1)) continue;
        const int k16 = round_up(g.k, 16), all_rows = form == 2 ? g.h : g.p;
        const int kts[4] = {form == 2 ? (g.k > 32 ? 64 : k16) : form ? std::min(k16, 256) : 128, 128, 64, 32};
        for (int ki = 0; ki < (form & 1 ? 4 : 1); ++ki) {
            if (ki > 0 && (kts[ki] >= kts[0] || kts[ki] >= k16)) continue;
            ClParams F = B;
            F.c_side = form & 1; F.row_atoms = form == 3; F.stack = form == 2; F.kt = kts[ki];
            const int kw = std::min(F.kt, k16);
            F.ka = kw > 32 ? 64 : kw > 16 ? 32 : 16;
            F.katoms = ceil_div(kw, F.ka);
            F.tiles_k = ceil_div(g.k, F.kt);
            // (M side output channels, wide filters: fewer channels a tile, so that all shifts fit the accumulators; up to 64 outputs stack:
            // 5x5 86->37 on 10x13, N = 67 19.8 us, 21.0 without)
            for (int ca = B.ca; ca >= ((form == 2 && g.s > 3) || (form == 0 && g.s * B.ca > kMaxCols && (g.k > 64 || g.stride_h > 1)) ? 16 : B.ca); ca /= 2)
            for (int na = 1; na <= 4; na *= 2) {
                F.ca = ca;
                if (na > 1 && (F.ca < 64 || (na - 1) * 64 >= g.c)) break;
                if (form == 1 && na > 2) break;
                if (form == 3 && na > 1) break;
                if (form != 1 && na > 2 && g.s > 1) break;
                F.na = na; F.ct = na * F.ca;
                F.merged = na > 1 && (form == 1 || g.s == 1) ? 1 : 0;
                F.tiles_c = ceil_div(g.c, F.ct);
                for (int rc = form >= 2 ? 2 : 1; rc <= (form == 2 ? std::min(g.r, 128 / F.ka) : form == 3 ? std::min(g.r, 128 / F.ca) : g.r); ++rc) {
                    F.rc = rc; F.tiles_r = ceil_div(g.r, rc);
                    if (rc > 1 && ceil_div(g.r, rc) == ceil_div(g.r, rc - 1)) continue;
                    F.row_tiles = F.stride > 1 ? rc : 1;
                    if (F.stride == 1) F.phases = 1;
                    // part of the accumulator block that stands for elements of dW
                    const double share = (double)g.k * g.c * g.r * g.s / ((double)F.tiles_k * F.tiles_c * F.tiles_r * 128);
                    for (int mode = kFlat; mode <= kImages; ++mode) {
                        if ((mode == kPaired || mode == kPixels) && g.q % 8 != 0) continue;
                        // (small maps: one order for every layout of dY, so that its results do not depend on it either)
                        if (mode == kPixels && (form == 2 || H.f32 || H.dy_npqk || g.p * g.q < 64)) continue;
                        if (mode == kImages && g.n < 5) continue;
                        auto consider = [&](int ci, int bp, bool bare) {
                            ClParams C = F;
                            if (!shape_chunk(C, ci, bp, mode, bare)) return mode == kPixels && bp * C.q % 16 != 0;
#ifdef GACONV_TUNING
                            if (const char* e = getenv("GACONV_CL_KS")) if (C.ksteps < atoi(e)) return true;
                            if (const char* e = getenv("GACONV_CL_KSMAX")) if (C.ksteps > atoi(e)) return true;
                            if (const char* e = getenv("GACONV_CL_FORM")) if (C.c_side != atoi(e)) return true;
                            if (const char* e = getenv("GACONV_CL_RC")) if (C.rc != atoi(e)) return true;
                            if (const char* e = getenv("GACONV_CL_KT")) if (C.kt != atoi(e)) return true;
                            if (const char* e = getenv("GACONV_CL_MODE")) if (mode != atoi(e)) return true;
                            if (const char* e = getenv("GACONV_CL_STACK")) if (C.stack != atoi(e)) return true;
                            if (const char* e = getenv("GACONV_CL_BARE")) if ((C.x_pre > 0) != (atoi(e) != 0)) return true;
                            if (const char* e = getenv("GACONV_CL_NA")) if (C.na != atoi(e)) return true;
#endif
                            const size_t copies = x_copy + (mode == kPixels ? 0 : dy_copy);
                            if (copies > limit) return true;
                            Cost c = cost_of(C, sms, std::min(1.0, 1.3 * share / C.cols), limit - copies);
                            if (form == 2) c.cycles *= 1.07;          // (by a few per cent the other forms are as quick or quicker)
                            if (mode != kPixels) c.cycles += dy_pass;
                            if (c.cycles < best_cycles) { best_cycles = c.cycles; C.splits = c.splits; best = C; }
                            return true;
                        };
                        if (mode == kImages) {
                            for (int ci = 8; ci <= 64 && ci < 2 * g.n; ci *= 2) {
                                int last_bp = 0;
                                for (int parts = all_rows; parts >= 1; --parts) {
                                    const int bp = ceil_div(all_rows, parts);
                                    if (bp == last_bp) continue;
                                    last_bp = bp;
                                    if (!consider(ci, bp, false)) break;
                                }
                                // no halo columns: one MMA a k-step, of shifts alone, a first pixel with every shift inside or to the left, and
                                // no pixel without any (its window in the padding altogether)
                                if (g.pad_w < g.s && form != 1 && ci >= 16 && na == 1 && (rc == 1 || form == 2) && F.stride == 1 && g.s > 1 && g.s * F.ca <= kMaxCols && g.w >= g.s - g.pad_w && g.pad_w < g.w) {
                                    last_bp = 0;
                                    for (int parts = all_rows; parts >= 1; --parts) {
                                        const int bp = ceil_div(all_rows, parts);
                                        if (bp == last_bp) continue;
                                        last_bp = bp;
                                        if (!consider(ci, bp, true)) break;
                                    }
                                }
                            }
                            continue;
                        }
                        int last_bp = 0;
                        for (int parts = all_rows; parts >= 1; --parts) {      // fewer and fewer, larger and larger bands
                            int bp = ceil_div(all_rows, parts);
                            if (mode == kPaired) bp = round_up(bp, 2);
                            if (bp == last_bp) continue;
                            last_bp = bp;
                            if (!consider(1, bp, false)) break;
                        }
                        for (int ci = 2; ci <= 64 && ci <= g.n; ci = ci < 4 ? ci + 1 : ci + ci / 2)
                            if (!consider(ci, all_rows, false)) break;
                    }
                }
            }
        }
    }
    if (best_cycles >= 1e30) return false;
    best.chunk_base = best.chunks / best.splits;
    best.chunk_rem = best.chunks - best.chunk_base * best.splits;
    // fp32 accumulators, bf16 operands, both MN-major (dY K-major where it is read as it lies), M = 128; N is the group's
    best.idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | (8u << 24);
    if (best.order == kPixels) { best.idesc &= ~(best.c_side ? 1u << 16 : 1u << 15); H.pack_dy = false; }
    H.p = best;
    // second kernel: at most eight loads a thread, a block of at most 32 warps, and as many blocks as there are SMs where the
    // columns allow it
    H.groups = 1;
    while (H.groups < 32 && H.groups * 8 < best.splits) H.groups *= 2;
    H.log_cb = 4;
    while (H.log_cb > 0 && ((H.groups << H.log_cb) > 32 || best.tiles_k * best.tiles_c * best.tiles_r * ceil_div(best.cols, 1 << H.log_cb) < sms)) --H.log_cb;
    H.reduce.by_r = fast_div(best.tiles_r); H.reduce.by_c = fast_div(best.tiles_c);
    H.reduce.ws_c = (int)best.ws_c; H.reduce.atom_step = (int)(best.row_atoms ? best.ws_r : best.stride * best.ws_s);
    for (int e = 0; e < best.cols; ++e) {       // columns in the order of dW, see written_column
        const ClGroup* gr = best.g;
        while (gr + 1 < best.g + best.ngroups && e >= gr[1].col) ++gr;
        int j = e - gr->col;
        if (!best.c_side && best.s_inner) { const int atoms = gr->n / best.ca, c = j / atoms; j = (j - c * atoms) * best.ca + c; }
        const int a = best.c_side || best.merged ? 0 : j / best.ca, k = best.c_side ? j : 0, c = gr->cbase + (best.c_side ? 0 : best.merged ? j : j - a * best.ca);
        const int vs = vc != 0 ? c / vc : 0;
        H.reduce.col[e].off = (int)(k * best.ws_k + (c - vs * vc) * best.ws_c + (best.stack ? 0 : gr->r) * best.ws_r + (gr->s0 + best.stride * a + vs) * best.ws_s);
        H.reduce.col[e].info = (uint32_t)(gr->col + j) | (uint32_t)c << 8 | (uint32_t)gr->cnt << 16 | (uint32_t)gr->r << 20 | (uint32_t)k << 24;
    }
    const int tiles = best.tiles_k * best.tiles_c * best.tiles_r;
    H.lean = g.sm_budget > 0 || tiles * ceil_div(best.cols, 1 << H.log_cb) > sms * (65536 / (64 * 32 * H.groups << H.log_cb));
    if (tiles > 65535 || best.splits > 65535) return false;
    out->cycles = best_cycles;
    out->dy_pass = best.order == kPixels ? 0.0 : dy_pass;
    out->windows = vc != 0;
    out->partial_bytes = best.splits == 1 ? 0 : (size_t)tiles * best.splits * best.cols * 512;
    for (int wide = 0; wide < 2; ++wide) {
        H.xch[wide] = wide && H.pack_x && !H.f32 ? wide_pitch(g.c, best.ca) : round_up(g.c, 8);
        H.dych[wide] = wide && H.pack_dy && !H.f32 ? wide_pitch(g.k, best.ka) : round_up(g.k, 8);
        out->x_bytes[wide] = H.pack_x ? align_up(x_px * H.xch[wide] * 2 * best.planes, 256) : 0;
        out->dy_bytes[wide] = H.pack_dy ? align_up(dy_px * H.dych[wide] * 2 * best.planes, 256) : 0;
    }
    memcpy(out->opaque, &H, sizeof(H));
    return true;
}
}  // namespace

// Few input channels (image stems) leave most of an atom of 16 idle.  With stride 1 the columns of a window can stand in for channels: the
// packing pass, which such inputs need anyway, gathers s x c of them for every output column, and the filter becomes one of s = 1, whose
// rows are the atoms of one c-side MMA a k-step.  (Bound by operand reads before, with one MMA a filter row; us, plain / gathered: bf16 on
// 32x32 5x5 3->64, N = 128 25.1 / 15.4, 3x3 N = 256 23.9 / 20.8, 7x7 3->64 on 40x40, N = 50 19.2 / 15.2, fp32 5x5 3->64, N = 128 54.7 / 37.5,
// 3x3 3->40 on 30x30, N = 40 29.3 / 19.2.)  The gathered operand is longer, and so is its pass: a tenth of the estimate has to be gained
// (less lost: bf16 5x5 3->48 on 17x17, N = 30 12.2 / 13.1, estimated 11,100 / 10,100 cycles).  What both forms spend on packing dY is left out: it
// is there or not by the memory order of dY, which must not decide how its products are summed.  (Of 60 stems for which that moves the line, N = 9
// to 244, 36 gain more than 2 % from it, up to a quarter, 11 lose as much; geometric mean 0.96.)
bool plan_cl(const Geom& g, bool dy_npqk, size_t limit, ClPlan* out)
{
    const bool plain = plan_problem(g, dy_npqk, 0, 0, 0, limit, out);
    if (g.c > 4 || g.s < 2 || g.s * g.c > 32 || g.stride_h != 1 || g.stride_w != 1) return plain;
#ifdef GACONV_TUNING
    if (const char* e = getenv("GACONV_CL_VC")) if (atoi(e) == 0) return plain;
#endif
    Geom v = g;
    v.c = g.s * g.c; v.s = 1; v.w = g.q; v.pad_w = 0;
    ClPlan gathered;
    if (!plan_problem(v, dy_npqk, g.c, g.w, g.pad_w, limit, &gathered)) return plain;
    const double same = std::min(gathered.dy_pass, out->dy_pass);
    if (plain && 10 * (gathered.cycles - same) >= 9 * (out->cycles - same)) return plain;
    *out = gathered;
    return true;
}

cudaError_t launch_cl(const void* x, const void* dy, float* dw, float* partial, void* x_scratch, void* dy_scratch, uint32_t* status,
                      const ClPlan& plan, bool wide, cudaStream_t stream)
{
    ClHost H;
    memcpy(&H, plan.opaque, sizeof(H));
    const ClParams& P = H.p;
    cudaError_t err;
    const ClSource src{x, dy, H.f32, H.x_nhwc, H.dy_npqk};
    const int xch = H.xch[wide], dych = H.dych[wide];
    if (H.pack_x || H.pack_dy) {
        PackOp ox{}, od{};
        const int tile_px = H.f32 ? kPackPx<float> : kPackPx<unsigned short>;
        if (H.pack_x) ox = pack_op(x, x_scratch, P.c, xch, P.h * P.w, P.n, H.x_nhwc, tile_px);
        if (P.vc != 0) {
            ox.vc = P.vc; ox.vw = P.vw; ox.vpad = P.vpad; ox.q = P.w; ox.h = P.h;
            ox.blocks = (int)(((size_t)P.n * P.h * P.w * (ox.chp / 8) + 511) / 512);
        }
        if (H.pack_dy) od = pack_op(dy, dy_scratch, P.k, dych, P.p * P.q, P.n, H.dy_npqk, tile_px);
        const dim3 grid((unsigned)(ox.blocks + od.blocks));
        auto kern = H.f32 ? (P.vc ? pack_kernel<float, true> : pack_kernel<float, false>) : (P.vc ? pack_kernel<unsigned short, true> : pack_kernel<unsigned short, false>);
        err = launch_kernel(kern, grid, dim3(256), 0, stream, dim3(1, 1, 1), ox, od);
        if (err != cudaSuccess) return err;
        note_launch();
        if (H.pack_x) x = x_scratch;
        if (H.pack_dy) dy = dy_scratch;
    }
    // tensor maps over (channel, column, row, image, plane), the rows of a box in the order of the reduction; box extents count the pixels stepped over at the conv stride
    auto encode = [&](CUtensorMap* map, const void* base, int ch, int pitch, int w, int h, int atom, int bw, int bh, int st) {
        const cuuint64_t row = (cuuint64_t)pitch * 2;
        cuuint64_t dims[5] = {(cuuint64_t)ch, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)P.n, (cuuint64_t)P.planes};
        cuuint64_t strides[4] = {row, row * w, row * w * h, row * w * h * P.n};
        cuuint32_t box[5] = {(cuuint32_t)atom, (cuuint32_t)((bw - 1) * st + 1), (cuuint32_t)((bh - 1) * st + 1), (cuuint32_t)P.ci, 1};
        cuuint32_t es[5] = {1, (cuuint32_t)st, (cuuint32_t)st, 1, 1};
        if (P.order == kImages) {        // (channel, image, column, row, plane)
            for (int i : {2, 1}) { std::swap(dims[i], dims[i + 1]); std::swap(strides[i - 1], strides[i]); std::swap(box[i], box[i + 1]); std::swap(es[i], es[i + 1]); }
        }
        const CUtensorMapSwizzle swz = atom == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : atom == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
        return encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    CUtensorMap map_dy, map_x;
    auto encode_pixels = [&](CUtensorMap* map) {              // dY as (pixel, channel, image)
        const cuuint64_t pq = (cuuint64_t)P.p * P.q;
        cuuint64_t dims[3] = {pq, (cuuint64_t)P.k, (cuuint64_t)P.n}, strides[2] = {pq * 2, pq * P.k * 2};
        cuuint32_t box[3] = {64, (cuuint32_t)std::min(P.kt, P.k), 1}, es[3] = {1, 1, 1};
        return encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(dy), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    if (!(P.order == kPixels ? encode_pixels(&map_dy) : encode(&map_dy, dy, P.k, dych, P.q, P.p, P.ka, P.dy_pitch, P.dy_img / P.dy_pitch, 1)) ||
        !encode(&map_x, x, P.c, xch, P.w, P.h, P.ca, P.x_pitch, P.x_img / P.x_pitch, P.stride))
        return cudaErrorInvalidValue;
    // the stages; at the end they hold the accumulator block
    const size_t smem = std::max((size_t)P.stages * P.stage_bytes + P.slack, (size_t)P.cols * 512) + 1024;
    const dim3 grid((unsigned)(P.tiles_k * P.tiles_c * P.tiles_r), (unsigned)P.splits);
    ClKernel kern = kernel_for(P.ngroups, H.f32, P.c_side != 0);
    static std::atomic<unsigned long long> ready[kMaxGroups][2][2];
    if ((err = allow_shared_memory((const void*)kern, ready[P.ngroups > 9 ? kMaxGroups - 1 : P.ngroups - 1][H.f32][P.c_side])) != cudaSuccess) return err;
    if ((err = launch_kernel(kern, grid, dim3(kThreads), smem, stream, dim3(1, 1, 1), map_dy, map_x, dw, partial, status, P, src)) != cudaSuccess) return err;
    note_launch();
    if (P.splits == 1) return cudaSuccess;
    const dim3 rgrid((unsigned)ceil_div(P.cols, 1 << H.log_cb), grid.x);
    err = launch_kernel(H.lean ? cl_reduce_kernel<true> : cl_reduce_kernel<false>, rgrid, dim3(32u * H.groups << H.log_cb), 0, stream, dim3(1, 1, 1), static_cast<const float*>(partial), dw,
                        static_cast<const ClShape&>(P), src, H.reduce, H.log_cb, H.groups);
    if (err != cudaSuccess) return err;
    note_launch();
    return cudaSuccess;
}

}  // namespace gaconv

#ifdef GACONV_TUNING
extern "C" int gaconv_tuning_read_cl(long long* host) { return (int)cudaMemcpyFromSymbol(host, gaconv_tuning_cl, sizeof(gaconv_tuning_cl)); }
// tuning builds: the plan of a problem, as launch_cl would use it
extern "C" int gaconv_tuning_plan_cl(const int* v, int bf16, int x_nhwc, int npqk, int budget, void* out, int size)
{
    using namespace gaconv;
    Geom g{};
    g.n = v[0]; g.c = v[1]; g.h = v[2]; g.w = v[3]; g.k = v[4]; g.r = v[5]; g.s = v[6]; g.stride_h = g.stride_w = v[7]; g.pad_h = g.pad_w = v[8];
    g.p = (g.h + 2 * g.pad_h - g.r) / g.stride_h + 1; g.q = (g.w + 2 * g.pad_w - g.s) / g.stride_w + 1;
    g.xs_c = x_nhwc ? 1 : 2;
    g.ws_c = 1; g.ws_s = g.c; g.ws_r = g.s * g.c; g.ws_k = g.r * g.s * g.c;
    g.bf16 = bf16 != 0; g.alpha = 1.f; g.sm_budget = budget;
    ClPlan P;
    if (!plan_cl(g, npqk != 0, kNoLimit, &P) || size < (int)sizeof(ClHost)) return -1;
    memcpy(out, P.opaque, sizeof(ClHost));
    return (int)P.cycles;
}
#endif
