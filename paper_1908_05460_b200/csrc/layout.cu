// Operands given in the other order are brought into the kernels' own by one pass through shared memory into the
// caller's workspace: activations N x C x H x W -> N x H x W x C (what the tensor-core, stem and gather kernels are
// built for), output gradients N x P x Q x K -> N x K x P x Q.  (The paper's own kernel expects channels-last
// activations as well and pays the same transposition, Sections 2.4 and 3.1.)
#include "gaconv_internal.h"

#include <type_traits>

namespace gaconv {
namespace {

// out[b][j][i] = in[b][i][j] for i < c, j < hw.  A block turns a 32 x 32 tile; both the reads (along j) and the
// writes (along i) are contiguous.
template <typename T>
__global__ void __launch_bounds__(256)
transpose_batched_kernel(const T* __restrict__ in, T* __restrict__ out, int c, int hw)
{
    __shared__ T tile[32][33];
    pdl_release_next_grid();
    pdl_wait_prior_grid();
    const int n = blockIdx.z, j0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
    const T* src = in + (size_t)n * c * hw;
    T* dst = out + (size_t)n * c * hw;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int cc = ty; cc < 32; cc += 8)
        if (c0 + cc < c && j0 + tx < hw) tile[cc][tx] = src[(size_t)(c0 + cc) * hw + j0 + tx];
    __syncthreads();
    for (int jj = ty; jj < 32; jj += 8)
        if (j0 + jj < hw && c0 + tx < c) dst[(size_t)(j0 + jj) * c + c0 + tx] = tile[tx][jj];
}

// c a multiple of 16 bytes: a block turns 64 rows x 64 columns, all the loads of a thread in flight and 16-byte stores.
// A 32 x 32 tile with eight narrow loads a thread left too few bytes in flight.  (fp32, 22 MB of 24x24 maps with 240 channels:
// 16.5 -> 8.8 us; bf16, 12 MB of 26x17 maps with 496 channels: 15 -> 7.8 us.)
template <typename T>
__global__ void __launch_bounds__(256)
transpose_tiled_kernel(const T* __restrict__ in, T* __restrict__ out, int c, int hw)
{
    constexpr int V = 16 / sizeof(T);                    // elements of a store
    typedef typename std::conditional<sizeof(T) == 4, float4, uint2>::type Quad;
    __shared__ __align__(16) T tile[64][sizeof(T) == 4 ? 65 : 66];
    pdl_release_next_grid();
    const int n = blockIdx.z, j0 = blockIdx.x * 64, c0 = blockIdx.y * 64, rows = min(64, c - c0), cols = min(64, hw - j0);
    const T* src = in + ((size_t)n * c + c0) * hw + j0;
    T* dst = out + ((size_t)n * hw + j0) * c + c0;
    pdl_wait_prior_grid();
    if ((hw & 3) == 0) {
        const int q = threadIdx.x & 15, r0 = threadIdx.x >> 4;
        Quad v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            v[i] = r0 + 16 * i < rows && 4 * q < cols ? __ldg(reinterpret_cast<const Quad*>(src + (size_t)(r0 + 16 * i) * hw) + q) : Quad{};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            T* t = &tile[r0 + 16 * i][4 * q];
            const T* e = reinterpret_cast<const T*>(&v[i]);
            t[0] = e[0]; t[1] = e[1]; t[2] = e[2]; t[3] = e[3];
        }
    } else {
        const int x = threadIdx.x & 63, r0 = threadIdx.x >> 6;
        T v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = r0 + 4 * i < rows && x < cols ? __ldg(src + (size_t)(r0 + 4 * i) * hw + x) : T(0);
#pragma unroll
        for (int i = 0; i < 16; ++i) tile[r0 + 4 * i][x] = v[i];
    }
    __syncthreads();
    const int q = threadIdx.x % (64 / V), x0 = threadIdx.x / (64 / V);
#pragma unroll
    for (int x = x0; x < 64; x += 4 * V) {
        if (x < cols && V * q < rows) {
            float4 o;
            T* e = reinterpret_cast<T*>(&o);
#pragma unroll
            for (int i = 0; i < V; ++i) e[i] = tile[V * q + i][x];
            *reinterpret_cast<float4*>(dst + (size_t)x * c + V * q) = o;
        }
    }
}

}  // namespace

cudaError_t launch_transpose_batched(const void* in, void* out, int rows, int cols, int batch, bool bf16, cudaStream_t stream)
{
    if (rows % (bf16 ? 8 : 4) == 0 && batch <= 65535 && (rows + 63) / 64 <= 65535) {
        const dim3 grid((unsigned)((cols + 63) / 64), (unsigned)((rows + 63) / 64), (unsigned)batch);
        note_launch();
        return bf16 ? launch_kernel(transpose_tiled_kernel<unsigned short>, grid, dim3(256), 0, stream, dim3(1, 1, 1),
                                    static_cast<const unsigned short*>(in), static_cast<unsigned short*>(out), rows, cols)
                    : launch_kernel(transpose_tiled_kernel<float>, grid, dim3(256), 0, stream, dim3(1, 1, 1),
                                    static_cast<const float*>(in), static_cast<float*>(out), rows, cols);
    }
    const dim3 grid((unsigned)((cols + 31) / 32), (unsigned)((rows + 31) / 32), (unsigned)batch);
    if (grid.y > 65535u || grid.z > 65535u) return cudaErrorInvalidValue;
    note_launch();
    if (bf16)
        return launch_kernel(transpose_batched_kernel<__nv_bfloat16>, grid, dim3(256), 0, stream, dim3(1, 1, 1),
                             static_cast<const __nv_bfloat16*>(in), static_cast<__nv_bfloat16*>(out), rows, cols);
    return launch_kernel(transpose_batched_kernel<float>, grid, dim3(256), 0, stream, dim3(1, 1, 1), static_cast<const float*>(in),
                         static_cast<float*>(out), rows, cols);
}

}  // namespace gaconv
