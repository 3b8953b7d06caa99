// Copies within the GPU: strided blocks between the caller's contiguous buffers and the per-policy sub-workspaces, and single blobs.
#include "common.cuh"

namespace anakin {

// rows blocks of `words` words, dst and src advancing by their own pitch (in words).  One CTA column walks a block in steps of
// four words per thread; consecutive threads touch consecutive words, so either side is coalesced whatever its alignment.
// Bound by HBM on the parameter-sized blobs.  It replaces one memcpy per policy: 1024 policies x 42 KB took 3.6 ms (each copy
// costs 3.5 us on the stream), one launch takes 20 us.
template <class W>
__global__ void __launch_bounds__(256) k_copy_blocks(W* dst, size_t dpitch, const W* src, size_t spitch, size_t words, size_t rows) {
    PDL_START();
    for (size_t r = blockIdx.y; r < rows; r += gridDim.y) {
        const W* s = src + r * spitch;
        W* o = dst + r * dpitch;
        for (size_t i = (size_t)blockIdx.x * 1024 + threadIdx.x; i < words; i += (size_t)gridDim.x * 1024) {
            W v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i + 256 * q < words) v[q] = s[i + 256 * q];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i + 256 * q < words) o[i + 256 * q] = v[q];
        }
    }
}

cudaError_t launch_copy_blocks(void* dst, size_t dpitch, const void* src, size_t spitch, size_t bytes, size_t rows, cudaStream_t s) {
    if (rows == 0 || bytes == 0) return cudaSuccess;
    const bool w4 = (((uintptr_t)dst | (uintptr_t)src | dpitch | spitch | bytes) & 3) == 0;
    const size_t words = w4 ? bytes / 4 : bytes;
    const size_t gx = (words + 1023) / 1024;
    const dim3 grid((unsigned)(gx < 1024 ? gx : 1024), (unsigned)(rows < 65535 ? rows : 65535));
    if (w4) launch<k_copy_blocks<uint32_t>>(grid, 256, 0, s, (uint32_t*)dst, dpitch / 4, (const uint32_t*)src, spitch / 4, words, rows);
    else launch<k_copy_blocks<uint8_t>>(grid, 256, 0, s, (uint8_t*)dst, dpitch, (const uint8_t*)src, spitch, words, rows);
    return cudaGetLastError();
}

// One block of `n` words of W, four in flight a thread.  For blobs of up to a few megabytes, where a memcpy's own cost on the stream (3.5 us
// each, and the gaps around it: it is no programmatic dependent) is most of the time: see COPY_KERNEL_MAX.
template <class W>
__global__ void __launch_bounds__(256) k_copy_flat(W* __restrict__ dst, const W* __restrict__ src, size_t n, uint8_t* dst_tail, const uint8_t* src_tail, int tail) {
    PDL_START();
    for (size_t i = (size_t)blockIdx.x * 1024 + threadIdx.x; i < n; i += (size_t)gridDim.x * 1024) {
        W v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (i + 256 * q < n) v[q] = src[i + 256 * q];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (i + 256 * q < n) dst[i + 256 * q] = v[q];
    }
    if (blockIdx.x == 0 && (int)threadIdx.x < tail) dst_tail[threadIdx.x] = src_tail[threadIdx.x];
}

cudaError_t launch_copy_flat(void* dst, const void* src, size_t bytes, cudaStream_t s) {
    const uintptr_t both = (uintptr_t)dst | (uintptr_t)src;
    const size_t w = (both & 15) == 0 ? 16 : (both & 3) == 0 ? 4 : 1, n = bytes / w, gx = (n + 1023) / 1024;
    const int tail = (int)(bytes - n * w);
    uint8_t* dt = static_cast<uint8_t*>(dst) + n * w;
    const uint8_t* st = static_cast<const uint8_t*>(src) + n * w;
    const unsigned grid = (unsigned)(gx < 1 ? 1 : gx < 148 * 8 ? gx : 148 * 8);
    if (w == 16) launch<k_copy_flat<uint4>>(grid, 256, 0, s, (uint4*)dst, (const uint4*)src, n, dt, st, tail);
    else if (w == 4) launch<k_copy_flat<uint32_t>>(grid, 256, 0, s, (uint32_t*)dst, (const uint32_t*)src, n, dt, st, tail);
    else launch<k_copy_flat<uint8_t>>(grid, 256, 0, s, (uint8_t*)dst, (const uint8_t*)src, n, dt, st, tail);
    return cudaGetLastError();
}

}  // namespace anakin
