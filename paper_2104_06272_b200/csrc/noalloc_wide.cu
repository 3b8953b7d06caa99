// Scratch of anakin_rollout_noalloc above 256 hidden units: those layers run the tcgen05 GEMMs of the handle-based rollout on one
// step's activations (h1 as three bf16 terms, h2) and three planes of W2.  2730 envs, H = 384, T = 24: 0.41 ms; on a plain FMA kernel
// that needs none of it 4.8 ms.  A file of its own is a module of its own: its 16 MiB are not loaded for narrower layers.
#include "common.cuh"

namespace anakin {

namespace {

constexpr size_t kMaxBH = ANAKIN_NOALLOC_MAX_BH, kMaxH = 1024;
constexpr size_t kH1Bytes = 3 * kMaxBH * 2, kH2Bytes = kMaxBH * 4, kW2Bytes = 3 * kMaxH * kMaxH * 2;
constexpr int kMaxDevices = 64;

// [ h1: three planes | h2 | W2: three planes ]
static __device__ __align__(256) unsigned char g_noalloc_wide[kH1Bytes + kH2Bytes + kW2Bytes];

unsigned char* g_wide_ptr[kMaxDevices] = {nullptr};  // device address of the array, per device ordinal

}  // namespace

// Points b's h1, h2 and W2 planes into the current device's array (the first call on a device resolves its address).
cudaError_t noalloc_wide_scratch(Buffers* b) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (!g_wide_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_wide);
        if (e != cudaSuccess) return e;
        g_wide_ptr[dev] = static_cast<unsigned char*>(p);
    }
    unsigned char* w = g_wide_ptr[dev];
    b->h1 = reinterpret_cast<float*>(w);
    b->h2 = reinterpret_cast<float*>(w + kH1Bytes);
    b->w2p_hi = reinterpret_cast<uint16_t*>(w + kH1Bytes + kH2Bytes);
    return cudaSuccess;
}

}  // namespace anakin
