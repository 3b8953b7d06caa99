// Agent plane of dW1 and S = sum over t of dh1 in one pass over dh1 (Podracer paper, Section 3.1: part of the batch-mean
// gradient), for the wide hidden layers whose dh1 goes through HBM.
//
// The agent plane of the observation is one-hot, so its weight gradient is a sum of dh1 rows by agent cell:
//   dW1[C + c] = sum over rows with pos = c of dh1[row].
// A warp owns 32 hidden units and walks tiles of eight envs over all steps: the row's values go into the warp's own [C][32]
// accumulator in shared memory (lane = unit: no conflicts, no atomics, fixed order) and into eight registers for S.  Plain fp32
// additions, exact inputs, one read of dh1.  Bound by the latency of its loads (each warp keeps 32 rows in flight) beside the
// read-modify-write chain: 48 us for 48,000 rows x 512 on 121 cells (2 TB/s), where the FFMA form of the one-hot product and the
// separate sum over t took 486 us.  (The bf16 workload keeps its tensor-core one-hot GEMM: at 256 cells only six such warps fit
// on an SM and the same sums took 1.2 ms against 0.38 ms.)
#include "env_step.cuh"

namespace anakin {

namespace {

constexpr int AG_ENVS = 8;

// Warps per CTA: two CTAs per SM, each warp (C + 1) x 128 bytes of accumulator.
int agent_warps(int C) {
    const int w = (113 * 1024) / ((C + 1) * 128);
    return w < 1 ? 1 : w > 8 ? 8 : w;
}

__global__ void __launch_bounds__(256) k_agent_plane(LearnArgs a, float* part, size_t stride) {
    PDL_START();
    extern __shared__ float s_acc[];  // [warps][C + 1][32]
    const Dims& d = a.d;
    const Buffers& b = a.b;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int H = d.H, C = d.C, B = d.B, T = a.T;
    const int col = blockIdx.x * 32 + lane;
    float* acc = s_acc + (size_t)wid * (C + 1) * 32 + lane;  // row C takes what belongs to no cell
    for (int i = threadIdx.x; i < nw * (C + 1) * 32; i += blockDim.x) s_acc[i] = 0.f;
    __syncthreads();
    const int ntiles = (B + AG_ENVS - 1) / AG_ENVS;
    uint16_t* S = reinterpret_cast<uint16_t*>(b.S);
    const size_t SP = (size_t)B * H;  // elements of one plane of S
    for (int tile = blockIdx.y * nw + wid; tile < ntiles; tile += gridDim.y * nw) {
        const int e0 = tile * AG_ENVS, n = min(AG_ENVS, B - e0);
        // DEPTH steps of loads stay in flight: a slot is refilled as soon as its values have been added.  Loads past the last
        // step or env repeat a valid row (no branches around them) and go to row C.
        constexpr int DEPTH = 4;
        float s[AG_ENVS], v[DEPTH][AG_ENVS];
        int pos[DEPTH];
#pragma unroll
        for (int q = 0; q < AG_ENVS; ++q) s[q] = 0.f;
        const float* src = b.dh1 + (size_t)e0 * H + col;
        auto load = [&](int t, float (&x)[AG_ENVS], int& p) {
            const size_t i0 = (size_t)min(t, T - 1) * B;
            p = b.tpos[i0 + e0 + min(lane, n - 1)];  // lane q holds env q's cell
#pragma unroll
            for (int q = 0; q < AG_ENVS; ++q) x[q] = __ldg(src + (i0 + min(q, n - 1)) * H);
        };
#pragma unroll
        for (int k = 0; k < DEPTH; ++k) load(k, v[k], pos[k]);
        for (int t0 = 0; t0 < T; t0 += DEPTH) {
#pragma unroll
            for (int k = 0; k < DEPTH; ++k) {
                if (t0 + k < T) {
                    const int pk = (lane < n && pos[k] < C) ? pos[k] : C;
#pragma unroll
                    for (int h = 0; h < AG_ENVS; h += 4) {
                        int c[4];
                        float x[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            c[q] = __shfl_sync(0xFFFFFFFFu, pk, h + q) * 32;
                            x[q] = v[k][h + q];
                            s[h + q] += x[q];
                        }
                        // four different cells: the read-modify-writes overlap; otherwise one after the other (same order)
                        if (c[0] != c[1] && c[0] != c[2] && c[0] != c[3] && c[1] != c[2] && c[1] != c[3] && c[2] != c[3]) {
                            float o[4];
#pragma unroll
                            for (int q = 0; q < 4; ++q) o[q] = acc[c[q]];
#pragma unroll
                            for (int q = 0; q < 4; ++q) acc[c[q]] = o[q] + x[q];
                        } else {
#pragma unroll
                            for (int q = 0; q < 4; ++q) acc[c[q]] += x[q];
                        }
                    }
                }
                load(t0 + k + DEPTH, v[k], pos[k]);
            }
        }
#pragma unroll
        for (int q = 0; q < AG_ENVS; ++q) {
            if (q < n) {  // S as its three bf16 terms
                uint32_t tm[3];
                split3(s[q], 0.f, tm);
                for (int p = 0; p < 3; ++p) S[p * SP + (size_t)(e0 + q) * H + col] = (uint16_t)tm[p];
            }
        }
    }
    __syncthreads();
    float* out = part + (size_t)blockIdx.y * stride + blockIdx.x * 32;
    for (int i = threadIdx.x; i < C * 32; i += blockDim.x) {
        float v = s_acc[i];
        for (int w = 1; w < nw; ++w) v += s_acc[(size_t)w * (C + 1) * 32 + i];  // in warp order
        out[(size_t)(i >> 5) * H + (i & 31)] = v;
    }
}

}  // namespace

// Env groups (= partials): two CTAs per SM over the H / 32 column groups, no more than there are env tiles.
int agent_plane_splits(const Dims& d) {
    const int cols = d.H / 32, tiles = (d.B + AG_ENVS - 1) / AG_ENVS, w = agent_warps(d.C);
    int ns = 2 * 148 / cols;
    const int cap = (tiles + w - 1) / w;
    if (ns > cap) ns = cap;
    return ns < 1 ? 1 : ns;
}

cudaError_t launch_agent_plane(const LearnArgs& a, int ns, float* part, size_t stride, const Ctx& c) {
    const int w = agent_warps(a.d.C);
    const size_t smem = (size_t)w * (a.d.C + 1) * 128;
    Scope sc(c, K_DW1_AGENT);
    return launch<k_agent_plane>(dim3(a.d.H / 32, ns), 32 * w, smem, c.s, a, part, stride);
}

}  // namespace anakin
