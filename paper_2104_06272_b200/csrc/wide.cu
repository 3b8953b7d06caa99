// Wide-network path (hidden widths 384, 512, 768, 1024, both precisions): the layer-2 products of the Anakin minimal unit
// (Podracer paper, Section 3.1; Figure 2, top) as large GEMMs on the 5th-generation tensor cores.
//
// With a hidden layer this wide W2 no longer fits on chip next to a CTA's activations, so the acting half runs as two
// launches per environment step instead of one persistent kernel, after one for the first step's h1:
//   k_h1_wide      h1 = relu(base[env] + W1[agent row])                        gather-add, HBM-bound (first step, replays)
//   GEMM           h2 = relu(h1 W2 + b2)                                       tcgen05, persistent, bias/ReLU epilogue
//   k_heads_wide   out = h2 Wh + bh, softmax / Philox sample / env step, then h1 of the next step
// h1 and h2 of every recorded row stay in HBM for the update, which runs the GEMM once more for dh1 = (dh2 W2^T) gated by
// h1 > 0 over all B*T rows.  In bf16 the GEMM is k_gemm_nt_tc (below) or the CTA-pair kernel (wide2.cu), activations are one bf16
// plane and k_sum_t_wide forms S = sum over t of dh1; fp32 runs x3_gemm.cu on three bf16 terms and k_agent_plane for S.
//
// k_gemm_nt_tc: C[m][n] = sum_k A[m][k] Bop[k][n] with A row-major (K-major for the MMA).  One persistent CTA per SM walks
// 128 x 256 output tiles (n fastest, so that the CTAs running together share A tiles through L2):
//   warp 0 (one lane)  TMA producer: 64-wide k chunks of A (128 rows) and B (256 columns) into a 3-stage ring
//   warp 1             tcgen05.mma issuer (the whole warp walks the loop, an elected lane issues), four k16 MMAs per chunk into one of two 256-column fp32 accumulators in TMEM
//   warps 2-9          epilogue of tile i while the MMAs of tile i+1 run: tcgen05.ld, bias + ReLU (or gate), bf16, store
// B is either K-major (rows = n: W2 as stored, for dh2 W2^T) or MN-major (rows = k: W2 as stored, for h1 W2).
// Every wait is bounded; a timeout raises DEV_E_WAIT_TIMEOUT and the CTA unwinds (tensor memory freed).
#include <cstring>

#include "wide_gemm.cuh"

namespace anakin {

// Hidden layers too wide for the persistent rollouts, in either precision (bf16 at 512 / 1024 is the headline form).
bool wide_supported(int H) { return H == 384 || H == 512 || H == 768 || H == 1024; }

namespace {

using namespace widegemm;

template <int BN_>
struct NtCfg {
    static constexpr int BM = 128, BN = BN_, KC = 64, STAGES = BN == 256 ? 3 : BN == 128 ? 5 : 6, THREADS = 320, MAXN = NT_MAXN;
    static constexpr int A_BYTES = BM * KC * 2, B_BYTES = BN * KC * 2, STAGE = A_BYTES + B_BYTES;
    static constexpr size_t smem_bytes = (size_t)STAGES * STAGE + 1024 /*alignment slack*/ + 256 /*barriers, tmem slot*/ + MAXN * 4 + NT_EPI_WARPS * NT_STAGE_BYTES;
};

template <int EPI, bool B_MN, int BN_>
__global__ void __launch_bounds__(320, 1) k_gemm_nt_tc(const __grid_constant__ NtMaps maps, NtArgs g) {
    using Cfg = NtCfg<BN_>;
    constexpr int BM = Cfg::BM, BN = Cfg::BN, KC = Cfg::KC, STAGES = Cfg::STAGES;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);  // the swizzle needs 1024-byte alignment
    uint64_t* bars = (uint64_t*)(base + STAGES * Cfg::STAGE);
    uint64_t* full = bars;                // [STAGES]
    uint64_t* empty = bars + STAGES;      // [STAGES]
    uint64_t* tfull = bars + 2 * STAGES;  // [2] accumulator written
    uint64_t* tempty = tfull + 2;         // [2] accumulator drained (4 epilogue warps arrive)
    uint32_t* tmem_slot = (uint32_t*)(tempty + 2);
    float* s_bias = (float*)(base + STAGES * Cfg::STAGE + 256);
    unsigned char* s_stage = (unsigned char*)(s_bias + NT_MAXN);  // [NT_EPI_WARPS][NT_STAGE_BYTES]
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const int nt = (g.N + BN - 1) / BN, mt = (g.M + BM - 1) / BM, ntiles = mt * nt, nch = g.K / KC;

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) { tc::mbar_init(&full[s], 1); tc::mbar_init(&empty[s], 1); }
        for (int i = 0; i < 2; ++i) { tc::mbar_init(&tfull[i], 1); tc::mbar_init(&tempty[i], NT_EPI_WARPS); }
        tc::mbar_fence_init();
    }
    if (wid == 2) tc::tmem_alloc(tmem_slot, 2 * BN);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();  // (the set-up above runs under the predecessor's tail)
    if (EPI != EPI_GATE) {
        for (int i = tid; i < g.N; i += Cfg::THREADS) s_bias[i] = g.bias[i];
        __syncthreads();
    }
    bool ok = true;

    if (wid == 0) {
        if (lane == 0) {  // ---- TMA producer
            int c = 0;
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
                const int m0 = (tile / nt) * BM, n0 = (tile % nt) * BN;
                for (int kc = 0; kc < nch; ++kc, ++c) {
                    const int s = c % STAGES;
                    if (c >= STAGES) ok = tc::mbar_wait(&empty[s], ((c / STAGES) - 1) & 1);
                    if (!ok) break;
                    unsigned char* sa = base + s * Cfg::STAGE;
                    unsigned char* sb = sa + Cfg::A_BYTES;
                    tc::mbar_expect_tx(&full[s], Cfg::STAGE);
                    // rows past M belong to later rows of the buffer or are zero-filled; the epilogue drops them
                    tc::tma_load_2d(sa, &maps.a, &full[s], kc * KC, g.row0 + m0);
                    if (B_MN) {
#pragma unroll
                        for (int bx = 0; bx < BN / 64; ++bx) tc::tma_load_2d(sb + bx * 8192, &maps.b, &full[s], n0 + 64 * bx, kc * KC);
                    } else {
#pragma unroll
                        for (int bx = 0; bx < BN; bx += 128) tc::tma_load_2d(sb + bx * 128, &maps.b, &full[s], kc * KC, n0 + bx);  // boxes of 128 rows (n), 64 for a 64-wide tile
                    }
                }
            }
            if (!ok) atomicOr(g.status, DEV_E_WAIT_TIMEOUT);
        }
    } else if (wid == 1) {
        {  // ---- MMA issuer: the whole warp walks the loop, one elected lane issues
            const uint32_t idesc = tc::umma_idesc<1>(BM, BN, false, B_MN);
            int c = 0, u = 0;
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++u) {
                const int buf = u & 1;
                if (u >= 2) ok = tc::warp_all(tc::mbar_wait(&tempty[buf], ((u >> 1) - 1) & 1));  // the epilogue of tile u-2 has drained it
                if (!ok) break;
                tc::tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)(buf * BN);
                for (int kc = 0; kc < nch; ++kc, ++c) {
                    const int s = c % STAGES;
                    ok = tc::warp_all(tc::mbar_wait(&full[s], (c / STAGES) & 1));
                    if (!ok) break;
                    tc::tc_fence_after();
                    unsigned char* sa = base + s * Cfg::STAGE;
                    unsigned char* sb = sa + Cfg::A_BYTES;
                    if (tc::elect_one()) {
#pragma unroll
                    for (int k16 = 0; k16 < KC / 16; ++k16) {
                        // K-major: 16 k = 32 bytes along the swizzled 128-byte rows; MN-major: 16 k rows = 2048 bytes
                        const uint64_t ad = tc::umma_desc(sa + k16 * 32, 16, 1024);
                        const uint64_t bd = B_MN ? tc::umma_desc(sb + k16 * 2048, 8192, 1024) : tc::umma_desc(sb + k16 * 32, 16, 1024);
                        tc::umma(acc, ad, bd, idesc, (kc > 0 || k16 > 0) ? 1u : 0u);
                    }
                    tc::umma_commit(&empty[s]);
                    if (kc == nch - 1) tc::umma_commit(&tfull[buf]);
                    }
                    __syncwarp();
                }
            }
            if (!ok && lane == 0) atomicOr(g.status, DEV_E_WAIT_TIMEOUT);
        }
    } else {
        // ---- epilogue warps: accumulator lanes 32*(wid%4)..+31 = output rows
        const int q = wid & 3, half = (wid - 2) >> 2;
        int u = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++u) {
            const int buf = u & 1;
            const int m0 = (tile / nt) * BM, n0 = (tile % nt) * BN;
            const int m = m0 + 32 * q + lane;
            const bool valid = m < g.M;
            const size_t gi = ((size_t)g.row0 + (valid ? m : 0)) * g.N + n0;
            if (EPI == EPI_GATE && valid) nt_prefetch_gate(g, gi, g.N - n0 < BN ? g.N - n0 : BN);  // towards L2 while the MMAs run
            ok = tc::mbar_wait(&tfull[buf], (u >> 1) & 1);
            if (!ok) break;
            tc::tc_fence_after();
            constexpr int HW = BN >= 128 ? BN / 2 : 64;  // two column halves; the epilogue takes 64 columns at a time, so a 64-wide tile is one half's
            nt_epilogue_warp<EPI>(g, s_bias, s_stage + (wid - 2) * NT_STAGE_BYTES, tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * BN), m - lane, n0, lane,
                                  half * HW, (half + 1) * HW < BN ? (half + 1) * HW : BN);
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&tempty[buf]);  // the issuer may overwrite this accumulator now
        }
        if (!ok && lane == 0) atomicOr(g.status, DEV_E_WAIT_TIMEOUT);
    }
    tc::tc_fence_before();
    __syncthreads();
    if (wid == 2) tc::tmem_dealloc(tmem, 2 * BN);
}

template <int EPI, bool B_MN, int BN>
cudaError_t launch_nt_t(const NtMaps& maps, const NtArgs& g, int ntiles, cudaStream_t s) {
    using Cfg = NtCfg<BN>;
    return launch<k_gemm_nt_tc<EPI, B_MN, BN>>(ntiles < 148 ? ntiles : 148, Cfg::THREADS, Cfg::smem_bytes, s, maps, g);
}

// B: MN-major [K][N] (boxes of 64 x 64) or K-major [N][K].  The CTA-pair kernel (256 x 256 tiles) halves the operand traffic and takes
// every launch that gives its 74 pairs work; with fewer tiles than half of that, smaller tiles on more SMs are quicker.
template <int EPI, bool B_MN>
cudaError_t launch_nt(const void* A, size_t a_rows, const void* B, const NtArgs& g, cudaStream_t s) {
    if (g.N % 64 != 0 || g.K % 64 != 0 || g.N > NT_MAXN || g.M < 1) return cudaErrorNotSupported;
    auto tiles = [&](int bm, int bn) { return ((g.M + bm - 1) / bm) * ((g.N + bn - 1) / bn); };
    const int np = tiles(256, 256), n128 = tiles(128, 128), n64 = tiles(128, 64);
    const int bn = EPI == EPI_BASE || np > 37 ? 256 : n64 <= 148 ? 64 : 128;
    NtMaps maps;
    memset(&maps, 0, sizeof(maps));
    if (!make_tensor_map_2d(&maps.a, A, a_rows, g.K, 128, true)) return cudaErrorNotSupported;
    if (!make_tensor_map_2d(&maps.b, B, B_MN ? g.K : g.N, B_MN ? g.N : g.K, B_MN || bn == 64 ? 64 : 128, true)) return cudaErrorNotSupported;
    if (bn == 256 && g.M >= 256) return launch_nt_pair(EPI, B_MN, maps, g, s);
    if constexpr (EPI != EPI_BASE) {
        if (bn == 64) return launch_nt_t<EPI, B_MN, 64>(maps, g, n64, s);
        if (bn == 128) return launch_nt_t<EPI, B_MN, 128>(maps, g, n128, s);
    }
    return launch_nt_t<EPI, B_MN, 256>(maps, g, tiles(128, 256), s);
}

// Elements between the bf16 planes of h1 in the fp32 form: the recorded rows and the B rows of the bootstrap step.
// First activation row of step t.  Tmax = 0: h1 and h2 hold the rows of one step only (acting without a workspace).
__host__ __device__ inline size_t step_row0(const Dims& d, int t) { return d.Tmax ? (size_t)t * d.B : 0; }
__host__ __device__ inline size_t h1_plane(const Dims& d) { return ((size_t)d.B * d.Tmax + d.B) * d.H; }

// Eight consecutive hidden units of one row of h1 = relu(base + W1 row): bf16-rounded (one plane), or exact as three planes.
template <bool F32>
__device__ __forceinline__ void h1_store8(uint16_t* out, size_t plane, const float4& b0, const float4& b1, const float4& w0, const float4& w1) {
    const float x[8] = {fmaxf(b0.x + w0.x, 0.f), fmaxf(b0.y + w0.y, 0.f), fmaxf(b0.z + w0.z, 0.f), fmaxf(b0.w + w0.w, 0.f),
                        fmaxf(b1.x + w1.x, 0.f), fmaxf(b1.y + w1.y, 0.f), fmaxf(b1.z + w1.z, 0.f), fmaxf(b1.w + w1.w, 0.f)};
    if (F32) {
        uint32_t t[4][3];
#pragma unroll
        for (int q = 0; q < 4; ++q) split3(x[2 * q], x[2 * q + 1], t[q]);
#pragma unroll
        for (int p = 0; p < 3; ++p) *reinterpret_cast<uint4*>(out + p * plane) = make_uint4(t[0][p], t[1][p], t[2][p], t[3][p]);
    } else {
        uint32_t o[4], unused;
#pragma unroll
        for (int q = 0; q < 4; ++q) split2<1>(x[2 * q], x[2 * q + 1], o[q], unused);
        *reinterpret_cast<uint4*>(out) = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// h1 rows: 8 hidden units per thread.  pos[i] is the agent cell of row i (env = i mod B).
template <bool F32>
__global__ void __launch_bounds__(256) k_h1_wide(Dims d, Buffers b, const uint8_t* pos, size_t rows, size_t row0) {
    PDL_START();
    const int H = d.H, H8 = H / 8;
    const float* W1a = b.theta_c + d.oW1 + (size_t)d.C * H;  // agent plane of W1
    uint16_t* out = reinterpret_cast<uint16_t*>(b.h1) + row0 * H;
    const size_t total = rows * H8;
    for (size_t idx = (size_t)blockIdx.x * 256 + threadIdx.x; idx < total; idx += (size_t)gridDim.x * 256) {
        const size_t i = idx / H8;
        const int j8 = (int)(idx - i * H8);
        const int env = (int)(i % d.B);
        const int p = min((int)pos[i], d.C - 1);  // a position handed in from outside stays inside the plane
        const float4* bp = reinterpret_cast<const float4*>(b.base + (size_t)env * H) + 2 * j8;
        const float4* wp = reinterpret_cast<const float4*>(W1a + (size_t)p * H) + 2 * j8;
        h1_store8<F32>(out + idx * 8, h1_plane(d), bp[0], bp[1], __ldg(wp), __ldg(wp + 1));
    }
}

// Heads, sampling and env step for HW_ROWS = 32 or 8 rows per CTA (eight where 32 would leave SMs without a CTA: a step is a
// dependent launch, so its latency counts): eight warps share the rows for the head products, then warp 0
// takes one row per lane for the per-env part (its env state and wall words were requested at kernel start).
//   mode 0: step t of the rollout (row = env): saves the head outputs and the value, samples, steps the env, records.
//   mode 1: bootstrap forward after the last step: saves the value only.
//   mode 2: replay of recorded rows (row = t*B + env): saves the head outputs only.
//   mode 3: forward of the current env state under the current parameters: saves the value to vboot.
template <int H, bool F32, int HW_ROWS>
__global__ void __launch_bounds__(256, HW_ROWS >= 16 && H >= 768 ? 4 : 5) k_heads_wide(RolloutArgs a, int t, int mode, size_t rows, size_t row0) {
    PDL_START();
    constexpr int TRIPS = H / 128;   // a lane covers four consecutive hidden units per trip
    extern __shared__ __align__(16) float s_wh[];  // [H][5] as stored
    __shared__ float s_out[HW_ROWS][8];
    __shared__ uint32_t s_walls[HW_ROWS][8];
    const Dims& d = a.d;
    const Buffers& b = a.b;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const size_t i0 = (size_t)blockIdx.x * HW_ROWS;
    {   // Wh: straight 16-byte copies (the parameter block starts on a 16-byte boundary for these H)
        const float4* src = reinterpret_cast<const float4*>(b.theta_c + d.oWh);
        float4* dst = reinterpret_cast<float4*>(s_wh);
#pragma unroll
        for (int q = 0; q < (5 * H / 4 + 255) / 256; ++q)
            if (tid + 256 * q < 5 * H / 4) dst[tid + 256 * q] = __ldg(src + tid + 256 * q);
    }
    EnvLane es;
    es.pos = es.tep = es.start = es.goal = 0;
    if (mode == 0) {
        if (tid < HW_ROWS && i0 + tid < rows) {
            es.pos = b.pos[i0 + tid];
            es.tep = b.tep[i0 + tid];
            es.start = b.start[i0 + tid];
            es.goal = b.goal[i0 + tid];
        }
        for (int idx = tid; idx < HW_ROWS * d.W; idx += 256) {
            const int e = idx / d.W, wi = idx - e * d.W;
            if (i0 + e < rows) s_walls[e][wi] = b.walls[(i0 + e) * d.W + wi];
        }
    }
    const uint16_t* h2b = reinterpret_cast<const uint16_t*>(b.h2);
    // A warp walks rows wid, wid + 8, ...; WIN trips of h2 are in flight.  In CTAs of 32 rows it takes two at a time, so that a piece of
    // Wh read from shared memory serves both (B200, one row / two: bf16 H = 1024, 16384 rows 39.8 / 34.8 us, 768 32.5 / 27.4, 512, 20000
    // rows 26.6 / 22.8, 384 21.4 / 18.0; fp32 H = 1024, 12000 rows 39.4 / 34.2).  In fp32 below 768 the second row's registers cost
    // what it gains in the largest batches (H = 512, 12000 rows 24.2 / 22.4, 120000 rows 138.8 / 142.0), so those keep one.
    constexpr int RB = HW_ROWS >= 16 && (H >= 768 || !F32) ? 2 : 1, WIN = RB == 2 && F32 ? (TRIPS % 2 == 0 ? 2 : 3) : TRIPS % 4 == 0 ? 4 : 3;
    using H2x4 = typename std::conditional<F32, float4, uint2>::type;  // four consecutive units of h2: fp32, or bf16
    static_assert(TRIPS % WIN == 0, "a trip keeps its slot from one pass to the next");
    H2x4 v[WIN][RB];
    auto load_trip = [&](int r, int q, H2x4 (&dst)[RB]) {
#pragma unroll
        for (int k = 0; k < RB; ++k) {
            const size_t i = i0 + r + 8 * k, off = (row0 + (i < rows ? i : 0)) * H;
            const H2x4* hp = F32 ? reinterpret_cast<const H2x4*>(b.h2 + off) : reinterpret_cast<const H2x4*>(h2b + off);
            dst[k] = i < rows ? __ldg(hp + lane + 32 * q) : H2x4{};
        }
    };
#pragma unroll
    for (int q = 0; q < WIN; ++q) load_trip(wid, q, v[q]);
    __syncthreads();
#pragma unroll 1
    for (int r = wid; r < HW_ROWS; r += 8 * RB) {
        float acc[RB][5];
#pragma unroll
        for (int k = 0; k < RB; ++k)
#pragma unroll
            for (int c = 0; c < 5; ++c) acc[k][c] = 0.f;
#pragma unroll
        for (int q = 0; q < TRIPS; ++q) {
            // this lane's four units are 20 consecutive floats of Wh (80-byte lane stride: conflict-free 16-byte reads)
            const float4* wp = reinterpret_cast<const float4*>(s_wh + 20 * (lane + 32 * q));
            float w[20];
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                const float4 f = wp[j];
                w[4 * j] = f.x; w[4 * j + 1] = f.y; w[4 * j + 2] = f.z; w[4 * j + 3] = f.w;
            }
#pragma unroll
            for (int k = 0; k < RB; ++k) {
                const H2x4 y = v[q % WIN][k];
                float x[4];
                if constexpr (F32) {
                    x[0] = y.x; x[1] = y.y; x[2] = y.z; x[3] = y.w;
                } else {
                    x[0] = __uint_as_float(y.x << 16);
                    x[1] = __uint_as_float(y.x & 0xFFFF0000u);
                    x[2] = __uint_as_float(y.y << 16);
                    x[3] = __uint_as_float(y.y & 0xFFFF0000u);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int c = 0; c < 5; ++c) acc[k][c] = fmaf(x[u], w[5 * u + c], acc[k][c]);
            }
            if (q + WIN < TRIPS) load_trip(r, q + WIN, v[q % WIN]);
            else if (r + 8 * RB < HW_ROWS) load_trip(r + 8 * RB, (q + WIN) % TRIPS, v[q % WIN]);  // (the next rows' first trips)
        }
        // sums over the lanes; two rows: the first round of the tree hands each half of the warp one of them
        float o5[5];
        const bool up = lane & 16;
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            if constexpr (RB == 2) o5[c] = (up ? acc[1][c] : acc[0][c]) + __shfl_xor_sync(0xFFFFFFFFu, up ? acc[0][c] : acc[1][c], 16);
            else o5[c] = acc[0][c] + __shfl_xor_sync(0xFFFFFFFFu, acc[0][c], 16);
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) o5[c] += __shfl_xor_sync(0xFFFFFFFFu, o5[c], off);
        }
        if ((lane & 15) == 0 && (RB == 2 || lane == 0)) {
#pragma unroll
            for (int c = 0; c < 5; ++c) s_out[r + (RB == 2 && up ? 8 : 0)][c] = o5[c] + b.theta_c[d.obh + c];
        }
    }
    __syncthreads();
    __shared__ int s_pos[HW_ROWS];
    if (tid < 32) {  // (the whole warp: the counters below are folded over its lanes)
    const size_t i = i0 + tid;
    const bool valid = tid < HW_ROWS && i < rows;
    unsigned long long n_ep = 0, n_goal = 0, n_steps = 0;
    int bad = 0;
    if (valid) {
        const float o0 = s_out[tid][0], o1 = s_out[tid][1], o2 = s_out[tid][2], o3 = s_out[tid][3], v4 = s_out[tid][4];
        if (mode == 1) {
            b.tval[(size_t)a.T * d.B + i] = v4;
        } else if (mode == 3) {
            b.vboot[i] = v4;
        } else {
            const size_t row = mode == 0 ? (size_t)t * d.B + i : i;
            if (b.out5) {
                float4* o = reinterpret_cast<float4*>(b.out5 + row * 8);
                o[0] = make_float4(o0, o1, o2, o3);
                o[1] = make_float4(v4, 0.f, 0.f, 0.f);
            }
            if (mode == 0) {
                b.tval[row] = v4;
                const int env = (int)i;
                es.n_episodes = es.n_goals = es.n_epsteps = 0;
                es.bad = 0;
                check_env_state(es, d.C, s_walls[tid]);
                act_and_step(es, a, env, t, o0, o1, o2, o3, s_walls[tid]);
                b.pos[env] = (uint8_t)es.pos;
                b.tep[env] = (uint8_t)es.tep;
                s_pos[tid] = es.pos;
                n_ep = es.n_episodes; n_goal = es.n_goals; n_steps = es.n_epsteps; bad = es.bad;
            }
        }
    }
    if (mode == 0) {
    // fold the warp's counters and add them with integer atomics (order-free totals)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        n_ep += __shfl_xor_sync(0xFFFFFFFFu, n_ep, off);
        n_goal += __shfl_xor_sync(0xFFFFFFFFu, n_goal, off);
        n_steps += __shfl_xor_sync(0xFFFFFFFFu, n_steps, off);
        bad |= __shfl_xor_sync(0xFFFFFFFFu, bad, off);
    }
    if (lane == 0) {
        if (n_ep) atomicAdd((unsigned long long*)&b.stats->episodes, n_ep);
        if (n_goal) atomicAdd((unsigned long long*)&b.stats->goals, n_goal);
        if (n_steps) atomicAdd((unsigned long long*)&b.stats->episode_steps, n_steps);
        if (blockIdx.x == 0 && tid == 0) atomicAdd((unsigned long long*)&b.stats->frames, (unsigned long long)d.B);
        if (bad) atomicOr(b.status, bad);
    }
    }
    }
    if (mode != 0) return;
    // ---- layer 1 of the NEXT step for this CTA's envs, from the positions just produced (rows (t+1)*B + env):
    // 256 / HW_ROWS threads per env, 16-byte chunks interleaved so that a row's lanes read and write contiguous memory
    __syncthreads();
    {
        constexpr int TPR = 256 / HW_ROWS;
        const int rl = tid / TPR, q = tid % TPR;
        const size_t env = i0 + rl;
        if (env < rows) {
            const float4* bp = reinterpret_cast<const float4*>(b.base + env * H);
            const float4* wp = reinterpret_cast<const float4*>(b.theta_c + d.oW1 + ((size_t)d.C + s_pos[rl]) * H);
            uint16_t* out = reinterpret_cast<uint16_t*>(b.h1) + (step_row0(d, t + 1) + env) * H;
#pragma unroll 4
            for (int ch = q; ch < H / 8; ch += TPR)
                h1_store8<F32>(out + 8 * ch, h1_plane(d), bp[2 * ch], bp[2 * ch + 1], __ldg(wp + 2 * ch), __ldg(wp + 2 * ch + 1));
        }
    }
}

// S[env][j] = sum over t of dh1[t*B + env][j], kept as two bf16 terms (hi and lo planes) for the K = B GEMMs of dW1.
__global__ void __launch_bounds__(256) k_sum_t_wide(Dims d, Buffers b, int T) {
    PDL_START();
    const int H8 = d.H / 8;
    const size_t total = (size_t)d.B * H8;
    const size_t idx = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (idx >= total) return;
    const uint4* src = reinterpret_cast<const uint4*>(b.dh1) + idx;
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int t0 = 0; t0 < T; t0 += 8) {  // eight loads in flight
        uint4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = t0 + q < T ? __ldg(src + (size_t)(t0 + q) * total) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const uint32_t w[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                s[2 * e] += __uint_as_float(w[e] << 16);
                s[2 * e + 1] += __uint_as_float(w[e] & 0xFFFF0000u);
            }
        }
    }
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        __nv_bfloat16 h0, l0, h1, l1;
        split_bf16(s[2 * e], h0, l0);
        split_bf16(s[2 * e + 1], h1, l1);
        hi[e] = pack_bf16(h0, h1);
        lo[e] = pack_bf16(l0, l1);
    }
    uint4* S_hi = reinterpret_cast<uint4*>(b.S);
    uint4* S_lo = S_hi + total;
    S_hi[idx] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    S_lo[idx] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
}

// W2 as row-major bf16 planes: one (the values are bf16 already in the bf16 workload) or the three terms of fp32 weights.
template <bool F32>
__global__ void __launch_bounds__(256) k_pack_w2_wide(Dims d, Buffers b) {
    PDL_START();
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x, n = (size_t)d.H * d.H;
    if (2 * i >= n) return;
    const float2 w = reinterpret_cast<const float2*>(b.theta_c + d.oW2)[i];
    uint32_t t[3];
    split3(w.x, w.y, t);
    for (int p = 0; p < (F32 ? 3 : 1); ++p) reinterpret_cast<uint32_t*>(b.w2p_hi + p * n)[i] = t[p];
}

// Operands of the base GEMM: X[env][c] = 1 where cell c of the env is a wall (bf16), and the wall plane of W1 as bf16 planes
// (one where the weights are bf16 values, else three terms).  Columns / rows from C up to Cp, a multiple of 64, are zero.
template <bool F32>
__global__ void __launch_bounds__(256) k_expand_walls(Dims d, Buffers b, uint16_t* X, uint16_t* W1w, int Cp) {
    PDL_START();
    const size_t nx = (size_t)d.B * (Cp / 8), nw = (size_t)Cp * d.H / 2, real = (size_t)d.C * d.H / 2;
    for (size_t idx = (size_t)blockIdx.x * 256 + threadIdx.x; idx < nx + nw; idx += (size_t)gridDim.x * 256) {
        if (idx < nx) {
            const size_t e = idx / (Cp / 8);
            const int c8 = (int)(idx - e * (Cp / 8)), left = d.C - 8 * c8;  // cells of the board in this chunk
            uint32_t bits = left > 0 ? (b.walls[e * d.W + (c8 >> 2)] >> ((c8 & 3) * 8)) & 0xFFu : 0u;
            if (left < 8 && left > 0) bits &= (1u << left) - 1u;
            uint32_t o[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) o[q] = ((bits >> (2 * q)) & 1u ? 0x3F80u : 0u) | ((bits >> (2 * q + 1)) & 1u ? 0x3F800000u : 0u);
            for (int p = 0; p < (F32 ? 3 : 1); ++p) reinterpret_cast<uint4*>(X)[(e * (F32 ? 3 : 1) + p) * (Cp / 8) + c8] = make_uint4(o[0], o[1], o[2], o[3]);
        } else {
            const size_t i = idx - nx;
            const float2 w = i < real ? reinterpret_cast<const float2*>(b.theta_c + d.oW1)[i] : make_float2(0.f, 0.f);
            uint32_t t[3];
            split3(w.x, w.y, t);
            for (int p = 0; p < (F32 ? 3 : 1); ++p) reinterpret_cast<uint32_t*>(W1w)[(F32 ? 2 - p : 0) * nw + i] = t[p];
        }
    }
}

#define CKW(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) return e_; } while (0)

template <int H, bool F32>
cudaError_t heads_wide_t(const RolloutArgs& a, int t, int mode, size_t rows, size_t row0, cudaStream_t s) {
    const size_t smem = (size_t)5 * H * sizeof(float);
    if (rows < 148 * 2 * 32) launch<k_heads_wide<H, F32, 8>>((unsigned)((rows + 7) / 8), 256, smem, s, a, t, mode, rows, row0);
    else launch<k_heads_wide<H, F32, 32>>((unsigned)((rows + 31) / 32), 256, smem, s, a, t, mode, rows, row0);
    return cudaGetLastError();
}
cudaError_t heads_wide(const RolloutArgs& a, bool f32, int t, int mode, size_t rows, size_t row0, cudaStream_t s) {
    switch (a.d.H) {
        case 384: return f32 ? heads_wide_t<384, true>(a, t, mode, rows, row0, s) : heads_wide_t<384, false>(a, t, mode, rows, row0, s);
        case 512: return f32 ? heads_wide_t<512, true>(a, t, mode, rows, row0, s) : heads_wide_t<512, false>(a, t, mode, rows, row0, s);
        case 768: return f32 ? heads_wide_t<768, true>(a, t, mode, rows, row0, s) : heads_wide_t<768, false>(a, t, mode, rows, row0, s);
        case 1024: return f32 ? heads_wide_t<1024, true>(a, t, mode, rows, row0, s) : heads_wide_t<1024, false>(a, t, mode, rows, row0, s);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace

// fp32 workloads compute with the master parameters themselves.
static bool is_f32(const Buffers& b) { return b.theta_c == b.theta; }

cudaError_t launch_pack_w2_wide(const Dims& d, const Buffers& b, const Ctx& c) {
    Scope sc(c, K_PACK_W2);
    const unsigned nb = (unsigned)(((size_t)d.H * d.H / 2 + 255) / 256);
    if (is_f32(b)) launch<k_pack_w2_wide<true>>(nb, 256, 0, c.s, d, b);
    else launch<k_pack_w2_wide<false>>(nb, 256, 0, c.s, d, b);
    return cudaGetLastError();
}

size_t wide_scratch_bytes(const Dims& d) {
    const size_t Cp = (size_t)(d.C + 63) / 64 * 64;
    return 3 * ((size_t)d.B * Cp + Cp * d.H) * 2;
}
size_t wide_h1_rows(const Dims& d) { return (size_t)d.B * d.Tmax + d.B; }

// base = b1 + walls x W1[wall plane] + W1[goal row] as one GEMM (K = C cells, padded to a multiple of 64): the operand X is
// exact, W1 has one (bf16 workload) or three exact bf16 terms, the accumulation is fp32.  Three terms are one GEMM of three
// times the K: the smallest term's rows first, X repeated.  cudaErrorNotSupported for the
// buffers of other paths and for small batches, where the gather kernel's single launch is quicker (B H = 2^20: 11 us each): up to the
// sizes that act without a workspace, which has no room for the operands, so that both give the same bits.
// Uses the dh1 buffer (the one h2 is in) as scratch for the operands: base is computed ahead of the forward passes that fill it.
cudaError_t launch_env_base_wide(const Dims& d, const Buffers& b, const Ctx& c) {
    if (!b.w2p_hi || !wide_supported(d.H) || (size_t)d.B * d.H <= ANAKIN_NOALLOC_MAX_BH) return cudaErrorNotSupported;
    const bool f32 = is_f32(b);
    const int Cp = (d.C + 63) / 64 * 64, terms = f32 ? 3 : 1;
    uint16_t* X = reinterpret_cast<uint16_t*>(b.dh1);
    uint16_t* W1w = X + (size_t)d.B * Cp * terms;
    {
        Scope sc(c, K_ENV_BASE);
        if (f32) launch<k_expand_walls<true>>(148 * 8, 256, 0, c.s, d, b, X, W1w, Cp);
        else launch<k_expand_walls<false>>(148 * 8, 256, 0, c.s, d, b, X, W1w, Cp);
        CKW(cudaGetLastError());
    }
    Scope sc(c, K_ENV_BASE);
    NtArgs g;
    memset(&g, 0, sizeof(g));
    g.M = d.B; g.N = d.H; g.K = Cp * terms; g.row0 = 0;
    g.bias = b.theta_c + d.ob1;
    g.outf = b.base;
    g.addrows = b.theta_c + d.oW1;
    g.addidx = b.goal;
    g.addrow0 = 2 * d.C;
    g.addmax = d.C - 1;
    g.status = b.status;
    return launch_nt<EPI_BASE, true>(X, d.B, W1w, g, c.s);
}

template <bool F32>
static cudaError_t rollout_wide_t(const RolloutArgs& a, const Ctx& c) {
    const Dims& d = a.d;
    const Buffers& b = a.b;
    const int H = d.H, B = d.B;
    const size_t rows = wide_h1_rows(d);
    auto fwd = [&](size_t n, size_t row0) {  // h2 of n rows
        if constexpr (F32) {
            X3Args g;
            memset(&g, 0, sizeof(g));
            g.M = (int)n; g.N = g.K = H; g.row0 = (int)row0;
            g.arows = (int)rows; g.brows = H;
            g.out = b.h2;
            g.bias = b.theta_c + d.ob2;
            g.status = b.status;
            return launch_x3_nt(EPI_FWD, b.h1, 3 * rows, b.w2p_hi, g, c.s);
        } else {
            NtArgs g;
            memset(&g, 0, sizeof(g));
            g.M = (int)n; g.N = g.K = H; g.row0 = (int)row0;
            g.out = reinterpret_cast<uint16_t*>(b.h2);
            g.bias = b.theta_c + d.ob2;
            g.status = b.status;
            return launch_nt<EPI_FWD, true>(b.h1, rows, b.w2p_hi, g, c.s);
        }
    };
    auto h1_rows = [&](const uint8_t* pos, size_t n, size_t row0) {
        return launch<k_h1_wide<F32>>((unsigned)((n * (H / 8) + 255) / 256), 256, 0, c.s, d, b, pos, n, row0);
    };
    // forward of n rows from row0: (h1,) h2, heads in the given mode
    auto replay = [&](const uint8_t* pos, size_t n, size_t row0, int mode) {
        {
            Scope sc(c, K_REPLAY);
            CKW(h1_rows(pos, n, row0));
        }
        {
            Scope sc(c, K_REPLAY);
            CKW(fwd(n, row0));
        }
        Scope sc(c, K_REPLAY);
        return heads_wide(a, F32, 0, mode, n, row0, c.s);
    };
    if (a.replay) {
        const size_t R = (size_t)B * a.T;
        CKW(replay(b.tpos, R, 0, 2));
        if (a.replay == 2) CKW(replay(b.pos, B, R, 3));  // and the env state as it stands, in the B rows after the recorded ones
        return cudaSuccess;
    }
    for (int t = 0; t <= a.T; ++t) {
        const size_t row0 = step_row0(d, t);
        if (t == 0) {  // later steps: the heads kernel of step t-1 writes the h1 rows of step t
            Scope sc(c, K_H1);
            CKW(h1_rows(b.pos, B, row0));
        }
        {
            Scope sc(c, K_FWD2);
            CKW(fwd(B, row0));
        }
        {
            Scope sc(c, K_ROLLOUT);
            CKW(heads_wide(a, F32, t, t == a.T ? 1 : 0, B, row0, c.s));
        }
    }
    return cudaSuccess;
}
// T+1 forward passes (or, in replay mode, one pass over the recorded rows).
cudaError_t launch_rollout_wide(const RolloutArgs& a, const Ctx& c) { return is_f32(a.b) ? rollout_wide_t<true>(a, c) : rollout_wide_t<false>(a, c); }

// dh1 = (dh2 W2^T) gated by h1 > 0 over all R rows: fp32 (the agent-plane kernel reads it and forms S), or one bf16 plane and S.
template <bool F32>
static cudaError_t dh1_wide_t(const LearnArgs& a, const Ctx& c) {
    const Dims& d = a.d;
    const Buffers& b = a.b;
    const int H = d.H;
    const size_t R = (size_t)d.B * a.T, plane = (size_t)d.B * d.Tmax;  // (dh2 planes)
    if constexpr (F32) {
        Scope sc(c, K_DH1);
        X3Args g;
        memset(&g, 0, sizeof(g));
        g.M = (int)R; g.N = g.K = H;
        g.arows = (int)plane; g.brows = H;
        g.out = b.dh1;
        g.gate = reinterpret_cast<const uint16_t*>(b.h1);
        g.status = b.status;
        return launch_x3_nt(EPI_GATE, b.dh2, 3 * plane, b.w2p_hi, g, c.s);
    } else {
        NtArgs g;
        memset(&g, 0, sizeof(g));
        g.M = (int)R; g.N = g.K = H;
        g.out = reinterpret_cast<uint16_t*>(b.dh1);
        g.gate = reinterpret_cast<const uint16_t*>(b.h1);
        g.status = b.status;
        {
            Scope sc(c, K_DH1);
            CKW((launch_nt<EPI_GATE, false>(b.dh2, R, b.w2p_hi, g, c.s)));
        }
        Scope sc(c, K_SUM_OVER_T);
        return launch<k_sum_t_wide>((unsigned)(((size_t)d.B * (H / 8) + 255) / 256), 256, 0, c.s, d, b, a.T);
    }
}
cudaError_t launch_dh1_wide(const LearnArgs& a, const Ctx& c) { return is_f32(a.b) ? dh1_wide_t<true>(a, c) : dh1_wide_t<false>(a, c); }

}  // namespace anakin
