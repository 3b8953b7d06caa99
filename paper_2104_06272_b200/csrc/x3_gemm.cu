// fp32 GEMMs of the wide hidden layers on the 5th-generation tensor cores:  C[m][n] = sum_k A[m][k] Bop[k][n]  with fp32 operands
// stored as three exact bf16 planes each (x = t0 + t1 + t2), six bf16 products per fp32 product, fp32 results.  The layer-2
// products of the Anakin minimal unit (Podracer paper, Section 3.1; Figure 2, top): h2 = relu(h1 W2 + b2) and
// dh1 = (dh2 W2^T) gated by h1 > 0.
//
// One pipeline stage holds all three planes of both operands for a 64-wide K chunk, so a byte staged by TMA feeds two MMAs instead
// of one.  The tensor core's fp32 accumulation rounds toward zero, once per MMA; a chunk is therefore an accumulator group of its
// own: its products go in smallest first (24 MMAs, of which only the last four round at full magnitude), the accumulator is read
// out, and the epilogue warps add the chunks with round-to-nearest in registers while the next chunk runs into the other
// accumulator.  The value error at H = 512 is 1.5e-7 relative, against 2.7e-7 of an fp32 FMA chain.
//
// PAIR: a cluster of two CTAs owns a 256 x 256 tile (cta_group::2), 96 KB per stage and CTA for 24 x 128 clocks of MMAs; otherwise
// one CTA owns 128 x BN (BN = 128, 64) for launches with few tiles.
//   warp 0 (one lane)        TMA producer (PAIR: of its CTA's halves, credited to the leader's barrier)
//   warp 1                   MMA issuer (PAIR: the leader's): the whole warp walks the loop, an elected lane issues
//   warps 2-9                accumulate the groups, then bias / ReLU / gate and store through a staging buffer, 64-byte row segments
// Every wait is bounded; a timeout raises DEV_E_WAIT_TIMEOUT and the CTA unwinds (tensor memory freed).
#include <cstring>

#include "wide_gemm.cuh"

namespace anakin {
namespace widegemm {

namespace {

template <bool PAIR, int BN>
struct X3Cfg {
    static constexpr int BM = 128, PM = PAIR ? 256 : 128, BNC = PAIR ? BN / 2 : BN, KC = 64, THREADS = 320, EPI_WARPS = 8;
    static constexpr int A_PLANE = BM * KC * 2, B_PLANE = BNC * KC * 2, STAGE = 3 * (A_PLANE + B_PLANE);
    static constexpr int STAGES = 2;
    static constexpr int MAXN = 1024, STG = 2048;  // bias floats; staging bytes per epilogue warp: 32 rows x 16 columns
    static constexpr size_t smem_bytes = (size_t)STAGES * STAGE + 1024 /*alignment slack*/ + 256 /*barriers, tmem slot*/ + MAXN * 4 + EPI_WARPS * STG;
    static_assert(smem_bytes <= 232448, "shared memory");
};

template <int EPI, bool B_MN, bool PAIR, int BN>
__device__ __forceinline__ void x3_body(const NtMaps& maps, const X3Args& g) {
    using Cfg = X3Cfg<PAIR, BN>;
    constexpr int BM = Cfg::BM, PM = Cfg::PM, BNC = Cfg::BNC, KC = Cfg::KC, STAGES = Cfg::STAGES, COLS = BN / 2;
    constexpr int LDC = COLS == 128 ? 16 : 32;  // accumulator columns per load (128 running sums leave few registers)
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);  // (the same offset in both CTAs of a pair)
    uint64_t* bars = (uint64_t*)(base + STAGES * Cfg::STAGE);
    uint64_t* full = bars;                // [STAGES] (PAIR: the leader's copy collects both CTAs' loads)
    uint64_t* empty = bars + STAGES;      // [STAGES]
    uint64_t* tfull = bars + 2 * STAGES;  // [2] accumulator written
    uint64_t* tempty = tfull + 2;         // [2] accumulator drained (PAIR: the leader's copy counts the warps of both CTAs)
    uint32_t* tmem_slot = (uint32_t*)(tempty + 2);
    float* s_bias = (float*)(base + STAGES * Cfg::STAGE + 256);
    unsigned char* s_stage = (unsigned char*)(s_bias + Cfg::MAXN);
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const int rank = PAIR ? (int)tc::cluster_ctarank() : 0;
    const bool leader = rank == 0;
    const int unit = PAIR ? blockIdx.x >> 1 : blockIdx.x, units = PAIR ? gridDim.x >> 1 : gridDim.x;
    const int nt = (g.N + BN - 1) / BN, mt = (g.M + PM - 1) / PM, ntiles = mt * nt, nkc = (g.K + KC - 1) / KC;  // (columns of A past K read as zeros)

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) { tc::mbar_init(&full[s], 1); tc::mbar_init(&empty[s], 1); }
        for (int i = 0; i < 2; ++i) { tc::mbar_init(&tfull[i], 1); tc::mbar_init(&tempty[i], (PAIR ? 2 : 1) * Cfg::EPI_WARPS); }
        tc::mbar_fence_init();
    }
    if (wid == 2) {
        if constexpr (PAIR) tc::tmem_alloc_pair(tmem_slot, 2 * BN);
        else tc::tmem_alloc(tmem_slot, 2 * BN);
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if constexpr (PAIR) tc::cluster_sync_all();  // both CTAs' barriers exist before either signals the other
    const uint32_t tmem = *tmem_slot;
    pdl_wait();  // (the set-up above runs under the predecessor's tail)
    if (EPI == EPI_FWD) {
        for (int i = tid; i < g.N; i += Cfg::THREADS) s_bias[i] = g.bias[i];
        __syncthreads();
    }
    bool ok = true;

    if (wid == 0) {
        if (lane == 0) {  // ---- TMA producer
            int c = 0;
            for (int tile = unit; tile < ntiles && ok; tile += units) {
                const int m0 = g.row0 + (tile / nt) * PM + BM * rank, n0 = (tile % nt) * BN + BNC * rank;
                for (int kc = 0; kc < nkc; ++kc, ++c) {
                    const int s = c % STAGES;
                    if (c >= STAGES) ok = tc::mbar_wait(&empty[s], ((c / STAGES) - 1) & 1);
                    if (!ok) break;
                    unsigned char* sa = base + s * Cfg::STAGE;
                    unsigned char* sb = sa + 3 * Cfg::A_PLANE;
                    if (leader) tc::mbar_expect_tx(&full[s], (PAIR ? 2 : 1) * Cfg::STAGE);
                    const uint32_t bar = PAIR ? tc::mapa(tc::smem_u32(&full[s]), 0) : 0u;
                    auto load = [&](void* dst, const CUtensorMap* m, int x, int y) {
                        if constexpr (PAIR) tc::tma_load_2d_pair(dst, m, bar, x, y);
                        else tc::tma_load_2d(dst, m, &full[s], x, y);
                    };
                    // rows past M belong to later rows or planes of the buffer or are zero-filled; the epilogue drops them
#pragma unroll
                    for (int p = 0; p < 3; ++p) {
                        load(sa + p * Cfg::A_PLANE, &maps.a, kc * KC, m0 + p * g.arows);
#pragma unroll
                        for (int bx = 0; bx < BNC / 64; ++bx) {
                            if (B_MN) load(sb + p * Cfg::B_PLANE + bx * 8192, &maps.b, n0 + 64 * bx, p * g.brows + kc * KC);
                            else load(sb + p * Cfg::B_PLANE + bx * 8192, &maps.b, kc * KC, p * g.brows + n0 + 64 * bx);
                        }
                    }
                }
            }
            if (!ok) atomicOr(g.status, DEV_E_WAIT_TIMEOUT);
        }
    } else if (wid == 1) {
        if (leader) {  // ---- MMA issuer: the whole warp walks the loop, one elected lane issues
            const uint32_t idesc = tc::umma_idesc<2>(PM, BN, false, B_MN);
            int c = 0;
            for (int tile = unit; tile < ntiles && ok; tile += units) {
                for (int kc = 0; kc < nkc; ++kc, ++c) {
                    const int s = c % STAGES, buf = c & 1;
                    if (c >= 2) ok = PAIR ? tc::mbar_wait_cluster(&tempty[buf], ((c >> 1) - 1) & 1) : tc::mbar_wait(&tempty[buf], ((c >> 1) - 1) & 1);
                    if (ok) ok = tc::mbar_wait(&full[s], (c / STAGES) & 1);
                    ok = tc::warp_all(ok);
                    if (!ok) break;
                    tc::tc_fence_after();
                    const uint32_t acc = tmem + (uint32_t)(buf * BN);
                    unsigned char* sa = base + s * Cfg::STAGE;
                    unsigned char* sb = sa + 3 * Cfg::A_PLANE;
                    // K-major: 16 k = 32 bytes along the swizzled 128-byte rows; MN-major: 16 k rows = 2048 bytes (the start address
                    // is the descriptor's low field, in 16-byte units)
                    const uint64_t a0 = tc::umma_desc(sa, 16, 1024), b0 = B_MN ? tc::umma_desc(sb, 8192, 1024) : tc::umma_desc(sb, 16, 1024);
                    if (tc::elect_one()) {
#pragma unroll
                        for (int i = 0; i < tc::X3_PAIRS; ++i) {
#pragma unroll
                            for (int k16 = 0; k16 < KC / 16; ++k16) {
                                const uint64_t ad = a0 + (uint64_t)(tc::x3_a(i) * (Cfg::A_PLANE >> 4) + k16 * 2);
                                const uint64_t bd = b0 + (uint64_t)(tc::x3_b(i) * (Cfg::B_PLANE >> 4) + k16 * (B_MN ? 128 : 2));
                                if constexpr (PAIR) tc::umma_pair(acc, ad, bd, idesc, (i > 0 || k16 > 0) ? 1u : 0u);
                                else tc::umma(acc, ad, bd, idesc, (i > 0 || k16 > 0) ? 1u : 0u);
                            }
                        }
                        if constexpr (PAIR) {
                            tc::umma_commit_pair(&empty[s], 3);
                            tc::umma_commit_pair(&tfull[buf], 3);
                        } else {
                            tc::umma_commit(&empty[s]);
                            tc::umma_commit(&tfull[buf]);
                        }
                    }
                    __syncwarp();
                }
            }
            if (!ok && lane == 0) atomicOr(g.status, DEV_E_WAIT_TIMEOUT);
        }
    } else {
        // ---- epilogue warps: accumulator lanes 32*(wid%4)..+31 = output rows, column half (wid-2)/4
        const int q = wid & 3, half = (wid - 2) >> 2, crow = lane >> 2, cch = lane & 3;
        unsigned char* stage = s_stage + (wid - 2) * Cfg::STG;
        int c = 0;
#pragma unroll 1
        for (int tile = unit; tile < ntiles && ok; tile += units) {
            const int mb = (tile / nt) * PM + BM * rank + 32 * q, n0 = (tile % nt) * BN + half * COLS;
            float sum[COLS];
#pragma unroll
            for (int j = 0; j < COLS; ++j) sum[j] = 0.f;
#pragma unroll 1
            for (int kc = 0; kc < nkc; ++kc, ++c) {
                const int buf = c & 1;
                ok = tc::mbar_wait(&tfull[buf], (c >> 1) & 1);
                if (!ok) break;
                tc::tc_fence_after();
                const uint32_t t = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * BN + half * COLS);
#pragma unroll
                for (int c0 = 0; c0 < COLS; c0 += LDC) {
                    uint32_t r[LDC];
                    if constexpr (LDC == 16) tc::tmem_ld16_nowait(t + (uint32_t)c0, r);
                    else tc::tmem_ld32_nowait(t + (uint32_t)c0, r);
                    tc::tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < LDC; ++j) sum[c0 + j] += __uint_as_float(r[j]);
                }
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) {  // the issuer may overwrite this accumulator now
                    if constexpr (PAIR) tc::mbar_arrive_remote_cta_release(tc::mapa(tc::smem_u32(&tempty[buf]), 0));
                    else tc::mbar_arrive(&tempty[buf]);
                }
            }
            if (!ok) break;
            // 16 columns at a time through the staging buffer (lane = row in, four lanes per row out; chunks XOR-swizzled)
            const int left = g.M - mb - crow;  // rows of this lane's out phase: crow, crow + 8, ... below M
            const size_t o0 = ((size_t)g.row0 + mb + crow) * g.N + n0 + 4 * cch;
            const float* src = reinterpret_cast<const float*>(stage + crow * 64 + ((cch ^ ((crow >> 1) & 3)) << 4));  // (8 rows on: the same swizzle)
            uint2 gt[4];  // gates of the next 16 columns: requested one round ahead
            auto load_gates = [&](int c0) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    gt[i] = 8 * i < left && n0 + c0 < g.N ? __ldg(reinterpret_cast<const uint2*>(g.gate + o0 + (size_t)(8 * i) * g.N + c0)) : make_uint2(0u, 0u);
            };
            if (EPI == EPI_GATE) load_gates(0);
#pragma unroll
            for (int c0 = 0; c0 < COLS; c0 += 16) {
                if (n0 + c0 < g.N) {  // (the matrix's width is a multiple of 32)
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch)
                        *reinterpret_cast<float4*>(stage + lane * 64 + ((ch ^ ((lane >> 1) & 3)) << 4)) =
                            make_float4(sum[c0 + 4 * ch], sum[c0 + 4 * ch + 1], sum[c0 + 4 * ch + 2], sum[c0 + 4 * ch + 3]);
                    __syncwarp();
                    uint32_t on = 0u;  // four gate bits per row: the first term of an activation is zero exactly where the activation is
                    if (EPI == EPI_GATE) {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            on |= (((gt[i].x & 0x00007FFFu) ? 1u : 0u) | ((gt[i].x & 0x7FFF0000u) ? 2u : 0u) | ((gt[i].y & 0x00007FFFu) ? 4u : 0u) |
                                   ((gt[i].y & 0x7FFF0000u) ? 8u : 0u)) << (4 * i);
                        if (c0 + 16 < COLS) load_gates(c0 + 16);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (8 * i < left) {
                            float4 v = *reinterpret_cast<const float4*>(src + i * 128);
                            if (EPI == EPI_FWD) {
                                const float4 bs = *reinterpret_cast<const float4*>(s_bias + n0 + c0 + 4 * cch);
                                v = make_float4(fmaxf(v.x + bs.x, 0.f), fmaxf(v.y + bs.y, 0.f), fmaxf(v.z + bs.z, 0.f), fmaxf(v.w + bs.w, 0.f));
                            } else {
                                v.x = (on >> (4 * i)) & 1u ? v.x : 0.f;
                                v.y = (on >> (4 * i)) & 2u ? v.y : 0.f;
                                v.z = (on >> (4 * i)) & 4u ? v.z : 0.f;
                                v.w = (on >> (4 * i)) & 8u ? v.w : 0.f;
                            }
                            *reinterpret_cast<float4*>(g.out + o0 + (size_t)(8 * i) * g.N + c0) = v;
                        }
                    }
                    __syncwarp();
                }
            }
        }
        if (!ok && lane == 0) atomicOr(g.status, DEV_E_WAIT_TIMEOUT);
    }
    // (a pair: neither CTA leaves or frees tensor memory while the other may still signal it or run MMAs that touch it)
    tc::tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) tc::cluster_sync_all();
    if (wid == 2) {
        if constexpr (PAIR) tc::tmem_dealloc_pair(tmem, 2 * BN);
        else tc::tmem_dealloc(tmem, 2 * BN);
    }
}

template <int EPI, bool B_MN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(320, 1) k_x3_pair(const __grid_constant__ NtMaps maps, X3Args g) {
    x3_body<EPI, B_MN, true, 256>(maps, g);
}
template <int EPI, bool B_MN, int BN>
__global__ void __launch_bounds__(320, 1) k_x3_one(const __grid_constant__ NtMaps maps, X3Args g) {
    x3_body<EPI, B_MN, false, BN>(maps, g);
}

template <int EPI, bool B_MN>
cudaError_t launch_x3_t(const NtMaps& maps, const X3Args& g, int bn, int tiles, cudaStream_t s) {
    if (bn == 256) return launch<k_x3_pair<EPI, B_MN>>(2 * (tiles < 74 ? tiles : 74), 320, X3Cfg<true, 256>::smem_bytes, s, maps, g);
    if (bn == 128) return launch<k_x3_one<EPI, B_MN, 128>>(tiles < 148 ? tiles : 148, 320, X3Cfg<false, 128>::smem_bytes, s, maps, g);
    return launch<k_x3_one<EPI, B_MN, 64>>(tiles < 148 ? tiles : 148, 320, X3Cfg<false, 64>::smem_bytes, s, maps, g);
}

}  // namespace

// Tile rule: no tile more than twice as wide as the matrix; pairs (256 x 256) while more than half of the 74 pairs get a tile; below that 128 x 128 tiles, or 128 x 64 where even
// those fit one wave (an idle SM costs more than a narrow MMA).
cudaError_t launch_x3_nt(int epi, const void* a, size_t a_rows_total, const void* b, const X3Args& g, cudaStream_t s) {
    if (g.N % 32 != 0 || g.K % 32 != 0 || g.N > X3Cfg<true, 256>::MAXN || g.M < 1) return cudaErrorNotSupported;
    auto tiles = [&](int bm, int bn) { return ((g.M + bm - 1) / bm) * ((g.N + bn - 1) / bn); };
    const int np = tiles(256, 256), n128 = tiles(128, 128), n64 = tiles(128, 64);
    const int bn = g.N <= 64 ? 64 : np > 37 && g.N > 128 ? 256 : n64 <= 148 ? 64 : 128, n = bn == 256 ? np : bn == 128 ? n128 : n64;
    const bool b_mn = epi == EPI_FWD;  // W2 as stored: rows = k for h1 W2, rows = n for dh2 W2^T
    NtMaps maps;
    memset(&maps, 0, sizeof(maps));
    if (!make_tensor_map_2d(&maps.a, a, a_rows_total, g.K, 128, true)) return cudaErrorNotSupported;
    if (!make_tensor_map_2d(&maps.b, b, (size_t)3 * g.brows, b_mn ? g.N : g.K, 64, true)) return cudaErrorNotSupported;
    return b_mn ? launch_x3_t<EPI_FWD, true>(maps, g, bn, n, s) : launch_x3_t<EPI_GATE, false>(maps, g, bn, n, s);
}

}  // namespace widegemm
}  // namespace anakin
