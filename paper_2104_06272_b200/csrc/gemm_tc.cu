// Weight-gradient GEMMs on the 5th-generation tensor cores:  C[m][n] = sum_k A[k][m] B[k][n],  K = B*T rows.
//
// These are the batch-mean reductions of the update (the single-device form of the paper's cross-core gradient average,
// Podracer paper, Section 3.1): dW2 = h1^T dh2 of the widths that have no fused kernel for it, the agent plane of dW1 =
// onehot(pos)^T dh1 of the bf16 widths outside 64, 128, 256, and the wall and goal planes of every width.  Both operands have the
// contraction index as their slow (row) index, i.e. they are "MN-major" for the MMA.
//
// One CTA owns a 128 x BN output tile (BN = the hidden width up to 256, else column tiles of 256; the accumulator
// columns live in tensor memory) and a
// K range (split-K; partials are summed later in a fixed order).  Per 64-row K chunk:
//   warp 0 (one lane)  issues TMA loads of the operand planes (64 x 64 boxes, 128-byte swizzle) into a ring of two to four stages,
//   warps 2-5          for the one-hot A operand: write the 0/1 tile straight into the swizzled layout instead of loading it,
//   warp 1             issues tcgen05.mma (the whole warp walks the loop, an elected lane issues): for fp32 workloads three MMAs per
//                      k16 (lo*hi, hi*lo, hi*hi fp16 terms) into one fp32 accumulator, six with three-term operands;
//                      the small terms of the wall and goal planes go into an accumulator of their own; commits free the stage,
//   warps 2-5          after the last chunk: tcgen05.ld the accumulator and store the partial tile.
// Long K ranges (plane operands): the tensor core's fp32 accumulation rounds toward zero, which biases a sum of many
// thousand MMAs by more than the fp32 workloads' 1e-4 bound (measured: -2e-4 after 65,536 rows; fp32 workloads only).  The K range of a CTA
// is therefore cut into groups of GROUP chunks; the groups alternate between two accumulators in tensor memory, and
// while the MMAs of one group run, warps 2-5 add the previous group's accumulator into the partial tile in global
// memory with ordinary (round-to-nearest) fp32 additions, in group order.
// Every wait is bounded; a timeout raises DEV_E_WAIT_TIMEOUT in the status word and the CTA unwinds (tensor memory freed).
#include <cstdio>
#include <cstring>

#include "tc_common.cuh"

namespace anakin {

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// (initialised once, by whichever thread is first; the others wait for it)
EncodeTiledFn encode_fn() {
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) return nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// A tensor map is a pure function of these values, and a training loop asks for the same dozen every iteration: each thread keeps
// the last 64 it encoded (an encode costs about a microsecond of host time, a tenth of tiny's launch work in all).
struct MapKey {
    const void* base;
    uint64_t dims[4], strides[3];  // innermost first; strides in bytes, of dimension 1 and up
    uint32_t box[4], rank, type;   // type: 0 = fp16, 1 = bf16 (both 128-byte swizzle), 2 = bytes
    bool operator==(const MapKey& o) const { return memcmp(this, &o, sizeof(MapKey)) == 0; }
};
static_assert(sizeof(MapKey) == 8 + 7 * 8 + 6 * 4, "compared as bytes: no padding");
struct MapSlot {
    MapKey key;
    CUtensorMap map;
};

bool encode_cached(CUtensorMap* map, const MapKey& k) {
    constexpr int SLOTS = 64;
    static thread_local MapSlot slots[SLOTS] = {};
    const uint64_t h = ((uint64_t)(uintptr_t)k.base * 0x9E3779B97F4A7C15ull) ^ (k.dims[1] * 0xC2B2AE3D27D4EB4Full) ^ (k.dims[0] << 7) ^ (k.box[1] << 3) ^ k.type;
    MapSlot& s = slots[(h ^ (h >> 29)) >> 20 & (SLOTS - 1)];
    if (s.key == k) { *map = s.map; return true; }
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint32_t estr[4] = {1, 1, 1, 1};
    cuuint64_t dims[4], strides[3];
    for (int i = 0; i < 4; ++i) dims[i] = k.dims[i];
    for (int i = 0; i < 3; ++i) strides[i] = k.strides[i];
    const CUtensorMapDataType type = k.type == 2 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : k.type == 1 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    if (enc(&s.map, type, k.rank, const_cast<void*>(k.base), dims, strides, k.box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            k.type == 2 ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
        s.key = MapKey{};
        return false;
    }
    s.key = k;
    *map = s.map;
    return true;
}

}  // namespace

bool make_tensor_map_2d(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows, bool bf16) {
    return encode_cached(map, MapKey{base, {cols, rows}, {cols * 2}, {64, box_rows}, 2, bf16 ? 1u : 0u});
}

bool make_tensor_map_4d(CUtensorMap* map, const void* base, uint64_t envs, uint64_t steps, uint64_t policies, uint64_t pol_stride, uint32_t box_envs,
                        uint32_t box_steps, bool bf16) {
    return encode_cached(map, MapKey{base, {64, envs, steps, policies}, {128, envs * 128, pol_stride}, {64, box_envs, box_steps, 1}, 4, bf16 ? 1u : 0u});
}

// The same over a row-major byte matrix [rows][cols] (cols a multiple of 16) with a box of box_cols x box_rows bytes, not swizzled.
bool make_tensor_map_u8(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows, uint32_t box_cols) {
    if (cols % 16 != 0 || box_cols % 16 != 0) return false;
    return encode_cached(map, MapKey{base, {cols, rows}, {cols}, {box_cols, box_rows}, 2, 2u});
}

// DEEP: as many stages as fit (plane operands, TMA-latency-bound); otherwise two, so that two CTAs share an SM (the
// synthesized-A modes are bound by their builder threads, and a second CTA hides them).
template <int BN, int APL, int BPL, bool DEEP, int PREC = 0>
struct GemmTcCfg {
    static constexpr int BM = 128, KC = 64, THREADS = DEEP && PREC == 2 ? 320 : 192;
    static constexpr int BOX = 64 * 64 * 2;                  // one 64 x 64 box of 16-bit elements
    static constexpr int A_PLANE = (BM / 64) * BOX;          // 16 KB
    static constexpr int B_PLANE = (BN / 64) * BOX;
    static constexpr int STAGE = APL * A_PLANE + BPL * B_PLANE;
    // as many stages as fit beside the slack (the loads are latency-bound: bytes in flight set the rate), at most 4
    static constexpr int FIT = (232448 - 1024 - 128) / STAGE;
    static constexpr int STAGES = !DEEP ? 2 : (FIT >= 4 ? 4 : (FIT >= 2 ? FIT : 2));
    static constexpr size_t smem_bytes = (size_t)STAGES * STAGE + 1024 /*alignment slack*/ + 128 /*barriers, tmem slot*/;
    // plane operands of the fp32 workloads: two accumulators, a group of GROUP 64-row chunks (4096 rows, 768 MMAs) each.
    // The bf16 workload's 2e-2 bound does not need it.
    static constexpr bool FLUSH = DEEP && PREC != 1;
    // fp32 as three bf16 terms (plane operands): a stage holds all three terms of both operands, so that a staged byte feeds two
    // MMAs; every 64-row chunk is an accumulator group of its own (products smallest first, four leading MMAs), and the groups
    // are added with round-to-nearest in the registers of eight epilogue warps.
    static constexpr bool X3 = PREC == 2 && DEEP;
    static constexpr int GROUP = X3 ? 1 : 64;
    static constexpr int EPI_THREADS = X3 ? 256 : 128;
    // several terms of B beside an exact synthesized A: the leading products in one accumulator, the small terms in a second one (every
    // MMA rounds toward zero at its accumulator's magnitude), added at the end.  8192 rows, the most that one split has, are then 512
    // MMAs in the accumulator that counts; in one for both terms they were 1024.  In time it is nothing: 65536 envs,
    // 10 x 10, H = 256 29.1 us with and without, 16384, 16 x 16, H = 1024 55.6, 303104, 12 x 12, H = 256 154.
    static constexpr bool SPLIT = !DEEP && BPL >= 2;
    static constexpr int TMEM_COLS = FLUSH || SPLIT ? 2 * BN : BN;
};

struct GemmTcMaps {
    CUtensorMap a_hi, a_lo, a_lo2, b_hi, b_lo, b_lo2;
};

template <int BN, int AMODE, int APL, int BPL, int PREC>
__global__ void __launch_bounds__((GemmTcCfg<BN, APL, BPL, AMODE == A_PLANES, PREC>::THREADS), 1) k_gemm_tn_tc(const __grid_constant__ GemmTcMaps maps, GemmTnArgs g, int* status) {
    using Cfg = GemmTcCfg<BN, APL, BPL, AMODE == A_PLANES, PREC>;
    constexpr int BM = Cfg::BM, KC = Cfg::KC, STAGES = Cfg::STAGES;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);  // the swizzle needs 1024-byte alignment
    uint64_t* bars = (uint64_t*)(base + STAGES * Cfg::STAGE);  // full[STAGES], empty[STAGES], accfull[2], accempty[2]
    uint64_t* accfull = bars + 2 * STAGES;
    uint64_t* accempty = accfull + 2;
    uint32_t* tmem_slot = (uint32_t*)(accempty + 2);
    constexpr bool FLUSH = Cfg::FLUSH;
    constexpr int GROUP = Cfg::GROUP;
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    // A_ENV: two groups of row tiles with different synthesized A operands (wall bits + ones row; one-hot of idx2), each with its
    // own M space
    const int wall_tiles = AMODE == A_ENV ? (g.M + BM - 1) / BM : 0;
    const bool second = AMODE == A_ENV && (int)blockIdx.x >= wall_tiles;
    const int amode = AMODE == A_ENV ? (second ? A_ONEHOT : A_WALLS) : AMODE;
    const int m0 = ((int)blockIdx.x - (second ? wall_tiles : 0)) * BM, n0 = blockIdx.y * BN, split = blockIdx.z;
    const uint8_t* oh_idx = (AMODE == A_ENV) ? g.idx2 : g.idx;
    const int kbeg = split * g.klen, kend = min(g.K, kbeg + g.klen);
    const int nchunks = kend > kbeg ? (kend - kbeg + KC - 1) / KC : 0;
    const int ngroups = FLUSH ? (nchunks + GROUP - 1) / GROUP : (nchunks > 0 ? 1 : 0);
    constexpr uint32_t NBUILD = AMODE == A_PLANES ? 0u : 128u;

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) { tc::mbar_init(&bars[s], 1 + NBUILD); tc::mbar_init(&bars[STAGES + s], 1); }
        for (int q = 0; q < 2; ++q) { tc::mbar_init(&accfull[q], 1); tc::mbar_init(&accempty[q], Cfg::EPI_THREADS); }
        tc::mbar_fence_init();
    }
    if (wid == 2) tc::tmem_alloc(tmem_slot, Cfg::TMEM_COLS);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (tid == 0) {
        tc::prefetch_map(&maps.b_hi);
        if (BPL >= 2) tc::prefetch_map(&maps.b_lo);
        if (AMODE == A_PLANES) tc::prefetch_map(&maps.a_hi);
    }
    pdl_wait();  // (the set-up above runs under the predecessor's tail)
    bool ok = true;

    if (wid == 0) {
        if (lane == 0) {  // ---- TMA producer
            for (int c = 0; c < nchunks && ok; ++c) {
                const int s = c % STAGES, k0 = kbeg + c * KC;
                if (c >= STAGES) ok = tc::mbar_wait(&bars[STAGES + s], ((c / STAGES) - 1) & 1);
                if (!ok) break;
                unsigned char* st = base + s * Cfg::STAGE;
                constexpr uint32_t tx = (AMODE == A_PLANES ? APL * Cfg::A_PLANE : 0) + BPL * Cfg::B_PLANE;
                tc::mbar_expect_tx(&bars[s], tx);
                if (AMODE == A_PLANES) {
#pragma unroll
                    for (int bx = 0; bx < BM / 64; ++bx) {
                        tc::tma_load_2d(st + bx * Cfg::BOX, &maps.a_hi, &bars[s], m0 + 64 * bx, k0);
                        if (APL == 3) tc::tma_load_2d(st + 2 * Cfg::A_PLANE + bx * Cfg::BOX, &maps.a_lo2, &bars[s], m0 + 64 * bx, k0);
                        if (APL >= 2) tc::tma_load_2d(st + Cfg::A_PLANE + bx * Cfg::BOX, &maps.a_lo, &bars[s], m0 + 64 * bx, k0);
                    }
                }
                unsigned char* sb = st + APL * Cfg::A_PLANE;
#pragma unroll
                for (int bx = 0; bx < BN / 64; ++bx) {
                    tc::tma_load_2d(sb + bx * Cfg::BOX, &maps.b_hi, &bars[s], n0 + 64 * bx, k0);
                    if (BPL >= 2) tc::tma_load_2d(sb + Cfg::B_PLANE + bx * Cfg::BOX, &maps.b_lo, &bars[s], n0 + 64 * bx, k0);
                    if (BPL == 3) tc::tma_load_2d(sb + 2 * Cfg::B_PLANE + bx * Cfg::BOX, &maps.b_lo2, &bars[s], n0 + 64 * bx, k0);
                }
            }
            pdl_trigger();  // (the last loads are on their way)
            if (!ok) atomicOr(status, DEV_E_WAIT_TIMEOUT);
        }
    } else if (wid == 1) {
        {  // ---- MMA issuer: the whole warp walks the loop, one elected lane issues
            const uint32_t idesc = tc::umma_idesc<PREC>(BM, BN, true, true);
            for (int c = 0; c < nchunks && ok; ++c) {
                const int s = c % STAGES;
                const int grp = FLUSH ? c / GROUP : 0, cg = FLUSH ? c - grp * GROUP : c;  // accumulator group, chunk within it
                const uint32_t acc = tmem + (uint32_t)((grp & 1) * BN);
                // the third and later groups reuse an accumulator: wait until the epilogue warps have read it out
                if (FLUSH && cg == 0 && grp >= 2) ok = tc::mbar_wait(&accempty[grp & 1], ((grp >> 1) - 1) & 1);
                ok = tc::warp_all(ok && tc::mbar_wait(&bars[s], (c / STAGES) & 1));
                if (!ok) break;
                tc::tc_fence_after();
                unsigned char* sa = base + s * Cfg::STAGE;
                unsigned char* sb = sa + APL * Cfg::A_PLANE;
                if (tc::elect_one()) {
                if constexpr (Cfg::X3) {
#pragma unroll
                    for (int i = 0; i < tc::X3_PAIRS; ++i)
#pragma unroll
                        for (int k16 = 0; k16 < KC / 16; ++k16)
                            tc::umma(acc, tc::umma_desc(sa + tc::x3_a(i) * Cfg::A_PLANE + k16 * 2048, Cfg::BOX, 1024),
                                     tc::umma_desc(sb + tc::x3_b(i) * Cfg::B_PLANE + k16 * 2048, Cfg::BOX, 1024), idesc, (i > 0 || k16 > 0) ? 1u : 0u);
                } else
#pragma unroll
                for (int k16 = 0; k16 < KC / 16; ++k16) {
                    // 16 k rows = two 8-row groups = 2048 bytes further into every box
                    const uint64_t a_hi = tc::umma_desc(sa + k16 * 2048, Cfg::BOX, 1024);
                    const uint64_t b_hi = tc::umma_desc(sb + k16 * 2048, Cfg::BOX, 1024);
                    uint32_t accum = (cg > 0 || k16 > 0) ? 1u : 0u;
                    if (APL == 2) { tc::umma(acc, tc::umma_desc(sa + Cfg::A_PLANE + k16 * 2048, Cfg::BOX, 1024), b_hi, idesc, accum); accum = 1u; }
                    if (Cfg::SPLIT) {
                        if (BPL == 3) tc::umma(acc + BN, a_hi, tc::umma_desc(sb + 2 * Cfg::B_PLANE + k16 * 2048, Cfg::BOX, 1024), idesc, accum);
                        tc::umma(acc + BN, a_hi, tc::umma_desc(sb + Cfg::B_PLANE + k16 * 2048, Cfg::BOX, 1024), idesc, BPL == 3 ? 1u : accum);
                    }
                    if (BPL == 2 && !Cfg::SPLIT) { tc::umma(acc, a_hi, tc::umma_desc(sb + Cfg::B_PLANE + k16 * 2048, Cfg::BOX, 1024), idesc, accum); accum = 1u; }
                    tc::umma(acc, a_hi, b_hi, idesc, accum);
                }
                tc::umma_commit(&bars[STAGES + s]);  // frees the stage when these MMAs are done
                if (c == nchunks - 1 || (FLUSH && cg == GROUP - 1)) tc::umma_commit(&accfull[grp & 1]);  // this group's sum is complete
                }
                __syncwarp();
            }
            if (!ok && lane == 0) atomicOr(status, DEV_E_WAIT_TIMEOUT);
        }
    } else {
        // ---- warps 2-5: builders of a synthesized A tile, then the epilogue
        const int bt = tid - 64;  // 0..127
        if (AMODE != A_PLANES) {
            // (after a timeout the loop keeps going without waiting, so that every thread still meets every bar.sync)
            for (int c = 0; c < nchunks; ++c) {
                const int s = c % STAGES, k0 = kbeg + c * KC;
                if (ok && c >= STAGES) ok = tc::mbar_wait(&bars[STAGES + s], ((c / STAGES) - 1) & 1);
                unsigned char* sa = base + s * Cfg::STAGE;
                // element (k, m) of the tile lives in box m/64 at byte  k*128 + (((m%64)/8) ^ (k%8))*16 + (m%8)*2
                if (amode == A_ONEHOT) {
                    uint4* z = reinterpret_cast<uint4*>(sa);
                    for (int i = bt; i < Cfg::A_PLANE / 16; i += 128) z[i] = make_uint4(0u, 0u, 0u, 0u);
                    asm volatile("bar.sync 1, 128;" ::: "memory");  // zeros before ones
                    if (bt < KC && k0 + bt < kend) {
                        const int m = (int)oh_idx[g.kmod ? (k0 + bt) % g.kmod : (k0 + bt)] - m0;
                        if (m >= 0 && m < BM) {
                            const int k = bt;
                            const uint32_t off = (m >> 6) * Cfg::BOX + k * 128 + ((((m & 63) >> 3) ^ (k & 7)) << 4) + (m & 7) * 2;
                            *reinterpret_cast<uint16_t*>(sa + off) = (uint16_t)one16<PREC>();
                        }
                    }
                } else {  // A_WALLS: thread = (k row, 64-wide box); it writes all eight 16-byte chunks of its row segment
                    const int k = bt >> 1, bx = bt & 1;
                    const int kk = k0 + k;
                    // the 64 cells m = mb .. mb + 63 of this box as one bit mask: wall bits below ones_row, the ones row itself
                    const int mb = m0 + 64 * bx;  // a multiple of 64: two whole words of the env's wall mask
                    unsigned long long bits = 0ull;
                    if (kk < kend) {
                        const uint32_t* wrow = g.walls + (size_t)(g.kmod ? kk % g.kmod : kk) * g.W;
                        const int w0 = mb >> 5;
                        const uint32_t lo32 = w0 < g.W ? wrow[w0] : 0u, hi32 = w0 + 1 < g.W ? wrow[w0 + 1] : 0u;
                        bits = (unsigned long long)lo32 | ((unsigned long long)hi32 << 32);
                        const int r1 = g.ones_row - mb;  // position of the ones row in this box
                        if (r1 <= 0) bits = 0ull;
                        else if (r1 < 64) bits &= (1ull << r1) - 1ull;
                        if (r1 >= 0 && r1 < 64) bits |= 1ull << r1;
                    }
                    const uint32_t one = one16<PREC>();
#pragma unroll
                    for (int c8 = 0; c8 < 8; ++c8) {
                        const uint32_t by = (uint32_t)(bits >> (8 * c8)) & 0xFFu;
                        uint32_t w[4];
#pragma unroll
                        for (int q2 = 0; q2 < 4; ++q2) w[q2] = ((by >> (2 * q2)) & 1u) * one | ((by >> (2 * q2 + 1)) & 1u) * (one << 16);
                        *reinterpret_cast<uint4*>(sa + bx * Cfg::BOX + k * 128 + ((c8 ^ (k & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                }
                tc::fence_proxy_async();  // generic-proxy stores -> visible to the tensor core
                tc::mbar_arrive(&bars[s]);
            }
            if (!ok && lane == 0) atomicOr(status, DEV_E_WAIT_TIMEOUT);
        }
        // epilogue: warp w reads accumulator lanes 32*(w%4)..+31 = output rows.  Group 0 writes the partial tile, every
        // later group adds to what this same thread wrote (program order; round-to-nearest additions in group order).
        const int q = wid & 3;
        const int m = m0 + 32 * q + lane;
        const int Mrows = second ? g.M2 : g.M;
        float* part = second ? g.part2 + (size_t)split * g.stride2 : g.part + (size_t)split * g.stride + g.off;
        bool got = true;
        if constexpr (Cfg::X3) {  // warps 2-9: column half (wid - 2) / 4 of the tile, sums in registers, one store at the end
            constexpr int COLS = BN / 2;
            const int half = (wid - 2) >> 2;
            float sum[COLS];
#pragma unroll
            for (int j = 0; j < COLS; ++j) sum[j] = 0.f;  // an empty K range contributes zeros
            for (int grp = 0; grp < ngroups && got; ++grp) {
                got = tc::mbar_wait(&accfull[grp & 1], (grp >> 1) & 1);
                tc::tc_fence_after();
                __syncwarp();
                const uint32_t acc = tmem + (uint32_t)((grp & 1) * BN + half * COLS) + ((uint32_t)(32 * q) << 16);
                if (got) {
#pragma unroll
                    for (int c0 = 0; c0 < COLS; c0 += 32) {
                        uint32_t r[32];
                        tc::tmem_ld32(acc + (uint32_t)c0, r);
#pragma unroll
                        for (int j = 0; j < 32; ++j) sum[c0 + j] += __uint_as_float(r[j]);
                    }
                }
                tc::tc_fence_before();
                if (grp + 2 < ngroups) tc::mbar_arrive(&accempty[grp & 1]);  // hand the accumulator back to the issuer
            }
            if (m < Mrows) {
                float4* dst = reinterpret_cast<float4*>(part + (size_t)m * g.ldc + n0 + half * COLS);
#pragma unroll
                for (int j = 0; j < COLS / 4; ++j)
                    if (n0 + half * COLS + 4 * j < g.N) dst[j] = make_float4(sum[4 * j], sum[4 * j + 1], sum[4 * j + 2], sum[4 * j + 3]);
            }
        } else
        for (int grp = 0; grp < (ngroups > 0 ? ngroups : 1); ++grp) {
            if (ngroups > 0 && got) got = tc::mbar_wait(&accfull[grp & 1], (grp >> 1) & 1);
            tc::tc_fence_after();
            __syncwarp();
            const uint32_t acc = tmem + (uint32_t)((grp & 1) * BN) + ((uint32_t)(32 * q) << 16);
            for (int c0 = 0; c0 < BN; c0 += 32) {
                uint32_t r[32];
                if (ngroups > 0 && got) {
                    tc::tmem_ld32(acc + (uint32_t)c0, r);
                    if constexpr (Cfg::SPLIT) {
                        uint32_t r2[32];
                        tc::tmem_ld32(acc + (uint32_t)(BN + c0), r2);
#pragma unroll
                        for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(r2[j]));
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j) r[j] = 0u;  // an empty K range contributes zeros
                }
                if (m < Mrows && n0 + c0 < g.N) {
                    float4* dst = reinterpret_cast<float4*>(part + (size_t)m * g.ldc + n0 + c0);
                    if (amode == A_WALLS && m == g.ones_row) dst = reinterpret_cast<float4*>(part - g.off + g.off_ones + n0 + c0);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float4 v = make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]), __uint_as_float(r[4 * j + 2]),
                                               __uint_as_float(r[4 * j + 3]));
                        if (grp > 0) {
                            const float4 o = dst[j];
                            v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
                        }
                        dst[j] = v;
                    }
                }
            }
            if (FLUSH && grp + 2 < ngroups) {  // hand the accumulator back to the issuer
                tc::tc_fence_before();
                tc::mbar_arrive(&accempty[grp & 1]);
            }
        }
        if (!got && lane == 0) atomicOr(status, DEV_E_WAIT_TIMEOUT);
    }
    tc::tc_fence_before();
    __syncthreads();
    if (wid == 2) tc::tmem_dealloc(tmem, Cfg::TMEM_COLS);
}

template <int BN, int AMODE, int APL, int BPL, int PREC>
static cudaError_t launch_t(const GemmTnArgs& g, int splits, int* status, cudaStream_t s) {
    using Cfg = GemmTcCfg<BN, APL, BPL, AMODE == A_PLANES, PREC>;
    GemmTcMaps maps;
    memset(&maps, 0, sizeof(maps));
    const bool bf = PREC >= 1;
    // (every term is a matrix of its own: rows past K read as zeros)
    auto map = [&](CUtensorMap* m, const __nv_bfloat16* p, int ld) { return make_tensor_map_2d(m, p, (uint64_t)g.K, (uint64_t)ld, 64, bf); };
    if (AMODE == A_PLANES) {
        if (!map(&maps.a_hi, g.Ahi, g.lda)) return cudaErrorNotSupported;
        if (APL >= 2 && !map(&maps.a_lo, g.Alo, g.lda)) return cudaErrorNotSupported;
        if (APL == 3 && !map(&maps.a_lo2, g.Alo + (g.Alo - g.Ahi), g.lda)) return cudaErrorNotSupported;
    }
    if (!map(&maps.b_hi, g.Bhi, g.ldb)) return cudaErrorNotSupported;
    if (BPL >= 2 && !map(&maps.b_lo, g.Blo, g.ldb)) return cudaErrorNotSupported;
    if (BPL == 3 && !map(&maps.b_lo2, g.Blo + (g.Blo - g.Bhi), g.ldb)) return cudaErrorNotSupported;
    dim3 grid((g.M + Cfg::BM - 1) / Cfg::BM + (AMODE == A_ENV ? (g.M2 + Cfg::BM - 1) / Cfg::BM : 0), (g.N + BN - 1) / BN, splits);
    return launch<k_gemm_tn_tc<BN, AMODE, APL, BPL, PREC>>(grid, Cfg::THREADS, Cfg::smem_bytes, s, maps, g, status);
}

template <int BN, int PREC>
static cudaError_t launch_bn(const GemmTnArgs& g, int amode, int splits, int* status, cudaStream_t s) {
    constexpr int PL = PREC == 1 ? 1 : PREC == 2 ? 3 : 2, SPL = PREC == 2 ? 3 : 2;  // terms of an activation, of S
    // (fp32 as three bf16 terms, plane operands: 128-column tiles, two stages of 96 KB)
    if (amode == A_PLANES) return launch_t<PREC == 2 ? 128 : BN, A_PLANES, PL, PL, PREC>(g, splits, status, s);
    if (amode == A_ENV) return launch_t<BN, A_ENV, 1, SPL, PREC>(g, splits, status, s);
    if constexpr (PREC == 1) {  // the agent plane of the wide layers
        if (amode == A_ONEHOT) return launch_t<BN, A_ONEHOT, 1, 1, PREC>(g, splits, status, s);
    }
    return cudaErrorNotSupported;
}

template <int PREC>
static cudaError_t launch_p(const GemmTnArgs& g, int amode, int splits, int* status, cudaStream_t s) {
    if (g.N > 128) return launch_bn<256, PREC>(g, amode, splits, status, s);
    if (g.N > 64) return launch_bn<128, PREC>(g, amode, splits, status, s);
    return launch_bn<64, PREC>(g, amode, splits, status, s);
}

// CTAs of the wall and goal planes' launch that an SM holds at once (its 228 KB of shared memory decide, 1 KB of them a CTA's own).
int gemm_tn_tc_env_per_sm(int H, bool three) {
    constexpr size_t sm = 228 * 1024;
    auto fit = [](size_t smem) { return (int)(sm / (smem + 1024)); };
    if (H > 128) return three ? fit(GemmTcCfg<256, 1, 3, false, 2>::smem_bytes) : fit(GemmTcCfg<256, 1, 2, false, 0>::smem_bytes);
    if (H > 64) return three ? fit(GemmTcCfg<128, 1, 3, false, 2>::smem_bytes) : fit(GemmTcCfg<128, 1, 2, false, 0>::smem_bytes);
    return three ? fit(GemmTcCfg<64, 1, 3, false, 2>::smem_bytes) : fit(GemmTcCfg<64, 1, 2, false, 0>::smem_bytes);
}

// Covered: N = ldb a multiple of 32 (column tiles of 64, 128 or 256; columns past N read as zeros and are not stored), klen a
// multiple of 64, the planes of the workload's precision.
cudaError_t launch_gemm_tn_tc(const GemmTnArgs& g, int amode, int prec, int splits, int* status, cudaStream_t s) {
    if (g.N != g.ldb || g.N % 32 != 0 || g.klen % 64 != 0 || (amode == A_PLANES && g.lda % 32 != 0)) return cudaErrorNotSupported;
    return prec == 2 ? launch_p<2>(g, amode, splits, status, s) : prec == 1 ? launch_p<1>(g, amode, splits, status, s) : launch_p<0>(g, amode, splits, status, s);
}

}  // namespace anakin
