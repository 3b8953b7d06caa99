// Backward pass through the second layer at hidden width 64 in one tcgen05 kernel: dh1 = (dh2 W2^T) gated by h1 > 0, S = sum
// over t of dh1, dW2 = h1^T dh2 and the agent plane of dW1 = onehot(pos)^T dh1 (the update half of the Anakin minimal unit,
// Podracer paper, Section 3.1).
//
// What bounds it: HBM.  At 64 columns every product of a row is small, so the cost of a separate kernel per product is its
// reads: dh1 written and read again, dh2 read twice.  Here a row of dh2 and of h1 is fetched once (8 bytes an element in fp32
// workloads) and dh1 exists only in shared memory.
//
// A tile is 128 rows: 128 envs of one step, or, for batches of up to 64 envs, several steps of all of them.  With the rows as
// accumulator lanes one 128-byte-swizzled box [row][64 units] serves both ways: K-major for dh1 (k = unit), MN-major for the
// two gradients (k = row).  A CTA walks (env tile, slice of the steps) units; several policies take a slice of grid.z each.
//   warp 0      TMA: the dh2 and h1 planes of a tile into one stage (rows past the batch or the last step arrive as zeros)
//   warp 1      tcgen05.mma: the dh1 product (K = 64) into one of two accumulators; dW2 (K = 128 rows; the hi and the lo plane
//               of h1 are the two halves of M, so both terms of h1 cost one MMA); then, for the tile before, the agent plane
//               (A = one-hot cells, 128 or 256 of them; B = dh1)
//   warps 2-9   thread = (row, half of the units): tcgen05.ld, gate, S +=, 16-bit split; the dh1 planes go over the dh2 planes
//               of the same stage once dW2 has read them
// The tensor core rounds toward zero, so a long sum in one accumulator comes out low.  dW2 restarts its accumulator every FLUSH tiles
// (4096 rows, as in the plain GEMM) and the groups are added in registers; the agent plane restarts every AGENT_FLUSH tiles (768 MMAs
// an accumulator, fp32 workloads) and the groups are added in the CTA's partial.  Left to run, 142,000 rows a CTA on 2 x 2 cells came
// out 1.1e-4 low.
#include <cstring>

#include "tc_common.cuh"

namespace anakin {

namespace {

__device__ __forceinline__ void tmem_cols(uint32_t taddr, uint32_t (&r)[16]) { tc::tmem_ld16_nowait(taddr, r); }
__device__ __forceinline__ void tmem_cols(uint32_t taddr, uint32_t (&r)[32]) { tc::tmem_ld32_nowait(taddr, r); }

template <int PREC, int NC>
struct Back64Cfg {
    static constexpr int H = 64, BM = 128;
    static constexpr int PL = PREC == 1 ? 1 : 2;
    static constexpr int EPI_WARPS = 8, FIRST_EPI = 2, THREADS = 32 * (FIRST_EPI + EPI_WARPS);
    static constexpr int BOX = BM * 128;             // 128 rows x 64 16-bit elements
    static constexpr int STAGE = PL * BOX;           // the planes of one operand
    static constexpr int HST = PREC == 1 ? 3 : 2;    // h1 ring
    static constexpr int DST = PREC == 1 ? 4 : NC == 1 ? 3 : 2;  // dh2 ring (a stage then holds the dh1 planes: it is busy longer)
    static constexpr int W_BOX = H * 128, W_BYTES = PL * W_BOX;
    static constexpr int O_TILE = 2 * NC * BOX;      // one-hot: 128 rows x NC * 128 cells in 64-wide boxes
    static constexpr int FLUSH = 32;                 // tiles per dW2 accumulator
    // tiles per agent-plane accumulator, and of the first one.  Its last tile is never the one before a restart of dW2: there the issuer
    // waits for the epilogue of the new tile before it issues the agent MMAs of the old one, which that epilogue would be waiting for.
    static constexpr int AGENT_FLUSH = 96, AGENT_FIRST = 80;
    static_assert(AGENT_FLUSH % FLUSH == 0 && AGENT_FIRST % FLUSH != 0, "the agent plane and dW2 never restart at the same tile");
    // Two planes of the N operand are one MMA of 128 columns (half of them the lo plane's): the M operand is then read from shared
    // memory once, and shared memory is what bounds these products.  (At NC = 2 tensor memory has no room for it in dh1.)
    static constexpr int W2_N = PL * H, AGENT_N = PL * H, ACC_N = PL == 2 && NC == 1 ? 2 * H : H;
    static constexpr int ACC_COL = 0, W2_COL = 2 * ACC_N, AGENT_COL = W2_COL + W2_N, TMEM_COLS = 512;
    static_assert(AGENT_COL + NC * AGENT_N <= TMEM_COLS, "tensor memory");
    static constexpr size_t smem_bytes = (size_t)(HST + DST) * STAGE + W_BYTES + O_TILE + 256 + 1024;
    static_assert(smem_bytes <= 232448, "227 KB per CTA");
};

struct Back64Maps {
    CUtensorMap d_hi, d_lo, h_hi, h_lo;              // every policy but the last
    CUtensorMap ld_hi, ld_lo, lh_hi, lh_lo;          // the last policy (fewer envs)
};
struct Back64Args {
    LearnArgs a;
    float *part_w2, *part_agent;
    size_t stride_agent;
    int nx;  // CTAs per policy: one partial of dW2 and of the agent plane each
};

// LONG: a CTA may walk more than AGENT_FIRST tiles.
template <int PREC, int NC, bool GROUPED, bool LONG>
__global__ void __launch_bounds__(Back64Cfg<PREC, NC>::THREADS, 1) k_back64(const __grid_constant__ Back64Maps maps, const __grid_constant__ Back64Args in) {
    using Cfg = Back64Cfg<PREC, NC>;
    constexpr int H = Cfg::H, BM = Cfg::BM, PL = Cfg::PL, HST = Cfg::HST, DST = Cfg::DST, BOX = Cfg::BOX;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sH = base;                              // [HST] h1 planes
    unsigned char* sD = sH + HST * Cfg::STAGE;             // [DST] dh2 planes, then dh1 planes
    unsigned char* sW = sD + DST * Cfg::STAGE;             // W2 planes, 64 rows x 64 k each
    unsigned char* sO = sW + Cfg::W_BYTES;                 // one-hot tile
    uint64_t* bars = (uint64_t*)(sO + Cfg::O_TILE);
    uint64_t* hfull = bars;                // [HST] h1 planes landed
    uint64_t* hempty = hfull + HST;        // [HST] dW2 has read them (commit) and the gates have been taken (the epilogue warps arrive)
    uint64_t* full = hempty + HST;         // [DST] dh2 planes landed
    uint64_t* empty = full + DST;          // [DST] the agent MMAs of the tile have finished
    uint64_t* w2done = empty + DST;        // [DST] dW2 (and dh1) of the tile have finished: the dh2 planes may be overwritten
    uint64_t* tfull = w2done + DST;        // [2] dh1 accumulator written
    uint64_t* tempty = tfull + 2;          // [2] dh1 accumulator drained (the epilogue warps arrive)
    uint64_t* wfull = tempty + 2;          // W2 planes in shared memory (the epilogue warps arrive)
    uint64_t* tiles_full = wfull + 1;      // dh1 planes and one-hot of a tile written (the epilogue warps arrive)
    uint32_t* tmem_slot = (uint32_t*)(tiles_full + 1);

    const int pol = GROUPED ? (int)blockIdx.z : 0;
    const PolicyArgs<GROUPED, LearnArgs> pa(in.a, pol);
    const LearnArgs& a = pa.a;
    const Dims& d = a.d;
    const Buffers& b = a.b;
    const bool last = GROUPED && pol == in.a.d.npol - 1 && d.B_last != in.a.d.B;
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const int B = d.B, T = a.T, C = d.C;
    // rows of a tile: SP steps of TE envs
    const int SP = in.a.d.B <= BM / 2 ? min(BM / in.a.d.B, T) : 1, TE = SP > 1 ? B : BM;
    const int m_tiles = SP > 1 ? 1 : (B + BM - 1) / BM;
    const int nx = in.nx, xi = blockIdx.x, units = m_tiles * a.ts;
    const int tl = ((T + a.ts - 1) / a.ts + SP - 1) / SP * SP;  // steps of a slice
    auto t_begin = [&](int u) { return min((u / m_tiles) * tl, T); };
    auto t_end = [&](int u) { return min((u / m_tiles) * tl + tl, T); };

    if (tid == 0) {
        for (int s = 0; s < HST; ++s) { tc::mbar_init(&hfull[s], 1); tc::mbar_init(&hempty[s], 1 + Cfg::EPI_WARPS); }
        for (int s = 0; s < DST; ++s) { tc::mbar_init(&full[s], 1); tc::mbar_init(&empty[s], 1); tc::mbar_init(&w2done[s], 1); }
        for (int i = 0; i < 2; ++i) { tc::mbar_init(&tfull[i], 1); tc::mbar_init(&tempty[i], Cfg::EPI_WARPS); }
        tc::mbar_init(wfull, Cfg::EPI_WARPS);
        tc::mbar_init(tiles_full, Cfg::EPI_WARPS);
        tc::mbar_fence_init();
    }
    if (wid == 1) tc::tmem_alloc(tmem_slot, Cfg::TMEM_COLS);
    // the one-hot tile starts all zero (every tile clears the elements of the one before); so do the rows that no box fills
    for (int i = tid; i < Cfg::O_TILE / 16; i += Cfg::THREADS) reinterpret_cast<uint4*>(sO)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (SP * TE < BM)
        for (int i = tid; i < (HST + DST) * Cfg::STAGE / 16; i += Cfg::THREADS) reinterpret_cast<uint4*>(sH)[i] = make_uint4(0u, 0u, 0u, 0u);
    tc::fence_proxy_async();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (tid == 0) {
        tc::prefetch_map(last ? &maps.ld_hi : &maps.d_hi);
        tc::prefetch_map(last ? &maps.lh_hi : &maps.h_hi);
        if (PL == 2) { tc::prefetch_map(last ? &maps.ld_lo : &maps.d_lo); tc::prefetch_map(last ? &maps.lh_lo : &maps.h_lo); }
    }
    pdl_wait();  // (the set-up above runs under the predecessor's tail)
    int G = 0;  // tiles of this CTA
    for (int u = xi; u < units; u += nx) G += (t_end(u) - t_begin(u) + SP - 1) / SP;
    bool ok = true;

    if (wid == 0) {
        if (lane == 0) {  // ---- TMA producer
            const CUtensorMap* mh = last ? &maps.lh_hi : &maps.h_hi;
            const CUtensorMap* ml = last ? &maps.lh_lo : &maps.h_lo;
            const CUtensorMap* dh = last ? &maps.ld_hi : &maps.d_hi;
            const CUtensorMap* dl = last ? &maps.ld_lo : &maps.d_lo;
            const int w = last ? 0 : pol;
            const uint32_t bytes = PL * (uint32_t)(SP * TE) * 128u;
            int g = 0;
            for (int u = xi; u < units && ok; u += nx) {
                const int env0 = (u % m_tiles) * BM, t1 = t_end(u);
                for (int t = t_begin(u); t < t1; t += SP, ++g) {
                    const int hs = g % HST, ds = g % DST, tp = t + DST * SP;
                    if (tp < t1) {  // pull a later tile of this unit towards L2
                        tc::tma_prefetch_4d(dh, 0, env0, tp, w);
                        tc::tma_prefetch_4d(mh, 0, env0, tp, w);
                        if (PL == 2) { tc::tma_prefetch_4d(dl, 0, env0, tp, w); tc::tma_prefetch_4d(ml, 0, env0, tp, w); }
                    }
                    if (g >= DST) ok = tc::mbar_wait(&empty[ds], (uint32_t)(g / DST - 1) & 1u);
                    if (!ok) break;
                    tc::mbar_expect_tx(&full[ds], bytes);
                    tc::tma_load_4d(sD + ds * Cfg::STAGE, dh, &full[ds], 0, env0, t, w);
                    if (PL == 2) tc::tma_load_4d(sD + ds * Cfg::STAGE + BOX, dl, &full[ds], 0, env0, t, w);
                    if (g >= HST) ok = tc::mbar_wait(&hempty[hs], (uint32_t)(g / HST - 1) & 1u);
                    if (!ok) break;
                    tc::mbar_expect_tx(&hfull[hs], bytes);
                    tc::tma_load_4d(sH + hs * Cfg::STAGE, mh, &hfull[hs], 0, env0, t, w);
                    if (PL == 2) tc::tma_load_4d(sH + hs * Cfg::STAGE + BOX, ml, &hfull[hs], 0, env0, t, w);
                }
            }
            pdl_trigger();  // (the last loads are on their way)
            if (!ok) atomicOr(b.status, DEV_E_WAIT_TIMEOUT);
        }
    } else if (wid == 1) {  // ---- MMA issuer: the whole warp walks the loop, one elected lane issues
        const uint32_t id_dh1 = tc::umma_idesc<PREC>(BM, H, false, false), id_dh1_2 = tc::umma_idesc<PREC>(BM, 2 * H, false, false);
        const uint32_t id_w2 = tc::umma_idesc<PREC>(128, Cfg::W2_N, true, true), id_agent = tc::umma_idesc<PREC>(128, Cfg::AGENT_N, true, true);
        auto agent_mma = [&](int v) {  // 16 rows = 2048 bytes further in the MN-major boxes; the lo plane of dh1 one box on
            const int s = v % DST;
            ok = tc::warp_all(tc::mbar_wait(tiles_full, (uint32_t)v & 1u));
            if (!ok) return;
            tc::tc_fence_after();
            if (tc::elect_one()) {
#pragma unroll
                for (int k16 = 0; k16 < BM / 16; ++k16) {
                    const uint64_t dd = tc::umma_desc(sD + s * Cfg::STAGE + k16 * 2048, BOX, 1024);
#pragma unroll
                    for (int c = 0; c < NC; ++c)
                        tc::umma(tmem + (uint32_t)(Cfg::AGENT_COL + Cfg::AGENT_N * c), tc::umma_desc(sO + 2 * c * BOX + k16 * 2048, BOX, 1024), dd, id_agent,
                                 (v > 0 && !(LONG && v % Cfg::AGENT_FLUSH == Cfg::AGENT_FIRST)) || k16 > 0);  // (a group's first MMA restarts the sum)
                }
                tc::umma_commit(&empty[s]);
            }
            __syncwarp();
        };
        ok = tc::warp_all(tc::mbar_wait(wfull, 0));
        for (int g = 0; g < G && ok; ++g) {
            const int hs = g % HST, ds = g % DST, buf = g & 1;
            if (g >= 2) ok = tc::warp_all(tc::mbar_wait(&tempty[buf], (uint32_t)((g >> 1) - 1) & 1u));
            if (ok) ok = tc::warp_all(tc::mbar_wait(&full[ds], (uint32_t)(g / DST) & 1u));
            if (!ok) break;
            tc::tc_fence_after();
            const unsigned char* sh = sH + hs * Cfg::STAGE;
            const unsigned char* sd = sD + ds * Cfg::STAGE;
            if (tc::elect_one()) {
                const uint32_t acc = tmem + (uint32_t)(Cfg::ACC_COL + Cfg::ACC_N * buf);
                // dh1 per k16 (32 bytes along the swizzled rows): dh2 hi x [W hi | W lo] where there is room for both halves (they
                // are added in the epilogue), dh2 lo x W hi
#pragma unroll
                for (int k16 = 0; k16 < H / 16; ++k16) {
                    const uint64_t d_hi = tc::umma_desc(sd + k16 * 32, 16, 1024), w_hi = tc::umma_desc(sW + k16 * 32, 16, 1024);
                    if (PL == 1) {
                        tc::umma(acc, d_hi, w_hi, id_dh1, k16 > 0);
                    } else {
                        const uint64_t d_lo = tc::umma_desc(sd + BOX + k16 * 32, 16, 1024);
                        if (NC == 1) {
                            tc::umma(acc, d_hi, w_hi, id_dh1_2, k16 > 0);
                            tc::umma(acc, d_lo, w_hi, id_dh1, 1u);
                        } else {
                            tc::umma(acc, d_hi, tc::umma_desc(sW + Cfg::W_BOX + k16 * 32, 16, 1024), id_dh1, k16 > 0);
                            tc::umma(acc, d_lo, w_hi, id_dh1, 1u);
                            tc::umma(acc, d_hi, w_hi, id_dh1, 1u);
                        }
                    }
                }
                tc::umma_commit(&tfull[buf]);
            }
            __syncwarp();
            ok = tc::warp_all(tc::mbar_wait(&hfull[hs], (uint32_t)(g / HST) & 1u));
            // a new group of dW2: the accumulator of the one before has been read (the epilogue does so ahead of its own dh1)
            if (ok && g > 0 && g % Cfg::FLUSH == 0) ok = tc::warp_all(tc::mbar_wait(&tempty[buf], (uint32_t)(g >> 1) & 1u));
            if (!ok) break;
            tc::tc_fence_after();
            if (tc::elect_one()) {
                // dW2: M = units of the hi plane of h1, then of the lo plane one box on (bf16: whatever follows, 64 lanes that are not
                // read); N = units of dh2, the lo plane's behind the hi plane's
                const uint32_t acc2 = tmem + (uint32_t)Cfg::W2_COL;
#pragma unroll
                for (int k16 = 0; k16 < BM / 16; ++k16)
                    tc::umma(acc2, tc::umma_desc(sh + k16 * 2048, BOX, 1024), tc::umma_desc(sd + k16 * 2048, BOX, 1024), id_w2, g % Cfg::FLUSH != 0 || k16 > 0);
                tc::umma_commit(&w2done[ds]);
                tc::umma_commit(&hempty[hs]);
            }
            __syncwarp();
            if (g >= 1) agent_mma(g - 1);
        }
        if (ok && G > 0) agent_mma(G - 1);
        if (!ok && lane == 0) atomicOr(b.status, DEV_E_WAIT_TIMEOUT);
    } else {
        // ---- epilogue: thread = row r (accumulator lane) x 32 of the 64 units
        const int q = wid & 3, r = 32 * q + lane, half = (wid - Cfg::FIRST_EPI) >> 2, etid = tid - 32 * Cfg::FIRST_EPI;
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        {   // W2 rows, 16-byte pieces permuted by row % 8
            constexpr int TRIPS = PL * H * 8 / 256;
            uint4 v[TRIPS];
#pragma unroll
            for (int k = 0; k < TRIPS; ++k) {
                const int i = etid + 256 * k;
                v[k] = __ldg(reinterpret_cast<const uint4*>((i / (H * 8) ? b.w2p_lo : b.w2p_hi) + ((i / 8) % H) * H) + (i & 7));
            }
#pragma unroll
            for (int k = 0; k < TRIPS; ++k) {
                const int i = etid + 256 * k, row = (i / 8) % H;
                *reinterpret_cast<uint4*>(sW + (i / (H * 8)) * Cfg::W_BOX + row * 128 + (((i & 7) ^ (row & 7)) << 4)) = v[k];
            }
        }
        tc::fence_proxy_async();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(wfull);
        const int row_e = SP > 1 ? r % TE : r, row_dt = SP > 1 ? r / TE : 0;  // env of the tile, step of the tile
        int prev_off = -1;  // byte offset of the one-hot element this thread set for the tile before
        int g = 0;
        float w_acc[32], s_acc[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) w_acc[i] = 0.f;
        uint16_t* const S_hi = reinterpret_cast<uint16_t*>(b.S);
        uint16_t* const S_lo = S_hi + (size_t)a.ts * B * H;
        // 32 columns of this thread's lane: those of the hi half of the accumulator and, behind them, of the lo half, added
        auto read_pair = [&](uint32_t col, bool two, float (&v)[32]) {
            uint32_t x0[32], x1[32];
            tc::tmem_ld32_nowait(tmem + lane_base + col + 32 * half, x0);
            if (two) tc::tmem_ld32_nowait(tmem + lane_base + col + 64 + 32 * half, x1);
            tc::tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = two ? __uint_as_float(x0[i]) + __uint_as_float(x1[i]) : __uint_as_float(x0[i]);
        };
        auto add_w2 = [&]() {  // += this thread's 32 columns of the finished dW2 accumulator
            float v[32];
            read_pair(Cfg::W2_COL, PL == 2, v);
#pragma unroll
            for (int i = 0; i < 32; ++i) w_acc[i] += v[i];
        };
        // The agent accumulators (lane = cell, column = unit) into this CTA's partial: the first group is written, every later one added
        // to what this same thread wrote.  The MMAs of the tiles so far have been waited for; no other is issued before this warp's
        // next arrival on tiles_full.
        // W columns at a time: 16 inside the loop, which leaves few registers; 32 and unrolled at the end, where nothing runs beside it.
        auto drain_agent = [&](auto width, bool first, bool got) {
            constexpr int W = decltype(width)::value, PIECES = NC * (32 / W);
            float* pagent = in.part_agent + (size_t)xi * in.stride_agent;
            if (GROUPED) pagent = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(pagent) + (size_t)pol * in.a.d.pstride);
            tc::tc_fence_after();
            __syncwarp();
#pragma unroll(W == 32 ? PIECES : 1)
            for (int k = 0; k < PIECES; ++k) {
                const int c = k / (32 / W), cell = 128 * c + r, c0 = 32 * half + W * (k % (32 / W));
                float v[W];
#pragma unroll
                for (int i = 0; i < W; ++i) v[i] = 0.f;
                if (got) {
                    uint32_t x0[W], x1[W];
                    const uint32_t at = tmem + lane_base + (uint32_t)(Cfg::AGENT_COL + Cfg::AGENT_N * c + c0);
                    tmem_cols(at, x0);
                    if (PL == 2) tmem_cols(at + 64, x1);
                    tc::tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < W; ++i) v[i] = PL == 2 ? __uint_as_float(x0[i]) + __uint_as_float(x1[i]) : __uint_as_float(x0[i]);
                }
                if (cell < C) {
                    float4* p = reinterpret_cast<float4*>(pagent + (size_t)cell * H + c0);
                    if (!first) {
#pragma unroll
                        for (int i = 0; i < W / 4; ++i) {
                            const float4 o = p[i];
                            v[4 * i] += o.x; v[4 * i + 1] += o.y; v[4 * i + 2] += o.z; v[4 * i + 3] += o.w;
                        }
                    }
#pragma unroll
                    for (int i = 0; i < W / 4; ++i) p[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                }
            }
            tc::tc_fence_before();
        };
        auto store_S = [&](size_t row, const float (&v)[32]) {  // 32 units of one row, two 16-bit planes
            uint32_t hi[16], lo[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                if (PREC == 1) {
                    __nv_bfloat16 h0, l0, h1, l1;
                    split_bf16(v[2 * i], h0, l0);
                    split_bf16(v[2 * i + 1], h1, l1);
                    hi[i] = pack_bf16(h0, h1);
                    lo[i] = pack_bf16(l0, l1);
                } else {
                    split2<0>(v[2 * i], v[2 * i + 1], hi[i], lo[i]);
                }
            }
            uint4* ph = reinterpret_cast<uint4*>(S_hi + row * H + 32 * half);
            uint4* pl = reinterpret_cast<uint4*>(S_lo + row * H + 32 * half);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                ph[i] = make_uint4(hi[4 * i], hi[4 * i + 1], hi[4 * i + 2], hi[4 * i + 3]);
                pl[i] = make_uint4(lo[4 * i], lo[4 * i + 1], lo[4 * i + 2], lo[4 * i + 3]);
            }
        };
        for (int u = xi; u < units && ok; u += nx) {
            const int env = (u % m_tiles) * BM + row_e, t1 = t_end(u);
            const bool have = env < B && row_dt < SP;
#pragma unroll
            for (int i = 0; i < 32; ++i) s_acc[i] = 0.f;
            for (int t = t_begin(u); t < t1; t += SP, ++g) {
                const int buf = g & 1, s = g % DST, hs = g % HST;
                if (LONG && g % Cfg::AGENT_FLUSH == Cfg::AGENT_FIRST) {  // a whole group of the agent plane
                    ok = tc::mbar_wait(&empty[(g - 1) % DST], (uint32_t)((g - 1) / DST) & 1u);
                    if (!ok) break;
                    drain_agent(std::integral_constant<int, 16>{}, g == Cfg::AGENT_FIRST, true);
                }
                const int cell = half == 0 && have && t + row_dt < t1 ? (int)b.tpos[(size_t)(t + row_dt) * B + env] : -1;
                ok = tc::mbar_wait(&tfull[buf], (uint32_t)(g >> 1) & 1u);
                if (!ok) break;
                tc::tc_fence_after();
                if (g > 0 && g % Cfg::FLUSH == 0) add_w2();  // (finished: w2done of the tile before was waited for)
                float x[32];
                read_pair((uint32_t)(Cfg::ACC_COL + Cfg::ACC_N * buf), Cfg::ACC_N > H, x);
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&tempty[buf]);
                ok = tc::mbar_wait(&hfull[hs], (uint32_t)(g / HST) & 1u);  // (the loads themselves, for this thread's own reads)
                if (!ok) break;
                uint32_t hi[16];
                uint32_t lo[16];
#pragma unroll
                for (int c = 0; c < 4; ++c) {  // 16-byte chunks of 8 units: gate, S, split
                    const uint4 gt = *reinterpret_cast<const uint4*>(sH + hs * Cfg::STAGE + r * 128 + (((4 * half + c) ^ (r & 7)) << 4));
                    const uint32_t gw[4] = {gt.x, gt.y, gt.z, gt.w};
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const int i = 8 * c + 2 * p;
                        const float v0 = rnd<PREC>((gw[p] & 0x00007FFFu) ? x[i] : 0.f);
                        const float v1 = rnd<PREC>((gw[p] & 0x7FFF0000u) ? x[i + 1] : 0.f);
                        s_acc[i] += v0;
                        s_acc[i + 1] += v1;
                        split2<PREC>(v0, v1, hi[i / 2], lo[i / 2]);
                    }
                }
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&hempty[hs]);
                ok = tc::mbar_wait(&w2done[s], (uint32_t)(g / DST) & 1u);
                if (ok && g >= 1) ok = tc::mbar_wait(&empty[(g - 1) % DST], (uint32_t)((g - 1) / DST) & 1u);  // the one-hot tile is free
                if (!ok) break;
                unsigned char* drow = sD + s * Cfg::STAGE + r * 128;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int off = ((4 * half + c) ^ (r & 7)) << 4;
                    *reinterpret_cast<uint4*>(drow + off) = make_uint4(hi[4 * c], hi[4 * c + 1], hi[4 * c + 2], hi[4 * c + 3]);
                    if (PL == 2) *reinterpret_cast<uint4*>(drow + BOX + off) = make_uint4(lo[4 * c], lo[4 * c + 1], lo[4 * c + 2], lo[4 * c + 3]);
                }
                if (prev_off >= 0) *reinterpret_cast<uint16_t*>(sO + prev_off) = 0;
                prev_off = -1;
                if (cell >= 0 && cell < 128 * NC) {
                    // element (k = row, m = cell) of the MN-major tile: byte k*128 + ((m/8) ^ (k%8))*16 + (m%8)*2 of its 64-cell box
                    prev_off = (cell >> 6) * BOX + r * 128 + ((((cell & 63) >> 3) ^ (r & 7)) << 4) + (cell & 7) * 2;
                    *reinterpret_cast<uint16_t*>(sO + prev_off) = (uint16_t)one16<PREC>();
                }
                tc::fence_proxy_async();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(tiles_full);
            }
            if (ok && SP == 1 && have) store_S((size_t)(u / m_tiles) * B + env, s_acc);
        }
        if (!ok && lane == 0) atomicOr(b.status, DEV_E_WAIT_TIMEOUT);
        bool got = ok && G > 0;
        if (got) got = tc::mbar_wait(&empty[(G - 1) % DST], (uint32_t)((G - 1) / DST) & 1u);  // the last MMAs; the stages are idle now
        if (!got && ok && G > 0 && lane == 0) atomicOr(b.status, DEV_E_WAIT_TIMEOUT);
        tc::tc_fence_after();
        __syncwarp();
        if (got) add_w2();
        // the lo half of dW2 (lanes 64..) and, where a tile holds several steps, S go through the idle stages
        float* const x_w2 = reinterpret_cast<float*>(sH);             // [64][64 + 4]
        float* const x_s = reinterpret_cast<float*>(sH + 2 * BOX);    // [128][64]
        if (PL == 2 && q >= 2) {
#pragma unroll
            for (int i = 0; i < 32; i += 4)
                *reinterpret_cast<float4*>(x_w2 + (r - 64) * 68 + 32 * half + i) = make_float4(w_acc[i], w_acc[i + 1], w_acc[i + 2], w_acc[i + 3]);
        }
        if (SP > 1) {
#pragma unroll
            for (int i = 0; i < 32; i += 4)
                *reinterpret_cast<float4*>(x_s + r * 64 + 32 * half + i) = make_float4(s_acc[i], s_acc[i + 1], s_acc[i + 2], s_acc[i + 3]);
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (q < 2) {
            float* dst = in.part_w2 + (size_t)xi * (H * H);
            if (GROUPED) dst = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(dst) + (size_t)pol * in.a.d.pstride);
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
                float4 v = make_float4(w_acc[i], w_acc[i + 1], w_acc[i + 2], w_acc[i + 3]);
                if (PL == 2) {
                    const float4 l = *reinterpret_cast<const float4*>(x_w2 + r * 68 + 32 * half + i);
                    v.x += l.x; v.y += l.y; v.z += l.z; v.w += l.w;
                }
                *reinterpret_cast<float4*>(dst + r * H + 32 * half + i) = v;
            }
        }
        if (SP > 1 && ok && xi < units && r < B) {  // (one unit per CTA: its slice of the steps) sum over the tile's steps, in step order
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
                for (int k = 1; k < SP; ++k) {
                    const float4 o = *reinterpret_cast<const float4*>(x_s + (k * TE + r) * 64 + 32 * half + i);
                    s_acc[i] += o.x; s_acc[i + 1] += o.y; s_acc[i + 2] += o.z; s_acc[i + 3] += o.w;
                }
            }
            store_S((size_t)(xi / m_tiles) * B + r, s_acc);
        }
        drain_agent(std::integral_constant<int, 32>{}, !LONG || G <= Cfg::AGENT_FIRST, got);  // the last group (or zeros)
    }
    tc::tc_fence_before();
    __syncthreads();
    if (wid == 1) tc::tmem_dealloc(tmem, Cfg::TMEM_COLS);
}

template <int PREC, int NC>
cudaError_t launch_t(const LearnArgs& a, int nx, float* part_w2, float* part_agent, size_t stride_agent, cudaStream_t s) {
    using Cfg = Back64Cfg<PREC, NC>;
    const Dims& d = a.d;
    const Buffers& b = a.b;
    constexpr bool bf = PREC == 1;
    const int sp = d.B <= Cfg::BM / 2 ? (Cfg::BM / d.B < a.T ? Cfg::BM / d.B : a.T) : 1;
    Back64Maps maps;
    memset(&maps, 0, sizeof(maps));
    const size_t RH = (size_t)d.B * d.Tmax * Cfg::H;
    const uint64_t ps = d.npol > 1 ? d.pstride : RH * 2;
    const uint16_t *h1 = reinterpret_cast<const uint16_t*>(b.h1), *dh2 = reinterpret_cast<const uint16_t*>(b.dh2);
    auto map = [&](CUtensorMap* m, const uint16_t* p, int envs, int pols) {
        return make_tensor_map_4d(m, p, (uint64_t)envs, (uint64_t)a.T, (uint64_t)pols, ps, (uint32_t)(sp > 1 ? envs : Cfg::BM), (uint32_t)sp, bf);
    };
    if (!map(&maps.h_hi, h1, d.B, d.npol) || !map(&maps.d_hi, dh2, d.B, d.npol)) return cudaErrorNotSupported;
    if (Cfg::PL == 2 && (!map(&maps.h_lo, h1 + RH, d.B, d.npol) || !map(&maps.d_lo, dh2 + RH, d.B, d.npol))) return cudaErrorNotSupported;
    if (d.npol > 1 && d.B_last != d.B) {
        const size_t off = (size_t)(d.npol - 1) * d.pstride / 2, RHl = (size_t)d.B_last * d.Tmax * Cfg::H;
        if (!map(&maps.lh_hi, h1 + off, d.B_last, 1) || !map(&maps.ld_hi, dh2 + off, d.B_last, 1)) return cudaErrorNotSupported;
        if (Cfg::PL == 2 && (!map(&maps.lh_lo, h1 + off + RHl, d.B_last, 1) || !map(&maps.ld_lo, dh2 + off + RHl, d.B_last, 1))) return cudaErrorNotSupported;
    }
    const Back64Args in{a, part_w2, part_agent, stride_agent, nx};
    // The restarts cost registers in the tile loop (1024 policies x 64 envs, 8 tiles a CTA: 191 -> 195 us), so launches without a CTA that
    // needs them do without.  Where they are taken: 131072 envs, 9 cells, T = 60 747 -> 740 us, 25 cells, T = 16 237 -> 229 us, 144
    // cells, T = 16 303 -> 311 us.
    const int m_tiles = sp > 1 ? 1 : (d.B + Cfg::BM - 1) / Cfg::BM, steps = (a.T + sp - 1) / sp;
    const bool many = (m_tiles * a.ts + nx - 1) / nx * ((steps + a.ts - 1) / a.ts) > Cfg::AGENT_FIRST;
    const dim3 grid(nx, 1, d.npol);
    if constexpr (PREC == 1) {
        if (d.npol > 1) return cudaErrorNotSupported;
        return launch<k_back64<1, NC, false, false>>(grid, Cfg::THREADS, Cfg::smem_bytes, s, maps, in);
    } else {
        if (d.npol > 1 && many) return launch<k_back64<0, NC, true, true>>(grid, Cfg::THREADS, Cfg::smem_bytes, s, maps, in);
        if (d.npol > 1) return launch<k_back64<0, NC, true, false>>(grid, Cfg::THREADS, Cfg::smem_bytes, s, maps, in);
        if (many) return launch<k_back64<0, NC, false, true>>(grid, Cfg::THREADS, Cfg::smem_bytes, s, maps, in);
        return launch<k_back64<0, NC, false, false>>(grid, Cfg::THREADS, Cfg::smem_bytes, s, maps, in);
    }
}

}  // namespace

// CTAs per policy (all policies together fill the GPU once where there are fewer than 148) and slices of the steps; one slice per
// CTA where a tile holds several steps.
void back64_shape(const Dims& d, int T, int* nx, int* ts) {
    const int cap = 148 / d.npol > 0 ? 148 / d.npol : 1;
    const int sp = d.B <= 64 ? (128 / d.B < T ? 128 / d.B : T) : 1, m_tiles = sp > 1 ? 1 : (d.B + 127) / 128, steps = (T + sp - 1) / sp;
    int most = most_slices(m_tiles, cap);
    if (sp > 1 && most > cap) most = cap;
    *ts = slices_for(m_tiles, cap, steps, most);
    const int units = m_tiles * *ts;
    *nx = units < cap ? units : cap;
}

// a.ts slices and nx CTAs per policy from back64_shape; partial x of dW2 goes to part_w2[x * 4096], of the agent plane to
// part_agent[x * stride_agent].
cudaError_t launch_back64(const LearnArgs& a, int prec, int nx, float* part_w2, float* part_agent, size_t stride_agent, cudaStream_t s) {
    if (prec == 1) return a.d.C > 128 ? launch_t<1, 2>(a, nx, part_w2, part_agent, stride_agent, s) : launch_t<1, 1>(a, nx, part_w2, part_agent, stride_agent, s);
    return a.d.C > 128 ? launch_t<0, 2>(a, nx, part_w2, part_agent, stride_agent, s) : launch_t<0, 1>(a, nx, part_w2, part_agent, stride_agent, s);
}

}  // namespace anakin
