// The whole backward pass above the first layer at hidden width 128 in one tcgen05 kernel: softmax, losses and output gradients
// from the saved head outputs, dWh, db2, dbh, dh2 = (dOut Wh^T) gated by h2 > 0, dW2 = h1^T dh2, dh1 = (dh2 W2^T) gated by h1 > 0,
// S = sum over t of dh1, and the agent plane of dW1 = onehot(pos)^T dh1 (the update half of the Anakin minimal unit, Podracer paper,
// Section 3.1; Figure 2, top).  h1 and h2 of a row are fetched once, 8 bytes a hidden unit in fp32 workloads; dh2 and dh1 never
// leave the chip.
//
// A tile is 64 envs of one step.  The dh1 product is taken transposed, dh1^T[unit][env] = W2[unit][:] . dh2[env][:], with W2 (both
// 16-bit planes) in TENSOR memory as the A operand; the epilogue writes the gated, split dh1^T back over the accumulator it came from
// (sixteen columns of fp32 = eight of hi pairs and eight of lo pairs), where it is the A operand of the agent-plane product.  One
// 128-byte-swizzled box of dh2 [env][64 units] serves as the K-major operand of dh1 (k = unit) and as the MN-major one of dW2 (k = env).
//   warp 0       loads: W2 once; per tile h1 (TMA boxes), h2 and the layer-1 gates (bulk copies)
//   warp 1       tcgen05.mma issuer: dW2 and dh1 of a tile, then the agent plane of the tile before
//   warps 2, 3   lane = row of a tile: softmax, loss terms, output gradients
//   warps 4-11   builders, thread = (four units, eight rows): dh2 into its operand box, running sums of dWh and db2; every GROUP tiles
//                they add the dW2 accumulator to this CTA's partial
//   warps 12-19  epilogue, thread = (unit, half of the envs): tcgen05.ld, gate, S +=, 16-bit split, tcgen05.st; the one-hot rows
// Tensor memory: [W2 planes | two dh1 accumulators | dW2 | agent plane] = 128 + 128 + 128 + 128 columns (128 cells at most).
// The tensor core rounds toward zero, so dW2 restarts its accumulator every 3584 rows and the agent plane every 768 MMAs; the
// groups are added with round-to-nearest.
// Every wait is bounded; a timeout raises DEV_E_WAIT_TIMEOUT and the CTA unwinds.
//
// What bounds it: no single thing.  A tile takes about 4200 clocks; HBM is half busy; the tensor pipe is taken for 2600 of them (20 MMAs
// with N = 128 at 64 clocks, and the 24 of dh1, N = 64, at the 55 that one takes instead of 32; its counter, of useful clocks, says 47 %),
// and the issuer, the builders and the epilogue are each at work for 3200 (with the builders' loop cut to an
// eighth, or most MMAs left out, 2.25 ms become 2.1).  B200, 131072 envs, 8 x 8, T = 64, fp32: the two kernels this one replaces (heads with
// dW2; dh1 with the agent plane; dh2 out to HBM and back) 2.18 + 1.19 ms, this one 2.25; the whole iteration 5.94 -> 4.95 ms.  2500 envs,
// 9 x 9, T = 24: 26 + 19 -> 33 us; rollout and four PPO epochs 420 -> 367 us.  Tried: sixteen builder warps 2.39 ms (fewer registers);
// 24 warps with more row warps and a loader for h1 2.30; an L2 prefetch two, four or eight tiles ahead 2.53, 2.62 and 2.81; scalar
// products in the builders 2.56.  The roles run side by side, so their code shares one instruction cache: with the row warps' code
// twice and every loop unrolled the warps waited for instructions (2.53), hence the plain loops in the issuer.
#include <cstring>

#include "tc_common.cuh"

namespace anakin {

namespace {

template <int PREC>
struct Back128Cfg {
    static constexpr int H = 128, BM = 64;
    static constexpr int PL = PREC == 1 ? 1 : 2;
    static constexpr int BUILD_WARPS = 8, EPI_WARPS = 8, FIRST_ROW = 2, FIRST_BUILD = 4, FIRST_EPI = FIRST_BUILD + BUILD_WARPS, THREADS = 32 * (FIRST_EPI + EPI_WARPS);
    // Registers a thread: 96 at launch (20 warps), then so many for the first four warps, the builders and the epilogue.  setmaxnreg.inc
    // may draw on no more than the block was launched with, and .dec may not raise (an illegal instruction).
    static constexpr int REGS = 96, REGS_FIRST = 72, REGS_BUILD = 88, REGS_EPI = 112;
    static_assert(REGS_FIRST <= REGS && REGS_BUILD <= REGS && REGS_EPI >= REGS, "directions of the changes");
    static_assert(FIRST_BUILD * REGS_FIRST + BUILD_WARPS * REGS_BUILD + EPI_WARPS * REGS_EPI <= (FIRST_EPI + EPI_WARPS) * REGS, "registers of the block");
    static constexpr int BOX = BM * 128;              // 64 rows x 64 16-bit elements
    static constexpr int TILE = PL * 2 * BOX;         // one operand of a tile: [plane][64-unit box]
    static constexpr int HST = PREC == 1 ? 4 : 2;     // h1 ring
    static constexpr int P_TILE = BM * H * 4, PST = PREC == 1 ? 3 : 2;  // h2 ring
    static constexpr int O_TILE = 2 * BOX;            // one-hot: 64 k-rows (envs) x 128 cells, MN-major
    static constexpr int G_TILE = BM * (H / 8), GST = 4;  // layer-1 gates
    static constexpr int DO_ROW = 32, DO_TILE = BM * DO_ROW;  // output gradients of a row
    static constexpr int W_BOX = H * 128;             // W2: 128 rows x 64 k, staged where dh2 goes later
    static_assert(PL * 2 * W_BOX == 2 * TILE, "W2 fills the two dh2 tiles");
    static constexpr int W_COL = 0, ACC_COL = PL * H / 2, W2_COL = ACC_COL + 2 * BM, AGENT_COL = W2_COL + H, TMEM_COLS = 512;
    static_assert(AGENT_COL + 128 <= TMEM_COLS, "tensor memory");
    // Tiles of a dW2 accumulator.  A CTA's tiles are consecutive steps of the same envs, whose products partly have one sign, so that an
    // accumulator loses more than over as many rows from all over the batch: 2-norm of the error of 20,000 envs, 8 x 8, T = 64 1.9e-5 with 64
    // tiles, 1.5e-5 with 56 (1.7e-5 as a sum of the heads kernel, whose rows are those of one step).  131,072 envs 4.79 / 4.80 ms an
    // iteration, 20,000 1.03 / 1.02; with 32 tiles 9e-6, 4.89 and 1.04.
    static constexpr int GROUP = PREC == 1 ? (1 << 30) : 56;
    static constexpr int AGENT_GROUP = PREC == 1 ? (1 << 30) : 96;   // ... of an agent-plane accumulator
    static constexpr int BARS = 512;
    static constexpr size_t smem_bytes = (size_t)HST * TILE + PST * P_TILE + 2 * TILE + O_TILE + GST * G_TILE + 2 * DO_TILE + BARS + 1024;
    static_assert(smem_bytes <= 232448, "227 KB per CTA");
};

struct Back128Maps {
    CUtensorMap h_hi, h_lo, w_hi, w_lo;
};

template <int PREC>
__global__ void __launch_bounds__(Back128Cfg<PREC>::THREADS, 1)
    k_back128(const __grid_constant__ Back128Maps maps, const __grid_constant__ LearnArgs a, float* part_w2, float* part_agent, size_t stride_agent) {
    using Cfg = Back128Cfg<PREC>;
    constexpr int H = Cfg::H, BM = Cfg::BM, PL = Cfg::PL, HST = Cfg::HST, PST = Cfg::PST, GST = Cfg::GST, BOX = Cfg::BOX, TILE = Cfg::TILE;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sH = base;                          // [HST] h1 planes
    unsigned char* sD = sH + HST * TILE;               // [2] dh2 planes (W2 on its way to tensor memory first)
    unsigned char* sO = sD + 2 * TILE;                 // one-hot tile
    unsigned char* sP = sO + Cfg::O_TILE;              // [PST] h2 rows
    unsigned char* sG = sP + PST * Cfg::P_TILE;        // [GST] layer-1 gates
    unsigned char* sQ = sG + GST * Cfg::G_TILE;          // [2] output gradients
    uint64_t* bars = (uint64_t*)(sQ + 2 * Cfg::DO_TILE);
    uint64_t* hfull = bars;                // [HST] h1 landed
    uint64_t* hempty = hfull + HST;        // [HST] dW2 has read it (commit)
    uint64_t* pfull = hempty + HST;        // [PST] h2 landed
    uint64_t* pempty = pfull + PST;        // [PST] ... and read (the builder warps arrive)
    uint64_t* gfull = pempty + PST;        // [GST] gates landed
    uint64_t* gempty = gfull + GST;        // [GST] ... and read (the epilogue warps arrive)
    uint64_t* qfull = gempty + GST;         // [2] output gradients written (the row warps arrive)
    uint64_t* qempty = qfull + 2;          // [2] ... and read (the builder warps arrive)
    uint64_t* dfull = qempty + 2;          // [2] dh2 written (the builder warps arrive)
    uint64_t* mdone = dfull + 2;           // [2] dW2 and dh1 of a tile have finished
    uint64_t* tiles_full = mdone + 2;      // dh1^T and the one-hot of a tile written (the epilogue warps arrive)
    uint64_t* tiles_free = tiles_full + 1; // the agent MMAs of a tile have finished
    uint64_t* wstage = tiles_free + 1;     // W2 landed in its staging boxes
    uint64_t* wfull = wstage + 1;          // ... and is in tensor memory (the epilogue warps arrive)
    uint32_t* tmem_slot = (uint32_t*)(wfull + 1);
    float* s_fin = (float*)(tmem_slot + 1);  // [8] sums of the second row warp
    static_assert((2 * HST + 2 * PST + 2 * GST + 14) * 8 + 4 + 32 <= Cfg::BARS, "room for the barriers");

    const Dims& d = a.d;
    const Buffers& b = a.b;
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const int B = d.B, T = a.T, C = d.C;
    const int m_tiles = (B + BM - 1) / BM, tl = (T + a.ts - 1) / a.ts, units = m_tiles * a.ts;
    const int xi = blockIdx.x, nx = gridDim.x;
    int* status = b.status;
    // this CTA's units u = xi, xi + nx, ...: 64 envs, a slice of the steps
    auto t_begin = [&](int u) { return min((u / m_tiles) * tl, T); };
    auto t_end = [&](int u) { return min((u / m_tiles) * tl + tl, T); };

    if (tid == 0) {
        for (int s = 0; s < HST; ++s) { tc::mbar_init(&hfull[s], 1); tc::mbar_init(&hempty[s], 1); }
        for (int s = 0; s < PST; ++s) { tc::mbar_init(&pfull[s], 1); tc::mbar_init(&pempty[s], Cfg::BUILD_WARPS); }
        for (int s = 0; s < GST; ++s) { tc::mbar_init(&gfull[s], 1); tc::mbar_init(&gempty[s], Cfg::EPI_WARPS); }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&qfull[i], 2);
            tc::mbar_init(&qempty[i], Cfg::BUILD_WARPS);
            tc::mbar_init(&dfull[i], Cfg::BUILD_WARPS);
            tc::mbar_init(&mdone[i], 1);
        }
        tc::mbar_init(tiles_full, Cfg::EPI_WARPS);
        tc::mbar_init(tiles_free, 1);
        tc::mbar_init(wstage, 1);
        tc::mbar_init(wfull, Cfg::EPI_WARPS);
        tc::mbar_fence_init();
    }
    if (wid == 1) tc::tmem_alloc(tmem_slot, Cfg::TMEM_COLS);
    // the one-hot tile starts all zero (a tile clears the elements of the one before); so do the h2 tiles: rows past the last one
    // are never filled, and their products with zero gradients must be zero
    for (int i = tid; i < (Cfg::O_TILE + PST * Cfg::P_TILE) / 16; i += Cfg::THREADS) reinterpret_cast<uint4*>(sO)[i] = make_uint4(0u, 0u, 0u, 0u);
    tc::fence_proxy_async();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (tid == 0) {
        tc::prefetch_map(&maps.w_hi);
        tc::prefetch_map(&maps.h_hi);
        if (PL == 2) { tc::prefetch_map(&maps.w_lo); tc::prefetch_map(&maps.h_lo); }
    }
    pdl_wait();  // (the set-up above runs under the predecessor's tail)
    int G = 0;  // tiles of this CTA
    for (int u = xi; u < units; u += nx) G += t_end(u) - t_begin(u);
    bool ok = true;

    if (wid < Cfg::FIRST_BUILD) {
        tc::regs_dec<Cfg::REGS_FIRST>();
        if (wid == 0) {
            if (lane == 0) {  // ---- loads
                tc::mbar_expect_tx(wstage, PL * 2 * Cfg::W_BOX);
#pragma unroll
                for (int pl = 0; pl < PL; ++pl)
#pragma unroll
                    for (int kc = 0; kc < 2; ++kc) tc::tma_load_2d(sD + (pl * 2 + kc) * Cfg::W_BOX, pl ? &maps.w_lo : &maps.w_hi, wstage, kc * 64, 0);
                const size_t R = (size_t)B * T;
                int g = 0;
                for (int u = xi; u < units && ok; u += nx) {
                    const int env0 = (u % m_tiles) * BM, t1 = t_end(u);
                    for (int t = t_begin(u); t < t1; ++t, ++g) {
                        // rows t*B + env0 .. +63: those past the batch end are the next step's and carry zero gradients
                        const size_t row = (size_t)t * B + env0;
                        const int ps = g % PST, hs = g % HST, gs = g % GST;
                        const uint32_t n = (uint32_t)min(R - row, (size_t)BM);
                        if (g >= PST) ok = tc::mbar_wait(&pempty[ps], (uint32_t)(g / PST - 1) & 1u);
                        if (!ok) break;
                        tc::mbar_expect_tx(&pfull[ps], n * H * 4);
                        tc::bulk_load(sP + ps * Cfg::P_TILE, b.h2 + row * H, &pfull[ps], n * H * 4);
                        if (g >= HST) ok = tc::mbar_wait(&hempty[hs], (uint32_t)(g / HST - 1) & 1u);
                        if (!ok) break;
                        tc::mbar_expect_tx(&hfull[hs], TILE);
#pragma unroll
                        for (int bx = 0; bx < 2; ++bx) {  // (TMA fills rows past the last one with zeros)
                            tc::tma_load_2d(sH + hs * TILE + bx * BOX, &maps.h_hi, &hfull[hs], 64 * bx, (int)row);
                            if (PL == 2) tc::tma_load_2d(sH + hs * TILE + (2 + bx) * BOX, &maps.h_lo, &hfull[hs], 64 * bx, (int)row);
                        }
                        if (g >= GST) ok = tc::mbar_wait(&gempty[gs], (uint32_t)(g / GST - 1) & 1u);
                        if (!ok) break;
                        tc::mbar_expect_tx(&gfull[gs], n * (H / 8));
                        tc::bulk_load(sG + gs * Cfg::G_TILE, b.gate1 + row * (H / 8), &gfull[gs], n * (H / 8));
                    }
                }
                pdl_trigger();  // (the last loads are on their way)
                if (!ok) atomicOr(status, DEV_E_WAIT_TIMEOUT);
            }
        } else if (wid == 1) {  // ---- MMA issuer: the whole warp walks the loop, one elected lane issues
            const uint32_t id_w2 = tc::umma_idesc<PREC>(128, H, true, true), id_dh1 = tc::umma_idesc<PREC>(128, BM, false, false);
            const uint32_t id_agent = tc::umma_idesc<PREC>(128, 128, false, true);
            auto agent_mma = [&](int v) {
                ok = tc::warp_all(tc::mbar_wait(tiles_full, (uint32_t)v & 1u));
                if (!ok) return;
                tc::tc_fence_after();
                if (tc::elect_one()) {
                    const uint32_t at = tmem + (uint32_t)(Cfg::ACC_COL + BM * (v & 1));
#pragma unroll 1
                    for (int k16 = 0; k16 < BM / 16; ++k16) {  // 16 env rows = 2048 bytes further, cells 64.. one box further
                        const uint64_t od = tc::umma_desc(sO + k16 * 2048, BOX, 1024);
#pragma unroll
                        for (int pl = 0; pl < PL; ++pl)
                            tc::umma_ta(tmem + (uint32_t)Cfg::AGENT_COL, at + (uint32_t)(16 * k16 + 8 * pl), od, id_agent,
                                        v % Cfg::AGENT_GROUP > 0 || pl > 0 || k16 > 0);  // (a group's first MMA restarts the sum)
                    }
                    tc::umma_commit(tiles_free);
                }
                __syncwarp();
            };
            ok = tc::warp_all(tc::mbar_wait(wfull, 0));
            for (int g = 0; g < G && ok; ++g) {
                const int hs = g % HST, buf = g & 1;
                ok = tc::mbar_wait(&dfull[buf], (uint32_t)(g >> 1) & 1u);
                ok = tc::warp_all(ok && tc::mbar_wait(&hfull[hs], (uint32_t)(g / HST) & 1u));
                if (!ok) break;
                tc::tc_fence_after();
                const unsigned char* sh = sH + hs * TILE;
                const unsigned char* sd = sD + buf * TILE;
                if (tc::elect_one()) {
                    // dW2[i][j] += sum over the 64 rows of h1[r][i] dh2[r][j]: both MN-major, 16 rows = 2048 bytes further
                    const uint32_t acc = tmem + (uint32_t)Cfg::W2_COL;
#pragma unroll 1
                    for (int k16 = 0; k16 < BM / 16; ++k16) {
                        const uint64_t h_hi = tc::umma_desc(sh + k16 * 2048, BOX, 1024), d_hi = tc::umma_desc(sd + k16 * 2048, BOX, 1024);
                        uint32_t accum = (g % Cfg::GROUP > 0 || k16 > 0) ? 1u : 0u;
                        if (PL == 2) {
                            tc::umma(acc, tc::umma_desc(sh + 2 * BOX + k16 * 2048, BOX, 1024), d_hi, id_w2, accum);
                            tc::umma(acc, h_hi, tc::umma_desc(sd + 2 * BOX + k16 * 2048, BOX, 1024), id_w2, 1u);
                            accum = 1u;
                        }
                        tc::umma(acc, h_hi, d_hi, id_w2, accum);
                    }
                    tc::umma_commit(&hempty[hs]);
                }
                __syncwarp();
                // the accumulator of two tiles ago, with the dh1^T that lies over it, has been used
                if (g >= 2) ok = tc::warp_all(tc::mbar_wait(tiles_free, (uint32_t)g & 1u));
                if (!ok) break;
                tc::tc_fence_after();
                if (tc::elect_one()) {
                    const uint32_t acc = tmem + (uint32_t)(Cfg::ACC_COL + BM * buf);
#pragma unroll 1
                    for (int kc = 0; kc < 2; ++kc)
#pragma unroll 1
                        for (int k16 = 0; k16 < 4; ++k16) {
                            // W2 in tensor memory: 16 k = 8 columns; dh2 (K-major): 16 k = 32 bytes along the swizzled rows
                            const uint32_t w_hi = tmem + (uint32_t)(Cfg::W_COL + kc * 32 + k16 * 8);
                            const uint64_t d_hi = tc::umma_desc(sd + kc * BOX + k16 * 32, 16, 1024);
                            tc::umma_ta(acc, w_hi, d_hi, id_dh1, kc > 0 || k16 > 0);
                            if (PL == 2) {
                                tc::umma_ta(acc, w_hi + (uint32_t)(H / 2), d_hi, id_dh1, 1u);
                                tc::umma_ta(acc, w_hi, tc::umma_desc(sd + (2 + kc) * BOX + k16 * 32, 16, 1024), id_dh1, 1u);
                            }
                        }
                    tc::umma_commit(&mdone[buf]);
                }
                __syncwarp();
                if (g >= 1) agent_mma(g - 1);  // queued behind this tile's products: the tensor pipe stays busy
            }
            if (ok && G > 0) agent_mma(G - 1);
            if (!ok && lane == 0) atomicOr(status, DEV_E_WAIT_TIMEOUT);
        } else {
            // ---- row warps: lane = row of a tile; a row's loads are requested a tile ahead
            const int rr = 32 * (wid - Cfg::FIRST_ROW) + lane;
            const float invR = a.gscale / (float)((size_t)B * T);  // output gradients are carried times gscale
            float a_bh[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
            float l_pg = 0.f, l_v = 0.f, l_ent = 0.f;
            struct RowIn { float4 o4; float v, adv, ret, lpo; int act; bool ok; };
            int lu = xi, lt = t_begin(xi);  // the tile whose rows are requested next
            auto row_load = [&](RowIn& in) {
                while (lu < units && lt >= t_end(lu)) { lu += nx; lt = t_begin(lu); }
                const int env = (lu % m_tiles) * BM + rr;
                in.ok = lu < units && env < B;
                in.o4 = make_float4(0.f, 0.f, 0.f, 0.f);
                in.v = in.adv = in.ret = in.lpo = 0.f;
                in.act = 0;
                if (in.ok) {
                    const size_t i = (size_t)lt * B + env;
                    in.o4 = *reinterpret_cast<const float4*>(b.out5 + i * 8);
                    in.v = b.out5[i * 8 + 4];
                    in.adv = b.adv[i];
                    in.lpo = a.ppo_clip > 0.f ? b.tlogp[i] : 0.f;
                    in.ret = b.ret[i];
                    in.act = b.tact[i];
                }
                ++lt;
            };
            auto row_out = [&](const RowIn& in, int g) {
                const int buf = g & 1;
                float dO[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
                if (in.ok) {
                    const float o[4] = {in.o4.x, in.o4.y, in.o4.z, in.o4.w};
                    const float mx = fmaxf(fmaxf(o[0], o[1]), fmaxf(o[2], o[3]));
                    float ex[4], Z = 0.f;
#pragma unroll
                    for (int c = 0; c < 4; ++c) { ex[c] = expf(o[c] - mx); Z += ex[c]; }
                    const float logZ = logf(Z);
                    float p[4], lp[4], ent = 0.f;
#pragma unroll
                    for (int c = 0; c < 4; ++c) { p[c] = ex[c] / Z; lp[c] = (o[c] - mx) - logZ; ent -= p[c] * lp[c]; }
                    const float A = in.adv, err = in.v - in.ret;
                    const float pf = policy_term(A, in.act == 0 ? lp[0] : in.act == 1 ? lp[1] : in.act == 2 ? lp[2] : lp[3], in.lpo, a.ppo_clip, l_pg);
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        dO[c] = rnd<PREC>((-A * pf * ((c == in.act ? 1.f : 0.f) - p[c]) + a.c_e * p[c] * (lp[c] + ent)) * invR);
                    dO[4] = rnd<PREC>(2.f * a.c_v * err * invR);
                    l_v += err * err;
                    l_ent += ent;
#pragma unroll
                    for (int c = 0; c < 5; ++c) a_bh[c] += dO[c];
                }
                if (g >= 2) ok = tc::mbar_wait(&qempty[buf], (uint32_t)((g >> 1) - 1) & 1u);
                float4* q4 = reinterpret_cast<float4*>(sQ + buf * Cfg::DO_TILE + rr * Cfg::DO_ROW);
                q4[0] = make_float4(dO[0], dO[1], dO[2], dO[3]);
                q4[1].x = dO[4];
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&qfull[buf]);
            };
            RowIn in;
            row_load(in);
#pragma unroll 1
            for (int g = 0; g < G && ok; ++g) {
                row_out(in, g);
                row_load(in);  // (used a tile on; moved through a second set of registers it would be waited for here)
            }
            // dbh and the loss terms of this CTA: a fixed shuffle tree over the lanes, then the second warp's sums on top of the first's
            float vals[8] = {a_bh[0], a_bh[1], a_bh[2], a_bh[3], a_bh[4], l_pg, l_v, l_ent};
#pragma unroll
            for (int c = 0; c < 8; ++c)
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) vals[c] += __shfl_xor_sync(0xFFFFFFFFu, vals[c], off);
            if (wid > Cfg::FIRST_ROW && lane == 0) {
#pragma unroll
                for (int c = 0; c < 8; ++c) s_fin[c] = vals[c];
            }
            asm volatile("bar.sync 2, 64;" ::: "memory");
            if (wid == Cfg::FIRST_ROW) {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    if (lane == c) {
                        const float v = vals[c] + s_fin[c];
                        if (c < 5) a.part_small[(size_t)xi * a.small_stride + (size_t)H * 6 + c] = v;
                        else b.loss_part[(size_t)xi * 4 + (c - 5)] = v;
                    }
                }
            }
            if (!ok && lane == 0) atomicOr(status, DEV_E_WAIT_TIMEOUT);
        }
    } else if (wid < Cfg::FIRST_EPI) {
        tc::regs_dec<Cfg::REGS_BUILD>();
        // ---- builders: a warp takes eight rows of a tile, a lane four units (two register pairs) of each
        const int rg = wid - Cfg::FIRST_BUILD, u0 = 4 * lane;
        uint64_t wh[2][5], a_wh[2][5], a_b2[2];
        {
            const float* w = b.theta_c + d.oWh + (size_t)u0 * 5;
#pragma unroll
            for (int p = 0; p < 2; ++p) {
#pragma unroll
                for (int c = 0; c < 5; ++c) { wh[p][c] = pack_f32x2(__ldg(w + 10 * p + c), __ldg(w + 10 * p + 5 + c)); a_wh[p][c] = 0ull; }
                a_b2[p] = 0ull;
            }
        }
        // This CTA's partial of dW2: accumulator lane = row of dW2, column = its column; a warp reads lane quarter wid % 4 and one half
        // of the columns.  The first group is written, every later one added to what this same thread wrote.
        auto dw2_out = [&](bool first, bool got) {
            tc::tc_fence_after();
            __syncwarp();
            const int q = wid & 3, col = 64 * ((wid - Cfg::FIRST_BUILD) >> 2);
            float* const row = part_w2 + (size_t)xi * H * H + (size_t)(32 * q + lane) * H + col;
#pragma unroll 1
            for (int c0 = 0; c0 < 64; c0 += 16) {
                uint32_t r[16];
                if (got) {
                    tc::tmem_ld16_nowait(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(Cfg::W2_COL + col + c0), r);
                    tc::tmem_ld_wait();
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i) r[i] = 0u;
                }
                float4* dst = reinterpret_cast<float4*>(row + c0);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float4 v = make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]), __uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3]));
                    if (!first) {
                        const float4 o = dst[i];
                        v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
                    }
                    dst[i] = v;
                }
            }
            tc::tc_fence_before();
        };
        // four units' place in row k of the MN-major (and K-major) tile: byte k*128 + ((unit/8) ^ (k%8))*16 + (unit%8)*2 of box unit/64
        const int tcol = (lane >> 4) * BOX + (lane & 1) * 8, chunk = (lane & 15) >> 1;
        ok = tc::mbar_wait(wfull, 0);  // (W2 came through the dh2 tiles)
        for (int g = 0; g < G && ok; ++g) {
            const int buf = g & 1, ps = g % PST;
            ok = tc::mbar_wait(&qfull[buf], (uint32_t)(g >> 1) & 1u);
            if (ok && g >= 2) ok = tc::mbar_wait(&mdone[buf], (uint32_t)((g >> 1) - 1) & 1u);  // the products of two tiles ago have read this tile's place
            if (ok) ok = tc::mbar_wait(&pfull[ps], (uint32_t)(g / PST) & 1u);
            if (!ok) break;
            const uint32_t h2t = tc::lds_base(sP + ps * Cfg::P_TILE + (rg * 8) * H * 4 + u0 * 4);
            const uint32_t qt = tc::lds_base(sQ + buf * Cfg::DO_TILE + (rg * 8) * Cfg::DO_ROW);
            unsigned char* out = sD + buf * TILE + tcol + (rg * 8) * 128;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                uint64_t hp[2], dd[5];
                tc::lds_2b64(h2t + r * H * 4, hp[0], hp[1]);
                const float4 d4 = tc::lds_f4(qt + r * Cfg::DO_ROW);
                const float d5 = tc::lds_f1(qt + r * Cfg::DO_ROW + 16);
                dd[0] = pack_f32x2(d4.x, d4.x); dd[1] = pack_f32x2(d4.y, d4.y); dd[2] = pack_f32x2(d4.z, d4.z); dd[3] = pack_f32x2(d4.w, d4.w);
                dd[4] = pack_f32x2(d5, d5);
                uint32_t hi[2], lo[2];
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    uint64_t v = mul_f32x2(dd[0], wh[p][0]);
#pragma unroll
                    for (int c = 1; c < 5; ++c) v = fma_f32x2(dd[c], wh[p][c], v);
#pragma unroll
                    for (int c = 0; c < 5; ++c) a_wh[p][c] = fma_f32x2(hp[p], dd[c], a_wh[p][c]);
                    const float2 hv = unpack_f32x2(hp[p]), x = unpack_f32x2(v);
                    const float x0 = rnd<PREC>(hv.x > 0.f ? x.x : 0.f), x1 = rnd<PREC>(hv.y > 0.f ? x.y : 0.f);
                    a_b2[p] = add_f32x2(a_b2[p], pack_f32x2(x0, x1));
                    split2<PREC>(x0, x1, hi[p], lo[p]);
                }
                unsigned char* o = out + r * 128 + ((chunk ^ r) << 4);  // (the row's place among eight is r)
                *reinterpret_cast<uint2*>(o) = make_uint2(hi[0], hi[1]);
                if (PL == 2) *reinterpret_cast<uint2*>(o + 2 * BOX) = make_uint2(lo[0], lo[1]);
            }
            // after a group's last tile the accumulator goes to this CTA's partial, before any MMA of the next tile is issued
            if (g % Cfg::GROUP == 0 && g > 0) {
                ok = tc::mbar_wait(&mdone[(g - 1) & 1], (uint32_t)((g - 1) >> 1) & 1u);
                if (!ok) break;
                dw2_out(g == Cfg::GROUP, true);
            }
            tc::fence_proxy_async();  // generic-proxy stores -> visible to the tensor core
            __syncwarp();
            if (lane == 0) {
                tc::mbar_arrive(&dfull[buf]);
                tc::mbar_arrive(&pempty[ps]);
                tc::mbar_arrive(&qempty[buf]);
            }
        }
        // ---- this CTA's dWh and db2: the row groups are added, in order, through the idle h2 ring
        {
            uint64_t* red = reinterpret_cast<uint64_t*>(sP);  // [row group 1..7][pair of a lane][6][32]
            asm volatile("bar.sync 1, 256;" ::: "memory");
            if (rg > 0) {
#pragma unroll
                for (int p = 0; p < 2; ++p) {
#pragma unroll
                    for (int c = 0; c < 5; ++c) red[(((rg - 1) * 2 + p) * 6 + c) * 32 + lane] = a_wh[p][c];
                    red[(((rg - 1) * 2 + p) * 6 + 5) * 32 + lane] = a_b2[p];
                }
            }
            asm volatile("bar.sync 1, 256;" ::: "memory");
            if (rg == 0) {
                float* part = a.part_small + (size_t)xi * a.small_stride;
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    for (int q = 0; q < Cfg::BUILD_WARPS - 1; ++q) {
#pragma unroll
                        for (int c = 0; c < 5; ++c) a_wh[p][c] = add_f32x2(a_wh[p][c], red[((q * 2 + p) * 6 + c) * 32 + lane]);
                        a_b2[p] = add_f32x2(a_b2[p], red[((q * 2 + p) * 6 + 5) * 32 + lane]);
                    }
#pragma unroll
                    for (int c = 0; c < 5; ++c) {
                        const float2 v = unpack_f32x2(a_wh[p][c]);
                        part[(size_t)(u0 + 2 * p) * 5 + c] = v.x;
                        part[(size_t)(u0 + 2 * p + 1) * 5 + c] = v.y;
                    }
                    *reinterpret_cast<float2*>(part + (size_t)H * 5 + u0 + 2 * p) = unpack_f32x2(a_b2[p]);
                }
            }
        }
        bool got = ok && G > 0;
        if (got) got = tc::mbar_wait(&mdone[(G - 1) & 1], (uint32_t)((G - 1) >> 1) & 1u);
        if (!got && G > 0 && lane == 0) atomicOr(status, DEV_E_WAIT_TIMEOUT);
        dw2_out(PREC == 1 || G <= Cfg::GROUP, got);
    } else {
        tc::regs_inc<Cfg::REGS_EPI>();
        // ---- epilogue: thread = hidden unit j (accumulator lane) x 32 of the tile's 64 envs
        const int q = wid & 3, j = 32 * q + lane, half = (wid - Cfg::FIRST_EPI) >> 2;
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        // W2 into tensor memory: row j = lane j, two k per column, the hi plane, then the lo plane.  Its boxes of 64 k have their 16-byte
        // pieces permuted by row % 8.
        if ((ok = tc::mbar_wait(wstage, 0))) {
#pragma unroll 1
            for (int pl = 0; pl < PL; ++pl) {
                const unsigned char* row = sD + (pl * 2 + half) * Cfg::W_BOX + j * 128;
                uint32_t r[32];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint4 v = *reinterpret_cast<const uint4*>(row + ((c ^ (j & 7)) << 4));
                    r[4 * c] = v.x; r[4 * c + 1] = v.y; r[4 * c + 2] = v.z; r[4 * c + 3] = v.w;
                }
                tc::tmem_st32(tmem + lane_base + (uint32_t)(Cfg::W_COL + pl * (H / 2) + half * 32), r);
            }
        }
        tc::tmem_st_wait();
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(wfull);
        float* const part = part_agent + (size_t)xi * stride_agent + j;
        // The agent accumulator (lane = unit, column = cell) into this CTA's partial, as the builders do with dW2.  The MMAs of the tiles so
        // far have been waited for; no other is issued before this warp's next arrival on tiles_full.
        auto drain_agent = [&](bool first, bool got) {
            tc::tc_fence_after();
            __syncwarp();
#pragma unroll 1
            for (int c0 = 64 * half; c0 < 64 * half + 64 && c0 < C; c0 += 16) {
                float* const p = part + (size_t)c0 * H;
                uint32_t r[16];
                if (got) {
                    tc::tmem_ld16_nowait(tmem + lane_base + (uint32_t)(Cfg::AGENT_COL + c0), r);
                    tc::tmem_ld_wait();
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i) r[i] = 0u;
                }
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    if (c0 + i < C) p[(size_t)i * H] = (first ? 0.f : p[(size_t)i * H]) + __uint_as_float(r[i]);
            }
            tc::tc_fence_before();
        };
        int prev_off = -1;  // byte offset of the one-hot element this thread set for the tile before
        int g = 0;
        for (int u = xi; u < units && ok; u += nx) {
            const int env0 = (u % m_tiles) * BM, t1 = t_end(u);
            const int nvalid = min(32, max(0, B - env0 - 32 * half));  // envs of this thread's half that exist
            const uint32_t valid = nvalid >= 32 ? 0xFFFFFFFFu : (1u << nvalid) - 1u;
            float s_acc[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) s_acc[i] = 0.f;
            for (int t = t_begin(u); t < t1; ++t, ++g) {
                const int buf = g & 1;
                const int cell = half == 0 && j < BM && env0 + j < B ? (int)b.tpos[(size_t)t * B + env0 + j] : -1;  // env j of the tile
                // Layer-1 gates: lane e fetches the word of units 32 q .. +31 of env 32 half + e; transposed across the warp, lane = unit
                ok = tc::mbar_wait(&gfull[g % GST], (uint32_t)(g / GST) & 1u);
                if (!ok) break;
                uint32_t gate = *reinterpret_cast<const uint32_t*>(sG + (g % GST) * Cfg::G_TILE + (32 * half + lane) * (H / 8) + 4 * q);
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&gempty[g % GST]);
                gate = transpose_bits32(gate, lane) & valid;
                if (PREC != 1 && g > 0 && g % Cfg::AGENT_GROUP == 0) {  // a whole group of the agent plane
                    ok = tc::mbar_wait(tiles_free, (uint32_t)(g - 1) & 1u);
                    if (!ok) break;
                    drain_agent(g == Cfg::AGENT_GROUP, true);
                }
                ok = tc::mbar_wait(&mdone[buf], (uint32_t)(g >> 1) & 1u);
                if (!ok) break;
                tc::tc_fence_after();
#pragma unroll
                for (int k = 0; k < 2; ++k) {  // sixteen envs: their columns become eight of hi pairs and eight of lo pairs
                    const uint32_t acc = tmem + lane_base + (uint32_t)(Cfg::ACC_COL + BM * buf + 32 * half + 16 * k);
                    uint32_t r[16], hi[8], lo[8];
                    tc::tmem_ld16_nowait(acc, r);
                    tc::tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int e = 16 * k + 2 * i;
                        const float v0 = rnd<PREC>((gate >> e) & 1u ? __uint_as_float(r[2 * i]) : 0.f);
                        const float v1 = rnd<PREC>((gate >> (e + 1)) & 1u ? __uint_as_float(r[2 * i + 1]) : 0.f);
                        s_acc[e] += v0;
                        s_acc[e + 1] += v1;
                        split2<PREC>(v0, v1, hi[i], lo[i]);
                    }
                    tc::tmem_st8(acc, hi);
                    if (PL == 2) tc::tmem_st8(acc + 8, lo);
                }
                tc::tmem_st_wait();
                // The MMAs of the tile before have read the one-hot tile.  Every warp waits for every tile's, also those that write no row of it: a
                // wait for a phase is only right from the one before it (two behind, it returns at once, and the accumulator would be read
                // before its last MMAs), and no warp arrives for a tile before all have for the one before.
                if (g >= 1) ok = tc::mbar_wait(tiles_free, (uint32_t)(g - 1) & 1u);
                if (half == 0 && q < BM / 32) {  // the one-hot row of env j
                    if (prev_off >= 0) *reinterpret_cast<uint16_t*>(sO + prev_off) = 0;
                    prev_off = -1;
                    if (cell >= 0 && cell < 128) {
                        // element (k = env j, n = cell) of the MN-major tile: byte k*128 + ((n/8) ^ (k%8))*16 + (n%8)*2 of box n/64
                        prev_off = (cell >> 6) * BOX + j * 128 + ((((cell & 63) >> 3) ^ (j & 7)) << 4) + (cell & 7) * 2;
                        *reinterpret_cast<uint16_t*>(sO + prev_off) = (uint16_t)one16<PREC>();
                    }
                    tc::fence_proxy_async();  // generic-proxy stores -> visible to the tensor core
                }
                tc::tc_fence_before();
                __syncwarp();
                if (!ok) break;
                if (lane == 0) tc::mbar_arrive(tiles_full);
            }
            // S (sum over t of dh1) as two 16-bit planes [ts*B][H]: an fp32 sum keeps two terms in either workload
            if (ok) {
                uint16_t* S_hi = reinterpret_cast<uint16_t*>(b.S);
                uint16_t* S_lo = S_hi + (size_t)a.ts * B * H;
                const size_t si = ((size_t)(u / m_tiles) * B + env0 + 32 * half) * H + j;  // an empty slice writes zeros
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    if (i < nvalid) {
                        uint16_t hi, lo;
                        if (PREC == 1) {
                            __nv_bfloat16 h0, l0;
                            split_bf16(s_acc[i], h0, l0);
                            hi = __bfloat16_as_ushort(h0);
                            lo = __bfloat16_as_ushort(l0);
                        } else {
                            split1<0>(s_acc[i], hi, lo);
                        }
                        S_hi[si + (size_t)i * H] = hi;
                        S_lo[si + (size_t)i * H] = lo;
                    }
                }
            }
        }
        if (!ok && lane == 0) atomicOr(status, DEV_E_WAIT_TIMEOUT);
        bool got = ok && G > 0;
        if (got) got = tc::mbar_wait(tiles_free, (uint32_t)(G - 1) & 1u);
        if (!got && ok && G > 0 && lane == 0) atomicOr(status, DEV_E_WAIT_TIMEOUT);
        drain_agent(PREC == 1 || G <= Cfg::AGENT_GROUP, got);  // the last group (or zeros)
    }
    tc::tc_fence_before();
    __syncthreads();
    if (wid == 1) tc::tmem_dealloc(tmem, Cfg::TMEM_COLS);
}

template <int PREC>
cudaError_t launch_t(const LearnArgs& a, int nx, float* part_w2, float* part_agent, size_t stride_agent, cudaStream_t s) {
    using Cfg = Back128Cfg<PREC>;
    const Dims& d = a.d;
    const Buffers& b = a.b;
    constexpr bool bf = PREC == 1;
    const size_t R = (size_t)d.B * a.T, RH = (size_t)d.B * d.Tmax * Cfg::H;
    Back128Maps maps;
    memset(&maps, 0, sizeof(maps));
    const uint16_t* h1 = reinterpret_cast<const uint16_t*>(b.h1);
    if (!make_tensor_map_2d(&maps.h_hi, h1, R, Cfg::H, Cfg::BM, bf)) return cudaErrorNotSupported;
    if (!make_tensor_map_2d(&maps.w_hi, b.w2p_hi, Cfg::H, Cfg::H, 128, bf)) return cudaErrorNotSupported;
    if (Cfg::PL == 2) {
        if (!make_tensor_map_2d(&maps.h_lo, h1 + RH, R, Cfg::H, Cfg::BM, bf)) return cudaErrorNotSupported;
        if (!make_tensor_map_2d(&maps.w_lo, b.w2p_lo, Cfg::H, Cfg::H, 128, bf)) return cudaErrorNotSupported;
    }
    return launch<k_back128<PREC>>(dim3(nx), Cfg::THREADS, Cfg::smem_bytes, s, maps, a, part_w2, part_agent, stride_agent);
}

}  // namespace

bool back128_supported(const Dims& d) { return d.H == 128 && d.C <= 128 && d.npol <= 1; }

// CTAs (one partial of everything each) and slices of the steps.
void back128_shape(const Dims& d, int T, int* nx, int* ts) {
    const int m_tiles = (d.B + 63) / 64;
    *ts = slices_for(m_tiles, 148, T, most_slices(m_tiles, 148));
    const int units = m_tiles * *ts;
    *nx = units < 148 ? units : 148;
}

// a.ts slices and nx CTAs from back128_shape; partial x of dW2 goes to part_w2[x * 16384], of the agent plane to
// part_agent[x * stride_agent], of dWh, db2, dbh to a.part_small and of the loss terms to loss_part.
cudaError_t launch_back128(const LearnArgs& a, int prec, int nx, float* part_w2, float* part_agent, size_t stride_agent, cudaStream_t s) {
    if (!back128_supported(a.d) || !a.b.gate1) return cudaErrorNotSupported;
    return prec == 1 ? launch_t<1>(a, nx, part_w2, part_agent, stride_agent, s) : launch_t<0>(a, nx, part_w2, part_agent, stride_agent, s);
}

}  // namespace anakin
