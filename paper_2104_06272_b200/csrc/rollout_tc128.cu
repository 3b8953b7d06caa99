// Persistent rollout on the 5th-generation tensor cores for hidden width 128 and large batches: one CTA owns 128 envs
// for all T+1 forward passes of a rollout and keeps the whole second layer on chip.
//
// Acting half of the Anakin minimal unit (Podracer paper, Section 3.1; Figure 2, top); the fp32 form (bf16 workloads have one
// plane of each operand and one MMA per k16).  With many envs per
// SM the rollout is a throughput problem, but a single env group still walks a strictly serial chain per step (gather the
// agent's first-layer row -> tensor cores -> heads -> sample -> next gather).  The CTA therefore holds TWO independent
// groups of 64 envs, each with eight worker warps of its own, so that one group's tensor-core phase and sampling phase
// fall into the other group's gather and heads phases.  Per group and step:
//   layer 1   h1 = relu(base + W1[agent row])       gather-add; the fp16 (hi, lo) terms go straight into the swizzled
//                                                   K-major operand tile [64 hi rows | 64 lo rows] x 128 k
//   layer 2   transposed, D[j][env] = sum_k W2[k][j] h1[env][k], M = 128 hidden units: two tcgen05 MMAs per k16,
//             W2hi x [h1hi | h1lo] (N = 128) and W2lo x h1hi (N = 64), fp32 accumulators in tensor memory beside both
//             planes of W2 (the A operand, transposed into it once: shared memory then holds the agent rows of W1 and is left
//             to the workers; 2336 -> 2118 us on 131072 envs, T = 64, with one proxy fence a step); a dedicated warp issues the MMAs of both groups
//   heads     a worker thread = one hidden unit j (its accumulator lane): bias, ReLU, h2 stores (one 128-byte line per
//             env and warp); the warp's 32 units x 32 envs go to shared memory as fp16 (hi, lo) terms and come back
//             transposed (ldmatrix.trans) as A fragments of warp-level MMAs against Wh; the four 32-unit partials of an
//             env are summed by its owner thread in a fixed order
//   env       (owner warps) one thread per env: softmax, Philox inverse-CDF sample, gridworld step, time-major records;
//             the new position is published before the records are written
// The phases meet through mbarriers only (operand blocks written -> issuer; MMAs finished -> workers; partials stored ->
// owners; positions published -> workers).  Every wait is bounded; a timeout raises DEV_E_WAIT_TIMEOUT and the threads
// keep walking through the barriers to the exit, where tensor memory is freed.
#include <type_traits>

#include "tc_common.cuh"

namespace anakin {

namespace {

struct Tc128Cfg {
    static constexpr int H = 128, NE = 64, NG = 2, NWORK = 8;   // NWORK worker warps per group
    static constexpr int NWT = NG * NWORK * 32;                 // worker threads
    static constexpr int NOWN = NG * NE;                        // owner threads: one per env
    static constexpr int THREADS = NWT + NOWN + 32;             // + the issuer warp
    static constexpr int B_CHUNK = 2 * NE * 128;                // 128 operand rows (64 hi + 64 lo) x 64 k: 16 KB
    static constexpr int B_BYTES = (H / 64) * B_CHUNK;          // a group's operand tile: 32 KB
    static constexpr int ACC = 192;                             // TMEM columns of a group: [0,128) W2hi x [hi|lo], [128,192) W2lo x hi
    static constexpr int W_COL = NG * ACC, TMEM_COLS = 512;     // W2: 64 columns a plane (two k per column), hi then lo
    static constexpr size_t fixed_bytes =
        (size_t)NG * B_BYTES + (size_t)NG * NE * H * 4                        // operand tiles, base
        + 256                                                                 // barriers, tensor-memory slot
        + (size_t)NG * 4 * NE * 5 * 4                                         // head partials: 4 blocks of 32 hidden units
        + 8 * 4 + (size_t)NOWN * 8 * 4 + NOWN * 4;                            // bh, walls, pos
    static constexpr size_t gae_bytes(int T) { return (size_t)(T + 1) * NOWN * 4 + (size_t)T * NOWN; }
};

// W1S: the agent rows of W1 in shared memory too (512 bytes a cell; larger boards gather from L2).
template <int PREC, bool REPLAY, bool W1S>
__global__ void __launch_bounds__(Tc128Cfg::THREADS, 1) k_rollout_tc128(RolloutArgs a) {
    using Cfg = Tc128Cfg;
    constexpr int H = Cfg::H, NE = Cfg::NE, NG = Cfg::NG, NWT = Cfg::NWT, NOWN = Cfg::NOWN;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);  // the swizzle needs 1024-byte alignment
    unsigned char* s_bop = sm;                                                       // [NG] operand tiles
    float* s_base = reinterpret_cast<float*>(s_bop + NG * Cfg::B_BYTES);             // [NG][NE][H]
    uint64_t* wbar = reinterpret_cast<uint64_t*>(s_base + NG * NE * H);              // the agent rows of W1 landed
    uint64_t* tfull = wbar + 1;     // [NG] this step's MMAs of the group finished
    uint64_t* ready = tfull + NG;   // [NG] the group's operand rows written (8 worker warps arrive)
    uint64_t* pdone = ready + NG;  // [NG] the four head partials of every env of the group are stored (8 warps arrive)
    uint64_t* posrdy = pdone + NG;     // [NG] the group's positions for the next step are published (2 owner warps arrive)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(posrdy + NG);
    float* s_red = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(wbar) + 256);  // [NG][4][NE][5]
    float* s_bh = s_red + NG * 4 * NE * 5;                                           // [8]
    uint32_t* s_walls = reinterpret_cast<uint32_t*>(s_bh + 8);                       // [NOWN][8]
    int* s_pos = reinterpret_cast<int*>(s_walls + NOWN * 8);                         // [NOWN]
    float* s_w1 = reinterpret_cast<float*>(s_pos + NOWN);                            // [C][H] (W1S only)
    float* s_gv = s_w1 + (W1S ? a.d.C * H : 0);                                      // [T+1][NOWN] (a.gae_smem only)
    uint8_t* s_gc = reinterpret_cast<uint8_t*>(s_gv + (a.T + 1) * NOWN);             // [T][NOWN]

    const Dims& d = a.d;
    const Buffers& b = a.b;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int e0 = blockIdx.x * NOWN;  // this CTA's first env; group g owns envs e0 + g*NE ..
    const int B = d.B, C = d.C;
    const float* W1 = b.theta_c + d.oW1;
    const bool worker = tid < NWT;
    const bool ownerw = tid >= NWT && tid < NWT + NOWN;  // a thread of the owner warps
    const bool issuer = tid == NWT + NOWN;               // lane 0 of the last warp

    // ---- prologue
    if (tid == 0) {
        tc::mbar_init(wbar, 1);
        for (int g = 0; g < NG; ++g) {
            tc::mbar_init(&tfull[g], 1);
            tc::mbar_init(&ready[g], Cfg::NWORK);
            tc::mbar_init(&pdone[g], Cfg::NWORK);
            tc::mbar_init(&posrdy[g], NE / 32);
        }
        tc::mbar_fence_init();
    }
    if (wid == (NWT + NOWN) / 32) tc::tmem_alloc(tmem_slot, Cfg::TMEM_COLS);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    PDL_START();  // (the set-up above runs under the predecessor's tail)
    // Replay recomputes the T recorded rows (mode 2: and the current state), in independent slices of steps (grid.y).
    const int t_last = REPLAY && a.replay == 1 ? a.T - 1 : a.T, t_len = REPLAY ? (t_last + (int)gridDim.y) / (int)gridDim.y : 0;
    const int t_beg = REPLAY ? (int)blockIdx.y * t_len : 0, t_end = REPLAY ? min(t_last, t_beg + t_len - 1) : t_last;
    if (W1S && issuer) {
        tc::mbar_expect_tx(wbar, (uint32_t)(C * H * 4));
        tc::bulk_load(s_w1, W1 + (size_t)C * H, wbar, (uint32_t)(C * H * 4));
    }
    // worker constants: hidden unit of this thread in the heads phase (its accumulator lane) and the env half it reads
    const int wg = worker ? wid / Cfg::NWORK : 0;   // the worker's group
    const int wl = wid % Cfg::NWORK;                // its warp within the group
    const int tidg = tid % (Cfg::NWORK * 32);       // its thread index within the group
    const int q = wl & 3, half = (wl >> 2) & 1;
    const int j = 32 * q + lane;
    float b2j = 0.f;
    uint32_t whf_hi[2][2], whf_lo[2][2];  // Wh rows of this warp's 32 hidden units as mma B fragments (k16 x n8), two k steps
    EnvLane s;
    s.pos = s.tep = s.start = s.goal = 0;
    s.n_episodes = s.n_goals = s.n_epsteps = 0;
    s.bad = 0;
    const int ow = tid - NWT;              // owner threads: env e0 + ow, group ow / NE
    const int og = ownerw ? ow / NE : 0;   // the owner's group
    const bool owner = ownerw && e0 + ow < B;
    if (worker) {
        for (int i = tid; i < NG * NE * H / 4; i += NWT) {
            const int e = i / (H / 4), k = 4 * (i - e * (H / 4));
            const bool okb = e0 + e < B;
            cp_async16(s_base + e * H + k, b.base + (size_t)(okb ? e0 + e : 0) * H + k, okb ? 16 : 0);
        }
        cp_async_commit();
        {   // W2 into tensor memory, transposed: lane = hidden unit j, 32-bit column = k 2c (low half), 2c + 1; the four warps of a
            // lane quarter take half a plane each
            const int pc = wid >> 2, col0 = 32 * (pc & 1);
            if (PREC == 0 || pc < 2) {
                const uint16_t* src = ((pc >> 1) ? b.w2p_lo : b.w2p_hi) + (size_t)(2 * col0) * H + j;
                uint32_t r[32];
#pragma unroll
                for (int c = 0; c < 32; ++c) r[c] = (uint32_t)__ldg(src + (size_t)(2 * c) * H) | ((uint32_t)__ldg(src + (size_t)(2 * c + 1) * H) << 16);
                tc::tmem_st32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(Cfg::W_COL + 64 * (pc >> 1) + col0), r);
                tc::tmem_st_wait();
            }
            tc::tc_fence_before();
        }
        b2j = b.theta_c[d.ob2 + j];
        {   // fragment element (k, n): lane = 4n + t holds k = 2t, 2t+1 (first register) and 2t+8, 2t+9 (second)
            const int n = lane >> 2, t4 = lane & 3;
#pragma unroll
            for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const int jj = 32 * q + 16 * ks + 8 * hh + 2 * t4;
                    const float w0 = n < 5 ? b.theta_c[d.oWh + (size_t)jj * 5 + n] : 0.f;
                    const float w1 = n < 5 ? b.theta_c[d.oWh + (size_t)(jj + 1) * 5 + n] : 0.f;
                    split2<PREC>(w0, w1, whf_hi[ks][hh], whf_lo[ks][hh]);
                }
        }
        if (tid < 5) s_bh[tid] = b.theta_c[d.obh + tid];
        cp_async_wait<0>();
    } else if (ownerw) {
        for (int wi = 0; wi < 8; ++wi) s_walls[ow * 8 + wi] = (owner && wi < d.W) ? b.walls[(size_t)(e0 + ow) * d.W + wi] : 0u;
        if (owner) {
            s.pos = b.pos[e0 + ow];
            s.tep = b.tep[e0 + ow];
            s.start = b.start[e0 + ow];
            s.goal = b.goal[e0 + ow];
            check_env_state(s, C, s_walls + ow * 8);
            if (REPLAY) s.pos = min((int)(t_beg < a.T ? b.tpos[(size_t)t_beg * B + e0 + ow] : b.pos[e0 + ow]), C - 1);  // the slice's first position
        }
        s_pos[ow] = s.pos;
    }
    bool ok = true;
    if (W1S && worker) ok = tc::mbar_wait(wbar, 0);
    __syncthreads();
    tc::tc_fence_after();

    __nv_bfloat16* g_h1hi = reinterpret_cast<__nv_bfloat16*>(b.h1);
    __nv_bfloat16* g_h1lo = g_h1hi + (size_t)B * d.Tmax * H;

    if (wid == (NWT + NOWN) / 32) {
        // ---- layer 2: one warp drives the tensor core for both groups (an elected lane issues), in the order the groups' operand
        // tiles are written (group 0, then group 1, every step).  A tile's eight arrivals also say that those warps have read the
        // group's accumulators of the step before.
        const uint32_t idesc_w = tc::umma_idesc<PREC>(128, 128, false, false), idesc_n = tc::umma_idesc<PREC>(128, 64, false, false);
        for (int t = t_beg; t <= t_end; ++t) {
            for (int g = 0; g < NG; ++g) {
                const uint32_t acc = tmem + (uint32_t)(g * Cfg::ACC);
                unsigned char* bop = s_bop + g * Cfg::B_BYTES;
                ok = tc::warp_all(ok && tc::mbar_wait(&ready[g], (uint32_t)(t - t_beg) & 1u));
                tc::tc_fence_after();
                if (tc::elect_one()) {
#pragma unroll
                    for (int k16 = 0; k16 < 8; ++k16) {
                        // A: 16 k = 8 columns.  B (K-major): 16 k = 32 bytes along the swizzled rows, 1024 bytes between 8-row groups
                        const uint32_t ahi = tmem + (uint32_t)(Cfg::W_COL + 8 * k16);
                        const uint64_t bd = tc::umma_desc(bop + (k16 >> 2) * Cfg::B_CHUNK + (k16 & 3) * 32, 16, 1024);
                        if (PREC == 0) {
                            tc::umma_ta(acc, ahi, bd, idesc_w, k16 ? 1u : 0u);
                            tc::umma_ta(acc + 128u, ahi + 64u, bd, idesc_n, k16 ? 1u : 0u);
                        } else {  // bf16 operands: one product, the hi rows of the operand tile only
                            tc::umma_ta(acc, ahi, bd, idesc_n, k16 ? 1u : 0u);
                        }
                    }
                    tc::umma_commit(&tfull[g]);
                }
                __syncwarp();
            }
        }
    } else if (worker) {
        // ---- layer 1 of group g for step t: 16-byte chunks of eight hidden units; all gathers of the agents' W1 rows are
        // in flight before any is used.  Thread (e, c8) covers chunk c8 of both k blocks of envs e and e + 32 (eight lanes
        // read 256 contiguous bytes of one row): chunk c8 goes to operand row (hi) and 64 + row (lo) of its block, at the
        // 16-byte position c8 ^ (row % 8) of the 128-byte row (the 128-byte swizzle of a K-major operand).  The finished
        // tile is announced to the issuer.
        auto gather = [&](int g, int t) {
            // (lanes 4-7 of an env read their two 16-byte pieces of a row in the other order: the eight lanes cover all banks)
            const int e = tidg >> 3, c8 = tidg & 7, sw = (c8 >> 2) & 1;
            unsigned char* bop = s_bop + g * Cfg::B_BYTES;
            float4 w[2][2][2];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const int pos = s_pos[g * NE + e + 32 * p];
                const float* wrow = (W1S ? s_w1 + pos * H : W1 + (size_t)(C + pos) * H) + 8 * c8;
#pragma unroll
                for (int kb = 0; kb < 2; ++kb)
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        const float4* wp = reinterpret_cast<const float4*>(wrow + 64 * kb + 4 * (sw ^ x));
                        w[kb][p][x] = W1S ? *wp : __ldg(wp);
                    }
            }
            tc::tc_fence_before();  // this thread's reads of the group's accumulators precede the arrivals below
            uint4 hi[2][2], lo[2][2];
#pragma unroll
            for (int kb = 0; kb < 2; ++kb) {
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const int er = e + 32 * p, k = 64 * kb + 8 * c8;  // row within the group
                    const float* bp = s_base + (g * NE + er) * H + k;
                    const float4 b0 = *reinterpret_cast<const float4*>(bp + 4 * sw), b1 = *reinterpret_cast<const float4*>(bp + 4 * (sw ^ 1));
                    const float4 w0 = w[kb][p][0], w1 = w[kb][p][1];
                    uint2 h0, h1, l0, l1;
                    split2<PREC>(fmaxf(b0.x + w0.x, 0.f), fmaxf(b0.y + w0.y, 0.f), h0.x, l0.x);
                    split2<PREC>(fmaxf(b0.z + w0.z, 0.f), fmaxf(b0.w + w0.w, 0.f), h0.y, l0.y);
                    split2<PREC>(fmaxf(b1.x + w1.x, 0.f), fmaxf(b1.y + w1.y, 0.f), h1.x, l1.x);
                    split2<PREC>(fmaxf(b1.z + w1.z, 0.f), fmaxf(b1.w + w1.w, 0.f), h1.y, l1.y);
                    hi[kb][p] = sw ? make_uint4(h1.x, h1.y, h0.x, h0.y) : make_uint4(h0.x, h0.y, h1.x, h1.y);
                    lo[kb][p] = sw ? make_uint4(l1.x, l1.y, l0.x, l0.y) : make_uint4(l0.x, l0.y, l1.x, l1.y);
                    unsigned char* row = bop + kb * Cfg::B_CHUNK + er * 128 + ((c8 ^ (er & 7)) << 4);
                    *reinterpret_cast<uint4*>(row) = hi[kb][p];
                    if (PREC == 0) *reinterpret_cast<uint4*>(row + NE * 128) = lo[kb][p];
                }
            }
            tc::fence_proxy_async();  // ordinary stores -> visible to the tensor core (once: it costs some 300 clocks)
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&ready[g]);
            // the copies for the update leave after the arrivals
            if (b.h1 != nullptr && t < a.T) {
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const int env = e0 + g * NE + e + 32 * p;
                    if (env < B) {
#pragma unroll
                        for (int kb = 0; kb < 2; ++kb) {
                            const size_t gi = ((size_t)t * B + env) * H + 64 * kb + 8 * c8;
                            *reinterpret_cast<uint4*>(g_h1hi + gi) = hi[kb][p];
                            if (PREC == 0) *reinterpret_cast<uint4*>(g_h1lo + gi) = lo[kb][p];
                            if (b.gate1) b.gate1[gi >> 3] = (uint8_t)nonzero_bits16(hi[kb][p]);  // the gates of these eight units
                        }
                    }
                }
            }
        };
        // ---- heads of group g for step t: thread = hidden unit j, the 32 envs of its half of the group
        auto heads = [&](int g, int t) {
            if (ok) ok = tc::mbar_wait(&tfull[g], (uint32_t)(t - t_beg) & 1u);
            tc::tc_fence_after();
            // sixteen envs at a time (registers): accumulator columns -> bias, ReLU -> the h2 rows for the update -> the
            // fp16 (hi, lo) terms for the head products.  The group's operand tile is free once the step's MMAs have
            // finished: warp w keeps [32 units][32 envs] fp16 hi and lo planes in its 4 KB of it, rows of 64 bytes whose
            // 16-byte chunks are XOR-swizzled by (row / 2) % 4 (conflict-free both ways).
            unsigned char* wsm = s_bop + g * Cfg::B_BYTES + wl * 4096;
            const int env0 = e0 + g * NE + 32 * half;  // first env of the block this warp holds
            const bool save_h2 = b.h2 != nullptr && t < a.T;
            const uint32_t lanes = tmem + (uint32_t)(g * Cfg::ACC) + ((uint32_t)(32 * q) << 16);
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                float v[16];
                {
                    uint32_t r0[16], r1[16], r2[16];
                    tc::tmem_ld16_nowait(lanes + (uint32_t)(32 * half + 16 * hf), r0);             // W2hi x h1hi
                    if (PREC == 0) {
                        tc::tmem_ld16_nowait(lanes + (uint32_t)(NE + 32 * half + 16 * hf), r1);         // W2hi x h1lo
                        tc::tmem_ld16_nowait(lanes + 128u + (uint32_t)(32 * half + 16 * hf), r2);  // W2lo x h1hi
                    }
                    tc::tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        float z = __uint_as_float(r0[e]);
                        if (PREC == 0) z = (z + __uint_as_float(r1[e])) + __uint_as_float(r2[e]);
                        v[e] = rnd<PREC>(fmaxf(z + b2j, 0.f));
                    }
                }
                if (save_h2) {  // one 128-byte line per env and warp
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        if (env0 + 16 * hf + e < B) b.h2[((size_t)t * B + env0 + 16 * hf + e) * H + j] = v[e];
                }
#pragma unroll
                for (int c2 = 0; c2 < 2; ++c2) {
                    const int c4 = 2 * hf + c2;
                    uint4 hi, lo;
                    split2<PREC>(v[8 * c2 + 0], v[8 * c2 + 1], hi.x, lo.x);
                    split2<PREC>(v[8 * c2 + 2], v[8 * c2 + 3], hi.y, lo.y);
                    split2<PREC>(v[8 * c2 + 4], v[8 * c2 + 5], hi.z, lo.z);
                    split2<PREC>(v[8 * c2 + 6], v[8 * c2 + 7], hi.w, lo.w);
                    const int off = lane * 64 + ((c4 ^ ((lane >> 1) & 3)) << 4);
                    *reinterpret_cast<uint4*>(wsm + off) = hi;
                    if (PREC == 0) *reinterpret_cast<uint4*>(wsm + 2048 + off) = lo;
                }
            }
            __syncwarp();
            float acc[2][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[mt][i] = 0.f;
            {
                // A fragment (row = env, k = unit) from the [unit][env] tile: matrix i of the x4 load covers units
                // 16ks + 8(i/2) .., envs 16mt + 8(i%2) ..; the transposing load hands out the fragment's register order
                const int mi = lane >> 3, r8 = lane & 7;
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    const int krow = 16 * ks + 8 * (mi >> 1) + r8;
#pragma unroll
                    for (int mt = 0; mt < 2; ++mt) {
                        const int chunk = 2 * mt + (mi & 1);
                        const int off = krow * 64 + ((chunk ^ ((krow >> 1) & 3)) << 4);
                        uint32_t ahi[4], alo[4];
                        ldmatrix_x4_trans(ahi, wsm + off);
                        if (PREC == 0) ldmatrix_x4_trans(alo, wsm + 2048 + off);
                        if (PREC == 0) {
                            mma16816<PREC>(acc[mt], alo, whf_hi[ks][0], whf_hi[ks][1]);
                            mma16816<PREC>(acc[mt], ahi, whf_lo[ks][0], whf_lo[ks][1]);
                        }
                        mma16816<PREC>(acc[mt], ahi, whf_hi[ks][0], whf_hi[ks][1]);
                    }
                }
            }
            // accumulator element (row g8 + 8hh of tile mt, column 2 t4 + cc) = (env 16mt + 8hh + g8 of this half, head 2 t4 + cc)
            {
                const int g8 = lane >> 2, t4 = lane & 3;
                float* red = s_red + ((g * 4 + q) * NE + 32 * half) * 5;
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const int e = 16 * mt + 8 * hh + g8;
                        if (t4 < 3) red[e * 5 + 2 * t4] = acc[mt][2 * hh];
                        if (t4 < 2) red[e * 5 + 2 * t4 + 1] = acc[mt][2 * hh + 1];
                    }
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&pdone[g]);
        };
        // a group's eight warps walk its steps on their own; the two groups drift apart by themselves, so that one group's
        // tensor-core and sampling phases fall into the other's gather and heads phases
        if (t_beg <= t_end) gather(wg, t_beg);
        for (int t = t_beg; t <= t_end; ++t) {
            heads(wg, t);
            if (t < t_end) {
                if (ok) ok = tc::mbar_wait(&posrdy[wg], (uint32_t)(t - t_beg) & 1u);  // the owners have published the positions after step t
                gather(wg, t + 1);
            }
        }
    } else if (ownerw) {
        // ---- one thread per env
        const int env = e0 + ow;
        const int oe = ow - og * NE;  // env index within the group
        for (int t = t_beg; t <= t_end; ++t) {
            // the logits-independent half of the interaction, while the workers gather and the tensor core runs
            const bool acting = owner && !REPLAY && t < a.T;
            StepPre pre;
            if (acting) pre = step_prepare(s, a, env, t, s_walls + ow * 8);
            if (ok) ok = tc::mbar_wait(&pdone[og], (uint32_t)(t - t_beg) & 1u);
            float o[5];
#pragma unroll
            for (int c = 0; c < 5; ++c) o[c] = 0.f;
            ActOut ao;
            ao.la_mx = ao.Z = ao.rew = 0.f;
            ao.act = ao.done = ao.pos0 = 0;
            if (owner) {
#pragma unroll
                for (int blk = 0; blk < 4; ++blk)
#pragma unroll
                    for (int c = 0; c < 5; ++c) o[c] += s_red[((og * 4 + blk) * NE + oe) * 5 + c];
#pragma unroll
                for (int c = 0; c < 5; ++c) o[c] += s_bh[c];
                if (acting) {
                    ao = act_decide(s, a, env, t, o[0], o[1], o[2], o[3], pre);
                    s_pos[ow] = s.pos;
                } else if (REPLAY && t < t_end) {  // positions come from the recorded trajectory (row T: the env state as it stands)
                    s_pos[ow] = min((int)(t + 1 < a.T ? b.tpos[(size_t)(t + 1) * B + env] : b.pos[env]), C - 1);
                }
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&posrdy[og]);  // the workers may gather the group's next step
            if (owner) {
                if (b.out5 && t < a.T) {  // the update reuses the head outputs of every recorded row
                    float4* o5 = reinterpret_cast<float4*>(b.out5 + ((size_t)t * B + env) * 8);
                    o5[0] = make_float4(o[0], o[1], o[2], o[3]);
                    o5[1] = make_float4(o[4], 0.f, 0.f, 0.f);
                }
                if (REPLAY && a.replay == 2 && t == a.T) b.vboot[env] = o[4];
                if (!REPLAY) {
                    b.tval[(size_t)t * B + env] = o[4];
                    if (a.gae_smem) s_gv[t * NOWN + ow] = o[4];
                }
                if (acting) {
                    act_record(a, env, t, o[0], o[1], o[2], o[3], ao);
                    if (a.gae_smem) s_gc[t * NOWN + ow] = (uint8_t)(ao.done | (ao.rew != 0.f ? 2 : 0));
                }
            }
        }
        if (owner && !REPLAY) {
            b.pos[env] = (uint8_t)s.pos;
            b.tep[env] = (uint8_t)s.tep;
            if (a.gae_smem) gae_scan_env_smem(b, B, a.T, env, a.gamma, a.lambda, s_gv, s_gc, NOWN, ow);
            else if (a.fuse_gae) gae_scan_env(b, B, a.T, env, a.gamma, a.lambda);
        }
        if (!REPLAY) flush_env_stats(s, a, wid == NWT / 32);
    }
    if (!ok && lane == 0) atomicOr(b.status, DEV_E_WAIT_TIMEOUT);
    tc::tc_fence_before();
    __syncthreads();
    if (wid == (NWT + NOWN) / 32) tc::tmem_dealloc(tmem, Cfg::TMEM_COLS);
}

}  // namespace

// Hidden width 128 in either precision, on batches beyond one wave of the warp-level kernel and on replays of more than 64
// envs; anything else returns cudaErrorNotSupported and the caller takes the warp-level kernel.
cudaError_t launch_rollout_tc128(const RolloutArgs& a0, int prec, cudaStream_t s) {
    using Cfg = Tc128Cfg;
    if (a0.d.H != Cfg::H || !a0.b.w2p_hi || (prec == 0 && !a0.b.w2p_lo) || !a0.b.base || a0.d.npol > 1) return cudaErrorNotSupported;
    // Acting: beyond one wave of the warp-level kernel (two CTAs of 32 envs per SM), whose step takes 4.4 us against 5.8 us here.
    // Replay: whenever a CTA's two groups have envs.
    if (a0.replay ? a0.d.B <= Cfg::NE : a0.d.B <= 148 * 64) return cudaErrorNotSupported;
    RolloutArgs a = a0;
    size_t smem = Cfg::fixed_bytes + 1024;  // alignment slack
    const size_t w1 = (size_t)a.d.C * Cfg::H * 4;
    const bool w1s = smem + w1 <= 232448;
    if (w1s) smem += w1;
    a.gae_smem = 0;
    if (a.fuse_gae && !a.replay && smem + Cfg::gae_bytes(a.T) <= 232448) {
        a.gae_smem = 1;
        smem += Cfg::gae_bytes(a.T);
    }
    const int ctas = (a.d.B + Cfg::NOWN - 1) / Cfg::NOWN;
    const dim3 grid(ctas, replay_slices(a, ctas));
    auto go = [&](auto w) {
        constexpr bool W = decltype(w)::value;
        if (prec == 1) return a.replay ? launch<k_rollout_tc128<1, true, W>>(grid, Cfg::THREADS, smem, s, a) : launch<k_rollout_tc128<1, false, W>>(grid, Cfg::THREADS, smem, s, a);
        return a.replay ? launch<k_rollout_tc128<0, true, W>>(grid, Cfg::THREADS, smem, s, a) : launch<k_rollout_tc128<0, false, W>>(grid, Cfg::THREADS, smem, s, a);
    };
    return w1s ? go(std::true_type{}) : go(std::false_type{});
}

}  // namespace anakin
