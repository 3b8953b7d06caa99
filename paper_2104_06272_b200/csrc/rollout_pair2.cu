// Persistent rollout on the 5th-generation tensor cores for hidden width 256 and large batches: a pair of CTAs (a
// cluster of two, on neighbouring SMs) owns 128 envs for all T+1 forward passes, in TWO independent groups of 64.
//
// Acting half of the Anakin minimal unit (Podracer paper, Section 3.1; Figure 2, top); the fp32 form (bf16 workloads have one
// plane of each operand and one MMA per k16).  The layout of one
// group is that of the one-group CTA-pair kernel: layer 2 transposed, D[j][env] = sum_k W2[k][j] h1[env][k], as
// tcgen05.mma.cta_group::2 with M = 256 hidden units, each CTA keeping ITS 128 columns of W2 on chip (the fp16 hi
// plane transposed in tensor memory as the A operand, the lo plane in shared memory) and building the h1 rows of ITS 32 envs of the group.  With many envs per SM the rollout is a
// throughput problem, but one group walks a strictly serial chain per step (gather -> tensor cores -> heads -> sample);
// so a CTA holds two groups, each with eight worker warps and an owner warp of its own, and one group's tensor-core and
// sampling phases fall into the other's gather and heads phases.  Per group and step:
//   layer 1   h1 = relu(base + W1[agent row])       gather-add (base in shared memory); fp16 (hi, lo) terms straight into the swizzled
//                                                   K-major operand tile [32 hi rows | 32 lo rows] x 256 k
//   layer 2   two MMAs per k16:  W2hi x [h1hi | h1lo]  (N = 128 over the pair)  and  W2lo x h1hi  (N = 64), fp32
//             accumulators in tensor memory; one thread of the leader CTA's issuer warp drives both groups
//   heads     a worker thread = one hidden unit j: bias, ReLU, h2 stores, then 32 units x 32 envs through shared memory
//             (ldmatrix.trans) into warp-level MMAs against Wh; the eight 32-unit partials of an env meet in the shared
//             memory of the CTA that owns it, sent as asynchronous remote stores that count their bytes on its mbarrier
//   env       (owner warps) one thread per env: softmax, Philox inverse-CDF sample, gridworld step, time-major records;
//             the new position is published before the records are written
// (B200, 65536 envs, T = 32: 1450 us with both planes of W2 in shared memory, base read from L2, a proxy fence per k block and
// conflicting reads; 1120 us so.)
// The phases meet through mbarriers only; the cluster barrier is used at start and exit.  Every wait is bounded; a timeout
// raises DEV_E_WAIT_TIMEOUT and the threads keep walking through the barriers to the exit, where tensor memory is freed.
#include <cstring>

#include "tc_common.cuh"

namespace anakin {

namespace {

struct Pair2Cfg {
    static constexpr int H = 256, ME = 32, NG = 2, NWORK = 8;       // ME envs per CTA and group, NWORK worker warps per group
    static constexpr int NWT = NG * NWORK * 32;                     // worker threads
    static constexpr int NOWN = NG * ME;                            // owner threads: one per env of this CTA
    static constexpr int THREADS = NWT + NOWN + 32;                 // + the issuer warp
    static constexpr int BOX = 64 * 64 * 2;                         // one 64 x 64 box of 16-bit elements
    static constexpr int A_PLANE = (128 / 64) * (H / 64) * BOX;     // this CTA's 128 columns of W2, all k: 64 KB (the lo plane)
    static constexpr int B_CHUNK = 64 * 128;                        // 64 operand rows (32 hi + 32 lo) x 64 k
    static constexpr int B_BYTES = (H / 64) * B_CHUNK;              // a group's operand tile: 32 KB
    static constexpr int ACC = 192;                                 // TMEM columns of a group
    static constexpr int W_COL = NG * ACC, TMEM_COLS = 512;         // W2 hi: 128 columns (lane = hidden unit, two k per column)
    static constexpr size_t fixed_bytes =
        (size_t)A_PLANE + (size_t)NG * B_BYTES + (size_t)NG * ME * H * 4  // W2 lo, operand tiles, base
        + 256                                                       // barriers, tensor-memory slot
        + (size_t)NG * 8 * ME * 6 * 4                               // head partials: 8 blocks of 32 hidden units per group
        + 8 * 4 + (size_t)NOWN * 8 * 4 + NOWN * 4;                  // bh, walls, pos
    static constexpr size_t gae_bytes(int T) { return (size_t)(T + 1) * NOWN * 4 + (size_t)T * NOWN; }
};

struct Pair2Maps {
    CUtensorMap w_lo;  // W2 row-major [k][j], the fp16 lo plane, boxes of 64 j x 64 k
};

// Asynchronous store of two floats into the shared memory of a CTA of the cluster; when it has landed it counts its
// eight bytes on the mbarrier (same CTA as the destination), so the reader needs no fence from the writer.
__device__ __forceinline__ void st_async_f32x2(uint32_t cluster_addr, float v0, float v1, uint32_t cluster_bar_addr) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(cluster_addr), "f"(v0), "f"(v1),
                 "r"(cluster_bar_addr)
                 : "memory");
}

template <int PREC, bool REPLAY>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(Pair2Cfg::THREADS, 1) k_rollout_pair2(const __grid_constant__ Pair2Maps maps, RolloutArgs a) {
    using Cfg = Pair2Cfg;
    constexpr int H = Cfg::H, ME = Cfg::ME, NG = Cfg::NG, NWT = Cfg::NWT, NOWN = Cfg::NOWN;
    extern __shared__ unsigned char smem_raw[];
    // the dynamic shared memory starts at the same offset in both CTAs, so the rounded base does too
    unsigned char* sm = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* s_alo = sm;
    unsigned char* s_bop = s_alo + Cfg::A_PLANE;                                     // [NG] operand tiles
    float* s_base = reinterpret_cast<float*>(s_bop + NG * Cfg::B_BYTES);             // [NG][ME][H]
    uint64_t* wbar = reinterpret_cast<uint64_t*>(s_base + NG * ME * H);              // W2 lo landed
    uint64_t* tfull = wbar + 1;      // [NG] this step's MMAs of the group finished
    uint64_t* ready = tfull + NG;    // [NG][2] leader's copy: two k blocks of both CTAs' operand rows written (16 warps arrive)
    uint64_t* pfull = ready + NG * 2;  // [NG] the eight head partials of this CTA's envs of the group have landed (bytes)
    uint64_t* posrdy = pfull + NG;     // [NG] this CTA's positions of the group for the next step are published
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(posrdy + NG);
    float* s_red = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(wbar) + 256);  // [NG][8][ME][6]
    float* s_bh = s_red + NG * 8 * ME * 6;                                           // [8]
    uint32_t* s_walls = reinterpret_cast<uint32_t*>(s_bh + 8);                       // [NOWN][8]
    int* s_pos = reinterpret_cast<int*>(s_walls + NOWN * 8);                         // [NOWN]
    float* s_gv = reinterpret_cast<float*>(s_pos + NOWN);                            // [T+1][NOWN] (a.gae_smem only)
    uint8_t* s_gc = reinterpret_cast<uint8_t*>(s_gv + (a.T + 1) * NOWN);             // [T][NOWN]

    const Dims& d = a.d;
    const Buffers& b = a.b;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint32_t rank = tc::cluster_ctarank();
    const int pair = blockIdx.x >> 1;
    // the pair owns envs pair*128 ..: group g has 64 of them, CTA `rank` the 32 at pair*128 + g*64 + rank*32
    const int B = d.B, C = d.C;
    const float* W1 = b.theta_c + d.oW1;
    const bool worker = tid < NWT;
    const bool ownerw = tid >= NWT && tid < NWT + NOWN;
    const int iwarp = (NWT + NOWN) / 32;           // the issuer warp
    const bool issuer = tid == NWT + NOWN;

    // ---- prologue
    if (tid == 0) {
        tc::mbar_init(wbar, 1);
        for (int g = 0; g < NG; ++g) {
            tc::mbar_init(&tfull[g], 1);
            for (int i = 0; i < 2; ++i) tc::mbar_init(&ready[2 * g + i], 2 * Cfg::NWORK);
            tc::mbar_init(&pfull[g], 1);
            tc::mbar_init(&posrdy[g], 1);
        }
        tc::mbar_fence_init();
    }
    if (wid == iwarp) tc::tmem_alloc_pair(tmem_slot, Cfg::TMEM_COLS);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    PDL_START();  // (the set-up above runs under the predecessor's tail)
    // Replay recomputes the T recorded rows (mode 2: and the current state), in independent slices of steps (grid.y).
    const int t_last = REPLAY && a.replay == 1 ? a.T - 1 : a.T, t_len = REPLAY ? (t_last + (int)gridDim.y) / (int)gridDim.y : 0;
    const int t_beg = REPLAY ? (int)blockIdx.y * t_len : 0, t_end = REPLAY ? min(t_last, t_beg + t_len - 1) : t_last;
    if (PREC == 0 && issuer) {  // this CTA's 128 columns of the lo plane: box (kb, bx) = k rows 64kb.., columns 128 rank + 64 bx..
        tc::mbar_expect_tx(wbar, Cfg::A_PLANE);
#pragma unroll
        for (int kb = 0; kb < H / 64; ++kb)
#pragma unroll
            for (int bx = 0; bx < 2; ++bx) tc::tma_load_2d(s_alo + (kb * 2 + bx) * Cfg::BOX, &maps.w_lo, wbar, 128 * (int)rank + 64 * bx, 64 * kb);
    }
    // worker constants
    const int wg = worker ? wid / Cfg::NWORK : 0;   // the worker's group
    const int wl = wid % Cfg::NWORK;                // its warp within the group
    const int tidg = tid % (Cfg::NWORK * 32);       // its thread index within the group
    const int q = wl & 3, rE = (wl >> 2) & 1;       // accumulator lanes 32q.., envs of CTA rE
    const int j = 128 * (int)rank + 32 * q + lane;  // hidden unit of this thread in the heads phase
    float b2j = 0.f;
    uint32_t whf_hi[2][2], whf_lo[2][2];  // Wh rows of this warp's 32 hidden units as mma B fragments (k16 x n8), two k steps
    EnvLane s;
    s.pos = s.tep = s.start = s.goal = 0;
    s.n_episodes = s.n_goals = s.n_epsteps = 0;
    s.bad = 0;
    const int ow = tid - NWT;                  // owner threads: index into this CTA's envs, group ow / ME
    const int og = ownerw ? ow / ME : 0;
    const int oe = ow - og * ME;               // env index within the group's 32 of this CTA
    const int oenv = pair * (2 * NG * ME) + og * (2 * ME) + (int)rank * ME + oe;  // global env of an owner thread
    const bool owner = ownerw && oenv < B;
    if (worker) {
        for (int i = tid; i < NG * ME * H / 4; i += NWT) {
            const int e = i / (H / 4), k = 4 * (i - e * (H / 4));
            const int env = pair * (2 * NG * ME) + (e / ME) * (2 * ME) + (int)rank * ME + e % ME;
            cp_async16(s_base + e * H + k, b.base + (size_t)(env < B ? env : 0) * H + k, env < B ? 16 : 0);
        }
        cp_async_commit();
        {   // W2 hi into tensor memory, transposed: lane = hidden unit j, 32-bit column = k 2c (low half), 2c + 1; the four warps of a
            // lane quarter take 32 columns each
            const int col0 = 32 * (wid >> 2);
            const uint16_t* src = b.w2p_hi + (size_t)(2 * col0) * H + j;
            uint32_t r[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) r[c] = (uint32_t)__ldg(src + (size_t)(2 * c) * H) | ((uint32_t)__ldg(src + (size_t)(2 * c + 1) * H) << 16);
            tc::tmem_st32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(Cfg::W_COL + col0), r);
            tc::tmem_st_wait();
            tc::tc_fence_before();
        }
        b2j = b.theta_c[d.ob2 + j];
        {   // fragment element (k, n): lane = 4n + t holds k = 2t, 2t+1 (first register) and 2t+8, 2t+9 (second)
            const int n = lane >> 2, t4 = lane & 3;
#pragma unroll
            for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const int jj = 128 * (int)rank + 32 * q + 16 * ks + 8 * hh + 2 * t4;
                    const float w0 = n < 5 ? b.theta_c[d.oWh + (size_t)jj * 5 + n] : 0.f;
                    const float w1 = n < 5 ? b.theta_c[d.oWh + (size_t)(jj + 1) * 5 + n] : 0.f;
                    split2<PREC>(w0, w1, whf_hi[ks][hh], whf_lo[ks][hh]);
                }
        }
        if (tid < 5) s_bh[tid] = b.theta_c[d.obh + tid];
        cp_async_wait<0>();
    } else if (ownerw) {
        for (int wi = 0; wi < 8; ++wi) s_walls[ow * 8 + wi] = (owner && wi < d.W) ? b.walls[(size_t)oenv * d.W + wi] : 0u;
        if (owner) {
            s.pos = b.pos[oenv];
            s.tep = b.tep[oenv];
            s.start = b.start[oenv];
            s.goal = b.goal[oenv];
            check_env_state(s, C, s_walls + ow * 8);
            if (REPLAY) s.pos = min((int)(t_beg < a.T ? b.tpos[(size_t)t_beg * B + oenv] : b.pos[oenv]), C - 1);  // the slice's first position
        }
        s_pos[ow] = s.pos;
    }
    bool ok = true;
    if (PREC == 0 && issuer) ok = tc::mbar_wait(wbar, 0);  // the issuer's thread vouches for the weights of its CTA
    __syncthreads();
    tc::cluster_sync_all();  // both CTAs' barriers, tensor memory and weights exist before the first MMA
    tc::tc_fence_after();

    __nv_bfloat16* g_h1hi = reinterpret_cast<__nv_bfloat16*>(b.h1);
    __nv_bfloat16* g_h1lo = g_h1hi + (size_t)B * d.Tmax * H;

    if (wid == iwarp) {
        // ---- layer 2: this warp of the leader CTA drives both tensor cores for both groups (one elected lane issues), k block by k block, in the
        // order the groups' operand blocks are written.  A block's sixteen arrivals also say that those warps have read
        // the group's accumulators of the step before.
        if (rank == 0) {
            const uint32_t idesc_w = tc::umma_idesc<PREC>(256, 128, false, false), idesc_n = tc::umma_idesc<PREC>(256, 64, false, false);
            const uint32_t idesc_lo = tc::umma_idesc<PREC>(256, 64, true, false);
            for (int t = t_beg; t <= t_end; ++t) {
                for (int g = 0; g < NG; ++g) {
                    const uint32_t acc = tmem + (uint32_t)(g * Cfg::ACC);
                    unsigned char* bop = s_bop + g * Cfg::B_BYTES;
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        ok = tc::warp_all(ok && tc::mbar_wait_cluster(&ready[2 * g + i], (uint32_t)(t - t_beg) & 1u));
                        tc::tc_fence_after();
                        if (tc::elect_one()) {
#pragma unroll
                            for (int k16 = 8 * i; k16 < 8 * i + 8; ++k16) {
                                // A hi (tensor memory): 16 k = 8 columns.  A lo (MN-major): 16 k rows = 2048 bytes into each box, 8192
                                // bytes between the two 64-column boxes.  B (K-major): 16 k = 32 bytes along the swizzled rows
                                const uint32_t ahi = tmem + (uint32_t)(Cfg::W_COL + 8 * k16);
                                const uint64_t bd = tc::umma_desc(bop + (k16 >> 2) * Cfg::B_CHUNK + (k16 & 3) * 32, 16, 1024);
                                if (PREC == 0) {
                                    tc::umma_pair_ta(acc, ahi, bd, idesc_w, k16 ? 1u : 0u);
                                    tc::umma_pair(acc + 128u, tc::umma_desc(s_alo + (k16 >> 2) * 2 * Cfg::BOX + (k16 & 3) * 2048, Cfg::BOX, 1024), bd, idesc_lo, k16 ? 1u : 0u);
                                } else {  // bf16 operands: one product, the hi rows of the operand tile only
                                    tc::umma_pair_ta(acc, ahi, bd, idesc_n, k16 ? 1u : 0u);
                                }
                            }
                            if (i == 1) tc::umma_commit_pair(&tfull[g], 3);
                        }
                        __syncwarp();
                    }
                }
            }
        }
    } else if (worker) {
        // ---- layer 1 of group g for step t: 16-byte chunks of eight hidden units; two k blocks' gathers are in flight before any is
        // used.  Thread (e, c8) covers chunk c8 of the four k blocks of env e: the chunk goes to operand row e (hi) and
        // 32 + e (lo) of its block, at the 16-byte position c8 ^ (e % 8) of the 128-byte row (the 128-byte swizzle of a
        // K-major operand).  Two finished blocks at a time are announced to the leader's issuer (one proxy fence).  Lanes 4-7 of an
        // env read their two 16-byte pieces of a row in the other order, so that the eight lanes cover all banks.
        auto gather = [&](int g, int t) {
            const int e = tidg >> 3, c8 = tidg & 7, sw = (c8 >> 2) & 1;
            const int env = pair * (2 * NG * ME) + g * (2 * ME) + (int)rank * ME + e;
            unsigned char* bop = s_bop + g * Cfg::B_BYTES;
            const float* wrow = W1 + (size_t)(C + s_pos[g * ME + e]) * H + 8 * c8;
            const float* brow = s_base + (g * ME + e) * H + 8 * c8;
            uint4 hi[4], lo[4];
            float4 w[4][2];
#pragma unroll
            for (int kb = 0; kb < 4; ++kb)
#pragma unroll
                for (int x = 0; x < 2; ++x) w[kb][x] = __ldg(reinterpret_cast<const float4*>(wrow + 64 * kb + 4 * (sw ^ x)));
            tc::tc_fence_before();  // this thread's reads of the group's accumulators precede the arrivals below
#pragma unroll
            for (int kb = 0; kb < 4; ++kb) {
                const float4 b0 = *reinterpret_cast<const float4*>(brow + 64 * kb + 4 * sw), b1 = *reinterpret_cast<const float4*>(brow + 64 * kb + 4 * (sw ^ 1));
                uint2 h0, h1, l0, l1;
                split2<PREC>(fmaxf(b0.x + w[kb][0].x, 0.f), fmaxf(b0.y + w[kb][0].y, 0.f), h0.x, l0.x);
                split2<PREC>(fmaxf(b0.z + w[kb][0].z, 0.f), fmaxf(b0.w + w[kb][0].w, 0.f), h0.y, l0.y);
                split2<PREC>(fmaxf(b1.x + w[kb][1].x, 0.f), fmaxf(b1.y + w[kb][1].y, 0.f), h1.x, l1.x);
                split2<PREC>(fmaxf(b1.z + w[kb][1].z, 0.f), fmaxf(b1.w + w[kb][1].w, 0.f), h1.y, l1.y);
                hi[kb] = sw ? make_uint4(h1.x, h1.y, h0.x, h0.y) : make_uint4(h0.x, h0.y, h1.x, h1.y);
                lo[kb] = sw ? make_uint4(l1.x, l1.y, l0.x, l0.y) : make_uint4(l0.x, l0.y, l1.x, l1.y);
                unsigned char* row = bop + kb * Cfg::B_CHUNK + e * 128 + ((c8 ^ (e & 7)) << 4);
                *reinterpret_cast<uint4*>(row) = hi[kb];
                if (PREC == 0) *reinterpret_cast<uint4*>(row + ME * 128) = lo[kb];
                if (kb & 1) {
                    tc::fence_proxy_async();  // ordinary stores -> visible to the tensor cores
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive_remote_cta_release(tc::mapa(tc::smem_u32(&ready[2 * g + (kb >> 1)]), 0));
                }
            }
            // the copies for the update leave after the arrivals (their CTA-scope release does not wait for global stores)
            if (b.h1 != nullptr && t < a.T && env < B) {
#pragma unroll
                for (int kb = 0; kb < 4; ++kb) {
                    const size_t gi = ((size_t)t * B + env) * H + 64 * kb + 8 * c8;
                    *reinterpret_cast<uint4*>(g_h1hi + gi) = hi[kb];
                    if (PREC == 0) *reinterpret_cast<uint4*>(g_h1lo + gi) = lo[kb];
                    if (b.gate1) b.gate1[gi >> 3] = (uint8_t)nonzero_bits16(hi[kb]);  // the gates of these eight units
                }
            }
        };
        // ---- heads of group g for step t: thread = hidden unit j, the group's 32 envs of CTA rE
        auto heads = [&](int g, int t) {
            if (ok) ok = tc::mbar_wait(&tfull[g], (uint32_t)(t - t_beg) & 1u);
            tc::tc_fence_after();
            // sixteen envs at a time (registers): accumulator columns -> bias, ReLU -> the h2 rows for the update -> the
            // fp16 (hi, lo) terms for the head products.  The group's operand tile is free once the step's MMAs have
            // finished: warp w keeps [32 units][32 envs] fp16 hi and lo planes in its 4 KB of it, rows of 64 bytes whose
            // 16-byte chunks are XOR-swizzled by (row / 2) % 4 (conflict-free both ways).
            unsigned char* wsm = s_bop + g * Cfg::B_BYTES + wl * 4096;
            const int env0 = pair * (2 * NG * ME) + g * (2 * ME) + rE * ME;  // first env of the block this warp holds
            const bool save_h2 = b.h2 != nullptr && t < a.T;
            const uint32_t lanes = tmem + (uint32_t)(g * Cfg::ACC) + ((uint32_t)(32 * q) << 16);
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                float v[16];
                {
                    uint32_t r0[16], r1[16], r2[16];
                    tc::tmem_ld16_nowait(lanes + (uint32_t)((PREC == 0 ? 64 : 32) * rE + 16 * hf), r0);             // W2hi x h1hi
                    if (PREC == 0) {
                        tc::tmem_ld16_nowait(lanes + (uint32_t)(64 * rE + 32 + 16 * hf), r1);         // W2hi x h1lo
                        tc::tmem_ld16_nowait(lanes + 128u + (uint32_t)(32 * rE + 16 * hf), r2);  // W2lo x h1hi
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
            // every warp of the group is done with its staging area before any of them writes the operand tile again (the
            // partials below only tell an owner about the four warps of each CTA that hold ITS envs); named barrier 1 + g
            asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "n"(Cfg::NWORK * 32) : "memory");
            // accumulator element (row g8 + 8hh of tile mt, column 2 t4 + cc) = (env 16mt + 8hh + g8 of CTA rE's block, head 2 t4 + cc)
            {
                const int g8 = lane >> 2, t4 = lane & 3;
                const uint32_t pbar = tc::mapa(tc::smem_u32(&pfull[g]), (uint32_t)rE);
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const int e = 16 * mt + 8 * hh + g8;
                        const uint32_t dst = tc::mapa(tc::smem_u32(s_red + (((g * 8) + 4 * (int)rank + q) * ME + e) * 6 + 2 * t4), (uint32_t)rE);
                        if (t4 < 3) st_async_f32x2(dst, acc[mt][2 * hh], acc[mt][2 * hh + 1], pbar);
                    }
            }
        };
        // a group's eight warps walk its steps on their own
        if (t_beg <= t_end) gather(wg, t_beg);
        for (int t = t_beg; t <= t_end; ++t) {
            heads(wg, t);
            if (t < t_end) {
                if (ok) ok = tc::mbar_wait(&posrdy[wg], (uint32_t)(t - t_beg) & 1u);  // the owners have published the positions after step t
                gather(wg, t + 1);
            }
        }
    } else if (ownerw) {
        // ---- one thread per env of this CTA (owner warp og serves group og)
        for (int t = t_beg; t <= t_end; ++t) {
            if (lane == 0) tc::mbar_expect_tx(&pfull[og], 8 * ME * 6 * 4);  // this step's head partials, counted as they land
            const bool acting = owner && !REPLAY && t < a.T;
            StepPre pre;
            if (acting) pre = step_prepare(s, a, oenv, t, s_walls + ow * 8);
            if (ok) ok = tc::mbar_wait_cluster(&pfull[og], (uint32_t)(t - t_beg) & 1u);
            float o[5];
#pragma unroll
            for (int c = 0; c < 5; ++c) o[c] = 0.f;
            ActOut ao;
            ao.la_mx = ao.Z = ao.rew = 0.f;
            ao.act = ao.done = ao.pos0 = 0;
            if (owner) {
#pragma unroll
                for (int blk = 0; blk < 8; ++blk)
#pragma unroll
                    for (int c = 0; c < 5; ++c) o[c] += s_red[((og * 8 + blk) * ME + oe) * 6 + c];
#pragma unroll
                for (int c = 0; c < 5; ++c) o[c] += s_bh[c];
                if (acting) {
                    ao = act_decide(s, a, oenv, t, o[0], o[1], o[2], o[3], pre);
                    s_pos[ow] = s.pos;
                } else if (REPLAY && t < t_end) {  // positions come from the recorded trajectory (row T: the env state as it stands)
                    s_pos[ow] = min((int)(t + 1 < a.T ? b.tpos[(size_t)(t + 1) * B + oenv] : b.pos[oenv]), C - 1);
                }
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&posrdy[og]);  // the group's workers of this CTA may gather the next step
            if (owner) {
                if (b.out5 && t < a.T) {  // the update reuses the head outputs of every recorded row
                    float4* o5 = reinterpret_cast<float4*>(b.out5 + ((size_t)t * B + oenv) * 8);
                    o5[0] = make_float4(o[0], o[1], o[2], o[3]);
                    o5[1] = make_float4(o[4], 0.f, 0.f, 0.f);
                }
                if (REPLAY && a.replay == 2 && t == a.T) b.vboot[oenv] = o[4];
                if (!REPLAY) {
                    b.tval[(size_t)t * B + oenv] = o[4];
                    if (a.gae_smem) s_gv[t * NOWN + ow] = o[4];
                }
                if (acting) {
                    act_record(a, oenv, t, o[0], o[1], o[2], o[3], ao);
                    if (a.gae_smem) s_gc[t * NOWN + ow] = (uint8_t)(ao.done | (ao.rew != 0.f ? 2 : 0));
                }
            }
        }
        if (owner && !REPLAY) {
            b.pos[oenv] = (uint8_t)s.pos;
            b.tep[oenv] = (uint8_t)s.tep;
            if (a.gae_smem) gae_scan_env_smem(b, B, a.T, oenv, a.gamma, a.lambda, s_gv, s_gc, NOWN, ow);
            else if (a.fuse_gae) gae_scan_env(b, B, a.T, oenv, a.gamma, a.lambda);
        }
        if (!REPLAY) flush_env_stats(s, a, wid == NWT / 32);
    }
    if (!ok && lane == 0) atomicOr(b.status, DEV_E_WAIT_TIMEOUT);
    // neither CTA frees tensor memory or leaves while the other may still signal it
    tc::tc_fence_before();
    __syncthreads();
    tc::cluster_sync_all();
    if (wid == iwarp) tc::tmem_dealloc_pair(tmem, Cfg::TMEM_COLS);
}

}  // namespace

// Hidden width 256 in either precision, on batches beyond one wave of the one-group kernel and on replays of 128 envs and more;
// anything else returns cudaErrorNotSupported and the caller takes the one-group CTA-pair kernel.
cudaError_t launch_rollout_pair2(const RolloutArgs& a0, int prec, cudaStream_t s) {
    using Cfg = Pair2Cfg;
    constexpr int PER_PAIR = 2 * Cfg::NG * Cfg::ME;
    if (a0.d.H != Cfg::H || !a0.b.w2p_hi || (prec == 0 && !a0.b.w2p_lo) || !a0.b.base || a0.d.npol > 1) return cudaErrorNotSupported;
    // Acting: beyond one wave of the one-group kernel (74 pairs of 64 envs), whose second wave would cost more than the longer
    // steps here (5.2 us for 128 envs against 3.6 us for 64).  Replay: whenever a pair has its two groups.
    if (a0.replay ? a0.d.B < PER_PAIR : a0.d.B <= 74 * PER_PAIR / 2) return cudaErrorNotSupported;
    RolloutArgs a = a0;
    size_t smem = Cfg::fixed_bytes + 1024;  // alignment slack
    a.gae_smem = 0;
    if (a.fuse_gae && !a.replay && smem + Cfg::gae_bytes(a.T) <= 232448) {
        a.gae_smem = 1;
        smem += Cfg::gae_bytes(a.T);
    }
    Pair2Maps maps;
    memset(&maps, 0, sizeof(maps));
    if (prec == 0 && !make_tensor_map_2d(&maps.w_lo, a.b.w2p_lo, Cfg::H, Cfg::H, 64, false)) return cudaErrorNotSupported;
    const int pairs = (a.d.B + PER_PAIR - 1) / PER_PAIR;
    const dim3 grid(2 * pairs, replay_slices(a, 2 * pairs));
    if (prec == 1) return a.replay ? launch<k_rollout_pair2<1, true>>(grid, Cfg::THREADS, smem, s, maps, a) : launch<k_rollout_pair2<1, false>>(grid, Cfg::THREADS, smem, s, maps, a);
    return a.replay ? launch<k_rollout_pair2<0, true>>(grid, Cfg::THREADS, smem, s, maps, a) : launch<k_rollout_pair2<0, false>>(grid, Cfg::THREADS, smem, s, maps, a);
}

}  // namespace anakin
