// Persistent rollout on the 5th-generation tensor cores: a pair of CTAs (a cluster of two, on neighbouring SMs) owns
// 64 envs for all T+1 forward passes of a rollout and shares the second-layer weights between its two SMs.
//
// Acting half of the Anakin minimal unit (Podracer paper, Section 3.1; Figure 2, top), hidden width 256; the fp32 form
// (bf16 workloads have one plane of each operand and one MMA per k16).
// The second layer is computed transposed,  D[j][env] = sum_k W2[k][j] h1[env][k],  as tcgen05.mma.cta_group::2 with
// M = 256 hidden units, so that each CTA keeps only ITS 128 columns of W2 on chip (two fp16 planes in TENSOR memory, the A
// operand of every MMA, transposed into it once) and builds only the h1 rows of ITS 32 envs; the tensor cores of the pair read
// both CTAs' h1 rows, and each CTA receives its 128 hidden units x all 64 envs in its own tensor memory.  What bounds a step
// is the chain gather -> layer 1 -> MMAs -> heads -> action, so the agent rows of W1 stay in shared memory on boards of up to
// 144 cells (with W2 in shared memory and these rows in L2 the gather was 950-1900 and the MMAs 2200 clocks of 7400).  Per step:
//   layer 1   h1 = relu(base + W1[agent row])       gather-add; the fp16 (hi, lo) terms go straight into the swizzled
//                                                   K-major operand tile [32 hi rows | 32 lo rows] x 256 k
//   layer 2   two MMAs per k16:  W2hi x [h1hi | h1lo]  (N = 128 over the pair)  and  W2lo x h1hi  (N = 64), fp32
//             accumulators in tensor memory; one thread of the leader CTA issues them for the pair
//   heads     a thread = one hidden unit j: bias, ReLU, h2 stores (one 128-byte line per env and warp); the warp's
//             32 units x 32 envs go to shared memory as fp16 (hi, lo) terms and come back transposed (ldmatrix.trans)
//             as A fragments of warp-level MMAs against Wh: out[env][c] = sum_j h2[j][env] Wh[j][c]; the eight 32-unit
//             partials of an env meet in the shared memory of the CTA that owns it, sent as asynchronous remote stores
//             that count their bytes on the owner's mbarrier
//   env       (ninth warp) one thread per env: softmax, Philox inverse-CDF sample, gridworld step, time-major records
// Inside a step the CTAs of a pair meet only through mbarriers (operand blocks written -> issuer; MMAs finished ->
// workers; partials landed -> owners) and each CTA has one barrier of its own (new positions); the cluster barrier is
// used at start and exit only.  Every mbarrier wait is bounded; a timeout raises DEV_E_WAIT_TIMEOUT and the threads keep
// walking through the barriers to the exit, where tensor memory is freed.
#include <type_traits>

#include "tc_common.cuh"

namespace anakin {

namespace {

// ME: envs per CTA, 32 or 16.  A smaller batch takes 16: the chain of a step has half the operand rows to build, half the MMA
// columns and half the head work, on twice the SMs.
template <int ME_>
struct PairCfg {
    static constexpr int H = 256, ME = ME_, NWORK = 8, THREADS = (NWORK + 1) * 32;
    static constexpr int B_CHUNK = 2 * ME * 128;              // operand rows (ME hi + ME lo) x 64 k
    static constexpr int B_BYTES = (H / 64) * B_CHUNK;
    // [0, 4 ME): W2hi x [hi|lo] of both CTAs, [128, 128 + 2 ME): W2lo x hi; then this CTA's 128 columns of W2 as rows (lane = hidden unit, two
    // k per 32-bit column), hi plane and lo plane
    static constexpr int W_COL = 256, TMEM_COLS = 512;
    static constexpr int W1_CELLS = ME == 32 ? 144 : 169;     // boards whose agent rows of W1 fit in shared memory
    static constexpr size_t fixed_bytes =
        (size_t)B_BYTES + (size_t)ME * H * 4                  // operand tile, base
        + 64                                                  // barriers, tensor-memory slot
        + (size_t)8 * ME * 6 * 4                              // head partials: 8 blocks of 32 hidden units
        + 8 * 4 + (size_t)ME * 8 * 4 + ME * 4;                // bh, walls, pos
    static constexpr size_t gae_bytes(int T) { return (size_t)(T + 1) * ME * 4 + (size_t)T * ME; }
};

// Asynchronous store of two floats into the shared memory of a CTA of the cluster; when it has landed it counts its
// eight bytes on the mbarrier (same CTA as the destination), so the reader needs no fence from the writer.
__device__ __forceinline__ void st_async_f32x2(uint32_t cluster_addr, float v0, float v1, uint32_t cluster_bar_addr) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(cluster_addr), "f"(v0), "f"(v1),
                 "r"(cluster_bar_addr)
                 : "memory");
}

template <int ME_, int PREC, bool REPLAY, bool W1S>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PairCfg<ME_>::THREADS, 1) k_rollout_pair(RolloutArgs a) {
    using Cfg = PairCfg<ME_>;
    constexpr int H = Cfg::H, ME = Cfg::ME, NWT = Cfg::NWORK * 32;
    extern __shared__ unsigned char smem_raw[];
    // the dynamic shared memory starts at the same offset in both CTAs, so the rounded base does too
    unsigned char* sm = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* s_bop = sm;
    float* s_base = reinterpret_cast<float*>(s_bop + Cfg::B_BYTES);                 // [ME][H]
    uint64_t* wbar = reinterpret_cast<uint64_t*>(s_base + ME * H);                  // the agent rows of W1 landed
    uint64_t* tfull = wbar + 1;                                                     // this step's MMAs finished
    uint64_t* ready = tfull + 1;   // [2] leader's copy: k blocks 2i, 2i + 1 of both CTAs' operand rows written (16 warps arrive)
    uint64_t* pfull = ready + 2;   // the eight head partials of this CTA's envs have landed (counted in bytes)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(pfull + 1);
    float* s_red = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(wbar) + 64);  // [8][ME][6]
    float* s_bh = s_red + 8 * ME * 6;                                               // [8]
    uint32_t* s_walls = reinterpret_cast<uint32_t*>(s_bh + 8);                      // [ME][8]
    int* s_pos = reinterpret_cast<int*>(s_walls + ME * 8);                          // [ME]
    float* s_w1 = reinterpret_cast<float*>(s_pos + ME);                             // [C][H] (W1S only)
    float* s_gv = s_w1 + (W1S ? a.d.C * H : 0);                                     // [T+1][ME] (a.gae_smem only)
    uint8_t* s_gc = reinterpret_cast<uint8_t*>(s_gv + (a.T + 1) * ME);              // [T][ME]

    const Dims& d = a.d;
    const Buffers& b = a.b;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint32_t rank = tc::cluster_ctarank();
    const int pair = blockIdx.x >> 1;
    const int e0 = pair * 2 * ME + (int)rank * ME;  // this CTA's first env
    const int B = d.B, C = d.C;
    const float* W1 = b.theta_c + d.oW1;
    const bool worker = wid < Cfg::NWORK;

    // ---- prologue
    if (tid == 0) {
        tc::mbar_init(wbar, 1);
        tc::mbar_init(tfull, 1);
        for (int i = 0; i < 2; ++i) tc::mbar_init(&ready[i], 2 * Cfg::NWORK);
        tc::mbar_init(pfull, 1);
        tc::mbar_fence_init();
    }
    if (wid == Cfg::NWORK) tc::tmem_alloc_pair(tmem_slot, Cfg::TMEM_COLS);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    PDL_START();  // (the set-up above runs under the predecessor's tail)
    if (W1S && tid == NWT) {
        tc::mbar_expect_tx(wbar, (uint32_t)(C * H * 4));
        tc::bulk_load(s_w1, W1 + (size_t)C * H, wbar, (uint32_t)(C * H * 4));
    }
    // hidden unit of this thread in the heads phase, and its constants
    const int q = wid & 3, rE = (wid >> 2) & 1;  // accumulator lanes 32q.., envs of CTA rE
    const int j = 128 * (int)rank + 32 * q + lane;
    float b2j = 0.f;
    uint32_t whf_hi[2][2], whf_lo[2][2];  // Wh rows of this warp's 32 hidden units as mma B fragments (k16 x n8), two k steps
    EnvLane s;
    s.pos = s.tep = s.start = s.goal = 0;
    s.n_episodes = s.n_goals = s.n_epsteps = 0;
    s.bad = 0;
    const int ow = tid - NWT;  // warp 8: lane = env of this CTA (its lane 0 also issues the pair's MMAs)
    const bool owner = ow >= 0 && ow < ME && e0 + ow < B;
    if (worker) {
        for (int i = tid; i < ME * H / 4; i += NWT) {
            const int e = i / (H / 4), k = 4 * (i - e * (H / 4));
            const bool okb = e0 + e < B;
            cp_async16(s_base + e * H + k, b.base + (size_t)(okb ? e0 + e : 0) * H + k, okb ? 16 : 0);
        }
        cp_async_commit();
        // W2 into tensor memory, transposed: lane = hidden unit j, 32-bit column = k 2c (low half), 2c + 1.  The two warps of a lane
        // quarter take 64 columns each of every plane.
#pragma unroll 1
        for (int pc = 0; pc < (PREC == 0 ? 4 : 2); ++pc) {
            const int col0 = 64 * rE + 32 * (pc & 1);
            const uint16_t* src = ((pc >> 1) ? b.w2p_lo : b.w2p_hi) + (size_t)(2 * col0) * H + j;
            uint32_t r[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) r[c] = (uint32_t)__ldg(src + (size_t)(2 * c) * H) | ((uint32_t)__ldg(src + (size_t)(2 * c + 1) * H) << 16);
            tc::tmem_st32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(Cfg::W_COL + 128 * (pc >> 1) + col0), r);
        }
        tc::tmem_st_wait();
        tc::tc_fence_before();
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
    } else {
        if (ow < ME)
            for (int wi = 0; wi < 8; ++wi) s_walls[ow * 8 + wi] = (owner && wi < d.W) ? b.walls[(size_t)(e0 + ow) * d.W + wi] : 0u;
        if (owner) {
            s.pos = b.pos[e0 + ow];
            s.tep = b.tep[e0 + ow];
            s.start = b.start[e0 + ow];
            s.goal = b.goal[e0 + ow];
            check_env_state(s, C, s_walls + ow * 8);
        }
        if (ow < ME) s_pos[ow] = s.pos;
    }
    bool ok = true;
    if (W1S) ok = tc::mbar_wait(wbar, 0);
    __syncthreads();
    tc::cluster_sync_all();  // both CTAs' barriers, tensor memory and weights exist before the first MMA
    tc::tc_fence_after();

    __nv_bfloat16* g_h1hi = reinterpret_cast<__nv_bfloat16*>(b.h1);
    __nv_bfloat16* g_h1lo = g_h1hi + (size_t)B * d.Tmax * H;
    const uint32_t idesc_w = tc::umma_idesc<PREC>(256, 4 * ME, false, false), idesc_n = tc::umma_idesc<PREC>(256, 2 * ME, false, false);

    // Replay recomputes the T recorded rows (mode 2: and the current state), in independent slices of steps (grid.y).
    const int t_last = REPLAY && a.replay == 1 ? a.T - 1 : a.T, t_len = REPLAY ? (t_last + (int)gridDim.y) / (int)gridDim.y : 0;
    const int t_beg = REPLAY ? (int)blockIdx.y * t_len : 0, t_end = REPLAY ? min(t_last, t_beg + t_len - 1) : t_last;
    for (int t = t_beg; t <= t_end; ++t) {
        if (REPLAY) {  // positions come from the recorded trajectory
            if (ow >= 0 && ow < ME) s_pos[ow] = owner ? min((int)(t < a.T ? b.tpos[(size_t)t * B + e0 + ow] : b.pos[e0 + ow]), C - 1) : 0;
            __syncthreads();
        }
        if (tid == NWT) tc::mbar_expect_tx(pfull, 8 * ME * 6 * 4);  // this step's head partials, counted as they land
        // ---- layer 1 (workers): 16-byte chunks of eight hidden units.  Trip kb covers k block kb (64 hidden units of layer 1)
        // (ME = 16: warps 0-3 the even blocks, warps 4-7 the odd ones) of all envs: chunk c8 of env e goes to operand row e (hi)
        // and ME + e (lo) of that block, at the 16-byte position
        // c8 ^ (e % 8) of the 128-byte row (the 128-byte swizzle of a K-major operand).  Two finished blocks are announced to
        // the issuer together (the proxy fence costs some 300 clocks each time), so the tensor cores start on the first two
        // while the others are being written.  Lanes 4-7 of an env read their two 16-byte pieces of a row in the other order,
        // so that the eight lanes cover all banks.
        if (worker) {
            const int e = (tid >> 3) % ME, c8 = tid & 7, sw = (c8 >> 2) & 1;
            constexpr int NB = ME / 8;  // chunks of this thread: block kb_of(0), kb_of(1), ...
            auto kb_of = [&](int i) { return ME == 32 ? i : 2 * i + (wid >> 2); };
            uint4 hi[NB], lo[NB];
            const float* wrow = (W1S ? s_w1 + (size_t)s_pos[e] * H : W1 + (size_t)(C + s_pos[e]) * H) + 8 * c8;
            const float* brow = s_base + e * H + 8 * c8;
            float4 w[NB][2];
            if (!W1S) {  // all gathers of the agent's W1 row are in flight before any is used
#pragma unroll
                for (int i = 0; i < NB; ++i) {
                    w[i][0] = __ldg(reinterpret_cast<const float4*>(wrow + 64 * kb_of(i) + 4 * sw));
                    w[i][1] = __ldg(reinterpret_cast<const float4*>(wrow + 64 * kb_of(i) + 4 * (sw ^ 1)));
                }
            }
            tc::tc_fence_before();  // this thread's reads of last step's accumulators precede the arrivals below
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const int kb = kb_of(i);
                if (W1S) {
                    w[i][0] = *reinterpret_cast<const float4*>(wrow + 64 * kb + 4 * sw);
                    w[i][1] = *reinterpret_cast<const float4*>(wrow + 64 * kb + 4 * (sw ^ 1));
                }
                const float4 b0 = *reinterpret_cast<const float4*>(brow + 64 * kb + 4 * sw);
                const float4 b1 = *reinterpret_cast<const float4*>(brow + 64 * kb + 4 * (sw ^ 1));
                uint2 h0, h1, l0, l1;
                split2<PREC>(fmaxf(b0.x + w[i][0].x, 0.f), fmaxf(b0.y + w[i][0].y, 0.f), h0.x, l0.x);
                split2<PREC>(fmaxf(b0.z + w[i][0].z, 0.f), fmaxf(b0.w + w[i][0].w, 0.f), h0.y, l0.y);
                split2<PREC>(fmaxf(b1.x + w[i][1].x, 0.f), fmaxf(b1.y + w[i][1].y, 0.f), h1.x, l1.x);
                split2<PREC>(fmaxf(b1.z + w[i][1].z, 0.f), fmaxf(b1.w + w[i][1].w, 0.f), h1.y, l1.y);
                hi[i] = sw ? make_uint4(h1.x, h1.y, h0.x, h0.y) : make_uint4(h0.x, h0.y, h1.x, h1.y);
                lo[i] = sw ? make_uint4(l1.x, l1.y, l0.x, l0.y) : make_uint4(l0.x, l0.y, l1.x, l1.y);
                unsigned char* row = s_bop + kb * Cfg::B_CHUNK + e * 128 + ((c8 ^ (e & 7)) << 4);
                *reinterpret_cast<uint4*>(row) = hi[i];
                if (PREC == 0) *reinterpret_cast<uint4*>(row + ME * 128) = lo[i];
                if (ME == 16 || (i & 1)) {
                    tc::fence_proxy_async();  // ordinary stores -> visible to the tensor cores
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive_remote_cta_release(tc::mapa(tc::smem_u32(&ready[ME == 16 ? i : i >> 1]), 0));
                }
            }
            // the copies for the update leave after the arrivals (their CTA-scope release does not wait for global stores)
            if (b.h1 != nullptr && t < a.T && e0 + e < B) {
#pragma unroll
                for (int i = 0; i < NB; ++i) {
                    const size_t gi = ((size_t)t * B + e0 + e) * H + 64 * kb_of(i) + 8 * c8;
                    *reinterpret_cast<uint4*>(g_h1hi + gi) = hi[i];
                    if (PREC == 0) *reinterpret_cast<uint4*>(g_h1lo + gi) = lo[i];
                    if (b.gate1) b.gate1[gi >> 3] = (uint8_t)nonzero_bits16(hi[i]);  // the gates of these eight units
                }
            }
        }
        // the logits-independent half of the interaction, taken by the owner warp while the workers gather
        const bool acting = owner && !REPLAY && t < a.T;
        StepPre pre;
        if (acting) pre = step_prepare(s, a, e0 + ow, t, s_walls + ow * 8);
        // ---- layer 2: the leader's owner warp drives both tensor cores, two k blocks at a time (the whole warp waits, one elected
        // lane issues).  Their sixteen arrivals also say that those warps have read last step's accumulators.
        if (!worker && rank == 0) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                ok = tc::warp_all(ok && tc::mbar_wait_cluster(&ready[i], (uint32_t)(t - t_beg) & 1u));
                tc::tc_fence_after();
                if (tc::elect_one()) {
#pragma unroll
                    for (int k16 = 8 * i; k16 < 8 * i + 8; ++k16) {
                        // A: 16 k = 8 columns.  B (K-major): 16 k = 32 bytes along the swizzled rows, 1024 bytes between 8-row groups
                        const uint32_t ahi = tmem + (uint32_t)(Cfg::W_COL + 8 * k16), alo = ahi + 128u;
                        const uint64_t bd = tc::umma_desc(s_bop + (k16 >> 2) * Cfg::B_CHUNK + (k16 & 3) * 32, 16, 1024);
                        if (PREC == 0) {
                            tc::umma_pair_ta(tmem, ahi, bd, idesc_w, k16 ? 1u : 0u);
                            tc::umma_pair_ta(tmem + 128u, alo, bd, idesc_n, k16 ? 1u : 0u);
                        } else {  // bf16 operands: one product, the hi rows of the operand tile only
                            tc::umma_pair_ta(tmem, ahi, bd, idesc_n, k16 ? 1u : 0u);
                        }
                    }
                    if (i == 1) tc::umma_commit_pair(tfull, 3);
                }
                __syncwarp();
            }
        }
        // ---- heads (workers): thread = hidden unit j, the ME envs of CTA rE
        if (worker) {
            if (ok) ok = tc::mbar_wait(tfull, (uint32_t)(t - t_beg) & 1u);
            tc::tc_fence_after();
            float v[ME];
            {
                uint32_t r0[ME], r1[ME], r2[ME];
                const uint32_t lanes = tmem + ((uint32_t)(32 * q) << 16);
                auto load = [&](uint32_t col, uint32_t (&x)[ME]) {
                    if constexpr (ME == 32) tc::tmem_ld32_nowait(lanes + col, x);
                    else tc::tmem_ld16_nowait(lanes + col, x);
                };
                load((uint32_t)((PREC == 0 ? 2 * ME : ME) * rE), r0);  // W2hi x h1hi
                if (PREC == 0) {
                    load((uint32_t)(2 * ME * rE + ME), r1);    // W2hi x h1lo
                    load(128u + (uint32_t)(ME * rE), r2);      // W2lo x h1hi
                }
                tc::tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < ME; ++e) {
                    float z = __uint_as_float(r0[e]);
                    if (PREC == 0) z = (z + __uint_as_float(r1[e])) + __uint_as_float(r2[e]);
                    v[e] = rnd<PREC>(fmaxf(z + b2j, 0.f));
                }
            }
            // head partials over this warp's 32 hidden units on the warp-level tensor path.  The operand tile is free
            // once the step's MMAs have finished: warp w keeps [32 units][ME envs] fp16 hi and lo planes in its eighth of it,
            // rows of 64 (32) bytes whose 16-byte chunks are XOR-swizzled by (row / 2) % 4 ((row / 4) % 2): conflict-free both ways.
            unsigned char* wsm = s_bop + wid * (Cfg::B_BYTES / 8);
            constexpr int PLANE = 32 * 2 * ME;
            auto stage_off = [](int unit, int chunk) { return unit * (2 * ME) + ((ME == 32 ? chunk ^ ((unit >> 1) & 3) : chunk ^ ((unit >> 2) & 1)) << 4); };
#pragma unroll
            for (int c4 = 0; c4 < ME / 8; ++c4) {
                uint4 hi, lo;
                split2<PREC>(v[8 * c4 + 0], v[8 * c4 + 1], hi.x, lo.x);
                split2<PREC>(v[8 * c4 + 2], v[8 * c4 + 3], hi.y, lo.y);
                split2<PREC>(v[8 * c4 + 4], v[8 * c4 + 5], hi.z, lo.z);
                split2<PREC>(v[8 * c4 + 6], v[8 * c4 + 7], hi.w, lo.w);
                const int off = stage_off(lane, c4);
                *reinterpret_cast<uint4*>(wsm + off) = hi;
                if (PREC == 0) *reinterpret_cast<uint4*>(wsm + PLANE + off) = lo;
            }
            __syncwarp();
            constexpr int MT = ME / 16;
            float acc[MT][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
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
                    for (int mt = 0; mt < MT; ++mt) {
                        const int chunk = 2 * mt + (mi & 1);
                        const int off = stage_off(krow, chunk);
                        uint32_t ahi[4], alo[4];
                        ldmatrix_x4_trans(ahi, wsm + off);
                        if (PREC == 0) ldmatrix_x4_trans(alo, wsm + PLANE + off);
                        // the x4 order above is (k lo, m lo), (k lo, m hi), (k hi, m lo), (k hi, m hi) = a0, a1, a2, a3
                        if (PREC == 0) {
                            mma16816<PREC>(acc[mt], alo, whf_hi[ks][0], whf_hi[ks][1]);
                            mma16816<PREC>(acc[mt], ahi, whf_lo[ks][0], whf_lo[ks][1]);
                        }
                        mma16816<PREC>(acc[mt], ahi, whf_hi[ks][0], whf_hi[ks][1]);
                    }
                }
            }
            // accumulator element (row g + 8hh of tile mt, column 2 t4 + cc) = (env 16mt + 8hh + g, head 2 t4 + cc)
            {
                const int g = lane >> 2, t4 = lane & 3;
                const uint32_t pbar = tc::mapa(tc::smem_u32(pfull), (uint32_t)rE);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const int e = 16 * mt + 8 * hh + g;
                        const uint32_t dst = tc::mapa(tc::smem_u32(s_red + ((4 * (int)rank + q) * ME + e) * 6 + 2 * t4), (uint32_t)rE);
                        if (t4 < 3) st_async_f32x2(dst, acc[mt][2 * hh], acc[mt][2 * hh + 1], pbar);
                    }
            }
            // h2 for the update: one 128-byte line per env
            const int env0 = pair * 2 * ME + rE * ME;  // first env of the block this warp holds
            if (b.h2 != nullptr && t < a.T) {
#pragma unroll
                for (int e = 0; e < ME; ++e)
                    if (env0 + e < B) b.h2[((size_t)t * B + env0 + e) * H + j] = v[e];
            }
        }
        // ---- one thread per env: once the eight partials are in, their fixed-order sum, then act and step
        if (!worker && ok) ok = tc::mbar_wait_cluster(pfull, (uint32_t)(t - t_beg) & 1u);
        // The new positions are all the next step's gather needs: the owners publish them and release the workers (named
        // barrier 1: the workers wait on it, the owner warp only arrives, once and as a whole warp) before they write the
        // step's records.
        if (!worker) {
            float o[5];
#pragma unroll
            for (int c = 0; c < 5; ++c) o[c] = 0.f;
            ActOut ao;
            ao.la_mx = ao.Z = ao.rew = 0.f;
            ao.act = ao.done = ao.pos0 = 0;
            const int env = e0 + ow;
            if (owner) {
#pragma unroll
                for (int blk = 0; blk < 8; ++blk) {
                    const float2* p2 = reinterpret_cast<const float2*>(s_red + (blk * ME + ow) * 6);
                    const float2 x0 = p2[0], x1 = p2[1];
                    o[0] += x0.x; o[1] += x0.y; o[2] += x1.x; o[3] += x1.y;
                    o[4] += s_red[(blk * ME + ow) * 6 + 4];
                }
#pragma unroll
                for (int c = 0; c < 5; ++c) o[c] += s_bh[c];
                if (acting) {
                    ao = act_decide(s, a, env, t, o[0], o[1], o[2], o[3], pre);
                    s_pos[ow] = s.pos;
                }
            }
            __syncwarp();
            asm volatile("bar.arrive 1, %0;" ::"n"(Cfg::THREADS) : "memory");
            if (owner) {
                if (b.out5 && t < a.T) {  // the update reuses the head outputs of every recorded row
                    float4* o5 = reinterpret_cast<float4*>(b.out5 + ((size_t)t * B + env) * 8);
                    o5[0] = make_float4(o[0], o[1], o[2], o[3]);
                    o5[1] = make_float4(o[4], 0.f, 0.f, 0.f);
                }
                if (REPLAY && a.replay == 2 && t == a.T) b.vboot[env] = o[4];
                if (!REPLAY) {
                    b.tval[(size_t)t * B + env] = o[4];
                    if (a.gae_smem) s_gv[t * ME + ow] = o[4];
                }
                if (acting) {
                    act_record(a, env, t, o[0], o[1], o[2], o[3], ao);
                    if (a.gae_smem) s_gc[t * ME + ow] = (uint8_t)(ao.done | (ao.rew != 0.f ? 2 : 0));
                }
            }
        } else {
            // every worker is done with its staging area in the operand tile, and the positions are in place
            asm volatile("bar.sync 1, %0;" ::"n"(Cfg::THREADS) : "memory");
        }
    }
    if (owner && !REPLAY) {
        b.pos[e0 + ow] = (uint8_t)s.pos;
        b.tep[e0 + ow] = (uint8_t)s.tep;
        if (a.gae_smem) gae_scan_env_smem(b, B, a.T, e0 + ow, a.gamma, a.lambda, s_gv, s_gc, ME, ow);
        else if (a.fuse_gae) gae_scan_env(b, B, a.T, e0 + ow, a.gamma, a.lambda);
    }
    if (!worker && !REPLAY) flush_env_stats(s, a);
    if (!ok && lane == 0) atomicOr(b.status, DEV_E_WAIT_TIMEOUT);
    // neither CTA frees tensor memory or leaves while the other may still signal it
    tc::tc_fence_before();
    __syncthreads();
    tc::cluster_sync_all();
    if (wid == Cfg::NWORK) tc::tmem_dealloc_pair(tmem, Cfg::TMEM_COLS);
}

}  // namespace

template <int ME>
static cudaError_t launch_pair(const RolloutArgs& a0, int prec, cudaStream_t s) {
    using Cfg = PairCfg<ME>;
    RolloutArgs a = a0;
    const bool w1s = a.d.C <= Cfg::W1_CELLS;  // (larger boards gather from L2)
    size_t smem = Cfg::fixed_bytes + 1024 /*alignment slack*/ + (w1s ? (size_t)a.d.C * Cfg::H * 4 : 0);
    a.gae_smem = 0;
    if (a.fuse_gae && !a.replay && smem + Cfg::gae_bytes(a.T) <= 232448) {
        a.gae_smem = 1;
        smem += Cfg::gae_bytes(a.T);
    }
    const int pairs = (a.d.B + 2 * ME - 1) / (2 * ME);
    const dim3 grid(2 * pairs, replay_slices(a, 2 * pairs));
    auto go = [&](auto w1) {
        constexpr bool W = decltype(w1)::value;
        if constexpr (ME == 32) {
            if (a.replay) return prec == 1 ? launch<k_rollout_pair<ME, 1, true, W>>(grid, Cfg::THREADS, smem, s, a) : launch<k_rollout_pair<ME, 0, true, W>>(grid, Cfg::THREADS, smem, s, a);
        }
        return prec == 1 ? launch<k_rollout_pair<ME, 1, false, W>>(grid, Cfg::THREADS, smem, s, a) : launch<k_rollout_pair<ME, 0, false, W>>(grid, Cfg::THREADS, smem, s, a);
    };
    return w1s ? go(std::true_type{}) : go(std::false_type{});
}

// Hidden width 256 in either precision, given the row-major 16-bit planes of W2; cudaErrorNotSupported otherwise.
cudaError_t launch_rollout_pair(const RolloutArgs& a, int prec, cudaStream_t s) {
    if (a.d.H != 256 || !a.b.w2p_hi || (prec == 0 && !a.b.w2p_lo) || !a.b.base) return cudaErrorNotSupported;
    // 16 envs per CTA while one wave of pairs covers the batch
    return !a.replay && a.d.B <= 74 * 32 ? launch_pair<16>(a, prec, s) : launch_pair<32>(a, prec, s);
}

}  // namespace anakin
