// Persistent rollout on the tensor pipe (warp-level mma.sync), second-layer weights resident on chip: hidden widths 32, 64, 96, 128
// and 192, and many policies.  (128 beyond one wave of batches: rollout_tc128.cu; 256: rollout_pair.cu, rollout_pair2.cu.)
//
// Acting half of the Anakin minimal unit (Podracer paper, Section 3.1; Figure 2, top).  A CTA owns 32 envs, or 16 in small batches,
// for all T+1 forward passes of a rollout; nothing is exchanged between CTAs.  Per step:
//   layer 1   h1 = relu(base + W1[agent row])            gather-add, written to smem as 16-bit (hi, lo) planes
//   layer 2   h2 = relu(h1 W2 + b2)                      mma.sync m16n8k16; warp w owns output columns [NC*w, NC*w+NC)
//   heads     out = h2 Wh + bh                           fp32 FMA on the accumulator fragments, fixed-order reduction
//   env       softmax, Philox inverse-CDF sample, gridworld step, time-major records   (one thread per env)
// fp32 workloads at 64 and 128 use a two-term fp16 split of both operands and three MMAs per product (hi*hi + lo*hi + hi*lo,
// fp32 accumulate), at 32, 96 and 192 three bf16 terms and six MMAs.  W2's leading B-fragments stay in shared memory and those of
// its last term in registers for the whole kernel, so after the prologue the loop touches no weight bytes beyond the
// agent's W1 row (from L2, or from shared memory where the launch says so).  The bf16 workload needs one MMA per product.
#include "env_step.cuh"

namespace anakin {

// B fragments of W2 for mma.m16n8k16 (.col B): entry [(ks*(H/8) + nt)*32 + lane] holds, for g = lane/4, t = lane%4,
// n = 8*nt + g:  x = {W2[16ks+2t][n], W2[16ks+2t+1][n]},  y = {W2[16ks+2t+8][n], W2[16ks+2t+9][n]}  (low half first).
template <int PREC, bool GROUPED>
__global__ void __launch_bounds__(256) k_pack_w2(DimsBuffers in) {
    PDL_START();
    const PolicyArgs<GROUPED, DimsBuffers> pa(in, blockIdx.y);  // many policies: grid.y = policy
    const Dims& d = pa.a.d;
    const Buffers& b = pa.a.b;
    const int H = d.H;
    const int total = H * H / 4;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int lane = idx & 31, nt = (idx >> 5) % (H / 8), ks = (idx >> 5) / (H / 8);
    const int g = lane >> 2, t = lane & 3;
    const int n = nt * 8 + g, k0 = ks * 16 + 2 * t;
    const float* W2 = b.theta_c + d.oW2;
    if (b.w2f_hi) {
        const int ks4[4] = {k0, k0 + 1, k0 + 8, k0 + 9};
        if constexpr (PREC == 2) {
            uint32_t x[3], y[3];
            split3(W2[(size_t)ks4[0] * H + n], W2[(size_t)ks4[1] * H + n], x);
            split3(W2[(size_t)ks4[2] * H + n], W2[(size_t)ks4[3] * H + n], y);
            b.w2f_hi[idx] = make_uint2(x[0], y[0]);
            b.w2f_lo[idx] = make_uint2(x[1], y[1]);
            b.w2f_lo2[idx] = make_uint2(x[2], y[2]);
        } else {
            uint2 hi, lo;
            split2<PREC>(W2[(size_t)ks4[0] * H + n], W2[(size_t)ks4[1] * H + n], hi.x, lo.x);
            split2<PREC>(W2[(size_t)ks4[2] * H + n], W2[(size_t)ks4[3] * H + n], hi.y, lo.y);
            b.w2f_hi[idx] = hi;
            b.w2f_lo[idx] = lo;
        }
    }
    // and W2 itself as row-major hi / lo planes: this thread covers elements 4*idx .. 4*idx+3
    if (!b.w2p_hi || (PREC != 2 && !b.w2p_lo)) return;
    if constexpr (PREC == 2) {  // three planes one after the other
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            uint32_t tm[3];
            split3(W2[(size_t)4 * idx + 2 * q], W2[(size_t)4 * idx + 2 * q + 1], tm);
            for (int p = 0; p < 3; ++p) reinterpret_cast<uint32_t*>(b.w2p_hi + (size_t)p * H * H)[2 * idx + q] = tm[p];
        }
    } else
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint16_t h16, l16;
        split1<PREC == 1 ? 1 : 0>(W2[(size_t)4 * idx + q], h16, l16);
        b.w2p_hi[(size_t)4 * idx + q] = h16;
        b.w2p_lo[(size_t)4 * idx + q] = l16;
    }
}

cudaError_t launch_pack_w2(const Dims& d, const Buffers& b, int prec, const Ctx& c) {
    if (!b.w2f_hi && !b.w2p_hi) return cudaSuccess;
    Scope sc(c, K_PACK_W2);
    const unsigned nb = (d.H * d.H / 4 + 255) / 256;
    if (d.npol > 1) {
        if (prec == 1) return cudaErrorNotSupported;
        launch<k_pack_w2<0, true>>(dim3(nb, d.npol), 256, 0, c.s, DimsBuffers{d, b});
    } else if (prec == 1) launch<k_pack_w2<1, false>>(nb, 256, 0, c.s, DimsBuffers{d, b});
    else if (three_terms(d.H, prec)) launch<k_pack_w2<2, false>>(nb, 256, 0, c.s, DimsBuffers{d, b});
    else launch<k_pack_w2<0, false>>(nb, 256, 0, c.s, DimsBuffers{d, b});
    return cudaGetLastError();
}

template <int H, int NW, int PREC, int ME_ = 32>
struct RolloutMmaCfg {
    static constexpr int ME = ME_;           // envs per CTA (two m16 tiles, or one: see the launch)
    static constexpr int MT = ME / 16;
    static constexpr int NC = H / NW;        // output columns per warp
    static constexpr int NT = NC / 8;        // n8 tiles per warp
    static constexpr int KS = H / 16;        // k16 steps
    static constexpr int LD = H + 8;         // bf16 row pitch of the h1 planes (16-byte skew: conflict-free ldmatrix)
    static constexpr int PLANES = PREC == 1 ? 1 : PREC == 2 ? 3 : 2;
    static constexpr int WSM = PREC == 2 ? 2 : 1;  // planes of W2 fragments in shared memory (the last plane: registers)
    static constexpr size_t smem_bytes =
        (size_t)H * H * 2 * WSM              // W2 leading fragments
        + (size_t)ME * H * 4                 // base
        + (size_t)PLANES * ME * LD * 2       // h1 hi (and lo)
        + (size_t)NW * ME * 5 * 4            // per-warp head partials
        + (size_t)(H * 5 + H + 8) * 4        // Wh, b2, bh
        + (size_t)ME * 8 * 4 + ME * 4        // walls, pos
        + (size_t)ME * 8;                    // prepared half of the next interaction
    // values and outcomes of the CTA's envs for the GAE scan at the end (only when the scan is fused and they fit)
    static constexpr size_t gae_bytes(int T) { return (size_t)(T + 1) * ME * 4 + (size_t)T * ME; }
};

// OWN: the per-env part of a step (one lane per env) has a warp of its own beside the NW workers, which meets them at named
// barriers: the logits-independent half of an interaction runs under the gather, and the records are written after the workers
// have been given the new positions.  Otherwise warp 0 does both (the wide kernels' registers leave no room for another warp).
// W1S: the agent rows of W1 in shared memory (the gather from L2 is a quarter of a small batch's step).
template <int H, int NW, int PREC, bool GROUPED, int MINB, bool OWN, bool REPLAY, int ME_, bool W1S>
__global__ void __launch_bounds__(NW * 32 + (OWN ? 32 : 0), MINB) k_rollout_mma(RolloutArgs a_in) {
    pdl_wait();
    const PolicyArgs<GROUPED, RolloutArgs> pa(a_in, blockIdx.y);  // many policies: grid.y = policy
    const RolloutArgs& a = pa.a;
    using Cfg = RolloutMmaCfg<H, NW, PREC, ME_>;
    constexpr int ME = Cfg::ME, MT = Cfg::MT, NT = Cfg::NT, KS = Cfg::KS, LD = Cfg::LD, NTHREADS = NW * 32 /*workers*/, NALL = NTHREADS + (OWN ? 32 : 0);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint2* s_w2hi = reinterpret_cast<uint2*>(smem_raw);                        // [KS][H/8][32]
    uint2* s_w2mid = s_w2hi + (size_t)H * H / 4;                               // (PREC 2) the second terms
    float* s_base = reinterpret_cast<float*>(smem_raw + (size_t)H * H * 2 * Cfg::WSM);  // [ME][H]
    __nv_bfloat16* s_h1hi = reinterpret_cast<__nv_bfloat16*>(s_base + ME * H); // [ME][LD]
    __nv_bfloat16* s_h1lo = s_h1hi + (PREC == 1 ? 0 : ME * LD);               // [ME][LD] (fp32 workloads only)
    __nv_bfloat16* s_h1lo2 = s_h1hi + (PREC == 2 ? 2 * ME * LD : 0);           // (PREC 2)
    float* s_red = reinterpret_cast<float*>(s_h1hi + Cfg::PLANES * ME * LD);   // [NW][ME][5]
    float* s_wh = s_red + NW * ME * 5;                                         // [H][5]
    float* s_b2 = s_wh + H * 5;                                                // [H]
    float* s_bh = s_b2 + H;                                                    // [8]
    uint32_t* s_walls = reinterpret_cast<uint32_t*>(s_bh + 8);                 // [ME][8]
    int* s_pos = reinterpret_cast<int*>(s_walls + ME * 8);                     // [ME]
    uint2* s_pre = reinterpret_cast<uint2*>(s_pos + ME);                       // [ME]
    float* s_gv = reinterpret_cast<float*>(s_pre + ME);                        // [T+1][ME] (a.gae_smem only)
    uint8_t* s_gc = reinterpret_cast<uint8_t*>(s_gv + (a.T + 1) * ME);         // [T][ME]
    float* s_w1 = a.gae_smem ? reinterpret_cast<float*>(s_gc + a.T * ME) : s_gv;  // [C][H] (W1S only)

    const Dims& d = a.d;
    const Buffers& b = a.b;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int g = lane >> 2, t4 = lane & 3;
    const int e0 = blockIdx.x * ME;
    const int B = d.B, C = d.C;
    const float* W1 = b.theta_c + d.oW1;

    const int ow = OWN ? tid - NTHREADS : tid;  // env of this thread (0 .. ME-1: an owner)
    const bool worker = !OWN || tid < NTHREADS, ownw = ow >= 0 && ow < ME;

    // ---- prologue: weights and per-env constants on chip
    // asynchronous copies: every 16-byte chunk is in flight at once, nothing is staged in registers
    for (int i = tid; i < H * H * 2 / 16; i += NALL) cp_async16(reinterpret_cast<uint4*>(s_w2hi) + i, reinterpret_cast<const uint4*>(b.w2f_hi) + i, 16);
    if (PREC == 2)
        for (int i = tid; i < H * H * 2 / 16; i += NALL) cp_async16(reinterpret_cast<uint4*>(s_w2mid) + i, reinterpret_cast<const uint4*>(b.w2f_lo) + i, 16);
    for (int i = tid; i < ME * H / 4; i += NALL) {
        const int e = i / (H / 4), j = 4 * (i - e * (H / 4));
        const bool ok = e0 + e < B;
        cp_async16(s_base + e * H + j, b.base + (size_t)(ok ? e0 + e : 0) * H + j, ok ? 16 : 0);
    }
    if (W1S)
        for (int i = tid; i < C * H / 4; i += NALL) cp_async16(s_w1 + 4 * i, W1 + (size_t)C * H + 4 * i, 16);
    cp_async_commit();
    for (int i = tid; i < H * 5; i += NALL) s_wh[i] = b.theta_c[d.oWh + i];
    for (int i = tid; i < H; i += NALL) s_b2[i] = b.theta_c[d.ob2 + i];
    if (tid < 5) s_bh[tid] = b.theta_c[d.obh + tid];
    uint2 blo[PREC == 1 ? 1 : KS][NT];
    if (PREC != 1 && worker) {
        const uint2* last = PREC == 2 ? b.w2f_lo2 : b.w2f_lo;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int j = 0; j < NT; ++j) blo[ks][j] = last[(ks * (H / 8) + wid * NT + j) * 32 + lane];
    }
    EnvLane s;
    s.pos = s.tep = s.start = s.goal = 0;
    s.n_episodes = s.n_goals = s.n_epsteps = 0;
    s.bad = 0;
    const bool owner = ownw && e0 + ow < B;
    if (ownw) {
        for (int wi = 0; wi < 8; ++wi) s_walls[ow * 8 + wi] = (owner && wi < d.W) ? b.walls[(size_t)(e0 + ow) * d.W + wi] : 0u;
        if (owner) {
            s.pos = b.pos[e0 + ow];
            s.tep = b.tep[e0 + ow];
            s.start = b.start[e0 + ow];
            s.goal = b.goal[e0 + ow];
            check_env_state(s, C, s_walls + ow * 8);
        }
        s_pos[ow] = s.pos;
    }
    cp_async_wait<0>();
    __syncthreads();

    // Saved activations (the update reuses the policy's forward pass: Section 3.1): row i = t*B + env.
    __nv_bfloat16* g_h1hi = reinterpret_cast<__nv_bfloat16*>(b.h1);
    const size_t h1_plane = (size_t)B * d.Tmax * H;
    // Replay recomputes the T recorded rows (mode 2: and the current state).  Its steps are independent of one another, so a
    // launch for few envs cuts them into slices (grid.y).
    constexpr bool SLICED = REPLAY && !GROUPED;
    const int t_last = REPLAY && a.replay == 1 ? a.T - 1 : a.T, t_len = SLICED ? (t_last + (int)gridDim.y) / (int)gridDim.y : 0;
    const int t_beg = SLICED ? (int)blockIdx.y * t_len : 0, t_end = SLICED ? min(t_last, t_beg + t_len - 1) : t_last;
    auto recorded_pos = [&](int t) {  // replay: the position of this thread's env at step t (row T: the env state as it stands)
        return owner ? min((int)(t < a.T ? b.tpos[(size_t)t * B + e0 + ow] : b.pos[e0 + ow]), C - 1) : 0;
    };
    if (REPLAY) {
        if (ownw) s_pos[ow] = recorded_pos(t_beg);
        __syncthreads();
    }
    auto layer1 = [&](int t) {
        // ---- layer 1: eight consecutive hidden units per thread and trip.  All gathers of the agent's W1 row are issued
        // before any is used (one L2 round trip per step, not one per trip); the fp16 planes go to shared memory for
        // the MMAs and, for the update's reuse, straight to global memory (16 bytes per lane).
        {
            constexpr int TRIPS = ME * H / 8 / NTHREADS;
            static_assert(TRIPS * NTHREADS == ME * H / 8, "layer-1 trips must tile the h1 block");
            const bool save_h1 = b.h1 != nullptr && t < a.T;
            float4 w[TRIPS][2];
#pragma unroll
            for (int i = 0; i < TRIPS; ++i) {
                const int p = tid + i * NTHREADS;
                const int e = p / (H / 8), k = 8 * (p - e * (H / 8));
                if (W1S) {
                    const float4* wp = reinterpret_cast<const float4*>(s_w1 + s_pos[e] * H + k);
                    w[i][0] = wp[0];
                    w[i][1] = wp[1];
                } else {
                    const float4* wp = reinterpret_cast<const float4*>(W1 + (size_t)(C + s_pos[e]) * H + k);
                    w[i][0] = __ldg(wp);
                    w[i][1] = __ldg(wp + 1);
                }
            }
#pragma unroll
            for (int i = 0; i < TRIPS; ++i) {
                const int p = tid + i * NTHREADS;
                const int e = p / (H / 8), k = 8 * (p - e * (H / 8));
                const float4 b0 = *reinterpret_cast<const float4*>(s_base + e * H + k);
                const float4 b1 = *reinterpret_cast<const float4*>(s_base + e * H + k + 4);
                const bool save = save_h1 && e0 + e < B;
                const size_t gi = ((size_t)t * B + e0 + e) * H + k;
                if constexpr (PREC == 2) {
                    uint32_t x[4][3];
                    split3(fmaxf(b0.x + w[i][0].x, 0.f), fmaxf(b0.y + w[i][0].y, 0.f), x[0]);
                    split3(fmaxf(b0.z + w[i][0].z, 0.f), fmaxf(b0.w + w[i][0].w, 0.f), x[1]);
                    split3(fmaxf(b1.x + w[i][1].x, 0.f), fmaxf(b1.y + w[i][1].y, 0.f), x[2]);
                    split3(fmaxf(b1.z + w[i][1].z, 0.f), fmaxf(b1.w + w[i][1].w, 0.f), x[3]);
#pragma unroll
                    for (int p3 = 0; p3 < 3; ++p3) {
                        const uint4 v = make_uint4(x[0][p3], x[1][p3], x[2][p3], x[3][p3]);
                        *reinterpret_cast<uint4*>(s_h1hi + p3 * ME * LD + e * LD + k) = v;
                        if (save) *reinterpret_cast<uint4*>(g_h1hi + p3 * h1_plane + gi) = v;
                    }
                } else {
                    uint4 hi, lo;
                    split2<PREC>(fmaxf(b0.x + w[i][0].x, 0.f), fmaxf(b0.y + w[i][0].y, 0.f), hi.x, lo.x);
                    split2<PREC>(fmaxf(b0.z + w[i][0].z, 0.f), fmaxf(b0.w + w[i][0].w, 0.f), hi.y, lo.y);
                    split2<PREC>(fmaxf(b1.x + w[i][1].x, 0.f), fmaxf(b1.y + w[i][1].y, 0.f), hi.z, lo.z);
                    split2<PREC>(fmaxf(b1.z + w[i][1].z, 0.f), fmaxf(b1.w + w[i][1].w, 0.f), hi.w, lo.w);
                    if (PREC == 0) *reinterpret_cast<uint4*>(s_h1lo + e * LD + k) = lo;
                    *reinterpret_cast<uint4*>(s_h1hi + e * LD + k) = hi;
                    if (save) {
                        *reinterpret_cast<uint4*>(g_h1hi + gi) = hi;
                        if (PREC == 0) *reinterpret_cast<uint4*>(g_h1hi + h1_plane + gi) = lo;
                        if (b.gate1) b.gate1[gi >> 3] = (uint8_t)nonzero_bits16(hi);  // the gates of these eight units
                    }
                }
            }
        }
    };
    auto layer2_heads = [&](int t) {
        // ---- layer 2 on the tensor pipe: acc[mt][j] = rows 16mt.. x columns 8(wid*NT+j)..
        float acc[MT][NT][4];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[mt][j][q] = 0.f;
        {
            // PREC 2: the leading products and the others in accumulators of their own (the tensor core rounds toward zero
            // at every MMA: the small terms do that at their own magnitude)
            float accx[PREC == 2 ? MT : 1][PREC == 2 ? NT : 1][4];
            if (PREC == 2) {
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int j = 0; j < NT; ++j)
#pragma unroll
                        for (int q = 0; q < 4; ++q) accx[mt][j][q] = 0.f;
            }
            const int arow = (lane & 7) + ((lane >> 3) & 1) * 8, acol = (lane >> 4) * 8;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                uint32_t ahi[MT][4], alo[MT][4], alo2[MT][4];
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    ldmatrix_x4(ahi[mt], s_h1hi + (16 * mt + arow) * LD + 16 * ks + acol);
                    if (PREC != 1) ldmatrix_x4(alo[mt], s_h1lo + (16 * mt + arow) * LD + 16 * ks + acol);
                    if (PREC == 2) ldmatrix_x4(alo2[mt], s_h1lo2 + (16 * mt + arow) * LD + 16 * ks + acol);
                }
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    const uint2 bhi = s_w2hi[(ks * (H / 8) + wid * NT + j) * 32 + lane];
                    uint2 bmid = make_uint2(0u, 0u);
                    if (PREC == 2) bmid = s_w2mid[(ks * (H / 8) + wid * NT + j) * 32 + lane];
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        if (PREC == 2) {
                            mma16816<PREC>(accx[mt][j], alo2[mt], bhi.x, bhi.y);
                            mma16816<PREC>(accx[mt][j], ahi[mt], blo[ks][j].x, blo[ks][j].y);
                            mma16816<PREC>(accx[mt][j], alo[mt], bmid.x, bmid.y);
                            mma16816<PREC>(accx[mt][j], alo[mt], bhi.x, bhi.y);
                            mma16816<PREC>(accx[mt][j], ahi[mt], bmid.x, bmid.y);
                        }
                        if (PREC == 0) {
                            mma16816<PREC>(acc[mt][j], alo[mt], bhi.x, bhi.y);
                            mma16816<PREC>(acc[mt][j], ahi[mt], blo[ks][j].x, blo[ks][j].y);
                        }
                        mma16816<PREC>(acc[mt][j], ahi[mt], bhi.x, bhi.y);
                    }
                }
            }
            if (PREC == 2) {
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int j = 0; j < NT; ++j)
#pragma unroll
                        for (int q = 0; q < 4; ++q) acc[mt][j][q] += accx[mt][j][q];
            }
        }
        // ---- epilogue: bias, ReLU, head partials over this warp's columns
        {
            float ps[2 * MT][5];  // rows g, g+8, (16+g, 24+g)
#pragma unroll
            for (int r = 0; r < 2 * MT; ++r)
#pragma unroll
                for (int c = 0; c < 5; ++c) ps[r][c] = 0.f;
            const bool save_h2 = b.h2 != nullptr && t < a.T;
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                const int col0 = (wid * NT + j) * 8 + 2 * t4;
#pragma unroll
                for (int cc = 0; cc < 2; ++cc) {
                    const float bias = s_b2[col0 + cc];
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                        for (int hh = 0; hh < 2; ++hh) acc[mt][j][2 * hh + cc] = rnd<PREC>(fmaxf(acc[mt][j][2 * hh + cc] + bias, 0.f));
                }
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const int row = 16 * mt + 8 * hh + g;
                        if (save_h2 && e0 + row < B)
                            *reinterpret_cast<float2*>(b.h2 + ((size_t)t * B + e0 + row) * H + col0) =
                                make_float2(acc[mt][j][2 * hh], acc[mt][j][2 * hh + 1]);
                    }
#pragma unroll
                for (int cc = 0; cc < 2; ++cc) {
                    float wh[5];
#pragma unroll
                    for (int c = 0; c < 5; ++c) wh[c] = s_wh[(col0 + cc) * 5 + c];
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                        for (int hh = 0; hh < 2; ++hh) {
                            const float h2 = acc[mt][j][2 * hh + cc];
#pragma unroll
                            for (int c = 0; c < 5; ++c) ps[2 * mt + hh][c] = fmaf(h2, wh[c], ps[2 * mt + hh][c]);
                        }
                }
            }
            // sum over the four lanes of a quad with a transposing exchange: after two rounds lane t4 holds the total
            // of ONE of the four rows (15 shuffles instead of 40; ME = 16: of one of two), and every lane stores its row
            const bool b0 = t4 & 1, b1 = t4 & 2;
            if constexpr (MT == 2) {
                float q2[2][5];
#pragma unroll
                for (int c = 0; c < 5; ++c) {
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const float send = b0 ? ps[i][c] : ps[2 + i][c];
                        const float keep = b0 ? ps[2 + i][c] : ps[i][c];
                        q2[i][c] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 1);
                    }
                }
                const int r = (b0 ? 2 : 0) + (b1 ? 1 : 0);
                const int row = 16 * (r >> 1) + 8 * (r & 1) + g;
#pragma unroll
                for (int c = 0; c < 5; ++c) {
                    const float send = b1 ? q2[0][c] : q2[1][c];
                    const float keep = b1 ? q2[1][c] : q2[0][c];
                    s_red[(wid * ME + row) * 5 + c] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 2);
                }
            } else {
                const int row = 8 * b0 + g;
#pragma unroll
                for (int c = 0; c < 5; ++c) {
                    float x = (b0 ? ps[1][c] : ps[0][c]) + __shfl_xor_sync(0xFFFFFFFFu, b0 ? ps[0][c] : ps[1][c], 1);
                    x += __shfl_xor_sync(0xFFFFFFFFu, x, 2);
                    if (!b1) s_red[(wid * ME + row) * 5 + c] = x;
                }
            }
        }
    };
    // ---- one thread per env: fixed-order sum of the warps' partials, then act and step; `publish` comes between the new
    // position and the records
    auto per_env = [&](int t, bool acting, const StepPre& pre, auto&& publish) {
        float o[5];
        ActOut ao;
        ao.la_mx = ao.Z = ao.rew = 0.f;
        ao.act = ao.done = ao.pos0 = 0;
        if (owner) {
#pragma unroll
            for (int c = 0; c < 5; ++c) o[c] = 0.f;
#pragma unroll
            for (int w = 0; w < NW; ++w)
#pragma unroll
                for (int c = 0; c < 5; ++c) o[c] += s_red[(w * ME + ow) * 5 + c];
#pragma unroll
            for (int c = 0; c < 5; ++c) o[c] += s_bh[c];
            if (acting) {
                ao = act_decide(s, a, e0 + ow, t, o[0], o[1], o[2], o[3], pre);
                s_pos[ow] = s.pos;
            }
        }
        if (REPLAY && ownw && t < t_end) s_pos[ow] = recorded_pos(t + 1);
        publish();
        if (owner) {
            const int env = e0 + ow;
            if (b.out5 && t < a.T) {  // the update reuses the head outputs of every recorded row
                float4* o5 = reinterpret_cast<float4*>(b.out5 + ((size_t)t * B + env) * 8);
                o5[0] = make_float4(o[0], o[1], o[2], o[3]);
                o5[1] = make_float4(o[4], 0.f, 0.f, 0.f);
            }
            if (REPLAY && a.replay == 2 && t == a.T) b.vboot[env] = o[4];
            if (!REPLAY) {
                b.tval[(size_t)t * B + env] = o[4];
                if (a.gae_smem) s_gv[t * ME + ow] = o[4];
                if (acting) {
                    act_record(a, env, t, o[0], o[1], o[2], o[3], ao);
                    if (a.gae_smem) s_gc[t * ME + ow] = (uint8_t)(ao.done | (ao.rew != 0.f ? 2 : 0));
                }
            }
        }
    };
    if constexpr (OWN) {
        // Named barriers: 3 = the workers have written the h1 tile; 2 = head partials written (workers arrive, the owner warp
        // waits); 1 = positions published and every worker past its reads of the h1 tile (the owner warp arrives).
        if (worker) {
            for (int t = t_beg; t <= t_end; ++t) {
                layer1(t);
                asm volatile("bar.sync 3, %0;" ::"n"(NTHREADS) : "memory");
                layer2_heads(t);
                asm volatile("bar.arrive 2, %0;" ::"n"(NALL) : "memory");
                asm volatile("bar.sync 1, %0;" ::"n"(NALL) : "memory");
            }
        } else {
            for (int t = t_beg; t <= t_end; ++t) {
                const bool acting = owner && !REPLAY && t < a.T;
                StepPre pre;
                if (acting) pre = step_prepare(s, a, e0 + ow, t, s_walls + ow * 8);
                asm volatile("bar.sync 2, %0;" ::"n"(NALL) : "memory");
                per_env(t, acting, pre, [&]() {
                    __syncwarp();
                    asm volatile("bar.arrive 1, %0;" ::"n"(NALL) : "memory");
                });
            }
        }
    } else {
        for (int t = t_beg; t <= t_end; ++t) {
            layer1(t);
            __syncthreads();
            // the logits-independent half of the interaction waits in shared memory (two words per env) rather than in
            // registers, which the MMA loop needs
            const bool acting = owner && !REPLAY && t < a.T;
            if (acting) {
                const StepPre pre = step_prepare(s, a, e0 + ow, t, s_walls + ow * 8);
                s_pre[ow] = make_uint2(__float_as_uint(pre.u), (uint32_t)pre.np[0] | ((uint32_t)pre.np[1] << 8) | ((uint32_t)pre.np[2] << 16) | ((uint32_t)pre.np[3] << 24));
            }
            layer2_heads(t);
            __syncthreads();
            StepPre pre;
            if (acting) {
                const uint2 pk = s_pre[ow];
                pre.u = __uint_as_float(pk.x);
#pragma unroll
                for (int q = 0; q < 4; ++q) pre.np[q] = (pk.y >> (8 * q)) & 0xFF;
            }
            per_env(t, acting, pre, []() {});
            __syncthreads();
        }
    }
    pdl_trigger();
    if (REPLAY) return;
    if (owner) {
        b.pos[e0 + ow] = (uint8_t)s.pos;
        b.tep[e0 + ow] = (uint8_t)s.tep;
        // the owner thread wrote this env's rewards, values and done flags itself: it can scan them right away
        if (a.gae_smem) gae_scan_env_smem(b, B, a.T, e0 + ow, a.gamma, a.lambda, s_gv, s_gc, ME, ow);
        else if (a.fuse_gae) gae_scan_env(b, B, a.T, e0 + ow, a.gamma, a.lambda);
    }
    if (OWN ? !worker : tid < 32) flush_env_stats(s, a);
}

constexpr size_t MAX_DYN_SMEM = 232448;  // 227 KB of dynamic shared memory per CTA

template <int H, int NW, int PREC, bool GROUPED, int MINB, bool OWN>
static cudaError_t launch_k(const RolloutArgs& a, dim3 grid, size_t smem, cudaStream_t s) {
    if (a.replay) return launch<k_rollout_mma<H, NW, PREC, GROUPED, MINB, OWN, true, 32, false>>(grid, NW * 32 + (OWN ? 32 : 0), smem, s, a);
    return launch<k_rollout_mma<H, NW, PREC, GROUPED, MINB, OWN, false, 32, false>>(grid, NW * 32 + (OWN ? 32 : 0), smem, s, a);
}

// Small batches: 16 envs per CTA, half the chain of a step for each, while every CTA finds an SM of its own (the narrow widths:
// up to three to an SM; bf16 at 96: two).  B200, T = 16, 64 and 2368 envs: H = 32 22 -> 15 and 17 us, 64 24 -> 18 and 22, 96 49 -> 30
// and 31, 128 43 -> 29 and 30, 192 113 -> 63 and 65; past the line (3000 envs): 96 50 -> 59, 128 44 -> 56, 192 116 -> 126.
template <int H, int PREC> constexpr int small_ctas() { return H <= 64 ? 444 : H == 96 && PREC == 1 ? 296 : 148; }
template <int H, int NW, int PREC>
static cudaError_t launch_small(RolloutArgs a, cudaStream_t s) {
    using Cfg = RolloutMmaCfg<H, NW, PREC, 16>;
    size_t smem = Cfg::smem_bytes;
    a.gae_smem = a.fuse_gae && smem + Cfg::gae_bytes(a.T) <= MAX_DYN_SMEM;
    if (a.gae_smem) smem += Cfg::gae_bytes(a.T);
    const unsigned ctas = (a.d.B + 15) / 16;
    const size_t w1 = (size_t)a.d.C * H * 4;
    if (smem + w1 <= MAX_DYN_SMEM) return launch<k_rollout_mma<H, NW, PREC, false, 1, true, false, 16, true>>(ctas, NW * 32 + 32, smem + w1, s, a);
    return launch<k_rollout_mma<H, NW, PREC, false, 1, true, false, 16, false>>(ctas, NW * 32 + 32, smem, s, a);
}

template <int H, int NW, int PREC, bool GROUPED = false>
static cudaError_t launch_t(const RolloutArgs& a0, cudaStream_t s) {
    using Cfg = RolloutMmaCfg<H, NW, PREC>;
    RolloutArgs a = a0;
    if constexpr (!GROUPED)
        if (!a.replay && a.d.B <= 16 * small_ctas<H, PREC>()) return launch_small<H, NW, PREC>(a, s);
    size_t smem = Cfg::smem_bytes;
    a.gae_smem = 0;
    if (a.fuse_gae && !a.replay && smem + Cfg::gae_bytes(a.T) <= MAX_DYN_SMEM) {
        a.gae_smem = 1;
        smem += Cfg::gae_bytes(a.T);
    }
    const int ctas = (a.d.B + Cfg::ME - 1) / Cfg::ME;
    const int slices = GROUPED ? 1 : replay_slices(a, ctas, H <= 32 ? 4 : H <= 64 ? 3 : H <= 128 ? 2 : 1 /*as many as an SM holds*/, true);
    const dim3 grid(ctas, GROUPED ? a.d.npol : slices);
    // Three-term operands at H = 96, a CTA to an SM: the registers of a whole SM, and the agent rows of W1 (B200, T = 16, 4736 envs:
    // 70 -> 48 us; the other widths and bf16 gain nothing from these rows, their gathers hide behind twice the MMAs).
    const size_t w1 = (size_t)a.d.C * H * 4;
    if constexpr (!GROUPED && H == 96 && PREC == 2)
        if (!a.replay && ctas <= 148 && smem + w1 <= MAX_DYN_SMEM) return launch<k_rollout_mma<H, NW, PREC, false, 1, true, false, 32, true>>(grid, NW * 32 + 32, smem + w1, s, a);
    // The owner warp costs a CTA of the 128-wide kernel its second place on an SM: only where every CTA gets an SM of its own.
    // (H = 64: three CTAs per SM where there are that many)
    // ... in fp32 with the agent rows of W1 beside them where the GPU is full more than once and the rollout is ten steps or longer: a CTA
    // loads them once and gathers from them every step.  B200, gather from shared memory / from L2, 14300 to 131072 envs on 9 to 121 cells:
    // T = 2, 4 0.99 to 1.13, T = 6, 8 0.92 to 1.05, T = 12 0.90 to 0.98, T = 16 to 64 0.85 to 1.00 of the time, whatever the board (30000
    // envs, 81 cells, T = 16: 128 -> 116 us).  Up to 444 CTAs 0.94 to 1.08 without a pattern; bf16 loses (44158 envs, T = 45: 333 ->
    // 345 us).
    if constexpr (H == 64 && PREC == 0) {
        const size_t w1b = (size_t)a.d.C * H * 4;
        if (!a.replay && (size_t)grid.x * grid.y > 444 && a.T >= 10 && smem + w1b <= 75 * 1024)
            return launch<k_rollout_mma<H, NW, PREC, GROUPED, 3, true, false, 32, true>>(grid, NW * 32 + 32, smem + w1b, s, a);
    }
    if constexpr (H == 64)
        if ((size_t)grid.x * grid.y > 296) return launch_k<H, NW, PREC, GROUPED, 3, true>(a, grid, smem, s);
    if constexpr (H < 128) return launch_k<H, NW, PREC, GROUPED, 2, true>(a, grid, smem, s);
    else if constexpr (H == 128) {
        if ((size_t)grid.x * grid.y <= 148) return launch_k<H, NW, PREC, GROUPED, 1, true>(a, grid, smem, s);
        return launch_k<H, NW, PREC, GROUPED, 2, false>(a, grid, smem, s);
    } else return launch_k<H, NW, PREC, GROUPED, 1, H == 192>(a, grid, smem, s);
}

// Hidden widths whose second-layer weights fit on chip beside a CTA's activations.
bool rollout_mma_supported(int H) { return H == 32 || H == 64 || H == 96 || H == 128 || H == 192 || H == 256; }
// fp32 operands as three exact bf16 terms (the widths beside 64, 128 and 256, which take two fp16 terms).
bool three_terms(int H, int prec) { return prec == 0 && !(H == 64 || H == 128 || H == 256); }
// H = 256 runs the CTA-pair tcgen05 kernels, which read the row-major planes of W2 only.
bool rollout_uses_fragments(int H) { return rollout_mma_supported(H) && H != 256; }

// Returns cudaErrorNotSupported when the shape is not covered by the tensor-pipe kernel.
cudaError_t launch_rollout_mma(const RolloutArgs& a, int prec, cudaStream_t s) {
    if (!rollout_mma_supported(a.d.H)) return cudaErrorNotSupported;
    if (a.d.npol <= 1 && a.d.H == 256) {  // the CTA-pair kernels on the 5th-generation tensor cores
        const cudaError_t e = launch_rollout_pair2(a, prec, s);  // large batches: two env groups per pair
        if (e != cudaErrorNotSupported) return e;
        return launch_rollout_pair(a, prec, s);
    }
    if (a.d.npol <= 1 && a.d.H == 128) {  // large batches: two env groups per CTA on the 5th-generation tensor cores
        const cudaError_t e = launch_rollout_tc128(a, prec, s);
        if (e != cudaErrorNotSupported) return e;
    }
    if (!a.b.w2f_hi) return cudaErrorNotSupported;
    if (a.d.npol > 1) {  // many policies: one grid slice per policy, each with its own weights on chip
        if (prec != 0) return cudaErrorNotSupported;
        switch (a.d.H) {
            case 64: return launch_t<64, 4, 0, true>(a, s);
            case 128: return launch_t<128, 8, 0, true>(a, s);
        }
        return cudaErrorNotSupported;
    }
    if (prec == 1) {
        switch (a.d.H) {
            case 32: return launch_t<32, 2, 1>(a, s);
            case 64: return launch_t<64, 4, 1>(a, s);
            case 96: return launch_t<96, 6, 1>(a, s);
            case 128: return launch_t<128, 8, 1>(a, s);
            case 192: return launch_t<192, 12, 1>(a, s);
        }
    } else {
        switch (a.d.H) {
            case 32: return launch_t<32, 2, 2>(a, s);
            case 64: return launch_t<64, 4, 0>(a, s);
            case 96: return launch_t<96, 6, 2>(a, s);
            case 128: return launch_t<128, 8, 0>(a, s);
            case 192: return launch_t<192, 12, 2>(a, s);
        }
    }
    return cudaErrorNotSupported;
}

}  // namespace anakin
