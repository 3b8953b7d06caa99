// Acting half of the Anakin minimal unit (Podracer paper, Section 3.1; Figure 2, top): T interactions of
// every env with the policy, fused into one persistent kernel.  A CTA owns ME envs for the whole rollout,
// so there is no inter-CTA dependency and no grid-wide wait anywhere.
#include "env_step.cuh"

namespace anakin {

// base[b][j] = b1[j] + sum over wall cells c (ascending) of W1[c][j] + W1[2C+goal_b][j].
// The wall and goal planes of the observation do not change during an env's life, so their contribution
// to the first layer is computed once per parameter version instead of once per step.
// One thread owns four hidden units of one env; the W1 rows are fetched eight at a time (independent loads) and added in
// ascending cell order, the goal row last.
template <bool GROUPED>
__global__ void __launch_bounds__(256) k_env_base(DimsBuffers in) {
    pdl_wait();
    const PolicyArgs<GROUPED, DimsBuffers> pa(in, blockIdx.y);  // many policies: grid.y = policy
    const Dims& d = pa.a.d;
    const Buffers& b = pa.a.b;
    const int H4 = d.H / 4;
    const size_t idx = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (idx >= (size_t)d.B * H4) return;
    const int e = (int)(idx / H4), j4 = (int)(idx - (size_t)e * H4);
    const uint32_t* w = b.walls + (size_t)e * d.W;
    const float4* W1 = reinterpret_cast<const float4*>(b.theta_c + d.oW1) + j4;
    const int goal_row = 2 * d.C + min((int)b.goal[e], d.C - 1);  // (the rollout flags a goal outside the board)
    float4 acc = reinterpret_cast<const float4*>(b.theta_c + d.ob1)[j4];
    int wi = 0;
    uint32_t bits = w[0];
    bool goal_done = false;
    auto next_row = [&]() -> int {  // next wall cell in ascending order, then the goal row, then -1
        while (!bits && wi + 1 < d.W) bits = w[++wi];
        if (bits) {
            const int c = wi * 32 + (__ffs(bits) - 1);
            bits &= bits - 1;
            return c;
        }
        if (!goal_done) { goal_done = true; return goal_row; }
        return -1;
    };
    for (;;) {
        int rows[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) rows[q] = next_row();
        float4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = rows[q] >= 0 ? __ldg(W1 + (size_t)rows[q] * H4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (rows[q] >= 0) { acc.x += v[q].x; acc.y += v[q].y; acc.z += v[q].z; acc.w += v[q].w; }
        }
        if (rows[7] < 0) break;
    }
    pdl_trigger();
    reinterpret_cast<float4*>(b.base)[idx] = acc;
}

cudaError_t launch_env_base(const Dims& d, const Buffers& b, const Ctx& c) {
    if (d.npol <= 1) {
        const cudaError_t ew = launch_env_base_wide(d, b, c);  // tensor-core form where it applies
        if (ew != cudaErrorNotSupported) return ew;
    }
    Scope sc(c, K_ENV_BASE);
    const unsigned nb = (unsigned)(((size_t)d.B * (d.H / 4) + 255) / 256);
    if (d.npol > 1) launch<k_env_base<true>>(dim3(nb, d.npol), 256, 0, c.s, DimsBuffers{d, b});
    else launch<k_env_base<false>>(nb, 256, 0, c.s, DimsBuffers{d, b});
    return cudaGetLastError();
}

cudaError_t launch_rollout(const RolloutArgs& a, int prec, const Ctx& c) {
    if (wide_supported(a.d.H)) return launch_rollout_wide(a, c);  // two launches per step
    Scope sc(c, K_ROLLOUT);
    return launch_rollout_mma(a, prec, c.s);
}

// ----------------------------------------------------------------------------------------------------
// The two reverse scans over the recorded steps, x_t = delta_t + coef_t x_{t+1}.  A CTA takes 32 envs and up to 64 steps at a time: eight
// warps fetch the rows and form delta and coef (lane = env, a warp every eighth step, so that all of a chunk's loads are in flight at
// once), one warp walks the chain through shared memory, the eight write the results.  One thread per env with four or eight steps in
// flight pays a memory round trip and the exponentials of each group one after the other, on a few SMs.  B200 (events included): V-trace of
// 6000 envs, T = 20 17.8 -> 10.6 us; GAE of 16384 envs, T = 32 23.8 -> 10.6, of 3000, T = 16 12.8 -> 8.8.
// Where the batch alone fills the GPU, a thread per env (k_gae_each, k_vtrace_each) has as many loads in flight without the shared memory
// and the barriers, and with few steps no warp without a row: chunk / each, GAE of 16384 envs T = 4 8 / 9, T = 64 13 / 40; of 32768 T = 4
// 10 / 9, T = 16 11 / 15; of 65536 T = 8 13 / 11, T = 16 15 / 15, T = 32 20 / 26; of 98304 T = 8 17 / 12, T = 64 44 / 46; of 131072 T = 8 20 /
// 11, T = 64 52 / 48.  V-trace (32 bytes of head outputs a row, the exponentials) of 16384 envs T = 4 14 / 10, T = 16 13 / 18; of 24576 T = 8
// 14 / 11, T = 16 17 / 17, T = 64 35 / 46; of 32768 T = 16 19 / 17, T = 64 45 / 48; of 49152 T = 64 64 / 44; of 131072 T = 64 141 / 77.
// Either form takes the same operations in the same order.
// ----------------------------------------------------------------------------------------------------
static bool gae_in_chunks(long long envs, int T) { return envs <= 98304 && envs < 4096LL * T; }
static bool vtrace_in_chunks(int envs, int T) { return envs <= 24576 && envs <= 1024LL * T; }

constexpr int SCAN_ENVS = 32, SCAN_WARPS = 8, SCAN_STEPS = 64, SCAN_ROWS = SCAN_STEPS / SCAN_WARPS;

struct ScanShared {
    float v[SCAN_STEPS + 1][SCAN_ENVS];      // values; row n: the value after the chunk's last step
    float x[SCAN_STEPS + 1][SCAN_ENVS];      // results of the chain; row n: the one after the chunk
    float delta[SCAN_STEPS][SCAN_ENVS], coef[SCAN_STEPS][SCAN_ENVS];
};

// The chain of one chunk of n steps; the caller synchronises on both sides.
__device__ __forceinline__ void scan_chain(ScanShared& s, int n, int lane) {
    float x = s.x[n][lane];
    for (int k = n - 1; k >= 0; --k) {
        x = __fmaf_rn(s.coef[k][lane], x, s.delta[k][lane]);
        s.x[k][lane] = x;
    }
}

// GAE: d_t = 1 - done_t; delta_t = r_t + gamma d_t V_{t+1} - V_t; A_t = delta_t + gamma lambda d_t A_{t+1}; ret = A + V.  The operations
// of gae_scan_env_smem, which the rollouts that keep their values on chip run: the same bits.
template <bool GROUPED>
__global__ void __launch_bounds__(32 * SCAN_WARPS) k_gae(DimsBuffers in, int T, float gamma, float lambda) {
    __shared__ ScanShared s;
    pdl_wait();
    const PolicyArgs<GROUPED, DimsBuffers> pa(in, blockIdx.y);
    const Buffers& b = pa.a.b;
    const int B = pa.a.d.B, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, env = blockIdx.x * SCAN_ENVS + lane;
    const bool have = env < B;
    const float gl = __fmul_rn(gamma, lambda);
    for (int tb = T; tb > 0; tb -= SCAN_STEPS) {
        const int t0 = max(tb - SCAN_STEPS, 0), n = tb - t0;
        float r[SCAN_ROWS], nd[SCAN_ROWS];
        float vn = 0.f, xn = 0.f;  // after the chunk: the bootstrap value, then the first row of the chunk before
        if (wid == 0) {
            vn = tb == T ? (have ? b.tval[(size_t)T * B + env] : 0.f) : s.v[0][lane];
            xn = tb == T ? 0.f : s.x[0][lane];
        }
        if (tb < T) __syncthreads();  // (every warp is done with the chunk before)
        if (wid == 0) {
            s.v[n][lane] = vn;
            s.x[n][lane] = xn;
        }
        float v[SCAN_ROWS];
#pragma unroll
        for (int q = 0; q < SCAN_ROWS; ++q) {
            const int k = wid + SCAN_WARPS * q;
            v[q] = r[q] = nd[q] = 0.f;
            if (k < n && have) {
                const size_t i = (size_t)(t0 + k) * B + env;
                v[q] = b.tval[i];
                r[q] = b.trew[i];
                nd[q] = b.tdone[i] ? 0.f : 1.f;
            }
        }
#pragma unroll
        for (int q = 0; q < SCAN_ROWS; ++q)
            if (wid + SCAN_WARPS * q < n) s.v[wid + SCAN_WARPS * q][lane] = v[q];
        __syncthreads();
#pragma unroll
        for (int q = 0; q < SCAN_ROWS; ++q) {
            const int k = wid + SCAN_WARPS * q;
            if (k < n) {
                s.delta[k][lane] = __fsub_rn(__fmaf_rn(__fmul_rn(gamma, nd[q]), s.v[k + 1][lane], r[q]), v[q]);
                s.coef[k][lane] = __fmul_rn(gl, nd[q]);
            }
        }
        __syncthreads();
        if (wid == 0) scan_chain(s, n, lane);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < SCAN_ROWS; ++q) {
            const int k = wid + SCAN_WARPS * q;
            if (k < n && have) {
                const size_t i = (size_t)(t0 + k) * B + env;
                const float A = s.x[k][lane];
                b.adv[i] = A;
                b.ret[i] = __fadd_rn(A, v[q]);
            }
        }
    }
}

// ... thread = env.
template <bool GROUPED>
__global__ void __launch_bounds__(128) k_gae_each(DimsBuffers in, int T, float gamma, float lambda) {
    pdl_wait();
    const PolicyArgs<GROUPED, DimsBuffers> pa(in, blockIdx.y);
    const Dims& d = pa.a.d;
    const int e = blockIdx.x * 128 + threadIdx.x;
    if (e < d.B) gae_scan_env(pa.a.b, d.B, T, e, gamma, lambda);
}

cudaError_t launch_gae(const Dims& d, const Buffers& b, int T, float gamma, float lambda, const Ctx& c) {
    Scope sc(c, K_GAE);
    const DimsBuffers db{d, b};
    const bool chunks = gae_in_chunks((long long)d.B * d.npol, T);
    const unsigned per = chunks ? SCAN_ENVS : 128, threads = chunks ? 32 * SCAN_WARPS : 128;
    const dim3 grid((unsigned)(d.B + per - 1) / per, d.npol);
    if (d.npol > 1) return chunks ? launch<k_gae<true>>(grid, threads, 0, c.s, db, T, gamma, lambda) : launch<k_gae_each<true>>(grid, threads, 0, c.s, db, T, gamma, lambda);
    return chunks ? launch<k_gae<false>>(grid, threads, 0, c.s, db, T, gamma, lambda) : launch<k_gae_each<false>>(grid, threads, 0, c.s, db, T, gamma, lambda);
}

// V-trace targets (Espeholt et al. 2018, IMPALA, Eq. 1; recursive form).  mu = the policy that acted (recorded log-probabilities),
// pi = the current parameters (head outputs of the recorded rows in out5):
//   w = exp(logp_pi - logp_mu); rho = min(rho_bar, w); c = min(c_bar, w); d = 1 - done
//   delta = rho (r + gamma d V' - V);  e = delta + gamma d c e';  ret = V + e;  adv = rho (r + gamma d (V' + e') - V)
struct VtraceRow {  // what a recorded row brings
    float4 lg;
    float v, r, lmu;
    int act, done;
};
__device__ __forceinline__ VtraceRow vtrace_row(const Buffers& b, size_t i) {
    const float4* o = reinterpret_cast<const float4*>(b.out5 + i * 8);
    return VtraceRow{o[0], o[1].x, b.trew[i], b.tlogp[i], b.tact[i], b.tdone[i]};
}
__device__ __forceinline__ float vtrace_ratio(const VtraceRow& x) {
    const float l0 = x.lg.x, l1 = x.lg.y, l2 = x.lg.z, l3 = x.lg.w;
    const float mx = fmaxf(fmaxf(l0, l1), fmaxf(l2, l3));
    const float Z = ((expf(l0 - mx) + expf(l1 - mx)) + expf(l2 - mx)) + expf(l3 - mx);
    const float la = x.act == 0 ? l0 : x.act == 1 ? l1 : x.act == 2 ? l2 : l3;
    return expf(((la - mx) - logf(Z)) - x.lmu);
}
// rho (r + gamma d x - V): delta with x = V', the advantage with x = V' + e'
__device__ __forceinline__ float vtrace_term(float rho, float r, float gd, float x, float v) {
    return __fmul_rn(rho, __fsub_rn(__fmaf_rn(gd, x, r), v));
}

__global__ void __launch_bounds__(32 * SCAN_WARPS) k_vtrace(Dims d, Buffers b, int T, float gamma, float rho_bar, float c_bar, const float* boot) {
    __shared__ ScanShared s;
    pdl_wait();  // (no early trigger: the next kernel's CTAs would crowd in beside this one's)
    const int B = d.B, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, env = blockIdx.x * SCAN_ENVS + lane;
    const bool have = env < B;
    for (int tb = T; tb > 0; tb -= SCAN_STEPS) {
        const int t0 = max(tb - SCAN_STEPS, 0), n = tb - t0;
        float vn = 0.f, xn = 0.f;  // after the chunk: the bootstrap value, then the first row of the chunk before
        if (wid == 0) {
            vn = tb == T ? (have ? boot[env] : 0.f) : s.v[0][lane];
            xn = tb == T ? 0.f : s.x[0][lane];
        }
        if (tb < T) __syncthreads();  // (every warp is done with the chunk before)
        if (wid == 0) {
            s.v[n][lane] = vn;
            s.x[n][lane] = xn;
        }
        float v[SCAN_ROWS], r[SCAN_ROWS], gd[SCAN_ROWS], rho[SCAN_ROWS];
#pragma unroll
        for (int h = 0; h < SCAN_ROWS; h += 4) {  // four rows' loads at a time
            VtraceRow x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = wid + SCAN_WARPS * (h + q);
                x[q] = VtraceRow{make_float4(0.f, 0.f, 0.f, 0.f), 0.f, 0.f, 0.f, 0, 0};
                if (k < n && have) x[q] = vtrace_row(b, (size_t)(t0 + k) * B + env);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = wid + SCAN_WARPS * (h + q);
                v[h + q] = x[q].v;
                r[h + q] = x[q].r;
                gd[h + q] = x[q].done ? 0.f : gamma;
                if (k < n) {
                    const float w = vtrace_ratio(x[q]);
                    rho[h + q] = fminf(rho_bar, w);
                    s.coef[k][lane] = __fmul_rn(gd[h + q], fminf(c_bar, w));
                    s.v[k][lane] = x[q].v;
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < SCAN_ROWS; ++q) {
            const int k = wid + SCAN_WARPS * q;
            if (k < n) s.delta[k][lane] = vtrace_term(rho[q], r[q], gd[q], s.v[k + 1][lane], v[q]);
        }
        __syncthreads();
        if (wid == 0) scan_chain(s, n, lane);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < SCAN_ROWS; ++q) {
            const int k = wid + SCAN_WARPS * q;
            if (k < n && have) {
                const size_t i = (size_t)(t0 + k) * B + env;
                b.adv[i] = vtrace_term(rho[q], r[q], gd[q], __fadd_rn(s.v[k + 1][lane], s.x[k + 1][lane]), v[q]);
                b.ret[i] = __fadd_rn(v[q], s.x[k][lane]);
            }
        }
    }
}

// ... thread = env, four steps per memory round trip.
__global__ void __launch_bounds__(128) k_vtrace_each(Dims d, Buffers b, int T, float gamma, float rho_bar, float c_bar, const float* boot) {
    pdl_wait();  // (no early trigger: 37 us alone, 61 us with the next kernel's CTAs beside it)
    const int env = blockIdx.x * 128 + threadIdx.x, B = d.B;
    if (env >= B) return;
    float e = 0.f, vnext = boot[env];
    for (int tb = T; tb > 0; tb -= 4) {
        VtraceRow x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (tb - 1 - q >= 0) x[q] = vtrace_row(b, (size_t)(tb - 1 - q) * B + env);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (tb - 1 - q >= 0) {
                const size_t i = (size_t)(tb - 1 - q) * B + env;
                const float w = vtrace_ratio(x[q]), rho = fminf(rho_bar, w), gd = x[q].done ? 0.f : gamma;
                b.adv[i] = vtrace_term(rho, x[q].r, gd, __fadd_rn(vnext, e), x[q].v);
                e = __fmaf_rn(__fmul_rn(gd, fminf(c_bar, w)), e, vtrace_term(rho, x[q].r, gd, vnext, x[q].v));
                b.ret[i] = __fadd_rn(x[q].v, e);
                vnext = x[q].v;
            }
        }
    }
}

cudaError_t launch_vtrace(const Dims& d, const Buffers& b, int T, float gamma, float rho_bar, float c_bar, const float* boot, const Ctx& c) {
    Scope sc(c, K_VTRACE);
    if (!vtrace_in_chunks(d.B, T)) return launch<k_vtrace_each>((d.B + 127) / 128, 128, 0, c.s, d, b, T, gamma, rho_bar, c_bar, boot);
    return launch<k_vtrace>((d.B + SCAN_ENVS - 1) / SCAN_ENVS, 32 * SCAN_WARPS, 0, c.s, d, b, T, gamma, rho_bar, c_bar, boot);
}

}  // namespace anakin
