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
// GAE reverse scan: lane = env, so every load and store of a warp is one contiguous segment per t.
//   d_t = 1 - done_t; delta_t = r_t + gamma d_t V_{t+1} - V_t; A_t = delta_t + gamma lambda d_t A_{t+1}; ret = A + V
// ----------------------------------------------------------------------------------------------------
template <bool GROUPED>
__global__ void __launch_bounds__(128) k_gae(DimsBuffers in, int T, float gamma, float lambda) {
    pdl_wait();
    const PolicyArgs<GROUPED, DimsBuffers> pa(in, blockIdx.y);
    const Dims& d = pa.a.d;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= d.B) return;
    gae_scan_env(pa.a.b, d.B, T, e, gamma, lambda);
}

cudaError_t launch_gae(const Dims& d, const Buffers& b, int T, float gamma, float lambda, const Ctx& c) {
    Scope sc(c, K_GAE);
    if (d.npol > 1) launch<k_gae<true>>(dim3((d.B + 127) / 128, d.npol), 128, 0, c.s, DimsBuffers{d, b}, T, gamma, lambda);
    else launch<k_gae<false>>((d.B + 127) / 128, 128, 0, c.s, DimsBuffers{d, b}, T, gamma, lambda);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------------------------
// V-trace targets (Espeholt et al. 2018, IMPALA, Eq. 1; recursive form), lane = env, reverse scan over t.  mu = the policy
// that acted (recorded log-probabilities), pi = the current parameters (head outputs of the recorded rows in out5):
//   w = exp(logp_pi - logp_mu); rho = min(rho_bar, w); c = min(c_bar, w); d = 1 - done
//   delta = rho (r + gamma d V' - V);  e = delta + gamma d c e';  ret = V + e;  adv = rho (r + gamma d (V' + e') - V)
// Four steps per memory round trip.
// ----------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(128) k_vtrace(Dims d, Buffers b, int T, float gamma, float rho_bar, float c_bar, const float* boot) {
    pdl_wait();  // (no early trigger: 37 us alone, 61 us with the next kernel's CTAs beside it)
    const int env = blockIdx.x * blockDim.x + threadIdx.x;
    if (env >= d.B) return;
    const int B = d.B;
    float e_next = 0.f, v_next = boot[env];
    for (int tb = T; tb > 0; tb -= 4) {
        float4 lg[4];
        float v[4], r[4], nd[4], lmu[4];
        int act[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int t = tb - 1 - q;
            if (t >= 0) {
                const size_t i = (size_t)t * B + env;
                const float4* o = reinterpret_cast<const float4*>(b.out5 + i * 8);
                lg[q] = o[0];
                v[q] = o[1].x;
                r[q] = b.trew[i];
                nd[q] = b.tdone[i] ? 0.f : 1.f;
                lmu[q] = b.tlogp[i];
                act[q] = b.tact[i];
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int t = tb - 1 - q;
            if (t >= 0) {
                const size_t i = (size_t)t * B + env;
                const float l0 = lg[q].x, l1 = lg[q].y, l2 = lg[q].z, l3 = lg[q].w;
                const float mx = fmaxf(fmaxf(l0, l1), fmaxf(l2, l3));
                const float Z = ((expf(l0 - mx) + expf(l1 - mx)) + expf(l2 - mx)) + expf(l3 - mx);
                const float la = act[q] == 0 ? l0 : act[q] == 1 ? l1 : act[q] == 2 ? l2 : l3;
                const float lpi = (la - mx) - logf(Z);
                const float w = expf(lpi - lmu[q]);
                const float rho = fminf(rho_bar, w), c = fminf(c_bar, w);
                const float gd = gamma * nd[q];
                const float delta = rho * ((r[q] + gd * v_next) - v[q]);
                const float e = delta + gd * c * e_next;
                b.adv[i] = rho * ((r[q] + gd * (v_next + e_next)) - v[q]);
                b.ret[i] = v[q] + e;
                e_next = e;
                v_next = v[q];
            }
        }
    }
}

cudaError_t launch_vtrace(const Dims& d, const Buffers& b, int T, float gamma, float rho_bar, float c_bar, const float* boot, const Ctx& c) {
    Scope sc(c, K_VTRACE);
    return launch<k_vtrace>((d.B + 127) / 128, 128, 0, c.s, d, b, T, gamma, rho_bar, c_bar, boot);
}

}  // namespace anakin
