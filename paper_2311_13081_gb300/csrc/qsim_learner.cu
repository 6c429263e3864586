// qsim_learner.cu -- asymmetric TD3 learner (Sec. IV; TD3 of Fujimoto et al. 2018) and the
// batched multi-run training kernel.
//
// One run is processed by a thread-block cluster of S CTAs.  Each CTA owns B/S samples of
// the minibatch: it gathers them from the replay ring, rebuilds the actor and privileged
// critic observations, and runs every forward / backward GEMM of its slice: on the tensor
// cores when it holds whole 128-sample tiles (td3_update_tc, qsim_tcmlp.cuh), else in shared
// memory (td3_update_smem, qsim_smlp.cuh) or, for odd shapes, with activations in its own
// L2-resident scratch (td3_update).  Weight gradients are reduced across the
// cluster in a fixed order (deterministic, no float atomics): each CTA sums one slice of
// the parameter vector over the S partials and applies Adam (and Polyak) to that slice,
// with hardware cluster barriers between phases.  A persistent grid of clusters walks a
// host-computed longest-processing-time-first list of runs; each run advances n_iters
// iterations of {env step of its envs, updates_per_step updates} before the cluster moves
// to its next run.  The same kernel launched for one run and one iteration is the plain
// (one-run-per-launch) form.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <mutex>
#include <numeric>
#include <vector>

#include <cooperative_groups.h>

#include "qsim_gemm.cuh"
#include "qsim_smlp.cuh"
#include "qsim_internal.h"
#include "qsim_recalc.cuh"
#include "qsim_staging.h"
#include "qsim_tcgen05.cuh"
#include "qsim_tcmlp.cuh"

namespace cg = cooperative_groups;

namespace qsim {


constexpr int SMEM_ENGINE = smlp::floats() > smlp::floats2() ? smlp::floats() : smlp::floats2();
constexpr int SMEM_TC = (tce::SMEM_BYTES + 3) / 4;
constexpr int SMEM_MAIN = SMEM_TC > SMEM_ENGINE ? SMEM_TC : (GEMM_SMEM > SMEM_ENGINE ? GEMM_SMEM : SMEM_ENGINE);
static_assert(4 * (SMEM_MAIN + 32) <= 227 * 1024, "learner shared memory");
// the small-run env step keeps an actor of hidden <= 128 and <= 128 inputs in shared memory
static_assert(SMEM_MAIN >= 128 * 128 + 128 + 128 * 128 + 128 + 4 * 128 + 4 + 4 + 8 * (132 + 2 * 132 + 4 + 32),
              "learner shared memory too small for the small-run env step");

struct LearnHyper {
    float gamma, tau, lr, beta1, beta2, eps, sigma_t, noise_clip;
    int policy_delay, updates_per_step;
};

// Everything the training kernel knows about one run.  Counters are updated in place by
// the kernel so that a captured graph can be replayed.
struct RunDesc {
    EnvCfg C;
    EnvPtrs E;
    int64_t capacity, head, size, t_now;
    int64_t next_curr, curr_interval;
    float cf[7], ct[7];
    float sig_f, sig_min;
    int recalc;
    int n_env;
    float *actor, *actor_t, *c1, *c1_t, *c2, *c2_t;
    float *m_a, *v_a, *m_c1, *v_c1, *m_c2, *v_c2;
    float* stats;
    int H, B, DA, DC, PA, PC;
    int64_t t_a, t_c, u;
    int64_t start_updates;
    LearnHyper hp;
    uint32_t* idx_log;  // [B] flat replay indices of the latest update, or null
};

// Forward of in -> H (ReLU) -> H (ReLU) -> out (tanh or linear) for M rows of X [M][ldx].
__device__ __noinline__ void mlp_fwd(const float* W, int in, int H, int out, const float* X, int ldx, int M,
                        float* H1, float* H2, float* Y, int ldy, bool tanh_out, float* sm) {
    const float* W1 = W;
    const float* b1 = W1 + H * in;
    const float* W2 = b1 + H;
    const float* b2 = W2 + H * H;
    const float* W3 = b2 + H;
    const float* b3 = W3 + out * H;
    cta_gemm(M, H, in, Mat{X, ldx, 1}, Mat{W1, 1, in}, sm,
             [&](int m, int n, float v) { H1[m * H + n] = fmaxf(v, 0.0f); }, b1);
    cta_gemm(M, H, H, Mat{H1, H, 1}, Mat{W2, 1, H}, sm,
             [&](int m, int n, float v) { H2[m * H + n] = fmaxf(v, 0.0f); }, b2);
    cta_gemm(M, out, H, Mat{H2, H, 1}, Mat{W3, 1, H}, sm, [&](int m, int n, float v) {
        Y[m * ldy + n] = tanh_out ? tanhf(v) : v;
    }, b3);
}

// Reverse through the MLP for M rows.  dZ3 [M][out] holds dLoss/d(pre-activation of the
// output layer).  Writes the parameter gradient (this CTA's partial) into G (layout of
// W) and, if dX != nullptr, dLoss/dX [M][in] (only columns [x_lo, in) are needed).
__device__ __noinline__ void mlp_bwd(const float* W, int in, int H, int out, const float* X, int ldx, int M,
                        const float* H1, const float* H2, const float* dZ3, float* dZ2,
                        float* dZ1, float* G, float* dX, int x_lo, float* sm) {
    const float* W2 = W + H * in + H;
    const float* W3 = W2 + H * H + H;
    float* gW1 = G;
    float* gb1 = gW1 + H * in;
    float* gW2 = gb1 + H;
    float* gb2 = gW2 + H * H;
    float* gW3 = gb2 + H;
    float* gb3 = gW3 + out * H;
    // dW3 = dZ3^T H2 ; db3 = colsum dZ3
    if (G) {
        cta_gemm(out, H, M, Mat{dZ3, 1, out}, Mat{H2, H, 1}, sm,
                 [&](int m, int n, float v) { gW3[m * H + n] = v; });
        for (int n = threadIdx.x; n < out; n += LT) {
            float s = 0.0f;
            for (int m = 0; m < M; ++m) s += ldcg(dZ3 + m * out + n);
            gb3[n] = s;
        }
    }
    // dZ2 = (dZ3 W3) * (H2 > 0)
    cta_gemm(M, H, out, Mat{dZ3, out, 1}, Mat{W3, H, 1}, sm, [&](int m, int n, float v) {
        dZ2[m * H + n] = H2[m * H + n] > 0.0f ? v : 0.0f;  // written by this CTA
    });
    if (G) {
        cta_gemm(H, H, M, Mat{dZ2, 1, H}, Mat{H1, H, 1}, sm,
                 [&](int m, int n, float v) { gW2[m * H + n] = v; });
        for (int n = threadIdx.x; n < H; n += LT) {
            float s = 0.0f;
            for (int m = 0; m < M; ++m) s += ldcg(dZ2 + m * H + n);
            gb2[n] = s;
        }
    }
    // dZ1 = (dZ2 W2) * (H1 > 0)
    cta_gemm(M, H, H, Mat{dZ2, H, 1}, Mat{W2, H, 1}, sm, [&](int m, int n, float v) {
        dZ1[m * H + n] = H1[m * H + n] > 0.0f ? v : 0.0f;  // written by this CTA
    });
    if (G) {
        cta_gemm(H, in, M, Mat{dZ1, 1, H}, Mat{X, ldx, 1}, sm,
                 [&](int m, int n, float v) { gW1[m * in + n] = v; });
        for (int n = threadIdx.x; n < H; n += LT) {
            float s = 0.0f;
            for (int m = 0; m < M; ++m) s += ldcg(dZ1 + m * H + n);
            gb1[n] = s;
        }
    }
    if (dX) {
        const float* W1 = W;
        cta_gemm(M, in - x_lo, H, Mat{dZ1, H, 1}, Mat{W1 + x_lo, in, 1}, sm,
                 [&](int m, int n, float v) { dX[m * in + x_lo + n] = v; });
    }
    __syncthreads();
}

// -------------------------------------------------------------------- cluster helpers
__device__ __forceinline__ void cluster_sync_all(int S) {
    if (S > 1) {
        __threadfence();
        cg::this_cluster().sync();
    } else {
        __syncthreads();
    }
}

// Scratch layout of one CTA (floats), for Bc samples.
struct Scr {
    float *oa, *oa2, *oc, *oc2, *r, *term, *y, *q1, *q2, *mu, *da, *dz3, *X1, *X2, *H1a, *H2a,
        *H1b, *H2b, *dZ2, *dZ1, *ga, *g1, *g2, *loss, *env_obs, *env_h1, *env_h2, *env_mu;
    // tensor-core passes (in the place of X1 .. dZ1): this CTA's share of the six networks'
    // halves (net_img), and o_c in FP32 rows [Bc][critic input] with their sums of magnitudes [Bc]
    float *img, *x32, *xn;
};
enum Net { N_ACTOR, N_ACTOR_T, N_C1, N_C1_T, N_C2, N_C2_T };

// Halves of network n of a run (for the tensor-core passes), from any CTA of its cluster.
__device__ __forceinline__ unsigned char* net_img(const Scr& S, float* scr_base, size_t scr_stride, int rk, int nS, int H,
                                                  int n) {
    const ptrdiff_t at = (ptrdiff_t)(n % nS - rk) * (ptrdiff_t)scr_stride + (S.img - scr_base) +
                         (ptrdiff_t)(n / nS) * tce::img_floats(H);
    return reinterpret_cast<unsigned char*>(scr_base + at);
}

// Networks' halves per CTA of a cluster of nS: network n lies in the scratch of rank n mod nS.
__host__ __device__ constexpr int imgs_per_cta(int nS) { return (6 + nS - 1) / nS; }

// (tiles: as the tensor-core passes lay it out, else in FP32 rows)
__host__ __device__ inline size_t scratch_floats(int Bc, int H, int DA, int DC, int PA, int PC,
                                                 int n_env, int nS, bool tiles) {
    size_t f = 0;
    if (tiles) {
        f += 4 * (size_t)(Bc / tce::TR) * tce::TILE_FLOATS;              // oa oa2 oc oc2: input tiles
        f += (size_t)(tce::KP + 1) * Bc;                                 // x32 xn
        f += (size_t)imgs_per_cta(nS) * tce::img_floats(H);              // img
    } else {
        f += 2 * (size_t)Bc * DA + 2 * (size_t)Bc * DC;  // oa oa2 oc oc2
        f += 8 * (size_t)Bc * H;                         // X1 X2 H1a H2a H1b H2b dZ2 dZ1
    }
    f += 5 * (size_t)Bc;                              // r term y q1 q2
    f += 3 * 4 * (size_t)Bc;                          // mu da dz3
    f += (size_t)PA + 2 * (size_t)PC + 8;             // partial grads + loss
    f += (size_t)n_env * (DA + 2 * H + 4);            // env-step tile
    return (f + 31) & ~(size_t)31;
}

__host__ __device__ inline size_t scratch_floats(int Bc, int H, int DA, int DC, int PA, int PC, int n_env, int nS) {
    return scratch_floats(Bc, H, DA, DC, PA, PC, n_env, nS, tce::shape_ok(Bc, H, DA, DC));
}

__device__ Scr carve(float* base, int Bc, int H, int DA, int DC, int PA, int PC, int n_env, int nS, bool tiles) {
    Scr s;
    float* p = base;
    auto take = [&](size_t n) { float* q = p; p += n; return q; };
    if (tiles) {  // (all multiples of 32 floats from a 128-byte aligned base)
        const size_t nt = (size_t)(Bc / tce::TR) * tce::TILE_FLOATS;
        s.oa = take(nt); s.oa2 = take(nt); s.oc = take(nt); s.oc2 = take(nt);
        s.img = take((size_t)imgs_per_cta(nS) * tce::img_floats(H));
        s.x32 = take((size_t)tce::KP * Bc); s.xn = take(Bc);
        s.X1 = s.X2 = s.H1a = s.H2a = s.H1b = s.H2b = s.dZ2 = s.dZ1 = nullptr;
    } else {
        s.oa = take((size_t)Bc * DA); s.oa2 = take((size_t)Bc * DA);
        s.oc = take((size_t)Bc * DC); s.oc2 = take((size_t)Bc * DC);
        s.X1 = take((size_t)Bc * H); s.X2 = take((size_t)Bc * H);
        s.H1a = take((size_t)Bc * H); s.H2a = take((size_t)Bc * H);
        s.H1b = take((size_t)Bc * H); s.H2b = take((size_t)Bc * H);
        s.dZ2 = take((size_t)Bc * H); s.dZ1 = take((size_t)Bc * H);
        s.img = s.x32 = s.xn = nullptr;
    }
    s.r = take(Bc); s.term = take(Bc); s.y = take(Bc); s.q1 = take(Bc); s.q2 = take(Bc);
    s.mu = take(4 * (size_t)Bc); s.da = take(4 * (size_t)Bc); s.dz3 = take(4 * (size_t)Bc);
    s.ga = take(PA); s.g1 = take(PC); s.g2 = take(PC); s.loss = take(8);
    s.env_obs = take((size_t)n_env * DA); s.env_h1 = take((size_t)n_env * H);
    s.env_h2 = take((size_t)n_env * H); s.env_mu = take((size_t)n_env * 4);
    return s;
}

// ------------------------------------------------------------------- env-step helpers
__device__ __forceinline__ void load_env(const RunDesc& R, int e, float* s, float* d, Prm& P) {
    const int ld = R.C.ld;
#pragma unroll
    for (int i = 0; i < NS; ++i) s[i] = ldcg(R.E.state + i * ld + e);
#pragma unroll
    for (int i = 0; i < 6; ++i) d[i] = ldcg(R.E.dist + i * ld + e);
    const float* pr = R.E.prm;
    P = make_prm(ldcg(pr + e), ldcg(pr + ld + e), ldcg(pr + 2 * ld + e), ldcg(pr + 3 * ld + e),
                 ldcg(pr + 4 * ld + e), ldcg(pr + 5 * ld + e), ldcg(pr + 6 * ld + e));
}

// Actor forward for a handful of rows (n <= 8, hidden <= 64, input <= 128): one warp per
// output unit, lanes split the inputs, every weight load of a warp in flight at once, rows
// reduced with warp shuffles.  x, h: shared memory; the tanh outputs go to Y (global [n][4]).
template <int JT, int KC>
__device__ __forceinline__ void small_layer(const float* Wl, const float* bl, int in, int nout,
                                            const float* x, int ldx, int n, float* y, int ldy,
                                            bool last) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float w[JT][KC], bv[JT];
#pragma unroll
    for (int t = 0; t < JT; ++t) {
        const int j = warp + (LT / 32) * t;
#pragma unroll
        for (int c = 0; c < KC; ++c) {
            const int k = lane + 32 * c;
            w[t][c] = j < nout && k < in ? ldcg(Wl + (size_t)j * in + k) : 0.0f;
        }
        bv[t] = j < nout ? ldcg(bl + j) : 0.0f;
    }
    for (int r = 0; r < n; ++r) {
        float xv[KC];
#pragma unroll
        for (int c = 0; c < KC; ++c) xv[c] = lane + 32 * c < in ? x[r * ldx + lane + 32 * c] : 0.0f;
#pragma unroll
        for (int t = 0; t < JT; ++t) {
            const int j = warp + (LT / 32) * t;
            if (j >= nout) continue;
            float acc = 0.0f;
#pragma unroll
            for (int c = 0; c < KC; ++c) acc = fmaf(w[t][c], xv[c], acc);
            acc = smlp::warp_sum(acc) + bv[t];
            if (lane == 0) y[r * ldy + j] = last ? tanhf(acc) : fmaxf(acc, 0.0f);
        }
    }
}

__device__ __noinline__ void actor_small(const float* W, int in, int H, const float* X, int n,
                                         float* Y, float* sm) {
    constexpr int LX = 132, LH = 68;
    float* xs = sm;
    float* h1 = xs + 8 * LX;
    float* h2 = h1 + 8 * LH;
    for (int i = threadIdx.x; i < n * in; i += LT) xs[(i / in) * LX + i % in] = ldcg(X + i);
    __syncthreads();
    const float* b1 = W + (size_t)H * in;
    const float* W2 = b1 + H;
    const float* b2 = W2 + (size_t)H * H;
    const float* W3 = b2 + H;
    const float* b3 = W3 + 4 * H;
    small_layer<8, 4>(W, b1, in, H, xs, LX, n, h1, LH, false);
    __syncthreads();
    small_layer<8, 2>(W2, b2, H, H, h1, LH, n, h2, LH, false);
    __syncthreads();
    small_layer<1, 2>(W3, b3, H, 4, h2, LH, n, Y, 4, true);
    __syncthreads();
}

// Actor forward of n rows through the shared-memory engine (hidden <= 64).
__device__ __noinline__ void actor_smem(const float* W, int in, int H, const float* X, int n,
                                        float* Y, float* sm) {
    const smlp::Buf b = smlp::carve(sm);
    smlp::stage(W, in, H, 4, b);
    for (int r0 = 0; r0 < n; r0 += smlp::MC)
        smlp::forward(in, H, 4, X, in, r0, min(smlp::MC, n - r0), b, Y, 4, true);
}

// One env step of all envs of run R (executed by one CTA): observation, actor forward
// (generic GEMM path), warm-up / exploration, RK4, reward, termination, record write,
// history update and reset.
__device__ __noinline__ void env_step_cta(RunDesc& R, const Scr& S, uint32_t t, int64_t slot, float* sm) {
    const EnvCfg& C = R.C;
    const int ld = C.ld, n = R.n_env, DA = R.DA, H = R.H;
    const bool warm = (int64_t)t < (int64_t)C.learning_starts;
    if (!warm) {
        for (int e = threadIdx.x; e < n; e += LT) {
            float s[NS], o[18];
#pragma unroll
            for (int i = 0; i < NS; ++i) s[i] = ldcg(R.E.state + i * ld + e);
            obs_state(s, o);
            if (C.any_noise) {
                float nz[18];
                obs_noise(C, (uint32_t)e, t, nz);
#pragma unroll
                for (int k = 0; k < 18; ++k) o[k] += nz[k];
            }
            float* row = S.env_obs + (size_t)e * DA;
#pragma unroll
            for (int k = 0; k < 18; ++k) row[k] = o[k];
            // history loads in two halves, each all in flight before its stores
            const int nh4 = 4 * C.n_hist;
#pragma unroll 1
            for (int h0 = 0; h0 < 4 * HMAX; h0 += 2 * HMAX) {
                float hv[2 * HMAX];
#pragma unroll
                for (int k = 0; k < 2 * HMAX; ++k)
                    hv[k] = h0 + k < nh4 ? ldcg(R.E.hist + (h0 + k) * ld + e) : 0.0f;
#pragma unroll
                for (int k = 0; k < 2 * HMAX; ++k)
                    if (h0 + k < nh4) row[18 + h0 + k] = hv[k];
            }
        }
        __syncthreads();
        if (n <= 8 && H <= 64 && DA <= 128) {
            actor_small(R.actor, DA, H, S.env_obs, n, S.env_mu, sm);
        } else if (H <= smlp::HP && DA <= smlp::INP) {
            actor_smem(R.actor, DA, H, S.env_obs, n, S.env_mu, sm);
        } else {
            mlp_fwd(R.actor, DA, H, 4, S.env_obs, DA, n, S.env_h1, S.env_h2, S.env_mu, 4, true, sm);
        }
    }
    const float sigma = ldcg(R.E.rewardC + 7);
    float Cr[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) Cr[i] = ldcg(R.E.rewardC + i);
    for (int e = threadIdx.x; e < n; e += LT) {
        float s[NS], d[6], a[4];
        Prm P;
        load_env(R, e, s, d, P);
        // episode counters: loads in flight across the integration
        const uint32_t ep_step = ldcg(R.E.ep_step + e);
        const float ret0 = ldcg(R.E.ep_ret + e);
        if (warm) {
            const uint4 r = draw(C, (uint32_t)e, t, TAG_WARM, 0);
            a[0] = 2.0f * u01(r.x) - 1.0f; a[1] = 2.0f * u01(r.y) - 1.0f;
            a[2] = 2.0f * u01(r.z) - 1.0f; a[3] = 2.0f * u01(r.w) - 1.0f;
        } else {
            float mu[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) mu[j] = ldcg(S.env_mu + e * 4 + j);
            if (sigma > 0.0f) {
                const uint4 r0 = draw(C, (uint32_t)e, t, TAG_EXPL, 0);
                const uint4 r1 = draw(C, (uint32_t)e, t, TAG_EXPL, 1);
                a[0] = clampf(fmaf(sigma, gauss(r0.x, r0.y), mu[0]), -1.0f, 1.0f);
                a[1] = clampf(fmaf(sigma, gauss(r0.z, r0.w), mu[1]), -1.0f, 1.0f);
                a[2] = clampf(fmaf(sigma, gauss(r1.x, r1.y), mu[2]), -1.0f, 1.0f);
                a[3] = clampf(fmaf(sigma, gauss(r1.z, r1.w), mu[3]), -1.0f, 1.0f);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) a[j] = clampf(mu[j], -1.0f, 1.0f);
            }
        }
        float u[4], s2[NS];
        action_to_rpm(C.veh, a, u);
#pragma unroll
        for (int i = 0; i < NS; ++i) s2[i] = s[i];
        motor_lag_off(C, u, s2);
        rk4(C.veh, C.dt, C.renorm, s2, u, P, d);
        const float r = reward(Cr, s2, a);
        const bool term = terminated(C, s2);
        const uint32_t ep_after = ep_step + 1;
        const bool trunc = !term && (int)ep_after >= C.episode_len;
        if (R.capacity > 0 && in_bounds(R.E.status, slot, R.E.rows, SITE_RING_WRITE) &&
            in_bounds(R.E.status, e, ld, SITE_SOA)) {
            float* rec = R.E.rec + (size_t)slot * C.F * ld + e;
#pragma unroll
            for (int i = 0; i < NS; ++i) rec[i * ld] = s[i];
#pragma unroll
            for (int i = 0; i < 4; ++i) rec[(17 + i) * ld] = a[i];
            rec[21 * ld] = r;
            rec[22 * ld] = __uint_as_float(pack_flags(term, trunc, ep_step));
            if (C.n_priv) {
                float pv[NPRIV];
                priv_vals(C, P, d, pv);
#pragma unroll
                for (int k = 0; k < NPRIV; ++k) rec[(23 + k) * ld] = pv[k];
            }
            if (term || trunc) {
                float* sd = R.E.side + ((size_t)slot * ld + e) * NS;
#pragma unroll
                for (int i = 0; i < NS; ++i) sd[i] = s2[i];
            }
        }
        {
            // shift the history (newest first) in two halves, the older half first so that
            // no entry is overwritten before it has been loaded: entries [h0, h0 + 30) move
            // to [h0 + 4, h0 + 34)
            const int nh4 = 4 * C.n_hist;
            constexpr int HH = 2 * HMAX - 2;
#pragma unroll 1
            for (int h0 = HH; h0 >= 0; h0 -= HH) {
                float hv[HH];
#pragma unroll
                for (int k = 0; k < HH; ++k)
                    hv[k] = h0 + k + 4 < nh4 ? ldcg(R.E.hist + (h0 + k) * ld + e) : 0.0f;
#pragma unroll
                for (int k = 0; k < HH; ++k)
                    if (h0 + k + 4 < nh4) R.E.hist[(h0 + k + 4) * ld + e] = hv[k];
            }
            if (C.n_hist > 0)
                for (int c = 0; c < 4; ++c) R.E.hist[c * ld + e] = a[c];
        }
        float ret = ret0 + r;
        uint32_t eps = ep_after;
        if (term || trunc) {
            R.E.n_done[e] = ldcg(R.E.n_done + e) + 1;
            R.E.len_sum[e] = ldcg(R.E.len_sum + e) + ep_after;
            R.E.ret_sum[e] = ldcg(R.E.ret_sum + e) + ret;
            const uint32_t epi = ldcg(R.E.ep_index + e) + 1;
            R.E.ep_index[e] = epi;
            float prm7[7];
            reset_env(C, (uint32_t)e, epi, s2, prm7, d);
            for (int i = 0; i < 7; ++i) R.E.prm[i * ld + e] = prm7[i];
            for (int i = 0; i < 6; ++i) R.E.dist[i * ld + e] = d[i];
            for (int i = 0; i < 4 * HMAX; ++i) R.E.hist[i * ld + e] = 0.0f;
            ret = 0.0f;
            eps = 0;
        }
        R.E.ep_ret[e] = ret;
        R.E.ep_step[e] = eps;
#pragma unroll
        for (int i = 0; i < NS; ++i) R.E.state[i * ld + e] = s2[i];
    }
    __syncthreads();
}

// Env step of a run with at most 8 envs (one CTA; a single run's env step sits on the
// critical path of every update): the actor's weights are copied into shared memory
// asynchronously (cp.async, L2 -> shared) while each env's thread loads its state and
// history and builds its observation in shared memory; the three layers then read
// shared memory only; the env's data stay in registers from the observation to the
// write-back, and the history shift reads the observation row already in shared memory.
__device__ __noinline__ void env_step_small(RunDesc& R, uint32_t t, int64_t slot, float* sm) {
    const EnvCfg& C = R.C;
    const int ld = C.ld, n = R.n_env, DA = R.DA, H = R.H, PA = R.PA;
    const bool warm = (int64_t)t < (int64_t)C.learning_starts;
    constexpr int LX = 132, LH = 132;
    float* Ws = sm;                                   // actor parameters, as stored
    float* xs = sm + ((PA + 3) & ~3);                 // [8][LX] observations
    float* h1 = xs + 8 * LX;                          // [8][LH]
    float* h2 = h1 + 8 * LH;                          // [8][LH]
    float* mus = h2 + 8 * LH;                         // [8][4]
    float* park = mus + 8 * 4;                        // [8][32]: env data across the layers
    if (!warm) {
        // 16-byte copies need a 16-byte aligned source (the actor opens the learner's
        // allocation, so it is); otherwise every element goes through the tail loop
        const int nv = ((uintptr_t)R.actor & 15u) == 0 ? PA >> 2 : 0;
        const uint32_t sW = (uint32_t)__cvta_generic_to_shared(Ws);
        for (int v = threadIdx.x; v < nv; v += LT)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(sW + 16u * (uint32_t)v),
                         "l"(R.actor + 4 * v) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
        for (int i = 4 * nv + threadIdx.x; i < PA; i += LT) Ws[i] = ldcg(R.actor + i);
    }
    const int e = threadIdx.x;
    const bool mine = e < n;
    if (mine) {
        // the env's data wait in shared memory while the layers run (no long live ranges)
        float* pk = park + 32 * e;
        float s[NS];
#pragma unroll
        for (int i = 0; i < NS; ++i) s[i] = pk[i] = ldcg(R.E.state + i * ld + e);
#pragma unroll
        for (int i = 0; i < 6; ++i) pk[NS + i] = ldcg(R.E.dist + i * ld + e);
#pragma unroll
        for (int i = 0; i < 7; ++i) pk[NS + 6 + i] = ldcg(R.E.prm + i * ld + e);
        pk[30] = __uint_as_float(ldcg(R.E.ep_step + e));
        pk[31] = ldcg(R.E.ep_ret + e);
        float* row = xs + e * LX;
        const int nh4 = 4 * C.n_hist;
        // history in two halves, each with all its loads in flight before its stores
#pragma unroll 1
        for (int h0 = 0; h0 < 4 * HMAX; h0 += 2 * HMAX) {
            float hv[2 * HMAX];
#pragma unroll
            for (int k = 0; k < 2 * HMAX; ++k) hv[k] = h0 + k < nh4 ? ldcg(R.E.hist + (h0 + k) * ld + e) : 0.0f;
#pragma unroll
            for (int k = 0; k < 2 * HMAX; ++k) row[18 + h0 + k] = hv[k];
        }
        float o[18];
        obs_state(s, o);
        if (!warm && C.any_noise) {
            float nz[18];
            obs_noise(C, (uint32_t)e, t, nz);
#pragma unroll
            for (int k = 0; k < 18; ++k) o[k] += nz[k];
        }
#pragma unroll
        for (int k = 0; k < 18; ++k) row[k] = o[k];
    }
    if (!warm) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        // layers: one warp per output unit; the warp's lanes split into n groups of L (one
        // group per env), each group's lanes over the inputs, group-wide shuffle sums
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const int L = n <= 1 ? 32 : (n <= 2 ? 16 : (n <= 4 ? 8 : 4));
        const int r = lane / L, kq = lane - r * L;
        const bool on = r < n;
        auto gsum = [&](float v) {
            for (int o = L >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            return v;
        };
        const float* b1 = Ws + H * DA;
        const float* W2 = b1 + H;
        const float* b2 = W2 + H * H;
        const float* W3 = b2 + H;
        const float* b3 = W3 + 4 * H;
        for (int j = warp; j < H; j += LT / 32) {
            float acc = 0.0f;
            if (on)
                for (int k = kq; k < DA; k += L) acc = fmaf(Ws[j * DA + k], xs[r * LX + k], acc);
            acc = gsum(acc) + b1[j];
            if (on && kq == 0) h1[r * LH + j] = fmaxf(acc, 0.0f);
        }
        __syncthreads();
        for (int j = warp; j < H; j += LT / 32) {
            float acc = 0.0f;
            if (on)
                for (int k = kq; k < H; k += L) acc = fmaf(W2[j * H + k], h1[r * LH + k], acc);
            acc = gsum(acc) + b2[j];
            if (on && kq == 0) h2[r * LH + j] = fmaxf(acc, 0.0f);
        }
        __syncthreads();
        if (warp < 4) {
            const int o = warp;
            float acc = 0.0f;
            if (on)
                for (int k = kq; k < H; k += L) acc = fmaf(W3[o * H + k], h2[r * LH + k], acc);
            acc = gsum(acc) + b3[o];
            if (on && kq == 0) mus[r * 4 + o] = tanhf(acc);
        }
    }
    __syncthreads();
    if (!mine) return;
    float s[NS], d[6];
    const float* pk = park + 32 * e;
#pragma unroll
    for (int i = 0; i < NS; ++i) s[i] = pk[i];
#pragma unroll
    for (int i = 0; i < 6; ++i) d[i] = pk[NS + i];
    const Prm P = make_prm(pk[23], pk[24], pk[25], pk[26], pk[27], pk[28], pk[29]);
    const uint32_t ep_step = __float_as_uint(pk[30]);
    const float ret0 = pk[31];
    const float sigma = ldcg(R.E.rewardC + 7);
    float Cr[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) Cr[i] = ldcg(R.E.rewardC + i);
    float a[4];
    if (warm) {
        const uint4 r = draw(C, (uint32_t)e, t, TAG_WARM, 0);
        a[0] = 2.0f * u01(r.x) - 1.0f; a[1] = 2.0f * u01(r.y) - 1.0f;
        a[2] = 2.0f * u01(r.z) - 1.0f; a[3] = 2.0f * u01(r.w) - 1.0f;
    } else {
        const float* mu = mus + e * 4;
        if (sigma > 0.0f) {
            const uint4 r0 = draw(C, (uint32_t)e, t, TAG_EXPL, 0);
            const uint4 r1 = draw(C, (uint32_t)e, t, TAG_EXPL, 1);
            a[0] = clampf(fmaf(sigma, gauss(r0.x, r0.y), mu[0]), -1.0f, 1.0f);
            a[1] = clampf(fmaf(sigma, gauss(r0.z, r0.w), mu[1]), -1.0f, 1.0f);
            a[2] = clampf(fmaf(sigma, gauss(r1.x, r1.y), mu[2]), -1.0f, 1.0f);
            a[3] = clampf(fmaf(sigma, gauss(r1.z, r1.w), mu[3]), -1.0f, 1.0f);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) a[j] = clampf(mu[j], -1.0f, 1.0f);
        }
    }
    float u[4], s2[NS];
    action_to_rpm(C.veh, a, u);
#pragma unroll
    for (int i = 0; i < NS; ++i) s2[i] = s[i];
    motor_lag_off(C, u, s2);
    rk4(C.veh, C.dt, C.renorm, s2, u, P, d);
    const float r = reward(Cr, s2, a);
    const bool term = terminated(C, s2);
    const uint32_t ep_after = ep_step + 1;
    const bool trunc = !term && (int)ep_after >= C.episode_len;
    if (R.capacity > 0 && in_bounds(R.E.status, slot, R.E.rows, SITE_RING_WRITE) &&
        in_bounds(R.E.status, e, ld, SITE_SOA)) {
        float* rec = R.E.rec + (size_t)slot * C.F * ld + e;
#pragma unroll
        for (int i = 0; i < NS; ++i) rec[i * ld] = s[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) rec[(17 + i) * ld] = a[i];
        rec[21 * ld] = r;
        rec[22 * ld] = __uint_as_float(pack_flags(term, trunc, ep_step));
        if (C.n_priv) {
            float pv[NPRIV];
            priv_vals(C, P, d, pv);
#pragma unroll
            for (int k = 0; k < NPRIV; ++k) rec[(23 + k) * ld] = pv[k];
        }
        if (term || trunc) {
            float* sd = R.E.side + ((size_t)slot * ld + e) * NS;
#pragma unroll
            for (int i = 0; i < NS; ++i) sd[i] = s2[i];
        }
    }
    float ret = ret0 + r;
    uint32_t eps = ep_after;
    if (term || trunc) {
        R.E.n_done[e] = ldcg(R.E.n_done + e) + 1;
        R.E.len_sum[e] = ldcg(R.E.len_sum + e) + ep_after;
        R.E.ret_sum[e] = ldcg(R.E.ret_sum + e) + ret;
        const uint32_t epi = ldcg(R.E.ep_index + e) + 1;
        R.E.ep_index[e] = epi;
        float prm7[7];
        reset_env(C, (uint32_t)e, epi, s2, prm7, d);
        for (int i = 0; i < 7; ++i) R.E.prm[i * ld + e] = prm7[i];
        for (int i = 0; i < 6; ++i) R.E.dist[i * ld + e] = d[i];
        for (int i = 0; i < 4 * HMAX; ++i) R.E.hist[i * ld + e] = 0.0f;
        ret = 0.0f;
        eps = 0;
    } else {
        // history newest first: a_t, then the previous entries (from the observation row)
        const int nh4 = 4 * C.n_hist;
        const float* row = xs + e * LX + 18;
        for (int k = nh4 - 1; k >= 4; --k) R.E.hist[k * ld + e] = row[k - 4];
        if (C.n_hist > 0)
#pragma unroll
            for (int c = 0; c < 4; ++c) R.E.hist[c * ld + e] = a[c];
    }
    R.E.ep_ret[e] = ret;
    R.E.ep_step[e] = eps;
#pragma unroll
    for (int i = 0; i < NS; ++i) R.E.state[i * ld + e] = s2[i];
}

// ------------------------------------------------------------------------- TD3 update
// Ring index a mod m for a in [-m, 2m).
__device__ __forceinline__ int64_t ring(int64_t a, int64_t m) {
    return a < 0 ? a + m : (a >= m ? a - m : a);
}

// ------------------------------------------------------------------------ replay gather
// Rebuilds o_a, o_a', o_c (with the stored action), o_c' (action slot filled later), r and
// the termination flag of this CTA's samples from the compact replay records, up to GS
// samples a pass.  A sample is ~110 scattered 4-byte values (state, successor state, 17
// actions), each its own 32-byte sector and, with rings beyond L2, its own DRAM access: what
// bounds the pass is how many of them are in flight.  So all samples' indices and flags
// come first (one round trip), then every value goes straight from the ring to shared
// memory with asynchronous copies (no registers, nothing waited for in between; entries
// before the episode start are zero-filled by the copy), and only then the observations are
// formed and written out as coalesced rows.  256 samples on one CTA, values alone: 107 us
// with the ring in DRAM and every SM at it, 27 us from L2 (two cycles a sector, the rate of
// the load path); with the rows 140 and 57 us, against 177 and 72 us for one group of 32
// samples after another through registers.  Prefetching the same sectors into L2 first, as
// tensor-map boxes or line by line, did not shorten it (102 and 119 us for the values).
namespace gat {
constexpr int GS = 256, GP = GS + 1;  // samples a pass; row stride (odd: lanes along rows are conflict-free)
// rows of the shared tile [row][sample]: s, s', a_t, the lags, privileged values, reward,
// then the 18 observation entries of s and s' without and with the actor's noise
constexpr int R_S = 0, R_S2 = NS, R_A = 2 * NS, R_L = R_A + 4, R_PV = R_L + 4 * HMAX, R_R = R_PV + NPRIV,
              R_O = R_R + 1, R_O2 = R_O + 18, R_ON = R_O2 + 18, R_ON2 = R_ON + 18, ROWS = R_ON2 + 18;
constexpr int MAPS = 128;  // entries of a column map (input widths are below that)
constexpr int XE = 4;      // passes of the largest batch
static_assert(GS == tce::TILES_X * tce::TR, "an exponent a pass");
static_assert(ROWS * GP + 3 * GS + 4 * MAPS / 2 <= SMEM_MAIN, "gather tile");

// 4 bytes global -> shared, zero when !ok (nothing is read then)
__device__ __forceinline__ void cp4(float* dst, const float* src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;"
                 :: "r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 4 : 0));
}
}  // namespace gat

template <bool TILES>
__device__ __noinline__ void gather_pass(const RunDesc& R, int j0, int Bc, int g0, int G, uint32_t u, int64_t head,
                                         int64_t size, int64_t t_now, const Scr& S, float* sm, bool need_oa,
                                         int* xe, bool plain_next) {
    using namespace gat;
    const EnvCfg& C = R.C;
    const int ld = C.ld, F = C.F, NE = R.n_env, DA = R.DA, DC = R.DC, nh = C.n_hist;
    const int64_t CAP = R.capacity;
    const int tid = threadIdx.x;
    float* tile = sm;
    int* m_env = reinterpret_cast<int*>(sm + ROWS * GP);                 // sample's env (-1: skipped),
    uint32_t* m_slot = reinterpret_cast<uint32_t*>(m_env + GS);          // slot,
    uint32_t* m_flag = m_slot + GS;                                      // and flags
    int16_t* map = reinterpret_cast<int16_t*>(m_flag + GS);              // tile row of o_a, o_a', o_c, o_c' column k
    // (out of the descriptor once: it lies in global memory)
    int* const bst = R.E.status;
    const float *const ring_rec = R.E.rec, *const ring_side = R.E.side;
    const int64_t rows = R.E.rows;
    const int n_priv = C.n_priv;
    const int64_t lost = size == CAP ? nh : 0;
    const int64_t first = head - size + lost;  // ring position of sample index 0 (before wrapping)
    // ---- column maps
    for (int k = tid; k < MAPS; k += LT) {
        const bool noisy = C.any_noise != 0;
        map[k] = (int16_t)(k < 18 ? (noisy ? R_ON : R_O) + k : R_L + k - 18);
        map[MAPS + k] = (int16_t)(k < 18 ? (noisy ? R_ON2 : R_O2) + k : R_A + k - 18);
        int c = -1, c2 = -1;
        const int act = k - (DC - 4);
        if (act >= 0) {
            c = R_A + act;  // o_c' gets the target action later
        } else if (C.critic_layout == 3) {
            c = map[k];
            c2 = map[MAPS + k];
        } else {
            const int x = k - (C.critic_layout == 2 ? 18 : DA);  // position past observation (and history)
            if (k < 18) { c = R_O + k; c2 = R_O2 + k; }
            else if (x < 0) { c = R_L + k - 18; c2 = R_A + k - 18; }
            else if (x < 4) { c = R_S + 13 + x; c2 = R_S2 + 13 + x; }
            else { c = c2 = R_PV + x - 4; }
        }
        map[2 * MAPS + k] = (int16_t)c;
        map[3 * MAPS + k] = (int16_t)c2;
    }
    // ---- indices and flags
    for (int jl = tid; jl < G; jl += LT) {
        const int j = j0 + g0 + jl;
        const uint32_t nvalid = (uint32_t)((size - 1 - lost) * NE);
        const uint4 rr = draw(C, (uint32_t)j >> 2, u, TAG_REPLAY, 0);
        const uint32_t x = (j & 3) == 0 ? rr.x : ((j & 3) == 1 ? rr.y : ((j & 3) == 2 ? rr.z : rr.w));
        const uint32_t idx = (uint32_t)(((uint64_t)x * (uint64_t)nvalid) >> 32);
        if (R.idx_log) R.idx_log[j] = idx;
        const uint32_t k = idx / (uint32_t)NE;
        const int env = (int)(idx - k * (uint32_t)NE);
        const int64_t slot = ring(first + k, CAP);
        // (debug builds) a slot or env outside the ring skips the sample, status set
        const bool ok = in_bounds(bst, slot, rows, SITE_RING_READ) && in_bounds(bst, env, ld, SITE_SOA);
        m_env[jl] = ok ? env : -1;
        m_slot[jl] = (uint32_t)slot;
        const uint32_t fl = ok ? __float_as_uint(ldcg(ring_rec + ((size_t)slot * F + 22) * ld + env)) : 0u;
        m_flag[jl] = fl;
        S.term[g0 + jl] = (fl & 1u) ? 1.0f : 0.0f;
    }
    __syncthreads();
    // ---- every value of every sample, asynchronously: tps threads share a sample
    int gp = 16;  // samples covered by the CTA at once (a power of two)
    while (gp < G) gp *= 2;
    const int tps = LT / gp, jl = tid & (gp - 1), sub = tid / gp;
    if (jl < G && m_env[jl] >= 0) {
        const int env = m_env[jl];
        const int64_t slot = m_slot[jl];
        const uint32_t fl = m_flag[jl], ep = fl >> 8;
        const bool done = (fl & 3u) != 0;
        const int64_t nslot = ring(slot + 1, CAP);
        const bool nxt_ok = done || in_bounds(bst, nslot, rows, SITE_RING_READ);
        float* T = tile + jl;
        const float* rec = ring_rec + (size_t)slot * F * ld + env;
        // the side slot is env-major (an env's 17 values contiguous), the records field-major
        const float* src2 = done ? ring_side + ((size_t)slot * ld + env) * NS : ring_rec + (size_t)nslot * F * ld + env;
        const size_t st2 = done ? 1 : (size_t)ld;
        for (int i = sub; i < NS; i += tps) {
            cp4(T + (R_S + i) * GP, rec + (size_t)i * ld, true);
            cp4(T + (R_S2 + i) * GP, nxt_ok ? src2 + i * st2 : rec, nxt_ok);
        }
        // a_t and the lags i = 1..n_hist; zeros before the episode start
        for (int i = sub; i <= nh; i += tps) {
            const int64_t sl = ring(slot - i, CAP);
            const bool ok = i == 0 || ((uint32_t)i <= ep && in_bounds(bst, sl, rows, SITE_RING_READ));
            const float* ap = ok ? ring_rec + ((size_t)sl * F + 17) * ld + env : rec;
#pragma unroll
            for (int c = 0; c < 4; ++c) cp4(T + (R_A + 4 * i + c) * GP, ap + (ok ? c * ld : 0), ok);
        }
        if (sub == tps - 1) {
            cp4(T + R_R * GP, rec + (size_t)21 * ld, true);
            for (int k = 0; k < n_priv; ++k) cp4(T + (R_PV + k) * GP, rec + (size_t)(23 + k) * ld, true);
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // ---- observations, one (sample, side) per thread
    for (int i = tid; i < 2 * G; i += LT) {
        const int side = i >= G, js = i - side * G;
        if (m_env[js] < 0) continue;
        float* T = tile + js;
        float* st = T + (side ? R_S2 : R_S) * GP;
        float sv[NS], o[18];
#pragma unroll
        for (int q = 0; q < NS; ++q) sv[q] = st[q * GP];
        obs_state(sv, o);
        float* ot = T + (side ? R_O2 : R_O) * GP;
#pragma unroll
        for (int q = 0; q < 18; ++q) ot[q * GP] = o[q];
#pragma unroll
        for (int q = 0; q < 4; ++q) st[(13 + q) * GP] = rpm_norm(C.veh, sv[13 + q]);
        if (side == 0) S.r[g0 + js] = T[R_R * GP];
    }
    __syncthreads();
    if (C.any_noise) {
        // the actor's observation noise of s_t (side 0, step t_rec) and s_{t+1} (side 1, step
        // t_rec + 1): 9 Philox blocks per side
        for (int i = tid; i < 18 * G; i += LT) {
            const int pr = i / G, js = i - pr * G, side = pr >= 9, blk = pr - 9 * side;
            if (m_env[js] < 0) continue;
            int64_t k = (int64_t)m_slot[js] - first;  // sample index's time slot
            while (k < 0) k += CAP;
            while (k >= CAP) k -= CAP;
            float n0, n1;
            obs_noise_pair(C, (uint32_t)m_env[js], (uint32_t)(t_now - size + lost + k) + (uint32_t)side, blk, n0, n1);
            const float* ot = tile + ((side ? R_O2 : R_O) + 2 * blk) * GP + js;
            float* nt = tile + ((side ? R_ON2 : R_ON) + 2 * blk) * GP + js;
            nt[0] = ot[0] + n0;
            nt[GP] = ot[GP] + n1;
        }
        __syncthreads();
    }
    // ---- rows of the scratch
    const int warp = tid >> 5, lane = tid & 31;
    if constexpr (TILES) {
        // input tiles of the tensor-core passes: lane = sample, 8 columns of one matrix at a
        // time as hi / lo halves (zero past the input width; a core matrix row is 16 bytes,
        // 8 samples make 128); o_c' gets the target action later.  A warp keeps a column
        // group's tile rows for all of its samples.
        constexpr int KC = tce::KC1;
        const bool need_oc = need_oa || R.H == 128;  // hidden <= 64: o_c's tile is read on the actor's step only
        // The power of two that this pass's samples are scaled by, one for o_a and o_c and one
        // for o_a' and o_c' (none where the passes take them plain): their largest magnitude
        // goes below 2^X_TOP.  Actions that are put in later are at most 1.
        float mx = 1.0f, mx2 = 1.0f;
        for (int js = tid; js < G; js += LT) {
            if (m_env[js] < 0) continue;
            const float* T = tile + js;
            if (need_oc) {
                float n = 0.0f;
#pragma unroll 8
                for (int k = 0; k < DC; ++k) {
                    const float v = fabsf(T[map[2 * MAPS + k] * GP]);
                    n += v;
                    mx = fmaxf(mx, v);
                }
                if (R.H == 128) S.xn[g0 + js] = n;
            }
            // (o_a has o_c's columns but for the noise, unless the critic sees no history)
            if (need_oa)
#pragma unroll 8
                for (int k = 0; k < DA; ++k) mx = fmaxf(mx, fabsf(T[map[k] * GP]));
            if (!plain_next) {
#pragma unroll 8
                for (int k = 0; k < DA; ++k) mx2 = fmaxf(mx2, fabsf(T[map[MAPS + k] * GP]));
#pragma unroll 8
                for (int k = 0; k < DC - 4; ++k) mx2 = fmaxf(mx2, fabsf(T[map[3 * MAPS + k] * GP]));
            }
        }
        {
            float* red = sm + SMEM_MAIN;
            for (int o = 16; o > 0; o >>= 1) {
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                mx2 = fmaxf(mx2, __shfl_xor_sync(0xffffffffu, mx2, o));
            }
            if (lane == 0) {
                red[warp] = mx;
                red[8 + warp] = mx2;
            }
            __syncthreads();
            for (int i = 0; i < LT / 32; ++i) {
                mx = fmaxf(mx, red[i]);
                mx2 = fmaxf(mx2, red[8 + i]);
            }
        }
        const int e_cur = tce::scale_max(tce::X_TOP, mx), e_next = plain_next ? 0 : tce::scale_max(tce::X_TOP, mx2);
        if (tid == 0) {
            xe[g0 / GS] = e_cur;
            xe[XE + g0 / GS] = e_next;
        }
        const float x_cur = tce::exp2i(e_cur), x_next = tce::exp2i(e_next);
        // o_c in FP32 rows for the critics' regression, a warp per sample
        float* const x32 = S.x32;
        for (int js = warp; js < G; js += LT / 32) {
            if (m_env[js] < 0) continue;
            float v[3];
#pragma unroll
            for (int e = 0; e < 3; ++e) v[e] = lane + 32 * e < DC ? tile[map[2 * MAPS + lane + 32 * e] * GP + js] : 0.0f;
#pragma unroll
            for (int e = 0; e < 3; ++e)
                if (lane + 32 * e < DC) x32[(size_t)(g0 + js) * DC + lane + 32 * e] = v[e];
        }
        float *const t_oa = S.oa, *const t_oa2 = S.oa2, *const t_oc = S.oc, *const t_oc2 = S.oc2;
        for (int q = (need_oa ? 0 : KC) + warp; q < 4 * KC; q += LT / 32) {
            if (!need_oc && q / KC == 2) continue;
            const int mat = q / KC, kc = q - mat * KC;
            const int w = mat < 2 ? DA : (mat == 2 ? DC : DC - 4);
            float* const d = mat == 0 ? t_oa : (mat == 1 ? t_oa2 : (mat == 2 ? t_oc : t_oc2));
            int row8[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) row8[e] = 8 * kc + e < w ? map[mat * MAPS + 8 * kc + e] * GP : -1;
#pragma unroll 2
            for (int s0 = 0; s0 < G; s0 += 32) {
                const int js = s0 + lane, j = g0 + js;
                float v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = row8[e] >= 0 ? tile[row8[e] + js] * (mat & 1 ? x_next : x_cur) : 0.0f;
                if (m_env[js] < 0) continue;
                unsigned char* t = reinterpret_cast<unsigned char*>(d + (size_t)(j / tce::TR) * tce::TILE_FLOATS);
                tce::put8(t, t + 2 * tce::TILE_HALVES, KC, j % tce::TR, 8 * kc, v);
            }
        }
    } else {
        // FP32 rows, a warp per sample, 4 columns per lane and matrix in flight
        for (int js = warp; js < G; js += LT / 32) {
            if (m_env[js] < 0) continue;
            const size_t j = (size_t)(g0 + js);
            const float* T = tile + js;
#pragma unroll
            for (int mat = 0; mat < 4; ++mat) {
                const int w = mat < 2 ? DA : DC, n = mat == 3 ? DC - 4 : w;
                float* d = (mat == 0 ? S.oa : (mat == 1 ? S.oa2 : (mat == 2 ? S.oc : S.oc2))) + j * w;
                float v[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = lane + 32 * e < n ? T[map[mat * MAPS + lane + 32 * e] * GP] : 0.0f;
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (lane + 32 * e < n) d[lane + 32 * e] = v[e];
            }
        }
    }
    __syncthreads();
}

// Gather of this CTA's Bc samples (sm: shared memory, free at this point); need_oa: whether this
// update reads o_a (the actor's step).  In tiles: xe gets the passes' exponents, plain_next
// leaves those of s_{t+1} at zero.
template <bool TILES>
__device__ __forceinline__ void gather_all(const RunDesc& R, int j0, int Bc, uint32_t u,
                                           int64_t head, int64_t size, int64_t t_now,
                                           const Scr& S, float* sm, bool need_oa = true, int* xe = nullptr,
                                           bool plain_next = true) {
    for (int g0 = 0; g0 < Bc; g0 += gat::GS)
        gather_pass<TILES>(R, j0, Bc, g0, min(gat::GS, Bc - g0), u, head, size, t_now, S, sm, need_oa, xe, plain_next);
}

// Adam on parameters [lo, hi) from the sum of S gradient partials (partial s at
// gpart_base + s * part_stride + goff, summed in the order s = 0..S-1); with tg != nullptr
// the target copy also takes its Polyak step tg = tau th + (1 - tau) tg from the new th
// (the fused form of polyak_slice, for steps that update the targets).  img / timg: halves
// of the network and its target for the tensor-core passes, kept in step.
// Bound by issue and the latency of its loads: 10,500 parameters on one CTA take 20,000 cycles
// (9.7 us), 12,500 without the two divisions by the bias corrections, the quotient and the
// root, whose roundings the weights keep; the halves add 8,000.  Loads of the next block
// ahead of this block's arithmetic were slower (61 against 52 us for two critics).
__device__ void adam_slice(float* th, const float* gpart_base, size_t part_stride, int S,
                           int goff, float* m, float* v, int lo, int hi, int64_t t,
                           const LearnHyper& hp, float gscale, float* tg = nullptr,
                           const tce::Img img = tce::Img(), const tce::Img timg = tce::Img()) {
    const float beta1 = hp.beta1, beta2 = hp.beta2, lr = hp.lr, eps = hp.eps, tau = hp.tau;
    const float bc1 = 1.0f - powf(beta1, (float)t);
    const float bc2 = 1.0f - powf(beta2, (float)t);
    // U elements per thread per pass, all their loads issued before the arithmetic (8 was
    // measured no faster on the batched runs and 2.4 % slower on the single run).  The loop is
    // the same for every thread of the CTA: put_lanes needs whole warps.
    constexpr int U = 4;
    for (int b = lo; b < hi; b += U * LT) {
        float g[U], mo[U], vo[U], to[U], tt[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int i = b + (int)threadIdx.x + k * LT;
            g[k] = 0.0f; mo[k] = 0.0f; vo[k] = 0.0f; to[k] = 0.0f; tt[k] = 0.0f;
            if (i < hi) {
                mo[k] = m[i]; vo[k] = v[i]; to[k] = th[i];
                if (tg) tt[k] = tg[i];
            }
        }
        // partials in batches of 4 (4 x U loads in flight)
        for (int s0 = 0; s0 < S; s0 += 4) {
            float x[4][U];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float* gp = gpart_base + (size_t)(s0 + q) * part_stride + goff;
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    const int i = b + (int)threadIdx.x + k * LT;
                    x[q][k] = s0 + q < S && i < hi ? ldcg(gp + i) : 0.0f;
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int k = 0; k < U; ++k)
                    if (s0 + q < S) g[k] += x[q][k];
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const float gk = g[k] * gscale;
            const float mi = fmaf(beta1, mo[k], (1.0f - beta1) * gk);
            const float vi = fmaf(beta2, vo[k], (1.0f - beta2) * gk * gk);
            mo[k] = mi;
            vo[k] = vi;
            to[k] = to[k] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
            tt[k] = fmaf(tau, to[k], (1.0f - tau) * tt[k]);
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int i = b + (int)threadIdx.x + k * LT;
            if (i < hi) {
                m[i] = mo[k];
                v[i] = vo[k];
                th[i] = to[k];
                if (tg) tg[i] = tt[k];
            }
            if (img.p) img.put_lanes(i, hi, to[k]);
            if (tg && timg.p) timg.put_lanes(i, hi, tt[k]);
        }
    }
}

__device__ void polyak_slice(float* tg, const float* src, int lo, int hi, float tau) {
    constexpr int U = 4;
    for (int i0 = lo + threadIdx.x; i0 < hi; i0 += U * LT) {
        float a[U], b[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int i = i0 + k * LT;
            a[k] = i < hi ? ldcg(src + i) : 0.0f;
            b[k] = i < hi ? tg[i] : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < U; ++k)
            if (i0 + k * LT < hi) tg[i0 + k * LT] = fmaf(tau, a[k], (1.0f - tau) * b[k]);
    }
}

// Block-wide sum of v over threads (fixed order).
__device__ float block_sum(float v, float* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    float s = 0.0f;
    for (int i = 0; i < LT / 32; ++i) s += red[i];
    __syncthreads();
    return s;
}

// One TD3 update of run R by the cluster (rank `rk` of S).
__device__ __noinline__ void td3_update(RunDesc& R, int64_t head, int64_t size, int64_t t_now, uint32_t u,
                           int64_t& t_a, int64_t& t_c, const Scr& S, float* scr_base,
                           size_t scr_stride, int cl_base, int rk, int nS, float* sm) {
    const int B = R.B, Bc = B / nS, H = R.H, DA = R.DA, DC = R.DC, PA = R.PA, PC = R.PC;
    const LearnHyper& hp = R.hp;
    const int j0 = rk * Bc;
    // a9: gather
    gather_all<false>(R, j0, Bc, u, head, size, t_now, S, sm);
    __syncthreads();
    // a10: target actor + smoothing
    mlp_fwd(R.actor_t, DA, H, 4, S.oa2, DA, Bc, S.X1, S.X2, S.mu, 4, true, sm);
    for (int jl = threadIdx.x; jl < Bc; jl += LT) {
        const uint32_t j = (uint32_t)(j0 + jl);
        const uint4 r0 = draw(R.C, j, u, TAG_SMOOTH, 0), r1 = draw(R.C, j, u, TAG_SMOOTH, 1);
        const float z[4] = {gauss(r0.x, r0.y), gauss(r0.z, r0.w), gauss(r1.x, r1.y), gauss(r1.z, r1.w)};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float eps = clampf(hp.sigma_t * z[i], -hp.noise_clip, hp.noise_clip);
            S.oc2[(size_t)jl * DC + DC - 4 + i] = clampf(S.mu[jl * 4 + i] + eps, -1.0f, 1.0f);
        }
    }
    __syncthreads();
    // a11: twin target critics, clipped double-Q target
    mlp_fwd(R.c1_t, DC, H, 1, S.oc2, DC, Bc, S.X1, S.X2, S.q1, 1, false, sm);
    mlp_fwd(R.c2_t, DC, H, 1, S.oc2, DC, Bc, S.X1, S.X2, S.q2, 1, false, sm);
    for (int jl = threadIdx.x; jl < Bc; jl += LT) {
        const float qmin = fminf(S.q1[jl], S.q2[jl]);
        S.y[jl] = S.r[jl] + (S.term[jl] != 0.0f ? 0.0f : hp.gamma * qmin);
    }
    __syncthreads();
    // a12: critic regression, forward + backward on this CTA's samples
    mlp_fwd(R.c1, DC, H, 1, S.oc, DC, Bc, S.H1a, S.H2a, S.q1, 1, false, sm);
    mlp_fwd(R.c2, DC, H, 1, S.oc, DC, Bc, S.H1b, S.H2b, S.q2, 1, false, sm);
    float lsum = 0.0f;
    for (int jl = threadIdx.x; jl < Bc; jl += LT) {
        const float e1 = S.q1[jl] - S.y[jl], e2 = S.q2[jl] - S.y[jl];
        S.dz3[jl] = 2.0f * e1 / (float)B;
        S.da[jl] = 2.0f * e2 / (float)B;
        lsum += (e1 * e1 + e2 * e2) / (float)B;
    }
    lsum = block_sum(lsum, sm + SMEM_MAIN);
    if (threadIdx.x == 0) S.loss[0] = lsum;
    __syncthreads();
    mlp_bwd(R.c1, DC, H, 1, S.oc, DC, Bc, S.H1a, S.H2a, S.dz3, S.dZ2, S.dZ1, S.g1, nullptr, 0, sm);
    mlp_bwd(R.c2, DC, H, 1, S.oc, DC, Bc, S.H1b, S.H2b, S.da, S.dZ2, S.dZ1, S.g2, nullptr, 0, sm);
    cluster_sync_all(nS);
    // a14 (critics): reduce the partials over the cluster and apply Adam to this slice
    t_c += 1;
    {
        const size_t g1off = (size_t)(S.g1 - scr_base), g2off = (size_t)(S.g2 - scr_base);
        const float* cl0 = scr_base - (size_t)rk * scr_stride;  // scratch of cluster rank 0
        const int lo = (int)((int64_t)PC * rk / nS), hi = (int)((int64_t)PC * (rk + 1) / nS);
        adam_slice(R.c1, cl0, scr_stride, nS, (int)g1off, R.m_c1, R.v_c1, lo, hi, t_c, hp, 1.0f);
        adam_slice(R.c2, cl0, scr_stride, nS, (int)g2off, R.m_c2, R.v_c2, lo, hi, t_c, hp, 1.0f);
        if (rk == 0 && threadIdx.x == 0) {
            float l = 0.0f;
            for (int s = 0; s < nS; ++s) l += ldcg(cl0 + (size_t)s * scr_stride + (S.loss - scr_base));
            R.stats[0] = l;
        }
    }
    cluster_sync_all(nS);
    // a13: delayed actor update through the updated first critic
    if ((int64_t)(u % (uint32_t)hp.policy_delay) != (int64_t)(hp.policy_delay - 1)) return;
    mlp_fwd(R.actor, DA, H, 4, S.oa, DA, Bc, S.X1, S.X2, S.mu, 4, true, sm);
    for (int i = threadIdx.x; i < Bc * 4; i += LT) {
        const int jl = i >> 2, c = i & 3;
        S.oc[(size_t)jl * DC + DC - 4 + c] = S.mu[i];
    }
    __syncthreads();
    mlp_fwd(R.c1, DC, H, 1, S.oc, DC, Bc, S.H1a, S.H2a, S.q1, 1, false, sm);
    float qs = 0.0f;
    for (int jl = threadIdx.x; jl < Bc; jl += LT) {
        S.dz3[jl] = -1.0f / (float)B;
        qs += -S.q1[jl] / (float)B;
    }
    qs = block_sum(qs, sm + SMEM_MAIN);
    if (threadIdx.x == 0) S.loss[1] = qs;
    __syncthreads();
    // dQ1/d(input) restricted to the action columns [DC-4, DC) -> dX stored in oc2 rows
    mlp_bwd(R.c1, DC, H, 1, S.oc, DC, Bc, S.H1a, S.H2a, S.dz3, S.dZ2, S.dZ1, nullptr, S.oc2, DC - 4, sm);
    for (int i = threadIdx.x; i < Bc * 4; i += LT) {
        const int jl = i >> 2, c = i & 3;
        const float m = S.mu[i];
        S.da[i] = S.oc2[(size_t)jl * DC + DC - 4 + c] * (1.0f - m * m);
    }
    __syncthreads();
    mlp_bwd(R.actor, DA, H, 4, S.oa, DA, Bc, S.X1, S.X2, S.da, S.dZ2, S.dZ1, S.ga, nullptr, 0, sm);
    cluster_sync_all(nS);
    t_a += 1;
    {
        const size_t gaoff = (size_t)(S.ga - scr_base);
        const float* cl0 = scr_base - (size_t)rk * scr_stride;
        const int lo = (int)((int64_t)PA * rk / nS), hi = (int)((int64_t)PA * (rk + 1) / nS);
        adam_slice(R.actor, cl0, scr_stride, nS, (int)gaoff, R.m_a, R.v_a, lo, hi, t_a, hp, 1.0f);
        if (rk == 0 && threadIdx.x == 0) {
            float l = 0.0f;
            for (int s = 0; s < nS; ++s) l += ldcg(cl0 + (size_t)s * scr_stride + (S.loss - scr_base) + 1);
            R.stats[1] = l;
        }
        __syncthreads();
        polyak_slice(R.actor_t, R.actor, lo, hi, hp.tau);
        const int clo = (int)((int64_t)PC * rk / nS), chi = (int)((int64_t)PC * (rk + 1) / nS);
        polyak_slice(R.c1_t, R.c1, clo, chi, hp.tau);
        polyak_slice(R.c2_t, R.c2, clo, chi, hp.tau);
    }
    cluster_sync_all(nS);
}

// One TD3 update with every network pass resident in shared memory (hidden <= 64, or the
// 128-wide engine shape for HT = 128): same phases and cluster reduction as td3_update.  HT/DAT/DCT fix the hidden width and the
// actor/critic input widths at compile time (0: taken from the run descriptor), so that the
// common shapes get fully unrolled shared-memory GEMMs.
template <int HT, int DAT, int DCT>
__device__ __noinline__ void td3_update_smem(RunDesc& R, int64_t head, int64_t size, int64_t t_now,
                                             uint32_t u, int64_t& t_a, int64_t& t_c, const Scr& S,
                                             float* scr_base, size_t scr_stride, int rk, int nS,
                                             float* sm) {
    using namespace smlp;
    const int B = R.B, Bc = B / nS, PA = R.PA, PC = R.PC;
    const int H = HT ? HT : R.H, DA = DAT ? DAT : R.DA, DC = DCT ? DCT : R.DC;
    const LearnHyper& hp = R.hp;
    const int j0 = rk * Bc;
    Buf b = HT == 128 ? carve2(sm) : carve(sm);  // the 64-wide shape is never re-bound
    const int MC = b.mc;
    float* red = sm + SMEM_MAIN;
    // a9: gather
    gather_all<false>(R, j0, Bc, u, head, size, t_now, S, sm);
    __syncthreads();
    // With an even cluster whose CTA pairs' rows fit one chunk, the twin critics are split
    // over the two halves: CTA rk runs critic cs = rk / half (target and current) on the
    // rows of the pair (rr, rr + half), rr = rk mod half, read from both owners' scratch.
    const int half = nS >> 1;
    const bool split = half > 0 && (nS & 1) == 0 && 2 * Bc <= MC;
    const int cs = split ? rk / half : 0, rr = split ? rk - cs * half : rk;
    const ptrdiff_t d0 = (ptrdiff_t)(rr - rk) * (ptrdiff_t)scr_stride;
    const ptrdiff_t d1 = (ptrdiff_t)(rr + half - rk) * (ptrdiff_t)scr_stride;
    // a10: target actor + smoothing
    stage(R.actor_t, DA, H, 4, b);
    for (int r0 = 0; r0 < Bc; r0 += MC) forward(DA, H, 4, S.oa2, DA, r0, min(MC, Bc - r0), b, S.mu, 4, true);
    for (int jl = threadIdx.x; jl < Bc; jl += LT) {
        const uint32_t j = (uint32_t)(j0 + jl);
        const uint4 r0 = draw(R.C, j, u, TAG_SMOOTH, 0), r1 = draw(R.C, j, u, TAG_SMOOTH, 1);
        const float z[4] = {gauss(r0.x, r0.y), gauss(r0.z, r0.w), gauss(r1.x, r1.y), gauss(r1.z, r1.w)};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float eps = clampf(hp.sigma_t * z[i], -hp.noise_clip, hp.noise_clip);
            S.oc2[(size_t)jl * DC + DC - 4 + i] = clampf(S.mu[jl * 4 + i] + eps, -1.0f, 1.0f);
        }
    }
    __syncthreads();
    // a11: twin target critics
    if (split) {
        cluster_sync_all(nS);  // the pair's o_c' rows are complete
        float* qt = cs ? S.q2 : S.q1;
        stage(cs ? R.c2_t : R.c1_t, DC, H, 1, b);
        forward2(DC, H, 1, S.oc2 + d0, S.oc2 + d1, DC, Bc, 2 * Bc, b, qt + d0, qt + d1, 1, false);
        cluster_sync_all(nS);  // both target values of the pair's rows are complete
    } else {
        stage(R.c1_t, DC, H, 1, b);
        for (int r0 = 0; r0 < Bc; r0 += MC) forward(DC, H, 1, S.oc2, DC, r0, min(MC, Bc - r0), b, S.q1, 1, false);
        stage(R.c2_t, DC, H, 1, b);
        for (int r0 = 0; r0 < Bc; r0 += MC) forward(DC, H, 1, S.oc2, DC, r0, min(MC, Bc - r0), b, S.q2, 1, false);
    }
    if (!split) {
        for (int jl = threadIdx.x; jl < Bc; jl += LT) {
            const float qmin = fminf(S.q1[jl], S.q2[jl]);
            S.y[jl] = S.r[jl] + (S.term[jl] != 0.0f ? 0.0f : hp.gamma * qmin);
        }
    }
    __syncthreads();
    // a12: critic regression, forward + backward chunk by chunk
    float lsum = 0.0f;
    if (split) {
        // one chunk: the pair's 2 Bc rows through critic cs; Q into dz3 (scratch of this CTA)
        float* g = cs ? S.g2 : S.g1;
        stage(cs ? R.c2 : R.c1, DC, H, 1, b);
        if constexpr (HT == 128) bind_grads(b, g, DC, H, 1);
        forward2(DC, H, 1, S.oc + d0, S.oc + d1, DC, Bc, 2 * Bc, b, S.dz3, S.dz3 + Bc, 1, false);
        for (int r = threadIdx.x; r < 2 * Bc; r += LT) {
            const ptrdiff_t o = (r < Bc ? d0 : d1) + (r < Bc ? r : r - Bc);
            const float qmin = fminf(S.q1[o], S.q2[o]);
            const float y = S.r[o] + (S.term[o] != 0.0f ? 0.0f : hp.gamma * qmin);
            const float e = S.dz3[r] - y;
            b.dZ3s[r * 4] = 2.0f * e / (float)B;
            lsum += e * e / (float)B;
        }
        __syncthreads();
        backward(DC, H, 1, 0, 2 * Bc, b, true, true, nullptr, 0, 0);
        store_grads(g, DC, H, 1, b);
    }
    for (int c = 0; c < (split ? 0 : 2); ++c) {
        const float* W = c ? R.c2 : R.c1;
        float* q = c ? S.q2 : S.q1;
        stage(W, DC, H, 1, b);
        if constexpr (HT == 128) bind_grads(b, c ? S.g2 : S.g1, DC, H, 1);
        for (int r0 = 0; r0 < Bc; r0 += MC) {
            const int mc = min(MC, Bc - r0);
            forward(DC, H, 1, S.oc, DC, r0, mc, b, q, 1, false);
            for (int r = threadIdx.x; r < mc; r += LT) {
                const float e = q[r0 + r] - S.y[r0 + r];
                b.dZ3s[r * 4] = 2.0f * e / (float)B;
                lsum += e * e / (float)B;
            }
            __syncthreads();
            backward(DC, H, 1, r0, mc, b, r0 == 0, true, nullptr, 0, 0);
        }
        store_grads(c ? S.g2 : S.g1, DC, H, 1, b);
    }
    lsum = block_sum(lsum, red);
    if (threadIdx.x == 0) S.loss[0] = lsum;
    __syncthreads();
    cluster_sync_all(nS);
    // a14 (critics): reduce the partials over the cluster and apply Adam to this slice
    t_c += 1;
    {
        const size_t g1off = (size_t)(S.g1 - scr_base), g2off = (size_t)(S.g2 - scr_base);
        const float* cl0 = scr_base - (size_t)rk * scr_stride;
        const int lo = (int)((int64_t)PC * rk / nS), hi = (int)((int64_t)PC * (rk + 1) / nS);
        // split: critic 1's partials are in CTAs [0, half), critic 2's in [half, nS)
        const int np = split ? half : nS;
        // on steps that update the actor, the critics' targets take their Polyak step here
        // (the actor phase reads the critics, not their targets)
        const bool pol = (int64_t)(u % (uint32_t)hp.policy_delay) == (int64_t)(hp.policy_delay - 1);
        adam_slice(R.c1, cl0, scr_stride, np, (int)g1off, R.m_c1, R.v_c1, lo, hi, t_c, hp, 1.0f,
                   pol ? R.c1_t : nullptr);
        adam_slice(R.c2, cl0 + (split ? (size_t)half * scr_stride : 0), scr_stride, np, (int)g2off,
                   R.m_c2, R.v_c2, lo, hi, t_c, hp, 1.0f, pol ? R.c2_t : nullptr);
        if (rk == 0 && threadIdx.x == 0) {
            float l = 0.0f;
            for (int s2 = 0; s2 < nS; ++s2) l += ldcg(cl0 + (size_t)s2 * scr_stride + (S.loss - scr_base));
            R.stats[0] = l;
        }
    }
    cluster_sync_all(nS);
    // a13: delayed actor update through the updated first critic
    if ((int64_t)(u % (uint32_t)hp.policy_delay) != (int64_t)(hp.policy_delay - 1)) return;
    // mu(o_a) alone (no activations kept)
    stage(R.actor, DA, H, 4, b);
    for (int r0 = 0; r0 < Bc; r0 += MC) forward(DA, H, 4, S.oa, DA, r0, min(MC, Bc - r0), b, S.mu, 4, true);
    for (int i = threadIdx.x; i < Bc * 4; i += LT) {
        const int jl = i >> 2, c = i & 3;
        S.oc[(size_t)jl * DC + DC - 4 + c] = S.mu[i];
    }
    __syncthreads();
    stage(R.c1, DC, H, 1, b);
    float qs = 0.0f;
    for (int r0 = 0; r0 < Bc; r0 += MC) {
        const int mc = min(MC, Bc - r0);
        forward(DC, H, 1, S.oc, DC, r0, mc, b, S.q1, 1, false);
        for (int r = threadIdx.x; r < mc; r += LT) {
            b.dZ3s[r * 4] = -1.0f / (float)B;
            qs += -S.q1[r0 + r] / (float)B;
        }
        __syncthreads();
        // dQ1/d(action columns) -> oc2 rows
        backward(DC, H, 1, r0, mc, b, false, false, S.oc2, DC, DC - 4);
    }
    qs = block_sum(qs, red);
    if (threadIdx.x == 0) S.loss[1] = qs;
    for (int i = threadIdx.x; i < Bc * 4; i += LT) {
        const int jl = i >> 2, c = i & 3;
        const float m = S.mu[i];
        S.da[i] = S.oc2[(size_t)jl * DC + DC - 4 + c] * (1.0f - m * m);
    }
    __syncthreads();
    stage(R.actor, DA, H, 4, b);
    if constexpr (HT == 128) bind_grads(b, S.ga, DA, H, 4);
    for (int r0 = 0; r0 < Bc; r0 += MC) {
        const int mc = min(MC, Bc - r0);
        forward(DA, H, 4, S.oa, DA, r0, mc, b, S.mu, 4, true);
        for (int i = threadIdx.x; i < mc * 4; i += LT) b.dZ3s[i] = S.da[r0 * 4 + i];
        __syncthreads();
        backward(DA, H, 4, r0, mc, b, r0 == 0, true, nullptr, 0, 0);
    }
    store_grads(S.ga, DA, H, 4, b);
    cluster_sync_all(nS);
    t_a += 1;
    {
        const size_t gaoff = (size_t)(S.ga - scr_base);
        const float* cl0 = scr_base - (size_t)rk * scr_stride;
        const int lo = (int)((int64_t)PA * rk / nS), hi = (int)((int64_t)PA * (rk + 1) / nS);
        adam_slice(R.actor, cl0, scr_stride, nS, (int)gaoff, R.m_a, R.v_a, lo, hi, t_a, hp, 1.0f, R.actor_t);
        if (rk == 0 && threadIdx.x == 0) {
            float l = 0.0f;
            for (int s2 = 0; s2 < nS; ++s2) l += ldcg(cl0 + (size_t)s2 * scr_stride + (S.loss - scr_base) + 1);
            R.stats[1] = l;
        }
    }
    cluster_sync_all(nS);
}

// Critic regression of a CTA's rows on the shared-memory engine (hidden <= 64), forward and
// backward chunk by chunk; IN: the critic's input width (0: in), fixed for the widths that
// td3_update_smem is compiled for as well: 90 (16 actions of history) at hidden 32 and 64, and
// 96 (the privileged critic) at 64.  Returns this thread's part of the loss.
template <int H, int IN>
__device__ __noinline__ float critics_smem(const RunDesc& R, const Scr& S, int Bc, int in, float* sm) {
    using namespace smlp;
    const int DC = IN ? IN : in, B = R.B;
    const Buf b = carve(sm);
    float lsum = 0.0f;
    for (int c = 0; c < 2; ++c) {
        float* q = c ? S.q2 : S.q1;
        stage(c ? R.c2 : R.c1, DC, H, 1, b);
        for (int r0 = 0; r0 < Bc; r0 += MC) {
            const int mc = min(MC, Bc - r0);
            forward(DC, H, 1, S.x32, DC, r0, mc, b, q, 1, false);
            for (int r = threadIdx.x; r < mc; r += LT) {
                const float e = q[r0 + r] - S.y[r0 + r];
                b.dZ3s[r * 4] = 2.0f * e / (float)B;
                lsum += e * e / (float)B;
            }
            __syncthreads();
            backward(DC, H, 1, r0, mc, b, r0 == 0, true, nullptr, 0, 0);
        }
        store_grads(c ? S.g2 : S.g1, DC, H, 1, b);
    }
    return lsum;
}

// What a CTA keeps about the tensor-core passes in shared memory, alike in a cluster: the
// networks' exponents (of the images), the gathered samples', and whether a wait ran out.
struct TcState {
    tce::NetScale net[6];
    int xe[2 * gat::XE];
    int dead;
};

// Whether the passes of the target networks take their operands as they are and in one chain: at
// hidden 32 and 64, where they feed the critics' FP32 regression and keep the bits they had.
__host__ __device__ constexpr bool plain_targets(int H) { return H != 128; }

__device__ __forceinline__ float2 block_max2(float a, float b, float* red) {
    for (int o = 16; o > 0; o >>= 1) {
        a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
        b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, o));
    }
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5] = a;
        red[8 + (threadIdx.x >> 5)] = b;
    }
    __syncthreads();
    for (int i = 0; i < LT / 32; ++i) {
        a = fmaxf(a, red[i]);
        b = fmaxf(b, red[8 + i]);
    }
    __syncthreads();
    return make_float2(a, b);
}

// Largest magnitudes of a network's W1 and W2, 16 loads in flight.
__device__ __noinline__ float2 net_max(const float* W, int in, int H, float* red) {
    auto largest = [](const float* p, int n) {
        float m = 0.0f;
        for (int i = threadIdx.x; i < n; i += 16 * LT) {
            float v[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = i + e * LT < n ? ldcg(p + i + e * LT) : 0.0f;
#pragma unroll
            for (int e = 0; e < 16; ++e) m = fmaxf(m, fabsf(v[e]));
        }
        return m;
    };
    const float a = largest(W, H * in), b = largest(W + H * in + H, H * H);
    return block_max2(a, b, red);
}

// Largest magnitudes of W1 and W2 of a network whose image a pass is about to read.  An image
// whose halves have left their range since it was made (Adam and Polyak keep its exponents)
// is made again, by its owner; every CTA of the cluster calls and finds the same.
template <int H>
__device__ __noinline__ float2 net_check(tce::NetScale& ns, unsigned char* img, const float* W, int in, bool owner, int nS,
                                         float* red) {
    using namespace tce;
    const NetScale e = ns;
    const float2 m = block_max2(max_half<H * KP>(img), max_half<H * H>(img + 4 * H * KP), red);
    if (m.x >= kScaleLow && m.x < kScaleTop && m.y >= kScaleLow && m.y < kScaleTop)
        return make_float2(m.x * exp2i(-e.e1), m.y * exp2i(-e.e2));
    const float2 w = net_max(W, in, H, red);
    const NetScale f{scale_max(W_TOP, w.x), scale_max(W_TOP, w.y)};
    if (f.e1 != e.e1 || f.e2 != e.e2) {
        if (threadIdx.x == 0) ns = f;
        cluster_sync_all(nS);  // every CTA has read the image
        if (owner) img_make(img, W, in, H, f);
        cluster_sync_all(nS);
    }
    return w;
}

// One TD3 update with its network passes on the tensor cores (tce::pass): a CTA holds whole
// 128-sample tiles, at most 96 inputs.  Same phases, random streams and cluster reduction as
// td3_update.  The critics' regression runs there at hidden 128 only; at 32 and 64 it keeps the
// shared-memory engine's FP32 sums in their order, and the target passes the order of their
// MMAs, so that a critic's weights are bit for bit what they were until the actor's first step
// (whose gradient is rounded differently, and whose target every later regression sees).  A
// unit that passes the ReLU on one side of a rounding and not on the other moves a weight by a
// sample's whole share, and over 16 updates of 128 runs one such unit in the regression was
// enough to be a thousandth of the weights' size.  At hidden 128 a unit's share is smaller,
// exact_unit1/2 settle the doubtful ones, and the regression was a third of the whole step.
// The actor's passes settle none: they are as close to 64 bits as FP32 (qsim_tcmlp.cuh), so
// that no more of their units fall on the other side than in FP32.
// 512 mixed runs x 4 steps 12.6 ms on the FP32 engines, 9.4 here; 128 privileged runs x 16
// updates 9.4 and 7.9.
// False (on every CTA of the cluster) when a wait for the tensor cores ran out on one of them:
// the networks whose gradients were not complete by then are left as they were.
template <int H>
__device__ __noinline__ bool td3_update_tc(RunDesc& R, int64_t head, int64_t size, int64_t t_now, uint32_t u,
                                           int64_t& t_a, int64_t& t_c, const Scr& S, float* scr_base,
                                           size_t scr_stride, int rk, int nS, float* sm, uint32_t tmem, TcState& tcs) {
    using namespace tce;
    const int B = R.B, Bc = B / nS, PA = R.PA, PC = R.PC, DA = R.DA, DC = R.DC;
    const LearnHyper& hp = R.hp;
    const int j0 = rk * Bc;
    int* const st = R.E.status;
    float* red = sm + SMEM_MAIN;
    const float invB = 1.0f / (float)B;
    const bool pol = (int64_t)(u % (uint32_t)hp.policy_delay) == (int64_t)(hp.policy_delay - 1);
    constexpr bool plain = plain_targets(H);
    gather_all<true>(R, j0, Bc, u, head, size, t_now, S, sm, pol, tcs.xe, plain);
    // target actor + smoothing; the target action goes into o_c' tiles' last columns
    const float* cl0 = scr_base - (size_t)rk * scr_stride;  // scratch of cluster rank 0
    auto img = [&](Net n) { return net_img(S, scr_base, scr_stride, rk, nS, H, n); };
    Args f{};
    f.Bc = Bc;
    f.limit = R.C.wait_limit;
    f.dead = &tcs.dead;
    // (a pass ends with a barrier of the CTA, so that all of its threads see the flag alike)
    auto alive = [&] { return *reinterpret_cast<volatile int*>(&tcs.dead) == 0; };
    // Before a cluster barrier each CTA posts its flag; after it, whether all are alive.
    auto post = [&](int k) {
        if (nS > 1 && threadIdx.x == 0) S.loss[k] = alive() ? 0.0f : 1.0f;
    };
    auto all_alive = [&](int k) {
        if (nS == 1) return alive();
        const float* p = cl0 + (size_t)(threadIdx.x < (unsigned)nS ? threadIdx.x : 0) * scr_stride + (S.loss - scr_base);
        return __syncthreads_or(ldcg(p + k) != 0.0f) == 0;
    };
    f.x32 = S.x32;
    f.xn = S.xn;
    f.invB = invB;
    // network n with weights W, for a pass with scaled operands
    auto use = [&](Net n, float* W, int in) {
        f.W = W; f.img = img(n); f.in = in;
        const float2 m = net_check<H>(tcs.net[n], img(n), W, in, n % nS == rk, nS, red);
        f.w1m = m.x; f.w2m = m.y; f.e = tcs.net[n];
    };
    // a target network
    auto target = [&](Net n, float* W, int in) {
        if constexpr (plain) {
            f.W = W; f.img = img(n); f.in = in;
            if (alive()) pass<H, FWD>(f, sm, tmem, st);
        } else {
            use(n, W, in);
            if (alive()) pass<H, FWDX>(f, sm, tmem, st);
        }
    };
    f.xe = tcs.xe + gat::XE;
    f.out = 4; f.X = S.oa2; f.Y = S.mu; f.tanh_out = true;
    target(N_ACTOR_T, R.actor_t, DA);
    for (int jl = threadIdx.x; jl < Bc; jl += LT) {
        const uint32_t j = (uint32_t)(j0 + jl);
        const uint4 r0 = draw(R.C, j, u, TAG_SMOOTH, 0), r1 = draw(R.C, j, u, TAG_SMOOTH, 1);
        const float z[4] = {gauss(r0.x, r0.y), gauss(r0.z, r0.w), gauss(r1.x, r1.y), gauss(r1.z, r1.w)};
        float a2[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float eps = clampf(hp.sigma_t * z[i], -hp.noise_clip, hp.noise_clip);
            a2[i] = clampf(ldcg(S.mu + jl * 4 + i) + eps, -1.0f, 1.0f);
        }
        unsigned char* t = reinterpret_cast<unsigned char*>(S.oc2 + (size_t)(jl / TR) * TILE_FLOATS);
        const float sx = exp2i(tcs.xe[gat::XE + jl / gat::GS]);
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
            uint32_t h, l;
            tc::split2(sx * a2[i], sx * a2[i + 1], h, l);
            const int at = 2 * tc::cano16(jl % TR, DC - 4 + i, KC1);
            *reinterpret_cast<uint32_t*>(t + at) = h;
            *reinterpret_cast<uint32_t*>(t + 2 * TILE_HALVES + at) = l;
        }
    }
    __syncthreads();
    // twin target critics, clipped double-Q target
    f.out = 1; f.X = S.oc2; f.tanh_out = false;
    f.Y = S.q1;
    target(N_C1_T, R.c1_t, DC);
    f.Y = S.q2;
    target(N_C2_T, R.c2_t, DC);
    for (int jl = threadIdx.x; jl < Bc; jl += LT) {
        const float qmin = fminf(ldcg(S.q1 + jl), ldcg(S.q2 + jl));
        S.y[jl] = S.r[jl] + (S.term[jl] != 0.0f ? 0.0f : hp.gamma * qmin);
    }
    __syncthreads();
    // critic regression
    float lsum = 0.0f;
    if constexpr (H == 128) {
        f.X = S.oc; f.y = S.y; f.xe = tcs.xe;
        use(N_C1, R.c1, DC);
        f.G = S.g1;
        if (alive()) lsum = pass<H, CRIT>(f, sm, tmem, st);
        use(N_C2, R.c2, DC);
        f.G = S.g2;
        if (alive()) lsum += pass<H, CRIT>(f, sm, tmem, st);
    } else if (DC == 90) {
        lsum = critics_smem<H, 90>(R, S, Bc, DC, sm);
    } else if (H == 64 && DC == 96) {
        lsum = critics_smem<H, H == 64 ? 96 : 0>(R, S, Bc, DC, sm);
    } else {
        lsum = critics_smem<H, 0>(R, S, Bc, DC, sm);
    }
    lsum = block_sum(lsum, red);
    if (threadIdx.x == 0) S.loss[0] = lsum;
    post(2);
    cluster_sync_all(nS);
    if (!all_alive(2)) return false;
    t_c += 1;
    {
        const int lo = (int)((int64_t)PC * rk / nS), hi = (int)((int64_t)PC * (rk + 1) / nS);
        // on steps that update the actor, the critics' targets take their Polyak step here
        // (at hidden <= 64 only those steps read critic 1's halves, and none critic 2's)
        adam_slice(R.c1, cl0, scr_stride, nS, (int)(S.g1 - scr_base), R.m_c1, R.v_c1, lo, hi, t_c, hp, 1.0f,
                   pol ? R.c1_t : nullptr, H == 128 || pol ? Img(img(N_C1), DC, H, tcs.net[N_C1]) : Img(),
                   Img(img(N_C1_T), DC, H, tcs.net[N_C1_T]));
        adam_slice(R.c2, cl0, scr_stride, nS, (int)(S.g2 - scr_base), R.m_c2, R.v_c2, lo, hi, t_c, hp, 1.0f,
                   pol ? R.c2_t : nullptr, H == 128 ? Img(img(N_C2), DC, H, tcs.net[N_C2]) : Img(),
                   Img(img(N_C2_T), DC, H, tcs.net[N_C2_T]));
        if (rk == 0 && threadIdx.x == 0) {
            float l = 0.0f;
            for (int s2 = 0; s2 < nS; ++s2) l += ldcg(cl0 + (size_t)s2 * scr_stride + (S.loss - scr_base));
            R.stats[0] = l;
        }
    }
    cluster_sync_all(nS);
    if (!pol) return true;
    // delayed actor update through the updated first critic
    f.xe = tcs.xe;
    f.out = 4; f.X = S.oa; f.Y = S.mu; f.tanh_out = true;
    use(N_ACTOR, R.actor, DA);
    const Args fa = f;
    pass<H, FWDX>(f, sm, tmem, st);
    f.out = 1; f.X = S.oc; f.mu = S.mu; f.da = S.da;
    use(N_C1, R.c1, DC);
    float qs = alive() ? pass<H, DQ>(f, sm, tmem, st) : 0.0f;
    f.W = fa.W; f.img = fa.img; f.in = DA; f.e = fa.e; f.w1m = fa.w1m; f.w2m = fa.w2m;
    f.out = 4; f.X = S.oa; f.G = S.ga;
    if (alive()) pass<H, ACT>(f, sm, tmem, st);
    qs = block_sum(qs, red);
    if (threadIdx.x == 0) S.loss[1] = qs;
    post(3);
    cluster_sync_all(nS);
    if (!all_alive(3)) return false;
    t_a += 1;
    {
        const int lo = (int)((int64_t)PA * rk / nS), hi = (int)((int64_t)PA * (rk + 1) / nS);
        adam_slice(R.actor, cl0, scr_stride, nS, (int)(S.ga - scr_base), R.m_a, R.v_a, lo, hi, t_a, hp, 1.0f, R.actor_t,
                   Img(img(N_ACTOR), DA, H, tcs.net[N_ACTOR]), Img(img(N_ACTOR_T), DA, H, tcs.net[N_ACTOR_T]));
        if (rk == 0 && threadIdx.x == 0) {
            float l = 0.0f;
            for (int s2 = 0; s2 < nS; ++s2) l += ldcg(cl0 + (size_t)s2 * scr_stride + (S.loss - scr_base) + 1);
            R.stats[1] = l;
        }
    }
    cluster_sync_all(nS);
    return true;
}

// Curriculum change + reward recalculation over the run's buffer, split over the cluster.
__device__ __noinline__ void curriculum_step(RunDesc& R, int64_t head, int64_t size, int rk, int nS) {
    if (rk == 0 && threadIdx.x == 0) {
        for (int i = 0; i < 7; ++i) {
            const float c = R.E.rewardC[i], x = c * R.cf[i];
            R.E.rewardC[i] = R.cf[i] >= 1.0f ? fminf(x, R.ct[i]) : fmaxf(x, R.ct[i]);
        }
        R.E.rewardC[7] = fmaxf(R.E.rewardC[7] * R.sig_f, R.sig_min);
    }
    cluster_sync_all(nS);
    if (!R.recalc || R.capacity == 0) return;
    float Cr[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) Cr[i] = ldcg(R.E.rewardC + i);
    recalc_range(R.C, R.E, Cr, head, size, R.capacity, (uint64_t)rk * LT + threadIdx.x, (uint64_t)nS * LT);
    cluster_sync_all(nS);
}

// Persistent training kernel.  Cluster c walks runs order[off[c] .. off[c+1]).
__global__ void __launch_bounds__(LT) k_train(RunDesc* runs, const int* order, const int* off,
                                              int n_iters, int do_env, float* scratch,
                                              size_t scr_stride, int nS, int use_tc) {
    extern __shared__ __align__(16) float sm[];
    // tensor memory for the tensor-core passes, when some run of the launch has them
    __shared__ uint32_t tmem_slot;
    __shared__ TcState tcs;
    if (use_tc) {
        if ((threadIdx.x >> 5) == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                         :: "r"(tc::smem_u32(&tmem_slot)), "r"(tce::TMEM_COLS) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
    }
    const uint32_t tmem = use_tc ? tmem_slot : 0u;
    const int rk = nS > 1 ? (int)cg::this_cluster().block_rank() : 0;
    const int cl = blockIdx.x / nS;
    float* my = scratch + (size_t)blockIdx.x * scr_stride;
    for (int oi = off[cl]; oi < off[cl + 1]; ++oi) {
        RunDesc& R = runs[order[oi]];
        int64_t head = R.head, size = R.size, t_now = R.t_now, t_a = R.t_a, t_c = R.t_c, u = R.u;
        int64_t next_curr = R.next_curr;
        const int Bc = R.B / nS;
        const bool tiles = use_tc && tce::shape_ok(Bc, R.H, R.DA, R.DC);  // tensor-core passes
        const Scr S = carve(my, Bc, R.H, R.DA, R.DC, R.PA, R.PC, R.n_env, nS, tiles);
        bool updating = true;  // until a wait runs out: the launch's other updates of the run are then left out
        if (tiles) {
            if (threadIdx.x == 0) tcs.dead = 0;
            // the networks' halves for the tensor-core passes, shared out over the cluster; their
            // exponents, by every CTA for itself (critic 2's are read at hidden 128 only)
            const float* nets[6] = {R.actor, R.actor_t, R.c1, R.c1_t, R.c2, R.c2_t};
            const bool plain = plain_targets(R.H);
            for (int n = 0; n < 6; ++n) {
                tce::NetScale e{0, 0};
                if (n & 1 ? !plain : n != N_C2 || R.H == 128) {
                    const float2 m = net_max(nets[n], n < 2 ? R.DA : R.DC, R.H, sm + SMEM_MAIN);
                    e = tce::NetScale{tce::scale_max(tce::W_TOP, m.x), tce::scale_max(tce::W_TOP, m.y)};
                }
                if (threadIdx.x == 0) tcs.net[n] = e;
                if (n % nS == rk) tce::img_make(net_img(S, my, scr_stride, rk, nS, R.H, n), nets[n], n < 2 ? R.DA : R.DC, R.H, e);
            }
            cluster_sync_all(nS);
        }
        for (int it = 0; it < n_iters; ++it) {
            int n_upd = 1;
            if (do_env) {
                if (rk == 0) {
                    if (R.n_env <= 8 && R.H <= 128 && R.DA <= 128)
                        env_step_small(R, (uint32_t)t_now, head, sm);
                    else
                        env_step_cta(R, S, (uint32_t)t_now, head, sm);
                }
                t_now += 1;
                if (R.capacity > 0) {
                    head = head + 1 == R.capacity ? 0 : head + 1;
                    if (size < R.capacity) size += 1;
                }
                cluster_sync_all(nS);
                if (R.curr_interval > 0 && t_now * (int64_t)R.n_env >= next_curr) {
                    curriculum_step(R, head, size, rk, nS);
                    next_curr += R.curr_interval;
                }
                n_upd = t_now >= R.start_updates ? R.hp.updates_per_step : 0;
            }
            const bool resident = R.H <= smlp::HP && R.DC <= smlp::INP && R.DA <= smlp::INP;
            const bool resident128 = R.H == 128 && R.DA == 82 && R.DC == 90;
            for (int k = 0; k < n_upd; ++k) {
                if (tiles) {
                    // (the counters advance as the host expects, whatever became of the update)
                    const int64_t a1 = t_a + ((uint32_t)u % (uint32_t)R.hp.policy_delay == (uint32_t)(R.hp.policy_delay - 1));
                    const int64_t c1 = t_c + 1;
                    if (updating)
                        updating = R.H == 64   ? td3_update_tc<64>(R, head, size, t_now, (uint32_t)u, t_a, t_c, S, my,
                                                                   scr_stride, rk, nS, sm, tmem, tcs)
                                   : R.H == 32 ? td3_update_tc<32>(R, head, size, t_now, (uint32_t)u, t_a, t_c, S, my,
                                                                   scr_stride, rk, nS, sm, tmem, tcs)
                                               : td3_update_tc<128>(R, head, size, t_now, (uint32_t)u, t_a, t_c, S, my,
                                                                    scr_stride, rk, nS, sm, tmem, tcs);
                    t_a = a1;
                    t_c = c1;
                } else if (resident) {
                    // specialised shapes: hidden 64 or 32 over 16 actions of history, and the
                    // privileged critic (82 + 4 + 6 motor/parameter inputs + 4 actions)
                    const int key = R.H * 1000000 + R.DA * 1000 + R.DC;
                    if (key == 64082090)
                        td3_update_smem<64, 82, 90>(R, head, size, t_now, (uint32_t)u, t_a, t_c, S,
                                                    my, scr_stride, rk, nS, sm);
                    else if (key == 32082090)
                        td3_update_smem<32, 82, 90>(R, head, size, t_now, (uint32_t)u, t_a, t_c, S,
                                                    my, scr_stride, rk, nS, sm);
                    else if (key == 64082096)
                        td3_update_smem<64, 82, 96>(R, head, size, t_now, (uint32_t)u, t_a, t_c, S,
                                                    my, scr_stride, rk, nS, sm);
                    else
                        td3_update_smem<0, 0, 0>(R, head, size, t_now, (uint32_t)u, t_a, t_c, S,
                                                 my, scr_stride, rk, nS, sm);
                } else if (resident128) {
                    // hidden 128 with 16 actions of history: the 128-wide engine shape
                    td3_update_smem<128, 82, 90>(R, head, size, t_now, (uint32_t)u, t_a, t_c, S, my,
                                                 scr_stride, rk, nS, sm);
                } else
                    td3_update(R, head, size, t_now, (uint32_t)u, t_a, t_c, S, my, scr_stride,
                               blockIdx.x - rk, rk, nS, sm);
                u += 1;
            }
        }
        cluster_sync_all(nS);
        if (rk == 0 && threadIdx.x == 0) {
            R.head = head; R.size = size; R.t_now = t_now; R.t_a = t_a; R.t_c = t_c; R.u = u;
            R.next_curr = next_curr;
        }
        cluster_sync_all(nS);
    }
    if (use_tc) {
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        if ((threadIdx.x >> 5) == 0)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(tce::TMEM_COLS) : "memory");
    }
}

// ------------------------------------------------------------------- initialisation
__global__ void k_init_params(float* P, int in, int h, int out, uint32_t net_id, uint32_t k0,
                              uint32_t k1, uint32_t run) {
    const int total = psize(in, h, out);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int sizes[6] = {h * in, h, h * h, h, out * h, out};
    const int fan[6] = {in, in, h, h, h, h};
    int blk = 0, acc = 0;
    while (blk < 5 && i >= acc + sizes[blk]) { acc += sizes[blk]; ++blk; }
    const float bound = 1.0f / sqrtf((float)fan[blk]);
    const uint4 r = philox((uint32_t)i >> 2, net_id, (TAG_INIT << 24), run, k0, k1);
    const uint32_t x = (i & 3) == 0 ? r.x : ((i & 3) == 1 ? r.y : ((i & 3) == 2 ? r.z : r.w));
    P[i] = bound * (2.0f * u01(x) - 1.0f);
}

static int grid_for(int64_t n, int b) { return (int)((n + b - 1) / b); }

static size_t learner_smem() { return sizeof(float) * (size_t)(SMEM_MAIN + 32); }


}  // namespace qsim

using namespace qsim;

// ---------------------------------------------------------------------------- ABI
static qsim_status fill_desc(ac_handle* a, qsim_handle* e, RunDesc& R) {
    memset(&R, 0, sizeof(R));
    if (!a || !e) return fail(QSIM_EINVAL, "null handle");
    R.C = e->dc;
    R.E = e->p;
    R.capacity = e->capacity; R.head = e->head; R.size = e->size; R.t_now = e->t_now;
    R.curr_interval = e->cfg.curriculum_interval;
    R.next_curr = e->next_curriculum;
    for (int i = 0; i < 7; ++i) { R.cf[i] = e->cfg.curriculum_factor[i]; R.ct[i] = e->cfg.curriculum_target[i]; }
    R.sig_f = e->cfg.sigma_factor; R.sig_min = e->cfg.sigma_min; R.recalc = e->cfg.recalc_rewards;
    R.n_env = e->n;
    R.actor = a->actor; R.actor_t = a->actor_t; R.c1 = a->c1; R.c1_t = a->c1_t; R.c2 = a->c2; R.c2_t = a->c2_t;
    R.m_a = a->m_a; R.v_a = a->v_a; R.m_c1 = a->m_c1; R.v_c1 = a->v_c1; R.m_c2 = a->m_c2; R.v_c2 = a->v_c2;
    R.stats = a->stats;
    R.H = a->hidden; R.B = a->batch; R.DA = a->obs_dim; R.DC = a->critic_in;
    R.PA = a->n_actor; R.PC = a->n_critic;
    R.t_a = a->t_actor; R.t_c = a->t_critic; R.u = a->updates;
    const int64_t lost = e->cfg.n_hist;
    R.start_updates = std::max<int64_t>((int64_t)e->cfg.learning_starts, 2 + lost);
    const ac_config& c = a->cfg;
    R.hp = LearnHyper{c.gamma, c.tau, c.lr, c.beta1, c.beta2, c.eps, c.sigma_target, c.noise_clip,
                      c.policy_delay, c.updates_per_step};
    R.idx_log = a->idx_log;
    return QSIM_OK;
}

static void read_back(ac_handle* a, qsim_handle* e, const RunDesc& R) {
    e->head = R.head; e->size = R.size; e->t_now = R.t_now; e->next_curriculum = R.next_curr;
    a->t_actor = R.t_a; a->t_critic = R.t_c; a->updates = R.u;
}

// Advances the counters of a run descriptor exactly as k_train does over n_iters
// iterations, so that the host knows them without reading the descriptor back.
static void advance_desc(RunDesc& R, int64_t n_iters, int do_env) {
    for (int64_t it = 0; it < n_iters; ++it) {
        int n_upd = 1;
        if (do_env) {
            R.t_now += 1;
            if (R.capacity > 0) {
                R.head = R.head + 1 == R.capacity ? 0 : R.head + 1;
                if (R.size < R.capacity) R.size += 1;
            }
            if (R.curr_interval > 0 && R.t_now * (int64_t)R.n_env >= R.next_curr) R.next_curr += R.curr_interval;
            n_upd = R.t_now >= R.start_updates ? R.hp.updates_per_step : 0;
        }
        for (int k = 0; k < n_upd; ++k) {
            R.t_c += 1;
            if ((int64_t)((uint32_t)R.u % (uint32_t)R.hp.policy_delay) == (int64_t)(R.hp.policy_delay - 1))
                R.t_a += 1;
            R.u += 1;
        }
    }
}

static int pick_cluster(const ac_handle* a, int n_runs) {
    if (a->cfg.cluster > 0) return a->cfg.cluster;
    if (n_runs >= 64) return 1;
    // a few runs: the widest cluster (16 CTAs, non-portable) that leaves each CTA >= 16
    // samples; at batch 256 that is 111.5 us per env step + update against 135.9 at 8 CTAs
    const int b = a->batch;
    int s = n_runs > 8 ? 2 : 16;
    while (s > 1 && (b % s || b / s < 16)) s >>= 1;
    return s;
}

static qsim_status validate_pair(const ac_handle* a, const qsim_handle* e) {
    if (!a || !e) return fail(QSIM_EINVAL, "null handle");
    int dev = -1;
    QCHECK_CUDA(cudaGetDevice(&dev));
    if (dev != a->device || dev != e->device)
        return fail(QSIM_EINVAL, "the current device (%d) is not the one the learner (%d) and env set (%d) "
                    "were created on", dev, a->device, e->device);
    if (e->capacity < 2) return fail(QSIM_ESTATE, "env set has no replay buffer");
    if (e->capacity < e->cfg.n_hist + 2)
        return fail(QSIM_EINVAL, "replay capacity %lld must exceed the history length + 1",
                    (long long)e->capacity);
    if (a->obs_dim != e->dc.obs_dim || a->critic_in != e->dc.cobs_dim + 4)
        return fail(QSIM_EINVAL, "learner and env set have different observation layouts");
    return QSIM_OK;
}

// Launch geometry of one run by itself: cluster size and per-CTA scratch (floats).
struct SingleRun {
    int nS = 1;
    size_t stride = 0;
};

// Checks shared by every single-run launch (ac_update, ac_update_static and the plain
// forms of ac_train).  do_env = 0: n_iters updates from the buffer as it is, which must
// already allow sampling.
static qsim_status prepare_single(const ac_handle* a, const qsim_handle* env, int do_env,
                                  int64_t n_iters, const char* who, SingleRun* out) {
    qsim_status s = validate_pair(a, env);
    if (s != QSIM_OK) return s;
    if (n_iters < 0) return fail(QSIM_EINVAL, "%s: negative count", who);
    if ((uint64_t)env->capacity * (uint64_t)env->n >= (1ull << 32))
        return fail(QSIM_EINVAL, "%s: replay buffer exceeds 2^32 transitions", who);
    if (do_env) {
        if (((env->t_now + n_iters) >> 32) != 0) return fail(QSIM_ESTATE, "%s: step counter exhausted", who);
    } else {
        const int64_t lost = env->size == env->capacity ? env->cfg.n_hist : 0;
        if (env->size - 1 - lost < 1)
            return fail(QSIM_ESTATE, "%s: replay buffer too small to sample (size=%lld)", who,
                        (long long)env->size);
        if (((a->updates + n_iters) >> 32) != 0) return fail(QSIM_ESTATE, "%s: update counter exhausted", who);
    }
    out->nS = pick_cluster(a, 1);
    if (a->batch % out->nS)
        return fail(QSIM_EINVAL, "%s: batch %d not divisible by cluster %d", who, a->batch, out->nS);
    out->stride = scratch_floats(a->batch / out->nS, a->hidden, a->obs_dim, a->critic_in, a->n_actor,
                                 a->n_critic, env->n, out->nS);
    return QSIM_OK;
}

// Device image of one run's launch: the descriptor and a one-run schedule.
struct PackedRun {
    RunDesc run;
    int order[1];
    int off[2];
};
static_assert(sizeof(PackedRun) <= QSIM_STATIC_DESC_BYTES, "run descriptor exceeds its static area");
constexpr size_t kPackedBytes = (sizeof(PackedRun) + 255) & ~(size_t)255;

// Whether the run's updates go to the tensor cores (a launch then allocates tensor memory).
static bool tc_wanted(const RunDesc& R, int nS) { return tce::shape_ok(R.B / nS, R.H, R.DA, R.DC); }

static qsim_status launch_k_train(int grid, int nS, cudaStream_t st, RunDesc* d_runs, const int* d_order,
                                  const int* d_off, int64_t n_iters, int do_env, float* scratch,
                                  size_t stride, int use_tc) {
    if (n_iters > INT32_MAX) return fail(QSIM_EINVAL, "too many steps for one launch");
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(grid);
    lc.blockDim = dim3(LT);
    lc.dynamicSmemBytes = learner_smem();
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = nS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    if (nS > 8) QCHECK_CUDA(cudaFuncSetAttribute(k_train, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    QCHECK_CUDA(cudaLaunchKernelEx(&lc, k_train, d_runs, d_order, d_off, (int)n_iters, do_env, scratch,
                                   stride, nS, use_tc));
    return QSIM_OK;
}

// Host to device copy of pageable `src`, which may go when this returns.  Outside stream capture
// the copy is staged by then; a captured copy reads its source at every replay, so that the
// bytes then belong to the graph.
static cudaError_t upload_pageable(void* dst, const void* src, size_t bytes, cudaStream_t st) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamGetCaptureInfo(st, &status, nullptr, &graph);
    if (e != cudaSuccess) return e;
    if (status == cudaStreamCaptureStatusActive) {
        void* own = malloc(bytes);
        if (!own) return cudaErrorMemoryAllocation;
        memcpy(own, src, bytes);
        cudaUserObject_t obj;
        e = cudaUserObjectCreate(&obj, own, free, 1, cudaUserObjectNoDestructorSync);
        if (e != cudaSuccess) {
            free(own);
            return e;
        }
        e = cudaGraphRetainUserObject(graph, obj, 1, cudaGraphUserObjectMove);
        if (e != cudaSuccess) {
            cudaUserObjectRelease(obj, 1);
            return e;
        }
        src = own;
    }
    return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
}

// One run, one launch of n_iters iterations.  desc_dev holds a PackedRun; when `mirror`
// is given it is the host copy of what desc_dev holds once the stream's earlier work has
// run, and the descriptor is uploaded only if the handles' state differs from it.
static qsim_status run_single(ac_handle* a, qsim_handle* env, int64_t n_iters, int do_env,
                              const SingleRun& L, unsigned char* desc_dev, float* scratch,
                              RunDesc* mirror, cudaStream_t st) {
    PackedRun pk;
    memset(&pk, 0, sizeof(pk));
    qsim_status s = fill_desc(a, env, pk.run);
    if (s != QSIM_OK) return s;
    pk.off[1] = 1;
    PackedRun* d_pk = reinterpret_cast<PackedRun*>(desc_dev);
    if (!mirror || memcmp(&pk.run, mirror, sizeof(RunDesc)) != 0) {
        QCHECK_CUDA(upload_pageable(d_pk, &pk, sizeof(pk), st));
    }
    s = launch_k_train(L.nS, L.nS, st, &d_pk->run, d_pk->order, d_pk->off, n_iters, do_env, scratch, L.stride,
                       tc_wanted(pk.run, L.nS) ? 1 : 0);
    if (s != QSIM_OK) {
        if (mirror) memset(mirror, 0xff, sizeof(RunDesc));  // unknown device state: upload next time
        return s;
    }
    advance_desc(pk.run, n_iters, do_env);
    read_back(a, env, pk.run);
    if (mirror) *mirror = pk.run;
    return QSIM_OK;
}

// The learner's own workspace for single-run launches: [PackedRun | scratch of the
// cluster], kept between calls, grown when a launch needs more.
struct LearnerCache {
    unsigned char* dev = nullptr;
    size_t bytes = 0;
    RunDesc mirror;
    LearnerCache() { memset(&mirror, 0xff, sizeof(mirror)); }
};

static qsim_status learner_run(ac_handle* a, qsim_handle* env, int64_t n_iters, int do_env,
                               const SingleRun& L, cudaStream_t st) {
    LearnerCache* c = static_cast<LearnerCache*>(a->cache);
    const size_t need = kPackedBytes + sizeof(float) * L.stride * (size_t)L.nS;
    if (c->bytes < need) {
        if (c->dev) {
            QCHECK_CUDA(cudaStreamSynchronize(st));
            cudaFree(c->dev);
            c->dev = nullptr;
            c->bytes = 0;
        }
        if (cudaMalloc((void**)&c->dev, need) != cudaSuccess) {
            cudaGetLastError();
            return fail(QSIM_ENOMEM, "learner workspace of %zu bytes", need);
        }
        c->bytes = need;
        memset(&c->mirror, 0xff, sizeof(RunDesc));
    }
    return run_single(a, env, n_iters, do_env, L, c->dev, reinterpret_cast<float*>(c->dev + kPackedBytes),
                      &c->mirror, st);
}

// All runs in one persistent launch (clusters walk a longest-processing-time-first list).
// Estimated time of one training iteration of a run (microseconds; a fit to the persistent
// kernel's measured step times at one CTA per run and 8 envs, hidden 32-128, batch
// 128-512): the env step plus updates_per_step x (a part fixed per update: Adam over the
// parameters, barriers, weight staging; and a part per sample on a CTA: gather, the
// networks' passes).  Only its ratios matter: it balances the longest-processing-time-first
// assignment of runs to clusters, where a pure FLOP count left the small runs' fixed costs
// out and piled them onto the same clusters.  The tensor-core passes have their own fit
// (256 samples, hidden 32 / 64 / 128: 45 / 81 / 190 us fixed and 90 / 113 / 175 us a tile).
static double run_cost(const ac_handle* a, const qsim_handle* e, int nS) {
    const double h = a->hidden, b = (double)a->batch / std::max(1, nS);
    // the small-run env step (<= 8 envs, one env per lane group) or the CTA-wide one
    const double env = e->n <= 8 && a->hidden <= 128 ? 13.0 + 0.1 * h : 16.0 + 0.34 * h;
    double upd;
    if (tce::shape_ok(a->batch / std::max(1, nS), a->hidden, a->obs_dim, a->critic_in)) {
        upd = 20.0 + 0.6 * h + 0.0057 * h * h + b / tce::TR * (66.0 + 0.68 * h + 0.0013 * h * h);
    } else {
        const double per_sample = 1.042 + 3.98e-5 * (h * (a->obs_dim + a->critic_in) + 3.0 * h * h);
        upd = 32.3 + 0.71 * h + 0.0109 * h * h + b * per_sample;
    }
    return env + std::max(1, (int)a->cfg.updates_per_step) * upd;
}

static qsim_status launch_train(std::vector<ac_handle*>& A, std::vector<qsim_handle*>& E,
                                int64_t n_iters, int do_env, int nS, cudaStream_t st,
                                int n_clusters_in) {
    const int n = (int)A.size();
    std::vector<RunDesc> D(n);
    size_t stride = 0;
    for (int i = 0; i < n; ++i) {
        qsim_status s = fill_desc(A[i], E[i], D[i]);
        if (s != QSIM_OK) return s;
        if (A[i]->batch % nS) return fail(QSIM_EINVAL, "batch %d not divisible by cluster %d", A[i]->batch, nS);
        stride = std::max(stride, scratch_floats(A[i]->batch / nS, A[i]->hidden, A[i]->obs_dim,
                                                 A[i]->critic_in, A[i]->n_actor, A[i]->n_critic, E[i]->n, nS));
    }
    const int n_clusters = std::max(1, std::min(n, n_clusters_in));
    std::vector<int> order(n), off(n_clusters + 1, 0);
    {
        std::vector<double> cost(n);
        for (int i = 0; i < n; ++i) cost[i] = run_cost(A[i], E[i], nS);
        std::vector<int> idx(n);
        std::iota(idx.begin(), idx.end(), 0);
        std::stable_sort(idx.begin(), idx.end(), [&](int x, int y) { return cost[x] > cost[y]; });
        std::vector<double> load(n_clusters, 0.0);
        std::vector<std::vector<int>> lists(n_clusters);
        for (int i : idx) {
            int best = 0;
            for (int c = 1; c < n_clusters; ++c)
                if (load[c] < load[best]) best = c;
            load[best] += cost[i];
            lists[best].push_back(i);
        }
        int k = 0;
        for (int c = 0; c < n_clusters; ++c) {
            off[c] = k;
            for (int i : lists[c]) order[k++] = i;
        }
        off[n_clusters] = k;
    }
    // device copies and scratch: one stream-ordered allocation, freed in stream order after
    // the launch
    auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t o_order = up(sizeof(RunDesc) * n), o_off = o_order + up(sizeof(int) * n),
                 o_scr = o_off + up(sizeof(int) * (n_clusters + 1));
    unsigned char* dev;
    QCHECK_CUDA(cudaMallocAsync((void**)&dev, o_scr + sizeof(float) * stride * (size_t)n_clusters * nS, st));
    // (not under capture: the staging is reused, and a replay reads the copy's source again)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(st, &cap);
    std::vector<unsigned char> pageable;
    Staging* const staging = cap == cudaStreamCaptureStatusNone ? staging_slot() : nullptr;
    unsigned char* host = staging ? (unsigned char*)staging->take(o_scr) : nullptr;
    const bool pinned = host != nullptr;
    if (!pinned) {
        pageable.resize(o_scr);
        host = pageable.data();
    }
    memcpy(host, D.data(), sizeof(RunDesc) * n);
    memcpy(host + o_order, order.data(), sizeof(int) * n);
    memcpy(host + o_off, off.data(), sizeof(int) * (n_clusters + 1));
    const cudaError_t ce = pinned ? cudaMemcpyAsync(dev, host, o_scr, cudaMemcpyHostToDevice, st)
                                  : upload_pageable(dev, host, o_scr, st);
    if (pinned) staging->used(st);
    if (ce != cudaSuccess) {
        cudaFreeAsync(dev, st);
        return cuda_fail(ce, "ac_train: descriptors");
    }
    int use_tc = 0;
    for (int i = 0; i < n; ++i) use_tc |= tc_wanted(D[i], nS) ? 1 : 0;
    qsim_status s = launch_k_train(n_clusters * nS, nS, st, reinterpret_cast<RunDesc*>(dev),
                                   reinterpret_cast<int*>(dev + o_order), reinterpret_cast<int*>(dev + o_off), n_iters,
                                   do_env, reinterpret_cast<float*>(dev + o_scr), stride, use_tc);
    cudaFreeAsync(dev, st);
    if (s != QSIM_OK) return s;
    for (int i = 0; i < n; ++i) {
        advance_desc(D[i], n_iters, do_env);
        read_back(A[i], E[i], D[i]);
    }
    return QSIM_OK;
}

extern "C" qsim_status ac_create(const ac_config* cfg, const qsim_handle* env, ac_handle** out) {
    if (!cfg || !env || !out) return fail(QSIM_EINVAL, "ac_create: null pointer");
    *out = nullptr;
    if (cfg->hidden < 4 || cfg->hidden > 128 || (cfg->hidden % 4))
        return fail(QSIM_EINVAL, "ac_create: hidden=%d must be a multiple of 4 in [4,128]", cfg->hidden);
    if (cfg->batch < 1 || cfg->batch > 1024) return fail(QSIM_EINVAL, "ac_create: batch out of range");
    if (cfg->policy_delay < 1) return fail(QSIM_EINVAL, "ac_create: policy_delay < 1");
    if (cfg->cluster < 0 || cfg->cluster > 16 || (cfg->cluster & (cfg->cluster - 1)))
        return fail(QSIM_EINVAL, "ac_create: cluster must be 0 or a power of two <= 16");
    int dev = -1;
    QCHECK_CUDA(cudaGetDevice(&dev));
    if (dev != env->device)
        return fail(QSIM_EINVAL, "ac_create: the current device (%d) is not the env set's (%d)", dev, env->device);
    // the learner kernel needs more than the default 48 KB of dynamic shared memory (set on
    // the current device, where every launch for this learner happens)
    QCHECK_CUDA(cudaFuncSetAttribute(k_train, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)learner_smem()));
    ac_handle* a = new ac_handle();
    a->cfg = *cfg;
    if (a->cfg.updates_per_step < 1) a->cfg.updates_per_step = 1;
    a->device = dev;
    a->cache = new LearnerCache();
    a->idx_log = nullptr;
    a->obs_dim = env->dc.obs_dim;
    a->critic_in = env->dc.cobs_dim + 4;
    a->hidden = cfg->hidden;
    a->batch = cfg->batch;
    a->n_actor = a->hidden * a->obs_dim + a->hidden + a->hidden * a->hidden + a->hidden + 4 * a->hidden + 4;
    a->n_critic = a->hidden * a->critic_in + a->hidden + a->hidden * a->hidden + a->hidden + a->hidden + 1;
    a->t_actor = a->t_critic = a->updates = 0;
    const size_t PA = a->n_actor, PC = a->n_critic;
    const size_t total = 4 * PA + 8 * PC + 8;
    if (cudaMalloc((void**)&a->base, total * 4) != cudaSuccess ||
        cudaMalloc((void**)&a->status, 4) != cudaSuccess) {
        cudaGetLastError();
        ac_destroy(a);
        return fail(QSIM_ENOMEM, "ac_create: allocation failed");
    }
    cudaMemset(a->base, 0, total * 4);
    cudaMemset(a->status, 0, 4);
    float* p = a->base;
    a->actor = p; p += PA; a->actor_t = p; p += PA;
    a->c1 = p; p += PC; a->c1_t = p; p += PC; a->c2 = p; p += PC; a->c2_t = p; p += PC;
    a->m_a = p; p += PA; a->v_a = p; p += PA;
    a->m_c1 = p; p += PC; a->v_c1 = p; p += PC; a->m_c2 = p; p += PC; a->v_c2 = p; p += PC;
    a->stats = p;
    const uint32_t k0 = env->dc.key0, k1 = env->dc.key1, run = env->dc.run_id;
    k_init_params<<<grid_for(PA, 256), 256>>>(a->actor, a->obs_dim, a->hidden, 4, 0, k0, k1, run);
    k_init_params<<<grid_for(PC, 256), 256>>>(a->c1, a->critic_in, a->hidden, 1, 1, k0, k1, run);
    k_init_params<<<grid_for(PC, 256), 256>>>(a->c2, a->critic_in, a->hidden, 1, 2, k0, k1, run);
    cudaMemcpy(a->actor_t, a->actor, PA * 4, cudaMemcpyDeviceToDevice);
    cudaMemcpy(a->c1_t, a->c1, PC * 4, cudaMemcpyDeviceToDevice);
    cudaMemcpy(a->c2_t, a->c2, PC * 4, cudaMemcpyDeviceToDevice);
    cudaError_t err = cudaDeviceSynchronize();
    if (err != cudaSuccess) {
        ac_destroy(a);
        return cuda_fail(err, "ac_create: init");
    }
    *out = a;
    return QSIM_OK;
}

extern "C" qsim_status ac_destroy(ac_handle* a) {
    if (!a) return QSIM_OK;
    LearnerCache* c = static_cast<LearnerCache*>(a->cache);
    if (c) {
        if (c->dev) {
            cudaDeviceSynchronize();
            cudaFree(c->dev);
        }
        delete c;
    }
    if (a->base) cudaFree(a->base);
    if (a->status) cudaFree(a->status);
    delete a;
    return QSIM_OK;
}

extern "C" qsim_status ac_info_get(const ac_handle* a, ac_info* o) {
    if (!a || !o) return fail(QSIM_EINVAL, "ac_info_get: null pointer");
    o->obs_dim = a->obs_dim; o->critic_in = a->critic_in; o->hidden = a->hidden; o->batch = a->batch;
    o->n_actor = a->n_actor; o->n_critic = a->n_critic;
    o->t_actor = a->t_actor; o->t_critic = a->t_critic; o->updates = a->updates;
    o->actor = a->actor; o->actor_t = a->actor_t; o->c1 = a->c1; o->c1_t = a->c1_t;
    o->c2 = a->c2; o->c2_t = a->c2_t; o->m_a = a->m_a; o->v_a = a->v_a;
    o->m_c1 = a->m_c1; o->v_c1 = a->v_c1; o->m_c2 = a->m_c2; o->v_c2 = a->v_c2;
    o->stats = a->stats;
    return QSIM_OK;
}

extern "C" qsim_status ac_set_counters(ac_handle* a, int64_t t_actor, int64_t t_critic, int64_t updates) {
    if (!a || t_actor < 0 || t_critic < 0 || updates < 0 || (updates >> 32))
        return fail(QSIM_EINVAL, "ac_set_counters: bad argument");
    a->t_actor = t_actor; a->t_critic = t_critic; a->updates = updates;
    return QSIM_OK;
}

extern "C" int32_t ac_set_cluster(ac_handle* a, int32_t cluster) {
    if (!a) return fail(QSIM_EINVAL, "ac_set_cluster: null handle");
    if (cluster < 0 || cluster > 16 || (cluster & (cluster - 1)))
        return fail(QSIM_EINVAL, "ac_set_cluster: cluster must be 0 or a power of two <= 16");
    const int32_t prev = a->cfg.cluster;
    a->cfg.cluster = cluster;
    return prev;
}

extern "C" qsim_status ac_set_index_log(ac_handle* a, uint32_t* idx) {
    if (!a) return fail(QSIM_EINVAL, "ac_set_index_log: null handle");
    if (reinterpret_cast<uintptr_t>(idx) & 3u) return fail(QSIM_EINVAL, "ac_set_index_log: misaligned pointer");
    a->idx_log = idx;
    return QSIM_OK;
}

extern "C" qsim_status ac_update(ac_handle* a, qsim_handle* env, int32_t n_updates, void* stream) {
    SingleRun L;
    qsim_status s = prepare_single(a, env, 0, n_updates, "ac_update", &L);
    if (s != QSIM_OK || n_updates == 0) return s;
    return learner_run(a, env, n_updates, 0, L, (cudaStream_t)stream);
}

// ------------------------------------------------- allocation-free learner update
// Scratch for ac_update_static(): a library-owned array in every device's global memory
// (held from library load until process exit), plus room for the run descriptor.
// Host code must not pass the symbol itself to a kernel (in host code it names a host-side
// stand-in); the device address comes from cudaGetSymbolAddress, looked up once per device.
// A run fits if its scratch in FP32 rows does, or that in tiles: the tensor-core passes' tiles and
// halves take up to 0.7 MiB more than the rows (181,248 floats at hidden 32, batch 1,024, no
// history, cluster 4; all shapes ac_create takes), for which the array has room.
constexpr size_t kStaticArea = QSIM_STATIC_SCRATCH_BYTES + (1u << 20);
static __device__ __align__(256) float g_static_scratch[kStaticArea / sizeof(float)];
static __device__ __align__(256) unsigned char g_static_desc[QSIM_STATIC_DESC_BYTES];

namespace {
struct StaticSlot {
    float* scratch = nullptr;
    unsigned char* desc = nullptr;
    bool ready = false;
};
constexpr int kMaxDevices = 64;
StaticSlot g_static_slots[kMaxDevices];
std::mutex g_static_mutex;

// Resolves the device addresses of the static arrays for the current device (first call
// on each device only).
qsim_status static_slot(int device, StaticSlot** out) {
    if (device < 0 || device >= kMaxDevices) return fail(QSIM_EINVAL, "ac_update_static: device id %d", device);
    std::lock_guard<std::mutex> lock(g_static_mutex);
    StaticSlot& s = g_static_slots[device];
    if (!s.ready) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "ac_update_static: cudaGetSymbolAddress(scratch)");
        s.scratch = static_cast<float*>(p);
        e = cudaGetSymbolAddress(&p, g_static_desc);
        if (e != cudaSuccess) return cuda_fail(e, "ac_update_static: cudaGetSymbolAddress(desc)");
        s.desc = static_cast<unsigned char*>(p);
        s.ready = true;
    }
    *out = &s;
    return QSIM_OK;
}
}  // namespace

extern "C" qsim_status ac_update_static(ac_handle* a, qsim_handle* env, int32_t n_updates,
                                        void* stream) {
    SingleRun L;
    qsim_status st = prepare_single(a, env, 0, n_updates, "ac_update_static", &L);
    if (st != QSIM_OK || n_updates == 0) return st;
    const size_t per_cta = std::min(L.stride, scratch_floats(a->batch / L.nS, a->hidden, a->obs_dim, a->critic_in,
                                                             a->n_actor, a->n_critic, env->n, L.nS, false));
    const size_t need = per_cta * sizeof(float) * (size_t)L.nS;
    if (need > QSIM_STATIC_SCRATCH_BYTES || L.stride * sizeof(float) * (size_t)L.nS > kStaticArea)
        return fail(QSIM_EINVAL,
                    "ac_update_static: needs %zu bytes of scratch (batch %d, hidden %d, cluster %d), "
                    "more than the static maximum of %d bytes; use ac_update",
                    need, a->batch, a->hidden, L.nS, (int)QSIM_STATIC_SCRATCH_BYTES);
    StaticSlot* slot = nullptr;
    st = static_slot(a->device, &slot);
    if (st != QSIM_OK) return st;
    // the shared descriptor area is rewritten on every call (no mirror)
    return run_single(a, env, n_updates, 0, L, slot->desc, slot->scratch, nullptr, (cudaStream_t)stream);
}

extern "C" qsim_status ac_train(ac_handle* const* runs, qsim_handle* const* envs, int32_t n_runs,
                                int64_t steps_per_run, int32_t persistent, void* stream) {
    if (!runs || !envs || n_runs < 1 || steps_per_run < 0 || persistent < 0 || persistent > 2)
        return fail(QSIM_EINVAL, "ac_train: bad argument");
    std::vector<ac_handle*> A(runs, runs + n_runs);
    std::vector<qsim_handle*> E(envs, envs + n_runs);
    std::vector<SingleRun> L(n_runs);
    for (int i = 0; i < n_runs; ++i) {
        qsim_status s = prepare_single(A[i], E[i], 1, steps_per_run, "ac_train", &L[i]);
        if (s != QSIM_OK) return s;
    }
    if (steps_per_run == 0) return QSIM_OK;
    cudaStream_t st = (cudaStream_t)stream;
    if (persistent == 0) {
        // plain form: one launch per run and env step, each run on its own cluster size
        for (int64_t t = 0; t < steps_per_run; ++t)
            for (int i = 0; i < n_runs; ++i) {
                qsim_status s = learner_run(A[i], E[i], 1, 1, L[i], st);
                if (s != QSIM_OK) return s;
            }
        return QSIM_OK;
    }
    if (persistent == 2 || n_runs == 1) {
        // one launch per run for all its steps, runs one after another
        for (int i = 0; i < n_runs; ++i) {
            qsim_status s = learner_run(A[i], E[i], steps_per_run, 1, L[i], st);
            if (s != QSIM_OK) return s;
        }
        return QSIM_OK;
    }
    const int nS = pick_cluster(A[0], n_runs);
    for (int i = 1; i < n_runs; ++i)
        if (pick_cluster(A[i], n_runs) != nS) return fail(QSIM_EINVAL, "ac_train: runs need one cluster size");
    int max_clusters = 1;
    {
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3(nS * 1024);
        lc.blockDim = dim3(LT);
        lc.dynamicSmemBytes = learner_smem();
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = nS;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        lc.attrs = attr;
        lc.numAttrs = 1;
        if (nS > 8) cudaFuncSetAttribute(k_train, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (cudaOccupancyMaxActiveClusters(&max_clusters, k_train, &lc) != cudaSuccess || max_clusters < 1) {
            cudaGetLastError();
            int sms = 152;
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, A[0]->device);
            max_clusters = std::max(1, sms / nS);
        }
    }
    return launch_train(A, E, steps_per_run, 1, nS, st, max_clusters);
}

// Autotuner of the batched launch: the cluster size S (CTAs per run) is timed on the runs
// themselves, every candidate that divides each run's batch with >= 16 samples per CTA.
extern "C" int32_t ac_train_autotune(ac_handle* const* runs, qsim_handle* const* envs, int32_t n_runs,
                                     int32_t trial_steps, void* stream) {
    if (!runs || !envs || n_runs < 1 || trial_steps < 1)
        return fail(QSIM_EINVAL, "ac_train_autotune: bad argument");
    for (int i = 0; i < n_runs; ++i)
        if (!runs[i] || !envs[i]) return fail(QSIM_EINVAL, "ac_train_autotune: null handle");
    cudaStream_t st = (cudaStream_t)stream;
    std::vector<int> saved(n_runs);
    for (int i = 0; i < n_runs; ++i) saved[i] = runs[i]->cfg.cluster;
    auto restore = [&]() { for (int i = 0; i < n_runs; ++i) runs[i]->cfg.cluster = saved[i]; };
    // one untimed call with the current setting: first-launch costs stay out of the trials
    qsim_status s0 = ac_train(runs, envs, n_runs, trial_steps, 1, stream);
    if (s0 != QSIM_OK) return s0;
    cudaEvent_t e0, e1;
    QCHECK_CUDA(cudaEventCreate(&e0));
    QCHECK_CUDA(cudaEventCreate(&e1));
    float best = 1e30f;
    int best_s = 0;
    for (int cand : {1, 2, 4, 8, 16}) {
        bool ok = true;
        for (int i = 0; i < n_runs; ++i) {
            const int b = runs[i]->batch;
            if (b % cand || (cand > 1 && b / cand < 16)) ok = false;
        }
        if (!ok) continue;
        for (int i = 0; i < n_runs; ++i) runs[i]->cfg.cluster = cand;
        cudaEventRecord(e0, st);
        const qsim_status r = ac_train(runs, envs, n_runs, trial_steps, 1, stream);
        cudaEventRecord(e1, st);
        if (r != QSIM_OK) {
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
            restore();
            return r;
        }
        cudaEventSynchronize(e1);
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < best) {
            best = ms;
            best_s = cand;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    QCHECK_LAUNCH("ac_train_autotune");
    for (int i = 0; i < n_runs; ++i) runs[i]->cfg.cluster = best_s;
    return best_s;
}

// ------------------------------------------------------------ graph-captured plans
struct ac_plan {
    std::vector<ac_handle*> A;
    std::vector<qsim_handle*> E;
    RunDesc* d_runs = nullptr;
    int* d_order = nullptr;
    int* d_off = nullptr;
    float* scratch = nullptr;
    size_t stride = 0;
    int nS = 1, n_clusters = 1, chunk = 1;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    int64_t steps_run = 0;
};

extern "C" qsim_status ac_plan_destroy(ac_plan* p) {
    if (!p) return QSIM_OK;
    if (p->exec) cudaGraphExecDestroy(p->exec);
    if (p->graph) cudaGraphDestroy(p->graph);
    if (p->d_runs) cudaFree(p->d_runs);
    if (p->d_order) cudaFree(p->d_order);
    if (p->d_off) cudaFree(p->d_off);
    if (p->scratch) cudaFree(p->scratch);
    delete p;
    return QSIM_OK;
}

extern "C" qsim_status ac_plan_create(ac_handle* const* runs, qsim_handle* const* envs,
                                      int32_t n_runs, int32_t steps_per_chunk, ac_plan** out) {
    if (!runs || !envs || !out || n_runs < 1 || steps_per_chunk < 1)
        return fail(QSIM_EINVAL, "ac_plan_create: bad argument");
    *out = nullptr;
    ac_plan* p = new ac_plan();
    p->A.assign(runs, runs + n_runs);
    p->E.assign(envs, envs + n_runs);
    p->chunk = steps_per_chunk;
    for (int i = 0; i < n_runs; ++i) {
        qsim_status s = validate_pair(p->A[i], p->E[i]);
        if (s != QSIM_OK) { ac_plan_destroy(p); return s; }
        if ((uint64_t)p->E[i]->capacity * (uint64_t)p->E[i]->n >= (1ull << 32)) {
            ac_plan_destroy(p);
            return fail(QSIM_EINVAL, "ac_plan_create: replay buffer exceeds 2^32 transitions");
        }
    }
    p->nS = pick_cluster(p->A[0], n_runs);
    for (int i = 0; i < n_runs; ++i)
        if (pick_cluster(p->A[i], n_runs) != p->nS || p->A[i]->batch % p->nS) {
            ac_plan_destroy(p);
            return fail(QSIM_EINVAL, "ac_plan_create: runs need one cluster size dividing every batch");
        }
    const int nS = p->nS;
    int max_clusters = 1;
    {
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3(nS * 1024);
        lc.blockDim = dim3(LT);
        lc.dynamicSmemBytes = learner_smem();
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = nS;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        lc.attrs = attr;
        lc.numAttrs = 1;
        if (nS > 8) cudaFuncSetAttribute(k_train, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (cudaOccupancyMaxActiveClusters(&max_clusters, k_train, &lc) != cudaSuccess || max_clusters < 1) {
            cudaGetLastError();
            int sms = 152;
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->A[0]->device);
            max_clusters = std::max(1, sms / nS);
        }
    }
    const int n = n_runs;
    p->n_clusters = std::max(1, std::min(n, max_clusters));
    std::vector<RunDesc> D(n);
    for (int i = 0; i < n; ++i) {
        qsim_status s = fill_desc(p->A[i], p->E[i], D[i]);
        if (s != QSIM_OK) { ac_plan_destroy(p); return s; }
        p->stride = std::max(p->stride, scratch_floats(p->A[i]->batch / nS, p->A[i]->hidden,
                                                       p->A[i]->obs_dim, p->A[i]->critic_in,
                                                       p->A[i]->n_actor, p->A[i]->n_critic, p->E[i]->n, nS));
    }
    int use_tc = 0;
    for (int i = 0; i < n; ++i) use_tc |= tc_wanted(D[i], nS) ? 1 : 0;
    // longest-processing-time-first assignment of runs to clusters
    std::vector<int> order(n), off(p->n_clusters + 1, 0);
    {
        std::vector<double> cost(n);
        for (int i = 0; i < n; ++i) cost[i] = run_cost(p->A[i], p->E[i], nS);
        std::vector<int> idx(n);
        std::iota(idx.begin(), idx.end(), 0);
        std::stable_sort(idx.begin(), idx.end(), [&](int x, int y) { return cost[x] > cost[y]; });
        std::vector<double> load(p->n_clusters, 0.0);
        std::vector<std::vector<int>> lists(p->n_clusters);
        for (int i : idx) {
            int best = 0;
            for (int c = 1; c < p->n_clusters; ++c)
                if (load[c] < load[best]) best = c;
            load[best] += cost[i];
            lists[best].push_back(i);
        }
        int k = 0;
        for (int c = 0; c < p->n_clusters; ++c) {
            off[c] = k;
            for (int i : lists[c]) order[k++] = i;
        }
        off[p->n_clusters] = k;
    }
    const size_t scr_bytes = sizeof(float) * p->stride * (size_t)p->n_clusters * nS;
    if (cudaMalloc((void**)&p->d_runs, sizeof(RunDesc) * n) != cudaSuccess ||
        cudaMalloc((void**)&p->d_order, sizeof(int) * n) != cudaSuccess ||
        cudaMalloc((void**)&p->d_off, sizeof(int) * (p->n_clusters + 1)) != cudaSuccess ||
        cudaMalloc((void**)&p->scratch, scr_bytes) != cudaSuccess) {
        cudaGetLastError();
        ac_plan_destroy(p);
        return fail(QSIM_ENOMEM, "ac_plan_create: allocation failed");
    }
    cudaMemcpy(p->d_runs, D.data(), sizeof(RunDesc) * n, cudaMemcpyHostToDevice);
    cudaMemcpy(p->d_order, order.data(), sizeof(int) * n, cudaMemcpyHostToDevice);
    cudaMemcpy(p->d_off, off.data(), sizeof(int) * (p->n_clusters + 1), cudaMemcpyHostToDevice);
    // capture one chunk of the persistent launch
    cudaStream_t cs;
    QCHECK_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(p->n_clusters * nS);
    lc.blockDim = dim3(LT);
    lc.dynamicSmemBytes = learner_smem();
    lc.stream = cs;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = nS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess)
        e = cudaLaunchKernelEx(&lc, k_train, p->d_runs, (const int*)p->d_order, (const int*)p->d_off,
                               steps_per_chunk, 1, p->scratch, p->stride, nS, use_tc);
    cudaError_t e2 = cudaStreamEndCapture(cs, &p->graph);
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&p->exec, p->graph, 0);
    cudaStreamDestroy(cs);
    if (e != cudaSuccess) {
        ac_plan_destroy(p);
        return cuda_fail(e, "ac_plan_create: graph capture");
    }
    *out = p;
    return QSIM_OK;
}

extern "C" qsim_status ac_plan_run(ac_plan* p, int32_t n_chunks, void* stream) {
    if (!p || n_chunks < 0) return fail(QSIM_EINVAL, "ac_plan_run: bad argument");
    for (size_t i = 0; i < p->E.size(); ++i)
        if (((p->E[i]->t_now + p->steps_run + (int64_t)n_chunks * p->chunk) >> 32) != 0)
            return fail(QSIM_ESTATE, "ac_plan_run: step counter exhausted");
    for (int c = 0; c < n_chunks; ++c) QCHECK_CUDA(cudaGraphLaunch(p->exec, (cudaStream_t)stream));
    p->steps_run += (int64_t)n_chunks * p->chunk;
    return QSIM_OK;
}

extern "C" qsim_status ac_plan_sync(ac_plan* p, void* stream) {
    if (!p) return fail(QSIM_EINVAL, "ac_plan_sync: null plan");
    const size_t n = p->A.size();
    std::vector<RunDesc> D(n);
    QCHECK_CUDA(cudaMemcpyAsync(D.data(), p->d_runs, sizeof(RunDesc) * n, cudaMemcpyDeviceToHost,
                                (cudaStream_t)stream));
    QCHECK_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
    for (size_t i = 0; i < n; ++i) read_back(p->A[i], p->E[i], D[i]);
    p->steps_run = 0;
    return QSIM_OK;
}

extern "C" qsim_status ac_sync(ac_handle* a) {
    if (!a) return fail(QSIM_EINVAL, "ac_sync: null handle");
    QCHECK_CUDA(cudaDeviceSynchronize());
    return QSIM_OK;
}

// ------------------------------------------------------------------------ checkpoints
namespace {
struct CkptHeader {
    char magic[8];
    int32_t abi, obs_dim, critic_in, hidden, n_actor, n_critic, n_env, ld;
    int64_t t_actor, t_critic, updates, t_now, head, size, next_curr;
};
}  // namespace

extern "C" qsim_status ac_save(const ac_handle* a, const qsim_handle* e, const char* path) {
    if (!a || !e || !path) return fail(QSIM_EINVAL, "ac_save: null pointer");
    CkptHeader h;
    memset(&h, 0, sizeof(h));
    memcpy(h.magic, "QSIMCKP1", 8);
    h.abi = QSIM_ABI_VERSION; h.obs_dim = a->obs_dim; h.critic_in = a->critic_in; h.hidden = a->hidden;
    h.n_actor = a->n_actor; h.n_critic = a->n_critic; h.n_env = e->n; h.ld = e->ld;
    h.t_actor = a->t_actor; h.t_critic = a->t_critic; h.updates = a->updates;
    h.t_now = e->t_now; h.head = e->head; h.size = e->size; h.next_curr = e->next_curriculum;
    const size_t nparam = 4 * (size_t)a->n_actor + 8 * (size_t)a->n_critic;
    std::vector<float> w(nparam);
    QCHECK_CUDA(cudaDeviceSynchronize());
    QCHECK_CUDA(cudaMemcpy(w.data(), a->base, nparam * 4, cudaMemcpyDeviceToHost));
    const size_t ld = e->ld;
    std::vector<float> env_f((NS + 8 + 6 + 4 * HMAX + 2) * ld + 8);
    std::vector<uint32_t> env_u(4 * ld);
    float* f = env_f.data();
    QCHECK_CUDA(cudaMemcpy(f, e->p.state, NS * ld * 4, cudaMemcpyDeviceToHost)); f += NS * ld;
    QCHECK_CUDA(cudaMemcpy(f, e->p.prm, 8 * ld * 4, cudaMemcpyDeviceToHost)); f += 8 * ld;
    QCHECK_CUDA(cudaMemcpy(f, e->p.dist, 6 * ld * 4, cudaMemcpyDeviceToHost)); f += 6 * ld;
    QCHECK_CUDA(cudaMemcpy(f, e->p.hist, 4 * HMAX * ld * 4, cudaMemcpyDeviceToHost)); f += 4 * HMAX * ld;
    QCHECK_CUDA(cudaMemcpy(f, e->p.ep_ret, ld * 4, cudaMemcpyDeviceToHost)); f += ld;
    QCHECK_CUDA(cudaMemcpy(f, e->p.ret_sum, ld * 4, cudaMemcpyDeviceToHost)); f += ld;
    QCHECK_CUDA(cudaMemcpy(f, e->p.rewardC, 8 * 4, cudaMemcpyDeviceToHost));
    QCHECK_CUDA(cudaMemcpy(env_u.data(), e->p.ep_index, ld * 4, cudaMemcpyDeviceToHost));
    QCHECK_CUDA(cudaMemcpy(env_u.data() + ld, e->p.ep_step, ld * 4, cudaMemcpyDeviceToHost));
    QCHECK_CUDA(cudaMemcpy(env_u.data() + 2 * ld, e->p.n_done, ld * 4, cudaMemcpyDeviceToHost));
    QCHECK_CUDA(cudaMemcpy(env_u.data() + 3 * ld, e->p.len_sum, ld * 4, cudaMemcpyDeviceToHost));
    std::ofstream os(path, std::ios::binary);
    if (!os) return fail(QSIM_EINVAL, "ac_save: cannot open %s", path);
    os.write((const char*)&h, sizeof(h));
    os.write((const char*)w.data(), w.size() * 4);
    os.write((const char*)env_f.data(), env_f.size() * 4);
    os.write((const char*)env_u.data(), env_u.size() * 4);
    if (!os) return fail(QSIM_EINVAL, "ac_save: write failed");
    return QSIM_OK;
}

extern "C" qsim_status ac_load(ac_handle* a, qsim_handle* e, const char* path) {
    if (!a || !e || !path) return fail(QSIM_EINVAL, "ac_load: null pointer");
    std::ifstream is(path, std::ios::binary);
    if (!is) return fail(QSIM_EINVAL, "ac_load: cannot open %s", path);
    CkptHeader h;
    is.read((char*)&h, sizeof(h));
    if (!is || memcmp(h.magic, "QSIMCKP1", 8) != 0) return fail(QSIM_EVERSION, "ac_load: not a checkpoint");
    if (h.abi != QSIM_ABI_VERSION || h.obs_dim != a->obs_dim || h.critic_in != a->critic_in ||
        h.hidden != a->hidden || h.n_actor != a->n_actor || h.n_critic != a->n_critic ||
        h.n_env != e->n || h.ld != e->ld)
        return fail(QSIM_EVERSION, "ac_load: checkpoint layout does not match the handles");
    const size_t nparam = 4 * (size_t)a->n_actor + 8 * (size_t)a->n_critic;
    const size_t ld = e->ld;
    std::vector<float> w(nparam), env_f((NS + 8 + 6 + 4 * HMAX + 2) * ld + 8);
    std::vector<uint32_t> env_u(4 * ld);
    is.read((char*)w.data(), w.size() * 4);
    is.read((char*)env_f.data(), env_f.size() * 4);
    is.read((char*)env_u.data(), env_u.size() * 4);
    if (!is) return fail(QSIM_EVERSION, "ac_load: truncated checkpoint");
    QCHECK_CUDA(cudaDeviceSynchronize());
    QCHECK_CUDA(cudaMemcpy(a->base, w.data(), nparam * 4, cudaMemcpyHostToDevice));
    const float* f = env_f.data();
    QCHECK_CUDA(cudaMemcpy(e->p.state, f, NS * ld * 4, cudaMemcpyHostToDevice)); f += NS * ld;
    QCHECK_CUDA(cudaMemcpy(e->p.prm, f, 8 * ld * 4, cudaMemcpyHostToDevice)); f += 8 * ld;
    QCHECK_CUDA(cudaMemcpy(e->p.dist, f, 6 * ld * 4, cudaMemcpyHostToDevice)); f += 6 * ld;
    QCHECK_CUDA(cudaMemcpy(e->p.hist, f, 4 * HMAX * ld * 4, cudaMemcpyHostToDevice)); f += 4 * HMAX * ld;
    QCHECK_CUDA(cudaMemcpy(e->p.ep_ret, f, ld * 4, cudaMemcpyHostToDevice)); f += ld;
    QCHECK_CUDA(cudaMemcpy(e->p.ret_sum, f, ld * 4, cudaMemcpyHostToDevice)); f += ld;
    QCHECK_CUDA(cudaMemcpy(e->p.rewardC, f, 8 * 4, cudaMemcpyHostToDevice));
    QCHECK_CUDA(cudaMemcpy(e->p.ep_index, env_u.data(), ld * 4, cudaMemcpyHostToDevice));
    QCHECK_CUDA(cudaMemcpy(e->p.ep_step, env_u.data() + ld, ld * 4, cudaMemcpyHostToDevice));
    QCHECK_CUDA(cudaMemcpy(e->p.n_done, env_u.data() + 2 * ld, ld * 4, cudaMemcpyHostToDevice));
    QCHECK_CUDA(cudaMemcpy(e->p.len_sum, env_u.data() + 3 * ld, ld * 4, cudaMemcpyHostToDevice));
    a->t_actor = h.t_actor; a->t_critic = h.t_critic; a->updates = h.updates;
    e->t_now = h.t_now; e->head = h.head; e->size = h.size; e->next_curriculum = h.next_curr;
    return QSIM_OK;
}
