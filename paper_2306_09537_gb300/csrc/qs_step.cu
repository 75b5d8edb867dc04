// qs_step.cu -- the fused control step (S1..S13) on sm_103a, in two forms:
//
//  k_step<W>   one control step per launch (qs_step): state read from and
//              written back to HBM.
//  k_rollout   T control steps per launch (qs_rollout): a persistent kernel
//              whose CTAs pull tiles of envs from a work counter (widest,
//              costliest classes first) and keep each drone's state in
//              registers across the T steps; one launch covers envs of every
//              swarm size.
//
// Layout: a CTA processes env "slots" of one width class W (a power of two >=
// the env's swarm size N); thread `lane` of a slot carries drone `lane` of the
// env. For W > 1 the slot exchanges positions and velocities through shared
// memory for the O(N^2) pair pass (collisions, Sec. III-B) and the K-nearest
// neighbour selection (Sec. II-B, III-C), which each thread keeps as a sorted
// register list of 32-bit words (pair_scan).
#include <cuda_runtime.h>
#include <stdint.h>

#include "qs_device.cuh"
#include "qs_internal.h"
#include "qs_scenario.cuh"

namespace qsk {

constexpr int MAX_BLOCK = 256;
// dynamic shared memory of the step and rollout kernels, floats per thread:
// staged position (4: one 16-byte load a partner) and velocity (3) of the pair
// pass, swap key (1). The rollout stages by step parity in two such sets: a
// slot wider than a warp would otherwise stage step t + 1 over what its slower
// warps still read for step t's neighbour rows.
constexpr int SMEM_PLANES = 8;
// the rollout's observation rows in shared memory, floats per thread: a row and
// the padding of its block (RowMap)
constexpr int ROW_PAD = 6;
// and the most the kernels ask for
constexpr int STEP_SMEM_MAX =
    (int)sizeof(float) * MAX_BLOCK * (2 * SMEM_PLANES + GOAL_STRIDE + 18 + 6 * QS_MAX_K + ROW_PAD);

// The step kernels come in three instances, EXT = extended_instance(): 0 the
// common configuration (one goal, no downwash, the paper's discrete contacts)
// with all of it decided at compile time, so it keeps the smaller code and
// register budget and the substep's contact branch is straight-line code; 1
// with the training scenarios (per-drone goals) and the downwash term, decided
// at run time; 2 that with the smooth contacts in place of the discrete ones.
// (Deciding the contacts at run time too, the dynamics side of 1999 swarms of 7
// under every scenario took 4,600 cycles for its substeps against 3,700.)
inline int extended(const Consts& c) { return extended_instance(c); }

// Per-env values a thread keeps in registers.
struct EnvRegs {
    Prm p;
    float g0, g1, g2;
    int ep;
    uint32_t tick;
    int sel;       // active buffer of the env's scenario record
    bool redrawn;  // auto-reset drew new parameters / goal this launch
};

template <int EXT>
__device__ __forceinline__ void load_env(EnvRegs& er, const Consts& c, const Dev& dv, int e) {
    er.p = load_prm(c, dv.prm, dv.E, e);
    er.g0 = dv.goal[e];
    er.g1 = dv.goal[dv.E + e];
    er.g2 = dv.goal[2 * dv.E + e];
    er.ep = dv.ep[e];
    er.tick = dv.tick[e];
    er.sel = (EXT && (c.scn_mask & ~1u)) ? dv.scn_sel[e] : 0;
    er.redrawn = false;
}

// Written by lane 0 of the slot at the end of a launch.
template <int EXT>
__device__ __forceinline__ void store_env(const EnvRegs& er, const Dev& dv, int e) {
    dv.ep[e] = er.ep;
    dv.tick[e] = er.tick;
    if (er.redrawn) {
        const float v[NPRM_DEV] = {er.p.m, er.p.ixx, er.p.iyy, er.p.izz, er.p.t2w, er.p.tau, er.p.arm, er.p.fmax,
                                   er.p.alag, er.p.ans, er.p.inv_m, er.p.inv_ixx, er.p.inv_iyy, er.p.inv_izz,
                                   er.p.thr, er.p.prox};
        for (int k = 0; k < NPRM_DEV; ++k) dv.prm[(size_t)k * dv.E + e] = v[k];
        dv.goal[e] = er.g0;
        dv.goal[dv.E + e] = er.g1;
        dv.goal[2 * dv.E + e] = er.g2;
        if (EXT) dv.scn_sel[e] = (uint8_t)er.sel;
    }
}

// Goal slot of drone `lane` under an active swap: the rank of its key among
// the keys staged by its env's drones at skey[sbase .. sbase + N) (ties to
// the lower index).
__device__ __forceinline__ int swap_rank(const uint32_t* skey, int sbase, int N, int lane, uint32_t myk) {
    int slot = 0;
    for (int j = 0; j < N; ++j) {
        const uint32_t kj = skey[sbase + j];
        slot += (kj < myk || (kj == myk && j < lane)) ? 1 : 0;
    }
    return slot;
}

// Downwash over the control step (duration substeps * dt): v_z += T az plus
// acceleration noise, w += T * angular-acceleration noise.
__device__ __forceinline__ void apply_downwash(const Consts& c, Drone& s, uint32_t tick, int d, float az) {
    float n[6];
    six_normals(c, tick, (uint32_t)d, TAG_DOWNWASH, 0, n);
    const float Tc = c.dt * (float)c.substeps;
    s.v[0] = __fmaf_rn(Tc, __fmul_rn(c.dw_sa, n[0]), s.v[0]);
    s.v[1] = __fmaf_rn(Tc, __fmul_rn(c.dw_sa, n[1]), s.v[1]);
    s.v[2] = fmaf(Tc, fmaf(c.dw_sa, n[2], az), s.v[2]);
    const float tsw = __fmul_rn(Tc, c.dw_sw);
    comp_add_prod(s.w[0], s.wlo[0], tsw, n[3]);
    comp_add_prod(s.w[1], s.wlo[1], tsw, n[4]);
    comp_add_prod(s.w[2], s.wlo[2], tsw, n[5]);
}

// S13 reward of one drone (Sec. III-E): weighted state terms, event indicators
// and the proximity term over its keff neighbours (pos(k): position of the k-th).
template <class Pos>
__device__ __forceinline__ float compute_reward(const Consts& c, const Drone& s, float prox, const float g[3],
                                                const float fh[4], uint32_t ev, int keff, const Pos& pos) {
    // explicit roundings: the same bits from every kernel that computes it
    const float dgx = __fsub_rn(s.x[0], g[0]), dgy = __fsub_rn(s.x[1], g[1]), dgz = __fsub_rn(s.x[2], g[2]);
    float r = __fmul_rn(c.w[QS_W_POS], sqrt_approx(dot3(dgx, dgy, dgz, dgx, dgy, dgz)));
    r = __fmaf_rn(c.w[QS_W_VEL], sqrt_approx(dot3(s.v[0], s.v[1], s.v[2], s.v[0], s.v[1], s.v[2])), r);
    r = __fmaf_rn(c.w[QS_W_ORI], s.R[8], r);
    r = __fmaf_rn(c.w[QS_W_SPIN], sqrt_approx(dot3(s.w[0], s.w[1], s.w[2], s.w[0], s.w[1], s.w[2])), r);
    const float na = __fmaf_rn(fh[3], fh[3], dot3(fh[0], fh[1], fh[2], fh[0], fh[1], fh[2]));
    r = __fmaf_rn(c.w[QS_W_ACT], sqrt_approx(na), r);
    const float q0 = __fsub_rn(fh[0], s.fp[0]), q1 = __fsub_rn(fh[1], s.fp[1]), q2 = __fsub_rn(fh[2], s.fp[2]),
                q3 = __fsub_rn(fh[3], s.fp[3]);
    r = __fmaf_rn(c.w[QS_W_DACT], sqrt_approx(__fmaf_rn(q3, q3, dot3(q0, q1, q2, q0, q1, q2))), r);
    const float tr = __fsub_rn(__fadd_rn(__fadd_rn(s.R[0], s.R[4]), s.R[8]), 1.0f);
    r = __fmaf_rn(__fmul_rn(c.w[QS_W_ROT], 0.5f), tr, r);
    r = __fmaf_rn(c.w[QS_W_YAW], s.R[0], r);
    r = __fadd_rn(r, (ev & EV_HIT_FLOOR) ? c.w[QS_W_HIT_FLOOR] : 0.0f);
    r = __fadd_rn(r, (ev & EV_ON_FLOOR) ? c.w[QS_W_ON_FLOOR] : 0.0f);
    r = __fadd_rn(r, (ev & EV_HIT_WALL) ? c.w[QS_W_HIT_WALL] : 0.0f);
    r = __fadd_rn(r, (ev & EV_HIT_CEIL) ? c.w[QS_W_HIT_CEIL] : 0.0f);
    r = __fadd_rn(r, (ev & EV_HIT_QUAD) ? c.w[QS_W_HIT_QUAD] : 0.0f);
    if (keff > 0 && c.w[QS_W_NEAR] != 0.0f) {
        float near = 0.0f;
        const float inv_prox = __frcp_rn(prox);
#pragma unroll
        for (int k = 0; k < QS_MAX_K; ++k) {
            if (k < keff) {
                const float3 q = pos(k);
                float dx, dy, dz;
                const float key = pair_key(s.x[0], s.x[1], s.x[2], q.x, q.y, q.z, dx, dy, dz);
                near = __fadd_rn(near, fmaxf(__fmaf_rn(-sqrt_approx(key), inv_prox, 1.0f), 0.0f));
            }
        }
        r = __fmaf_rn(c.w[QS_W_NEAR], near, r);
    }
    return r;
}

// End of a control step: previous command, episode counter, done flag,
// Philox counter, in-place auto-reset, non-finite check.
template <int EXT>
__device__ __forceinline__ void end_step(const Consts& c, const Dev& dv, Drone& s, EnvRegs& er, const float fh[4],
                                         int lane, int e, int d, uint8_t* __restrict__ done) {
    s.fp[0] = fh[0];
    s.fp[1] = fh[1];
    s.fp[2] = fh[2];
    s.fp[3] = fh[3];
    const uint32_t tick = er.tick;
    const int ep = er.ep + 1;
    const bool is_done = ep >= c.episode_steps;
    if (lane == 0 && done) done[e] = is_done ? 1 : 0;
    er.ep = (is_done && (c.flags & QS_F_AUTO_RESET)) ? 0 : ep;
    er.tick = tick + 1;
    if (is_done && (c.flags & QS_F_AUTO_RESET)) {
        // the env starts a new episode in place (new randomisation and goal);
        // every lane draws the env's values itself, so no exchange is needed
        float p7[QS_PARAM_DIM], goal[3], full[NPRM_DEV];
        draw_env(c, c.key0, c.key1, tick, TAG_AUTO_ENV, e, p7, goal);
        derive(c, p7, full);
        er.p = prm_from(full);
        er.g0 = goal[0];
        er.g1 = goal[1];
        er.g2 = goal[2];
        er.redrawn = true;
        draw_drone(c, c.key0, c.key1, tick, TAG_AUTO_DRONE, d, p7[P_T2W], s);
        if (EXT && (c.scn_mask & ~1u)) {
            // the next episode's record goes to the other buffer: lanes of
            // this env may still be reading the current one for this step
            er.sel ^= 1;
            if (lane == 0) {
                float rec[QS_NSCN];
                draw_scenario(c, c.key0, c.key1, tick, TAG_AUTO_SCN, e, rec);
                store_scenario(dv, er.sel, e, rec);
            }
        }
    }
    if (!finite_state(s)) atomicOr(dv.status, 1);
}

// Observation rows of a warp's drones on their way to memory. A row is od
// floats and a lane owns one, so rows written lane by lane put every store of a
// warp into 32 distinct sectors (K = 6: 27 stores of 8 bytes, 864 sectors for
// 216), and the warp waits for them before it may overwrite the registers they
// read. The rollout puts the rows together in shared memory instead and hands
// each block of consecutive rows to one bulk asynchronous copy, which runs
// while the warp computes the next step. The drones of a warp usually follow
// one another and form one block; the envs of a mixed handle's tile need not,
// and then each slot is a block. A bulk copy moves 16-byte units between
// addresses of the same offset: a block starts at its destination's offset
// within 16 bytes, and the 8 bytes before or after the units are stored apart.
struct RowMap {
    int d0, n;   // first drone and rows of the lane's block
    int off;     // the block's floats in the warp's buffer start here (a multiple of 4)
    int rank;    // row of this lane's drone in it
    int gl, gs;  // this lane's place among the gs lanes that share the block
    bool lead;   // the lane that hands the block over
};

__device__ __forceinline__ RowMap map_rows(bool act, int d, int W, int od) {
    RowMap r;
    const uint32_t am = __ballot_sync(0xffffffffu, act);
    const int ln = threadIdx.x & 31, rank = __popc(am & ((1u << ln) - 1u)), lead = max(__ffs(am) - 1, 0);
    const int f0 = __shfl_sync(0xffffffffu, d - rank, lead);
    const bool one = __all_sync(0xffffffffu, !act || d - rank == f0);
    if (one) {
        r = RowMap{f0, __popc(am), 0, rank, ln, 32, act && ln == lead};
    } else {  // slots of one warp: W <= 16
        const int slot = ln / W, l0 = slot * W;
        r = RowMap{d - (ln - l0), __popc(am >> l0 & ((1u << W) - 1u)), slot * (((W * od + 3) & ~3) + 4), ln - l0,
                   ln - l0, W, act && ln == l0};
    }
    return r;
}

// Floats from the block's start to its first row: the offset of the destination within 16 bytes.
__device__ __forceinline__ int row_shift(const RowMap& r, const float* obs, int od) {
    return (int)((uintptr_t)(obs + (size_t)r.d0 * od) >> 2) & 3;
}

// Before the rows of another step are written: the copies have read the last one's.
__device__ __forceinline__ void rows_free(const RowMap& r) {
    if (r.lead) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    __syncwarp();
}

// Sends the warp's blocks on their way (every lane calls it): bulk copies, or
// without bulk (destinations that may lie in host memory) stores by the lanes
// that share a block, side by side.
__device__ __forceinline__ void send_rows(const RowMap& r, const float* rows, float* __restrict__ obs, int od,
                                          bool bulk) {
    const int sh = row_shift(r, obs, od);
    const int n = r.n * od - sh, m = n & ~3;  // floats past the 8 bytes before the units
    const float* src = rows + r.off + sh;
    float* dst = obs + (size_t)r.d0 * od;
    if (bulk) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (!bulk) {
        const float4* s4 = reinterpret_cast<const float4*>(src + sh);
        float4* d4 = reinterpret_cast<float4*>(dst + sh);
        for (int i = r.gl; i < (m >> 2); i += r.gs) d4[i] = s4[i];
    }
    if (r.lead) {
        if (sh) *reinterpret_cast<float2*>(dst) = *reinterpret_cast<const float2*>(src);
        if (n & 2) *reinterpret_cast<float2*>(dst + sh + m) = *reinterpret_cast<const float2*>(src + sh + m);
        if (bulk)
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n\tcp.async.bulk.commit_group;" ::"l"(
                             dst + sh),
                         "r"((uint32_t)__cvta_generic_to_shared(src + sh)), "r"(4 * m)
                         : "memory");
    }
}

// ROWS: the observation rows go through shared memory (the rollout), else each
// lane stores its own. Swarm rollouts take the former (4096 uneven swarms, 32
// steps, 358 -> 299 us; 256 x 128, 16 steps, 203 -> 183 us) and the single
// drones' step; single-drone rollouts with short rows keep their stores (9 at
// K = 0): addressing the block costs 95 instructions of 1,100 a step, more than
// the stores' waits (1,048,576 drones, 32 steps: 1696 against 1834 us; single_form).
template <int EXT, bool ROWS>
__device__ __forceinline__ void step_body(const int W, const Consts& c, const Dev& dv, Drone& s, EnvRegs& er,
                                          uint32_t& ev_out, float4* sp, float* sv, const bool act, const int lane,
                                          const int N, const int sbase, const int e, const int d, const float4 a,
                                          float* __restrict__ obs, float* __restrict__ rew, uint8_t* __restrict__ done,
                                          const int observe_only, GoalCache& gc, const RowMap& rm, float* rows,
                                          const bool bulk) {
    const int nt = blockDim.x;
    const int K = c.K;
    const int keff = min(K, N - 1);
    const uint32_t tick = er.tick;
    // the EXT = 0 instance carries neither scenario nor downwash code
    const bool scn = EXT && (c.scn_mask & ~1u) != 0;
    const bool dw = EXT && (c.flags & QS_F_DOWNWASH) != 0;
    const int tau = observe_only ? er.ep : er.ep + 1;  // the goal is the one at the step's end
    uint32_t* skey = reinterpret_cast<uint32_t*>(sv + 3 * nt);
    bool swp = false;
    uint32_t myk = 0;
    float fh[4] = {0.f, 0.f, 0.f, 0.f};
    uint32_t ev = 0;
    // smooth contacts of a swarm (general instance): the pair penalty from the
    // positions at each substep's start, staged like the pair pass (uniform
    // over the CTA: every thread meets the barriers)
    const bool spair = EXT == 2 && W > 1 && !observe_only;
    if (spair) {
        if (act) {
            fh[0] = command(c, a.x);
            fh[1] = command(c, a.y);
            fh[2] = command(c, a.z);
            fh[3] = command(c, a.w);
        }
        const float u[4] = {sqrt_approx(fh[0]), sqrt_approx(fh[1]), sqrt_approx(fh[2]), sqrt_approx(fh[3])};
        for (int sub = 0; sub < c.substeps; ++sub) {
            float pacc[3] = {0.f, 0.f, 0.f};
            if (act) sp[threadIdx.x] = make_float4(s.x[0], s.x[1], s.x[2], 0.f);
            __syncthreads();
            if (act && N > 1) pair_acc(c, s.x, sp, sbase, lane, N, er.p.arm, pacc);
            __syncthreads();
            if (act) ev |= substep<false, EXT == 2 ? 1 : 0>(s, er.p, c, u, tick, d, sub, pacc);
        }
    } else if (act && !observe_only) {
        fh[0] = command(c, a.x);
        fh[1] = command(c, a.y);
        fh[2] = command(c, a.z);
        fh[3] = command(c, a.w);
        const float u[4] = {sqrt_approx(fh[0]), sqrt_approx(fh[1]), sqrt_approx(fh[2]), sqrt_approx(fh[3])};
        const float zero3[3] = {0.f, 0.f, 0.f};
        for (int sub = 0; sub < c.substeps; ++sub)
            ev |= substep<false, EXT == 2 ? 1 : 0>(s, er.p, c, u, tick, d, sub, zero3);
    }

    // ---- pair pass: collisions (S9, S10) and K nearest neighbours (S11)
    NbrList nbrs = 0;
    if (W > 1) {
        if (act) {
            sp[threadIdx.x] = make_float4(s.x[0], s.x[1], s.x[2], 0.f);
            sv[threadIdx.x] = s.v[0];
            sv[nt + threadIdx.x] = s.v[1];
            sv[2 * nt + threadIdx.x] = s.v[2];
        }
        __syncthreads();
        float dvs[3] = {0.f, 0.f, 0.f};
        bool responded = false, dw_hit = false;
        float dw_az = 0.f;
        if (act && N > 1) {
            const bool coll = (c.flags & QS_F_COLLISIONS) && EXT != 2 && !observe_only;
            const bool flag_coll = (c.flags & QS_F_COLLISIONS) && !observe_only;
            responded = pair_scan<(EXT > 0)>(c, s, er.p.thr, lane, N, sbase, sp, sv, nt, keff, coll, flag_coll, ev,
                                             nbrs, dvs, dw && !observe_only, dw_az, dw_hit);
        }
        if (responded) apply_response(c, s, tick, d, dvs);
        if (dw && dw_hit && !observe_only) apply_downwash(c, s, tick, d, dw_az);
        __syncthreads();
        if (act) {  // post-collision velocities for the neighbour observation
            sv[threadIdx.x] = s.v[0];
            sv[nt + threadIdx.x] = s.v[1];
            sv[2 * nt + threadIdx.x] = s.v[2];
            if (scn && !goal_cached(gc, tau) && swap_active(dv, er.sel, e, tau)) {
                swp = true;
                myk = swap_key(c, scn_seed(dv, er.sel, e), lane);
                skey[threadIdx.x] = myk;
            }
        }
        __syncthreads();
    }
    if (!ROWS && !act) return;

    // ---- the drone's goal at the end of the step (Sec. III-D scenarios)
    float gl[3] = {er.g0, er.g1, er.g2};
    if (scn && act) {
        if (!goal_cached(gc, tau))
            goal_fill(gc, c, dv, er.sel, e, lane, N, tau, swp ? swap_rank(skey, sbase, N, lane, myk) : lane, gl);
        goal_at(gc, c, tau, gl);
    }

    // ---- S12 observation
    if (ROWS && obs) rows_free(rm);
    if (obs && act) {
        float ex[3] = {0.f, 0.f, 0.f}, evv[3] = {0.f, 0.f, 0.f}, ew[3] = {0.f, 0.f, 0.f};
        if (c.flags & QS_F_OBS_NOISE) obs_noise(c, tick, d, observe_only ? 1u : 0u, ex, evv, ew);
        float2* o2 = reinterpret_cast<float2*>(ROWS ? rows + rm.off + row_shift(rm, obs, c.obs_dim) + rm.rank * c.obs_dim
                                                    : obs + (size_t)d * c.obs_dim);
        o2[0] = make_float2(s.x[0] - gl[0] + ex[0], s.x[1] - gl[1] + ex[1]);
        o2[1] = make_float2(s.x[2] - gl[2] + ex[2], s.v[0] + evv[0]);
        o2[2] = make_float2(s.v[1] + evv[1], s.v[2] + evv[2]);
        o2[3] = make_float2(s.R[0], s.R[1]);
        o2[4] = make_float2(s.R[2], s.R[3]);
        o2[5] = make_float2(s.R[4], s.R[5]);
        o2[6] = make_float2(s.R[6], s.R[7]);
        o2[7] = make_float2(s.R[8], s.w[0] + ew[0]);
        o2[8] = make_float2(s.w[1] + ew[1], s.w[2] + ew[2]);
#pragma unroll
        for (int k = 0; k < QS_MAX_K; ++k) {
            if (k >= K) break;
            float2* on = o2 + 9 + 3 * k;
            if (W > 1 && k < keff) {
                const int tj = sbase + nbr_at(nbrs, k);
                const float4 q = sp[tj];
                on[0] = make_float2(q.x - s.x[0], q.y - s.x[1]);
                on[1] = make_float2(q.z - s.x[2], sv[tj] - s.v[0]);
                on[2] = make_float2(sv[nt + tj] - s.v[1], sv[2 * nt + tj] - s.v[2]);
            } else {
                on[0] = make_float2(0.f, 0.f);
                on[1] = make_float2(0.f, 0.f);
                on[2] = make_float2(0.f, 0.f);
            }
        }
    }
    if (ROWS && obs) send_rows(rm, rows, obs, c.obs_dim, bulk);
    if (!act || observe_only) return;

    if ((c.flags & QS_F_RECORD_KNN) && dv.knn) {
#pragma unroll
        for (int k = 0; k < QS_MAX_K; ++k)
            if (k < K) dv.knn[(size_t)k * dv.D + d] = (W > 1 && k < keff) ? (int16_t)nbr_at(nbrs, k) : (int16_t)-1;
    }
    ev_out = ev;

    // ---- S13 reward and done
    if (rew)
        rew[d] = compute_reward(c, s, er.p.prox, gl, fh, ev, W > 1 ? keff : 0, [&](int k) {
            const float4 q = sp[sbase + nbr_at(nbrs, k)];
            return make_float3(q.x, q.y, q.z);
        });
    end_step<EXT>(c, dv, s, er, fh, lane, e, d, done);
    if (scn && er.ep == 0) gc.until = -1;  // an auto-reset drew a new record
}

struct SlotMap {
    int slot, lane, e, d0, N, d, sbase;
    bool act;
};

__device__ __forceinline__ SlotMap map_slot(const Dev& dv, const Tile& tile, const int* __restrict__ perm, int W) {
    SlotMap m;
    m.slot = threadIdx.x / W;
    m.lane = threadIdx.x - m.slot * W;
    const SlotGeo g = slot_geometry(dv, perm, tile, m.slot, W, blockDim.x);
    m.e = g.e;
    m.d0 = g.d0;
    m.N = g.N;
    m.act = m.lane < m.N;
    m.d = m.d0 + m.lane;
    m.sbase = m.slot * W;
    return m;
}

// W = 1 (one drone per env) is HBM-bound at scale: capping it at 80 registers
// (a few dozen bytes of spills to L1) keeps 12 CTAs of 64 threads per SM in
// flight instead of 9, +18% at 1M envs. Swarms of up to 32 keep 96 (10 CTAs of
// 64 threads instead of 8; 131,072 x 8, K = 6, 191 -> 173 us a step, 32,768 x 8
// 62 -> 56), wider ones, whose pair pass is most of the step, what they need
// (64 x 256: 9.5 against 10.0 us). OVERLAP: launched overlapped with the
// stream's previous kernel, for up to STEP_OVERLAP_WAVES waves (65,536 single
// drones 10.3 -> 8.0 us a step, 262,144 28.7 -> 28.3); past them every CTA's
// wait costs more than the launch (1,048,576: 83.2 -> 87.9 us).
constexpr int STEP_OVERLAP_WAVES = 2;
template <int W, int EXT, bool OVERLAP = true, bool ROWS = (W == 1 && !EXT)>
__global__ void __maxnreg__(W == 1 ? 80 : W <= 32 && !EXT ? 96 : 168)
    k_step(const Consts c, const Dev dv, const Tile* __restrict__ tiles, const int* __restrict__ perm, const StepIO io,
           const int observe_only) {
    extern __shared__ float4 sm[];
    const SlotMap m = map_slot(dv, tile_at(dv, tiles, blockIdx.x, blockDim.x), perm, W);
    if (OVERLAP) await_previous();
    Drone s;
    EnvRegs er;
    uint32_t ev = 0;
    if (m.act) {
        load_drone(s, dv.st, dv.D, m.d);
        load_env<EXT>(er, c, dv, m.e);
    }
    const float4 a = (m.act && !observe_only) ? reinterpret_cast<const float4*>(io.act)[m.d]
                                              : make_float4(0.f, 0.f, 0.f, 0.f);
    float gv[GOAL_VALUES];
    GoalCache gc{gv, GOAL_FIXED, 0, -1};
    // single drones: rows of a warp as one block (see RowMap; 150,000 drones 15.6 ->
    // 13.5 us, 300,000 28.9 -> 26.0; from 600,000 on the state's traffic is what
    // counts: 1,048,576 81.0 and 80.5), or stored by the lanes (lane_rows)
    const RowMap rm = ROWS ? map_rows(m.act, m.d, 1, c.obs_dim) : RowMap();
    float* rows = reinterpret_cast<float*>(sm) + (threadIdx.x & ~31) * (c.obs_dim + ROW_PAD);
    step_body<EXT, ROWS>(W, c, dv, s, er, ev, sm, reinterpret_cast<float*>(sm + blockDim.x), m.act, m.lane, m.N,
                         m.sbase, m.e, m.d, a, io.obs, io.rew, io.done, observe_only, gc, rm, rows, io.bulk);
    if (m.act && !observe_only) {
        dv.ev[m.d] = ev;
        store_drone(s, dv.st, dv.D, m.d);
        if (m.lane == 0) store_env<EXT>(er, dv, m.e);
    }
    if (ROWS && rm.lead) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// T steps of one tile with the state in registers. W1: every tile of the
// launch holds single-drone slots (a compile-time width of 1: no pair pass,
// neighbour or staging code).
template <int EXT, bool W1>
__device__ __forceinline__ void rollout_tile(const Consts& c, const Dev& dv, const Tile& tile, const int* __restrict__ perm,
                                             float4* sm, const RolloutIO& io, int t0, int nsteps) {
    const int W = W1 ? 1 : tile.W;
    const SlotMap m = map_slot(dv, tile, perm, W);
    Drone s;
    EnvRegs er;
    uint32_t ev = 0;
    if (m.act) {
        load_drone(s, dv.st, dv.D, m.d);
        load_env<EXT>(er, c, dv, m.e);
    }
    const size_t D = dv.D, E = dv.E;
    const float4* act4 = reinterpret_cast<const float4*>(io.act) + m.d;
    // the commands of step t + 1 are loaded while step t computes, so their
    // HBM latency leaves each step's dependent chain
    float4 a_next = m.act ? *(act4 + (size_t)t0 * D) : make_float4(0.f, 0.f, 0.f, 0.f);
    // the general instances' goal values, after the staging planes
    float* goals = reinterpret_cast<float*>(sm + (W1 ? 0 : 2 * SMEM_PLANES / 4 * blockDim.x));
    GoalCache gc{goals + GOAL_STRIDE * threadIdx.x, GOAL_FIXED, 0, -1};
    const RowMap rm = W1 ? RowMap() : map_rows(m.act, m.d, W, c.obs_dim);
    float* rows = goals + (EXT ? GOAL_STRIDE * blockDim.x : 0) + (threadIdx.x & ~31) * (c.obs_dim + ROW_PAD);
    for (int t = t0; t < t0 + nsteps; ++t) {
        const float4 a = a_next;
        if (m.act && t + 1 < t0 + nsteps) a_next = *(act4 + (size_t)(t + 1) * D);
        float4* sp = sm + ((t - t0) & 1) * (SMEM_PLANES / 4) * blockDim.x;
        step_body<EXT, !W1>(W, c, dv, s, er, ev, sp, reinterpret_cast<float*>(sp + blockDim.x), m.act, m.lane, m.N,
                            m.sbase, m.e, m.d, a, io.obs ? io.obs + (size_t)t * D * c.obs_dim : nullptr,
                            io.rew ? io.rew + (size_t)t * D : nullptr, io.done ? io.done + (size_t)t * E : nullptr, 0,
                            gc, rm, rows, io.bulk);
    }
    if (!W1 && rm.lead) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (m.act) {
        dv.ev[m.d] = ev;
        store_drone(s, dv.st, dv.D, m.d);
        if (m.lane == 0) store_env<EXT>(er, dv, m.e);
    }
}

// Persistent rollout: CTAs take tiles from *counter until none is left; every
// CTA draws one number past the tiles, and the last of those puts the counter
// back to zero for the next launch (a memset before each launch cost a launch
// of its own). Tiles are ordered costliest first. The W1 instances (EXT = 0
// and 2) serve handles whose envs all hold one drone (single_form): for EXT = 0 107
// registers instead of 121 and no untaken swarm code in the step loop (with
// the smooth contacts compiled out of the EXT = 0 instances, batched
// 1,048,576 single-drone envs went from 1.75e10 to 1.90e10 quadrotor-steps/s,
// each change about half of it). Held to 104 registers it fits in 96 without a
// spill, five warps a scheduler instead of four (1,048,576 drones, 32 steps,
// 1687 -> 1632 us, in 32-thread CTAs 1593; at 88 registers 1644). Swarms spill
// below 128 (16,384 x 8, 64 steps: 128 registers 746 us, 112 799, 160 901).
// With smooth contacts the rows' way through shared memory cost single drones
// 8% (34,000 drones, 32 steps: 102 us before the rows went that way, 111 after,
// 96 in this instance, whose lanes store their own; 300,000 drones 579, 589, 532).
template <int EXT, bool W1>
__global__ void __maxnreg__(W1 && !EXT ? 104 : 128)
    k_rollout(const Consts c, const Dev dv, const Tile* __restrict__ tiles, const int n_tiles,
              const int* __restrict__ perm, int* __restrict__ counter, const RolloutIO io, const int t0,
              const int nsteps) {
    extern __shared__ float4 sm[];
    __shared__ int s_next;
    await_previous();
    for (;;) {
        if (threadIdx.x == 0) {
            s_next = atomicAdd(counter, 1);
            if (s_next == n_tiles + (int)gridDim.x - 1) *counter = 0;
        }
        __syncthreads();
        const int ti = s_next;
        __syncthreads();  // everyone has read s_next before thread 0 overwrites it
        if (ti >= n_tiles) {
            launch_next();
            return;
        }
        rollout_tile<EXT, W1>(c, dv, tile_at(dv, tiles, ti, blockDim.x), perm, sm, io, t0, nsteps);
    }
}

// ---------------------------------------------------------------- warp-specialised step
// A CTA of 2P warps steps up to 32P drones: slots of width W <= 32P laid over
// the drone lanes of warps 0 .. P-1 (dynamics), which carry one drone per lane
// through the substeps and the pair pass. Warps P .. 2P-1 (noise) draw the
// motor-noise normals of the first WS_SUB substeps into shared memory ahead of
// the dynamics, then the observation noise while the dynamics run, and finally
// put the observation rows of their drones together in shared memory and send
// them (RowMap). The two sides meet at two CTA barriers: after
// the motor normals (B1) and after the dynamics warps publish the final states
// (B2). This takes the Philox and Box-Muller work off each drone's dependent
// chain. With P = 2 (swarms of 33..64) the dynamics warps also meet at named
// barrier 1 between staging and reading each other's positions, and the noise
// warps at named barrier 2 between writing and reading swap keys.
constexpr int WS_SUB = 4;

// What the two sides exchange, one entry a drone lane, in 8- and 16-byte words
// (a warp's load or store of one is as many instructions as its words). The
// noise side's observation rows follow in dynamic shared memory (ws_smem).
template <int P>
struct WsShared {
    float4 nrm[2][WS_SUB][32 * P];  // motor-noise normals of the four rotors [buffer][substep]
    // the published end of a step (post-collision), [buffer] by step parity:
    float4 px[2][32 * P];           // x, y, z, v_x
    float2 vyz[2][32 * P];          // v_y, v_z
    float4 rw[2][3][32 * P];        // R row-major, w
    float4 gk[2][32 * P];           // goal, number of neighbours (bits)
    NbrList nb[2][32 * P];          // CTA drone lanes of the neighbours
    float4 fh[2][32 * P];           // reward inputs: command f^,
    float4 fp[2][32 * P];           //   previous command,
    float2 pe[2][32 * P];           //   proximity radius, event bits
    float4 sp[32 * P];              // pair-pass staging: positions
    float sv[3][32 * P];            //                    velocities
    uint32_t key[32 * P];           // swap keys
    float gv[32 * P][GOAL_STRIDE];  // goal values of each lane's drone (GoalCache)
};

// Dynamic shared memory of a warp-specialised CTA: the noise side's rows. With
// WsShared it passes the 48 KiB every kernel may have for 64 lanes and K = 8;
// such a kernel asks for the most any shape needs.
inline size_t ws_smem(const Consts& c, int P) { return sizeof(float) * 32 * P * (c.obs_dim + ROW_PAD); }
inline cudaError_t allow_ws_smem(const void* fn, const Consts& c, int P) {
    const size_t fixed = (P == 1 ? sizeof(WsShared<1>) : sizeof(WsShared<2>)) + 64;  // and a few words of the kernel's own
    if (fixed + ws_smem(c, P) <= 48u << 10) return cudaSuccess;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(sizeof(float) * 32 * P * (18 + 6 * QS_MAX_K + ROW_PAD)));
}

// Barrier among the P warps of one side (id 1: dynamics, id 2: noise); one
// warp only needs its own lanes converged.
template <int P>
__device__ __forceinline__ void side_sync(int id) {
    if (P == 1)
        __syncwarp();
    else
        asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(32 * P) : "memory");
}

// Slot geometry of a warp-specialised CTA: drone lane L (0 .. 32P-1) of both
// sides stands for slot-local drone `lane` of slot `slot` (W lanes per slot).
struct WsMap {
    int W, L, slot, lane, e, d0, N, d, sbase;
    bool act;
};

template <int P>
__device__ __forceinline__ WsMap ws_map(const Dev& dv, const Tile& tile, const int* __restrict__ perm) {
    WsMap m;
    m.W = tile.W;
    m.L = threadIdx.x & (32 * P - 1);
    m.slot = m.L / m.W;
    m.lane = m.L - m.slot * m.W;
    const SlotGeo g = slot_geometry(dv, perm, tile, m.slot, m.W, 32 * P);
    m.e = g.e;
    m.d0 = g.d0;
    m.N = g.N;
    m.act = m.lane < m.N;
    m.d = m.d0 + m.lane;
    m.sbase = m.slot * m.W;
    return m;
}

// Noise side: the motor-noise normals of the first WS_SUB substeps of the
// step at Philox counter `tick`, into shared-memory buffer nb.
template <int P>
__device__ __forceinline__ void ws_motor_normals(const Consts& c, WsShared<P>& sh, const WsMap& m, uint32_t tick,
                                                 int nb) {
    if (!m.act || !(c.flags & QS_F_MOTOR_NOISE)) return;
    const int nahead = min(c.substeps, WS_SUB);
    for (int sub = 0; sub < nahead; ++sub) {
        float n[4];
        motor_normals(c, tick, m.d, sub, n);
        sh.nrm[nb][sub][m.L] = make_float4(n[0], n[1], n[2], n[3]);
    }
}

// The goal of the lane's drone at control step tau under the scenario record in
// buffer sel (Sec. III-D scenarios); gl holds the env's single goal on entry.
// Every thread of the side (side_sync id) calls it.
template <int P>
__device__ __forceinline__ void ws_goal(const Consts& c, const Dev& dv, WsShared<P>& sh, const WsMap& m, int sel, int tau,
                                        GoalCache& gc, float gl[3], int id) {
    const bool hit = goal_cached(gc, tau);  // the same for every lane of an env
    bool swp = false;
    uint32_t myk = 0;
    if (m.W > 1) {
        if (m.act && !hit && swap_active(dv, sel, m.e, tau)) {
            swp = true;
            myk = swap_key(c, scn_seed(dv, sel, m.e), m.lane);
            sh.key[m.L] = myk;
        }
        side_sync<P>(id);
    }
    if (!m.act) return;
    if (!hit)
        goal_fill(gc, c, dv, sel, m.e, m.lane, m.N, tau, swp ? swap_rank(sh.key, m.sbase, m.N, m.lane, myk) : m.lane, gl);
    goal_at(gc, c, tau, gl);
}

// Dynamics side: one control step of the lane's drone with command a and the
// motor normals of buffer nb. Meets the noise side at B1 (motor normals ready)
// and B2 (post-step state, goal and neighbours published for the observation
// rows), then writes the knn record, reward and done and ends the step. Every
// thread of the dynamics warps calls it.
template <int EXT, int P, bool DEFER, bool W1 = false>
__device__ __forceinline__ void ws_dynamics_step(const Consts& c, const Dev& dv, WsShared<P>& sh, const WsMap& m,
                                                 Drone& s, EnvRegs& er, uint32_t& ev_out, const float4 a, const int nb,
                                                 float* __restrict__ rew, uint8_t* __restrict__ done, GoalCache& gc,
                                                 const bool b1 = true) {
    const int b = nb;  // the step's buffers: its motor normals and its published end
    const int W = W1 ? 1 : m.W, L = m.L, lane = m.lane, N = W1 ? 1 : m.N, e = m.e, d = m.d, sbase = m.sbase;
    const bool act = m.act;
    const int K = c.K;
    const int nahead = min(c.substeps, WS_SUB);
    const bool mnoise = (c.flags & QS_F_MOTOR_NOISE) != 0;
    const bool dw = EXT && (c.flags & QS_F_DOWNWASH) != 0;  // EXT = 0: no downwash or scenario code
    float fh[4] = {0.f, 0.f, 0.f, 0.f}, u[4] = {0.f, 0.f, 0.f, 0.f};
    uint32_t ev = 0;
    if (act) {
        fh[0] = command(c, a.x);
        fh[1] = command(c, a.y);
        fh[2] = command(c, a.z);
        fh[3] = command(c, a.w);
        u[0] = sqrt_approx(fh[0]);
        u[1] = sqrt_approx(fh[1]);
        u[2] = sqrt_approx(fh[2]);
        u[3] = sqrt_approx(fh[3]);
    }
    if (b1) __syncthreads();  // B1: motor normals ready (the rollout's later steps: drawn before the last B2)
    // smooth contacts of a swarm (general instance): the pair penalty from the
    // positions at each substep's start, staged like the pair pass
    const bool spair = EXT == 2 && W > 1;
    if (spair) {
        for (int sub = 0; sub < c.substeps; ++sub) {
            float pacc[3] = {0.f, 0.f, 0.f};
            if (act) sh.sp[L] = make_float4(s.x[0], s.x[1], s.x[2], 0.f);
            side_sync<P>(1);
            if (act && N > 1) pair_acc(c, s.x, sh.sp, sbase, lane, N, er.p.arm, pacc);
            side_sync<P>(1);
            if (act) {
                if (mnoise && sub < nahead) {
                    const float4 q = sh.nrm[nb][sub][L];
                    const float n[4] = {q.x, q.y, q.z, q.w};
                    ev |= substep<false, EXT == 2 ? 1 : 0>(s, er.p, c, u, er.tick, d, sub, pacc, n);
                } else {
                    ev |= substep<false, EXT == 2 ? 1 : 0>(s, er.p, c, u, er.tick, d, sub, pacc);
                }
            }
        }
    } else if (act) {
        const float zero3[3] = {0.f, 0.f, 0.f};
        for (int sub = 0; sub < c.substeps; ++sub) {
            if (mnoise && sub < nahead) {
                const float4 q = sh.nrm[nb][sub][L];
                const float n[4] = {q.x, q.y, q.z, q.w};
                ev |= substep<false, EXT == 2 ? 1 : 0>(s, er.p, c, u, er.tick, d, sub, zero3, n);
            } else {
                ev |= substep<false, EXT == 2 ? 1 : 0>(s, er.p, c, u, er.tick, d, sub, zero3);
            }
        }
    }
    const int keff = min(K, N - 1);
    NbrList nbrs = 0;
    if (W > 1) {
        if (act) {
            sh.sp[L] = make_float4(s.x[0], s.x[1], s.x[2], 0.f);
            sh.sv[0][L] = s.v[0];
            sh.sv[1][L] = s.v[1];
            sh.sv[2][L] = s.v[2];
        }
        side_sync<P>(1);
        float dvs[3] = {0.f, 0.f, 0.f};
        bool responded = false, dw_hit = false;
        float dw_az = 0.f;
        if (act && N > 1) {
            const bool coll = (c.flags & QS_F_COLLISIONS) && EXT != 2;
            const bool flag_coll = (c.flags & QS_F_COLLISIONS) != 0;
            responded = pair_scan<(EXT > 0)>(c, s, er.p.thr, lane, N, sbase, sh.sp, &sh.sv[0][0], 32 * P, keff, coll,
                                             flag_coll, ev, nbrs, dvs, dw, dw_az, dw_hit);
        }
        if (responded) apply_response(c, s, er.tick, d, dvs);
        if (dw && dw_hit) apply_downwash(c, s, er.tick, d, dw_az);
    }
    // the drone's goal at the end of the step; in the rollout the noise side
    // evaluates it
    float gl[3] = {er.g0, er.g1, er.g2};
    if (EXT && !DEFER && (c.scn_mask & ~1u)) ws_goal<P>(c, dv, sh, m, er.sel, er.ep + 1, gc, gl, 1);
    if (act) {  // publish the observed state (post-collision) for the noise side
        sh.px[b][L] = make_float4(s.x[0], s.x[1], s.x[2], s.v[0]);
        sh.vyz[b][L] = make_float2(s.v[1], s.v[2]);
        sh.rw[b][0][L] = make_float4(s.R[0], s.R[1], s.R[2], s.R[3]);
        sh.rw[b][1][L] = make_float4(s.R[4], s.R[5], s.R[6], s.R[7]);
        sh.rw[b][2][L] = make_float4(s.R[8], s.w[0], s.w[1], s.w[2]);
        sh.gk[b][L] = make_float4(gl[0], gl[1], gl[2], __int_as_float(W > 1 ? keff : 0));
        if (!W1) sh.nb[b][L] = nbrs + (NbrList)sbase * 0x0101010101010101ull;  // (fields past keff are not read)
        if (DEFER) {  // the noise side computes the reward from these
            sh.fh[b][L] = make_float4(fh[0], fh[1], fh[2], fh[3]);
            sh.fp[b][L] = make_float4(s.fp[0], s.fp[1], s.fp[2], s.fp[3]);
            sh.pe[b][L] = make_float2(er.p.prox, __uint_as_float(ev));
        }
    }
    __syncthreads();  // B2
    if (!act) return;
    if ((c.flags & QS_F_RECORD_KNN) && dv.knn) {
#pragma unroll
        for (int k = 0; k < QS_MAX_K; ++k)
            if (k < K) dv.knn[(size_t)k * dv.D + d] = (W > 1 && k < keff) ? (int16_t)nbr_at(nbrs, k) : (int16_t)-1;
    }
    if (!DEFER && rew)
        rew[d] = compute_reward(c, s, er.p.prox, gl, fh, ev, W > 1 ? keff : 0, [&](int k) {
            const float4 q = sh.sp[sbase + nbr_at(nbrs, k)];
            return make_float3(q.x, q.y, q.z);
        });
    end_step<EXT>(c, dv, s, er, fh, lane, e, d, done);
    if (EXT && !DEFER && er.ep == 0) gc.until = -1;  // an auto-reset drew a new record
    ev_out = ev;
}

// Noise side: finishes the step published in buffer b. The observation rows
// (with sensor noise ex, evv, ew) go to obs, and with rew the reward (the same
// compute_reward as the dynamics side) of the lane's drone; goal(gl) replaces
// the published single goal where scenarios are on; without BULK the rows are
// always stored by the lanes, at once (one step: nothing to wait for). Every
// thread of the side calls it. The rows took two thirds of the noise side's time, word by word:
// 3,800 of 7,200 cycles a step for swarms of 8 at K = 6 (two CTAs an SM).
template <int P, bool BULK = true, class Goal>
__device__ __forceinline__ void ws_finish(const Consts& c, WsShared<P>& sh, const WsMap& m, const RowMap& rm, float* rows,
                                          int b, float* __restrict__ obs, float* __restrict__ rew, bool bulk,
                                          const float ex[3], const float evv[3], const float ew[3], const Goal& goal) {
    const int L = m.L, od = c.obs_dim, K = c.K;
    Drone s;
    float gl[3] = {0.f, 0.f, 0.f};
    int keff = 0;
    NbrList nb = 0;
    if (m.act) {
        const float4 a = sh.px[b][L], r0 = sh.rw[b][0][L], r1 = sh.rw[b][1][L], r2 = sh.rw[b][2][L], g = sh.gk[b][L];
        const float2 v = sh.vyz[b][L];
        nb = sh.nb[b][L];
        s.x[0] = a.x; s.x[1] = a.y; s.x[2] = a.z;
        s.v[0] = a.w; s.v[1] = v.x; s.v[2] = v.y;
        s.R[0] = r0.x; s.R[1] = r0.y; s.R[2] = r0.z; s.R[3] = r0.w; s.R[4] = r1.x; s.R[5] = r1.y; s.R[6] = r1.z;
        s.R[7] = r1.w; s.R[8] = r2.x;
        s.w[0] = r2.y; s.w[1] = r2.z; s.w[2] = r2.w;
        gl[0] = g.x; gl[1] = g.y; gl[2] = g.z;
        keff = __float_as_int(g.w);
    }
    goal(gl);
    if (obs) {
        if (BULK) rows_free(rm);
        if (m.act) {
            float2* o2 = reinterpret_cast<float2*>(rows + rm.off + row_shift(rm, obs, od) + rm.rank * od);
            o2[0] = make_float2(s.x[0] - gl[0] + ex[0], s.x[1] - gl[1] + ex[1]);
            o2[1] = make_float2(s.x[2] - gl[2] + ex[2], s.v[0] + evv[0]);
            o2[2] = make_float2(s.v[1] + evv[1], s.v[2] + evv[2]);
            o2[3] = make_float2(s.R[0], s.R[1]);
            o2[4] = make_float2(s.R[2], s.R[3]);
            o2[5] = make_float2(s.R[4], s.R[5]);
            o2[6] = make_float2(s.R[6], s.R[7]);
            o2[7] = make_float2(s.R[8], s.w[0] + ew[0]);
            o2[8] = make_float2(s.w[1] + ew[1], s.w[2] + ew[2]);
#pragma unroll
            for (int k = 0; k < QS_MAX_K; ++k) {
                if (k >= K) break;
                float2* on = o2 + 9 + 3 * k;
                if (k < keff) {
                    const int j = nbr_at(nb, k);
                    const float4 q = sh.px[b][j];
                    const float2 v = sh.vyz[b][j];
                    on[0] = make_float2(q.x - s.x[0], q.y - s.x[1]);
                    on[1] = make_float2(q.z - s.x[2], q.w - s.v[0]);
                    on[2] = make_float2(v.x - s.v[1], v.y - s.v[2]);
                } else {
                    on[0] = make_float2(0.f, 0.f);
                    on[1] = make_float2(0.f, 0.f);
                    on[2] = make_float2(0.f, 0.f);
                }
            }
        }
        send_rows(rm, rows, obs, od, BULK && bulk);
    }
    if (rew && m.act) {
        const float4 f = sh.fh[b][L], p = sh.fp[b][L];
        const float2 pe = sh.pe[b][L];
        const float fh[4] = {f.x, f.y, f.z, f.w};
        s.fp[0] = p.x; s.fp[1] = p.y; s.fp[2] = p.z; s.fp[3] = p.w;
        rew[m.d] = compute_reward(c, s, pe.x, gl, fh, __float_as_uint(pe.y), keff, [&](int k) {
            const float4 q = sh.px[b][nbr_at(nb, k)];
            return make_float3(q.x, q.y, q.z);
        });
    }
}

// The noise warp's rows in dynamic shared memory.
__device__ __forceinline__ float* ws_rows(const Consts& c, int L) {
    extern __shared__ float4 sm[];
    return reinterpret_cast<float*>(sm) + (L & ~31) * (c.obs_dim + ROW_PAD);
}

// W1: every slot of the launch holds one drone (no pair pass: a smaller kernel to
// fetch when its instructions are cold). 8192 drones with L2 flushed before each
// step, where the fetch counts (means of processes, each a mix of modes 0.3 - 1
// us apart; sources that differ elsewhere in the library give 8.7 - 10.0 for the
// same kernel): 9.75 us without W1, 9.05 - 9.25 with it, 8.7 - 9.2 with the rows
// mapped ahead of B2 and no bulk-copy code in the step. Back to back in a stream
// 4.0 -> 3.8 (4.4 before launches overlapped).
template <int EXT, bool W1 = false>
__global__ void __launch_bounds__(64) k_step_ws(const Consts c, const Dev dv, const Tile* __restrict__ tiles,
                                                const int* __restrict__ perm, const StepIO io) {
    __shared__ WsShared<1> sh;
    const Tile tile = tile_at(dv, tiles, blockIdx.x, 32);
    const WsMap m = ws_map<1>(dv, tile, perm);
    await_previous();
    if (threadIdx.x >= 32) {
        // ---------------- noise warp
        const uint32_t tick = m.act ? dv.tick[m.e] : 0u;  // warp 0 writes it only after B2
        ws_motor_normals<1>(c, sh, m, tick, 0);
        __syncthreads();  // B1
        float ex[3] = {0.f, 0.f, 0.f}, evv[3] = {0.f, 0.f, 0.f}, ew[3] = {0.f, 0.f, 0.f};
        if (m.act && io.obs && (c.flags & QS_F_OBS_NOISE)) obs_noise(c, tick, m.d, 0u, ex, evv, ew);
        const RowMap rm = map_rows(m.act, m.d, m.W, c.obs_dim);  // while the dynamics run
        __syncthreads();  // B2
        launch_next();
        if (io.obs)
            ws_finish<1, false>(c, sh, m, rm, ws_rows(c, m.L), 0, io.obs, nullptr, false, ex, evv, ew, [](float*) {});
        return;
    }
    // ---------------- dynamics warp
    Drone s;
    EnvRegs er;
    uint32_t ev = 0;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (m.act) {
        load_drone(s, dv.st, dv.D, m.d);
        load_env<EXT>(er, c, dv, m.e);
        a = reinterpret_cast<const float4*>(io.act)[m.d];
    }
    GoalCache gc{sh.gv[m.L], GOAL_FIXED, 0, -1};
    ws_dynamics_step<EXT, 1, false, W1>(c, dv, sh, m, s, er, ev, a, 0, io.rew, io.done, gc);
    if (!m.act) return;
    dv.ev[m.d] = ev;
    store_drone(s, dv.st, dv.D, m.d);
    if (m.lane == 0) store_env<EXT>(er, dv, m.e);
}

// Persistent warp-specialised rollout for latency-bound handles (every swarm
// class at most 32P wide): one CTA per tile of 32P drone lanes runs steps
// t0 .. t0 + nsteps - 1 with the drones in the dynamics warps' registers.
// While the dynamics side integrates step t, the noise side draws step t's
// sensor noise and step t + 1's motor normals (double-buffered) and finishes
// step t - 1's rewards and observation rows. For single-drone slots the two
// sides meet once per step, at B2 (and at B1 before the first step): step
// t + 1's normals are drawn before B2 of step t, so the noise side's work for
// a step overlaps the dynamics side's end of the previous one (plain 8192 /
// 4864 / 2432 envs: +2% / +5% / +7%); swarm slots meet at B1 and B2 of every
// step (without B1, 3.56e9 -> 3.50e9 quadrotor-steps/s for 2048 x 8).
template <int EXT, int P>
__global__ void __launch_bounds__(64 * P, (P == 1 ? 6 : 1))
    k_rollout_ws(const Consts c, const Dev dv, const Tile* __restrict__ tiles, const int* __restrict__ perm,
                 const RolloutIO io, const int t0, const int nsteps) {
    __shared__ WsShared<P> sh;
    const Tile tile = tile_at(dv, tiles, blockIdx.x, 32 * P);
    const WsMap m = ws_map<P>(dv, tile, perm);
    const size_t D = dv.D, E = dv.E;
    await_previous();
    if (threadIdx.x >= 32 * P) {
        // ---------------- noise side; the env's Philox counter advances by one per step
        // Step t's observation rows and reward are finished during step t + 1's
        // dynamics, from the end of step t published in buffer t & 1.
        const uint32_t tick0 = m.act ? dv.tick[m.e] : 0u;  // the dynamics side writes it after the last step
        ws_motor_normals<P>(c, sh, m, tick0, 0);
        float px[3] = {0.f, 0.f, 0.f}, pv[3] = {0.f, 0.f, 0.f}, pw[3] = {0.f, 0.f, 0.f};  // step t-1's sensor noise
        // scenario goals: the episode step and record buffer of the step being
        // finished, advanced as the dynamics side advances them. A record is
        // drawn after B2 of the step that ends its predecessor's episode, into
        // the other buffer, and first read after the next B2.
        const bool scn = EXT && (c.scn_mask & ~1u) != 0;
        int ep = scn && m.act ? dv.ep[m.e] : 0, sel = scn && m.act ? dv.scn_sel[m.e] : 0;
        GoalCache gc{sh.gv[m.L], GOAL_FIXED, 0, -1};
        const RowMap rm = map_rows(m.act, m.d, m.W, c.obs_dim);
        float* rows = ws_rows(c, m.L);
        const auto finish = [&](int t) {
            ws_finish<P>(c, sh, m, rm, rows, t & 1, io.obs ? io.obs + (size_t)(t0 + t) * D * c.obs_dim : nullptr,
                         io.rew ? io.rew + (size_t)(t0 + t) * D : nullptr, io.bulk, px, pv, pw, [&](float* gl) {
                if (!scn) return;
                ws_goal<P>(c, dv, sh, m, sel, ep + 1, gc, gl, 2);
                ep = ep + 1;
                if (ep >= c.episode_steps && (c.flags & QS_F_AUTO_RESET)) {
                    ep = 0;
                    sel ^= 1;
                    gc.until = -1;
                }
            });
        };
        for (int t = 0; t < nsteps; ++t) {
            // buffer t & 1 holds step t's normals, drawn before B2 of step t - 1:
            // B1 is needed before the first step only; swarm slots (whose
            // dynamics side takes the longer step) keep it every step, measured
            // faster there
            if (t == 0 || m.W > 1) __syncthreads();  // B1
            const uint32_t tick = tick0 + (uint32_t)t;
            float ex[3] = {0.f, 0.f, 0.f}, evv[3] = {0.f, 0.f, 0.f}, ew[3] = {0.f, 0.f, 0.f};
            if (m.act && io.obs && (c.flags & QS_F_OBS_NOISE)) obs_noise(c, tick, m.d, 0u, ex, evv, ew);
            // the other buffer was last read by the dynamics side before B2 of step t - 1
            if (t + 1 < nsteps) ws_motor_normals<P>(c, sh, m, tick + 1, (t + 1) & 1);
            if (t > 0) finish(t - 1);
            for (int k = 0; k < 3; ++k) {
                px[k] = ex[k];
                pv[k] = evv[k];
                pw[k] = ew[k];
            }
            __syncthreads();  // B2 of step t
        }
        launch_next();
        if (nsteps > 0) finish(nsteps - 1);  // after the last B2
        if (rm.lead) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        return;
    }
    // ---------------- dynamics side
    Drone s;
    EnvRegs er;
    uint32_t ev = 0;
    if (m.act) {
        load_drone(s, dv.st, dv.D, m.d);
        load_env<EXT>(er, c, dv, m.e);
    }
    const float4* act4 = reinterpret_cast<const float4*>(io.act) + m.d;
    float4 a_next = m.act ? *(act4 + (size_t)t0 * D) : make_float4(0.f, 0.f, 0.f, 0.f);
    GoalCache gc{sh.gv[m.L], GOAL_FIXED, 0, -1};
    for (int t = 0; t < nsteps; ++t) {
        const float4 a = a_next;
        if (m.act && t + 1 < nsteps) a_next = *(act4 + (size_t)(t0 + t + 1) * D);
        ws_dynamics_step<EXT, P, true>(c, dv, sh, m, s, er, ev, a, t & 1,
                                 io.rew ? io.rew + (size_t)(t0 + t) * D : nullptr,
                                 io.done ? io.done + (size_t)(t0 + t) * E : nullptr, gc, t == 0 || m.W > 1);
    }
    if (!m.act) return;
    dv.ev[m.d] = ev;
    store_drone(s, dv.st, dv.D, m.d);
    if (m.lane == 0) store_env<EXT>(er, dv, m.e);
}

// ---------------------------------------------------------------- resident step server
// A synchronous host loop (post commands, wait, read the outputs) pays a
// launch and a completion round trip per step on the per-call path. The
// server is one cooperative launch of the warp-specialised CTAs that keeps the
// drones in the dynamics warps' registers and steps them each time the host
// posts a step, with commands read from and outputs written to page-locked
// host memory in place. Handshake words in page-locked host memory: `go`
// holds in its low half the steps the host has posted (SERVE_STOP: end the
// launch; SERVE_IDLE: the server retired after waiting too long) and in its
// high half the command slot of the last posted step; `fin` counts the
// steps completed, written by the last CTA to finish each step (found with a
// counter in device memory). Only CTA 0 polls `go` over the host link; it
// relays what it reads through a word in device memory that the other CTAs
// poll (one reader of the host's line instead of one per CTA). Measured on
// GB300 at 8192 single-drone envs: one system-scope fence per CTA instead of
// one per thread, and the relay instead of every CTA polling the host, took a
// posted step from 15.8 to 11.1 us, and an acquire-release count instead of
// a second system-scope fence in the last CTA a synchronous host loop from
// 11.5 to 11.0 us per step; a completion byte
// per CTA polled by the host instead of the counter and fin was slower (11.7
// us: 64 CTAs write each line the host re-reads), and so were several reads
// of go (or of the relay) kept in flight at once instead of one (7.2 -> 11.2
// us for a one-CTA server: the reads keep taking the line from the host
// while it posts).
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned long long ld_acquire_sys(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.sys.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_sys(int* p, int v) {
    asm volatile("st.release.sys.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ unsigned long long ld_acquire_gpu(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long atom_add_acq_rel_gpu(unsigned long long* p, unsigned long long v) {
    unsigned long long old;
    asm volatile("atom.acq_rel.gpu.global.add.u64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v) : "memory");
    return old;
}

__device__ __forceinline__ void st_release_gpu(unsigned long long* p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// The step count (or stop code) and the command slot of a go word.
__device__ __forceinline__ int go_steps(unsigned long long v) { return (int)(unsigned int)(v & 0xffffffffull); }
__device__ __forceinline__ int go_slot(unsigned long long v) { return (int)(unsigned int)(v >> 32); }

// Thread 0 of CTAs other than 0: the relayed value once it leaves `posted`.
// CTA 0 relays every value it acts on, so this wait ends once CTA 0's does;
// its bound (4 idle_ns + 1 s, well past CTA 0's) only guards against a CTA 0
// that stopped answering, after which the CTA stops as if the server had
// retired.
__device__ __forceinline__ unsigned long long serve_follow(const unsigned long long* relay, int posted, long long idle_ns) {
    const unsigned long long t0 = global_ns(), limit = 4ull * (unsigned long long)idle_ns + 1000000000ull;
    for (;;) {
        const unsigned long long v = ld_acquire_gpu(relay);
        if (go_steps(v) != posted) return v;
        if (global_ns() - t0 > limit) return (unsigned long long)(unsigned int)SERVE_IDLE;
        __nanosleep(64);
    }
}

// Thread 0 of CTA 0: the value of `go` once its step count leaves `posted`
// (the steps already run). After idle_ns without an answer the server retires
// by swapping go from the value it last read to SERVE_IDLE; the swap fails
// only when the host posted a step (or stopped) first, so every CTA of the
// launch sees one outcome.
__device__ __forceinline__ unsigned long long serve_wait(unsigned long long* go, int posted, long long idle_ns) {
    const unsigned long long t0 = global_ns();
    for (;;) {
        const unsigned long long v = ld_acquire_sys(go);
        if (go_steps(v) != posted) return v;
        if (global_ns() - t0 > (unsigned long long)idle_ns) {
            const unsigned long long idle = (v & ~0xffffffffull) | (unsigned long long)(unsigned int)SERVE_IDLE;
            const unsigned long long old = atomicCAS_system(go, v, idle);
            __threadfence_system();
            return old == v ? idle : old;
        }
        __nanosleep(32);
    }
}

// Step k of the launch (global step k0 + k): B0 (the host posted it; the
// noise side has drawn its motor normals into buffer k & 1), the per-call
// warp-specialised step (B1, B2) with the observation rows of step k stored
// by the noise side after B2 and the next step's normals drawn after them,
// then B3, after which thread 0 fences the CTA's host writes at system scope
// and counts the CTA done; the last CTA publishes fin = k0 + k + 1.
// The launch bound is how many CTAs an SM holds, and with it the largest handle
// qs_serve_begin accepts: a scheduler takes three warps of up to 168 registers.
// Left to itself the 64-lane common instance takes 193, two CTAs an SM; held to
// three it fits in 144 without a spill (the general ones take 208 and 226).
template <int EXT, int P>
__global__ void __launch_bounds__(64 * P, (P == 1 ? 6 : EXT == 0 ? 3 : 2))
    k_serve(const Consts c, const Dev dv, const Tile* __restrict__ tiles, const int* __restrict__ perm, const ServeIO io,
            const int k0) {
    __shared__ WsShared<P> sh;
    __shared__ unsigned long long s_go;
    const Tile tile = tile_at(dv, tiles, blockIdx.x, 32 * P);
    const WsMap m = ws_map<P>(dv, tile, perm);
    const bool noise = threadIdx.x >= 32 * P;
    const uint32_t tick0 = (noise && m.act) ? dv.tick[m.e] : 0u;  // the dynamics side writes it back at the end
    Drone s;
    EnvRegs er;
    uint32_t ev = 0;
    GoalCache gc{sh.gv[m.L], GOAL_FIXED, 0, -1};
    if (!noise && m.act) {
        load_drone(s, dv.st, dv.D, m.d);
        load_env<EXT>(er, c, dv, m.e);
    }
    const RowMap rm = map_rows(m.act, m.d, m.W, c.obs_dim);
    if (noise) ws_motor_normals<P>(c, sh, m, tick0, 0);
    for (int k = 0;; ++k) {
        if (threadIdx.x == 0) {
            if (blockIdx.x == 0) {
                s_go = serve_wait(io.go, k0 + k, io.idle_ns);
                st_release_gpu(io.relay, s_go);
            } else {
                s_go = serve_follow(io.relay, k0 + k, io.idle_ns);
            }
        }
        __syncthreads();  // B0
        const unsigned long long g = s_go;
        // SERVE_STOP, SERVE_IDLE, or a slot the host never checked
        if (go_steps(g) != k0 + k + 1 || go_slot(g) >= io.n_slots) break;
        const int b = k & 1;
        if (noise) {
            const uint32_t tick = tick0 + (uint32_t)k;
            __syncthreads();  // B1
            float ex[3] = {0.f, 0.f, 0.f}, evv[3] = {0.f, 0.f, 0.f}, ew[3] = {0.f, 0.f, 0.f};
            if (m.act && io.obs && (c.flags & QS_F_OBS_NOISE)) obs_noise(c, tick, m.d, 0u, ex, evv, ew);
            __syncthreads();  // B2
            if (io.obs)
                ws_finish<P>(c, sh, m, rm, ws_rows(c, m.L), b, io.obs, nullptr, false, ex, evv, ew, [](float*) {});
            ws_motor_normals<P>(c, sh, m, tick + 1, b ^ 1);
        } else {
            // the host's commands of this step: fetched again, never from a cached line
            const float4* act4 = reinterpret_cast<const float4*>(io.act + (size_t)go_slot(g) * 4 * dv.D) + m.d;
            const float4 a = m.act ? __ldcv(act4) : make_float4(0.f, 0.f, 0.f, 0.f);
            ws_dynamics_step<EXT, P, false>(c, dv, sh, m, s, er, ev, a, b, io.rew, io.done, gc);
        }
        __syncthreads();  // B3
        if (threadIdx.x == 0) {
            // the CTA's host writes of the step (ordered before it by B3) performed
            // at system scope before its count; the count's acquire side orders
            // every CTA's count before the last one's release of fin
            __threadfence_system();
            const unsigned long long n = atom_add_acq_rel_gpu(io.count, 1ull) + 1ull;
            if (n == (unsigned long long)gridDim.x * (unsigned long long)(k + 1)) st_release_sys(io.fin, k0 + k + 1);
        }
    }
    if (noise || !m.act) return;
    dv.ev[m.d] = ev;
    store_drone(s, dv.st, dv.D, m.d);
    if (m.lane == 0) store_env<EXT>(er, dv, m.e);
}

// The instance of a warp-specialised kernel for a handle (ext: extended()).
template <int P>
const void* serve_kernel(int ext) {
    return ext == 2 ? (const void*)k_serve<2, P> : ext == 1 ? (const void*)k_serve<1, P> : (const void*)k_serve<0, P>;
}
template <int P>
auto rollout_ws_kernel(int ext) {
    return ext == 2 ? k_rollout_ws<2, P> : ext == 1 ? k_rollout_ws<1, P> : k_rollout_ws<0, P>;
}

cudaError_t launch_serve(const Consts& c, const Dev& dv, const Tile* tiles, int n_tiles, int P, const int* perm,
                         const ServeIO& io, int k0, cudaStream_t st) {
    const int ext = extended(c);
    const void* fn = P == 1 ? serve_kernel<1>(ext) : serve_kernel<2>(ext);
    if (P != 1 && P != 2) return cudaErrorInvalidValue;
    Consts cc = c;
    Dev dd = dv;
    ServeIO ii = io;
    const Tile* tt = tiles;
    const int* pp = perm;
    int kk = k0;
    void* args[] = {&cc, &dd, &tt, &pp, &ii, &kk};
    const cudaError_t e = allow_ws_smem(fn, c, P);
    if (e != cudaSuccess) return e;
    return cudaLaunchCooperativeKernel(fn, dim3(n_tiles), dim3(64 * P), args, ws_smem(c, P), st);
}

int serve_resident_ctas(const Consts& c, int P) {
    int dev = 0, n_sm = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const int ext = extended(c);
    const void* fn = P == 1 ? serve_kernel<1>(ext) : serve_kernel<2>(ext);
    if (allow_ws_smem(fn, c, P) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, 64 * P, ws_smem(c, P)) != cudaSuccess)
        return 0;
    return occ * n_sm;
}

int rollout_ws_resident_ctas(const Consts& c, int P) {
    int dev = 0, n_sm = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const int ext = extended(c);
    const void* fn = P == 1 ? (const void*)rollout_ws_kernel<1>(ext) : (const void*)rollout_ws_kernel<2>(ext);
    if (allow_ws_smem(fn, c, P) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, 64 * P, ws_smem(c, P)) != cudaSuccess)
        return 0;
    return occ * n_sm;
}

// A kernel whose shared memory passes the 48 KiB every kernel may have (large
// CTAs with many neighbours) asks for the most any shape needs, so that no
// handle's call lowers another's.
cudaError_t allow_smem(const void* fn, size_t smem) {
    if (smem <= 48u << 10) return cudaSuccess;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, STEP_SMEM_MAX);
}

// CTAs of `block` threads of the single-drone step (80 registers) in a wave.
int step_wave(int block) {
    int dev = 0, n_sm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    return n_sm * (768 / block);
}

// Whether the lanes of the large single-drone step store their own rows. Held to
// 80 registers, the form that sends them spills twice the bytes, which its
// substeps load again: it pays while the rows weigh more than the substeps.
// Measured, us a step of 1,048,576 drones at K = 0, stored by the lane against
// sent: 2 substeps 81.0 and 80.5 (300,000 drones 28.9 and 25.9), 3 90.4 and 92.2,
// 4 103.0 and 107.0, 6 139.5 and 143.5; 600,000 drones at K = 1: 4 substeps 67.1
// and 67.4, 6 86.4 and 89.0.
bool lane_rows(const Consts& c) { return c.substeps > 2 + 2 * c.K; }

template <int EXT>
cudaError_t launch_k_step(const Consts& c, const Dev& dv, const ClassPlan& cp, const Tile* t, const int* perm,
                          const StepIO& io, int observe_only, size_t smem, cudaStream_t st) {
    const auto k = [&](auto kernel) {
        return launch_overlapped(kernel, cp.n_tiles, cp.block, smem, st, c, dv, t, perm, io, observe_only);
    };
    switch (cp.W) {
        case 1: {
            cudaError_t e = allow_smem((const void*)k_step<1, EXT>, smem);
            if (e == cudaSuccess) e = allow_smem((const void*)k_step<1, EXT, false>, smem);
            if (e != cudaSuccess) return e;
            if (cp.n_tiles <= STEP_OVERLAP_WAVES * step_wave(cp.block)) return k(k_step<1, EXT>);
            if (lane_rows(c))
                k_step<1, EXT, false, false><<<cp.n_tiles, cp.block, 0, st>>>(c, dv, t, perm, io, observe_only);
            else
                k_step<1, EXT, false><<<cp.n_tiles, cp.block, smem, st>>>(c, dv, t, perm, io, observe_only);
            return cudaGetLastError();
        }
        case 2: return k(k_step<2, EXT>);
        case 4: return k(k_step<4, EXT>);
        case 8: return k(k_step<8, EXT>);
        case 16: return k(k_step<16, EXT>);
        case 32: return k(k_step<32, EXT>);
        case 64: return k(k_step<64, EXT>);
        case 128: return k(k_step<128, EXT>);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_step(const Consts& c, const Dev& dv, const ClassPlan& cp, const Tile* tiles, const int* perm,
                        const StepIO& io, int observe_only, cudaStream_t st) {
    if (cp.n_tiles == 0) return cudaSuccess;
    const int ext = extended(c);
    if (cp.ws && !observe_only) {
        const auto k = ext == 2 ? k_step_ws<2> : ext == 1 ? k_step_ws<1> : cp.W == 1 ? k_step_ws<0, true> : k_step_ws<0>;
        return launch_overlapped(k, cp.n_tiles, 64, io.obs ? ws_smem(c, 1) : 0, st, c, dv, tiles + cp.tile_off, perm, io);
    }
    const size_t smem = cp.W > 1 ? sizeof(float) * SMEM_PLANES * cp.block
                        : ext     ? 0
                                  : sizeof(float) * cp.block * (c.obs_dim + ROW_PAD);
    const Tile* t = tiles + cp.tile_off;
    return ext == 2   ? launch_k_step<2>(c, dv, cp, t, perm, io, observe_only, smem, st)
           : ext == 1 ? launch_k_step<1>(c, dv, cp, t, perm, io, observe_only, smem, st)
                      : launch_k_step<0>(c, dv, cp, t, perm, io, observe_only, smem, st);
}

// Whether a handle's rollout takes the single-drone form of its instance (the
// common and the smooth one have it): every env holds one drone, and the rows'
// neighbour fields are few enough that a lane had better store its own row than
// send it through shared memory, whose addressing costs a step more but whose
// stores do not scatter. Measured with one drone an env, us for 12 steps, stored
// by the lane against sent: K = 3 24,000 drones 40 and 43, 32,000 48 and 43; K = 6
// 12,000 35 and 39, 16,384 39 and 39, 20,000 49 and 43, 100,000 270 and 96; K = 8
// 12,000 37 and 39, 16,384 45 and 40; smooth K = 6 16,384 38 and 43, 20,000 51 and
// 48. With K = 1 the lane's stores win at every size (1,048,576 drones, 4 steps 218
// and 226).
bool single_form(const Consts& c, int D, bool single) {
    if (!single || extended(c) == 1) return false;
    if (c.K < 2) return true;
    int dev = 0, n_sm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    return (long)D * c.K <= 640L * n_sm;
}

// The k_rollout instance for a handle of D drones.
auto rollout_kernel(const Consts& c, int D, bool single) {
    const bool form = single_form(c, D, single);
    switch (extended(c)) {
        case 2: return form ? k_rollout<2, true> : k_rollout<2, false>;
        case 1: return k_rollout<1, false>;
        default: return form ? k_rollout<0, true> : k_rollout<0, false>;
    }
}

// Its dynamic shared memory: goal values (general instances) and, but for the
// single-drone forms, two sets of staging planes and the CTA's observation rows.
size_t rollout_smem(const Consts& c, int D, int block, bool single) {
    const int goal = extended(c) ? GOAL_STRIDE : 0;
    return sizeof(float) * block * (single_form(c, D, single) ? goal : 2 * SMEM_PLANES + goal + c.obs_dim + ROW_PAD);
}

int rollout_grid(const Consts& c, int D, int block, bool single) {
    int dev = 0, n_sm = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const void* fn = (const void*)rollout_kernel(c, D, single);
    const size_t smem = rollout_smem(c, D, block, single);
    allow_smem(fn, smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, block, smem);
    return (occ > 0 ? occ : 1) * n_sm;
}

cudaError_t launch_rollout_ws(const Consts& c, const Dev& dv, const Tile* tiles, int n_tiles, int P, const int* perm,
                              const RolloutIO& io, int t0, int nsteps, cudaStream_t st) {
    if (n_tiles == 0) return cudaSuccess;
    const int ext = extended(c);
    if (P != 1 && P != 2) return cudaErrorInvalidValue;
    const auto k = P == 1 ? rollout_ws_kernel<1>(ext) : rollout_ws_kernel<2>(ext);
    const cudaError_t e = allow_ws_smem((const void*)k, c, P);
    if (e != cudaSuccess) return e;
    return launch_overlapped(k, n_tiles, 64 * P, ws_smem(c, P), st, c, dv, tiles, perm, io, t0, nsteps);
}

cudaError_t launch_rollout(const Consts& c, const Dev& dv, const Tile* tiles, int n_tiles, int block, const int* perm,
                           int* counter, const RolloutIO& io, int t0, int nsteps, int grid, bool single,
                           cudaStream_t st) {
    const size_t smem = rollout_smem(c, dv.D, block, single);
    const auto k = rollout_kernel(c, dv.D, single);
    const cudaError_t e = allow_smem((const void*)k, smem);
    if (e != cudaSuccess) return e;
    const int g = grid > 0 ? grid : n_tiles;
    const int grid_n = g < n_tiles ? g : n_tiles;
    return launch_overlapped(k, grid_n, block, smem, st, c, dv, tiles, n_tiles, perm, counter, io, t0, nsteps);
}

}  // namespace qsk
