// Closed-loop receding-horizon control (Sec. V-B): per control step c every
// scenario re-solves the ADMM of Sec. IV-B over the next N steps from its
// measured state, warm-started from the previous plan shifted by one step,
// with only the obstacles inside its sensing window; then the first control
// drives the plant one Euler step and the true state is checked for
// collision against every obstacle (scale LP, Sec. III-A).
#include "oca_common.cuh"
#include "oca_kernels.h"
#include "oca_models.cuh"
#include "oca_solvers.cuh"

namespace oca {

// horizon window of step c: reference rows, warm-start shift, measured
// state as s_0, sensing mask (one warp per scenario)
template <typename T, int KIND>
__global__ void __launch_bounds__(32) k_mpc_window(MpcArgs<T> a) {
    constexpr int NS = MDims<KIND>::NS, NU = MDims<KIND>::NU, D = MDims<KIND>::D;
    const int s = blockIdx.x, lane = threadIdx.x;
    const ScenMeta sm = a.meta[s];
    const int N = sm.N;
    const T *ref = a.ref + (long long)s * a.T_ref * NS;
    for (int e = lane; e < (N + 1) * NS; e += 32) {
        const int t = e / NS, i = e % NS;
        const int r = min(a.c + t, a.T_ref - 1);
        a.s_ref[(long long)(sm.state0 + t) * NS + i] = ref[(long long)r * NS + i];
    }
    if (a.c > 0) {
        // s_t <- s_{t+1} (t = 1..N-1), u_t <- u_{t+1} (t = 0..N-2); each lane
        // owns one component, so the in-place ascending copy is race-free
        if (lane < NS)
            for (int t = 1; t < N; ++t)
                a.s[(long long)(sm.state0 + t) * NS + lane] = a.s[(long long)(sm.state0 + t + 1) * NS + lane];
        if (lane < NU)
            for (int t = 0; t + 1 < N; ++t)
                a.u[(long long)(sm.ctrl0 + t) * NU + lane] = a.u[(long long)(sm.ctrl0 + t + 1) * NU + lane];
    }
    if (lane < NS) a.s[(long long)sm.state0 * NS + lane] = a.x[(long long)s * NS + lane];
    // sensing window: obstacle centres within +-win of the position
    for (int j = lane; j < sm.M; j += 32) {
        const int gm = sm.obs0 + j;
        bool in = true;
#pragma unroll
        for (int i = 0; i < D; ++i)
            if (a.win[i] > T(0)) in &= m_abs(a.obs_center[(long long)gm * D + i] - a.x[(long long)s * NS + i]) <= a.win[i];
        a.mask[gm] = in ? 1 : 0;
    }
}

// Pair arrays shifted one step along t: (y, zeta, xi) at (j, part, t) <- (j, part, t + 1)
// for t = 1..N-1, in place.  A copy bound by memory: a warp owns whole (obstacle, part)
// blocks of N consecutive pairs (as many as fill it), 32 pairs at a time in ascending
// order; its lanes read up to eight components of the following pair before any of them
// writes.  256 quadrotor runs of horizon 16 (393,216 pairs): 170 -> 41 us
// (a thread per block walked its N pairs alone).
constexpr int kShiftWarps = 4, kShiftU = 8;
template <typename T>
__global__ void __launch_bounds__(32 * kShiftWarps) k_mpc_shift_pairs(MpcArgs<T> a, int D) {
    const int s = blockIdx.y;
    const ScenMeta sm = a.meta[s];
    const int lane = threadIdx.x & 31, N = sm.N, per = max(1, 32 / N);  // blocks per warp
    const int n_blk = sm.M * sm.NP;
    const int first = (blockIdx.x * kShiftWarps + (threadIdx.x >> 5)) * per;
    if (first >= n_blk) return;
    const int n = min(per, n_blk - first) * N;  // this warp's pairs
    const long long P = a.P, p0 = sm.pair0 + (long long)first * N;
    for (int l0 = 0; l0 < n; l0 += 32) {
        const int l = l0 + lane, blk = first + l / N;
        const bool move = l < n && l % N + 1 < N;
        const int nr = move ? a.g.part_nf[sm.part0 + blk % sm.NP] : 0, no = move ? a.g.obs_nf[sm.obs0 + blk / sm.NP] : 0;
        const int nc = move ? nr + no + 2 + D : 0;  // lambda, mu, gamma, zeta, xi
        const long long p = p0 + l;
        auto at = [&](int e) -> T * {
            if (e < nr) return a.y + (long long)e * P + p;
            if (e < nr + no) return a.y + (long long)(a.FR + e - nr) * P + p;
            if (e == nr + no) return a.y + (long long)(a.FR + a.FO) * P + p;
            if (e == nr + no + 1) return a.zeta + p;
            return a.xi + (long long)(e - nr - no - 2) * P + p;
        };
        const int nmax = __reduce_max_sync(0xffffffffu, nc);
        for (int e0 = 0; e0 < nmax; e0 += kShiftU) {
            T v[kShiftU];
#pragma unroll
            for (int k = 0; k < kShiftU; ++k)
                if (e0 + k < nc) v[k] = at(e0 + k)[1];
            __syncwarp();
#pragma unroll
            for (int k = 0; k < kShiftU; ++k)
                if (e0 + k < nc) *at(e0 + k) = v[k];
            __syncwarp();
        }
    }
}

// plant: x <- x + dt f_c(x, u_0), u_0 the plan's first control clipped to
// the control box (zero where the solve left it non-finite); histories
template <typename T, int KIND>
__global__ void k_mpc_plant(MpcArgs<T> a, int n_scen) {
    constexpr int NS = MDims<KIND>::NS, NU = MDims<KIND>::NU;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_scen) return;
    const ScenMeta sm = a.meta[s];
    T x[NS], u0[NU], f[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) x[i] = a.x[(long long)s * NS + i];
    if (a.c == 0)
#pragma unroll
        for (int i = 0; i < NS; ++i) a.x_hist[(long long)s * (a.n_steps + 1) * NS + i] = x[i];
#pragma unroll
    for (int i = 0; i < NU; ++i) {
        T v = a.u[(long long)sm.ctrl0 * NU + i];
        if (!m_finite(v)) v = T(0);
        u0[i] = fmin(fmax(v, a.model.u_lo[i]), a.model.u_hi[i]);
        a.u_hist[((long long)s * a.n_steps + a.c) * NU + i] = u0[i];
    }
    dynamics<T, KIND>(a.model, x, u0, f, nullptr, nullptr);
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        x[i] += a.model.dt * f[i];
        a.x[(long long)s * NS + i] = x[i];
        a.x_hist[((long long)s * (a.n_steps + 1) + a.c + 1) * NS + i] = x[i];
    }
    a.iters_hist[(long long)s * a.n_steps + a.c] = a.iters[s];
}

// collision of the true state with every obstacle: alpha* < 1 for some
// (part, obstacle) marks the scenario with the first step it happened
// One thread per (obstacle, part) with its LP columns staged in shared memory (at most
// 32 KB), 32 threads a block: a latency chain of a few pivots, so the blocks spread.
constexpr int kCollideThreads = 32;
template <typename T, int KIND>
__global__ void __launch_bounds__(kCollideThreads) k_mpc_collide(MpcArgs<T> a) {
    constexpr int NS = MDims<KIND>::NS, D = MDims<KIND>::D;
    const int s = blockIdx.y;
    const ScenMeta sm = a.meta[s];
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= sm.M * sm.NP) return;
    const int j = e / sm.NP, part = e % sm.NP;
    const int gm = sm.obs0 + j, gp = sm.part0 + part;
    T x[NS], off[D];
    Lane<T, D> L;
#pragma unroll
    for (int i = 0; i < NS; ++i) x[i] = a.x[(long long)s * NS + i];
#pragma unroll
    for (int i = 0; i < D; ++i) off[i] = a.g.part_off[gp * D + i];
    part_pose<T, KIND>(a.model, a.g.part_link[gp], off, x, L.rho, L.R, nullptr, nullptr, nullptr);
    L.A = a.g.part_A + (long long)gp * a.g.FR * D;
    L.b = a.g.part_b + (long long)gp * a.g.FR;
    L.nr = a.g.part_nf[gp];
    L.C = a.g.obs_C + (long long)gm * a.g.FO * D;
    L.d = a.g.obs_d + (long long)gm * a.g.FO;
    L.no = a.g.obs_nf[gm];
    int bas[D + 1];
    T xB[D + 1], alpha;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *rec = reinterpret_cast<T *>(smem_raw) + threadIdx.x * kLpRec;
    const int stride = kCollideThreads * kLpRec;
    lp_stage_part<T, D>(L, rec, stride);
    lp_stage_obstacle<T, D>(L, rec, stride);
    lp_solve<T, D>(StagedCols<T, D>{rec, stride, L.nr, L.no}, bas, xB, alpha);
    if (alpha < T(1)) atomicCAS(a.collided + s, -1, a.c + 1);
}

template <typename T, int KIND>
cudaError_t mpc_launch_t(const MpcArgs<T> &a, int stage, int n_scen, int max_blk, cudaStream_t st) {
    switch (stage) {
        case 0: k_mpc_window<T, KIND><<<n_scen, 32, 0, st>>>(a); break;
        case 1: k_mpc_shift_pairs<T><<<dim3((max_blk + kShiftWarps - 1) / kShiftWarps, n_scen), 32 * kShiftWarps, 0, st>>>(a, MDims<KIND>::D); break;
        case 2: k_mpc_plant<T, KIND><<<(n_scen + 63) / 64, 64, 0, st>>>(a, n_scen); break;
        default:
            k_mpc_collide<T, KIND><<<dim3((max_blk + kCollideThreads - 1) / kCollideThreads, n_scen), kCollideThreads,
                                     sizeof(T) * kLpRec * kCollideThreads * (a.g.FR + a.g.FO), st>>>(a);
            break;
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_mpc(const MpcArgs<T> &a, int stage, int n_scen, int max_blk, cudaStream_t st) {
    if (n_scen <= 0) return cudaSuccess;
    switch (a.model.kind) {
        case 0: return mpc_launch_t<T, 0>(a, stage, n_scen, max_blk, st);
        case 1: return mpc_launch_t<T, 1>(a, stage, n_scen, max_blk, st);
        case 2: return mpc_launch_t<T, 2>(a, stage, n_scen, max_blk, st);
    }
    return cudaErrorInvalidValue;
}

template cudaError_t launch_mpc<float>(const MpcArgs<float> &, int, int, int, cudaStream_t);
template cudaError_t launch_mpc<double>(const MpcArgs<double> &, int, int, int, cudaStream_t);

}  // namespace oca
