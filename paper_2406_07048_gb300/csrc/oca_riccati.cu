// Trajectory step of the ADMM (Sec. IV-B eqn:ADMM_state_updates, one SQP
// QP per iteration) and the per-scenario stopping rule.  The state/control
// boxes of eqn:MPC_opt_origin are a further ADMM block: a bounded copy z of
// (s, u) with scaled dual w, so that the step stays an unconstrained LQ
// problem (Riccati) with the augmented term 0.5 rho_b |(s,u) - z + w|^2; a
// proximal term 0.5 damp |(s,u) - (s,u)^j|^2 damps the SQP step.
//
// At launch j every scenario
//   1. tests the stopping rule of iteration j-1 (Sec. IV-B):
//        r_pri  = sum dzeta^2 + |dxi|^2     (partials written by the pair kernel's head at j)
//        r_dual = sum |dlambda|^2 + |dmu|^2 (partials written by the pair kernel at j-1)
//      and retires the scenario when both are below their tolerances or j = max_iter;
//   2. otherwise assembles the LQ stage terms at (s^j, u^j): Euler dynamics
//      linearised (A_t, B_t, c_t), tracking cost of eqn:navigation_cost and
//      the Gauss-Newton model of sigma/2 sum |r_ijt(s_t)|^2 rebuilt from the
//      per-(part, t) statistics W, Wc, E through the pose Jacobians;
//   3. runs the backward Riccati recursion (factorisation precision F) and
//      the forward sweep, writing s^{j+1}, u^{j+1} and the new poses.
#include <algorithm>
#include <type_traits>

#include "oca_common.cuh"
#include "oca_fp64.cuh"
#include "oca_kernels.h"
#include "oca_ric.cuh"
#include "oca_ricprog.cuh"

namespace oca {

long long riccati_scratch_elems(int kind, int N) {
    switch (kind) {
        // the forward step's and the adjoint's share the block (12 states: the adjoint's is dense)
        case 0: return RicMap<0>::adj_size(N);
        case 1: return RicMap<1>::adj_size(N);
        default: return std::max(RicLayout<12, 4>::size(N), RicMap<2>::size(N));
    }
}

template <typename T, int KIND>
__device__ void finish_scenario(const RicArgs<T> &a, const ScenMeta &sm, int s, int status, int iters, double rp, double rd) {
    constexpr int NS = MDims<KIND>::NS, NU = MDims<KIND>::NU;
    const int lane = threadIdx.x;
    double F = 0.0;
    for (int t = lane; t <= sm.N; t += 32) {
        for (int i = 0; i < NS; ++i) {
            const double e = double(a.s[(long long)(sm.state0 + t) * NS + i]) - double(a.s_ref[(long long)(sm.state0 + t) * NS + i]);
            F += double(a.model.Qs[i]) * e * e;
        }
        if (t < sm.N)
            for (int i = 0; i < NU; ++i) {
                const double uu = double(a.u[(long long)(sm.ctrl0 + t) * NU + i]);
                F += double(a.model.Qu[i]) * uu * uu;
            }
    }
    F = warp_sum(F);
    if (lane == 0) {
        a.scen_status[s] = status;
        a.status_out[s] = status;
        a.iters_out[s] = iters;
        a.r_pri_out[s] = T(rp);
        a.r_dual_out[s] = T(rd);
        a.cost_out[s] = T(F);
        atomicSub(a.active_count, 1);
    }
}

// stopping rule of iteration j-1 (one warp): true when the scenario is done
template <typename T, int KIND>
__device__ bool stop_rule(const RicArgs<T> &a, const ScenMeta &sm, int s, int j) {
    const int lane = threadIdx.x;
    if (j >= 1) {
        const double *rcur = a.res + (size_t)(j & 1) * a.n_tiles * 2;
        const double *rprev = a.res + (size_t)((j - 1) & 1) * a.n_tiles * 2;
        double rp = 0.0, rd = 0.0;
        for (int k = lane; k < sm.ntile; k += 32) {
            rp += rcur[(size_t)(sm.tile0 + k) * 2];
            rd += rprev[(size_t)(sm.tile0 + k) * 2 + 1];
        }
        rp = warp_sum(rp) + a.box_res[2 * s];      // + box-block residuals of iteration j-1
        rd = warp_sum(rd) + a.box_res[2 * s + 1];
        const bool conv = rp <= double(a.eps_pri) && rd <= double(a.eps_dual);
        if (conv || j >= a.max_iter) {
            finish_scenario<T, KIND>(a, sm, s, conv ? OCA_SCEN_CONVERGED : OCA_SCEN_MAX_ITER, j, rp, rd);
            return true;
        }
    } else if (a.max_iter <= 0) {
        finish_scenario<T, KIND>(a, sm, s, OCA_SCEN_MAX_ITER, 0, 0.0, 0.0);
        return true;
    }
    return false;
}

template <typename T>
__device__ __forceinline__ void stage_inputs(const RicArgs<T> &a, StageParams<T> &sp, StageSrc<T> &src) {
    sp.model = a.model;
    sp.g = a.g;
    sp.sigma = a.sigma;
    sp.rho_box = a.rho_box;
    sp.damp = a.damp;
    sp.s_ref = a.s_ref;
    sp.Qtot = a.Qtot;
    src.s = a.s;
    src.u = a.u;
    src.zs = a.box_zs;
    src.ws = a.box_ws;
    src.zu = a.box_zu;
    src.wu = a.box_wu;
    src.stats = a.stats;
}

// Step t of the new iterate (st = s_{t+1}, ut = u_t as stored): box block
// z = clip(x + w), w += x - z of its components, poses of s_{t+1}.  Everything is
// loaded before the first store: each load costs most of a microsecond and the
// compiler may not move one past a store.
template <typename T, int KIND>
__device__ __forceinline__ void box_poses(const RicArgs<T> &a, const ScenMeta &sm, int t, const T *st, const T *ut, double &rpb,
                                          double &rdb) {
    constexpr int NS = MDims<KIND>::NS, NU = MDims<KIND>::NU, D = MDims<KIND>::D;
    const long long ks = (long long)(sm.state0 + t + 1) * NS, ku = (long long)(sm.ctrl0 + t) * NU;
    const bool box = a.rho_box > T(0);  // rho_box = 0: no box block
    T zs[NS], ws[NS], zu[NU], wu[NU];
    bool bs[NS], bu[NU];
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        bs[i] = box && bounded(a.model.s_lo[i], a.model.s_hi[i]);
        if (bs[i]) {
            zs[i] = a.box_zs[ks + i];
            ws[i] = a.box_ws[ks + i];
        }
    }
#pragma unroll
    for (int i = 0; i < NU; ++i) {
        bu[i] = box && bounded(a.model.u_lo[i], a.model.u_hi[i]);
        if (bu[i]) {
            zu[i] = a.box_zu[ku + i];
            wu[i] = a.box_wu[ku + i];
        }
    }
    for (int part = 0; part < sm.NP; ++part) {
        const int gp = sm.part0 + part;
        T off[D], rho[D], R[D * D];
#pragma unroll
        for (int i = 0; i < D; ++i) off[i] = ldg(a.g.part_off + gp * D + i);
        part_pose<T, KIND>(a.model, ldg(a.g.part_link + gp), off, st, rho, R, nullptr, nullptr, nullptr);
        const int col = sm.qbeg + part * sm.N + t;
#pragma unroll
        for (int i = 0; i < D; ++i) a.pose[(long long)i * a.Qtot + col] = rho[i];
#pragma unroll
        for (int i = 0; i < D * D; ++i) a.pose[(long long)(D + i) * a.Qtot + col] = R[i];
    }
    auto update = [&](T x, T lo, T hi, T z, T w, T *zo, T *wo) {
        const T zn = fmin(fmax(x + w, lo), hi);
        rdb += double(zn - z) * double(zn - z);
        rpb += double(x - zn) * double(x - zn);
        *zo = zn;
        *wo = w + (x - zn);
    };
#pragma unroll
    for (int i = 0; i < NS; ++i)
        if (bs[i]) update(st[i], a.model.s_lo[i], a.model.s_hi[i], zs[i], ws[i], a.box_zs + ks + i, a.box_ws + ks + i);
#pragma unroll
    for (int i = 0; i < NU; ++i)
        if (bu[i]) update(ut[i], a.model.u_lo[i], a.model.u_hi[i], zu[i], wu[i], a.box_zu + ku + i, a.box_wu + ku + i);
}

// ============================================================================
// Three kernels per trajectory step.
//   k_traj_stage   stopping rule and stage assembly, lanes over t (FP32 work with
//                  everything in registers, written as one packed record per stage)
//   k_traj_lq      backward recursion and forward sweep (the FP64 chain): 2-D models,
//                  L lanes per scenario, 32 / L scenarios per warp
//   k_traj_lq4     the same for the 12-state model, four warps per scenario
//   k_traj_apply   the new iterate in T, box block and poses, lanes over t
// The recursion is bound by FP64 issue (oca_ricprog.cuh), the other two by latency;
// apart, the recursion keeps one warp per scheduler busy with nothing but the
// recursion, and the assembly and the box block run over all horizon steps at once.
// 2,048 trailer scenarios, mean horizon 50: 34 + 138 + 18 us per step; one warp
// per scenario doing everything with dense products took 510 us.  A stage of the
// recursion takes 2,660 cycles (22 FP64 instructions: 1,408 of them), a step of the
// sweep 700; the 80-stage scenarios set the time.
// ============================================================================

// the lists of multiply-adds of the recursion's three products
template <int KIND, int L, int PHASE>
__device__ constexpr auto kRicTab = RicBuild<KIND>::template table<PHASE, L>();
template <int KIND>
__device__ constexpr auto kRicOut = RicBuild<KIND>::out_map();


// 8- or 4-byte access at a shared-memory byte address
__device__ __forceinline__ double lds(unsigned at, double) {
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(at) : "memory");
    return v;
}
__device__ __forceinline__ float lds(unsigned at, float) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
    return v;
}
__device__ __forceinline__ void sts(unsigned at, double v) { asm volatile("st.shared.f64 [%0], %1;" ::"r"(at), "d"(v) : "memory"); }
__device__ __forceinline__ void sts(unsigned at, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(at), "f"(v) : "memory"); }

// One product's slots of one lane: the four shared-memory addresses of each slot,
// decoded once (a warp alone on its scheduler pays several cycles for every
// instruction, so the step decodes nothing).
template <typename F, int SLOTS>
struct LqSlots {
    unsigned in[SLOTS], c[SLOTS], v[SLOTS], st[SLOTS];
    unsigned cont;  // bit i: slot i continues the accumulator of slot i - 1

    template <int L>
    __device__ __forceinline__ void load(const RicPhase<SLOTS, L> &tab, int lane, const F *region) {
        const unsigned base = (unsigned)__cvta_generic_to_shared(region);
        cont = 0;
#pragma unroll
        for (int i = 0; i < SLOTS; ++i) {
            const uint64_t w = tab.code[i][lane];
            const unsigned at = (unsigned)w & 0xffffu;
            const bool k = at == (unsigned)kRicCont;
            cont |= (k ? 1u : 0u) << i;
            in[i] = base + (k ? 0u : at) * (unsigned)sizeof(F);
            c[i] = base + ((unsigned)(w >> 16) & 0xffffu) * (unsigned)sizeof(F);
            v[i] = base + ((unsigned)(w >> 32) & 0xffffu) * (unsigned)sizeof(F);
            st[i] = base + ((unsigned)(w >> 48) & 0xffffu) * (unsigned)sizeof(F);
        }
    }
    // A product reads nothing that it writes, so all operands are loaded first and
    // the multiply-adds follow each other without a load's latency between them.
    __device__ __forceinline__ void run() const {
        F a[SLOTS], x[SLOTS], y[SLOTS];
#pragma unroll
        for (int i = 0; i < SLOTS; ++i) {
            a[i] = lds(in[i], F(0));
            x[i] = lds(c[i], F(0));
            y[i] = lds(v[i], F(0));
        }
#pragma unroll
        for (int i = 0; i < SLOTS; ++i) a[i] = fma(x[i], y[i], i > 0 && (cont >> i & 1u) ? a[i > 0 ? i - 1 : 0] : a[i]);
#pragma unroll
        for (int i = 0; i < SLOTS; ++i) sts(st[i], a[i]);
    }
};
template <typename F, class Tab>
struct LqSlotsOf;
template <typename F, int SLOTS, int L>
struct LqSlotsOf<F, RicPhase<SLOTS, L>> {
    using type = LqSlots<F, SLOTS>;
};

// threads per scenario of the per-step kernels: one per horizon step up to 96
constexpr int kTrajBlock = 96;
// shared elements per thread of k_traj_stage (the 12-state record is written directly)
template <typename F, int KIND>
constexpr int traj_rec_stride() { return KIND == 2 ? 0 : RicMap<KIND>::REC | 1; }

// Stage t of the 12-state model as a packed record, in T: only the entries of A and B
// that are not structurally 0 or 1, and the Gauss-Newton terms of the six coordinates
// (position, angles) that a part's pose depends on.  (The generic assembly over dense
// 12 x 12 arrays keeps 2 KB per thread in local memory.)
template <typename T, typename F>
__device__ void quad_record(const StageParams<T> &a, const StageSrc<T> &src, const ScenMeta &sm, int t, F *rec) {
    using Mp = RicMap<2>;
    constexpr int NS = 12, NU = 4;
    const DevModel<T> &m = a.model;
    const int N = sm.N;
    T st[NS];
    const long long ks = (long long)(sm.state0 + t) * NS;
#pragma unroll
    for (int i = 0; i < NS; ++i) st[i] = src.s[ks + i];
    T R[9], dR[3][9];
    rot3<T>(st[6], st[7], st[8], R, dR);
    if (t < N) {
        T ut[NU];
        const long long ku = (long long)(sm.ctrl0 + t) * NU;
#pragma unroll
        for (int i = 0; i < NU; ++i) ut[i] = src.u[ku + i];
        T f[NS];
        dynamics<T, 2>(m, st, ut, f, nullptr, nullptr);
        const T mass = m.p[0], Jx = m.p[2], Jy = m.p[3], Jz = m.p[4], arm = m.p[5], km = m.p[6], dt = m.dt;
        const T thrust = mass * m.p[1] + ut[0] + ut[1] + ut[2] + ut[3];
        const T p = st[9], q = st[10], r = st[11];
        const T cf = m_cos(st[6]), sf = m_sin(st[6]), ct = m_cos(st[7]), tt = m_tan(st[7]), sc = T(1) / ct;
        const T w1 = sf * q + cf * r, w2 = cf * q - sf * r;
        // df/ds and df/du in the order of RicSparse<2>
        T A[25], B[9];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (i < 2 || k < 2) A[i * 3 + k] = dt * (dR[k][i * 3 + 2] * thrust / mass);
            B[i] = dt * (R[i * 3 + 2] / mass);
        }
        A[8] = T(1) + dt * (w2 * tt);
        A[9] = dt * (w1 * sc * sc);
        A[10] = dt * (sf * tt);
        A[11] = dt * (cf * tt);
        A[12] = dt * -w1;
        A[13] = dt * cf;
        A[14] = dt * -sf;
        A[15] = dt * (w2 * sc);
        A[16] = dt * (w1 * sc * tt);
        A[17] = dt * (sf * sc);
        A[18] = dt * (cf * sc);
        A[19] = dt * (r * (Jy - Jz) / Jx);
        A[20] = dt * (q * (Jy - Jz) / Jx);
        A[21] = dt * (r * (Jz - Jx) / Jy);
        A[22] = dt * (p * (Jz - Jx) / Jy);
        A[23] = dt * (q * (Jx - Jy) / Jz);
        A[24] = dt * (p * (Jx - Jy) / Jz);
        B[3] = dt * (arm / Jx);
        B[4] = dt * (-arm / Jx);
        B[5] = dt * (-arm / Jy);
        B[6] = dt * (arm / Jy);
        B[7] = dt * (km / Jz);
        B[8] = dt * (-km / Jz);
        // c = s + dt f - A s - B u over the entries that are not 0, in column order
        T c[NS];
#pragma unroll
        for (int i = 0; i < NS; ++i) c[i] = st[i] + dt * f[i];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            c[i] -= st[i];
            c[i] -= dt * st[3 + i];
            c[3 + i] -= st[3 + i];
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (i < 2 || k < 2) c[3 + i] -= A[i * 3 + k] * st[6 + k];
#pragma unroll
            for (int k = 0; k < NU; ++k) c[3 + i] -= B[i] * ut[k];
        }
        c[6] -= A[8] * st[6];
        c[6] -= A[9] * st[7];
        c[6] -= dt * st[9];
        c[6] -= A[10] * st[10];
        c[6] -= A[11] * st[11];
        c[7] -= A[12] * st[6];
        c[7] -= st[7];
        c[7] -= A[13] * st[10];
        c[7] -= A[14] * st[11];
        c[8] -= A[15] * st[6];
        c[8] -= A[16] * st[7];
        c[8] -= st[8];
        c[8] -= A[17] * st[10];
        c[8] -= A[18] * st[11];
        c[9] -= st[9];
        c[9] -= A[19] * st[10];
        c[9] -= A[20] * st[11];
        c[9] -= B[3] * ut[1];
        c[9] -= B[4] * ut[3];
        c[10] -= A[21] * st[9];
        c[10] -= st[10];
        c[10] -= A[22] * st[11];
        c[10] -= B[5] * ut[0];
        c[10] -= B[6] * ut[2];
        c[11] -= A[23] * st[9];
        c[11] -= A[24] * st[10];
        c[11] -= st[11];
        c[11] -= B[7] * ut[0];
        c[11] -= B[8] * ut[1];
        c[11] -= B[7] * ut[2];
        c[11] -= B[8] * ut[3];
#pragma unroll
        for (int i = 0; i < 25; ++i) rec[Mp::rA + i] = F(A[i]);
#pragma unroll
        for (int i = 0; i < 9; ++i) rec[Mp::rB + i] = F(B[i]);
#pragma unroll
        for (int i = 0; i < NS; ++i) rec[Mp::rc + i] = F(c[i]);
#pragma unroll
        for (int i = 0; i < NU; ++i) {
            T acc = -a.damp * ut[i];
            if (bounded(m.u_lo[i], m.u_hi[i])) acc -= a.rho_box * (src.zu[ku + i] - src.wu[ku + i]);
            rec[Mp::rr + i] = F(acc);
        }
    }
    // diagonal and linear terms, and the 6 x 6 Gauss-Newton block over (position, angles)
    T Qd[NS], qr[NS], H[6][6];
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        Qd[i] = T(2) * m.Qs[i];
        qr[i] = -T(2) * m.Qs[i] * a.s_ref[ks + i];
        if (t >= 1) {
            Qd[i] += a.damp;
            qr[i] -= a.damp * st[i];
            if (bounded(m.s_lo[i], m.s_hi[i])) {
                Qd[i] += a.rho_box;
                qr[i] -= a.rho_box * (src.zs[ks + i] - src.ws[ks + i]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int k = 0; k < 6; ++k) H[i][k] = T(0);
    if (t >= 1) {
        for (int part = 0; part < sm.NP; ++part) {
            const int gp = sm.part0 + part;
            const long long col = sm.qbeg + part * N + (t - 1);
            T W[3][3], Wc[3], E[9], off[3], rho[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) off[i] = a.g.part_off[gp * 3 + i];
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int k = 0; k <= i; ++k) W[i][k] = W[k][i] = src.stats[(long long)(i * (i + 1) / 2 + k) * a.Qtot + col];
#pragma unroll
            for (int i = 0; i < 3; ++i) Wc[i] = src.stats[(long long)(6 + i) * a.Qtot + col];
#pragma unroll
            for (int i = 0; i < 9; ++i) E[i] = src.stats[(long long)(9 + i) * a.Qtot + col];
            T gv[3], WR[9];  // Wc - W rho, W R
#pragma unroll
            for (int i = 0; i < 3; ++i) rho[i] = st[i] + R[i * 3] * off[0] + R[i * 3 + 1] * off[1] + R[i * 3 + 2] * off[2];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                gv[i] = Wc[i] - W[i][0] * rho[0] - W[i][1] * rho[1] - W[i][2] * rho[2];
#pragma unroll
                for (int k = 0; k < 3; ++k) WR[i * 3 + k] = W[i][0] * R[k] + W[i][1] * R[3 + k] + W[i][2] * R[6 + k];
            }
            T Hp[6][6], g[6];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                g[i] = -gv[i];
#pragma unroll
                for (int k = 0; k < 3; ++k) Hp[i][k] = W[i][k];
            }
#pragma unroll
            for (int x = 0; x < 3; ++x) {
                T d[3], Wd[3], WD[9];  // drho/dangle_x, W d, W dR_x
#pragma unroll
                for (int i = 0; i < 3; ++i) d[i] = dR[x][i * 3] * off[0] + dR[x][i * 3 + 1] * off[1] + dR[x][i * 3 + 2] * off[2];
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    Wd[i] = W[i][0] * d[0] + W[i][1] * d[1] + W[i][2] * d[2];
                    Hp[i][3 + x] = Wd[i];
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        WD[i * 3 + k] = W[i][0] * dR[x][k] + W[i][1] * dR[x][3 + k] + W[i][2] * dR[x][6 + k];
                }
                T gx = -(d[0] * gv[0] + d[1] * gv[1] + d[2] * gv[2]);
#pragma unroll
                for (int i = 0; i < 9; ++i) gx += dR[x][i] * (E[i] + WR[i]);
                g[3 + x] = gx;
#pragma unroll
                for (int y = 0; y <= x; ++y) {
                    T v = T(0);
#pragma unroll
                    for (int i = 0; i < 3; ++i)
                        v += (dR[y][i * 3] * off[0] + dR[y][i * 3 + 1] * off[1] + dR[y][i * 3 + 2] * off[2]) * Wd[i];
#pragma unroll
                    for (int i = 0; i < 9; ++i) v += dR[y][i] * WD[i];
                    Hp[3 + y][3 + x] = v;
                }
            }
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                T hs = T(0);
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    const T h = i <= k ? Hp[i][k] : Hp[k][i];
                    hs += h * st[k < 3 ? k : 3 + k];
                    if (i <= k) H[i][k] += a.sigma * h;
                }
                qr[i < 3 ? i : 3 + i] += a.sigma * (g[i] - hs);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        rec[Mp::rq + i] = F(qr[i]);
#pragma unroll
        for (int k = i; k < NS; ++k) {
            const bool ci = i < 3 || (i >= 6 && i < 9), ck = k < 3 || (k >= 6 && k < 9);
            T v = i == k ? Qd[i] : T(0);
            if (ci && ck) v += H[i < 3 ? i : i - 3][k < 3 ? k : k - 3];
            rec[Mp::rQ + Mp::sym(i, k)] = F(v);
        }
    }
}

template <typename T, typename F, int KIND>
__global__ void __launch_bounds__(kTrajBlock) k_traj_stage(RicArgs<T> a) {
    constexpr int NS = MDims<KIND>::NS;
    using Mp = RicMap<KIND>;
    const int s = blockIdx.x, lane = threadIdx.x, NT = blockDim.x;
    const ScenMeta sm = a.meta[s];
    // one warp reads and writes the scenario's status; the others take its verdict
    __shared__ int s_skip;
    if (lane < 32) {
        const int j = *a.iter;
        const bool skip = a.scen_status[s] != kActive || j > a.max_iter || stop_rule<T, KIND>(a, sm, s, j);
        if (lane == 0) s_skip = skip;
    }
    __syncthreads();
    if (s_skip) return;
    F *scr = reinterpret_cast<F *>(a.scratch) + a.scratch0[s];
    StageParams<T> sp;
    StageSrc<T> src;
    stage_inputs(a, sp, src);
    if constexpr (KIND == 2) {
        for (int t = lane; t <= sm.N; t += NT) quad_record<T, F>(sp, src, sm, t, scr + Mp::rec(t));
    } else {
        struct Sink {
            F *r;
            __device__ void A(int i, int k, T v) {
                const int e = RicSparse<KIND>::a_slot(i, k);
                if (e >= 0) r[Mp::rA + e] = F(v);
            }
            __device__ void B(int i, int k, T v) {
                const int e = RicSparse<KIND>::b_slot(i, k);
                if (e >= 0) r[Mp::rB + e] = F(v);
            }
            __device__ void c(int i, T v) { r[Mp::rc + i] = F(v); }
            __device__ void u(int i, T v) { r[Mp::rr + i] = F(v); }
            __device__ void Q(int i, int k, T v) {
                if (i <= k) r[Mp::rQ + Mp::sym(i, k)] = F(v);
            }
            __device__ void q(int i, T v) { r[Mp::rq + i] = F(v); }
        };
        // records through shared memory (odd stride): written straight to the scratch,
        // every 8-byte store of a warp touches 32 sectors
        constexpr int RS = traj_rec_stride<F, KIND>();
        extern __shared__ __align__(16) unsigned char smem_raw[];
        F *rec = reinterpret_cast<F *>(smem_raw);  // [NT][RS]
        for (int t0 = 0; t0 <= sm.N; t0 += NT) {
            const int n = min(NT, sm.N + 1 - t0);
            if (lane < n) {
                Sink out{rec + lane * RS};
                assemble_terms<T, KIND>(sp, src, sm, t0 + lane, out);
            }
            __syncthreads();
            F *dst = scr + Mp::rec(t0);
            for (int e = lane; e < n * Mp::REC; e += NT) dst[e] = rec[e / Mp::REC * RS + e % Mp::REC];
            __syncthreads();
        }
    }
    if (lane < NS) scr[Mp::s0(sm.N) + lane] = F(a.s[(long long)sm.state0 * NS + lane]);
}

// What the recursion needs of a launch, free of the array type T.
template <typename F>
struct LqArgs2 {
    const ScenMeta *meta;
    const int *order;        // scenarios by descending horizon
    int n_scen;
    const int *scen_status;  // forward: scenarios with kActive are solved
    const int *iters;        // adjoint (not null): scenarios with k < iters
    int k;
    void *scratch;
    const long long *scratch0;
    F dt, ru[4];
    int *ok;                 // [S] out: factorisation and sweep finite and positive definite
    int *iter;               // advanced by one (null: none)

    __device__ __forceinline__ bool active(int s) const { return iters ? k < iters[s] : scen_status[s] == kActive; }
};

// One CTA per SM, two warps per scheduler.  A group of 32 / L scenarios (neighbours
// in the order, so of about the same horizon) takes one warp, L lanes each; the
// groups, longest first, are dealt to the K = 4 x CTAs schedulers back and forth
// (0..K-1, K-1..0, ...), so that the longest chains have a scheduler for themselves
// and the others share with short ones: two long chains on one scheduler would each
// run at half speed.  Per stage: the three products as slot lists, the 2 x 2
// inverse between them, the next record loaded meanwhile.  F = A + B K and f = c + B k
// are formed with P, by lanes that would otherwise idle, so that the sweep is one
// matrix-vector product per step (lane i owns s_i) instead of two dependent ones.
constexpr int kLqWarps = 8;
template <typename F, int KIND, int L>
__global__ void __launch_bounds__(32 * kLqWarps) k_traj_lq(LqArgs2<F> a) {
    using Mp = RicMap<KIND>;
    constexpr int NS = Mp::NS, NU = Mp::NU, G = 32 / L, REC = Mp::REC, OUT = Mp::OUT;
    static_assert(NU == 2, "2-D models");
    constexpr int PR = (REC + L - 1) / L, PO = (OUT + L - 1) / L, KE = NU * (NS + 1), PK = (KE + L - 1) / L;
    __shared__ F region[kLqWarps][G][Mp::SIZE];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane / L, li = lane % L;
    if (a.iter && blockIdx.x == 0 && threadIdx.x == 0) *a.iter += 1;
    const int n_group = (a.n_scen + G - 1) / G, K = 4 * gridDim.x, slot = (warp & 3) * gridDim.x + blockIdx.x;
    F *sm = region[warp][g];

    typename LqSlotsOf<F, std::remove_cv_t<decltype(kRicTab<KIND, L, 0>)>>::type prod_y;
    typename LqSlotsOf<F, std::remove_cv_t<decltype(kRicTab<KIND, L, 1>)>>::type prod_m;
    typename LqSlotsOf<F, std::remove_cv_t<decltype(kRicTab<KIND, L, 2>)>>::type prod_p;
    prod_y.load(kRicTab<KIND, L, 0>, li, sm);
    prod_m.load(kRicTab<KIND, L, 1>, li, sm);
    prod_p.load(kRicTab<KIND, L, 2>, li, sm);
    int om[PO];
#pragma unroll
    for (int r = 0; r < PO; ++r) om[r] = li + L * r < OUT ? kRicOut<KIND>.at[li + L * r] : 0;

    if (li == 0) {
        sm[Mp::ZERO] = F(0);
        sm[Mp::ONE] = F(1);
        sm[Mp::DT] = a.dt;
        for (int x = 0; x < NU; ++x) sm[Mp::RU + x] = a.ru[x];
    }
    for (int round = warp >> 2; round * K < n_group; round += kLqWarps / 4) {
    const int group = round & 1 ? (round + 1) * K - 1 - slot : round * K + slot;
    const int at = group * G + g;
    const int s = group < n_group && at < a.n_scen ? a.order[at] : -1;
    const bool live = s >= 0 && a.active(s);
    if (!__any_sync(0xffffffffu, live)) continue;
    const int N = live ? a.meta[s].N : 0;
    int Nm = N;
#pragma unroll
    for (int o = 16; o >= L; o >>= 1) Nm = max(Nm, __shfl_xor_sync(0xffffffffu, Nm, o));
    F *scr = reinterpret_cast<F *>(a.scratch) + (live ? a.scratch0[s] : 0);
    __syncwarp();
    if (live) {
        const F *rN = scr + Mp::rec(N), *r1 = scr + Mp::rec(N - 1);
        for (int e = li; e < Mp::NSYM; e += L) sm[Mp::P0 + e] = rN[Mp::rQ + e];
        for (int e = li; e < NS; e += L) sm[Mp::p0 + e] = rN[Mp::rq + e];
        for (int e = li; e < REC; e += L) sm[Mp::REC0 + e] = r1[e];
    }
    bool ok = true;
    for (int t = Nm - 1; t >= 0; --t) {
        const bool act = t < N;
        F nxt[PR];
        __syncwarp();
        if (act) {
            if (t >= 1) {
                const F *rn = scr + Mp::rec(t - 1);
#pragma unroll
                for (int r = 0; r < PR; ++r)
                    if (li + L * r < REC) nxt[r] = rn[li + L * r];
            }
            prod_y.run();
        }
        __syncwarp();
        if (act) prod_m.run();
        __syncwarp();
        if (act) {
            // K = -Quu^-1 [Qus | qu] by the 2 x 2 adjugate; Quu not positive definite: K = 0, the
            // scenario fails.  It also fails where u11 [Qus | qu] passes the largest number
            // (costs of 1e150): forming the inverse first would take one FP64 instruction more
            // a stage (trailer batch 3,844 -> 3,853 us, gradient call 1,610 -> 1,617).
            const F u00 = sm[Mp::U0], u01 = sm[Mp::U0 + 1], u11 = sm[Mp::U0 + 3];
            const F det = fma(u00, u11, -(u01 * u01));
            const bool pd = positive_finite(u00) && positive_finite(det);
            ok = ok && pd;
            const F id = pd ? -recip(det) : F(0);
#pragma unroll
            for (int r = 0; r < PK; ++r) {
                const int e = li + L * r;
                if (e < KE) {
                    const bool x1 = e >= NS + 1;
                    const F own = sm[Mp::H0 + e], other = sm[Mp::H0 + (x1 ? e - (NS + 1) : e + (NS + 1))];
                    sm[Mp::K0 + e] = fma(x1 ? u00 : u11, own, -(u01 * other)) * id;
                }
            }
        }
        __syncwarp();
        if (act) prod_p.run();
        __syncwarp();
        if (act) {
            F *o = scr + Mp::out(N, t);
#pragma unroll
            for (int r = 0; r < PO; ++r)
                if (li + L * r < OUT) o[li + L * r] = sm[om[r]];
        }
        __syncwarp();
        if (act && t >= 1) {
#pragma unroll
            for (int r = 0; r < PR; ++r)
                if (li + L * r < REC) sm[Mp::REC0 + li + L * r] = nxt[r];
        }
    }
    // forward sweep s_{t+1} = F_t s_t + f_t, u_t = K_t s_t + k_t: lane i owns row i of
    // [F; K] (the controls cost no instruction of their own); the next step's row is
    // loaded meanwhile
    __syncwarp();
    constexpr int NZ = Mp::NZ;
    static_assert(NZ <= L, "one row of [F; K] per lane");
    const bool own = live && li < NZ;
    F x = live && li < NS ? scr[Mp::s0(N) + li] : F(0);
    constexpr int AHEAD = 4;  // steps: a step takes about 500 cycles, a load from L2 up to 1,500
    F row[AHEAD][NS], fv[AHEAD];
    auto fetch = [&](int t, F (&r)[NS], F &f) {
#pragma unroll
        for (int k = 0; k < NS; ++k) r[k] = F(0);
        f = F(0);
        if (own && t < N) {
            const F *o = scr + Mp::out(N, t);
#pragma unroll
            for (int k = 0; k < NS; ++k) r[k] = o[li * NS + k];
            f = o[NZ * NS + li];
        }
    };
#pragma unroll
    for (int d = 0; d < AHEAD; ++d) fetch(d, row[d], fv[d]);
    bool fin = true;
    for (int t0 = 0; t0 < Nm; t0 += AHEAD) {
#pragma unroll
        for (int d = 0; d < AHEAD; ++d) {
            const int t = t0 + d;
            F v = fv[d];
#pragma unroll
            for (int k = 0; k < NS; ++k) v = fma(row[d][k], __shfl_sync(0xffffffffu, x, k, L), v);
            x = v;
            if (own && t < N) {
                scr[Mp::sol(N, t) + li] = v;
                fin = fin && finite(v);
            }
            fetch(t + AHEAD, row[d], fv[d]);
        }
    }
    const unsigned bad = __ballot_sync(0xffffffffu, live && !(ok && fin));
    const unsigned mine = L == 32 ? 0xffffffffu : ((1u << (L & 31)) - 1u) << (g * (L & 31));
    if (live && li == 0) a.ok[s] = (bad & mine) == 0u;
    }
}

// The 12-state model: one CTA of four warps (one per scheduler) per scenario.  Per
// stage 7 + 7 + 6 FP64 instructions of the three products on every warp and 29 of the
// 4 x 4 system on the first (Gauss-Jordan, a column of [Quu | Qus qu] per lane; dense
// products took 24 + 24 + 4 and the inverse about 60).  The sweep splits each of the
// 16 rows of [F; K] over two lanes.  One step of 64 scenarios of horizon 40 takes 31 +
// 134 + 10 us in the three kernels (390 in one kernel of dense products), 256 of
// horizon 16 take 30 + 62 + 10 (239).
template <typename F>
__global__ void __launch_bounds__(128) k_traj_lq4(LqArgs2<F> a) {
    using Mp = RicMap<2>;
    constexpr int NS = Mp::NS, NU = Mp::NU, NZ = Mp::NZ, REC = Mp::REC, OUT = Mp::OUT, NT = 128;
    constexpr int PR = (REC + NT - 1) / NT, PO = (OUT + NT - 1) / NT;
    __shared__ F sm[Mp::SIZE];
    const int tid = threadIdx.x, lane = tid & 31, s = a.order[blockIdx.x];
    if (a.iter && blockIdx.x == 0 && tid == 0) *a.iter += 1;
    if (!a.active(s)) return;
    const int N = a.meta[s].N;
    F *scr = reinterpret_cast<F *>(a.scratch) + a.scratch0[s];
    typename LqSlotsOf<F, std::remove_cv_t<decltype(kRicTab<2, NT, 0>)>>::type prod_y;
    typename LqSlotsOf<F, std::remove_cv_t<decltype(kRicTab<2, NT, 1>)>>::type prod_m;
    typename LqSlotsOf<F, std::remove_cv_t<decltype(kRicTab<2, NT, 2>)>>::type prod_p;
    prod_y.load(kRicTab<2, NT, 0>, tid, sm);
    prod_m.load(kRicTab<2, NT, 1>, tid, sm);
    prod_p.load(kRicTab<2, NT, 2>, tid, sm);
    int om[PO];
#pragma unroll
    for (int r = 0; r < PO; ++r) om[r] = tid + NT * r < OUT ? kRicOut<2>.at[tid + NT * r] : 0;
    if (tid == 0) {
        sm[Mp::ZERO] = F(0);
        sm[Mp::ONE] = F(1);
        sm[Mp::DT] = a.dt;
        for (int x = 0; x < NU; ++x) sm[Mp::RU + x] = a.ru[x];
    }
    const F *rN = scr + Mp::rec(N), *r1 = scr + Mp::rec(N - 1);
    for (int e = tid; e < Mp::NSYM; e += NT) sm[Mp::P0 + e] = rN[Mp::rQ + e];
    for (int e = tid; e < NS; e += NT) sm[Mp::p0 + e] = rN[Mp::rq + e];
    for (int e = tid; e < REC; e += NT) sm[Mp::REC0 + e] = r1[e];
    bool ok = true;
    for (int t = N - 1; t >= 0; --t) {
        F nxt[PR];
        __syncthreads();
        if (t >= 1) {
            const F *rn = scr + Mp::rec(t - 1);
#pragma unroll
            for (int r = 0; r < PR; ++r)
                if (tid + NT * r < REC) nxt[r] = rn[tid + NT * r];
        }
        prod_y.run();
        __syncthreads();
        prod_m.run();
        __syncthreads();
        if (tid < 32) {
            // [K | k] = -Quu^-1 [Qus | qu]: lane c < 4 holds column c of Quu, lane 4 + j
            // column j of [Qus | qu].  Quu is positive definite iff every pivot is
            // positive; 1 takes the place of one that is not, the scenario fails.
            const int j = lane - NU;
            F v[NU];
#pragma unroll
            for (int i = 0; i < NU; ++i)
                v[i] = sm[lane < NU ? Mp::U0 + (i <= lane ? i * NU + lane : lane * NU + i) : Mp::H0 + i * (NS + 1) + min(j, NS)];
            if (j == NS)
#pragma unroll
                for (int i = 0; i < NU; ++i) v[i] += sm[Mp::HQ1 + i];
#pragma unroll
            for (int c = 0; c < NU; ++c) {
                F col[NU];
#pragma unroll
                for (int i = 0; i < NU; ++i) col[i] = __shfl_sync(0xffffffffu, v[i], c);
                const bool pd = positive_finite(col[c]);
                ok = ok && pd;
                v[c] *= pd ? recip(col[c]) : F(1);
#pragma unroll
                for (int i = 0; i < NU; ++i)
                    if (i != c) v[i] = fma(-col[i], v[c], v[i]);
            }
            if (j >= 0 && j <= NS)
#pragma unroll
                for (int i = 0; i < NU; ++i) sm[Mp::K0 + i * (NS + 1) + j] = -v[i];
        }
        __syncthreads();
        prod_p.run();
        __syncthreads();
        F *o = scr + Mp::out(N, t);
#pragma unroll
        for (int r = 0; r < PO; ++r)
            if (tid + NT * r < OUT) o[tid + NT * r] = sm[om[r]];
        __syncthreads();
        if (t >= 1) {
#pragma unroll
            for (int r = 0; r < PR; ++r)
                if (tid + NT * r < REC) sm[Mp::REC0 + tid + NT * r] = nxt[r];
        }
    }
    __syncthreads();  // the outputs of every thread are visible to the sweep
    if (tid >= 32) return;
    // forward sweep: lanes i and 16 + i own row i of [F; K], half of the sum each
    constexpr int AHEAD = 4, HN = NS / 2;
    const int i = lane & 15, half = lane >> 4;
    F x = i < NS ? scr[Mp::s0(N) + i] : F(0);
    F row[AHEAD][HN], fv[AHEAD];
    auto fetch = [&](int t, F (&r)[HN], F &f) {
        const F *o = scr + Mp::out(N, min(t, N - 1));
#pragma unroll
        for (int k = 0; k < HN; ++k) r[k] = o[i * NS + half * HN + k];
        f = half ? F(0) : o[NZ * NS + i];
    };
#pragma unroll
    for (int d = 0; d < AHEAD; ++d) fetch(d, row[d], fv[d]);
    bool fin = true;
    for (int t0 = 0; t0 < N; t0 += AHEAD) {
#pragma unroll
        for (int d = 0; d < AHEAD; ++d) {
            const int t = t0 + d;
            F v = fv[d];
#pragma unroll
            for (int k = 0; k < HN; ++k) v = fma(row[d][k], __shfl_sync(0xffffffffu, x, half * HN + k), v);
            v += __shfl_xor_sync(0xffffffffu, v, 16);
            x = v;
            if (t < N) {
                if (!half) scr[Mp::sol(N, t) + i] = v;
                fin = fin && finite(v);
            }
            fetch(t + AHEAD, row[d], fv[d]);
        }
    }
    const bool good = __all_sync(0xffffffffu, ok && fin);
    if (lane == 0) a.ok[s] = good;
}

// s, u from the sweep, then the box block and the poses of the new iterate
template <typename T, typename F, int KIND>
__global__ void __launch_bounds__(kTrajBlock) k_traj_apply(RicArgs<T> a, const int *lq_ok) {
    constexpr int NS = MDims<KIND>::NS, NU = MDims<KIND>::NU, NZ = NS + NU;
    using Mp = RicMap<KIND>;
    const int s = blockIdx.x, lane = threadIdx.x, NT = blockDim.x;
    if (a.scen_status[s] != kActive) return;
    const ScenMeta sm = a.meta[s];
    const int N = sm.N;
    const F *scr = reinterpret_cast<const F *>(a.scratch) + a.scratch0[s];
    const bool ok = lq_ok[s] != 0;
    double rpb = 0.0, rdb = 0.0;
    for (int t = lane; t < N; t += NT) {
        const F *sol = scr + Mp::sol(N, t);
        F v[NZ];
        T st[NS], ut[NU];
#pragma unroll
        for (int i = 0; i < NZ; ++i) v[i] = sol[i];
#pragma unroll
        for (int i = 0; i < NS; ++i) a.s[(long long)(sm.state0 + t + 1) * NS + i] = st[i] = T(v[i]);
#pragma unroll
        for (int i = 0; i < NU; ++i) a.u[(long long)(sm.ctrl0 + t) * NU + i] = ut[i] = T(v[NS + i]);
        if (ok) box_poses<T, KIND>(a, sm, t, st, ut, rpb, rdb);
    }
    if (!ok) {
        // k_traj_lq has advanced the counter: iteration j is *iter - 1
        __syncthreads();
        if (lane < 32) finish_scenario<T, KIND>(a, sm, s, OCA_SCEN_FAILED, *a.iter - 1, 0.0, 0.0);
        return;
    }
    __shared__ double part[kTrajBlock / 32][2];
    rpb = warp_sum(rpb);
    rdb = warp_sum(rdb);
    if ((lane & 31) == 0) {
        part[lane >> 5][0] = rpb;
        part[lane >> 5][1] = rdb;
    }
    __syncthreads();
    if (lane == 0) {
        for (int w = 1; w < NT / 32; ++w) {
            rpb += part[w][0];
            rdb += part[w][1];
        }
        a.box_res[2 * s] = rpb;
        a.box_res[2 * s + 1] = rdb;
    }
}

// Lanes per scenario: a warp of the recursion issues 22 (L = 32) or 24 (L = 16)
// FP64 instructions per stage, so 16 lanes carry nearly twice the scenarios; with
// no more scenarios than schedulers (4 per SM) every one has its own warp and 32
// lanes are the shorter chain (256 scenarios of horizon 50: 2,290 cycles per stage).
// 2,048 scenarios: 138 us with 16 lanes, 174 with 32.
template <typename F, int KIND>
void launch_lq_solve(const LqArgs2<F> &l, int n_sm, cudaStream_t st) {
    if constexpr (KIND == 2) {
        k_traj_lq4<F><<<l.n_scen, 128, 0, st>>>(l);
    } else {
        const bool one = l.n_scen <= 4 * n_sm;
        const int groups = one ? l.n_scen : (l.n_scen + 1) / 2, ctas = std::min(n_sm, groups);
        if (one) k_traj_lq<F, KIND, 32><<<ctas, 32 * kLqWarps, 0, st>>>(l);
        else k_traj_lq<F, KIND, 16><<<ctas, 32 * kLqWarps, 0, st>>>(l);
    }
}

// dt and the diagonal of Ru
template <typename T, typename F>
void lq_constants(LqArgs2<F> &l, const DevModel<T> &m, T damp, T rho_box, int nu) {
    l.dt = F(m.dt);
    for (int i = 0; i < nu; ++i)
        l.ru[i] = F(2) * F(m.Qu[i]) + F(damp) + (m.u_lo[i] > T(-1e29) || m.u_hi[i] < T(1e29) ? F(rho_box) : F(0));
}

template <typename T, typename F, int KIND>
cudaError_t launch_traj(const RicArgs<T> &a, int *lq_ok, const int *order, int max_n, int n_sm, cudaStream_t st) {
    LqArgs2<F> l;
    l.meta = a.meta;
    l.order = order;
    l.n_scen = a.n_scen;
    l.scen_status = a.scen_status;
    l.iters = nullptr;
    l.k = 0;
    l.scratch = a.scratch;
    l.scratch0 = a.scratch0;
    lq_constants<T, F>(l, a.model, a.damp, a.rho_box, MDims<KIND>::NU);
    l.ok = lq_ok;
    l.iter = a.iter;
    const int steps = std::min(kTrajBlock, (max_n + 1 + 31) / 32 * 32);
    k_traj_stage<T, F, KIND><<<a.n_scen, steps, sizeof(F) * steps * traj_rec_stride<F, KIND>(), st>>>(a);
    launch_lq_solve<F, KIND>(l, n_sm, st);
    k_traj_apply<T, F, KIND><<<a.n_scen, steps, 0, st>>>(a, lq_ok);
    return cudaGetLastError();
}

template <typename T, typename F>
cudaError_t launch_riccati_f(const RicArgs<T> &a, int *lq_ok, const int *order, int max_n, int n_sm, cudaStream_t st) {
    switch (a.model.kind) {
        case 0: return launch_traj<T, F, 0>(a, lq_ok, order, max_n, n_sm, st);
        case 1: return launch_traj<T, F, 1>(a, lq_ok, order, max_n, n_sm, st);
        case 2: return launch_traj<T, F, 2>(a, lq_ok, order, max_n, n_sm, st);
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_adj_lq(const AdjTrajArgs<T> &a, int n_scen, int *lq_ok, const int *order, int n_sm, cudaStream_t st) {
    LqArgs2<double> l;
    l.meta = a.meta;
    l.order = order;
    l.n_scen = n_scen;
    l.scen_status = nullptr;
    l.iters = a.iters;
    l.k = a.k;
    l.scratch = a.scratch;
    l.scratch0 = a.scratch0;
    lq_constants<T, double>(l, a.model, a.damp, a.rho_box, 2);
    l.ok = lq_ok;
    l.iter = nullptr;
    if (a.model.kind == 0) launch_lq_solve<double, 0>(l, n_sm, st);
    else if (a.model.kind == 1) launch_lq_solve<double, 1>(l, n_sm, st);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}
template cudaError_t launch_adj_lq<float>(const AdjTrajArgs<float> &, int, int *, const int *, int, cudaStream_t);
template cudaError_t launch_adj_lq<double>(const AdjTrajArgs<double> &, int, int *, const int *, int, cudaStream_t);

template <typename T>
cudaError_t launch_riccati(const RicArgs<T> &a, bool f32, int *lq_ok, const int *order, int max_n, int n_sm, cudaStream_t st) {
    if (f32) return launch_riccati_f<T, float>(a, lq_ok, order, max_n, n_sm, st);
    return launch_riccati_f<T, double>(a, lq_ok, order, max_n, n_sm, st);
}

template cudaError_t launch_riccati<float>(const RicArgs<float> &, bool, int *, const int *, int, int, cudaStream_t);
template cudaError_t launch_riccati<double>(const RicArgs<double> &, bool, int *, const int *, int, int, cudaStream_t);

}  // namespace oca
