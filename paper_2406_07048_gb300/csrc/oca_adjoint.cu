// Adjoint of a taped ADMM solve (reverse mode through the unrolled
// iterations of Sec. IV-B).  One iteration k maps
//   (s^k, u^k, y^k, zeta^{k-1}, xi^{k-1}, z^k, w^k)
// through
//   head  zeta^k = zeta^{k-1} + T(s^k, y^k),  xi^k = xi^{k-1} + R(s^k, y^k)
//   QP    y^{k+1} = pair QP at (pose(s^k), zeta^k, xi^k) with proximal centre y^k
//   stats Gauss-Newton statistics of y^{k+1}, zeta^k, xi^k per (part, t)
//   LQ    (s^{k+1}, u^{k+1}) = trajectory step linearised at (s^k, u^k)
//   box   z^{k+1} = clip((s,u)^{k+1} + w^k),  w^{k+1} = w^k + (s,u)^{k+1} - z^{k+1}
// and the reverse step k runs these backwards:
//   launch_adj_traj  box and LQ adjoints (the adjoint LQ has the forward
//               problem's matrices), then the chain rule through the
//               linearisation point (second derivatives of the dynamics and
//               of the part poses by dual numbers);
//   k_adj_pair  per pair: statistics, pair QP (implicit differentiation of
//               its optimality conditions in the (D+1)-dimensional dual form
//               the forward solver uses) and head adjoints, reduced to pose
//               adjoints per (part, t) and offset adjoints per obstacle face.
// The pair QP is differentiated on its active set, which is locally constant
// at strictly complementary solutions.
#include <algorithm>

#include "oca_common.cuh"
#include "oca_dual.cuh"
#include "oca_kernels.h"
#include "oca_ric.cuh"
#include "oca_ricprog.cuh"
#include "oca_solvers.cuh"

namespace oca {

// ============================================================================
// chain rule through the linearisation point
// ============================================================================

// (sb, ub) += dt * d/d(s, u) [ sum At .* fs(s, u) + Bt .* fu(s, u) ]: the
// adjoint of A_t = I + dt fs, B_t = dt fu and c_t = s + dt f - A_t s - B_t u
// with respect to the linearisation point, given At = Abar - cbar s^T and
// Bt = Bbar - cbar u^T.
template <typename T, int KIND>
__device__ void dyn_vjp(const DevModel<T> &m, const T *st, const T *ut, const T *At, const T *Bt, T *sb, T *ub) {
    constexpr int NS = MDims<KIND>::NS, NU = MDims<KIND>::NU;
    const DevModel<Dual<T>> dm = dual_model(m);
    for (int e = 0; e < NS + NU; ++e) {
        Dual<T> sd[NS], ud[NU], f[NS], fs[NS * NS], fu[NS * NU];
#pragma unroll
        for (int i = 0; i < NS; ++i) sd[i] = Dual<T>(st[i], i == e ? T(1) : T(0));
#pragma unroll
        for (int i = 0; i < NU; ++i) ud[i] = Dual<T>(ut[i], i + NS == e ? T(1) : T(0));
        dynamics<Dual<T>, KIND>(dm, sd, ud, f, fs, fu);
        T acc = T(0);
        for (int i = 0; i < NS * NS; ++i) acc += At[i] * fs[i].d;
        for (int i = 0; i < NS * NU; ++i) acc += Bt[i] * fu[i].d;
        if (e < NS) sb[e] += m.dt * acc;
        else ub[e - NS] += m.dt * acc;
    }
}

// Adjoint of the Gauss-Newton stage terms sigma Hs, sigma (g - Hs s) of one
// part (gn_part) given Qbar and qbar of the stage: G = Qbar - qbar s^T.
//   sb    += d/ds  sigma [G : Hs + qbar . g] - sigma Hs^T qbar
//   statb  = d/dstats sigma [G : Hs + qbar . g]   (the terms are linear in them)
template <typename T, int KIND>
__device__ void gn_vjp(const DevModel<T> &m, int link, const T *off, const T *st, const T *Wl, const T *Wc,
                       const T *E, const T *G, const T *qb, T sigma, T *sb, T *statb) {
    constexpr int NS = MDims<KIND>::NS, D = MDims<KIND>::D;
    constexpr int NW = StatDims<D>::NW, NSTAT = StatDims<D>::NSTAT;
    const DevModel<Dual<T>> dm = dual_model(m);
    Dual<T> offd[D], sd[NS], stat[NSTAT], Hs[NS * NS], g[NS];
#pragma unroll
    for (int i = 0; i < D; ++i) offd[i] = Dual<T>(off[i]);
#pragma unroll
    for (int i = 0; i < NW; ++i) stat[i] = Dual<T>(Wl[i]);
#pragma unroll
    for (int i = 0; i < D; ++i) stat[NW + i] = Dual<T>(Wc[i]);
#pragma unroll
    for (int i = 0; i < D * D; ++i) stat[NW + D + i] = Dual<T>(E[i]);
    for (int e = 0; e < NS; ++e) {
#pragma unroll
        for (int i = 0; i < NS; ++i) sd[i] = Dual<T>(st[i], i == e ? T(1) : T(0));
        gn_part<Dual<T>, KIND>(dm, link, offd, sd, stat, stat + NW, stat + NW + D, Hs, g);
        T acc = T(0);
        for (int i = 0; i < NS * NS; ++i) acc += G[i] * Hs[i].d;
        for (int i = 0; i < NS; ++i) acc += qb[i] * (g[i].d - Hs[i * NS + e].v);
        sb[e] += sigma * acc;
    }
#pragma unroll
    for (int i = 0; i < NS; ++i) sd[i] = Dual<T>(st[i]);
    for (int kk = 0; kk < NSTAT; ++kk) {
        stat[kk].d = T(1);
        gn_part<Dual<T>, KIND>(dm, link, offd, sd, stat, stat + NW, stat + NW + D, Hs, g);
        stat[kk].d = T(0);
        T acc = T(0);
        for (int i = 0; i < NS * NS; ++i) acc += G[i] * Hs[i].d;
        for (int i = 0; i < NS; ++i) acc += qb[i] * g[i].d;
        statb[kk] = sigma * acc;
    }
}

// ============================================================================
// seed: adjoint of the trajectory cost F of eqn:navigation_cost at s^K, u^K
// ============================================================================
template <typename T, int KIND>
__global__ void __launch_bounds__(32) k_adj_seed(AdjTrajArgs<T> a) {
    constexpr int NS = MDims<KIND>::NS, NU = MDims<KIND>::NU;
    const int s = blockIdx.x, lane = threadIdx.x;
    const ScenMeta sm = a.meta[s];
    const int K = a.iters[s];
    const T *sK = a.tape.s + (long long)K * a.tape.s_slot, *uK = a.tape.u + (long long)K * a.tape.u_slot;
    const T gc = a.grad_cost[s];
    for (int t = lane; t <= sm.N; t += 32) {
        for (int i = 0; i < NS; ++i) {
            const long long k2 = (long long)(sm.state0 + t) * NS + i;
            const T v = gc * T(2) * a.model.Qs[i] * (sK[k2] - a.s_ref[k2]);
            if (t == 0) a.gs0[(long long)s * NS + i] += double(v);
            else a.sb[k2] = v;
        }
        if (t < sm.N)
            for (int i = 0; i < NU; ++i) {
                const long long k2 = (long long)(sm.ctrl0 + t) * NU + i;
                a.ub[k2] = gc * T(2) * a.model.Qu[i] * uK[k2];
            }
    }
}

// ============================================================================
// reverse step k of the trajectory side, 12-state model (one warp per scenario)
// ============================================================================
template <typename T, typename F, int KIND>
__global__ void __launch_bounds__(32) k_adj_traj(AdjTrajArgs<T> a) {
    constexpr int NS = MDims<KIND>::NS, NU = MDims<KIND>::NU, D = MDims<KIND>::D, NROT = MDims<KIND>::NROT;
    constexpr int NW = StatDims<D>::NW, NSTAT = StatDims<D>::NSTAT;
    using LY = RicLayout<NS, NU>;
    const int s = blockIdx.x, lane = threadIdx.x;
    const int k = a.k;
    if (k >= a.iters[s]) return;
    const ScenMeta sm = a.meta[s];
    const int N = sm.N;
    const TapeView<T> &tp = a.tape;
    const T *s_k = tp.s + (long long)k * tp.s_slot, *u_k = tp.u + (long long)k * tp.u_slot;
    const T *s_k1 = tp.s + (long long)(k + 1) * tp.s_slot, *u_k1 = tp.u + (long long)(k + 1) * tp.u_slot;
    const T *zs_k = tp.box + (long long)k * tp.box_slot;
    const T *ws_k = zs_k + tp.n_states * NS, *zu_k = ws_k + tp.n_states * NS, *wu_k = zu_k + tp.n_ctrls * NU;
    const T *stats_k = tp.stats + (long long)k * tp.stats_slot;
    F *scr = reinterpret_cast<F *>(a.scratch) + a.scratch0[s];

    // ---- 1. pose adjoints of s^{k+1} (pair side of iteration k+1) into sbar^{k+1}
    for (int t = 1 + lane; t <= N; t += 32) {
        T st[NS], acc[NS];
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            st[i] = s_k1[(long long)(sm.state0 + t) * NS + i];
            acc[i] = T(0);
        }
        for (int part = 0; part < sm.NP; ++part) {
            const int gp = sm.part0 + part;
            T off[D], rho[D], R[D * D], drho[D * NS], dR[NROT][D * D];
            int ridx[NROT];
#pragma unroll
            for (int i = 0; i < D; ++i) off[i] = a.g.part_off[gp * D + i];
            part_pose<T, KIND>(a.model, a.g.part_link[gp], off, st, rho, R, drho, dR, ridx);
            const long long col = sm.qbeg + part * N + (t - 1);
            for (int i = 0; i < D; ++i) {
                const T rb = a.poseb[(long long)i * a.Qtot + col];
                for (int e = 0; e < NS; ++e) acc[e] += rb * drho[i * NS + e];
            }
#pragma unroll
            for (int r = 0; r < NROT; ++r) {
                T v = T(0);
#pragma unroll
                for (int i = 0; i < D * D; ++i) v += a.poseb[(long long)(D + i) * a.Qtot + col] * dR[r][i];
                acc[ridx[r]] += v;
            }
        }
        for (int i = 0; i < NS; ++i) a.sb[(long long)(sm.state0 + t) * NS + i] += acc[i];
    }
    // ---- 2. box update of iteration k (z = clip(x + w), w += x - z)
    const int n_box = a.rho_box > T(0) ? N * NS + N * NU : 0;
    for (int e = lane; e < n_box; e += 32) {
        long long k2;
        T lo, hi, x, w;
        T *xb, *zb, *wb;
        if (e < N * NS) {
            const int t = 1 + e / NS, i = e % NS;
            lo = a.model.s_lo[i];
            hi = a.model.s_hi[i];
            k2 = (long long)(sm.state0 + t) * NS + i;
            x = s_k1[k2];
            w = ws_k[k2];
            xb = a.sb;
            zb = a.zsb;
            wb = a.wsb;
        } else {
            const int e2 = e - N * NS, t = e2 / NU, i = e2 % NU;
            lo = a.model.u_lo[i];
            hi = a.model.u_hi[i];
            k2 = (long long)(sm.ctrl0 + t) * NU + i;
            x = u_k1[k2];
            w = wu_k[k2];
            xb = a.ub;
            zb = a.zub;
            wb = a.wub;
        }
        if (!bounded(lo, hi)) continue;
        const T wbar = wb[k2], zp = zb[k2] - wbar, v = x + w;
        T xa = xb[k2] + wbar, wn = wbar;
        if (v > lo && v < hi) {
            xa += zp;
            wn += zp;
        }
        xb[k2] = xa;
        wb[k2] = wn;
        zb[k2] = T(0);
    }
    __syncwarp();
    // ---- 3. the LQ problem of iteration k, rebuilt from the tape
    StageParams<T> sp;
    sp.model = a.model;
    sp.g = a.g;
    sp.sigma = a.sigma;
    sp.rho_box = a.rho_box;
    sp.damp = a.damp;
    sp.s_ref = a.s_ref;
    sp.Qtot = a.Qtot;
    StageSrc<T> src;
    src.s = s_k;
    src.u = u_k;
    src.zs = zs_k;
    src.ws = ws_k;
    src.zu = zu_k;
    src.wu = wu_k;
    src.stats = stats_k;
    for (int t = lane; t <= N; t += 32) assemble_stage<T, F, KIND>(sp, src, sm, t, scr);
    __syncwarp();
    // ---- 4. costates of its solution (s^{k+1}, u^{k+1})
    {
        auto xf = [&](int t, int i) -> F { return F(s_k1[(long long)(sm.state0 + t) * NS + i]); };
        ric_costates<F, NS, NU, false>(scr, N, xf);
    }
    // ---- 5. adjoint LQ: same Q, Ru, A, B; linear terms -sbar, -ubar; c = 0; s_0 = 0
    for (int t = lane; t <= N; t += 32) {
        for (int i = 0; i < NS; ++i)
            scr[LY::q(N, t) + i] = t >= 1 ? -F(a.sb[(long long)(sm.state0 + t) * NS + i]) : F(0);
        if (t < N) {
            for (int i = 0; i < NU; ++i) scr[LY::r(N, t) + i] = -F(a.ub[(long long)(sm.ctrl0 + t) * NU + i]);
            for (int i = 0; i < NS; ++i) scr[LY::c(N, t) + i] = F(0);
        }
    }
    // sbar of the fixed initial state passes straight to the initial-state adjoint
    if (lane < NS) {
        const long long k2 = (long long)sm.state0 * NS + lane;
        a.gs0[(long long)s * NS + lane] += double(a.sb[k2]);
        a.sb[k2] = T(0);
    }
    __syncwarp();
    // diagonal of Ru in shared memory, as in the forward kernel
    __shared__ F ru_diag[NU];
    for (int i = lane; i < NU; i += 32)
        ru_diag[i] = F(2) * F(a.model.Qu[i]) + F(a.damp) +
                     (bounded(a.model.u_lo[i], a.model.u_hi[i]) ? F(a.rho_box) : F(0));
    __syncwarp();
    ric_factor<F, NS, NU>(scr, N, ru_diag);
    __shared__ F sc[NS];
    for (int i = lane; i < NS; i += 32) {
        sc[i] = F(0);
        scr[LY::xs(N, 0) + i] = F(0);
    }
    __syncwarp();
    struct Out {
        F *scr;
        int N;
        __device__ void put_u(int t, int i, F v) { scr[LY::xu(N, t) + i] = v; }
        __device__ void put_s(int t, int i, F v) { scr[LY::xs(N, t) + i] = v; }
    } out{scr, N};
    ric_sweep<F, NS, NU>(scr, N, sc, out);
    {
        auto xa = [&](int t, int i) -> F { return scr[LY::xs(N, t) + i]; };
        ric_costates<F, NS, NU, true>(scr, N, xa);
    }
    __syncwarp();
    // ---- 6. data adjoints of the LQ and the chain rule into iterate k
    //   Abar_t = -(pa_{t+1} s_t^T + pf_{t+1} xs_t^T), Bbar_t = -(pa_{t+1} u_t^T + pf_{t+1} xu_t^T),
    //   cbar_t = -pa_{t+1}, rbar_t = -xu_t, qbar_t = -xs_t, Qbar_t = -xs_t s_t^T
    // with (s, u) = (s^{k+1}, u^{k+1}), (xs, xu) the adjoint solution and
    // pf, pa the forward and adjoint costates.
    const T rho_b = a.rho_box, damp = a.damp;
    for (int t = lane; t <= N; t += 32) {
        T sbk[NS], ubk[NU], skt[NS], ukt[NU];
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            sbk[i] = T(0);
            skt[i] = s_k[(long long)(sm.state0 + t) * NS + i];
        }
#pragma unroll
        for (int i = 0; i < NU; ++i) {
            ubk[i] = T(0);
            ukt[i] = t < N ? u_k[(long long)(sm.ctrl0 + t) * NU + i] : T(0);
        }
        if (t < N) {
            F pf1[NS], pa1[NS], xt[NS], xh[NS], uh[NU], ut1[NU];
            for (int i = 0; i < NS; ++i) {
                pf1[i] = scr[LY::pf(N, t + 1) + i];
                pa1[i] = scr[LY::pa(N, t + 1) + i];
                xt[i] = F(s_k1[(long long)(sm.state0 + t) * NS + i]);
                xh[i] = scr[LY::xs(N, t) + i];
            }
            for (int i = 0; i < NU; ++i) {
                uh[i] = scr[LY::xu(N, t) + i];
                ut1[i] = F(u_k1[(long long)(sm.ctrl0 + t) * NU + i]);
            }
            T At[NS * NS], Bt[NS * NU];
            for (int i = 0; i < NS; ++i) {
                const F cb = -pa1[i];
                for (int j = 0; j < NS; ++j) At[i * NS + j] = T(-(pa1[i] * xt[j] + pf1[i] * xh[j]) - cb * F(skt[j]));
                for (int j = 0; j < NU; ++j) Bt[i * NU + j] = T(-(pa1[i] * ut1[j] + pf1[i] * uh[j]) - cb * F(ukt[j]));
            }
            dyn_vjp<T, KIND>(a.model, skt, ukt, At, Bt, sbk, ubk);
            for (int i = 0; i < NU; ++i) {
                const T rb = T(-uh[i]);
                ubk[i] -= damp * rb;
                if (rho_b > T(0) && bounded(a.model.u_lo[i], a.model.u_hi[i])) {
                    const long long k2 = (long long)(sm.ctrl0 + t) * NU + i;
                    a.zub[k2] = -rho_b * rb;
                    a.wub[k2] += rho_b * rb;
                }
            }
            if (t == 0) {
                // s_0 enters the first dynamics constraint as data: -A_0^T pa_1
                const F *A0 = scr + LY::A(N, 0);
                for (int j = 0; j < NS; ++j) {
                    F acc = F(0);
                    for (int i = 0; i < NS; ++i) acc -= A0[i * NS + j] * pa1[i];
                    sbk[j] += T(acc);
                }
            }
        }
        if (t >= 1) {
            T qb[NS], G[NS * NS];
            for (int i = 0; i < NS; ++i) {
                const F xh = scr[LY::xs(N, t) + i];
                qb[i] = T(-xh);
                for (int j = 0; j < NS; ++j)
                    G[i * NS + j] = T(-xh * F(s_k1[(long long)(sm.state0 + t) * NS + j])) - qb[i] * skt[j];
            }
            for (int i = 0; i < NS; ++i) {
                sbk[i] -= damp * qb[i];
                if (rho_b > T(0) && bounded(a.model.s_lo[i], a.model.s_hi[i])) {
                    const long long k2 = (long long)(sm.state0 + t) * NS + i;
                    a.zsb[k2] = -rho_b * qb[i];
                    a.wsb[k2] += rho_b * qb[i];
                }
            }
            for (int part = 0; part < sm.NP; ++part) {
                const int gp = sm.part0 + part;
                const long long col = sm.qbeg + part * N + (t - 1);
                T off[D], Wl[NW], Wc[D], E[D * D], statb[NSTAT];
#pragma unroll
                for (int i = 0; i < D; ++i) off[i] = a.g.part_off[gp * D + i];
#pragma unroll
                for (int i = 0; i < NW; ++i) Wl[i] = stats_k[(long long)i * a.Qtot + col];
#pragma unroll
                for (int i = 0; i < D; ++i) Wc[i] = stats_k[(long long)(NW + i) * a.Qtot + col];
#pragma unroll
                for (int i = 0; i < D * D; ++i) E[i] = stats_k[(long long)(NW + D + i) * a.Qtot + col];
                gn_vjp<T, KIND>(a.model, a.g.part_link[gp], off, skt, Wl, Wc, E, G, qb, a.sigma, sbk, statb);
#pragma unroll
                for (int i = 0; i < NSTAT; ++i) a.statsb[(long long)i * a.Qtot + col] = statb[i];
            }
        }
        if (t == 0) {
            for (int i = 0; i < NS; ++i) a.gs0[(long long)s * NS + i] += double(sbk[i]);
        } else {
            for (int i = 0; i < NS; ++i) a.sb[(long long)(sm.state0 + t) * NS + i] = sbk[i];
        }
        if (t < N)
            for (int i = 0; i < NU; ++i) a.ub[(long long)(sm.ctrl0 + t) * NU + i] = ubk[i];
    }
}

// ============================================================================
// reverse step k of the trajectory side, 2-D models: four kernels instead of one warp
// per scenario doing everything (the LQ solve is the forward step's k_traj_lq).
//   k_adj_pre      pose adjoints, box update, the stage records of the adjoint LQ
//                  (lanes over t)
//   k_traj_lq      its solution (xs, xu)
//   k_adj_costate  costates of the forward and the adjoint solution (a warp each)
//   k_adj_post     data adjoints and the chain rule into iterate k: a thread per
//                  (step, direction), and the statistics' adjoints in closed form
// Bound by FP64 issue in the chains.  256 trailer scenarios of horizon 50, a reverse
// step: 358 us as one kernel, now 18 + 60 + 37 + 32 (gradient call 2.13 -> 1.78 ms).
// ============================================================================
constexpr int kAdjBlock = 96;

template <typename T, typename F, int KIND>
__global__ void __launch_bounds__(kAdjBlock) k_adj_pre(AdjTrajArgs<T> a) {
    constexpr int NS = MDims<KIND>::NS, NU = MDims<KIND>::NU, D = MDims<KIND>::D, NROT = MDims<KIND>::NROT;
    using Mp = RicMap<KIND>;
    const int s = blockIdx.x, k = a.k;
    if (k >= a.iters[s]) return;
    const ScenMeta sm = a.meta[s];
    const int N = sm.N;
    const TapeView<T> &tp = a.tape;
    const T *s_k = tp.s + (long long)k * tp.s_slot, *u_k = tp.u + (long long)k * tp.u_slot;
    const T *s_k1 = tp.s + (long long)(k + 1) * tp.s_slot, *u_k1 = tp.u + (long long)(k + 1) * tp.u_slot;
    const T *zs_k = tp.box + (long long)k * tp.box_slot;
    const T *ws_k = zs_k + tp.n_states * NS, *zu_k = ws_k + tp.n_states * NS, *wu_k = zu_k + tp.n_ctrls * NU;
    F *scr = reinterpret_cast<F *>(a.scratch) + a.scratch0[s];
    StageParams<T> sp;
    sp.model = a.model;
    sp.g = a.g;
    sp.sigma = a.sigma;
    sp.rho_box = a.rho_box;
    sp.damp = a.damp;
    sp.s_ref = a.s_ref;
    sp.Qtot = a.Qtot;
    StageSrc<T> src;
    src.s = s_k;
    src.u = u_k;
    src.zs = zs_k;
    src.ws = ws_k;
    src.zu = zu_k;
    src.wu = wu_k;
    src.stats = tp.stats + (long long)k * tp.stats_slot;
    struct Sink {
        F *r;
        F x[NS], g[NS];  // s^{k+1}_t; Q x + q
        __device__ void A(int i, int j, T v) {
            const int e = RicSparse<KIND>::a_slot(i, j);
            if (e >= 0) r[Mp::rA + e] = F(v);
        }
        __device__ void B(int i, int j, T v) {
            const int e = RicSparse<KIND>::b_slot(i, j);
            if (e >= 0) r[Mp::rB + e] = F(v);
        }
        __device__ void c(int, T) {}
        __device__ void u(int, T) {}
        __device__ void Q(int i, int j, T v) {
            if (i <= j) r[Mp::rQ + Mp::sym(i, j)] = F(v);
            g[i] = j == 0 ? F(v) * x[0] : fma(F(v), x[j], g[i]);
        }
        __device__ void q(int i, T v) { g[i] += F(v); }
    };
    for (int t = threadIdx.x; t <= N; t += blockDim.x) {
        // pose adjoints of s^{k+1} (pair side of iteration k+1), then the box update of
        // iteration k (z = clip(x + w), w += x - z)
        const long long ks = (long long)(sm.state0 + t) * NS, ku = (long long)(sm.ctrl0 + t) * NU;
        T st[NS], sb[NS], ub[NU];
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            st[i] = s_k1[ks + i];
            sb[i] = a.sb[ks + i];
        }
        if (t >= 1) {
            T acc[NS];
#pragma unroll
            for (int i = 0; i < NS; ++i) acc[i] = T(0);
            for (int part = 0; part < sm.NP; ++part) {
                const int gp = sm.part0 + part;
                T off[D], rho[D], R[D * D], drho[D * NS], dR[NROT][D * D];
                int ridx[NROT];
#pragma unroll
                for (int i = 0; i < D; ++i) off[i] = a.g.part_off[gp * D + i];
                part_pose<T, KIND>(a.model, a.g.part_link[gp], off, st, rho, R, drho, dR, ridx);
                const long long col = sm.qbeg + part * N + (t - 1);
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    const T rb = a.poseb[(long long)i * a.Qtot + col];
#pragma unroll
                    for (int e = 0; e < NS; ++e) acc[e] += rb * drho[i * NS + e];
                }
                T v = T(0);
#pragma unroll
                for (int i = 0; i < D * D; ++i) v += a.poseb[(long long)(D + i) * a.Qtot + col] * dR[0][i];
#pragma unroll
                for (int e = 0; e < NS; ++e)
                    if (e == ridx[0]) acc[e] += v;
            }
#pragma unroll
            for (int i = 0; i < NS; ++i) sb[i] += acc[i];
        }
        const bool box = a.rho_box > T(0);
        auto unbox = [&](T x, T lo, T hi, T w, T *zb, T *wb, T &xb) {
            const T wbar = *wb, zp = *zb - wbar, v = x + w;
            T xa = xb + wbar, wn = wbar;
            if (v > lo && v < hi) {
                xa += zp;
                wn += zp;
            }
            xb = xa;
            *wb = wn;
            *zb = T(0);
        };
        if (t >= 1 && box)
#pragma unroll
            for (int i = 0; i < NS; ++i)
                if (bounded(a.model.s_lo[i], a.model.s_hi[i]))
                    unbox(st[i], a.model.s_lo[i], a.model.s_hi[i], ws_k[ks + i], a.zsb + ks + i, a.wsb + ks + i, sb[i]);
        F *rec = scr + Mp::rec(t);
        if (t < N) {
#pragma unroll
            for (int i = 0; i < NU; ++i) {
                ub[i] = a.ub[ku + i];
                if (box && bounded(a.model.u_lo[i], a.model.u_hi[i]))
                    unbox(u_k1[ku + i], a.model.u_lo[i], a.model.u_hi[i], wu_k[ku + i], a.zub + ku + i, a.wub + ku + i, ub[i]);
                rec[Mp::rr + i] = -F(ub[i]);
            }
#pragma unroll
            for (int i = 0; i < NS; ++i) rec[Mp::rc + i] = F(0);
        }
        // the adjoint LQ has the forward one's Q, Ru, A, B, linear terms -sbar, -ubar, c = 0
        // and s_0 = 0; sbar of the fixed initial state passes to the initial-state adjoint
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            rec[Mp::rq + i] = t >= 1 ? -F(sb[i]) : F(0);
            if (t == 0) {
                a.gs0[(long long)s * NS + i] += double(sb[i]);
                scr[Mp::s0(N) + i] = F(0);
            }
        }
        Sink out;
        out.r = rec;
#pragma unroll
        for (int i = 0; i < NS; ++i) out.x[i] = F(st[i]);
        assemble_terms<T, KIND>(sp, src, sm, t, out);
#pragma unroll
        for (int i = 0; i < NS; ++i) scr[Mp::adj(N, 0, t) + i] = out.g[i];
    }
}

// Costates pi_t = g_t + A_t^T pi_{t+1}, g_t = Q_t x_t + q_t, of the forward solution
// (g from k_adj_pre; warp 0) and of the adjoint one (g formed here first; warp 1).
// Lane i owns pi_i; the steps' coefficients are on their way four steps ahead.
template <typename F, int KIND>
__global__ void __launch_bounds__(64) k_adj_costate(const ScenMeta *meta, const int *iters, int k, void *scratch,
                                                    const long long *scratch0) {
    constexpr int NS = MDims<KIND>::NS, AHEAD = 4;
    using Mp = RicMap<KIND>;
    const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, which = tid >> 5;
    if (k >= iters[s]) return;
    const int N = meta[s].N;
    F *scr = reinterpret_cast<F *>(scratch) + scratch0[s];
    for (int e = tid; e < N * NS; e += 64) {
        const int t = 1 + e / NS, i = e % NS;
        const F *rec = scr + Mp::rec(t), *x = scr + Mp::sol(N, t - 1);  // xs_t
        F acc = rec[Mp::rq + i];
#pragma unroll
        for (int j = 0; j < NS; ++j) acc = fma(rec[Mp::rQ + Mp::sym(i, j)], x[j], acc);
        scr[Mp::adj(N, 1, t) + i] = acc;
    }
    __syncthreads();
    const int i = lane < NS ? lane : 0;
    int slot[NS];  // where A[l][i] is read: record entry, or -1: 0, -2: 1
#pragma unroll
    for (int l = 0; l < NS; ++l) {
        const int e = RicSparse<KIND>::a_slot(l, i);
        slot[l] = e >= 0 ? e : l == i ? -2 : -1;
    }
    F col[AHEAD][NS], g[AHEAD];
    auto fetch = [&](int t, F (&c)[NS], F &gt) {  // step t: pi_t from pi_{t+1}
        const int tc = max(t, 1);
        const F *rec = scr + Mp::rec(min(tc, N - 1));  // t = N: pi_{N+1} = 0
#pragma unroll
        for (int l = 0; l < NS; ++l) c[l] = slot[l] >= 0 ? rec[Mp::rA + slot[l]] : slot[l] == -2 ? F(1) : F(0);
        gt = scr[Mp::adj(N, which, tc) + i];
    };
    F pi = F(0);
#pragma unroll
    for (int d = 0; d < AHEAD; ++d) fetch(N - d, col[d], g[d]);
    for (int t0 = N; t0 >= 1; t0 -= AHEAD) {
#pragma unroll
        for (int d = 0; d < AHEAD; ++d) {
            const int t = t0 - d;
            F v = g[d];
#pragma unroll
            for (int l = 0; l < NS; ++l) v = fma(col[d][l], __shfl_sync(0xffffffffu, pi, l), v);
            if (t >= 1) {
                pi = v;
                if (lane < NS) scr[Mp::adj(N, 2 + which, t) + lane] = v;
            }
            fetch(t - AHEAD, col[d], g[d]);
        }
    }
}

// Per step t, with (s, u) = (s^{k+1}, u^{k+1}), (xs, xu) the adjoint solution, pf, pa the
// costates and the linearisation point (s^k, u^k):
//   At = Abar - cbar s_k^T, Bt = Bbar - cbar u_k^T (Abar = -(pa s^T + pf xs^T),
//   Bbar = -(pa u^T + pf xu^T), cbar = -pa), qb = -xs, G = -xs s^T - qb s_k^T,
// then a thread per (step, direction e) of (s^k, u^k): d/de of At : fs + Bt : fu (dual
// numbers), the damping and box terms, and for e in s^k the Gauss-Newton terms of every
// part; and a thread per (step, part) for the statistics' adjoints, in closed form since
// the terms are linear in W, Wc and E.
constexpr int kPostSteps = 32, kPostThreads = 256;
template <typename T, typename F, int KIND>
__global__ void __launch_bounds__(kPostThreads) k_adj_post(AdjTrajArgs<T> a) {
    constexpr int NS = MDims<KIND>::NS, NU = MDims<KIND>::NU, D = MDims<KIND>::D, NROT = MDims<KIND>::NROT, NZ = NS + NU;
    constexpr int NW = StatDims<D>::NW, NSTAT = StatDims<D>::NSTAT;
    constexpr int oB = NS * NS, oG = oB + NS * NU, oq = oG + NS * NS, W = (oq + NS) | 1;
    using Mp = RicMap<KIND>;
    __shared__ T mat[kPostSteps * W];  // At, Bt, G, qb of each step
    const int s = blockIdx.x, tid = threadIdx.x, k = a.k;
    if (k >= a.iters[s]) return;
    const ScenMeta sm = a.meta[s];
    const int N = sm.N, t0 = blockIdx.y * kPostSteps, nt = min(kPostSteps, N + 1 - t0);
    if (nt <= 0) return;
    const TapeView<T> &tp = a.tape;
    const T *s_k = tp.s + (long long)k * tp.s_slot, *u_k = tp.u + (long long)k * tp.u_slot;
    const T *s_k1 = tp.s + (long long)(k + 1) * tp.s_slot, *u_k1 = tp.u + (long long)(k + 1) * tp.u_slot;
    const T *stats_k = tp.stats + (long long)k * tp.stats_slot;
    const F *scr = reinterpret_cast<const F *>(a.scratch) + a.scratch0[s];
    // xs_t, xu_t: rows [s_{t+1}, u_t] of the solution
    auto xs = [&](int t, int i) -> F { return t >= 1 ? scr[Mp::sol(N, t - 1) + i] : F(0); };
    for (int e = tid; e < nt * NS; e += kPostThreads) {
        // row i of the matrices of step t
        const int t = t0 + e / NS, i = e % NS;
        T *m = mat + (t - t0) * W;
        const long long ks = (long long)(sm.state0 + t) * NS, ku = (long long)(sm.ctrl0 + t) * NU;
        if (t < N) {
            const F pf1 = scr[Mp::adj(N, 2, t + 1) + i], pa1 = scr[Mp::adj(N, 3, t + 1) + i], cb = -pa1;
#pragma unroll
            for (int j = 0; j < NS; ++j)
                m[i * NS + j] = T(-(pa1 * F(s_k1[ks + j]) + pf1 * xs(t, j)) - cb * F(s_k[ks + j]));
#pragma unroll
            for (int j = 0; j < NU; ++j)
                m[oB + i * NU + j] = T(-(pa1 * F(u_k1[ku + j]) + pf1 * scr[Mp::sol(N, t) + NS + j]) - cb * F(u_k[ku + j]));
        }
        const F xh = xs(t, i);
        const T qb = T(-xh);
        m[oq + i] = qb;
#pragma unroll
        for (int j = 0; j < NS; ++j) m[oG + i * NS + j] = T(-xh * F(s_k1[ks + j])) - qb * s_k[ks + j];
    }
    __syncthreads();
    const T rho_b = a.rho_box, damp = a.damp;
    const int n_dir = nt * NZ, n_item = n_dir + nt * sm.NP;
    for (int item = tid; item < n_item; item += kPostThreads) {
        const bool dir = item < n_dir;
        // directions of one kind side by side: the lanes of a warp share a path
        const int t = t0 + (dir ? item % nt : (item - n_dir) % nt);
        const T *m = mat + (t - t0) * W, *qb = m + oq, *G = m + oG;
        const long long ks = (long long)(sm.state0 + t) * NS, ku = (long long)(sm.ctrl0 + t) * NU;
        T st[NS];
#pragma unroll
        for (int i = 0; i < NS; ++i) st[i] = s_k[ks + i];
        if (!dir) {
            const int part = (item - n_dir) / nt;
            if (t == 0) continue;
            const int gp = sm.part0 + part;
            T off[D], rho[D], R[D * D], drho[D * NS], dR[NROT][D * D];
            int ridx[NROT];
#pragma unroll
            for (int i = 0; i < D; ++i) off[i] = a.g.part_off[gp * D + i];
            part_pose<T, KIND>(a.model, a.g.part_link[gp], off, st, rho, R, drho, dR, ridx);
            T v[D], qa = T(0), gaa = T(0), Wb[D][D];
#pragma unroll
            for (int i = 0; i < D; ++i) v[i] = T(0);
#pragma unroll
            for (int e = 0; e < NS; ++e) {
#pragma unroll
                for (int i = 0; i < D; ++i) v[i] += qb[e] * drho[i * NS + e];
                if (e == ridx[0]) {
                    qa = qb[e];
                    gaa = G[e * NS + e];
                }
            }
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    T acc = v[i] * rho[j];
#pragma unroll
                    for (int e = 0; e < NS; ++e) {
                        T gd = T(0);
#pragma unroll
                        for (int f = 0; f < NS; ++f) gd += G[e * NS + f] * drho[j * NS + f];
                        acc += drho[i * NS + e] * gd;
                    }
#pragma unroll
                    for (int l = 0; l < D; ++l) acc += dR[0][i * D + l] * (gaa * dR[0][j * D + l] + qa * R[j * D + l]);
                    Wb[i][j] = acc;
                }
            const long long col = sm.qbeg + part * N + (t - 1);
            int kk = 0;
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int j = 0; j <= i; ++j, ++kk)
                    a.statsb[(long long)kk * a.Qtot + col] = a.sigma * (i == j ? Wb[i][i] : Wb[i][j] + Wb[j][i]);
#pragma unroll
            for (int i = 0; i < D; ++i) a.statsb[(long long)(NW + i) * a.Qtot + col] = -a.sigma * v[i];
#pragma unroll
            for (int i = 0; i < D * D; ++i) a.statsb[(long long)(NW + D + i) * a.Qtot + col] = a.sigma * qa * dR[0][i];
            continue;
        }
        const int e = item / nt;
        T out = T(0);
        if (t < N) {
            const DevModel<Dual<T>> dm = dual_model(a.model);
            Dual<T> sd[NS], ud[NU], f[NS], fs[NS * NS], fu[NS * NU];
#pragma unroll
            for (int i = 0; i < NS; ++i) sd[i] = Dual<T>(st[i], i == e ? T(1) : T(0));
#pragma unroll
            for (int i = 0; i < NU; ++i) ud[i] = Dual<T>(u_k[ku + i], i + NS == e ? T(1) : T(0));
            dynamics<Dual<T>, KIND>(dm, sd, ud, f, fs, fu);
            T acc = T(0);
#pragma unroll
            for (int i = 0; i < NS * NS; ++i) acc += m[i] * fs[i].d;
#pragma unroll
            for (int i = 0; i < NS * NU; ++i) acc += m[oB + i] * fu[i].d;
            out += a.model.dt * acc;
        }
        if (e >= NS) {
            if (t == N) continue;
            const int i = e - NS;
            const T rb = T(-scr[Mp::sol(N, t) + NS + i]);
            out -= damp * rb;
            if (rho_b > T(0) && bounded(a.model.u_lo[i], a.model.u_hi[i])) {
                a.zub[ku + i] = -rho_b * rb;
                a.wub[ku + i] += rho_b * rb;
            }
            a.ub[ku + i] = out;
            continue;
        }
        if (t == 0) {
            // s_0 enters the first dynamics constraint as data: -A_0^T pa_1
            const F *rec = scr + Mp::rec(0);
            F acc = F(0);
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                const int sl = RicSparse<KIND>::a_slot(i, e);
                const F A0 = sl >= 0 ? rec[Mp::rA + sl] : i == e ? F(1) : F(0);
                acc -= A0 * scr[Mp::adj(N, 3, 1) + i];
            }
            out += T(acc);
            a.gs0[(long long)s * NS + e] += double(out);
            a.sb[ks + e] = T(0);
            continue;
        }
        const T qe = qb[e];
        out -= damp * qe;
        if (rho_b > T(0) && bounded(a.model.s_lo[e], a.model.s_hi[e])) {
            a.zsb[ks + e] = -rho_b * qe;
            a.wsb[ks + e] += rho_b * qe;
        }
        for (int part = 0; part < sm.NP; ++part) {
            const int gp = sm.part0 + part;
            const long long col = sm.qbeg + part * N + (t - 1);
            const DevModel<Dual<T>> dm = dual_model(a.model);
            Dual<T> offd[D], sd[NS], stat[NSTAT], Hs[NS * NS], g[NS];
#pragma unroll
            for (int i = 0; i < D; ++i) offd[i] = Dual<T>(a.g.part_off[gp * D + i]);
#pragma unroll
            for (int i = 0; i < NSTAT; ++i) stat[i] = Dual<T>(stats_k[(long long)i * a.Qtot + col]);
#pragma unroll
            for (int i = 0; i < NS; ++i) sd[i] = Dual<T>(st[i], i == e ? T(1) : T(0));
            gn_part<Dual<T>, KIND>(dm, a.g.part_link[gp], offd, sd, stat, stat + NW, stat + NW + D, Hs, g);
            T acc = T(0);
            for (int i = 0; i < NS * NS; ++i) acc += G[i] * Hs[i].d;
            for (int i = 0; i < NS; ++i) acc += qb[i] * (g[i].d - Hs[i * NS + e].v);
            out += a.sigma * acc;
        }
        a.sb[ks + e] = out;
    }
}

// ============================================================================
// reverse step k of the pair side.  Work decomposition of the forward pair
// kernel: a CTA owns 32 (part, t) lanes of one scenario, warp w takes the
// obstacles j = w, w+W, ...
//
// Bound by the latency of its loads: face by face, each value is used as soon as it
// is read (8.4 of 14.5 cycles per issue on the long scoreboard).  STAGED: a warp copies the columns of its
// next pair (y^{k+1}, y^k, ybar, zeta, xi and their adjoints, the obstacle's faces) to
// shared memory while it works on this one, and the offset adjoints of eight faces
// are summed over the lanes together instead of by five shuffles each.  Not STAGED
// (two pairs of W warps exceed kAdjStageMax bytes): every value from global memory.
// 256 trailer scenarios of 32 obstacles, FP32, 3-12 faces: 237 us a step, staged 160.
// ============================================================================
constexpr size_t kAdjStageMax = 200 * 1024;
// rows of 32 lanes of one staged pair
__host__ __device__ inline int adj_pair_rows(int FR, int FO, int D) {
    return 2 * (FR + FO + 1) + FO + 2 * (D + 1) + (FO * (D + 1) + 31) / 32;
}

template <typename T, int D, int NR, bool STAGED>
__global__ void __launch_bounds__(256) k_adj_pair(AdjPairArgs<T> a) {
    constexpr int V = D + 1, NW = StatDims<D>::NW, PK = D + D * D;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *red = reinterpret_cast<T *>(smem_raw);  // [W][PK][32]
    const Tile tile = a.tiles[blockIdx.x];
    const ScenMeta sm = a.meta[tile.scen];
    const int k = a.k;
    if (k >= a.iters[tile.scen]) return;
    const int lane = threadIdx.x, warp = threadIdx.y, W = blockDim.y;
    const int Q = sm.NP * sm.N;
    const int q = tile.q0 + lane;
    const bool valid = q < Q;
    const long long P = a.P;
    const int FR = a.g.FR, FO = a.g.FO;
    const T rho_p = a.prox;
    const bool head = k >= 1;
    T pb[PK];
#pragma unroll
    for (int i = 0; i < PK; ++i) pb[i] = T(0);

    {
        // lanes past the tile's end run on the last lane's data (the warp
        // reductions below need every lane) and write nothing
        const int col = sm.qbeg + (valid ? q : Q - 1);
        T rho[D], R[D * D];
#pragma unroll
        for (int i = 0; i < D; ++i) rho[i] = a.pose[(long long)i * a.Qtot + col];
#pragma unroll
        for (int i = 0; i < D * D; ++i) R[i] = a.pose[(long long)(D + i) * a.Qtot + col];
        const int gp = sm.part0 + (valid ? q : Q - 1) / sm.N;
        const int nr = a.g.part_nf[gp];
        T ak[NR][D], bk[NR], ia2[NR];
#pragma unroll
        for (int kk = 0; kk < NR; ++kk) {
            T s2 = T(0);
#pragma unroll
            for (int i = 0; i < D; ++i) {
                ak[kk][i] = kk < nr ? a.g.part_A[((long long)gp * FR + kk) * D + i] : T(0);
                s2 += ak[kk][i] * ak[kk][i];
            }
            bk[kk] = kk < nr ? a.g.part_b[(long long)gp * FR + kk] : T(1);
            ia2[kk] = s2 > T(0) ? T(1) / s2 : T(0);
        }
        // adjoint of this lane's statistics
        T Wlb[NW], Wcb[D], Eb[D * D];
#pragma unroll
        for (int i = 0; i < NW; ++i) Wlb[i] = a.statsb[(long long)i * a.Qtot + col];
#pragma unroll
        for (int i = 0; i < D; ++i) Wcb[i] = a.statsb[(long long)(NW + i) * a.Qtot + col];
#pragma unroll
        for (int i = 0; i < D * D; ++i) Eb[i] = a.statsb[(long long)(NW + D + i) * a.Qtot + col];

        // staged pair: rows of y^{k+1}, ybar, y^k (obstacle faces), (zeta, xi), their
        // adjoints, then the obstacle's [C | d]
        const int NY = FR + FO + 1, rY0 = 2 * NY, rZX = rY0 + FO, rZB = rZX + V, rOB = rZB + V;
        const int rows = STAGED ? adj_pair_rows(FR, FO, D) : 0;
        T *stage = red + (W * PK + warp * 2 * rows) * 32;
        auto fetch = [&](int j, T *buf) {
            const int gm = sm.obs0 + j, no = a.g.obs_nf[gm];
            const long long p = sm.pair0 + (long long)j * Q + (valid ? q : Q - 1);
            T *b = buf + lane;
            for (int kk = 0; kk < nr; ++kk) {
                cp_async_elem(b + kk * 32, a.y_k1 + p + (long long)kk * P);
                cp_async_elem(b + (NY + kk) * 32, a.ybar_in + p + (long long)kk * P);
            }
            for (int m = 0; m < no; ++m) {
                const long long at = p + (long long)(FR + m) * P;
                cp_async_elem(b + (FR + m) * 32, a.y_k1 + at);
                cp_async_elem(b + (NY + FR + m) * 32, a.ybar_in + at);
                cp_async_elem(b + (rY0 + m) * 32, a.y_k + at);
            }
            cp_async_elem(b + (NY - 1) * 32, a.y_k1 + p + (long long)(NY - 1) * P);
            cp_async_elem(b + (2 * NY - 1) * 32, a.ybar_in + p + (long long)(NY - 1) * P);
#pragma unroll
            for (int i = 0; i < V; ++i) cp_async_elem(b + (rZX + i) * 32, a.zx_k + p + (long long)i * P);
            cp_async_elem(b + rZB * 32, a.zb + p);
#pragma unroll
            for (int i = 0; i < D; ++i) cp_async_elem(b + (rZB + 1 + i) * 32, a.xb + p + (long long)i * P);
            for (int e = lane; e < no * D; e += 32) cp_async_elem(buf + rOB * 32 + e, a.g.obs_C + (long long)gm * FO * D + e);
            for (int e = lane; e < no; e += 32) cp_async_elem(buf + rOB * 32 + FO * D + e, a.g.obs_d + (long long)gm * FO + e);
            cp_async_commit();
        };
        int half = 0;
        if constexpr (STAGED)
            if (warp < sm.M) fetch(warp, stage);
        // y rows: of the staged pair, or of global memory
        const long long ys = STAGED ? 32 : P;
        for (int j = warp; j < sm.M; j += W) {
            const int gm = sm.obs0 + j;
            const int no = a.g.obs_nf[gm];
            const long long p = sm.pair0 + (long long)j * Q + (valid ? q : Q - 1);
            const T *C = a.g.obs_C + (long long)gm * FO * D, *dd = a.g.obs_d + (long long)gm * FO;
            const T *y1 = a.y_k1 + p, *y0 = a.y_k + p + (long long)FR * P, *yi = a.ybar_in + p;
            const T *zx = a.zx_k + p, *zbar = a.zb + p, *xbar = a.xb + p;
            T *buf = stage + half * rows * 32;
            if constexpr (STAGED) {
                cp_async_wait_all();
                __syncwarp();  // the obstacle's faces came by other lanes, which are also done with the other half
                if (j + W < sm.M) fetch(j + W, stage + (half ^ 1) * rows * 32);
                half ^= 1;
                C = buf + rOB * 32;
                dd = C + FO * D;
                y1 = buf + lane;
                yi = y1 + NY * 32;
                y0 = y1 + rY0 * 32;
                zx = y1 + rZX * 32;
                zbar = y1 + rZB * 32;
                xbar = zbar + 32;
            }
            T *yo = a.ybar_out + p;
            const T zeta = zx[0];
            T xi[D];
#pragma unroll
            for (int i = 0; i < D; ++i) xi[i] = zx[(1 + i) * ys];
            // ---- pass 1: sums of y^{k+1}
            T lp[NR], a1[D], w1w[D], Sd = T(0);
#pragma unroll
            for (int i = 0; i < D; ++i) {
                a1[i] = T(0);
                w1w[i] = T(0);
            }
#pragma unroll
            for (int kk = 0; kk < NR; ++kk) {
                lp[kk] = kk < nr ? y1[kk * ys] : T(0);
#pragma unroll
                for (int i = 0; i < D; ++i) a1[i] += lp[kk] * ak[kk][i];
            }
            for (int m = 0; m < no; ++m) {
                const T mp = y1[(FR + m) * ys];
#pragma unroll
                for (int i = 0; i < D; ++i) w1w[i] += mp * C[m * D + i];
                Sd += mp * dd[m];
            }
            const T gp1 = y1[(FR + FO) * ys];
            // ---- statistics adjoint: W += w w^T, Wc += c w, E += w e^T
            const T cc = T(1) + Sd + gp1 + zeta;
            T e[D], w1b[D], eb[D], ccb = T(0);
#pragma unroll
            for (int i = 0; i < D; ++i) {
                e[i] = a1[i] + xi[i];
                w1b[i] = Wcb[i] * cc;
                ccb += Wcb[i] * w1w[i];
            }
            {
                int kk = 0;
#pragma unroll
                for (int i = 0; i < D; ++i)
#pragma unroll
                    for (int jj = 0; jj <= i; ++jj) {
                        if (i == jj) {
                            w1b[i] += T(2) * Wlb[kk] * w1w[i];
                        } else {
                            w1b[i] += Wlb[kk] * w1w[jj];
                            w1b[jj] += Wlb[kk] * w1w[i];
                        }
                        ++kk;
                    }
            }
#pragma unroll
            for (int jj = 0; jj < D; ++jj) {
                T acc = T(0);
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    acc += Eb[i * D + jj] * w1w[i];
                    w1b[i] += Eb[i * D + jj] * e[jj];
                }
                eb[jj] = acc;
            }
            T zb = zbar[0] + ccb, xb[D];
#pragma unroll
            for (int i = 0; i < D; ++i) xb[i] = xbar[i * ys] + eb[i];
            // ---- the QP's dual point w* = K^T y^{k+1} + bq
            T wr = T(0);
#pragma unroll
            for (int i = 0; i < D; ++i) wr += w1w[i] * rho[i];
            const T w0 = T(1) + zeta + Sd - wr + gp1;
            T w1s[D], Rw1[D];
#pragma unroll
            for (int i = 0; i < D; ++i) {
                T acc = xi[i] + a1[i];
#pragma unroll
                for (int l = 0; l < D; ++l) acc += R[l * D + i] * w1w[l];
                w1s[i] = acc;
            }
#pragma unroll
            for (int i = 0; i < D; ++i) {
                T acc = T(0);
#pragma unroll
                for (int l = 0; l < D; ++l) acc += R[i * D + l] * w1s[l];
                Rw1[i] = acc;
            }
            // ---- H = rho (I - K^T dy/dw) and rr = -rho (dy/dw)^T ybar_out
            T H[V][V], rr[V];
#pragma unroll
            for (int i = 0; i < V; ++i) {
                rr[i] = T(0);
#pragma unroll
                for (int jj = 0; jj < V; ++jj) H[i][jj] = i == jj ? rho_p : T(0);
            }
            // lambda block (projection onto b^T lambda = 1 on the support S)
            T yol[NR], bb = T(0), byo = T(0), ba[D];
#pragma unroll
            for (int i = 0; i < D; ++i) ba[i] = T(0);
#pragma unroll
            for (int kk = 0; kk < NR; ++kk) {
                T v = kk < nr ? yi[kk * ys] : T(0);
#pragma unroll
                for (int i = 0; i < D; ++i) v += ak[kk][i] * eb[i];
                yol[kk] = v;
                if (kk < nr && lp[kk] > T(0)) {
                    bb += bk[kk] * bk[kk] * ia2[kk];
                    byo += bk[kk] * ia2[kk] * v;
#pragma unroll
                    for (int i = 0; i < D; ++i) {
                        ba[i] += bk[kk] * ak[kk][i] * ia2[kk];
#pragma unroll
                        for (int l = 0; l < D; ++l) H[1 + i][1 + l] += ak[kk][i] * ak[kk][l] * ia2[kk];
                    }
                }
            }
            const T ibb = bb > T(0) ? T(1) / bb : T(0);
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int l = 0; l < D; ++l) H[1 + i][1 + l] -= ba[i] * ba[l] * ibb;
#pragma unroll
            for (int kk = 0; kk < NR; ++kk) {
                if (kk < nr && lp[kk] > T(0)) {
                    const T zl = yol[kk] - bk[kk] * byo * ibb;
#pragma unroll
                    for (int i = 0; i < D; ++i) rr[1 + i] += zl * ak[kk][i] * ia2[kk];
                }
            }
            // slack gamma
            const T yog = yi[(FR + FO) * ys] + ccb;
            if (gp1 > T(0)) {
                H[0][0] += T(1);
                rr[0] += yog;
            }
            // ---- pass 2: active obstacle faces
            for (int m = 0; m < no; ++m) {
                const T mp = y1[(FR + m) * ys];
                if (!(mp > T(0))) continue;
                T c[D], cr = T(0), c2 = T(0), Km[V];
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    c[i] = C[m * D + i];
                    cr += c[i] * rho[i];
                    c2 += c[i] * c[i];
                }
                const T dm = dd[m], dpm = dm - cr;
                Km[0] = dpm;
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    T acc = T(0);
#pragma unroll
                    for (int l = 0; l < D; ++l) acc += R[l * D + i] * c[l];
                    Km[1 + i] = acc;
                }
                T yom = yi[(FR + m) * ys] + ccb * dm;
#pragma unroll
                for (int i = 0; i < D; ++i) yom += c[i] * w1b[i];
                const T iDg = T(1) / (dpm * dpm + c2);
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    rr[i] += yom * Km[i] * iDg;
#pragma unroll
                    for (int l = 0; l < V; ++l) H[i][l] += Km[i] * Km[l] * iDg;
                }
            }
            T u[V];
#pragma unroll
            for (int i = 0; i < V; ++i) u[i] = rr[i];
            if (chol_solve<T, V>(H, u, V, T(0))) {
#pragma unroll
                for (int i = 0; i < V; ++i) u[i] = -u[i];
            } else {
#pragma unroll
                for (int i = 0; i < V; ++i) u[i] = T(0);
            }
            zb += u[0];
#pragma unroll
            for (int i = 0; i < D; ++i) xb[i] += u[1 + i];
            // head of iteration k: T = 1 + d'^T mu^k + gamma^k, R = A^T lambda^k + R^T C^T mu^k
            T RRv[D];
#pragma unroll
            for (int i = 0; i < D; ++i) {
                T acc = T(0);
#pragma unroll
                for (int l = 0; l < D; ++l) acc += R[i * D + l] * xb[l];
                RRv[i] = acc;
            }
            // ---- pass 3: face outputs
            T ch[D], wk[D];
#pragma unroll
            for (int i = 0; i < D; ++i) {
                ch[i] = T(0);
                wk[i] = T(0);
            }
            for (int m = 0; m < no; ++m) {
                const T mp = y1[(FR + m) * ys], mk = y0[m * ys];
                T c[D], cr = T(0), c2 = T(0), cRw = T(0), cu = T(0), cRv = T(0), cw1b = T(0);
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    c[i] = C[m * D + i];
                    cr += c[i] * rho[i];
                    c2 += c[i] * c[i];
                    cRw += c[i] * Rw1[i];
                    cRv += c[i] * RRv[i];
                    cw1b += c[i] * w1b[i];
                }
                // (R^T c) . u1
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    T acc = T(0);
#pragma unroll
                    for (int l = 0; l < D; ++l) acc += R[l * D + i] * c[l];
                    cu += acc * u[1 + i];
                }
                const T dm = dd[m], dpm = dm - cr, Dg = dpm * dpm + c2;
                T dpb = mp * u[0];   // d/dd' of (K^T y).u at fixed y
                T ybo = T(0);
                if (mp > T(0)) {
                    const T yom = yi[(FR + m) * ys] + ccb * dm + cw1b;
                    const T yh = yom + dpm * u[0] + cu;
                    const T iDg = T(1) / (rho_p * Dg), h = dpm * w0 + cRw;
                    ybo = yh;
                    dpb += yh * (-w0 * iDg + T(2) * h * dpm * iDg / Dg);
#pragma unroll
                    for (int i = 0; i < D; ++i) ch[i] += yh * c[i] * iDg;
                }
                if (head) {
                    ybo += zb * dpm + cRv;
                    dpb += zb * mk;
#pragma unroll
                    for (int i = 0; i < D; ++i) wk[i] += mk * c[i];
                }
                if (valid) yo[(long long)(FR + m) * P] = ybo;
#pragma unroll
                for (int i = 0; i < D; ++i) pb[i] -= dpb * c[i];
                // offset adjoint: d' = d - c.rho, plus the statistics' c = 1 + d^T mu + ...
                T gdv = valid ? dpb + ccb * mp : T(0);
                if constexpr (STAGED) {
                    buf[(FR + m) * 32 + lane] = gdv;  // over y^{k+1}'s, which is not read again
                } else {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) gdv += __shfl_xor_sync(0xffffffffu, gdv, o);
                    if (lane == 0) atomicAdd(a.gd + (long long)gm * FO + m, double(gdv));
                }
            }
            if constexpr (STAGED) {
                // four lanes to a face, eight values to a lane; the start differs by face: no bank twice
                __syncwarp();
                for (int m0 = 0; m0 < no; m0 += 8) {
                    const int m = m0 + (lane >> 2);
                    T v = T(0);
                    if (m < no)
#pragma unroll
                        for (int i = 0; i < 8; ++i) v += buf[(FR + m) * 32 + (lane & 3) * 8 + ((i + (lane >> 2)) & 7)];
                    v += __shfl_xor_sync(0xffffffffu, v, 1);
                    v += __shfl_xor_sync(0xffffffffu, v, 2);
                    if (m < no && (lane & 3) == 0) atomicAdd(a.gd + (long long)gm * FO + m, double(v));
                }
            }
            // R adjoint: -sum_act yh c w1*^T / (rho Dg) + w+ u1^T + [head] w^k xi_bar^T
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int l = 0; l < D; ++l)
                    pb[D + i * D + l] += -ch[i] * w1s[l] + w1w[i] * u[1 + l] + (head ? wk[i] * xb[l] : T(0));
            // lambda outputs
            T byh = T(0);
#pragma unroll
            for (int kk = 0; kk < NR; ++kk) {
                if (kk < nr && lp[kk] > T(0)) {
                    T yh = yol[kk];
#pragma unroll
                    for (int i = 0; i < D; ++i) yh += ak[kk][i] * u[1 + i];
                    yol[kk] = yh;
                    byh += bk[kk] * ia2[kk] * yh;
                }
            }
#pragma unroll
            for (int kk = 0; kk < NR; ++kk) {
                if (kk < nr) {
                    T v = lp[kk] > T(0) ? yol[kk] - bk[kk] * byh * ibb : T(0);
                    if (head) {
#pragma unroll
                        for (int i = 0; i < D; ++i) v += ak[kk][i] * xb[i];
                    }
                    if (valid) yo[(long long)kk * P] = v;
                }
            }
            if (valid) {
                yo[(long long)(FR + FO) * P] = (gp1 > T(0) ? yog + u[0] : T(0)) + (head ? zb : T(0));
                a.zb[p] = zb;
#pragma unroll
                for (int i = 0; i < D; ++i) a.xb[(long long)i * P + p] = xb[i];
            }
        }
    }
    // ---- reduce the pose adjoints across the W warps
#pragma unroll
    for (int i = 0; i < PK; ++i) red[(warp * PK + i) * 32 + lane] = pb[i];
    __syncthreads();
    if (valid) {
        const int col = sm.qbeg + q;
        for (int i = warp; i < PK; i += W) {
            T acc = T(0);
            for (int w2 = 0; w2 < W; ++w2) acc += red[(w2 * PK + i) * 32 + lane];
            a.poseb[(long long)i * a.Qtot + col] = acc;
        }
    }
}


// ============================================================================
// alpha* of the returned trajectory (Sec. III-A eqn:scale_opt): by the LP
// envelope theorem, at the optimum (alpha*, x*; lambda*, mu*) of a pair
//   dalpha/dd_m = -mu_m,  dalpha/drho = C^T mu,  dalpha/dR = (C^T mu) x*^T
// (C' = C R, d' = d - C rho; the Lagrangian alpha + lambda^T (A x - alpha b)
// + mu^T (C' x - d') differentiated at fixed multipliers).  Writes the pose
// adjoints that seed the reverse sweep and adds the offset adjoints.
// ============================================================================
template <typename T, int D>
__global__ void __launch_bounds__(256) k_adj_alpha(AdjAlphaArgs<T> a) {
    constexpr int PK = D + D * D;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *red = reinterpret_cast<T *>(smem_raw);  // [W][PK][32]
    const Tile tile = a.tiles[blockIdx.x];
    const ScenMeta sm = a.meta[tile.scen];
    const int lane = threadIdx.x, warp = threadIdx.y, W = blockDim.y;
    const int Q = sm.NP * sm.N;
    const int q = tile.q0 + lane;
    const bool valid = q < Q;
    const int qc = valid ? q : Q - 1;
    const long long P = a.P;
    const int FR = a.g.FR, FO = a.g.FO;
    T pb[PK];
#pragma unroll
    for (int i = 0; i < PK; ++i) pb[i] = T(0);
    Lane<T, D> L;
    const int col = sm.qbeg + qc;
#pragma unroll
    for (int i = 0; i < D; ++i) L.rho[i] = a.pose[(long long)i * a.Qtot + col];
#pragma unroll
    for (int i = 0; i < D * D; ++i) L.R[i] = a.pose[(long long)(D + i) * a.Qtot + col];
    const int gp = sm.part0 + qc / sm.N;
    L.A = a.g.part_A + (long long)gp * FR * D;
    L.b = a.g.part_b + (long long)gp * FR;
    L.nr = a.g.part_nf[gp];
    for (int j = warp; j < sm.M; j += W) {
        const int gm = sm.obs0 + j;
        L.C = a.g.obs_C + (long long)gm * FO * D;
        L.d = a.g.obs_d + (long long)gm * FO;
        L.no = a.g.obs_nf[gm];
        const long long p = sm.pair0 + (long long)j * Q + qc;
        int bas[D + 1];
        T xB[D + 1], alpha, x[D];
        lp_solve<T, D>(LaneCols<T, D>(L), bas, xB, alpha);
        const bool okx = lp_primal<T, D>(L, bas, x);
        const T ga = valid && okx ? a.grad_alpha[p] : T(0);
        T w[D];
#pragma unroll
        for (int i = 0; i < D; ++i) w[i] = T(0);
        for (int m = 0; m < L.no; ++m) {
            T mu = T(0);
#pragma unroll
            for (int i = 0; i < D + 1; ++i)
                if (bas[i] == L.nr + m) mu = xB[i];
#pragma unroll
            for (int i = 0; i < D; ++i) w[i] += mu * L.C[m * D + i];
            T gdv = -ga * mu;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) gdv += __shfl_xor_sync(0xffffffffu, gdv, o);
            if (lane == 0) atomicAdd(a.gd + (long long)gm * FO + m, double(gdv));
        }
#pragma unroll
        for (int i = 0; i < D; ++i) {
            pb[i] += ga * w[i];
#pragma unroll
            for (int l = 0; l < D; ++l) pb[D + i * D + l] += ga * w[i] * x[l];
        }
    }
#pragma unroll
    for (int i = 0; i < PK; ++i) red[(warp * PK + i) * 32 + lane] = pb[i];
    __syncthreads();
    if (valid) {
        for (int i = warp; i < PK; i += W) {
            T acc = T(0);
            for (int w2 = 0; w2 < W; ++w2) acc += red[(w2 * PK + i) * 32 + lane];
            a.poseb[(long long)i * a.Qtot + sm.qbeg + q] = acc;
        }
    }
}

// returned states of every scenario (iterate iters[s] of the tape) into one array
template <typename T>
__global__ void k_adj_final_states(const ScenMeta *meta, const int *iters, const T *tape_s, long long s_slot, int NS,
                                   T *out) {
    const int s = blockIdx.y;
    const ScenMeta sm = meta[s];
    const T *src = tape_s + (long long)iters[s] * s_slot;
    const int n = (sm.N + 1) * NS;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const long long k2 = (long long)sm.state0 * NS + e;
        out[k2] = src[k2];
    }
}

template <typename T>
cudaError_t launch_adj_alpha(const AdjAlphaArgs<T> &a, int dim, int n_tiles, int W, const int *iters,
                             const T *tape_s, long long s_slot, int NS, int n_scen, T *states_out,
                             const PoseArgs<T> &pa, int maxQ, cudaStream_t st) {
    if (n_tiles <= 0) return cudaSuccess;
    k_adj_final_states<T><<<dim3(4, n_scen), 128, 0, st>>>(a.meta, iters, tape_s, s_slot, NS, states_out);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    PoseArgs<T> p2 = pa;
    p2.states = states_out;
    if ((e = launch_pose<T>(p2, maxQ, st)) != cudaSuccess) return e;
    const size_t sm = (size_t)W * (dim + dim * dim) * 32 * sizeof(T);
    if (dim == 2) k_adj_alpha<T, 2><<<n_tiles, dim3(32, W), sm, st>>>(a);
    else k_adj_alpha<T, 3><<<n_tiles, dim3(32, W), sm, st>>>(a);
    return cudaGetLastError();
}

// ============================================================================
// launchers
// ============================================================================
template <typename T>
cudaError_t launch_adj_seed(const AdjTrajArgs<T> &a, int n_scen, cudaStream_t st) {
    switch (a.model.kind) {
        case 0: k_adj_seed<T, 0><<<n_scen, 32, 0, st>>>(a); break;
        case 1: k_adj_seed<T, 1><<<n_scen, 32, 0, st>>>(a); break;
        case 2: k_adj_seed<T, 2><<<n_scen, 32, 0, st>>>(a); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename T, int KIND>
cudaError_t launch_adj_traj_2d(const AdjTrajArgs<T> &a, int n_scen, int *lq_ok, const int *order, int max_n, int n_sm,
                               cudaStream_t st) {
    const int steps = std::min(kAdjBlock, (max_n + 1 + 31) / 32 * 32);
    k_adj_pre<T, double, KIND><<<n_scen, steps, 0, st>>>(a);
    cudaError_t e = launch_adj_lq<T>(a, n_scen, lq_ok, order, n_sm, st);
    if (e != cudaSuccess) return e;
    k_adj_costate<double, KIND><<<n_scen, 64, 0, st>>>(a.meta, a.iters, a.k, a.scratch, a.scratch0);
    k_adj_post<T, double, KIND><<<dim3(n_scen, (max_n + kPostSteps) / kPostSteps), kPostThreads, 0, st>>>(a);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_adj_traj(const AdjTrajArgs<T> &a, int n_scen, int *lq_ok, const int *order, int max_n, int n_sm,
                            cudaStream_t st) {
    switch (a.model.kind) {
        case 0: return launch_adj_traj_2d<T, 0>(a, n_scen, lq_ok, order, max_n, n_sm, st);
        case 1: return launch_adj_traj_2d<T, 1>(a, n_scen, lq_ok, order, max_n, n_sm, st);
        case 2: k_adj_traj<T, double, 2><<<n_scen, 32, 0, st>>>(a); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename T, int D, int NR>
cudaError_t launch_adj_pair_t(const AdjPairArgs<T> &a, int n_tiles, int W, cudaStream_t st) {
    const size_t red = (size_t)W * (D + D * D) * 32 * sizeof(T);
    const size_t staged = red + (size_t)W * 2 * adj_pair_rows(a.g.FR, a.g.FO, D) * 32 * sizeof(T);
    if (staged <= kAdjStageMax) {
        const cudaError_t e = cudaFuncSetAttribute(k_adj_pair<T, D, NR, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   int(kAdjStageMax));
        if (e != cudaSuccess) return e;
        k_adj_pair<T, D, NR, true><<<n_tiles, dim3(32, W), staged, st>>>(a);
    } else {
        k_adj_pair<T, D, NR, false><<<n_tiles, dim3(32, W), red, st>>>(a);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_adj_pair(const AdjPairArgs<T> &a, int dim, int n_tiles, int W, cudaStream_t st) {
    if (n_tiles <= 0) return cudaSuccess;
    if (dim == 2) {
        if (a.g.FR <= 4) return launch_adj_pair_t<T, 2, 4>(a, n_tiles, W, st);
        if (a.g.FR <= 6) return launch_adj_pair_t<T, 2, 6>(a, n_tiles, W, st);
        return launch_adj_pair_t<T, 2, 8>(a, n_tiles, W, st);
    }
    if (a.g.FR <= 6) return launch_adj_pair_t<T, 3, 6>(a, n_tiles, W, st);
    return launch_adj_pair_t<T, 3, 8>(a, n_tiles, W, st);
}

// offsets and centres from the accumulated offset adjoints: an obstacle
// translated by delta has offsets d_m + c_m . delta, so dL/ddelta = C^T dL/dd
template <typename T>
__global__ void k_adj_finish(const double *gd, const T *obs_C, const int *obs_nf, int M_tot, int FO, int dim,
                             T *grad_d, T *grad_ctr) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M_tot) return;
    const int nf = obs_nf[j];
    double ctr[3] = {0.0, 0.0, 0.0};
    for (int m = 0; m < FO; ++m) {
        const double v = m < nf ? gd[(long long)j * FO + m] : 0.0;
        if (grad_d) grad_d[(long long)j * FO + m] = T(v);
        for (int i = 0; i < dim && m < nf; ++i) ctr[i] += double(obs_C[((long long)j * FO + m) * dim + i]) * v;
    }
    if (grad_ctr)
        for (int i = 0; i < dim; ++i) grad_ctr[(long long)j * dim + i] = T(ctr[i]);
}

template <typename T>
cudaError_t launch_adj_finish(const double *gd, const T *obs_C, const int *obs_nf, int M_tot, int FO, int dim,
                              T *grad_d, T *grad_ctr, cudaStream_t st) {
    if (M_tot <= 0) return cudaSuccess;
    k_adj_finish<T><<<(M_tot + 127) / 128, 128, 0, st>>>(gd, obs_C, obs_nf, M_tot, FO, dim, grad_d, grad_ctr);
    return cudaGetLastError();
}

template cudaError_t launch_adj_seed<float>(const AdjTrajArgs<float> &, int, cudaStream_t);
template cudaError_t launch_adj_seed<double>(const AdjTrajArgs<double> &, int, cudaStream_t);
template cudaError_t launch_adj_traj<float>(const AdjTrajArgs<float> &, int, int *, const int *, int, int, cudaStream_t);
template cudaError_t launch_adj_traj<double>(const AdjTrajArgs<double> &, int, int *, const int *, int, int, cudaStream_t);
template cudaError_t launch_adj_pair<float>(const AdjPairArgs<float> &, int, int, int, cudaStream_t);
template cudaError_t launch_adj_pair<double>(const AdjPairArgs<double> &, int, int, int, cudaStream_t);
template cudaError_t launch_adj_alpha<float>(const AdjAlphaArgs<float> &, int, int, int, const int *, const float *,
                                             long long, int, int, float *, const PoseArgs<float> &, int, cudaStream_t);
template cudaError_t launch_adj_alpha<double>(const AdjAlphaArgs<double> &, int, int, int, const int *, const double *,
                                              long long, int, int, double *, const PoseArgs<double> &, int,
                                              cudaStream_t);
template cudaError_t launch_adj_finish<float>(const double *, const float *, const int *, int, int, int, float *, float *,
                                              cudaStream_t);
template cudaError_t launch_adj_finish<double>(const double *, const double *, const int *, int, int, int, double *,
                                               double *, cudaStream_t);

}  // namespace oca
