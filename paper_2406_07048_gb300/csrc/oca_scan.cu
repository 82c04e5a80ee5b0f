// The step-2 LQ problem of the ADMM (Sec. IV-B, one SQP QP per iteration)
// solved for a batch of independent problems, in two forms:
//
//   OCA_LQ_SCAN        parallel in time.  The optimality conditions link each
//                      stage's state and costate lam_t = dV_t/ds_t linearly,
//                        s_{t+1} = A_t s_t + b_t - C_t lam_{t+1},
//                        lam_t   = J_t s_t - eta_t + A_t^T lam_{t+1},
//                      with b_t = c_t - B_t R_t^-1 r_t, C_t = B_t R_t^-1 B_t^T,
//                      J_t = Q_t, eta_t = -q_t, and lam_N = Q_N s_N + q_N as the
//                      element (0, 0, 0, Q_N, -q_N).  Two consecutive relations
//                      compose into one of the same form (eliminating the shared
//                      state and costate, M = (I + C1 J2)^-1):
//                        A = A2 M A1,  b = A2 M (b1 + C1 eta2) + b2,
//                        C = A2 M C1 A2^T + C2,  J = J1 + A1^T M^T J2 A1,
//                        eta = eta1 + A1^T M^T (eta2 - J2 b1),
//                      an associative operation, so every suffix e_t o ... o e_N
//                      (whose A is 0: lam_t = J s_t - eta, the value function
//                      P_t = J, p_t = -eta) is formed in ceil(log2(N + 1)) rounds
//                      in which element t takes element t + 2^r, one CTA per
//                      composition.  The gains K_t, k_t and the closed-loop maps
//                      A + B K, B k + c follow per stage in parallel.
//   OCA_LQ_SEQUENTIAL  the backward Riccati recursion over t (one CTA per
//                      problem), which forms the gains; the closed-loop maps
//                      follow per stage in parallel.
//
// The rollout s_{t+1} = (A + B K) s + B k + c is a dependent chain of matrix-vector
// products: one warp per problem, or for few problems of 64 steps and more a warp per
// chunk of steps, started from the products of the maps before its chunk.
//
// FP64 throughout.  One CTA per composition: its two elements and the augmented
// system [I + C1 J2 | A1, b1 + C1 eta2, C1 A2^T] live in shared memory; the system is
// reduced by Gauss-Jordan elimination with partial pivoting.
//
// Measured (GB300, 12 states, 4 inputs): one problem of 256 steps, scan 750 -> 240 us
// (a composition round 63 -> 19, gains 43 -> 15, rollout 169 -> 41); 256 problems of 64
// steps, sequential 2,900 -> 380 us (33 -> 4.9 us a stage, the closed-loop maps 730 ->
// 25).
#include <algorithm>
#include <cfloat>
#include <utility>

#include "oca_common.cuh"
#include "oca_fp64.cuh"
#include "oca_kernels.h"

namespace oca {

constexpr int kLqMaxS = 12;  // state dimension
constexpr int kLqMaxU = 4;   // input dimension

struct LqArgs {
    int n, m, N, S;              // state, input, horizon, problems
    const double *A, *B, *c;     // [S][N][n][n], [S][N][n][m], [S][N][n]
    const double *Q, *q;         // [S][N+1][n][n], [S][N+1][n]
    const double *R, *r;         // [S][N][m][m], [S][N][m]
    const double *s0;            // [S][n]
    double *s, *u;               // [S][N+1][n], [S][N][m]
    double *P, *p;               // [S][N+1][n][n], [S][N+1][n] or null
    int *status;                 // [S]: 0 solved, 1 singular or non-finite
    double *buf0, *buf1;         // element buffers [S][N+1][es]
    double *F, *f, *K, *k;       // closed-loop maps and gains [S][N][..]
};

__host__ __device__ inline int lq_es(int n) { return 3 * n * n + 2 * n; }

// FP64 issues one warp instruction per 64 cycles and scheduler, whatever its lanes
// do, so the kernels below count FP64 instructions per warp: products are dealt one
// entry to a thread, small systems are solved with one column per lane, compares
// run on the integer pipe and a reciprocal is three multiply-adds.

// order of |x| as an integer (NaN above infinity)
__device__ __forceinline__ unsigned long long abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

// Solve M X = V, M m x m (m <= 4), by Gauss-Jordan elimination with partial pivoting:
// lane j < m of the warp holds column j of M in v, the lanes from m on the columns of
// V; on return they hold the columns of X.  False if a pivot is not above 1e-300 +
// 1e-14 max |M| or M is not finite (1 takes the pivot's place).  The bound is relative to
// M alone, for every m: padding M to 4 x 4 with ones, as small systems of 1 to 3 inputs
// once were, makes 1e-14 the least of it and refuses a control cost of 1e-15.
__device__ __forceinline__ bool gj_columns(double (&v)[kLqMaxU], int m, int lane) {
    unsigned long long big = 0;
#pragma unroll
    for (int i = 0; i < kLqMaxU; ++i)
        if (lane < m && i < m && abs_bits(v[i]) > big) big = abs_bits(v[i]);
    // the largest of the m columns
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, big, o);
        if (other > big) big = other;
    }
    big = __shfl_sync(0xffffffffu, big, 0);
    bool ok = big < 0x7ff0000000000000ull;
    const unsigned long long floor = abs_bits(fma(1e-14, __longlong_as_double((long long)big), 1e-300));
#pragma unroll
    for (int c = 0; c < kLqMaxU; ++c) {
        if (c >= m) break;
        int pr = c;
        unsigned long long best = abs_bits(v[c]);
#pragma unroll
        for (int i = c + 1; i < kLqMaxU; ++i)
            if (i < m && abs_bits(v[i]) > best) {
                best = abs_bits(v[i]);
                pr = i;
            }
        pr = __shfl_sync(0xffffffffu, pr, c);
        best = __shfl_sync(0xffffffffu, best, c);
        const bool fine = best > floor;
        ok = ok && fine;
#pragma unroll
        for (int i = c + 1; i < kLqMaxU; ++i)
            if (i == pr) {
                const double x = v[c];
                v[c] = v[i];
                v[i] = x;
            }
        double col[kLqMaxU];
#pragma unroll
        for (int i = 0; i < kLqMaxU; ++i) col[i] = i < m ? __shfl_sync(0xffffffffu, v[i], c) : 0.0;
        v[c] *= recip(fine ? col[c] : 1.0);
#pragma unroll
        for (int i = 0; i < kLqMaxU; ++i)
            if (i != c && i < m) v[i] = fma(-col[i], v[c], v[i]);
    }
    return ok;
}

// entry e of an n x n upper triangle, row by row
__device__ __forceinline__ void upper_entry(int e, int n, int &i, int &j) {
    i = 0;
    while (e >= n - i) {
        e -= n - i;
        ++i;
    }
    j = i + e;
}

// sum over y < n of a[y * sa] * b[y * sb] + init; CN: n when known at compile time
template <int CN>
__device__ __forceinline__ double dot_strided(const double *a, int sa, const double *b, int sb, int n, double init) {
    if constexpr (CN > 0) {
#pragma unroll
        for (int y = 0; y < CN; ++y) init = fma(a[y * sa], b[y * sb], init);
    } else {
#pragma unroll 4
        for (int y = 0; y < n; ++y) init = fma(a[y * sa], b[y * sb], init);
    }
    return init;
}

// ---- stage elements (one warp per stage and problem)
template <int CN, int CM>
__global__ void __launch_bounds__(32) k_lq_elem(LqArgs a) {
    const int t = blockIdx.x, s = blockIdx.y, lane = threadIdx.x;
    const int n = CN ? CN : a.n, m = CM ? CM : a.m, N = a.N, nn = n * n, E = N + 1;
    double *e = a.buf0 + ((size_t)s * E + t) * lq_es(n);
    double *Ae = e, *be = e + nn, *Ce = be + n, *Je = Ce + nn, *he = Je + nn;
    const double *Qt = a.Q + ((size_t)s * E + t) * nn, *qt = a.q + ((size_t)s * E + t) * n;
    for (int k2 = lane; k2 < nn; k2 += 32) Je[k2] = Qt[k2];
    for (int i = lane; i < n; i += 32) he[i] = -qt[i];
    if (t == N) {
        for (int k2 = lane; k2 < nn; k2 += 32) {
            Ae[k2] = 0.0;
            Ce[k2] = 0.0;
        }
        for (int i = lane; i < n; i += 32) be[i] = 0.0;
        return;
    }
    const size_t st = (size_t)s * N + t;
    const double *At = a.A + st * nn, *Bt = a.B + st * n * m, *ct = a.c + st * n;
    const double *Rt = a.R + st * m * m, *rt = a.r + st * m;
    __shared__ double X[kLqMaxU * (kLqMaxS + 1)], Bs[kLqMaxS * kLqMaxU];  // X = R^-1 [B^T | r]
    double v[kLqMaxU];
    const int col = lane - m;
#pragma unroll
    for (int i = 0; i < kLqMaxU; ++i)
        v[i] = i >= m ? 0.0 : lane < m ? Rt[i * m + lane] : col < n ? Bt[col * m + i] : col == n ? rt[i] : 0.0;
    for (int k2 = lane; k2 < n * m; k2 += 32) Bs[k2] = Bt[k2];
    for (int k2 = lane; k2 < nn; k2 += 32) Ae[k2] = At[k2];
    const bool ok = gj_columns(v, m, lane);
    if (!ok && lane == 0) a.status[s] = 1;
    if (col >= 0 && col <= n)
#pragma unroll
        for (int i = 0; i < kLqMaxU; ++i)
            if (i < m) X[i * (n + 1) + col] = v[i];
    __syncwarp();
    for (int i = lane; i < n; i += 32) be[i] = ct[i] - dot_strided<CM>(Bs + i * m, 1, X + n, n + 1, m, 0.0);
    // C = B R^-1 B^T
    for (int k2 = lane; k2 < nn; k2 += 32)
        Ce[k2] = dot_strided<CM>(Bs + k2 / n * m, 1, X + k2 % n, n + 1, m, 0.0);
}

// ---- one round of compositions: nxt[t] = cur[t] o cur[t + d] (or cur[t])
constexpr int kLqThreads = 128;

// With M = (I + C1 J2)^-1 and X = M [A1 | b1 + C1 eta2 | C1 A2^T] = [XA | Xb | XC], one
// system gives the whole composition: M^T J2 = J2 M and M^T = I - J2 M C1 (C1, J2
// symmetric), so
//   A = A2 XA,  b = A2 Xb + b2,  C = A2 XC + C2,
//   J = J1 + A1^T (J2 XA),  eta = eta1 + A1^T (eta2 - J2 Xb).
// The system is held as columns [X | M columns from the last to the first]: pivot c is
// the last active column, so the active ones stay in front.  Elimination writes the
// other of two copies (one barrier per pivot); each warp finds the pivot row itself
// (largest |x| by its upper 32 bits, the lowest row on ties).
template <int CN>
__global__ void __launch_bounds__(kLqThreads) k_lq_compose(LqArgs a, const double *cur, double *nxt, int d) {
    const int t = blockIdx.x, s = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = CN ? CN : a.n, nn = n * n, E = a.N + 1, es = lq_es(n);
    const double *e1g = cur + ((size_t)s * E + t) * es;
    double *eo = nxt + ((size_t)s * E + t) * es;
    if (t + d >= E) {
        for (int k2 = tid; k2 < es; k2 += kLqThreads) eo[k2] = e1g[k2];
        return;
    }
    const double *e2g = cur + ((size_t)s * E + t + d) * es;
    constexpr int NM = CN ? CN : kLqMaxS, MES = 3 * NM * NM + 2 * NM, WM = 3 * NM + 1;
    __shared__ double e1[MES], e2[MES], G[2][NM * WM], T[NM * (NM + 1)];
    for (int k2 = tid; k2 < es; k2 += kLqThreads) {
        e1[k2] = e1g[k2];
        e2[k2] = e2g[k2];
    }
    __syncthreads();
    const double *A1 = e1, *b1 = e1 + nn, *C1 = b1 + n, *J1 = C1 + nn, *h1 = J1 + nn;
    const double *A2 = e2, *b2 = e2 + nn, *C2 = b2 + n, *J2 = C2 + nn, *h2 = J2 + nn;
    const int W = 3 * n + 1, NX = 2 * n + 1;  // columns: XA [n], XC [n], Xb, then M columns n-1 .. 0
    for (int k2 = tid; k2 < nn; k2 += kLqThreads) G[0][k2 / n * W + k2 % n] = A1[k2];
    for (int k2 = tid; k2 < n * NX; k2 += kLqThreads) {
        // C1 times a row of A2, eta2 or a column of J2: one product for all three
        const int i = k2 / NX, j = n + k2 % NX, c = W - 1 - j;
        const double *right = j < 2 * n ? A2 + (j - n) * n : j == 2 * n ? h2 : J2 + c;
        const double init = j < 2 * n ? 0.0 : j == 2 * n ? b1[i] : i == c ? 1.0 : 0.0;
        G[0][i * W + j] = dot_strided<CN>(C1 + i * n, 1, right, j <= 2 * n ? 1 : n, n, init);
    }
    bool bad = false;
    for (int c = 0; c < n; ++c) {
        __syncthreads();
        const double *S = G[c & 1];
        double *O = G[(c + 1) & 1];
        const int pc = W - 1 - c;  // the pivot's column; columns 0 .. pc - 1 stay active
        const double cv = lane < n ? S[lane * W + pc] : 0.0;
        const unsigned key = lane >= c && lane < n ? (unsigned)(__double2hiint(cv) & 0x7fffffff) : 0u;
        const unsigned top = __reduce_max_sync(0xffffffffu, key);
        const int px = __ffs(__ballot_sync(0xffffffffu, lane >= c && lane < n && key == top)) - 1;
        const double pv = S[px * W + pc];
        const bool fine = abs_bits(pv) > 0x01a56e1fc2f8f359ull && abs_bits(pv) < 0x7ff0000000000000ull;  // > 1e-300, finite
        bad = bad || !fine;
        const double ip = recip(fine ? pv : 1.0);
        // a lane per column (the columns past 32 in a second pass while they are
        // active), the rows dealt over the warps: the scaled pivot row is formed once
        // per column and warp
        for (int j = lane; j < pc; j += 32) {
            const double rj = S[px * W + j] * ip;
            for (int i = warp; i < n; i += kLqThreads / 32) {
                const int src = i == px ? c : i;
                O[i * W + j] = i == c ? rj : fma(-S[src * W + pc], rj, S[src * W + j]);
            }
        }
    }
    __syncthreads();
    const double *X = G[n & 1];
    if (bad && tid == 0) a.status[s] = 1;
    // T = [J2 XA | eta2 - J2 Xb]
    for (int k2 = tid; k2 < n * (n + 1); k2 += kLqThreads) {
        const int i = k2 / (n + 1), j = k2 % (n + 1);
        const double v = dot_strided<CN>(J2 + i * n, 1, X + (j < n ? j : 2 * n), W, n, 0.0);
        T[k2] = j < n ? v : h2[i] - v;
    }
    // A, b and the upper triangle of C while T settles (C and J are symmetric)
    double *Ao = eo, *bo = eo + nn, *Co = bo + n, *Jo = Co + nn, *ho = Jo + nn;
    const int nsym = n * (n + 1) / 2;
    for (int k2 = tid; k2 < nn + n + nsym; k2 += kLqThreads) {
        int i, j;  // row of A2, column of X
        if (k2 < nn + n) {
            i = k2 / (n + 1);
            j = k2 % (n + 1);
            if (j == n) j = 2 * n;
        } else {
            upper_entry(k2 - nn - n, n, i, j);
            j += n;
        }
        const double init = j < n ? 0.0 : j < 2 * n ? C2[i * n + j - n] : b2[i];
        const double v = dot_strided<CN>(A2 + i * n, 1, X + j, W, n, init);
        if (j < n) Ao[i * n + j] = v;
        else if (j < 2 * n) Co[i * n + j - n] = Co[(j - n) * n + i] = v;
        else bo[i] = v;
    }
    __syncthreads();
    for (int k2 = tid; k2 < nsym + n; k2 += kLqThreads) {
        int i, j;
        if (k2 < nsym) {
            upper_entry(k2, n, i, j);
        } else {
            i = k2 - nsym;
            j = n;
        }
        const double v = dot_strided<CN>(A1 + i, n, T + j, n + 1, n, j < n ? J1[i * n + j] : h1[i]);
        if (j < n) Jo[i * n + j] = Jo[j * n + i] = v;
        else ho[i] = v;
    }
}

// ---- gains of stage t from the value function of stage t + 1 (J, -eta of element
// t + 1 of vf):
//   K = -(R + B^T P B)^-1 B^T P A,  k = -(R + B^T P B)^-1 (B^T (P c + p) + r),
// and the closed-loop map s_{t+1} = F s_t + f, F = A + B K, f = c + B k.
// Every block also writes its stage's value function when requested.
constexpr int kLqGainThreads = 64;
template <int CN, int CM>
__global__ void __launch_bounds__(kLqGainThreads) k_lq_gains(LqArgs a, const double *vf) {
    const int t = blockIdx.x, s = blockIdx.y, tid = threadIdx.x;
    const int n = CN ? CN : a.n, m = CM ? CM : a.m, N = a.N, nn = n * n, E = N + 1, es = lq_es(n);
    const double *Pt = vf + ((size_t)s * E + t) * es + 2 * nn + n, *P1g = Pt + es;
    if (a.P)
        for (int k2 = tid; k2 < nn; k2 += kLqGainThreads) a.P[((size_t)s * E + t) * nn + k2] = Pt[k2];
    if (a.p)
        for (int i = tid; i < n; i += kLqGainThreads) a.p[((size_t)s * E + t) * n + i] = -Pt[nn + i];
    if (t == N) return;
    __shared__ double P[kLqMaxS * kLqMaxS], As[kLqMaxS * kLqMaxS], Bs[kLqMaxS * kLqMaxU], Y[kLqMaxS * (kLqMaxU + 1)],
        H[kLqMaxU * (kLqMaxU + kLqMaxS + 1)], Ks[kLqMaxU * (kLqMaxS + 1)];
    const size_t st = (size_t)s * N + t;
    const double *At = a.A + st * nn, *Bt = a.B + st * n * m, *ct = a.c + st * n;
    const double *Rt = a.R + st * m * m, *rt = a.r + st * m;
    for (int k2 = tid; k2 < nn; k2 += kLqGainThreads) {
        P[k2] = P1g[k2];
        As[k2] = At[k2];
    }
    for (int k2 = tid; k2 < n * m; k2 += kLqGainThreads) Bs[k2] = Bt[k2];
    __syncthreads();
    // Y = [P B | P c + p]
    for (int k2 = tid; k2 < n * (m + 1); k2 += kLqGainThreads) {
        const int i = k2 / (m + 1), x = k2 % (m + 1);
        Y[k2] = x < m ? dot_strided<CN>(P + i * n, 1, Bs + x, m, n, 0.0) : dot_strided<CN>(P + i * n, 1, ct, 1, n, -P1g[nn + i]);
    }
    __syncthreads();
    // H = [R + B^T P B | (P B)^T A | B^T (P c + p) + r]
    const int HW = m + n + 1;
    for (int k2 = tid; k2 < m * HW; k2 += kLqGainThreads) {
        const int x = k2 / HW, j = k2 % HW;
        double v;
        if (j < m) v = dot_strided<CN>(Bs + x, m, Y + j, m + 1, n, Rt[x * m + j]);
        else if (j < m + n) v = dot_strided<CN>(Y + x, m + 1, As + j - m, n, n, 0.0);
        else v = dot_strided<CN>(Bs + x, m, Y + m, m + 1, n, rt[x]);
        H[k2] = v;
    }
    __syncthreads();
    double *Ko = a.K + st * m * n, *ko = a.k + st * m, *Fo = a.F + st * nn, *fo = a.f + st * n;
    if (tid < 32) {
        double v[kLqMaxU];
#pragma unroll
        for (int i = 0; i < kLqMaxU; ++i) v[i] = i < m && tid < HW ? H[i * HW + tid] : 0.0;
        const bool ok = gj_columns(v, m, tid);
        if (!ok && tid == 0) a.status[s] = 1;
        const int j = tid - m;
        if (j >= 0 && j <= n)
#pragma unroll
            for (int i = 0; i < kLqMaxU; ++i)
                if (i < m) {
                    Ks[i * (n + 1) + j] = -v[i];
                    if (j < n) Ko[i * n + j] = -v[i];
                    else ko[i] = -v[i];
                }
    }
    __syncthreads();
    for (int k2 = tid; k2 < n * (n + 1); k2 += kLqGainThreads) {
        const int i = k2 / (n + 1), j = k2 % (n + 1);
        const double v = dot_strided<CM>(Bs + i * m, 1, Ks + j, n + 1, m, j < n ? As[i * n + j] : ct[i]);
        if (j < n) Fo[i * n + j] = v;
        else fo[i] = v;
    }
}

// ---- closed-loop maps F = A + B K, f = c + B k of the sequential form's gains
template <int CN, int CM>
__global__ void __launch_bounds__(kLqGainThreads) k_lq_closed(LqArgs a) {
    const int t = blockIdx.x, s = blockIdx.y, tid = threadIdx.x;
    const int n = CN ? CN : a.n, m = CM ? CM : a.m, nn = n * n;
    const size_t st = (size_t)s * a.N + t;
    const double *Bt = a.B + st * n * m, *Kt = a.K + st * m * n, *kt = a.k + st * m;
    for (int k2 = tid; k2 < nn + n; k2 += kLqGainThreads) {
        if (k2 < nn) {
            const int i = k2 / n, j = k2 % n;
            a.F[st * nn + k2] = dot_strided<CM>(Bt + i * m, 1, Kt + j, n, m, a.A[st * nn + k2]);
        } else {
            const int i = k2 - nn;
            a.f[st * n + i] = dot_strided<CM>(Bt + i * m, 1, kt, 1, m, a.c[st * n + i]);
        }
    }
}

// ---- closed-loop maps of whole chunks: s_{t0 + L} = G s_{t0} + g over the L steps of
// chunk blockIdx.x (one product of maps per step).  Behind G and g a 1 where the rollout may
// not use the map: a mode that feedback does not reach and that grows by more than
// kLqMapMax within the chunk.  Its state can be small all the same (0, or held by c), and
// then G s + g is a difference of large numbers, or inf * 0, where the steps are exact.
constexpr double kLqMapMax = 65536.0;  // 2^16 of 2^53: at most 1e-11 of the state is lost
__host__ __device__ inline int lq_map_size(int n) { return n * n + n + 1; }
template <int CN>
__global__ void __launch_bounds__(kLqThreads) k_lq_chunk(LqArgs a, double *maps, int L) {
    const int c = blockIdx.x, s = blockIdx.y, tid = threadIdx.x;
    const int n = CN ? CN : a.n, nn = n * n, w = nn + n;
    constexpr int NM = CN ? CN : kLqMaxS;
    __shared__ double Fs[2][NM * NM + NM], G[2][NM * NM + NM];
    const double *F0 = a.F + ((size_t)s * a.N + (size_t)c * L) * nn, *f0 = a.f + ((size_t)s * a.N + (size_t)c * L) * n;
    auto copy = [&](int t) {
        for (int e = tid; e < w; e += kLqThreads)
            cp_async_elem(&Fs[t & 1][e], e < nn ? F0 + (size_t)t * nn + e : f0 + (size_t)t * n + e - nn);
        cp_async_commit();
    };
    bool far = false;
    auto put = [&](double *o, int e, double v) {
        o[e] = v;
        far = far || !(e < nn ? abs_bits(v) <= abs_bits(kLqMapMax) : finite(v));
    };
    for (int e = tid; e < w; e += kLqThreads) put(G[0], e, e < nn ? F0[e] : f0[e - nn]);
    if (L > 1) copy(1);
    for (int t = 1; t < L; ++t) {
        cp_async_wait_all();
        __syncthreads();
        if (t + 1 < L) copy(t + 1);
        const double *S = Fs[t & 1], *X = G[(t - 1) & 1];
        double *O = G[t & 1];
        for (int e = tid; e < w; e += kLqThreads) {
            const int i = e < nn ? e / n : e - nn;
            put(O, e, e < nn ? dot_strided<CN>(S + i * n, 1, X + e % n, n, n, 0.0)
                             : dot_strided<CN>(S + i * n, 1, X + nn, 1, n, S[nn + i]));
        }
    }
    far = __syncthreads_or(far);
    double *out = maps + ((size_t)s * gridDim.x + c) * lq_map_size(n);
    for (int e = tid; e < w; e += kLqThreads) out[e] = G[(L - 1) & 1][e];
    if (tid == 0) out[w] = far ? 1.0 : 0.0;
}

// ---- rollout s_{t+1} = F_t s_t + f_t (one warp per chunk and problem): the state at
// the chunk's start through the maps of the chunks before it (or their steps, where a map
// may not be used), then the chunk's steps.
// Lane i and lane 16 + i own s_i and sum one half of its row each; the rows of the next
// four steps are on their way while a step runs (a step takes about 900 cycles, a load
// up to 1,500).
template <int CN>
__global__ void __launch_bounds__(32) k_lq_rollout(LqArgs a, const double *maps, int C, int L) {
    constexpr int AHEAD = 4, HM = kLqMaxS / 2;
    const int c = blockIdx.x, s = blockIdx.y, lane = threadIdx.x, i = lane & 15, half = lane >> 4;
    const int n = CN ? CN : a.n, N = a.N, nn = n * n, nh = (n + 1) / 2;
    const bool own = i < n;
    const int k0 = half * nh, kn = own ? (half ? n - nh : nh) : 0;  // this lane's terms k0 .. k0 + kn - 1
    double x = own ? a.s0[(size_t)s * n + i] : 0.0;
    if (c == 0 && own && !half) a.s[(size_t)s * (N + 1) * n + i] = x;
    double row[AHEAD][HM], fv[AHEAD];
    // steps x <- F x + f with F, f of step t at F0 + t * sF, f0 + t * sf; the states go to out
    auto roll = [&](const double *F0, size_t sF, const double *f0, size_t sf, int steps, double *out) {
        auto fetch = [&](int t, double (&r)[HM], double &f) {
#pragma unroll
            for (int k2 = 0; k2 < HM; ++k2) r[k2] = t < steps && k2 < kn ? F0[t * sF + i * n + k0 + k2] : 0.0;
            f = t < steps && own && !half ? f0[t * sf + i] : 0.0;
        };
#pragma unroll
        for (int d = 0; d < AHEAD; ++d) fetch(d, row[d], fv[d]);
        for (int t0 = 0; t0 < steps; t0 += AHEAD) {
#pragma unroll
            for (int d = 0; d < AHEAD; ++d) {
                const int t = t0 + d;
                double v = fv[d];
#pragma unroll
                for (int k2 = 0; k2 < HM; ++k2) {
                    if (CN && k2 >= (CN + 1) / 2) break;
                    v = fma(row[d][k2], __shfl_sync(0xffffffffu, x, min(k0 + k2, 15)), v);
                }
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                if (t < steps) {
                    x = v;
                    if (out && own && !half) out[(size_t)t * n + i] = x;
                }
                fetch(t + AHEAD, row[d], fv[d]);
            }
        }
    };
    const int w = lq_map_size(n), t0 = c * L;
    if (c > 0) {
        const double *m0 = maps + (size_t)s * C * w;
        bool far = false;  // a map before this chunk that may not be used
        for (int k2 = lane; k2 < c; k2 += 32) far = far || abs_bits(m0[(size_t)k2 * w + nn + n]) != 0;
        if (__any_sync(0xffffffffu, far)) roll(a.F + (size_t)s * N * nn, nn, a.f + (size_t)s * N * n, n, t0, nullptr);
        else roll(m0, w, m0 + nn, w, c, nullptr);
    }
    const size_t st = (size_t)s * N + t0;
    roll(a.F + st * nn, nn, a.f + st * n, n, min(L, N - t0), a.s + ((size_t)s * (N + 1) + t0 + 1) * n);
}

// ---- u_t = K_t s_t + k_t, one thread per control
__global__ void __launch_bounds__(128) k_lq_controls(LqArgs a) {
    const long long e = (long long)blockIdx.x * 128 + threadIdx.x;
    const int n = a.n, m = a.m, N = a.N;
    if (e >= (long long)a.S * N * m) return;
    const long long st = e / m, s = st / N, t = st % N;
    const double *Kt = a.K + e * n, *xt = a.s + (s * (N + 1) + t) * n;
    double v = a.k[e];
    for (int j = 0; j < n; ++j) v = fma(Kt[j], xt[j], v);
    a.u[e] = v;
}

// ---- sequential backward Riccati recursion (one CTA per problem): with
// G = [A | B | c] and Y = P G + [0 | 0 | p],
//   Qss = Q + A^T Y_A, qs = q + A^T Y_c, H = B^T Y_A, Quu = R + B^T Y_B,
//   qu = r + B^T Y_c, [K | k] = -Quu^-1 [H | qu], P_t = Qss + H^T K, p_t = qs + H^T k;
// P_N = Q_N, p_N = q_N.  Per stage: both products with one or two entries per thread
// (their positions found once), the m x m system by one warp with a column per lane,
// the next stage's data copied to the other shared buffer meanwhile.
template <int CN, int CM, int NT>
__global__ void __launch_bounds__(NT) k_lq_seq(LqArgs a) {
    const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = CN ? CN : a.n, m = CM ? CM : a.m, N = a.N, nn = n * n, E = N + 1;
    // the warp that solves the m x m system: another scheduler's in the second half of
    // the grid, whose CTAs share SMs with the first half's
    const int solver = NT > 64 && blockIdx.x >= gridDim.x / 2 ? 2 : 0;
    constexpr int NM = CN ? CN : kLqMaxS, MM = CM ? CM : kLqMaxU;
    constexpr int STG = 2 * NM * NM + NM * MM + 2 * NM + MM * MM + MM;
    __shared__ double P[NM * NM], pp[NM], Y[NM * (NM + MM + 1)], Ms[NM * NM], gs[NM], Hs[MM * (NM + MM + 1)],
        Ks[MM * (NM + 1)], stg[2][STG];
    const int W = n + m + 1, nY = n * W, nsym = n * (n + 1) / 2, nM = nsym + n + m * W, nP = nsym + n;
    // shared copy of a stage: A, B, c, Q, q, R, r
    const int oB = nn, oc = oB + n * m, oQ = oc + n, oq = oQ + nn, oR = oq + n, orr = oR + m * m, nst = orr + m;
    auto copy = [&](int t, double *dst) {
        const size_t st = (size_t)s * N + t, se = (size_t)s * E + t;
        for (int e = tid; e < nst; e += NT) {
            const double *src = e < oB    ? a.A + st * nn + e
                                : e < oc  ? a.B + st * n * m + (e - oB)
                                : e < oQ  ? a.c + st * n + (e - oc)
                                : e < oq  ? a.Q + se * nn + (e - oQ)
                                : e < oR  ? a.q + se * n + (e - oq)
                                : e < orr ? a.R + st * m * m + (e - oR)
                                          : a.r + st * m + (e - orr);
            cp_async_elem(dst + e, src);
        }
        cp_async_commit();
    };
    // Y entries: row i, column j of [A | B | c] (first element and stride in the stage)
    constexpr int PY = (NM * (NM + MM + 1) + NT - 1) / NT, PM = (NM * (NM + 1) / 2 + NM + MM * (NM + MM + 1) + NT - 1) / NT,
                  PP = (NM * (NM + 1) / 2 + NM + NT - 1) / NT;
    int yi[PY], yo[PY], ys[PY];
#pragma unroll
    for (int r = 0; r < PY; ++r) {
        const int e = tid + NT * r, i = e / W, j = e % W;
        yi[r] = e < nY ? i : -1;
        yo[r] = j < n ? j : j < n + m ? oB + j - n : oc;
        ys[r] = j < n ? n : j < n + m ? m : 1;
    }
    // stage-matrix entries: left column (first element, stride in the stage), right
    // column of Y, init in the stage (-1: none), result
    int ml[PM], ms[PM], mr[PM], mi[PM];
    double *mo[PM];
#pragma unroll
    for (int r = 0; r < PM; ++r) {
        // dealt from the last thread on: with Y's entries dealt from the first, the four
        // schedulers get the same number of products
        const int e = NT - 1 - tid + NT * r;
        ml[r] = -1;
        ms[r] = mr[r] = 0;
        mi[r] = -1;
        mo[r] = nullptr;
        if (e < nsym) {
            int i, j;
            upper_entry(e, n, i, j);
            ml[r] = i;
            ms[r] = n;
            mr[r] = j;
            mi[r] = oQ + i * n + j;
            mo[r] = Ms + i * n + j;
        } else if (e < nsym + n) {
            const int i = e - nsym;
            ml[r] = i;
            ms[r] = n;
            mr[r] = n + m;
            mi[r] = oq + i;
            mo[r] = gs + i;
        } else if (e < nM) {
            const int k2 = e - nsym - n, x = k2 / W, j = k2 % W;
            ml[r] = oB + x;
            ms[r] = m;
            mr[r] = j;
            mi[r] = j < n ? -1 : j < n + m ? oR + x * m + j - n : orr + x;
            mo[r] = Hs + k2;
        }
    }
    int pi_[PP], pj[PP];
#pragma unroll
    for (int r = 0; r < PP; ++r) {
        const int e = tid + NT * r;
        pi_[r] = pj[r] = -1;
        if (e < nsym) upper_entry(e, n, pi_[r], pj[r]);
        else if (e < nP) {
            pi_[r] = e - nsym;
            pj[r] = n;
        }
    }
    const size_t sN = (size_t)s * E + N;
    for (int k2 = tid; k2 < nn; k2 += NT) {
        P[k2] = a.Q[sN * nn + k2];
        if (a.P) a.P[sN * nn + k2] = P[k2];
    }
    for (int i = tid; i < n; i += NT) {
        pp[i] = a.q[sN * n + i];
        if (a.p) a.p[sN * n + i] = pp[i];
    }
    if (N > 0) copy(N - 1, stg[(N - 1) & 1]);
    bool ok = true;
    for (int t = N - 1; t >= 0; --t) {
        const double *S = stg[t & 1];
        cp_async_wait_all();
        __syncthreads();  // this stage's data, P and p are there; the other buffer is free
        if (t > 0) copy(t - 1, stg[(t - 1) & 1]);
#pragma unroll
        for (int r = 0; r < PY; ++r)
            if (yi[r] >= 0) {
                const int e = tid + NT * r;
                Y[e] = dot_strided<CN>(P + yi[r] * n, 1, S + yo[r], ys[r], n, yo[r] == oc && ys[r] == 1 ? pp[yi[r]] : 0.0);
            }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < PM; ++r)
            if (ml[r] >= 0) *mo[r] = dot_strided<CN>(S + ml[r], ms[r], Y + mr[r], W, n, mi[r] >= 0 ? S[mi[r]] : 0.0);
        __syncthreads();
        const size_t st = (size_t)s * N + t;
        if (warp == solver) {
            // columns: Quu [m], then H [n] and qu
            const int at = lane < m ? n + lane : lane - m < n ? lane - m : n + m;
            double v[kLqMaxU];
#pragma unroll
            for (int i = 0; i < kLqMaxU; ++i) v[i] = i < m && lane <= n + m ? Hs[i * W + at] : 0.0;
            ok = gj_columns(v, m, lane) && ok;
            const int j = lane - m;
            if (j >= 0 && j <= n)
#pragma unroll
                for (int i = 0; i < kLqMaxU; ++i)
                    if (i < m) {
                        Ks[i * (n + 1) + j] = -v[i];
                        if (j < n) a.K[(st * m + i) * n + j] = -v[i];
                        else a.k[st * m + i] = -v[i];
                    }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < PP; ++r) {
            const int i = pi_[r], j = pj[r];
            if (i < 0) continue;
            const double v = dot_strided<CM>(Hs + i, W, Ks + j, n + 1, m, j < n ? Ms[i * n + j] : gs[i]);
            const size_t se = (size_t)s * E + t;
            if (j < n) {
                P[i * n + j] = v;
                P[j * n + i] = v;
                if (a.P) {
                    a.P[se * nn + i * n + j] = v;
                    a.P[se * nn + j * n + i] = v;
                }
            } else {
                pp[i] = v;
                if (a.p) a.p[se * n + i] = v;
            }
        }
    }
    if (warp == solver && lane == 0 && !ok) a.status[s] = 1;
}

__global__ void k_lq_reset(int *status, int S) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < S) status[i] = 0;
}

// workspace: two element buffers (scan; unused by the sequential form),
// then K, k, F, f; every region 256-byte aligned
struct LqWork {
    size_t buf0, buf1, K, k, F, f, bytes;
};

static LqWork lq_work(int n, int m, int N, int S) {
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    LqWork w;
    const size_t E = (size_t)N + 1;
    size_t o = 0;
    w.buf0 = o;
    o += al(sizeof(double) * (size_t)S * E * lq_es(n));
    w.buf1 = o;
    o += al(sizeof(double) * (size_t)S * E * lq_es(n));
    w.K = o;
    o += al(sizeof(double) * (size_t)S * N * m * n);
    w.k = o;
    o += al(sizeof(double) * (size_t)S * N * m);
    w.F = o;
    o += al(sizeof(double) * (size_t)S * N * n * n);
    w.f = o;
    o += al(sizeof(double) * (size_t)S * N * n);
    w.bytes = o;
    return w;
}

size_t lq_workspace_bytes(int n, int m, int N, int S) { return lq_work(n, m, N, S).bytes; }

template <int CN, int CM>
static cudaError_t launch_lq_dims(const LqArgs &a, int method, int n_sm, cudaStream_t st) {
    const int E = a.N + 1, S = a.S, N = a.N;
    if (method == 0) {
        k_lq_elem<CN, CM><<<dim3(E, S), 32, 0, st>>>(a);
        double *cur = a.buf0, *nxt = a.buf1;
        for (int d = 1; d < E; d *= 2) {
            k_lq_compose<CN><<<dim3(E, S), kLqThreads, 0, st>>>(a, cur, nxt, d);
            std::swap(cur, nxt);
        }
        k_lq_gains<CN, CM><<<dim3(E, S), kLqGainThreads, 0, st>>>(a, cur);
    } else {
        // a problem's two products have up to 204 and 158 entries: eight warps for the
        // larger dimensions (one entry per thread), two for up to six states
        constexpr int NT = CN > 6 ? 256 : 64;
        if (CN > 0 || a.n <= 6) k_lq_seq<CN, CM, NT><<<S, NT, 0, st>>>(a);
        else if constexpr (CN == 0) k_lq_seq<0, 0, 256><<<S, 256, 0, st>>>(a);
        if (N > 0) k_lq_closed<CN, CM><<<dim3(N, S), kLqGainThreads, 0, st>>>(a);
    }
    // The rollout's chain: N steps of one warp, or chunks of L steps whose maps are
    // formed side by side (n times the arithmetic), C map steps and L steps.  Chunks pay
    // from about 64 steps on and while their CTAs fit the GPU at once (two per SM): one
    // problem of 256 steps and 12 states 115 -> 41 us.
    const int L = std::max(8, (N + 63) / 64), C = N / L;
    if (N >= 64 && (long long)S * C <= 2 * n_sm) {
        // the last chunk takes the remainder, its map is not needed
        k_lq_chunk<CN><<<dim3(C, S), kLqThreads, 0, st>>>(a, a.buf0, L);
        k_lq_rollout<CN><<<dim3((N + L - 1) / L, S), 32, 0, st>>>(a, a.buf0, C, L);
    } else {
        k_lq_rollout<CN><<<dim3(1, S), 32, 0, st>>>(a, nullptr, 0, N);
    }
    if (N > 0) k_lq_controls<<<(unsigned)(((long long)S * N * a.m + 127) / 128), 128, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_lq(int method, int n, int m, int N, int S, const double *A, const double *B, const double *c,
                      const double *Q, const double *q, const double *R, const double *r, const double *s0, double *s,
                      double *u, double *P, double *p, int *status, void *work, int n_sm, cudaStream_t st) {
    const LqWork w = lq_work(n, m, N, S);
    unsigned char *wb = static_cast<unsigned char *>(work);
    LqArgs a;
    a.n = n;
    a.m = m;
    a.N = N;
    a.S = S;
    a.A = A;
    a.B = B;
    a.c = c;
    a.Q = Q;
    a.q = q;
    a.R = R;
    a.r = r;
    a.s0 = s0;
    a.s = s;
    a.u = u;
    a.P = P;
    a.p = p;
    a.status = status;
    a.buf0 = reinterpret_cast<double *>(wb + w.buf0);
    a.buf1 = reinterpret_cast<double *>(wb + w.buf1);
    a.K = reinterpret_cast<double *>(wb + w.K);
    a.k = reinterpret_cast<double *>(wb + w.k);
    a.F = reinterpret_cast<double *>(wb + w.F);
    a.f = reinterpret_cast<double *>(wb + w.f);
    k_lq_reset<<<(S + 255) / 256, 256, 0, st>>>(status, S);
    // the dimensions of the three vehicle models have their loops unrolled
    if (n == 4 && m == 2) return launch_lq_dims<4, 2>(a, method, n_sm, st);
    if (n == 5 && m == 2) return launch_lq_dims<5, 2>(a, method, n_sm, st);
    if (n == 12 && m == 4) return launch_lq_dims<12, 4>(a, method, n_sm, st);
    return launch_lq_dims<0, 0>(a, method, n_sm, st);
}

}  // namespace oca

using namespace oca;

extern "C" oca_status oca_lq_workspace_bytes(int32_t ns, int32_t nu, int32_t N, int32_t n_problems, int64_t *bytes) {
    if (!bytes || ns < 1 || nu < 1 || N < 0 || n_problems < 1) return OCA_ERR_INVALID_ARGUMENT;
    if (ns > kLqMaxS || nu > kLqMaxU || N > OCA_MAX_LQ_HORIZON || n_problems > 65535) return OCA_ERR_CAPACITY;
    *bytes = (int64_t)lq_workspace_bytes(ns, nu, N, n_problems);
    return OCA_OK;
}

extern "C" oca_status oca_lq_solve(oca_ctx *ctx, int32_t method, int32_t ns, int32_t nu, int32_t N, int32_t n_problems,
                                   const double *A, const double *B, const double *c, const double *Q, const double *q,
                                   const double *R, const double *r, const double *s0, double *s, double *u, double *P,
                                   double *p, int32_t *status, void *work, int64_t work_bytes, void *stream) {
    if (!ctx || (method != OCA_LQ_SCAN && method != OCA_LQ_SEQUENTIAL)) return OCA_ERR_INVALID_ARGUMENT;
    if (ns < 1 || nu < 1 || N < 0 || n_problems < 1) return OCA_ERR_INVALID_ARGUMENT;
    if (ns > kLqMaxS || nu > kLqMaxU || N > OCA_MAX_LQ_HORIZON || n_problems > 65535) return OCA_ERR_CAPACITY;
    if (!Q || !q || !s0 || !s || !status || !work) return OCA_ERR_INVALID_ARGUMENT;
    if (N > 0 && (!A || !B || !c || !R || !r || !u)) return OCA_ERR_INVALID_ARGUMENT;
    if (reinterpret_cast<uintptr_t>(work) % 256 != 0) return OCA_ERR_INVALID_ARGUMENT;
    if (work_bytes < (int64_t)lq_workspace_bytes(ns, nu, N, n_problems)) return OCA_ERR_CAPACITY;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const cudaError_t e = launch_lq(method == OCA_LQ_SCAN ? 0 : 1, ns, nu, N, n_problems, A, B, c, Q, q, R, r, s0, s,
                                    u, P, p, status, work, ctx_sm_count(ctx), st);
    return e == cudaSuccess ? OCA_OK : OCA_ERR_CUDA;
}
