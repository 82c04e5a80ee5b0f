// The Riccati step of the trajectory problem as a schedule of FP64 multiply-adds.
//
// GB300 issues one FP64 warp instruction per 64 cycles and scheduler (about one
// per 16 to 19 cycles and SM), however many of its lanes are active and however
// independent they are (measured with a chain and with eight independent
// chains: both 64 cycles).  So the cost of a stage is the number of FP64
// instructions that the warp issues, and the step is written to need few:
//   - only the products with entries of A_t and B_t that are not structurally 0
//     or 1 are formed (trailer: 224 multiply-adds per stage instead of 484,
//     quadrotor: about 1,800 instead of 5,080);
//   - the entries of each product are dealt out over the lanes of a scenario so
//     that every lane has about the same number of multiply-adds.
// Each lane runs a list of slots, acc = init + coef * val with the four operands
// and the result in the scenario's shared-memory region; the lists are built at
// compile time from the sparsity of the model's Jacobians.  The shared loads of
// a slot are free beside the 64 cycles of its multiply-add.
#pragma once

#include <stdint.h>

#include "oca_common.cuh"

namespace oca {

// ---- sparsity of s + dt f_c(s, u): entries of A - I and B that are not 0.
// Source index: >= 0 an entry of the stage record (in this order), -1 the
// constant dt.  A diagonal entry listed here replaces the implicit 1.
struct SpEntry {
    int row, col, src;
};

template <int KIND> struct RicSparse;
template <> struct RicSparse<0> {
    static constexpr int NA = 5, NB = 2, REC_A = 5, REC_B = 1;
    static constexpr SpEntry A[NA] = {{0, 2, 0}, {1, 2, 1}, {0, 3, 2}, {1, 3, 3}, {2, 3, 4}};
    static constexpr SpEntry B[NB] = {{3, 0, -1}, {2, 1, 0}};
    // record entry of A[i][k], B[i][k], or -1 (the same pairs, for device code)
    OCA_HD static constexpr int a_slot(int i, int k) { return k == 2 && i < 2 ? i : k == 3 && i < 3 ? 2 + i : -1; }
    OCA_HD static constexpr int b_slot(int i, int k) { return i == 2 && k == 1 ? 0 : -1; }
};
template <> struct RicSparse<1> {
    static constexpr int NA = 8, NB = 3, REC_A = 8, REC_B = 2;
    static constexpr SpEntry A[NA] = {{0, 2, 0}, {1, 2, 1}, {4, 2, 2}, {0, 3, 3}, {1, 3, 4}, {2, 3, 5}, {4, 3, 6}, {4, 4, 7}};
    static constexpr SpEntry B[NB] = {{3, 0, -1}, {2, 1, 0}, {4, 1, 1}};
    OCA_HD static constexpr int a_slot(int i, int k) {
        return k == 2 ? (i < 2 ? i : i == 4 ? 2 : -1) : k == 3 ? (i < 3 ? 3 + i : i == 4 ? 6 : -1) : k == 4 && i == 4 ? 7 : -1;
    }
    OCA_HD static constexpr int b_slot(int i, int k) { return k == 1 ? (i == 2 ? 0 : i == 4 ? 1 : -1) : -1; }
};
// 12-state quadrotor: positions and velocities, ZYX angles (6..8), body rates.  The
// thrust column of B is the same for the four rotors.
template <> struct RicSparse<2> {
    static constexpr int NA = 29, NB = 20, REC_A = 25, REC_B = 9;
    static constexpr SpEntry A[NA] = {{0, 3, -1}, {1, 4, -1}, {2, 5, -1},
                                      {3, 6, 0}, {3, 7, 1}, {3, 8, 2}, {4, 6, 3}, {4, 7, 4}, {4, 8, 5}, {5, 6, 6}, {5, 7, 7},
                                      {6, 6, 8}, {6, 7, 9}, {6, 9, -1}, {6, 10, 10}, {6, 11, 11},
                                      {7, 6, 12}, {7, 10, 13}, {7, 11, 14},
                                      {8, 6, 15}, {8, 7, 16}, {8, 10, 17}, {8, 11, 18},
                                      {9, 10, 19}, {9, 11, 20}, {10, 9, 21}, {10, 11, 22}, {11, 9, 23}, {11, 10, 24}};
    static constexpr SpEntry B[NB] = {{3, 0, 0}, {3, 1, 0}, {3, 2, 0}, {3, 3, 0}, {4, 0, 1}, {4, 1, 1}, {4, 2, 1}, {4, 3, 1},
                                      {5, 0, 2}, {5, 1, 2}, {5, 2, 2}, {5, 3, 2}, {9, 1, 3}, {9, 3, 4}, {10, 0, 5}, {10, 2, 6},
                                      {11, 0, 7}, {11, 1, 8}, {11, 2, 7}, {11, 3, 8}};
};
template <int KIND>
constexpr bool ric_slots_agree() {
    using SP = RicSparse<KIND>;
    for (int i = 0; i < MDims<KIND>::NS; ++i) {
        for (int k = 0; k < MDims<KIND>::NS; ++k) {
            int at = -1;
            for (int e = 0; e < SP::NA; ++e)
                if (SP::A[e].row == i && SP::A[e].col == k && SP::A[e].src >= 0) at = SP::A[e].src;
            if (at != SP::a_slot(i, k)) return false;
        }
        for (int k = 0; k < MDims<KIND>::NU; ++k) {
            int at = -1;
            for (int e = 0; e < SP::NB; ++e)
                if (SP::B[e].row == i && SP::B[e].col == k && SP::B[e].src >= 0) at = SP::B[e].src;
            if (at != SP::b_slot(i, k)) return false;
        }
    }
    return true;
}
static_assert(ric_slots_agree<0>() && ric_slots_agree<1>(), "a_slot, b_slot and the entry lists");

// Offsets (elements) of one scenario's shared region and of a stage record.
// Record: [A entries][B entries][c NS][q NS][r NU][Q upper triangle].
template <int KIND>
struct RicMap {
    static constexpr int NS = MDims<KIND>::NS, NU = MDims<KIND>::NU;
    using SP = RicSparse<KIND>;
    static constexpr int NSYM = NS * (NS + 1) / 2;
    // long products with vectors (P c + p, A^T w, B^T w) are summed in WS parts
    static constexpr int WS = NS > 6 ? 2 : 1;
    static constexpr int rA = 0, rB = SP::REC_A, rc = rB + SP::REC_B, rq = rc + NS, rr = rq + NS, rQ = rr + NU;
    static constexpr int REC = (rQ + NSYM + 1) & ~1;
    // shared region
    static constexpr int ZERO = 0, ONE = 1, DT = 2, TRASH = 3, RU = 4, REC0 = RU + NU;
    static constexpr int P0 = REC0 + REC, p0 = P0 + NSYM;
    static constexpr int Y0 = p0 + NS;           // Y[k][j] = (P A)[k][j], row-major (columns equal to P's are not formed)
    static constexpr int YB0 = Y0 + NS * NS;     // (P B)[k][x], only the rows that B touches
    static constexpr int W0 = YB0 + NS * NU;     // P c + p [part][k]
    static constexpr int M0 = W0 + WS * NS;      // Qss, upper triangle
    static constexpr int H0 = M0 + NSYM;         // Qus [x][j], then qu [x] (its first part) in column NS
    static constexpr int HQ1 = H0 + NU * (NS + 1);  // qu's second part [x]
    static constexpr int G0 = HQ1 + (WS - 1) * NU;  // qs [part][i]
    static constexpr int U0 = G0 + WS * NS;      // Quu, row-major upper
    static constexpr int K0 = U0 + NU * NU;      // K [x][j], k [x] in column NS
    static constexpr int F0 = K0 + NU * (NS + 1);  // F = A + B K (rows that B touches), then f in column NS
    static constexpr int SIZE = F0 + NS * (NS + 1);
    // global output of a stage: the rows of [F; K] (NZ x NS), then [f; k] (NZ)
    static constexpr int NZ = NS + NU, OUT = NZ * (NS + 1);
    // scratch of one scenario: records t = 0..N, outputs t < N, then s_0 and the
    // solution rows [s_{t+1}, u_t] of t < N
    __host__ __device__ static long long rec(int t) { return (long long)t * REC; }
    __host__ __device__ static long long out(int N, int t) { return (long long)(N + 1) * REC + (long long)t * OUT; }
    __host__ __device__ static long long s0(int N) { return out(N, N); }
    __host__ __device__ static long long sol(int N, int t) { return s0(N) + NS + (long long)t * NZ; }
    __host__ __device__ static long long size(int N) { return sol(N, N); }
    // behind them, the adjoint's vectors of t = 0..N: which = 0, 1 the sources Q x + q of
    // the forward and adjoint costates, 2, 3 the costates
    __host__ __device__ static long long adj(int N, int which, int t) {
        return size(N) + ((long long)which * (N + 1) + t) * NS;
    }
    __host__ __device__ static long long adj_size(int N) { return adj(N, 4, 0); }
    static constexpr int sym(int i, int j) { return i <= j ? i * NS - i * (i - 1) / 2 + (j - i) : sym(j, i); }
};

constexpr int kRicTerms = 14, kRicOps = 256;
struct RicOp {
    int init, store, n;
    int c[kRicTerms], v[kRicTerms];
};
struct RicOps {
    RicOp op[kRicOps];
    int n;
};
constexpr uint64_t kRicCont = 0xffff;  // init field: continue the lane's accumulator

// slots of one phase over L lanes: fields init, coef, val, store (16 bits each)
template <int SLOTS, int L>
struct RicPhase {
    uint64_t code[SLOTS][L];
};

template <int KIND>
struct RicBuild {
    using Mp = RicMap<KIND>;
    using SP = RicSparse<KIND>;
    static constexpr int NS = Mp::NS, NU = Mp::NU;

    static constexpr int a_src(int i) { return SP::A[i].src < 0 ? Mp::DT : Mp::REC0 + Mp::rA + SP::A[i].src; }
    static constexpr int b_src(int i) { return SP::B[i].src < 0 ? Mp::DT : Mp::REC0 + Mp::rB + SP::B[i].src; }
    // a listed diagonal entry of column j (or -1: the implicit 1)
    static constexpr int diag(int j) {
        for (int i = 0; i < SP::NA; ++i)
            if (SP::A[i].row == j && SP::A[i].col == j) return i;
        return -1;
    }
    static constexpr bool plain(int j) {
        for (int i = 0; i < SP::NA; ++i)
            if (SP::A[i].col == j) return false;
        return true;
    }
    static constexpr bool b_row(int k, int x) {
        for (int i = 0; i < SP::NB; ++i)
            if (SP::B[i].row == k && (x < 0 || SP::B[i].col == x)) return true;
        return false;
    }
    static constexpr int Yat(int k, int j) { return plain(j) ? Mp::P0 + Mp::sym(k, j) : Mp::Y0 + k * NS + j; }
    static constexpr void term(RicOp &o, int c, int v) {
        o.c[o.n] = c;
        o.v[o.n] = v;
        ++o.n;
    }
    static constexpr RicOp start(int init, int store) {
        RicOp o{};
        o.init = init;
        o.store = store;
        o.n = 0;
        return o;
    }
    static constexpr void add(RicOps &l, const RicOp &o) {
        l.op[l.n] = o;
        ++l.n;
    }
    // phase 1: Y = P A, the needed entries of P B, w = P c + p
    static constexpr RicOps phase_y() {
        RicOps l{};
        for (int k = 0; k < NS; ++k) {
            for (int j = 0; j < NS; ++j) {
                if (plain(j)) continue;
                RicOp o = start(diag(j) < 0 ? Mp::P0 + Mp::sym(k, j) : Mp::ZERO, Mp::Y0 + k * NS + j);
                for (int i = 0; i < SP::NA; ++i)
                    if (SP::A[i].col == j) term(o, a_src(i), Mp::P0 + Mp::sym(k, SP::A[i].row));
                add(l, o);
            }
            for (int x = 0; x < NU; ++x) {
                // (P B)[k][x] enters Quu[y][x], y <= x, for the columns y that have row k
                bool need = false;
                for (int y = 0; y <= x; ++y) need = need || b_row(k, y);
                if (!need) continue;
                RicOp o = start(Mp::ZERO, Mp::YB0 + k * NU + x);
                for (int i = 0; i < SP::NB; ++i)
                    if (SP::B[i].col == x) term(o, b_src(i), Mp::P0 + Mp::sym(k, SP::B[i].row));
                add(l, o);
            }
            for (int w = 0; w < Mp::WS; ++w) {
                RicOp o = start(w == 0 ? Mp::p0 + k : Mp::ZERO, Mp::W0 + w * NS + k);
                for (int i = w * NS / Mp::WS; i < (w + 1) * NS / Mp::WS; ++i) term(o, Mp::REC0 + Mp::rc + i, Mp::P0 + Mp::sym(k, i));
                add(l, o);
            }
        }
        return l;
    }
    // row i of A^T times column vector v(l)
    static constexpr void at_terms(RicOp &o, int i, int base, int stride, int j) {
        for (int l = 0; l < NS; ++l) {
            if (l == i && diag(i) < 0) term(o, Mp::ONE, j >= 0 ? Yat(l, j) : base + l * stride);
            for (int e = 0; e < SP::NA; ++e)
                if (SP::A[e].row == l && SP::A[e].col == i) term(o, a_src(e), j >= 0 ? Yat(l, j) : base + l * stride);
        }
    }
    // phase 2: Qss (upper), Qus, Quu (upper), qs, qu
    static constexpr RicOps phase_m() {
        RicOps l{};
        for (int i = 0; i < NS; ++i) {
            for (int j = i; j < NS; ++j) {
                RicOp o = start(Mp::REC0 + Mp::rQ + Mp::sym(i, j), Mp::M0 + Mp::sym(i, j));
                at_terms(o, i, 0, 0, j);
                add(l, o);
            }
            for (int w = 0; w < Mp::WS; ++w) {
                RicOp o = start(w == 0 ? Mp::REC0 + Mp::rq + i : Mp::ZERO, Mp::G0 + w * NS + i);
                at_terms(o, i, Mp::W0 + w * NS, 1, -1);
                add(l, o);
            }
        }
        for (int x = 0; x < NU; ++x) {
            for (int j = 0; j <= NS; ++j) {
                RicOp o = start(j < NS ? Mp::ZERO : Mp::REC0 + Mp::rr + x, Mp::H0 + x * (NS + 1) + j);
                for (int i = 0; i < SP::NB; ++i)
                    if (SP::B[i].col == x) term(o, b_src(i), j < NS ? Yat(SP::B[i].row, j) : Mp::W0 + SP::B[i].row);
                add(l, o);
            }
            if (Mp::WS > 1) {
                RicOp o = start(Mp::ZERO, Mp::HQ1 + x);
                for (int i = 0; i < SP::NB; ++i)
                    if (SP::B[i].col == x) term(o, b_src(i), Mp::W0 + NS + SP::B[i].row);
                add(l, o);
            }
            for (int y = x; y < NU; ++y) {
                RicOp o = start(x == y ? Mp::RU + x : Mp::ZERO, Mp::U0 + x * NU + y);
                for (int i = 0; i < SP::NB; ++i)
                    if (SP::B[i].col == x) term(o, b_src(i), Mp::YB0 + SP::B[i].row * NU + y);
                add(l, o);
            }
        }
        return l;
    }
    // phase 3: P = Qss + Qus^T K, p = qs + Qus^T k, F = A + B K, f = c + B k
    static constexpr RicOps phase_p() {
        RicOps l{};
        for (int i = 0; i < NS; ++i) {
            for (int j = i; j < NS; ++j) {
                RicOp o = start(Mp::M0 + Mp::sym(i, j), Mp::P0 + Mp::sym(i, j));
                for (int x = 0; x < NU; ++x) term(o, Mp::H0 + x * (NS + 1) + i, Mp::K0 + x * (NS + 1) + j);
                add(l, o);
            }
            RicOp o = start(Mp::G0 + i, Mp::p0 + i);
            if (Mp::WS > 1) term(o, Mp::ONE, Mp::G0 + NS + i);
            for (int x = 0; x < NU; ++x) term(o, Mp::H0 + x * (NS + 1) + i, Mp::K0 + x * (NS + 1) + NS);
            add(l, o);
        }
        for (int i = 0; i < NS; ++i) {
            if (!b_row(i, -1)) continue;
            for (int j = 0; j <= NS; ++j) {
                RicOp o = start(j < NS ? a_at(i, j) : Mp::REC0 + Mp::rc + i, Mp::F0 + i * (NS + 1) + j);
                for (int e = 0; e < SP::NB; ++e)
                    if (SP::B[e].row == i) term(o, b_src(e), Mp::K0 + SP::B[e].col * (NS + 1) + j);
                add(l, o);
            }
        }
        return l;
    }
    // where A[i][j] is read
    static constexpr int a_at(int i, int j) {
        for (int e = 0; e < SP::NA; ++e)
            if (SP::A[e].row == i && SP::A[e].col == j) return a_src(e);
        return i == j ? Mp::ONE : Mp::ZERO;
    }
    // shared offset of element e of a stage's global output
    static constexpr int out_at(int e) {
        constexpr int NZ = Mp::NZ;
        const int i = e < NZ * NS ? e / NS : e - NZ * NS, j = e < NZ * NS ? e % NS : NS;
        if (i >= NS) return Mp::K0 + (i - NS) * (NS + 1) + j;
        if (b_row(i, -1)) return Mp::F0 + i * (NS + 1) + j;
        return j < NS ? a_at(i, j) : Mp::REC0 + Mp::rc + i;
    }

    static constexpr RicOps ops(int phase) { return phase == 0 ? phase_y() : phase == 1 ? phase_m() : phase_p(); }

    // longest-first onto the least loaded lane; returns the number of slots
    template <int L, class Put>
    static constexpr int deal(const RicOps &l, Put put) {
        int load[L] = {};
        bool done[kRicOps] = {};
        int slots = 0;
        for (int k = 0; k < l.n; ++k) {
            int best = -1;
            for (int e = 0; e < l.n; ++e)
                if (!done[e] && (best < 0 || l.op[e].n > l.op[best].n)) best = e;
            done[best] = true;
            int lane = 0;
            for (int q = 1; q < L; ++q)
                if (load[q] < load[lane]) lane = q;
            const RicOp &o = l.op[best];
            for (int i = 0; i < o.n; ++i) put(load[lane] + i, lane, o, i);
            load[lane] += o.n;
            if (load[lane] > slots) slots = load[lane];
        }
        return slots;
    }
    struct Count {
        constexpr void operator()(int, int, const RicOp &, int) const {}
    };
    template <int L>
    static constexpr int slots(int phase) {
        return deal<L>(ops(phase), Count{});
    }
    static constexpr uint64_t word(uint64_t init, uint64_t c, uint64_t v, uint64_t st) {
        return init | (c << 16) | (v << 32) | (st << 48);
    }
    template <int SLOTS, int L>
    struct Fill {
        RicPhase<SLOTS, L> *p;
        constexpr void operator()(int slot, int lane, const RicOp &o, int i) const {
            p->code[slot][lane] = word(i == 0 ? (uint64_t)o.init : kRicCont, o.c[i], o.v[i], i == o.n - 1 ? o.store : Mp::TRASH);
        }
    };
    template <int PHASE, int L>
    static constexpr auto table() {
        constexpr int SL = slots<L>(PHASE);
        RicPhase<SL, L> t{};
        for (int s = 0; s < SL; ++s)
            for (int q = 0; q < L; ++q) t.code[s][q] = word(Mp::ZERO, Mp::ZERO, Mp::ZERO, Mp::TRASH);
        deal<L>(ops(PHASE), Fill<SL, L>{&t});
        return t;
    }
    struct OutMap {
        uint16_t at[Mp::OUT];
    };
    static constexpr OutMap out_map() {
        OutMap m{};
        for (int e = 0; e < Mp::OUT; ++e) m.at[e] = (uint16_t)out_at(e);
        return m;
    }
};

}  // namespace oca
