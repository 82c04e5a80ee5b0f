// The slot lists of the trajectory recursion (oca_ricprog.cuh), run on the host
// lane by lane with random stage data, against dense products: P A, P B, P c + p,
// the stage matrix, P_t and the closed-loop rows.  Prints "kind lanes slots error"
// per schedule; exits 1 on an operand outside the region, a result stored twice or
// a difference above 1e-12.
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "oca_ricprog.cuh"

using namespace oca;

static double rnd() { return rand() / (double)RAND_MAX - 0.5; }
static double worst;
static void check(double a, double b, const char *what) {
    const double e = std::fabs(a - b);
    if (!(e < 1e-12)) {
        std::printf("%s: %g, dense %g\n", what, a, b);
        std::exit(1);
    }
    if (e > worst) worst = e;
}

template <int SLOTS, int L, int SIZE, int TRASH>
static void run(const RicPhase<SLOTS, L> &t, double *sm) {
    double out[SIZE];
    bool wrote[SIZE] = {};
    for (int l = 0; l < L; ++l) {
        double acc = NAN;
        for (int s = 0; s < SLOTS; ++s) {
            const uint64_t w = t.code[s][l];
            const int in = w & 0xffff, c = (w >> 16) & 0xffff, v = (w >> 32) & 0xffff, st = (int)(w >> 48);
            if (c >= SIZE || v >= SIZE || st >= SIZE || (in != (int)kRicCont && in >= SIZE)) {
                std::printf("operand outside the region\n");
                std::exit(1);
            }
            acc = std::fma(sm[c], sm[v], in == (int)kRicCont ? acc : sm[in]);
            if (st == TRASH) continue;
            if (wrote[st]) {
                std::printf("result %d stored twice\n", st);
                std::exit(1);
            }
            wrote[st] = true;
            out[st] = acc;
        }
    }
    for (int i = 0; i < SIZE; ++i)
        if (wrote[i]) sm[i] = out[i];
}

template <int KIND, int L>
static void test() {
    using Bd = RicBuild<KIND>;
    using Mp = RicMap<KIND>;
    constexpr int NS = Mp::NS, NU = Mp::NU;
    static constexpr auto ty = Bd::template table<0, L>();
    static constexpr auto tm = Bd::template table<1, L>();
    static constexpr auto tp = Bd::template table<2, L>();
    static constexpr auto om = Bd::out_map();
    worst = 0.0;
    double sm[Mp::SIZE];
    for (double &x : sm) x = NAN;
    sm[Mp::ZERO] = 0.0;
    sm[Mp::ONE] = 1.0;
    sm[Mp::DT] = 0.1;
    for (int i = 0; i < NU; ++i) sm[Mp::RU + i] = 5.0 + i;
    for (int i = 0; i < Mp::REC; ++i) sm[Mp::REC0 + i] = rnd();
    for (int i = 0; i < Mp::NSYM + NS; ++i) sm[Mp::P0 + i] = rnd();
    double A[NS][NS] = {}, B[NS][NU] = {}, P[NS][NS], Q[NS][NS], c[NS], q[NS], r[NU], p[NS];
    for (int i = 0; i < NS; ++i) {
        A[i][i] = 1.0;
        c[i] = sm[Mp::REC0 + Mp::rc + i];
        q[i] = sm[Mp::REC0 + Mp::rq + i];
        p[i] = sm[Mp::p0 + i];
        for (int j = 0; j < NS; ++j) {
            P[i][j] = sm[Mp::P0 + Mp::sym(i, j)];
            Q[i][j] = sm[Mp::REC0 + Mp::rQ + Mp::sym(i, j)];
        }
    }
    for (int i = 0; i < NU; ++i) r[i] = sm[Mp::REC0 + Mp::rr + i];
    for (const SpEntry &e : RicSparse<KIND>::A) A[e.row][e.col] = e.src < 0 ? 0.1 : sm[Mp::REC0 + Mp::rA + e.src];
    for (const SpEntry &e : RicSparse<KIND>::B) B[e.row][e.col] = e.src < 0 ? 0.1 : sm[Mp::REC0 + Mp::rB + e.src];
    run<sizeof(ty.code) / sizeof(ty.code[0]), L, Mp::SIZE, Mp::TRASH>(ty, sm);
    run<sizeof(tm.code) / sizeof(tm.code[0]), L, Mp::SIZE, Mp::TRASH>(tm, sm);
    double PA[NS][NS], w[NS];
    for (int i = 0; i < NS; ++i) {
        w[i] = p[i];
        for (int j = 0; j < NS; ++j) {
            w[i] += P[i][j] * c[j];
            PA[i][j] = 0.0;
            for (int l = 0; l < NS; ++l) PA[i][j] += P[i][l] * A[l][j];
        }
    }
    for (int i = 0; i < NS; ++i) {
        for (int j = i; j < NS; ++j) {
            double v = Q[i][j];
            for (int l = 0; l < NS; ++l) v += A[l][i] * PA[l][j];
            check(sm[Mp::M0 + Mp::sym(i, j)], v, "Qss");
        }
        double v = q[i];
        for (int l = 0; l < NS; ++l) v += A[l][i] * w[l];
        check(sm[Mp::G0 + i] + (Mp::WS > 1 ? sm[Mp::G0 + NS + i] : 0.0), v, "qs");
    }
    for (int x = 0; x < NU; ++x) {
        for (int j = 0; j < NS; ++j) {
            double v = 0.0;
            for (int l = 0; l < NS; ++l) v += B[l][x] * PA[l][j];
            check(sm[Mp::H0 + x * (NS + 1) + j], v, "Qus");
        }
        double v = r[x];
        for (int l = 0; l < NS; ++l) v += B[l][x] * w[l];
        check(sm[Mp::H0 + x * (NS + 1) + NS] + (Mp::WS > 1 ? sm[Mp::HQ1 + x] : 0.0), v, "qu");
        for (int y = x; y < NU; ++y) {
            double u = x == y ? 5.0 + x : 0.0;
            for (int l = 0; l < NS; ++l)
                for (int k = 0; k < NS; ++k) u += B[l][x] * P[l][k] * B[k][y];
            check(sm[Mp::U0 + x * NU + y], u, "Quu");
        }
    }
    for (int i = 0; i < NU * (NS + 1); ++i) sm[Mp::K0 + i] = rnd();
    double old[Mp::SIZE];
    for (int i = 0; i < Mp::SIZE; ++i) old[i] = sm[i];
    run<sizeof(tp.code) / sizeof(tp.code[0]), L, Mp::SIZE, Mp::TRASH>(tp, sm);
    auto K = [&](int x, int j) { return old[Mp::K0 + x * (NS + 1) + j]; };
    auto H = [&](int x, int j) { return old[Mp::H0 + x * (NS + 1) + j]; };
    for (int i = 0; i < NS; ++i) {
        for (int j = i; j < NS; ++j) {
            double v = old[Mp::M0 + Mp::sym(i, j)];
            for (int x = 0; x < NU; ++x) v += H(x, i) * K(x, j);
            check(sm[Mp::P0 + Mp::sym(i, j)], v, "P");
        }
        double v = old[Mp::G0 + i] + (Mp::WS > 1 ? old[Mp::G0 + NS + i] : 0.0);
        for (int x = 0; x < NU; ++x) v += H(x, i) * K(x, NS);
        check(sm[Mp::p0 + i], v, "p");
    }
    for (int e = 0; e < Mp::OUT; ++e) {
        const int i = e < Mp::NZ * NS ? e / NS : e - Mp::NZ * NS, j = e < Mp::NZ * NS ? e % NS : NS;
        double v;
        if (i >= NS) {
            v = K(i - NS, j);
        } else {
            v = j < NS ? A[i][j] : c[i];
            for (int x = 0; x < NU; ++x) v += B[i][x] * K(x, j);
        }
        check(sm[om.at[e]], v, "output row");
    }
    std::printf("%d %d %d %.2g\n", KIND, L,
                (int)((sizeof(ty.code) + sizeof(tm.code) + sizeof(tp.code)) / sizeof(ty.code[0])), worst);
}

int main() {
    test<0, 16>();
    test<0, 32>();
    test<1, 16>();
    test<1, 32>();
    test<2, 128>();
    return 0;
}
