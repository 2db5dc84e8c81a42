// Test helper: how far Green functions are from exact Sherman-Morrison updates after some sweeps.
//
// Every chain starts from given matrices and fields and is carried through nsweep sweeps twice, in
// 113-bit arithmetic, which makes the decisions, and in FP64 with one rounded multiply-add per element
// (the rank-1 update as the method states it).  Compiled with g++ by test_gpu_f64_accuracy.py.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <thread>
#include <vector>

#if defined(__aarch64__)
typedef long double Quad;   // IEEE binary128 there
#else
typedef __float128 Quad;
#endif

namespace {

struct Job {
    int L, nsweep;
    double a_p, a_m;       // e^{-2 lambda} - 1 (sigma s = +1), e^{+2 lambda} - 1 (= -1)
    const double* G0;      // [chain][2][L*L]
    const int8_t* s0;      // [chain][L]
    const double* u;       // [chain][nsweep][L]
    const double* G;       // [chain][2][L*L] the matrices to be judged
    double* err;           // [chain][2] max |G - exact| / max |exact|
    double* err64;         // [chain][2] the same of the FP64 updates
    int8_t* s;             // [chain][L] fields after the sweeps
};

void run(const Job& J, int c) {
    const int L = J.L, LL = L * L;
    std::vector<Quad> q[2], col(L), row(L);
    std::vector<double> d[2], dcol(L), drow(L);
    std::vector<int> s(J.s0 + c * L, J.s0 + (c + 1) * L);
    for (int sp = 0; sp < 2; ++sp) {
        const double* g = J.G0 + (static_cast<size_t>(c) * 2 + sp) * LL;
        q[sp].assign(g, g + LL);
        d[sp].assign(g, g + LL);
    }
    for (int w = 0; w < J.nsweep; ++w)
        for (int l = 0; l < L; ++l) {
            const double a[2] = {s[l] > 0 ? J.a_p : J.a_m, s[l] > 0 ? J.a_m : J.a_p};
            const Quad R[2] = {1 + (1 - q[0][l * L + l]) * Quad(a[0]), 1 + (1 - q[1][l * L + l]) * Quad(a[1])};
            if (!(Quad(J.u[(static_cast<size_t>(c) * J.nsweep + w) * L + l]) < R[0] * R[1])) continue;
            for (int sp = 0; sp < 2; ++sp) {
                const Quad f = Quad(a[sp]) / R[sp];
                const double f64 = a[sp] / (1.0 + (1.0 - d[sp][l * L + l]) * a[sp]);
                for (int i = 0; i < L; ++i) {
                    col[i] = f * (q[sp][i * L + l] - (i == l ? 1 : 0));
                    row[i] = q[sp][l * L + i];
                    dcol[i] = f64 * (d[sp][i * L + l] - (i == l ? 1.0 : 0.0));
                    drow[i] = d[sp][l * L + i];
                }
                for (int i = 0; i < L; ++i)
                    for (int j = 0; j < L; ++j) {
                        q[sp][i * L + j] += col[i] * row[j];
                        d[sp][i * L + j] = std::fma(dcol[i], drow[j], d[sp][i * L + j]);
                    }
            }
            s[l] = -s[l];
        }
    for (int sp = 0; sp < 2; ++sp) {
        const double* g = J.G + (static_cast<size_t>(c) * 2 + sp) * LL;
        double big = 0.0, e = 0.0, e64 = 0.0;
        for (int i = 0; i < LL; ++i) {
            big = std::max(big, std::fabs(static_cast<double>(q[sp][i])));
            const double x = std::fabs(static_cast<double>(Quad(g[i]) - q[sp][i]));
            e = x > e || x != x ? x : e;
            e64 = std::max(e64, std::fabs(static_cast<double>(Quad(d[sp][i]) - q[sp][i])));
        }
        J.err[c * 2 + sp] = e / big;
        J.err64[c * 2 + sp] = e64 / big;
    }
    for (int l = 0; l < L; ++l) J.s[c * L + l] = static_cast<int8_t>(s[l]);
}

}  // namespace

extern "C" void green_errors(int L, int nchain, int nsweep, double a_p, double a_m, const double* G0,
                             const int8_t* s0, const double* u, const double* G, double* err,
                             double* err64, int8_t* s) {
    const Job J{L, nsweep, a_p, a_m, G0, s0, u, G, err, err64, s};
    std::vector<std::thread> pool;
    const int nt = std::max(1, std::min<int>(16, std::thread::hardware_concurrency()));
    for (int t = 0; t < nt; ++t)
        pool.emplace_back([&J, t, nt, nchain] {
            for (int c = t; c < nchain; c += nt) run(J, c);
        });
    for (std::thread& t : pool) t.join();
}
