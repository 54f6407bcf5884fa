// Runs the FP64 right-hand side and steps (csrc/cme_fixed.cuh, fix_rk4ip_step, fix_strang_kerr) of
// one launch shape (log2 N = CASE_LOGN, CASE_R values per thread) on the host.  Built with overflow checks on every signed
// operation, it stops at the first sum, product or shift that leaves 64 bits.
//
//   fixed idft|rhs|rk4ip|strang <g0> <kappa> <pump> <h> <steps> <fields in> <fields out>
//
// Fields: N complex numbers each, transform order.  Detuning 1, flat dispersion.
#include <stdio.h>
#include <stdlib.h>

#include "cuda_runtime.h"

#define CME_HOST_PRIMITIVES
namespace cme {
inline namespace fp32_packed {
inline long long fwide(int a, int b) { return (long long)a * b; }
inline long long fmad(int a, int b, long long c) { return (long long)a * b + c; }
inline long long fshl(long long v, int s) { return v * (1LL << s); }
template <typename V> inline void park_store(V* p, V v) { *p = v; }
template <typename V> inline V park_load(const V* p) { return *p; }
}
}
#include "cme_step.cuh"

using namespace cme;
using GR = Group<double, CASE_LOGN, CASE_R>;
constexpr int N = GR::N, P = GR::P, T = P < 32 ? 32 : P, G = T / P;
inline int host_threads() { return T; }

static int4 limbs(double re, double im, long long one = 0)
{
    const fl r = fsplit(llrint(re * 0x1p62) + (one << 62)), i = fsplit(llrint(im * 0x1p62));
    return {r.h, r.l, i.h, i.l};
}

int main(int argc, char** argv)
{
    const bool idft = !strcmp(argv[1], "idft"), rhs = !strcmp(argv[1], "rhs"),
               strang = !strcmp(argv[1], "strang");
    const double g0 = atof(argv[2]), kappa = atof(argv[3]), pump = atof(argv[4]), h = atof(argv[5]);
    const int steps = atoi(argv[6]);
    std::vector<int4> tw(N), Ef(N);
    std::vector<cx<double>> E(N), e1(N), e2(N);
    const long double pi = acosl(-1.0L);
    const long double lr = -0.5L * kappa, li = -1.0L;
    const auto expm1c = [](long double x, long double y) -> cx<double> {
        const long double s = sinl(y / 2);
        return {(double)(expm1l(x) * cosl(y) - 2 * s * s), (double)(expl(x) * sinl(y))};
    };
    const cx<double> p1 = expm1c(lr * h / 2, li * h / 2), p2 = expm1c(lr * h, li * h);
    for (int k = 0; k < N; ++k) {
        tw[k] = limbs((double)cosl(2 * pi * k / N), (double)sinl(2 * pi * k / N));
        Ef[k] = limbs(p1.re, p1.im, 1);
        E[k] = {p1.re + 1.0, p1.im};
        e1[k] = p1;
        e2[k] = p2;
    }
    // pump increments of the split step: pump (exp(L t) - 1) / L, t = h/2 and h
    const auto over_L = [&](cx<double> e) -> cx<double> {
        const long double d = lr * lr + li * li;
        return {(double)(pump * (e.re * lr + e.im * li) / d),
                (double)(pump * (e.im * lr - e.re * li) / d)};
    };
    StepArgs a{};
    a.E = E.data();
    a.e1 = e1.data();
    a.e2 = e2.data();
    a.Ef = Ef.data();
    StepConsts<double> c{};
    c.pump = {pump, 0.0};
    c.cp = over_L(p1);
    c.cp2 = over_L(p2);
    c.gN = g0 / N;
    c.g0h = g0 * h * 0.5;
    c.h = h;
    c.hh = 0.5 * h;
    c.h6 = h / 6.0;

    FILE* in = fopen(argv[7], "rb");
    FILE* out = fopen(argv[8], "wb");
    std::vector<unsigned char> smem(G * group_smem_bytes(8, CASE_LOGN, CASE_R));
    std::vector<cx<double>> D(G * N);
    size_t n;
    while ((n = fread(D.data(), N * 16, G, in)) > 0) {
        for (size_t g = n; g < (size_t)G; ++g)
            std::copy_n(D.begin(), N, D.begin() + g * N);
        host::run_block(T, [&] {
            const int g = threadIdx.x / P;
            GR grp;
            grp.setup(smem.data(), g, threadIdx.x - g * P, tw.data());
            FieldState<double, CASE_LOGN, CASE_R> fs;
            fs.bind(grp);
            cx<double>* d = D.data() + g * N + grp.t;
            fs.load(d, d);
            Props<double, CASE_LOGN, CASE_R> pr;
            pr.init(a, 0, grp.t);
            if (idft) {
                grp.inverse(fs.Dh, 0);
            } else if (rhs) {
                grp.rhs(fs.Dh, c.gN, c.pump);
            } else if (strang) {
                strang_steps(grp, fs, pr, c, steps);
            } else {
                for (int k = 0; k < steps; ++k)
                    rk4ip_step<false, false>(grp, fs, pr, c, d, (cx<double>*)nullptr, 0);
            }
            fs.store(d, d);
        });
        fwrite(D.data(), N * 16, n, out);
    }
    return fclose(out);
}
