// Host check of the integer collision (csrc/lb_fixed.cuh): nodes of a given mean
// density (in units of 2^e) around rest, collided in integers, in FP64 and in
// quadruple precision.  Prints one line per density:
//   density, nodes taken by the integers, rms error of the integers and of FP64
//   (in units of the node's density), worst error of the integers in units of
//   2^(e - 60) beyond half a unit of the result's last place, mean change of the
//   mass in a step (integers, FP64).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "lb_fixed.cuh"
#include "lbmd_ctx.h"

using namespace lbmd;
#ifdef __aarch64__
typedef long double Quad;
#else
typedef __float128 Quad;
#endif

struct Noise {
    unsigned w[8];
    double g[Q];
    unsigned bits(int k) const { return ((k - 4) & 1) ? w[(k - 4) >> 1] >> 16 : w[(k - 4) >> 1] & 0xffffu; }
    double normal(int k) const { return g[k]; }
};

// The collision of lb_core.cuh from its formulas, mode by mode.
template <typename T>
static void collide_by_modes(const double f0[Q], const T J[3], const double g[3], double gs, const T xi[Q], bool C,
                             T out[Q]) {
    T f[Q], m[Q], rho = 0, j[3] = {0, 0, 0}, F[3];
    for (int i = 0; i < Q; ++i) {
        f[i] = f0[i];
        rho += f[i];
        j[0] += f[i] * CX(i);
        j[1] += f[i] * CY(i);
        j[2] += f[i] * CZ(i);
    }
    auto weight = [](int i) { return C2(i) == 0 ? (T)1 / 3 : C2(i) == 1 ? (T)1 / 18 : (T)1 / 36; };
    auto norm = [&](int k) {
        T b = 0;
        for (int i = 0; i < Q; ++i) b += weight(i) * EMODE(k, i) * EMODE(k, i);
        return b;
    };
    auto products = [](const T u[3], const T v[3], T h[10]) {
        const T uv = u[0] * v[0] + u[1] * v[1] + u[2] * v[2];
        h[4] = uv;
        h[5] = 3 * u[0] * v[0] - uv;
        h[6] = u[1] * v[1] - u[2] * v[2];
        h[7] = (u[0] * v[1] + u[1] * v[0]) / 2;
        h[8] = (u[0] * v[2] + u[2] * v[0]) / 2;
        h[9] = (u[1] * v[2] + u[2] * v[1]) / 2;
    };
    for (int k = 0; k < Q; ++k) {
        m[k] = 0;
        for (int i = 0; i < Q; ++i) m[k] += f[i] * EMODE(k, i);
    }
    T u[3], h[10];
    for (int c = 0; c < 3; ++c) F[c] = C ? (T)g[c] : J[c] + (T)g[c];
    if (C) {
        for (int c = 0; c < 3; ++c) u[c] = (j[c] + J[c] / 2) / rho;
        products(u, J, h);
        for (int c = 0; c < 3; ++c) j[c] += J[c];
        m[4] += h[4];
        for (int k = 5; k < 10; ++k) m[k] += (1 + (T)gs) * h[k];
    }
    for (int c = 0; c < 3; ++c) u[c] = (j[c] + F[c] / 2) / rho;
    T eq[10];
    products(u, u, eq);
    products(u, F, h);
    m[0] = rho;
    for (int c = 0; c < 3; ++c) m[1 + c] = j[c] + F[c];
    for (int k = 4; k < Q; ++k) {
        const T e = k < 10 ? rho * eq[k] : (T)0, gk = k >= 5 && k < 10 ? (T)gs : (T)0;
        m[k] = e + gk * (m[k] - e) + (k < 10 ? (1 + gk) * h[k] : (T)0) + xi[k];
    }
    for (int i = 0; i < Q; ++i) {
        T a = 0;
        for (int k = 0; k < Q; ++k) a += m[k] * EMODE(k, i) / norm(k);
        out[i] = weight(i) * a;
    }
}

static Quad quad_sqrt(Quad v) {
    Quad s = std::sqrt((double)v);
    for (int i = 0; i < 3; ++i) s = (s + v / s) / 2;
    return s;
}

template <bool C>
static void run(double rel, double rho0, int nodes, unsigned seed) {
    std::mt19937_64 gen(seed);
    std::uniform_real_distribution<double> U(-1, 1);
    int E;
    const int e = std::frexp(rho0, &E) == 0.5 ? E - 1 : E;
    const double unit = std::ldexp(1.0, e), mean = rel * unit;
    long taken = 0;
    double s = 0, s64 = 0, worst = 0, dm = 0, dm64 = 0;
    for (int t = 0; t < nodes; ++t) {
        LbCoeffs co;
        lb_coefficients(t % 2 ? 1.0 / 6 : 0.05, -1.0, 0.0, t % 3 ? 1e-3 : 1e-5, co);
        for (int k = 0; k < Q; ++k) co.noise_amp[k] *= std::sqrt(rho0);
        const double g[3] = {1e-5 * rho0, -2e-6 * rho0, 0.0};
        const FixedArgs a = fixed_constants(e, co.noise_amp, g);
        double f[Q], out[Q], xd[Q], Jd[3];
        for (int i = 0; i < Q; ++i) f[i] = mean * WEIGHT(i) * (1 + 0.05 * U(gen));
        long long J[3];
        for (auto &v : J) v = (long long)(U(gen) * std::ldexp(rel, 56) * 1e-3);
        Noise noise;
        for (auto &w : noise.w) w = (unsigned)gen();
        FixedMoments o;
        if (!a.usable || !fixed_moments_in_range(f, e, o)) continue;
        if (!collide_fixed<C, false>(o, J, co.gamma_shear, g, a, true, noise, out)) continue;
        ++taken;
        Quad Jq[3], xq[Q], oq[Q], rho = 0;
        double od[Q], rd = 0;
        for (int i = 0; i < Q; ++i) {
            rho += (Quad)f[i];
            rd += f[i];
        }
        const Quad sq = quad_sqrt(rho);
        for (int c = 0; c < 3; ++c) {
            Jd[c] = std::ldexp((double)J[c], e - 56);
            Jq[c] = (Quad)J[c] * (Quad)std::ldexp(1.0, e - 56);
        }
        for (int k = 0; k < Q; ++k) {
            xq[k] = xd[k] = 0;
            if (k < 4) continue;
            xq[k] = (Quad)co.noise_amp[k] * (2 * quad_sqrt((Quad)3)) * sq * ((Quad)noise.bits(k) - (Quad)32767.5) / 65536;
            xd[k] = co.noise_amp[k] * 3.4641016151377544 * 1.52587890625e-05 * std::sqrt(rd) * (noise.bits(k) - 32767.5);
        }
        collide_by_modes<Quad>(f, Jq, g, co.gamma_shear, xq, C, oq);
        collide_by_modes<double>(f, Jd, g, co.gamma_shear, xd, C, od);
        Quad m = 0, m64 = 0;
        for (int i = 0; i < Q; ++i) {
            const double d = (double)((Quad)out[i] - oq[i]), d64 = (double)((Quad)od[i] - oq[i]);
            s += d * d;
            s64 += d64 * d64;
            int x;
            std::frexp((double)oq[i], &x);
            const double half = std::ldexp(1.0, x - 54);  // half a unit of the last place
            worst = std::fmax(worst, (std::fabs(d) - half) / (unit * std::ldexp(1.0, -60)));
            m += (Quad)out[i];
            m64 += (Quad)od[i];
        }
        dm += (double)(m - rho) / (double)rho;
        dm64 += (double)(m64 - rho) / (double)rho;
    }
    const double n = taken ? taken : 1;
    std::printf("%.6f %ld %.4g %.4g %.4g %.3g %.3g\n", rel, taken, std::sqrt(s / (19 * n)) / mean,
                std::sqrt(s64 / (19 * n)) / mean, worst, dm / n, dm64 / n);
}

// rho_factors_fixed against quadruple precision over 2^lo .. 2^hi: the worst
// errors of 1/rho and sqrt(rho) in units of the last place of the result
static void factors(int lo, int hi, int count) {
    std::mt19937_64 gen(5);
    std::uniform_real_distribution<double> U(0, 1);
    double wi = 0, ws = 0;
    for (int t = 0; t < count; ++t) {
        const double rho = std::ldexp(1 + U(gen), lo + (int)(gen() % (unsigned)(hi - lo)));
        double inv, sq;
        rho_factors_fixed(rho, inv, sq);
        int x;
        std::frexp(inv, &x);
        wi = std::fmax(wi, std::fabs((double)((Quad)inv - 1 / (Quad)rho)) / std::ldexp(1.0, x - 53));
        std::frexp(sq, &x);
        ws = std::fmax(ws, std::fabs((double)((Quad)sq - quad_sqrt((Quad)rho))) / std::ldexp(1.0, x - 53));
    }
    std::printf("%.6f %.6f\n", wi, ws);
}

// product_fixed against quadruple precision (half away from zero, of at least 62
// leading bits), and the products it may not call fitting.  Prints the number of
// wrong answers of each kind.
static void products(int count) {
    std::mt19937_64 gen(7);
    std::uniform_real_distribution<double> U(-1, 1);
    long wrong = 0, outside = 0, unfit = 0;
    for (int t = 0; t < count; ++t) {
        const double a = std::ldexp(U(gen), -(int)(gen() % 80)), b = std::ldexp(U(gen), (int)(gen() % 70));
        const double z = t % 50 ? a : 0.0;
        bool fits;
        const long long v = product_fixed(z, b, &fits);
        const Quad x = (Quad)z * (Quad)b;
        const double mag = std::fabs((double)x);
        if (mag < std::ldexp(1.0, 61) && !fits) ++outside;
        if (fits) {
            const Quad d = (Quad)v - x, half = (Quad)0.5 + (Quad)mag * (Quad)std::ldexp(1.0, -62);
            if (d > half || d < -half) ++wrong;
        }
    }
    const double inf = HUGE_VAL, nan = std::nan(""), tiny = 4.9e-324, big = std::ldexp(1.0, 31);
    for (double s : {1.0, -1.0})
        for (double b : {inf, nan, -inf})
            for (double a : {0.0, -0.0, tiny, 2.2e-308, 1e-300, 0.5, 1.0, big, inf, nan}) {
                bool f1, f2;
                product_fixed(s * a, b, &f1);
                product_fixed(b, s * a, &f2);
                unfit += f1 + f2;
            }
    bool fits;
    product_fixed(big, big, &fits);
    unfit += fits;
    std::printf("%ld %ld %ld\n", wrong, outside, unfit);
}

int main(int argc, char **argv) {
    if (argc > 1 && argv[1][0] == 'p') {
        products(2000000);
        return 0;
    }
    if (argc > 1 && argv[1][0] == 'f') {
        factors(-65, 64, 2000000);
        return 0;
    }
    const int nodes = argc > 1 ? std::atoi(argv[1]) : 4000;
    const double rho0 = argc > 2 ? std::atof(argv[2]) : 1.0;
    for (double rel : {0.9, 0.7, 0.5, 0.4, 0.33, 0.32, 0.3, 0.2, 0.12, 0.04, 0.001}) {
        run<false>(rel, rho0, nodes, 1);
        run<true>(rel, rho0, nodes, 2);
    }
    return 0;
}
