// The FP64 quotient of the interpolation (csrc/particle_step.cuh) and 1/rho, sqrt(rho)
// of the integer collision (csrc/lb_fixed.cuh) on the device, against the IEEE
// operations of the host and against quadruple precision: of each, the worst
// distance from the IEEE result in units of the last place and the worst error in
// those units; then the worst error of the reciprocal's approximation (log2).
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "lb_fixed.cuh"
#include "lbmd_ctx.h"
#include "particle_core.cuh"
#include "particle_step.cuh"

#ifdef __aarch64__
typedef long double Quad;
#else
typedef __float128 Quad;
#endif

__global__ void evaluate(const double *a, const double *b, double *q, double *h, double *inv, double *sq, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    q[i] = lbmd::quotient(a[i], b[i]);
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b[i]));
    h[i] = fma(-b[i], y, 1.0);
    lbmd::rho_factors_fixed(b[i], inv[i], sq[i]);
}

static double distance(double x, double y) {
    int64_t p, q;
    std::memcpy(&p, &x, 8);
    std::memcpy(&q, &y, 8);
    return std::fabs((double)(p - q));
}

static double unit(double x) {  // of the last place
    int e;
    std::frexp(x, &e);
    return std::ldexp(1.0, e - 53);
}

int main() {
    const int n = 1 << 20;
    std::vector<double> a(n), b(n), q(n), h(n), inv(n), sq(n);
    std::mt19937_64 gen(11);
    std::uniform_real_distribution<double> U(0, 1);
    for (int i = 0; i < n; ++i) {
        // densities of any rho0 in 2^-60 .. 2^60, thin and thick nodes among them;
        // weights from 0 and products of small offsets to 1
        b[i] = std::ldexp(1 + U(gen), -66 + (int)(gen() % 131));
        a[i] = i % 16 == 0 ? (double)(gen() % 2) : i % 16 == 1 ? std::ldexp(1 + U(gen), -(int)(gen() % 160)) : U(gen) * U(gen) * U(gen);
        if (i % 64 == 5) b[i] = std::ldexp(1.0, -60 + (int)(gen() % 121));  // a power of two, and next to it
        if (i % 64 == 6) b[i] = std::nextafter(std::ldexp(1.0, -60 + (int)(gen() % 121)), i & 64 ? 0.0 : 1e300);
    }
    double *d[6];
    for (auto &p : d)
        if (cudaMalloc(&p, n * sizeof(double)) != cudaSuccess) return 1;
    cudaMemcpy(d[0], a.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    cudaMemcpy(d[1], b.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    evaluate<<<n / 256, 256>>>(d[0], d[1], d[2], d[3], d[4], d[5], n);
    std::vector<double> *out[4] = {&q, &h, &inv, &sq};
    for (int k = 0; k < 4; ++k)
        if (cudaMemcpy(out[k]->data(), d[2 + k], n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    double w[3] = {0, 0, 0}, err[3] = {0, 0, 0}, hw = 0;
    for (int i = 0; i < n; ++i) {
        const double got[3] = {q[i], inv[i], sq[i]}, ieee[3] = {a[i] / b[i], 1.0 / b[i], std::sqrt(b[i])};
        const Quad B = b[i];
        Quad root = ieee[2];
        for (int k = 0; k < 2; ++k) root = (root + B / root) / 2;
        const Quad exact[3] = {(Quad)a[i] / B, 1 / B, root};
        for (int k = 0; k < 3; ++k) {
            w[k] = std::fmax(w[k], distance(got[k], ieee[k]));
            if (got[k] != 0) err[k] = std::fmax(err[k], std::fabs((double)((Quad)got[k] - exact[k])) / unit((double)exact[k]));
        }
        hw = std::fmax(hw, std::fabs(h[i]));
    }
    std::printf("%g %g %g %.6f %.6f %.6f %.2f\n", w[0], w[1], w[2], err[0], err[1], err[2], std::log2(hw));
    return 0;
}
