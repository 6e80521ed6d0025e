// lb_fixed.cuh -- the collision of lb_core.cuh for FP64 storage with its linear
// parts in 64-bit integers.
//
// Why: this GPU issues 2 FP64 operations per SM and clock against 64 or more
// 32-bit integer ones, and the moments, the relaxation and the back-transform
// are sums with small integer coefficients -- about 400 of the ~470 FP64
// operations of a node.  A population becomes an integer in units of
// 2^(e - 59) (e = ceil(log2 rho0)): exact for values of at least 2^(e - 7),
// rounded once at 2^(e - 60) below; the sums are then exact, where FP64 sums
// of values near rho0 round at 2^(e - 54).  What is left in FP64 is the
// non-linear part (1/rho, sqrt(rho), the products of u; ~45 operations).
//
// The new populations are f' = f + (1/144) sum_k c_ik D_k with the changes D_k of
// the moments (at rest they are 0, so they are small) and integers c_ik =
// 144 w_i e_k(c_i) / b_k: each change is divided by 9 with rounding, in units
// of 2^(e - 60), and the sum shifted by 4.  The changes sum to zero over the
// populations exactly; only the last shift rounds.
//
// Range: every |f_i| below 2^(e - 1), a density of at least (5/16) 2^e (rho0 is
// above 2^(e - 1)) and every |D_k| below 0.375 2^e, else the node is left to the
// FP64 form (fluids far from rho0, non-finite values).  The units are absolute, so
// in a thin node FP64 is the more accurate.  Against quadruple precision, in units
// of the node's density: rms error of the new populations 4.6e-18 at 0.9 2^e,
// 4.6e-18 at 0.5, 5.1e-18 at 0.3, 1.6e-17 at 2^-4 and 2.5e-17 at 0.04 (FP64 form
// 1.4e-17 to 1.7e-17 throughout); mean change of the mass in a step 1e-18 to
// 3e-18 down to 0.3, as in FP64, and 3e-17 to 9e-17 from 0.2 on, where populations
// are below 2^(e - 7) and rounded.
#pragma once

#include <cmath>
#include <cstring>

#include "lb_core.cuh"
#include "lbmd_device.cuh"

namespace lbmd {

constexpr int FIX_F = 59;  // populations: units of 2^(e - FIX_F)
constexpr int FIX_D = 60;  // changes of the moments: units of 2^(e - FIX_D)

// what the collision needs beside the FP64 constants
struct FixedArgs {
    int e;
    int usable;              // the noise amplitudes fit their fixed-point form
    long long amp[9];        // sqrt(12) times the amplitude of each class of modes, see fixed_constants
    long long g[3];          // body force, units of 2^(e - FIX_D)
};

// Classes of modes with one noise amplitude: 4, 5, 6, 7-9, 10-12, 13-15, 16, 17, 18.
__host__ __device__ constexpr int AMP_CLASS(int k) {
    return k <= 6 ? k - 4 : k <= 9 ? 3 : k <= 12 ? 4 : k <= 15 ? 5 : k - 10;
}

// amp[c]: a_k = sqrt(12) amp_k 2^(h - e) in units of 2^-62, h = e / 2 rounded
// up, so that a_k times sqrt(rho) 2^-h is the noise in units of 2^e.
inline FixedArgs fixed_constants(int e, const double noise_amp[Q], const double g[3]) {
    FixedArgs a;
    a.e = e;
    a.usable = 1;
    const int h = (e + (e > 0)) / 2;
    for (int k = 4; k < Q; ++k) {
        const double v = noise_amp[k] * 3.4641016151377544 * std::ldexp(1.0, h - e);
        if (!(v < 1.0)) a.usable = 0;
        a.amp[AMP_CLASS(k)] = a.usable ? (long long)std::llrint(std::ldexp(v, 62)) : 0;
    }
    for (int d = 0; d < 3; ++d) {
        const double v = std::ldexp(g[d], FIX_D - e);
        if (!(std::fabs(v) < std::ldexp(1.0, FIX_D - 2))) a.usable = 0;
        a.g[d] = a.usable ? (long long)std::llrint(v) : 0;
    }
    return a;
}

__host__ __device__ __forceinline__ long long mul_hi64(long long a, long long b) {
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (long long)(((__int128)a * b) >> 64);
#endif
}
// Whether all populations are below 2^(e - 1): one compare on the largest
// exponent field (NaN and infinity have the largest).
__host__ __device__ __forceinline__ bool in_fixed_range(const double f[Q], int e) {
    unsigned top = 0u;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const unsigned t = (unsigned)(bits_of(f[i]) >> 32) & 0x7fffffffu;
        top = t > top ? t : top;
    }
    return (top >> 20) < (unsigned)(1023 + e - 1);
}

struct FixedMoments {
    long long n[Q];  // populations, units of 2^(e - FIX_F)
    long long rho, j[3];
};
constexpr long long FIX_RHO_MIN = 5ll << (FIX_F - 4);  // the smallest density, see above

__host__ __device__ __forceinline__ void fixed_moments(const double f[Q], int e, FixedMoments &o) {
    long long d[9];
#pragma unroll
    for (int i = 0; i < Q; ++i) o.n[i] = to_fixed(f[i], FIX_F - e);
    o.rho = o.n[0];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        o.rho += o.n[2 * p + 1] + o.n[2 * p + 2];
        d[p] = o.n[2 * p + 1] - o.n[2 * p + 2];
    }
    o.j[0] = d[0] + (d[3] + d[4]) + (d[5] + d[6]);
    o.j[1] = d[1] + (d[3] - d[4]) + (d[7] + d[8]);
    o.j[2] = d[2] + (d[5] - d[6]) + (d[7] - d[8]);
}

// The moments of a node that the integers take; false for any other.
__host__ __device__ __forceinline__ bool fixed_moments_in_range(const double f[Q], int e, FixedMoments &o) {
    if (!in_fixed_range(f, e)) return false;
    fixed_moments(f, e, o);
    return o.rho >= FIX_RHO_MIN;
}

// momentum in the node record's units of 2^(e - 56)
__host__ __device__ __forceinline__ long long record_momentum(long long j) {
    return (j + (1ll << (FIX_F - 56 - 1))) >> (FIX_F - 56);
}

// Density, momentum and the momentum in the node records' fixed point of the
// populations f (as the arithmetic takes them), the same wherever a record or
// the transfer (record - this) is formed.  FP64 populations within range are
// summed as integers (lb_fixed.cuh).
template <typename T>
struct NodeSums {
    T rho, rho_m, jx, jy, jz;
    typename Prec<T>::fix ix, iy, iz;
};
template <bool DEV, typename T>
__device__ __forceinline__ NodeSums<T> node_sums(const T f[Q], T rho_base, T fs, int e) {
    using P = Prec<T>;
    NodeSums<T> s;
    if constexpr (sizeof(T) == 8) {
        FixedMoments o;
        if (fixed_moments_in_range(f, e, o)) {
            s.rho = s.rho_m = from_fixed(o.rho, FIX_F - e);
            s.jx = from_fixed(o.j[0], FIX_F - e);
            s.jy = from_fixed(o.j[1], FIX_F - e);
            s.jz = from_fixed(o.j[2], FIX_F - e);
            s.ix = record_momentum(o.j[0]);
            s.iy = record_momentum(o.j[1]);
            s.iz = record_momentum(o.j[2]);
            return s;
        }
    }
    pop_moments<DEV>(f, rho_base, s.rho, s.rho_m, s.jx, s.jy, s.jz);
    s.ix = P::to_fix(s.jx, fs);
    s.iy = P::to_fix(s.jy, fs);
    s.iz = P::to_fix(s.jz, fs);
    return s;
}

// 1/rho and sqrt(rho) in 12 FP64 operations, a third of the IEEE division and
// square root, for rho in the FP32 range.  With y the FP32 approximation of
// rho^-1/2 and rho y^2 = 1 - h, rho^-1/2 is y (1 - h)^-1/2 = y (1 + h/2 + 3 h^2/8 + ...):
// the binomial series, cut after h^2 (|h| below 2^-21: 2^-64 of it is left; the
// third-order member of Householder's iterations).  y^2 and rho y are then 1/rho and
// sqrt(rho) to the roundings of a few operations, and one Newton step each, on the
// residual that a fused multiply-add forms (P. W. Markstein, IBM J. Res. Dev. 34
// (1990) 111), takes those away: errors below 0.51 units of the last place.
// (Goldschmidt's coupled form, sqrt(rho) carried beside y through the series, holds
// one value longer: 12 bytes of spills and 1 % of a cycle at 128^3 nodes.)
__host__ __device__ __forceinline__ void rho_factors_fixed(double rho, double &inv, double &sq) {
#ifdef __CUDA_ARCH__
    double y = (double)rsqrtf((float)rho);
#else
    double y = (double)(1.0f / sqrtf((float)rho));
#endif
    const double t = rho * y;
    const double h = fma(-t, y, 1.0);
    y = fma(y * h, fma(0.375, h, 0.5), y);
    inv = y * y;
    inv = fma(inv, fma(-rho, inv, 1.0), inv);
    sq = rho * y;
    sq = fma(0.5 * y, fma(-sq, sq, rho), sq);
}

// One noise term: b (units of 2^(e - FIX_D)) times (2 h - 65535) 2^-17.
__host__ __device__ __forceinline__ long long fixed_noise(long long b, unsigned h) {
    const int n = (int)(2u * h) - 65535;
    const long long hi = (long long)(int)(b >> 32) * n;
    const long long lo = (long long)(int)((unsigned)b >> 1) * n;
    return (hi << 15) + (lo >> 16);
}

// The collision (lb_core.cuh: collide, with gamma_bulk = gamma_ghost = 0) of the
// node whose populations are in `o`, for the transfer J (record units, 2^(e - 56)) and the
// body force; with C (variant C) the transfer enters the populations first
// (apply_transfer).  f gets the new populations; false if a change is out of
// range (f untouched).  xi: the 15 noise numbers' source (bits for the uniform
// variates, normals otherwise).
template <bool C, bool GAUSS, typename Noise>
__host__ __device__ __forceinline__ bool collide_fixed(const FixedMoments &o, const long long J[3], double gamma_shear,
                                                       const double g[3], const FixedArgs &a, bool noisy,
                                                       Noise &&noise, double f[Q]) {
    const int e = a.e;
    const long long *n = o.n;
    // a density in [(5/16) 2^e, 9.5 2^e) -- 19 populations below 2^(e - 1) -- and a
    // transfer below 2^(e - 1): then everything below is finite
    bool ok = o.rho >= FIX_RHO_MIN;
#pragma unroll
    for (int c = 0; c < 3; ++c) ok = ok && (unsigned long long)(J[c] + (1ll << 55)) < (1ull << 56);
    if (!ok) return false;
    const double rho = from_fixed(o.rho, FIX_F - e);
    double inv, sr;
    rho_factors_fixed(rho, inv, sr);
    // D[1..3]: the whole force; F: the force the collision sees
    long long D[Q];
    double F[3], T[6];  // T: xx, yy, zz, xy, xz, yz of the new stress terms
    double P[3];
    const double fs = 1.0 + gamma_shear, fm = 1.0 - gamma_shear;
    double hxx = 0.0, hyy = 0.0, hzz = 0.0, hxy = 0.0, hxz = 0.0, hyz = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        D[1 + c] = J[c] * (1ll << (FIX_D - 56)) + a.g[c];
        const double jc = from_fixed(o.j[c], FIX_F - e), Jc = from_fixed(J[c], 56 - e);
        if (C) {
            F[c] = g[c];
            T[c] = jc;
            T[3 + c] = Jc;
            P[c] = fma(0.5, g[c], jc + Jc);
        } else {
            F[c] = Jc + g[c];
            P[c] = fma(0.5, F[c], jc);
        }
    }
    if (C) {
        // the transfer's own products, with u = (j + J/2)/rho
        const double vx = fma(0.5, T[3], T[0]) * inv, vy = fma(0.5, T[4], T[1]) * inv, vz = fma(0.5, T[5], T[2]) * inv;
        hxx = vx * T[3];
        hyy = vy * T[4];
        hzz = vz * T[5];
        hxy = 0.5 * fma(vx, T[4], vy * T[3]);
        hxz = 0.5 * fma(vx, T[5], vz * T[3]);
        hyz = 0.5 * fma(vy, T[5], vz * T[4]);
    }
    const double u[3] = {P[0] * inv, P[1] * inv, P[2] * inv};
    // bulk: m'_4 = rho u.u + u.F
    double bulk = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) bulk = fma(u[c], fma(rho, u[c], F[c]), bulk);
    // shear: (1 - gamma) rho u u + (1 + gamma) (u F + F u)/2 = u q + q u, q = (1 - gamma) rho u/2 + (1 + gamma) F/2
    const double cu = 0.5 * fm * rho, cf = 0.5 * fs;
    double q[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) q[c] = fma(cu, u[c], cf * F[c]);
    double txx = 2.0 * (u[0] * q[0]), tyy = 2.0 * (u[1] * q[1]), tzz = 2.0 * (u[2] * q[2]);
    double txy = fma(u[0], q[1], u[1] * q[0]), txz = fma(u[0], q[2], u[2] * q[0]), tyz = fma(u[1], q[2], u[2] * q[1]);
    if (C) {
        // the transfer's stress, then relaxed: (1 + gamma) h - (1 - gamma) (1 + gamma) h = gamma (1 + gamma) h
        const double gh = gamma_shear * fs;
        txx = fma(gh, hxx, txx);
        tyy = fma(gh, hyy, tyy);
        tzz = fma(gh, hzz, tzz);
        txy = fma(gh, hxy, txy);
        txz = fma(gh, hxz, txz);
        tyz = fma(gh, hyz, tyz);
    }
    const double t6 = tyy - tzz, t5 = fma(2.0, txx, -(tyy + tzz));
    // moments
    long long s[9], d[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) {
        s[p] = n[2 * p + 1] + n[2 * p + 2];
        d[p] = n[2 * p + 1] - n[2 * p + 2];
    }
    const long long sxy = s[3] + s[4], sxz = s[5] + s[6], syz = s[7] + s[8];
    const long long A = s[0] + s[1] + s[2], G = sxy + sxz + syz;
    const long long a5 = 2 * s[0] - s[1] - s[2], g5 = sxy + sxz - 2 * syz, a6 = s[1] - s[2], g6 = sxy - sxz;
    const long long xy_x = d[3] + d[4], xy_y = d[3] - d[4], xz_x = d[5] + d[6], xz_z = d[5] - d[6],
                    yz_y = d[7] + d[8], yz_z = d[7] - d[8];
    long long m[Q];
    m[4] = G - n[0];
    m[5] = a5 + g5;
    m[6] = a6 + g6;
    m[7] = s[3] - s[4];
    m[8] = s[5] - s[6];
    m[9] = s[7] - s[8];
    m[10] = xy_x + xz_x - 2 * d[0];
    m[11] = xy_y + yz_y - 2 * d[1];
    m[12] = xz_z + yz_z - 2 * d[2];
    m[13] = xy_x - xz_x;
    m[14] = yz_y - xy_y;
    m[15] = xz_z - yz_z;
    m[16] = n[0] - 2 * A + G;
    m[17] = g5 - a5;
    m[18] = g6 - a6;
    // changes: bulk and ghosts relax fully, shear by 1 - gamma
    const double t[6] = {bulk, t5, t6, txy, txz, tyz};
    double big = 0.0;
#pragma unroll
    for (int k = 4; k <= 9; ++k) {
        double v = t[k - 4];
        if (k > 4) v = fma(-fm, from_fixed(m[k], FIX_F - e), v);
        big = fmax(big, fabs(v));
        D[k] = to_fixed(v, FIX_D - e);
        if (k == 4) D[4] -= m[4] * (1 << (FIX_D - FIX_F));
    }
#pragma unroll
    for (int k = 10; k < Q; ++k) D[k] = -m[k] * (1 << (FIX_D - FIX_F));
    if (noisy) {
        if (GAUSS) {
#pragma unroll
            for (int k = 4; k < Q; ++k) {
                const double v = noise.normal(k) * sr;
                big = fmax(big, fabs(v));
                D[k] += to_fixed(v, FIX_D - e);
            }
        } else {
            const int h = (e + (e > 0)) / 2;
            const long long sf = to_fixed(sr, 62 - 2 - h);  // sqrt(rho) 2^-h below sqrt(9.5) < 4: units of 2^-60
            long long b[9];
#pragma unroll
            for (int c = 0; c < 9; ++c) b[c] = mul_hi64(sf, a.amp[c]) * 4;
#pragma unroll
            for (int k = 4; k < Q; ++k) D[k] += fixed_noise(b[AMP_CLASS(k)], noise.bits(k));
        }
    }
    // in range: |D| < 0.375 2^e, and what was converted below 2^(e - 1)
    const unsigned long long lim = 3ull << (FIX_D - 3);
    ok = big < double_of((unsigned long long)(1022 + e) << 52);
#pragma unroll
    for (int k = 1; k < Q; ++k) ok = ok && (unsigned long long)(D[k] + (long long)lim) < 2ull * lim;
    if (!ok) return false;
    // changes over 9, rounded
#pragma unroll
    for (int k = 1; k < Q; ++k) D[k] = mul_hi64(D[k] + 4, 0x1C71C71C71C71C72ll);
    const int up = FIX_D - FIX_F;
    auto out = [&](int i, long long S) { f[i] = from_fixed(n[i] * (1 << up) + ((S + 8) >> 4), FIX_D - e); };
    out(0, 24 * D[16] - 72 * D[4]);
    {
        const long long a1 = D[5] - D[17], b1 = D[6] - D[18], g16 = 8 * D[16];
        const long long E[3] = {12 * a1 - g16, 18 * b1 - 6 * a1 - g16, -18 * b1 - 6 * a1 - g16};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const long long O = 24 * (D[1 + c] - D[10 + c]);
            out(2 * c + 1, E[c] + O);
            out(2 * c + 2, E[c] - O);
        }
    }
    const long long a2 = 3 * (D[5] + D[17]), b2 = 9 * (D[6] + D[18]), c2 = 6 * D[4] + 2 * D[16];
    const long long x0 = 12 * D[1] + 6 * D[10], y0 = 12 * D[2] + 6 * D[11], z0 = 12 * D[3] + 6 * D[12];
    const long long xd = 18 * D[13], yd = 18 * D[14], zd = 18 * D[15];
    const long long base[3] = {c2 + a2 + b2, c2 + a2 - b2, c2 - 2 * a2};  // xy, xz, yz
    const long long first[3] = {x0 + xd, x0 - xd, y0 + yd}, second[3] = {y0 - yd, z0 + zd, z0 - zd};
#pragma unroll
    for (int q2 = 0; q2 < 3; ++q2) {
        const long long w = 36 * D[7 + q2];
        const int i = 7 + 4 * q2;
        const long long o1 = first[q2] + second[q2], o2 = first[q2] - second[q2];
        out(i, base[q2] + w + o1);
        out(i + 1, base[q2] + w - o1);
        out(i + 2, base[q2] - w + o2);
        out(i + 3, base[q2] - w - o2);
    }
    return true;
}

}  // namespace lbmd
