// lb_core.cuh -- the MRT collision with thermal noise and forcing at one
// node (Sec. 2 collision operator, Sec. 3 forcing term), shared by the
// single-box LB kernel (lb.cu), the batched replicas (batch.cu) and the adjoint's
// forward pass (adjoint.cu), which run one instruction sequence -- but for the
// single box in FP64, whose nodes mostly take the integer form of lb_fixed.cuh
// (the same collision, other roundings).
#pragma once

#include "lbmd_device.cuh"

namespace lbmd {

// Reciprocal norms 1/b_k, exact binary fractions.
__host__ __device__ constexpr double INV_BNORM(int k) {
    constexpr double t[Q] = {1.0, 3.0, 3.0, 3.0, 1.5, 0.75, 2.25, 9.0, 9.0, 9.0,
                             1.5, 1.5, 1.5, 4.5, 4.5, 4.5, 0.5, 0.75, 2.25};
    return t[k];
}
// 1/b_k and the norms b_k of lbmd_device.cuh (which the host's noise
// amplitudes use) are one table: checked at compile time.
constexpr bool inv_bnorm_matches() {
    for (int k = 0; k < Q; ++k)
        if (BNORM(k) * INV_BNORM(k) != 1.0) return false;
    return true;
}
static_assert(inv_bnorm_matches(), "INV_BNORM(k) must be 1 / BNORM(k)");

// The D3Q19 order pairs every moving velocity with its opposite:
// c_{2p+2} = -c_{2p+1}, p = 0..8 (x, y, z, then the diagonals of the xy, xz and
// yz planes, two each).  Even modes (0, 4-9, 16-18) see only the pair sums s_p,
// odd modes (1-3, 10-15) only the differences d_p; the back-transform likewise
// returns an even part E and an odd part O with f_{2p+1} = E + O and f_{2p+2} =
// E - O.  Within each, the three axes and the three planes share their sums.
template <typename T>
struct PairSums {
    T s[9], d[9];
    __device__ __forceinline__ explicit PairSums(const T f[Q]) {
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            s[p] = f[2 * p + 1] + f[2 * p + 2];
            d[p] = f[2 * p + 1] - f[2 * p + 2];
        }
    }
};

// 1/rho and sqrt(rho): IEEE in FP64; in FP32 both from one reciprocal square
// root (at most a few ulp, far below the FP32 path's tolerance)
__device__ __forceinline__ void rho_factors(double rho, double &inv, double &sq) {
    inv = 1.0 / rho;
    sq = sqrt(rho);
}
__device__ __forceinline__ void rho_factors(float rho, float &inv, float &sq) {
    const float r = rsqrtf(rho);
    inv = r * r;
    sq = rho * r;
}

// (h - 32767.5) for a 16-bit h, exactly: FP32 builds 2^23 + h from its bit
// pattern (no int-to-float conversion), removes 2^23 and then 32767.5 (both
// subtractions exact); FP64 converts.
__device__ __forceinline__ float centred16(uint32_t h, float) {
    return (__int_as_float((int)(0x4B000000u | h)) - 8388608.0f) - 32767.5f;
}
__device__ __forceinline__ double centred16(uint32_t h, double) { return (double)h - 32767.5; }

// Variant C (Sec. 4): a momentum transfer F enters the populations f (density
// rho, momentum j) through the forcing part of the collision alone: mass
// unchanged, momentum + F, stress modes + (1 + gamma) times the symmetric
// products of u = (j + F/2)/rho and F (as in collide()), ghost modes unchanged.
//
// The paper does this after every MD step, with that step's transfer.  The
// density stays and the momentum grows by each transfer, so with j_s the
// momentum before step s, j_{s+1} = j_s + F_s, the products telescope,
//     u_s F_s + F_s u_s = (j_{s+1} j_{s+1} - j_s j_s) / rho,
// and the m updates of a cycle are one update by the cycle's sum: the same
// populations, up to rounding (fewer of them), and the node velocities the
// MD steps see, (j + sum of the transfers) / rho, are those of variant B.  So
// variant C keeps its transfers in variant B's records and applies this
// once, inside the LB step, which has the populations in registers; a sweep
// over the populations per MD step cost 24 us per MD step at 96 x 80 x 112
// nodes (5.1e4 particles, FP32) and 0.78 ms at 256^3 (10^6 particles).
template <typename T>
__device__ __forceinline__ void apply_transfer(T f[Q], T rho, T jx, T jy, T jz, T Fx, T Fy, T Fz, T gamma_bulk,
                                               T gamma_shear) {
    const T ir = T(1) / rho;
    const T ux = (jx + T(0.5) * Fx) * ir, uy = (jy + T(0.5) * Fy) * ir, uz = (jz + T(0.5) * Fz) * ir;
    const T uF = ux * Fx + uy * Fy + uz * Fz;
    const T fb = T(1) + gamma_bulk, fs = T(1) + gamma_shear;
    const T dm[10] = {T(0), Fx, Fy, Fz, fb * uF, fs * (T(3) * ux * Fx - uF), fs * (uy * Fy - uz * Fz),
                      fs * T(0.5) * (ux * Fy + uy * Fx), fs * T(0.5) * (ux * Fz + uz * Fx),
                      fs * T(0.5) * (uy * Fz + uz * Fy)};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        T acc = T(0);
#pragma unroll
        for (int k = 1; k <= 9; ++k) {
            const int e = EMODE(k, i);
            if (e != 0) acc += T(e) * dm[k] * T(INV_BNORM(k));
        }
        f[i] += T(WEIGHT(i)) * acc;
    }
}

// (2h + 1) - 65536 for a 16-bit h, the low (high = 0) or the high half of a
// word, exactly: twice h - 32767.5.  FP32 builds 2^23 + 2h + 1 from its bit
// pattern (no int-to-float conversion) and subtracts once; FP64 goes through
// its fields.
__device__ __forceinline__ float centred16x2(uint32_t word, int high, float) {
    const uint32_t t = high ? word >> 15 : word << 1;
    return __uint_as_float((t & 0x1fffeu) | 0x4B000001u) - 8454144.0f;
}
__device__ __forceinline__ double centred16x2(uint32_t word, int high, double) {
    const uint32_t h = high ? word >> 16 : word & 0xffffu;
    return from_fixed((long long)(2u * h) - 65535ll, 0);
}

// MRT collision with forcing and noise at one node; f holds f* on entry and
// f' on exit -- or, for a deviation storage form, f* - b and f' - b with b the
// stored rest values (see PopStore): the collision is linear in the moments,
// and the mass mode takes rho_m (the density, or its part sum_i (f*_i - b_i)),
// while u, the equilibria and the noise amplitudes take the density rho.  With
// sum_i w_i = 1 and sum_i w_i e_k(c_i) = 0 for k > 0 the deviations then keep
// their sum, so the mass is conserved up to the rounding of small numbers.
//
// RELAX_FULL: gamma_bulk = gamma_ghost = 0 (the default reading), so the
// bulk and ghost modes relax fully, m'_k = m^eq_k exactly, and their moments
// m_k are not needed.
// A: any struct with the members gamma_bulk, gamma_shear, gamma_ghost,
// amp16[Q] and noisy (the single-box, batched and adjoint kernels), and for
// GAUSS (normal variates) ampg[Q]; the Philox key (key0, key1) and counters
// (node, step) come as arguments.
//
// The kernels that call this issue instructions about as fast as they move
// bytes, so the operations are counted: ~250 besides the noise bits, against
// ~430 when every mode and every population was summed on its own.  The
// stress terms (1 - gamma) rho u u + (1 + gamma) (u F + F u)/2 are u q + q u with
// q = (1 - gamma) rho u/2 + (1 + gamma) F/2; the 1/b_k and weights are constants of the
// back-transform.  The rest weight is taken as 1 - 24/36 of what the moving
// populations got, so that the weights add up to one whatever their rounding.
// Explicit multiply-adds: every kernel rounds alike.
template <typename T, bool RELAX_FULL, typename A, bool GAUSS = false>
__device__ __forceinline__ void collide(T f[Q], T rho, T rho_m, T jx, T jy, T jz, T Fx, T Fy, T Fz, const A &a,
                                        uint32_t key0, uint32_t key1, uint32_t node, uint32_t step) {
    T inv_rho, sr;
    rho_factors(rho, inv_rho, sr);
    const T ux = fma(T(0.5), Fx, jx) * inv_rho;
    const T uy = fma(T(0.5), Fy, jy) * inv_rho;
    const T uz = fma(T(0.5), Fz, jz) * inv_rho;
    const T cu = (T(0.5) - T(0.5) * a.gamma_shear) * rho, cf = T(0.5) + T(0.5) * a.gamma_shear;
    const T qx = fma(cu, ux, cf * Fx), qy = fma(cu, uy, cf * Fy), qz = fma(cu, uz, cf * Fz);
    const T bu = RELAX_FULL ? rho : rho - a.gamma_bulk * rho, bf = RELAX_FULL ? T(1) : T(1) + a.gamma_bulk;
    const T bx = fma(bu, ux, RELAX_FULL ? Fx : bf * Fx), by = fma(bu, uy, RELAX_FULL ? Fy : bf * Fy),
            bz = fma(bu, uz, RELAX_FULL ? Fz : bf * Fz);

    // post-collision modes 4..18: equilibrium and forcing, what is left of the
    // moments m_k = sum_i e_k(c_i) f_i, noise
    T m[Q];
    m[4] = fma(uz, bz, fma(uy, by, ux * bx));
    {
        const T txx = T(2) * (ux * qx), tyy = T(2) * (uy * qy), tzz = T(2) * (uz * qz);
        m[5] = fma(T(2), txx, -(tyy + tzz));
        m[6] = tyy - tzz;
        m[7] = fma(ux, qy, uy * qx);
        m[8] = fma(ux, qz, uz * qx);
        m[9] = fma(uy, qz, uz * qy);
    }
    {
        const PairSums<T> v(f);
        const T *s = v.s, *d = v.d;
        const T sxy = s[3] + s[4], sxz = s[5] + s[6], syz = s[7] + s[8];
        const T a5 = fma(T(2), s[0], -(s[1] + s[2])), g5 = fma(T(-2), syz, sxy + sxz);
        const T a6 = s[1] - s[2], g6 = sxy - sxz;
        const T gs = a.gamma_shear;
        m[5] = fma(gs, a5 + g5, m[5]);
        m[6] = fma(gs, a6 + g6, m[6]);
        m[7] = fma(gs, s[3] - s[4], m[7]);
        m[8] = fma(gs, s[5] - s[6], m[8]);
        m[9] = fma(gs, s[7] - s[8], m[9]);
        if constexpr (RELAX_FULL) {
#pragma unroll
            for (int k = 10; k < Q; ++k) m[k] = T(0);
        } else {
            const T gg = a.gamma_ghost, A3 = (s[0] + s[1]) + s[2], G = (sxy + sxz) + syz;
            m[4] = fma(a.gamma_bulk, G - f[0], m[4]);
            const T xy_x = d[3] + d[4], xy_y = d[3] - d[4], xz_x = d[5] + d[6], xz_z = d[5] - d[6],
                    yz_y = d[7] + d[8], yz_z = d[7] - d[8];
            m[10] = gg * fma(T(-2), d[0], xy_x + xz_x);
            m[11] = gg * fma(T(-2), d[1], xy_y + yz_y);
            m[12] = gg * fma(T(-2), d[2], xz_z + yz_z);
            m[13] = gg * (xy_x - xz_x);
            m[14] = gg * (yz_y - xy_y);
            m[15] = gg * (xz_z - yz_z);
            m[16] = gg * (fma(T(-2), A3, f[0]) + G);
            m[17] = gg * (g5 - a5);
            m[18] = gg * (g6 - a6);
        }
    }
    if constexpr (GAUSS) {
        if (a.noisy) {
            // 15 normal variates from four Philox calls, a Box-Muller pair
            // per two words, in mode order k = 4..18
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q) {
                const U4 r = philox4x32_10(U4{node, step, 0u, q}, key0, key1);
                T g[4];
                box_muller(r.x, r.y, g[0], g[1]);
                box_muller(r.z, r.w, g[2], g[3]);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int k = 4 + 4 * (int)q + t;
                    if (k < Q) m[k] = fma(a.ampg[k] * sr, g[t], m[k]);
                }
            }
        }
    } else if (a.noisy) {
        // 15 variates from two Philox calls: two 16-bit halves per 32-bit
        // word, low half first, in mode order k = 4..18.  The variate
        // sqrt(12) ((h + 1/2) 2^-16 - 1/2) is (h - 32767.5) times
        // sqrt(12) 2^-16, folded into amp16[k] = amp[k] sqrt(12) 2^-16, the
        // same for the modes of a class (7-9, 10-12, 13-15).
        const T half = T(0.5) * sr;
        T amp[Q];
#pragma unroll
        for (int k = 4; k < Q; ++k) {
            const bool same = k == 8 || k == 9 || k == 11 || k == 12 || k == 14 || k == 15;
            amp[k] = same ? amp[k - 1] : a.amp16[k] * half;
        }
#pragma unroll
        for (uint32_t q = 0; q < 2; ++q) {
            const U4 r = philox4x32_10(U4{node, step, 0u, q}, key0, key1);
            const uint32_t bits[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int k = 4 + 8 * (int)q + t;
                if (k < Q) m[k] = fma(amp[k], centred16x2(bits[t >> 1], t & 1, T(0)), m[k]);
            }
        }
    }
    m[1] = jx + Fx;
    m[2] = jy + Fy;
    m[3] = jz + Fz;
    // back-transform f_i = w_i sum_k e_k(c_i) m_k / b_k
    const T r36 = rho_m * T(1.0 / 36.0), r18 = r36 + r36, r0 = fma(T(-24), r36, rho_m);
    f[0] = fma(m[16], T(1.0 / 6.0), fma(m[4], T(-0.5), r0));
    {
        const T base = fma(m[16], T(-1.0 / 18.0), r18), e5 = m[5] - m[17], e6 = m[6] - m[18];
        const T side = fma(e5, T(-0.75 / 18.0), base);
        const T E[3] = {fma(e5, T(1.5 / 18.0), base), fma(e6, T(2.25 / 18.0), side), fma(e6, T(-2.25 / 18.0), side)};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T o = m[1 + c] - m[10 + c];
            f[2 * c + 1] = fma(o, T(3.0 / 18.0), E[c]);
            f[2 * c + 2] = fma(o, T(-3.0 / 18.0), E[c]);
        }
    }
    {
        const T base = fma(m[16], T(0.5 / 36.0), fma(m[4], T(1.5 / 36.0), r36)), e5 = m[5] + m[17], e6 = m[6] + m[18];
        const T side = fma(e5, T(0.75 / 36.0), base);
        const T E[3] = {fma(e6, T(2.25 / 36.0), side), fma(e6, T(-2.25 / 36.0), side), fma(e5, T(-1.5 / 36.0), base)};
        T X[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) X[c] = fma(m[10 + c], T(1.5 / 36.0), m[1 + c] * T(3.0 / 36.0));
        const T k = T(4.5 / 36.0);
        const T first[3] = {fma(m[13], k, X[0]), fma(m[13], -k, X[0]), fma(m[14], k, X[1])};
        const T second[3] = {fma(m[14], -k, X[1]), fma(m[15], k, X[2]), fma(m[15], -k, X[2])};
#pragma unroll
        for (int p = 0; p < 3; ++p) {  // xy, xz, yz
            const T ep = fma(m[7 + p], T(9.0 / 36.0), E[p]), em = fma(m[7 + p], T(-9.0 / 36.0), E[p]);
            const T op = first[p] + second[p], om = first[p] - second[p];
            f[7 + 4 * p] = ep + op;
            f[8 + 4 * p] = ep - op;
            f[9 + 4 * p] = em + om;
            f[10 + 4 * p] = em - om;
        }
    }
}

}  // namespace lbmd
