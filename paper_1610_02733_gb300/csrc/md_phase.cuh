// md_phase.cuh -- several MD steps of Sec. 3 in one launch, one thread per
// particle, with the particle kept in registers between the steps.
//
// frozen_phase_kernel (variant A, ideal particles): the node velocities are
// frozen between two LB updates, so no particle of the phase waits for
// another one.  The thread reads the 8 corner records when the particle
// enters a cell (once per phase for nearly all of them), runs its MD steps on
// them, sums the fixed-point transfers of the steps per corner in registers,
// and adds the sums to the nodes with atomics when the particle leaves the
// cell and at the end.  The sums are integers: the same bits as one
// transfer at a time.
//
// team_phase_kernel (variants B and C, and particles with conservative forces
// of any variant): the particles see one another's transfers (positions) of the
// MD step before, so the blocks, all resident at once (cooperative launch),
// meet at a grid barrier after every particle has read the nodes and after all
// transfers.  A team of lanes steps one particle.  Few ideal particles of variant A
// take the teams without the barriers.
#pragma once

#include <type_traits>

#include "lbmd_ctx.h"
#include "lbmd_device.cuh"
#include "particle_core.cuh"
#include "particle_step.cuh"
#include "phase_barrier.cuh"

namespace lbmd {

// The records of a cell's 8 corners as the interpolation takes them, and the
// transfers to them not yet handed over.
template <typename T>
struct CornerCache {
    using P = Prec<T>;
    T rho[8], jx[8], jy[8], jz[8];
    typename P::fix tx[8], ty[8], tz[8];

    __device__ __forceinline__ void load(const PArgs<T> &a, const CellXYZ &c) {
        typename P::node4 n[8];
        corner_records(a, c, n);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            rho[k] = P::rho_of(n[k]);
            jx[k] = P::from_fix(P::jx_of(n[k]), a.fis);
            jy[k] = P::from_fix(P::jy_of(n[k]), a.fis);
            jz[k] = P::from_fix(P::jz_of(n[k]), a.fis);
            tx[k] = ty[k] = tz[k] = 0;
        }
    }

    // the transfer -delta_k dt F to every corner
    __device__ __forceinline__ void add(const PArgs<T> &a, T fx, T fy, T fz, T Fx, T Fy, T Fz) {
        const T wx[2] = {T(1) - fx, fx}, wy[2] = {T(1) - fy, fy}, wz[2] = {T(1) - fz, fz};
        const T sx = Fx * a.neg_scale_dt, sy = Fy * a.neg_scale_dt, sz = Fz * a.neg_scale_dt;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const T d = wx[k & 1] * wy[(k >> 1) & 1] * wz[k >> 2];
            tx[k] += P::to_fix_neg(d, sx);
            ty[k] += P::to_fix_neg(d, sy);
            tz[k] += P::to_fix_neg(d, sz);
        }
    }

    __device__ __forceinline__ void hand_over(const PArgs<T> &a, const CellXYZ &c) {
        uint32_t rows[4];
        corner_rows(c, a.ny, a.nz, rows);
        const int x1 = c.x + 1 == a.nx ? 0 : c.x + 1;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int xn = (k & 1) ? x1 : c.x;
            const uint32_t row = rows[k >> 1];
            const int sl = active_slot(a.occw[(size_t)row * (uint32_t)a.occ_words + (xn >> 5)], xn);
            typename P::node4 *rec =
                sl >= 0 ? &a.cact_acc[sl] : &a.inactive_acc[(size_t)row * (uint32_t)a.nx + xn];
            P::add_transfer(rec, tx[k], ty[k], tz[k]);
        }
    }
};

// Registers: the cache and the sums take 56 (FP32) / 112 (FP64), so fewer
// threads are resident than in couple_kernel, but the phase reads memory once
// instead of at every step and its steps are arithmetic.
template <typename T, bool HALF>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 5 : 2) frozen_phase_kernel(PArgs<T> a, int count) {
    using P = Prec<T>;
    // the row gather's migrant lists are not used in this phase: both empty
    // for the next MD step that uses one
    if (blockIdx.x == 0 && threadIdx.x < 2) a.migrant_count[threadIdx.x] = 0;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.np) return;
    const typename P::real4 R = a.pos4[p];
    typename P::real4 V = a.vel4[p];
    T fx = R.x, fy = R.y, fz = R.z;
    CellXYZ c = cell_xyz(P::cell_of(R), a.fd_nx, a.fd_ny), held = c;
    T Fx = T(0), Fy = T(0), Fz = T(0);
    if (HALF) {
        const typename P::real4 F = a.fc4[p];
        Fx = F.x;
        Fy = F.y;
        Fz = F.z;
    }
    const uint32_t id = (uint32_t)a.pid[p], step0 = md_step_index(a);
    const T hm = a.half_dt * V.w;  // V.w = 1 / mass
    CornerCache<T> corner;
    bool fresh = true;
    for (int s = 0; s < count; ++s) {
        if (HALF) {
            V.x = fma(hm, Fx, V.x);
            V.y = fma(hm, Fy, V.y);
            V.z = fma(hm, Fz, V.z);
            advance(fx, c.x, a.dt, V.x, a.nx);
            advance(fy, c.y, a.dt, V.y, a.ny);
            advance(fz, c.z, a.dt, V.z, a.nz);
        }
        if (fresh || c.x != held.x || c.y != held.y || c.z != held.z) {
            if (!fresh) corner.hand_over(a, held);
            corner.load(a, c);
            held = c;
            fresh = false;
        }
        T ux, uy, uz;
        interp_u_cached(fx, fy, fz, corner.rho, corner.jx, corner.jy, corner.jz, ux, uy, uz);
        coupling_force_id(a, id, step0 + (uint32_t)s, V, ux, uy, uz, Fx, Fy, Fz);
        corner.add(a, fx, fy, fz, Fx, Fy, Fz);
        if (!HALF) {
            V.x = fma(hm, Fx, V.x);
            V.y = fma(hm, Fy, V.y);
            V.z = fma(hm, Fz, V.z);
            advance(fx, c.x, a.dt, V.x, a.nx);
            advance(fy, c.y, a.dt, V.y, a.ny);
            advance(fz, c.z, a.dt, V.z, a.nz);
        }
        V.x = fma(hm, Fx, V.x);
        V.y = fma(hm, Fy, V.y);
        V.z = fma(hm, Fz, V.z);
    }
    corner.hand_over(a, held);
    a.pos4[p] = P::make_pos(fx, fy, fz, c.x + (int64_t)a.nx * (c.y + (int64_t)a.ny * c.z));
    a.vel4[p] = V;
    a.fc4[p] = P::make4(Fx, Fy, Fz, T(0));
}

template <typename T>
__device__ __forceinline__ T quiet_nan();
template <>
__device__ __forceinline__ float quiet_nan<float>() { return __int_as_float(0x7fc00000); }
template <>
__device__ __forceinline__ double quiet_nan<double>() { return __longlong_as_double(0x7ff8000000000000LL); }

// Separation of a bond partner (partner minus particle, minimum image): the
// rounded components and what the rounding left out.
template <typename T>
struct Separation {
    T x, y, z, lx, ly, lz;
};

// a - b and a + b with their rounding errors (Knuth's two-sum)
template <typename T>
__device__ __forceinline__ T two_sum(T a, T b, T &err) {
    const T s = a + b, t = s - a;
    err = (a - (s - t)) + (b - t);
    return s;
}

// One component: d whole cells plus the difference of the offsets.  The image is
// taken off the whole cells: off the rounded sum it would cost a bond across
// the periodic boundary the last bits of the box length.
template <typename T>
__device__ __forceinline__ T separation_component(int d, T there, T here, int n, T &lo) {
    T l1, l2;
    const T f = two_sum(there, -here, l1);
    d -= n * (int)rint((T(d) + f) / T(n));
    const T x = two_sum(T(d), f, l2);
    lo = l1 + l2;
    return x;
}

// Through the stored cell indices and offsets, for the partner in slot q of a
// particle at (R, c).  L2: the partner's position was written during the launch.
template <bool L2 = false, typename T>
__device__ __forceinline__ Separation<T> bond_separation(const PArgs<T> &a, const typename Prec<T>::real4 &R,
                                                         const CellXYZ &c, int64_t q) {
    using P = Prec<T>;
    const typename P::real4 S = L2 ? load_l2(&a.pos4[q]) : a.pos4[q];
    const CellXYZ d = cell_xyz(P::cell_of(S), a.fd_nx, a.fd_ny);
    Separation<T> v;
    v.x = separation_component(d.x - c.x, S.x, R.x, a.nx, v.lx);
    v.y = separation_component(d.y - c.y, S.y, R.y, a.ny, v.ly);
    v.z = separation_component(d.z - c.z, S.z, R.z, a.nz, v.lz);
    return v;
}

// Bond force g d on a particle from a partner at separation d, |d| = r, with
//   harmonic U = (k/2)(r - r0)^2               g = k (r - r0) / r   (0 at r = 0)
//   FENE     U = -(k/2) R0^2 ln(1 - (r/R0)^2)  g = k / (1 - (r/R0)^2), R0 = r0
// (Kremer-Grest springs, Sec. 4); a FENE bond at r >= R0 gives NaN.  The
// harmonic one, stiff and near r0, takes r - r0 = (r^2 - r0^2) / (r + r0) with the
// squares' and sums' rounding errors carried along -- for r0 > 0, where r + r0
// does not cancel, and while r0^2 stays in FP32's range; elsewhere r - r0 as it
// stands, which does not cancel there (r is at most a few thousand).  That choice
// is made by bond_form, outside the MD steps of a phase (inside them it cost 0.6 %
// of a cycle of 4,096 bonded particles).
constexpr uint8_t BOND_HARMONIC_PLAIN = 2;
template <typename T>
__device__ __forceinline__ uint8_t bond_form(uint8_t kind, T r0) {
    return kind == LBMD_BOND_HARMONIC && !(r0 > T(0x1p-40) && r0 < T(0x1p40)) ? BOND_HARMONIC_PLAIN : kind;
}
template <typename T>
__device__ __forceinline__ T bond_gain(uint8_t form, T k, T r0, const Separation<T> &d) {
    const T px = d.x * d.x, py = d.y * d.y, pz = d.z * d.z;
    if (form != LBMD_BOND_HARMONIC) {
        const T r2 = fma(d.z, d.z, fma(d.y, d.y, px));
        if (form == BOND_HARMONIC_PLAIN) {
            const T r = sqrt(r2);
            return r > T(0) ? k * (r - r0) / r : T(0);
        }
        const T x = r2 / (r0 * r0);
        return x < T(1) ? k / (T(1) - x) : quiet_nan<T>();
    }
    const T p0 = r0 * r0;
    T e1, e2, e3;
    const T s = two_sum(two_sum(two_sum(px, -p0, e1), py, e2), pz, e3);
    const T small = fma(T(2) * d.x, d.lx, fma(T(2) * d.y, d.ly, (T(2) * d.z) * d.lz));
    const T squares = (fma(d.x, d.x, -px) + fma(d.y, d.y, -py)) + (fma(d.z, d.z, -pz) - fma(r0, r0, -p0));
    const T e = s + ((((e1 + e2) + e3) + squares) + small);  // r^2 - r0^2
    const T r = sqrt(fma(d.z, d.z, fma(d.y, d.y, px)));
    return r > T(0) ? k * e / (r * (r + r0)) : T(0);
}

// Bond forces on particle `id` at (R, c), summed over its partners in a fixed
// order.
template <typename T>
__device__ __forceinline__ void bond_forces(const PArgs<T> &a, int64_t id, const typename Prec<T>::real4 &R,
                                            const CellXYZ &c, T &Fx, T &Fy, T &Fz) {
    Fx = Fy = Fz = T(0);
    const int nbond = a.bond_count[id];
    for (int b = 0; b < nbond; ++b) {
        const int64_t e = id * LBMD_MAX_BONDS_PER_PARTICLE + b;
        const Separation<T> d = bond_separation(a, R, c, a.slot_of[a.bond_partner[e]]);
        const T r0 = (T)a.bond_r0[e], g = bond_gain(bond_form(a.bond_kind[e], r0), (T)a.bond_k[e], r0, d);
        Fx = fma(g, d.x, Fx);
        Fy = fma(g, d.y, Fy);
        Fz = fma(g, d.z, Fz);
    }
}

// Lennard-Jones force on the particle at (R, c) from the one at S, if within the
// cut-off; explicit FMAs, so that every path rounds alike.
template <typename T>
__device__ __forceinline__ void pair_term(const PArgs<T> &a, const typename Prec<T>::real4 &R, const CellXYZ &c,
                                          const CellXYZ &d, T sx, T sy, T sz, T &Fx, T &Fy, T &Fz) {
    const T dx = T(nearest_image(d.x - c.x, a.nx)) + (sx - R.x);
    const T dy = T(nearest_image(d.y - c.y, a.ny)) + (sy - R.y);
    const T dz = T(nearest_image(d.z - c.z, a.nz)) + (sz - R.z);
    const T r2 = fma(dz, dz, fma(dy, dy, dx * dx));
    if (r2 < a.lj_rc2) {
        const T s = a.lj_sig2 / r2;
        const T t = s * s * s;
        const T g = -a.lj_eps24 * fma(T(2) * t, t, -t) / r2;
        Fx = fma(g, dx, Fx);
        Fy = fma(g, dy, Fy);
        Fz = fma(g, dz, Fz);
    }
}
template <typename T>
__device__ __forceinline__ void pair_term(const PArgs<T> &a, const typename Prec<T>::real4 &R, const CellXYZ &c,
                                          const typename Prec<T>::real4 &S, T &Fx, T &Fy, T &Fz) {
    pair_term(a, R, c, cell_xyz(Prec<T>::cell_of(S), a.fd_nx, a.fd_ny), S.x, S.y, S.z, Fx, Fy, Fz);
}

// The lane's share of the listed pairs of the particle with id i (ids = lane mod
// 32, ascending), four positions in flight.
template <bool L2 = false, typename T>
__device__ __forceinline__ void listed_pairs(const PArgs<T> &a, int64_t i, int lane, const typename Prec<T>::real4 &R,
                                             const CellXYZ &c, T &Fx, T &Fy, T &Fz) {
    const int32_t *L = a.nb_list + i * LBMD_NB_MAX;
    const int end = a.nb_end[i * 32 + lane];
    const int prev = __shfl_up_sync(0xffffffffu, end, 1);
    for (int e = lane ? prev : 0; e < end; e += 4) {
        typename Prec<T>::real4 S[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (e + k < end) S[k] = L2 ? load_l2(&a.pos4[L[e + k]]) : a.pos4[L[e + k]];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (e + k < end) pair_term(a, R, c, S[k], Fx, Fy, Fz);
    }
}

// Why teams: with few particles a step is a chain of dependent instructions
// (about 1100 per particle in FP32, at 4-5 cycles each for a lone warp) and
// memory round trips, not throughput.  Lane k (mod 8) of a team takes corner k: its
// record, quotient and transfer, and bond k; the sums over the corners run in
// the order of the other kernels (values broadcast by shuffles), so all paths
// give the same bits.  Teams of 8 lanes, of 32 with Lennard-Jones forces (the
// pairs go over all lanes).  Per cycle against the separate launches: 64^3 nodes,
// 4,096 bonded particles, m = 10, 131 -> 76 us; 2,560 with Lennard-Jones forces 190
// -> 138; one thread per particle instead of a team took 141 us in the first.
constexpr int PHASE_THREADS = 256;  // threads per block, or twice that to keep the blocks within one per SM
constexpr int PHASE_CLUSTER = 16;   // largest cluster

// Positions of the other particles staged for the all-pairs form.
template <typename T>
struct PairTile {
    static constexpr int N = sizeof(T) == 4 ? 1024 : 512;  // 40 / 26 KB of shared memory
    T f[3][N];
    int c[3][N];
    float4 abs[N];  // FP32 absolute positions, for the filter
};
struct NoTile {};

// All pairs of one particle per warp (id i at (R, c)): the block stages the
// other particles in tiles of ids (cell coordinates and offsets, decoded once
// per block instead of once per pair); lane l takes the ids l, l + 32, ... of
// the tile.  Block-uniform (barriers inside).
template <bool L2, typename T>
__device__ __forceinline__ void all_pairs(const PArgs<T> &a, PairTile<T> &t, int64_t i, bool live, int lane,
                                          const typename Prec<T>::real4 &R, const CellXYZ &c, T &Fx, T &Fy, T &Fz) {
    using P = Prec<T>;
    constexpr int TILE = PairTile<T>::N;
    const float xi = (float)(T(c.x) + R.x), yi = (float)(T(c.y) + R.y), zi = (float)(T(c.z) + R.z);
    const float fnx = (float)a.nx, fny = (float)a.ny, fnz = (float)a.nz;
    const float inx = 1.0f / fnx, iny = 1.0f / fny, inz = 1.0f / fnz;
    for (int64_t j0 = 0; j0 < a.np; j0 += TILE) {
        const int cnt = a.np - j0 < TILE ? (int)(a.np - j0) : TILE;
        __syncthreads();  // the previous tile is consumed
        for (int k = threadIdx.x; k < cnt; k += blockDim.x) {
            const typename P::real4 *q = &a.pos4[a.slot_of[j0 + k]];
            const typename P::real4 S = L2 ? load_l2(q) : *q;
            const CellXYZ d = cell_xyz(P::cell_of(S), a.fd_nx, a.fd_ny);
            t.f[0][k] = S.x;
            t.f[1][k] = S.y;
            t.f[2][k] = S.z;
            t.c[0][k] = d.x;
            t.c[1][k] = d.y;
            t.c[2][k] = d.z;
            t.abs[k] = make_float4((float)(T(d.x) + S.x), (float)(T(d.y) + S.y), (float)(T(d.z) + S.z), 0.0f);
        }
        __syncthreads();
        if (!live) continue;
        for (int k = lane; k < cnt; k += 32) {
            // filter on FP32 absolute positions: a pair whose approximate
            // distance is beyond the cut-off plus the rounding margin is
            // beyond the cut-off (the exact test would reject it too)
            const float4 A = t.abs[k];
            float ex = A.x - xi, ey = A.y - yi, ez = A.z - zi;
            ex -= fnx * rintf(ex * inx);
            ey -= fny * rintf(ey * iny);
            ez -= fnz * rintf(ez * inz);
            if (ex * ex + ey * ey + ez * ez >= a.lj_filter2) continue;
            if (j0 + k != i)
                pair_term(a, R, c, CellXYZ{t.c[0][k], t.c[1][k], t.c[2][k]}, t.f[0][k], t.f[1][k], t.f[2][k], Fx, Fy,
                          Fz);
        }
    }
}

// CONS: 0 ideal particles, 1 bonds, 2 Lennard-Jones and bonds.
template <typename T, bool HALF, int CONS, bool CLUSTER>
__global__ void __launch_bounds__(2 * PHASE_THREADS, sizeof(T) == 4 ? 2 : 1)
    team_phase_kernel(PArgs<T> a, int count, GridBarrier words) {
    using P = Prec<T>;
    constexpr int LANES = CONS == 2 ? 32 : 8;
    __shared__ typename std::conditional<CONS == 2, PairTile<T>, NoTile>::type tile;
    PhaseBarrier<CLUSTER> bar{words};
    if (blockIdx.x == 0 && threadIdx.x < 2) a.migrant_count[threadIdx.x] = 0;  // as in frozen_phase_kernel
    const int64_t p0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / LANES;
    const bool live = p0 < a.np;
    const int64_t p = live ? p0 : 0;  // a team without a particle follows particle 0 and writes nothing
    const int lane = (int)threadIdx.x & (LANES - 1), k = lane & 7;
    const int ox = k & 1, oy = (k >> 1) & 1, oz = k >> 2;
    T fx, fy, fz, Fx = T(0), Fy = T(0), Fz = T(0), Bx = T(0), By = T(0), Bz = T(0);
    typename P::real4 V = a.vel4[p];
    CellXYZ c;
    {
        const typename P::real4 R = a.pos4[p];
        fx = R.x;
        fy = R.y;
        fz = R.z;
        c = cell_xyz(P::cell_of(R), a.fd_nx, a.fd_ny);
    }
    const uint32_t id = (uint32_t)a.pid[p];
    if (HALF) {
        const typename P::real4 F = a.fc4[p];
        Fx = F.x;
        Fy = F.y;
        Fz = F.z;
    }
    int32_t partner = -1;
    T bond_k = T(0), bond_r0 = T(0);
    uint8_t form = 0;
    int nbond = 0;
    if (CONS) {
        const typename P::real4 B = a.fcons4[p];
        Bx = B.x;
        By = B.y;
        Bz = B.z;
        nbond = a.bond_count[id];
        if (lane < nbond) {
            const int64_t e = (int64_t)id * LBMD_MAX_BONDS_PER_PARTICLE + lane;
            partner = a.slot_of[a.bond_partner[e]];
            bond_k = (T)a.bond_k[e];
            bond_r0 = (T)a.bond_r0[e];
            form = bond_form(a.bond_kind[e], bond_r0);
        }
    }
    // ideal particles of variant A wait for nobody
    const bool coupled = CONS || a.variant != LBMD_VARIANT_A;
    const int no_list = CONS == 2 ? __syncthreads_or(a.nb_count[id] < 0) : 0;  // in this block
    const uint32_t step0 = md_step_index(a);
    const T hm = a.half_dt * V.w;  // V.w = 1 / mass
    for (int s = 0; s < count; ++s) {
        auto kick = [&](T Gx, T Gy, T Gz) {
            V.x = fma(hm, Gx, V.x);
            V.y = fma(hm, Gy, V.y);
            V.z = fma(hm, Gz, V.z);
        };
        auto kick_drift = [&]() {
            if (CONS)
                kick(Fx + Bx, Fy + By, Fz + Bz);
            else
                kick(Fx, Fy, Fz);
            advance(fx, c.x, a.dt, V.x, a.nx);
            advance(fy, c.y, a.dt, V.y, a.ny);
            advance(fz, c.z, a.dt, V.z, a.nz);
        };
        if (HALF) kick_drift();
        // the lane's corner: its record, weight and where its transfer goes
        const int xn = ox ? (c.x + 1 == a.nx ? 0 : c.x + 1) : c.x;
        const int yn = oy ? (c.y + 1 == a.ny ? 0 : c.y + 1) : c.y;
        const int zn = oz ? (c.z + 1 == a.nz ? 0 : c.z + 1) : c.z;
        const uint32_t row = (uint32_t)yn + (uint32_t)a.ny * (uint32_t)zn;
        const int sl = active_slot(a.occw[(size_t)row * (uint32_t)a.occ_words + (xn >> 5)], xn);
        const size_t r = (size_t)row * (uint32_t)a.nx + xn;
        const typename P::node4 n = load_l2(a.interp_compact && sl >= 0 ? &a.cact[sl] : &a.node[r]);
        typename P::node4 *to = sl >= 0 ? &a.cact_acc[sl] : &a.inactive_acc[r];
        const T delta = (ox ? fx : T(1) - fx) * (oy ? fy : T(1) - fy) * (oz ? fz : T(1) - fz);
        const T w = quotient(delta, P::rho_of(n));
        const T jx = P::from_fix(P::jx_of(n), a.fis), jy = P::from_fix(P::jy_of(n), a.fis),
                jz = P::from_fix(P::jz_of(n), a.fis);
        if (coupled) bar.arrive();  // while the force is computed
        T ux = T(0), uy = T(0), uz = T(0);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const T wq = __shfl_sync(0xffffffffu, w, q, LANES);
            ux = fma(wq, __shfl_sync(0xffffffffu, jx, q, LANES), ux);
            uy = fma(wq, __shfl_sync(0xffffffffu, jy, q, LANES), uy);
            uz = fma(wq, __shfl_sync(0xffffffffu, jz, q, LANES), uz);
        }
        coupling_force_id(a, id, step0 + (uint32_t)s, V, ux, uy, uz, Fx, Fy, Fz);
        if (!HALF) kick_drift();
        // every particle has read the nodes, and the others' positions of the
        // step before
        if (coupled && !bar.wait()) return;
        if (CONS) {
            if (live && lane == 0) {
                if (CONS == 2) check_list_skin(a, p, c, fx, fy, fz);
                a.pos4[p] = P::make_pos(fx, fy, fz, c.x + (int64_t)a.nx * (c.y + (int64_t)a.ny * c.z));
            }
        }
        if (live && lane < 8) {
            const T tx = Fx * a.neg_scale_dt, ty = Fy * a.neg_scale_dt, tz = Fz * a.neg_scale_dt;
            P::add_transfer(to, P::to_fix_neg(delta, tx), P::to_fix_neg(delta, ty), P::to_fix_neg(delta, tz));
        }
        // all transfers are in and all positions known
        if (coupled && (CONS || s + 1 < count) && !bar.meet()) return;
        if (CONS) {
            const typename P::real4 R = P::make_pos(fx, fy, fz, 0);
            T g = T(0), dx = T(0), dy = T(0), dz = T(0);
            if (lane < nbond) {
                const Separation<T> d = bond_separation<true>(a, R, c, partner);
                dx = d.x;
                dy = d.y;
                dz = d.z;
                g = bond_gain(form, bond_k, bond_r0, d);
            }
            Bx = By = Bz = T(0);
            if (CONS == 1) {
                for (int q = 0; q < LBMD_MAX_BONDS_PER_PARTICLE; ++q) {
                    const T gq = __shfl_sync(0xffffffffu, g, q, LANES), xq = __shfl_sync(0xffffffffu, dx, q, LANES),
                            yq = __shfl_sync(0xffffffffu, dy, q, LANES), zq = __shfl_sync(0xffffffffu, dz, q, LANES);
                    if (q < nbond) {
                        Bx = fma(gq, xq, Bx);
                        By = fma(gq, yq, By);
                        Bz = fma(gq, zq, Bz);
                    }
                }
            } else {
                if constexpr (CONS == 2) {
                    if (!no_list && __ldcg(a.nb_invalid) == 0)  // the same for the whole grid
                        listed_pairs<true>(a, id, lane, R, c, Bx, By, Bz);
                    else
                        all_pairs<true>(a, tile, id, live, lane, R, c, Bx, By, Bz);
                }
                if (lane < nbond) {
                    Bx = fma(g, dx, Bx);
                    By = fma(g, dy, By);
                    Bz = fma(g, dz, Bz);
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
                    Bx += __shfl_xor_sync(0xffffffffu, Bx, off);
                    By += __shfl_xor_sync(0xffffffffu, By, off);
                    Bz += __shfl_xor_sync(0xffffffffu, Bz, off);
                }
            }
            kick(Bx + Fx, By + Fy, Bz + Fz);
        } else {
            kick(Fx, Fy, Fz);
        }
    }
    bar.finish();
    if (!live || lane != 0) return;
    if (!CONS) a.pos4[p] = P::make_pos(fx, fy, fz, c.x + (int64_t)a.nx * (c.y + (int64_t)a.ny * c.z));
    a.vel4[p] = V;
    a.fc4[p] = P::make4(Fx, Fy, Fz, T(0));
    if (CONS) a.fcons4[p] = P::make4(Bx, By, Bz, T(0));
}

}  // namespace lbmd
