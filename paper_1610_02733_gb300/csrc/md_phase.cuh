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
#pragma once

#include "lbmd_ctx.h"
#include "lbmd_device.cuh"
#include "particle_core.cuh"
#include "particle_step.cuh"

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

}  // namespace lbmd
