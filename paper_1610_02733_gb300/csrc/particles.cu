// particles.cu -- the dissipative particle-fluid coupling of Sec. 3 on the GPU.
//
// couple_kernel (one thread per particle slot), one MD step of length dt:
//   * node velocities at the 8 corners of the particle's cell, trilinear
//     weights delta_k from the fractional position (Eq. (5));
//   * random force from Philox(id, md_step, 1, 0), friction against the
//     interpolated fluid velocity (Eq. (4)); Delta P = dt F (Eq. (6));
//   * velocity Verlet with F held fixed (second half-kick here for ideal
//     particles, in bond_kick_kernel when bonds exist);
//   * the start-of-step position and F are kept for spread_rows_kernel, which
//     adds the transfer -delta_k Delta P (Eqs. (7), (8)) once every particle
//     has read the nodes.
// Transfers are added as fixed-point integers with atomics, so the sum does
// not depend on the order of the particles (bitwise reproducible).
//
// Particle positions are stored as cell index + fractional offset in [0,1):
// the offset is exactly the interpolation coordinate, and its precision does
// not degrade with the box size.
//
// sort_*: once per LB step the particles are re-ordered by the lattice row
// (y, z) of their cell (counting sort: count, scan, scatter), so that a warp
// handles particles whose corner nodes lie in a few neighbouring rows.
//
// active_*: after each re-ordering: the corners of the particles' cells become the active nodes, numbered row by row into a compact array of
// node records (filled by the post-stream moments of the LB step).  Between
// LB updates the MD kernels read and update an active node through its
// compact record, which is about as large as the touched part of the lattice
// rather than the whole node field, and a node that is not active (one a
// particle reaches only after moving to another cell) through the node
// field, as before.
#include <algorithm>
#include <cmath>

#include "lbmd_ctx.h"
#include "lbmd_device.cuh"
#include "md_phase.cuh"
#include "particle_core.cuh"
#include "particle_step.cuh"

// the tiled variant-B MD step (md_tile.cu)
namespace lbmd {
template <typename T>
struct PArgs;
}
template <typename T>
cudaError_t md_tile_step(lbmd_ctx *ctx, const lbmd::PArgs<T> &a);

namespace lbmd {

// One MD step, coupling force from the start of the step (integrator START):
// F = -zeta (v - u(R)) + F_rand with R, v of the beginning of the step
// (Eqs. (4)-(6)), velocity Verlet with F held over both half-kicks (the
// second one here for particles without conservative forces, in the bond /
// pair kernel otherwise), transfer around the start position.
// The variant is a run-time flag (one instruction sequence for both
// variants, as in the LB kernel).  Bound by the latency of the scattered
// corner loads (16 B records; 34 % of the issue slots busy, 12 cycles of waiting on
// a load per instruction, DRAM at 31 %): 8 records in
// flight per thread (corner_records) need 64 registers, and 8 blocks of 128
// threads of them per SM measured faster (42 us at 256^3 nodes and 10^6
// particles, FP32) than 4 of 256 (44 us), 6 of 128 (45 us) or 5 of 256 with
// 48 registers (50 us; fetching the records row by row 48 us).
constexpr int COUPLE_THREADS = 128;

template <typename T, bool BONDS>
__global__ void __launch_bounds__(COUPLE_THREADS, sizeof(T) == 4 ? 8 : 4) couple_kernel(PArgs<T> a) {
    using P = Prec<T>;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.np) return;
    const typename P::real4 R = a.pos4[p];
    typename P::real4 V = a.vel4[p];
    const CellXYZ c = cell_xyz(P::cell_of(R), a.fd_nx, a.fd_ny);
    T ux, uy, uz, Fx, Fy, Fz;
    interp_u(a, c, R.x, R.y, R.z, ux, uy, uz);
    coupling_force(a, p, V, ux, uy, uz, Fx, Fy, Fz);
    // velocity Verlet with F held fixed over the step
    const T hm = a.half_dt * V.w;  // V.w = 1 / mass
    T Gx = Fx, Gy = Fy, Gz = Fz;
    if (BONDS) {
        const typename P::real4 Fc = a.fcons4[p];
        Gx += Fc.x;
        Gy += Fc.y;
        Gz += Fc.z;
    }
    V.x = fma(hm, Gx, V.x);
    V.y = fma(hm, Gy, V.y);
    V.z = fma(hm, Gz, V.z);
    T fx = R.x, fy = R.y, fz = R.z;
    int cx = c.x, cy = c.y, cz = c.z;
    advance(fx, cx, a.dt, V.x, a.nx);
    advance(fy, cy, a.dt, V.y, a.ny);
    advance(fz, cz, a.dt, V.z, a.nz);
    if (!BONDS) {
        V.x = fma(hm, Fx, V.x);
        V.y = fma(hm, Fy, V.y);
        V.z = fma(hm, Fz, V.z);
    }
    if (BONDS) check_list_skin(a, p, CellXYZ{cx, cy, cz}, fx, fy, fz);
    a.pos4[p] = P::make_pos(fx, fy, fz, cx + (int64_t)a.nx * (cy + (int64_t)a.ny * cz));
    a.vel4[p] = V;
    a.fc4[p] = P::make4(Fx, Fy, Fz, T(0));
    hand_over(a, p, R);
}

// One MD step, coupling force from the half-step velocity (integrator
// HALF_STEP): first half-kick with the previous step's F (kept in fc4) and
// the conservative force, drift, then F = -zeta (v_half - u(R')) + F_rand at
// the new position R', second half-kick (here without conservative forces,
// in the bond / pair kernel otherwise), transfer around R'.
template <typename T, bool BONDS>
__global__ void __launch_bounds__(COUPLE_THREADS, sizeof(T) == 4 ? 8 : 4) couple_half_kernel(PArgs<T> a) {
    using P = Prec<T>;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.np) return;
    const typename P::real4 R = a.pos4[p];
    typename P::real4 V = a.vel4[p];
    const CellXYZ c = cell_xyz(P::cell_of(R), a.fd_nx, a.fd_ny);
    const T hm = a.half_dt * V.w;  // V.w = 1 / mass
    typename P::real4 G = a.fc4[p];
    if (BONDS) {
        const typename P::real4 Fc = a.fcons4[p];
        G.x += Fc.x;
        G.y += Fc.y;
        G.z += Fc.z;
    }
    V.x = fma(hm, G.x, V.x);
    V.y = fma(hm, G.y, V.y);
    V.z = fma(hm, G.z, V.z);
    T fx = R.x, fy = R.y, fz = R.z;
    CellXYZ cn = c;
    advance(fx, cn.x, a.dt, V.x, a.nx);
    advance(fy, cn.y, a.dt, V.y, a.ny);
    advance(fz, cn.z, a.dt, V.z, a.nz);
    const typename P::real4 Rn = P::make_pos(fx, fy, fz, cn.x + (int64_t)a.nx * (cn.y + (int64_t)a.ny * cn.z));
    if (BONDS) check_list_skin(a, p, cn, fx, fy, fz);
    T ux, uy, uz, Fx, Fy, Fz;
    interp_u(a, cn, fx, fy, fz, ux, uy, uz);
    coupling_force(a, p, V, ux, uy, uz, Fx, Fy, Fz);
    if (!BONDS) {
        V.x = fma(hm, Fx, V.x);
        V.y = fma(hm, Fy, V.y);
        V.z = fma(hm, Fz, V.z);
    }
    a.pos4[p] = Rn;
    a.vel4[p] = V;
    a.fc4[p] = P::make4(Fx, Fy, Fz, T(0));
    hand_over(a, p, Rn);
}


// Atomic-free spreading: one warp per node row (y, z), four rows per block,
// rows in reverse order (the couple kernel touched the high rows last).  The
// row's nodes get transfers only from particles in the four cell rows
// (y - oy, z - oz), oy, oz in {0, 1}; with the particles bucketed by cell
// row, the warp reads those buckets and adds each particle's two
// contributions to this row (nodes x and x + 1, weight delta_k as in
// Eq. (5)) as fixed-point integers in shared memory, one entry per active
// node of the row; then it updates the row's compact records with plain
// loads and stores (no other warp writes them).  A contribution to an inactive node goes with atomics to the
// node field (B, C) or J_acc (A).  Particles that left their bucket's row are
// skipped here and spread by migrant_spread_kernel.
constexpr int GATHER_WARPS = 4;  // warps per block (fewer for very long rows)

// Shared-memory sums of the row gather: 3 per active node (odd stride, so
// the lanes' atomics spread over the banks), cleared with 16-byte stores; the
// per-warp area has room for 3 nx + 4 sums.
template <typename fix>
__host__ __device__ constexpr size_t acc_words(int nx) {
    return ((size_t)3 * nx + 4 + (16 / sizeof(fix)) - 1) / (16 / sizeof(fix)) * (16 / sizeof(fix));
}
template <typename fix>
__device__ __forceinline__ void acc_clear(fix *acc, int cnt, int lane) {
    constexpr int per = 16 / sizeof(fix);
    const int n4 = (3 * cnt + per - 1) / per;
    int4 *a4 = reinterpret_cast<int4 *>(acc);
    for (int k = lane; k < n4; k += 32) a4[k] = make_int4(0, 0, 0, 0);
}

// bytes of the active-word area of one block (rounded to 16)
__host__ __device__ inline size_t gather_occ_bytes(int warps, int W) {
    return ((size_t)warps * W * sizeof(uint2) + 15) & ~(size_t)15;
}

template <typename T>
__global__ void __launch_bounds__(32 * GATHER_WARPS) spread_rows_kernel(PArgs<T> a, int n_rows) {
    using P = Prec<T>;
    using fix = typename P::fix;
    using N4 = typename P::node4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warps = blockDim.x >> 5;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int W = a.occ_words;
    // per warp: the row's active words (slots relative to the row's first),
    // then the sums of the active nodes
    uint2 *occ = reinterpret_cast<uint2 *>(smem_raw) + (size_t)warp * W;
    fix *acc = reinterpret_cast<fix *>(smem_raw + gather_occ_bytes(warps, W)) + (size_t)warp * acc_words<fix>(a.nx);
    const int g = blockIdx.x * warps + warp;
    if (g >= n_rows) return;
    const int nrow = n_rows - 1 - g;
    const int z = (int)fdiv((uint32_t)nrow, a.fd_ny), y = nrow - z * a.ny;
    // the four cell rows (y - oy, z - oz), q = oy + 2 oz, as one run of
    // total = e[4] particle entries: entry t belongs to row q with
    // e[q] <= t < e[q + 1], at slot lo[q] + t - e[q]
    const int ym = y == 0 ? a.ny - 1 : y - 1, zm = z == 0 ? a.nz - 1 : z - 1;
    const int c0 = y + a.ny * z, c1 = ym + a.ny * z, c2 = y + a.ny * zm, c3 = ym + a.ny * zm;
    const int lo0 = a.row_start[c0], lo1 = a.row_start[c1], lo2 = a.row_start[c2], lo3 = a.row_start[c3];
    // (a re-ordering that the limit of a barrier ended may leave the starts of
    // two orderings: no row's count is taken as negative)
    const int e1 = max(a.row_start[c0 + 1] - lo0, 0);
    const int e2 = e1 + max(a.row_start[c1 + 1] - lo1, 0);
    const int e3 = e2 + max(a.row_start[c2 + 1] - lo2, 0);
    const int total = e3 + max(a.row_start[c3 + 1] - lo3, 0);
    const uint2 *wrow = a.occw + (size_t)nrow * W;
    const int base = (int)wrow[0].y;
    for (int w = lane; w < W; w += 32) {
        uint2 v = wrow[w];
        v.y -= (uint32_t)base;
        occ[w] = v;
    }
    const uint2 last = wrow[W - 1];
    const int cnt = (int)last.y - base + __popc(last.x);
    acc_clear(acc, cnt, lane);
    __syncwarp();
    N4 *rowp = a.inactive_acc + (size_t)a.nx * nrow;
    // entries in passes of 64, two per lane, both loaded before either is used
    for (int t0 = 0; t0 < total; t0 += 64) {
        typename P::real4 Rv[2], Fv[2];
        int crow[2];
        bool oyv[2], ozv[2], live[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = t0 + 32 * h + lane;
            live[h] = t < total;
            const bool b1 = t >= e1, b2 = t >= e2, b3 = t >= e3;
            const int slot0 = b3 ? lo3 - e3 : b2 ? lo2 - e2 : b1 ? lo1 - e1 : lo0;
            crow[h] = b3 ? c3 : b2 ? c2 : b1 ? c1 : c0;
            oyv[h] = b1 != b2 || b3;  // q = 1 or 3
            ozv[h] = b2;              // q = 2 or 3
            if (live[h]) {
                Rv[h] = a.old4[slot0 + t];
                Fv[h] = a.fc4[slot0 + t];
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (!live[h]) continue;
            const typename P::real4 R = Rv[h], F = Fv[h];
            // cell x within the bucket's row; anything else is a migrant
            const int cx = (int)((uint32_t)P::cell_of(R) - (uint32_t)crow[h] * (uint32_t)a.nx);
            if ((uint32_t)cx >= (uint32_t)a.nx) continue;
            const int x1 = cx + 1 == a.nx ? 0 : cx + 1;
            const T wx[2] = {T(1) - R.x, R.x};
            const T wy = oyv[h] ? R.y : T(1) - R.y;
            const T wz = ozv[h] ? R.z : T(1) - R.z;
            const T sx = F.x * a.neg_scale_dt, sy = F.y * a.neg_scale_dt, sz = F.z * a.neg_scale_dt;
#pragma unroll
            for (int ox = 0; ox < 2; ++ox) {
                const T d = wx[ox] * wy * wz;  // the corner weight delta_k of Eq. (5)
                const int xn = ox ? x1 : cx;
                const fix vx = P::to_fix_neg(d, sx), vy = P::to_fix_neg(d, sy), vz = P::to_fix_neg(d, sz);
                const int sl = active_slot(occ[xn >> 5], xn);
                if (sl >= 0) {
                    fix *ak = acc + 3 * sl;
                    fix_add(ak + 0, vx);
                    fix_add(ak + 1, vy);
                    fix_add(ak + 2, vz);
                } else {
                    P::add_transfer(&rowp[xn], vx, vy, vz);
                }
            }
        }
    }
    __syncwarp();
    // write-back in passes of 128 nodes, the four records loaded together
    N4 *crec = a.cact_acc + base;
    for (int k0 = 0; k0 < cnt; k0 += 128) {
        N4 rec[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int k = k0 + 32 * h + lane;
            if (k < cnt) rec[h] = crec[k];
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int k = k0 + 32 * h + lane;
            if (k >= cnt) continue;
            const fix dx = acc[3 * k], dy = acc[3 * k + 1], dz = acc[3 * k + 2];
            if (dx == 0 && dy == 0 && dz == 0) continue;
            P::add_transfer_reg(rec[h], dx, dy, dz);
            crec[k] = rec[h];
        }
    }
}

// Every particle's transfers with atomics (LBMD_SPREAD_ATOMIC), FP32: one thread
// per corner -- 8 times the threads for a kernel whose threads each wait on
// their loads and then queue 16 atomics (7 -> 4.5 us at 53,000 particles).  FP64,
// whose arithmetic would be repeated per corner on its slow pipe, keeps a
// thread per particle (128^3 nodes, 131,072 particles: 1032 us a cycle, 1121 with this).
template <typename T>
__global__ void __launch_bounds__(256) spread_all_kernel(PArgs<T> a) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < 2) a.migrant_count[t] = 0;  // the row gather's lists are not in use
    if ((t >> 3) < a.np) spread_corner_atomic(a, t >> 3, (int)t & 7);
}
// The migrants of this MD step, spread with atomics once the row gather is done
// (particle_step.cuh); in FP32 with a thread per corner (256^3 nodes, 10^6
// particles: the cycle 1670 -> 1655 us).  With `all` (FP64) every particle is
// spread this way and the row gather does not run (LBMD_SPREAD_ATOMIC).
template <typename T>
__global__ void __launch_bounds__(256) migrant_spread_kernel(PArgs<T> a, int all) {
    using P = Prec<T>;
    const int par = a.mig_par;
    const int n = all ? (int)a.np : a.migrant_count[par];
    // the other list serves the next MD step: empty it now (nobody uses it
    // during this one)
    if (blockIdx.x == 0 && threadIdx.x == 0) a.migrant_count[par ^ 1] = 0;
    const int32_t *list = a.migrant_slot + (int64_t)par * a.np_cap;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (sizeof(T) == 4 && !all) {  // a thread per corner, as in spread_all_kernel
        for (; t < 8 * (int64_t)n; t += stride) spread_corner_atomic(a, (int64_t)list[t >> 3], (int)t & 7);
    } else {
        for (; t < n; t += stride) spread_particle_atomic(a, all ? t : (int64_t)list[t]);
    }
}

// Bond forces (harmonic or FENE) at the current positions (minimum image),
// summed per particle over its partners in a fixed order; with KICK, also
// the second velocity-Verlet half-kick with the stored coupling force.
template <typename T, bool KICK>
__global__ void __launch_bounds__(256) bond_kick_kernel(PArgs<T> a) {
    using P = Prec<T>;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.np) return;
    const typename P::real4 R = a.pos4[p];
    const CellXYZ c = cell_xyz(P::cell_of(R), a.fd_nx, a.fd_ny);
    const int64_t id = a.pid[p];
    T Fx, Fy, Fz;
    bond_forces(a, id, R, c, Fx, Fy, Fz);
    a.fcons4[p] = P::make4(Fx, Fy, Fz, T(0));
    if (KICK) {
        typename P::real4 V = a.vel4[p];
        const typename P::real4 Fc = a.fc4[p];
        const T hm = a.half_dt * V.w;
        V.x = fma(hm, Fx + Fc.x, V.x);
        V.y = fma(hm, Fy + Fc.y, V.y);
        V.z = fma(hm, Fz + Fc.z, V.z);
        a.vel4[p] = V;
        // variant B, all atomics: every particle has read the nodes (couple
        // kernel), so the transfers can go in now
        if (a.kick_spreads) spread_particle_atomic(a, p);
    }
}


// Conservative forces with Lennard-Jones (Kremer-Grest monomers, Sec. 4):
// one warp per particle id i, eight per block.  The block stages the other
// particles in tiles of PairTile ids in shared memory (cell coordinates and
// offsets, decoded once per block instead of once per pair); the lanes then
// run over the tile (lane l takes ids l, l + 32, ...) and add the LJ force of
// every j within the cut-off,
//   F_i += g d,  g = -24 eps (2 t^2 - t) / r^2,  t = (sigma^2 / r^2)^3,
// d = R_j - R_i at the nearest image (cell offsets wrapped as integers, then
// the fractional offsets added: exact to the last bit of the offsets; every
// box edge is at least 2 r_cut + 2, so the nearest image is unique within
// the cut-off); lane b < n_bonds(i) adds bond b.  The lane sums are combined
// by a fixed butterfly, so the result does not depend on the slot order.
// With KICK, lane 0 also makes the second velocity-Verlet half-kick.
constexpr int PAIR_THREADS = 256;  // eight particles per block

template <typename T, bool KICK>
__global__ void __launch_bounds__(PAIR_THREADS) pair_kick_kernel(PArgs<T> a) {
    using P = Prec<T>;
    __shared__ PairTile<T> tile;
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const bool live = i < a.np;
    const int64_t p = live ? a.slot_of[i] : 0;
    const typename P::real4 R = a.pos4[p];
    const CellXYZ c = cell_xyz(P::cell_of(R), a.fd_nx, a.fd_ny);
    T Fx = T(0), Fy = T(0), Fz = T(0);
    // Verlet lists when they hold every pair within the cut-off (no particle
    // moved more than half the skin since the build, no list overflowed in
    // this block).  Lane l takes the listed ids j = l (mod 32) in ascending
    // order: the same terms in the same order as the all-pairs loop below,
    // so both give the same bits.
    int use_all = a.nb_list == nullptr || *a.nb_invalid != 0;
    if (!use_all && live && a.nb_count[i] < 0) use_all = 1;
    use_all = __syncthreads_or(use_all);
    if (!use_all && live) listed_pairs(a, i, lane, R, c, Fx, Fy, Fz);  // whole warps
    if (use_all) all_pairs<false>(a, tile, i, live, lane, R, c, Fx, Fy, Fz);
    if (!live) return;  // whole warps, after the block's last barrier
    if (lane < a.bond_count[i]) {
        const int64_t e = i * LBMD_MAX_BONDS_PER_PARTICLE + lane;
        const Separation<T> d = bond_separation(a, R, c, a.slot_of[a.bond_partner[e]]);
        const T r0 = (T)a.bond_r0[e], g = bond_gain(bond_form(a.bond_kind[e], r0), (T)a.bond_k[e], r0, d);
        Fx = fma(g, d.x, Fx);
        Fy = fma(g, d.y, Fy);
        Fz = fma(g, d.z, Fz);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        Fx += __shfl_xor_sync(0xffffffffu, Fx, off);
        Fy += __shfl_xor_sync(0xffffffffu, Fy, off);
        Fz += __shfl_xor_sync(0xffffffffu, Fz, off);
    }
    // variant B, all atomics: the couple kernel is done, so every particle
    // has read the nodes; lanes 0..7 hand over the 8 corner transfers
    if (KICK && a.kick_spreads && lane < 8) spread_corner_atomic(a, p, lane);
    if (lane != 0) return;
    a.fcons4[p] = P::make4(Fx, Fy, Fz, T(0));
    if (KICK) {
        typename P::real4 V = a.vel4[p];
        const typename P::real4 Fc = a.fc4[p];
        const T hm = a.half_dt * V.w;
        V.x = fma(hm, Fx + Fc.x, V.x);
        V.y = fma(hm, Fy + Fc.y, V.y);
        V.z = fma(hm, Fz + Fc.z, V.z);
        a.vel4[p] = V;
    }
}

// LJ Verlet lists, rebuilt after each re-ordering (rebuilding only voided
// lists made the all-pairs fallback frequent: the skin is then spent over
// several LB steps): one warp per slot q (particle i = pid[q]) builds i's
// list: the lanes run over the particles of the row buckets
// within ceil(r_list) rows in y and z (each distinct row once; the buckets'
// slot ranges are concatenated and shared out 32 at a time), keep the ids
// j != i closer than r_list = r_cut + skin, and write their slots (fixed until
// the next re-ordering) ordered by (id mod 32, id), so that a lane of the pair
// loop reads its own share and nothing else (each lane ranks its entries by
// counting the smaller ones).  A particle with
// more than LBMD_NB_MAX candidates gets count -1 (its block then uses all
// pairs).  The positions at the build are kept per id.
constexpr int NB_WARPS = 8;

template <typename T>
__global__ void __launch_bounds__(32 * NB_WARPS) nb_build_kernel(PArgs<T> a, T rlist2, int reach) {
    using P = Prec<T>;
    __shared__ int32_t s_ids[NB_WARPS][LBMD_NB_MAX], s_slots[NB_WARPS][LBMD_NB_MAX];
    __shared__ int s_cnt[NB_WARPS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t q = (int64_t)blockIdx.x * NB_WARPS + warp;
    if (q >= a.np) return;  // whole warps; no block barrier below
    const int32_t i = a.pid[q];
    const typename P::real4 R = a.pos4[q];
    const CellXYZ c = cell_xyz(P::cell_of(R), a.fd_nx, a.fd_ny);
    if (lane == 0) {
        s_cnt[warp] = 0;
        const_cast<typename P::real4 *>(a.nb_ref4)[i] = R;
    }
    __syncwarp();
    const int ny_rows = 2 * reach + 1 < a.ny ? 2 * reach + 1 : a.ny;
    const int nz_rows = 2 * reach + 1 < a.nz ? 2 * reach + 1 : a.nz;
    const int y0 = 2 * reach + 1 < a.ny ? c.y - reach + a.ny : 0;
    const int z0 = 2 * reach + 1 < a.nz ? c.z - reach + a.nz : 0;
    const int nrows = ny_rows * nz_rows;
    for (int r0 = 0; r0 < nrows; r0 += 32) {
        // lane r: the slot range of candidate row r0 + r, and its offset in
        // the concatenation of the ranges
        int lo = 0, cnt = 0;
        if (r0 + lane < nrows) {
            const int ky = (r0 + lane) % ny_rows, kz = (r0 + lane) / ny_rows;
            const int row = (y0 + ky) % a.ny + a.ny * ((z0 + kz) % a.nz);
            lo = a.row_start[row];
            cnt = max(a.row_start[row + 1] - lo, 0);  // (as in spread_rows_kernel)
        }
        int incl = cnt;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += v;
        }
        const int excl = incl - cnt;
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        for (int t0 = 0; t0 < total; t0 += 32) {
            const int t = t0 + lane;
            // the last row whose range starts at or before t
            int r = 0;
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                const int v = __shfl_sync(0xffffffffu, excl, r + step);
                if (v <= t) r += step;
            }
            const int lo_r = __shfl_sync(0xffffffffu, lo, r), ex_r = __shfl_sync(0xffffffffu, excl, r);
            if (t >= total) continue;
            const int sl = lo_r + (t - ex_r);
            const int32_t j = a.pid[sl];
            if (j == i) continue;
            const typename P::real4 S = a.pos4[sl];
            const CellXYZ d = cell_xyz(P::cell_of(S), a.fd_nx, a.fd_ny);
            const T dx = T(nearest_image(d.x - c.x, a.nx)) + (S.x - R.x);
            const T dy = T(nearest_image(d.y - c.y, a.ny)) + (S.y - R.y);
            const T dz = T(nearest_image(d.z - c.z, a.nz)) + (S.z - R.z);
            if (dx * dx + dy * dy + dz * dz < rlist2) {
                const int k = atomicAdd(&s_cnt[warp], 1);
                if (k < LBMD_NB_MAX) {
                    s_ids[warp][k] = j;
                    s_slots[warp][k] = sl;
                }
            }
        }
    }
    __syncwarp();
    const int cnt = s_cnt[warp];
    if (cnt > LBMD_NB_MAX) {
        if (lane == 0) const_cast<int32_t *>(a.nb_count)[i] = -1;
        return;
    }
    // slots by (id mod 32, id); the end of each class
    int32_t *L = const_cast<int32_t *>(a.nb_list) + (int64_t)i * LBMD_NB_MAX;
    for (int k = lane; k < cnt; k += 32) {
        const int32_t j = s_ids[warp][k];
        int rank = 0;
        for (int m = 0; m < cnt; ++m) {
            const int32_t o = s_ids[warp][m];
            rank += (o & 31) < (j & 31) || ((o & 31) == (j & 31) && o < j) ? 1 : 0;
        }
        L[rank] = s_slots[warp][k];
    }
    int end = 0;
    for (int m = 0; m < cnt; ++m) end += (s_ids[warp][m] & 31) <= lane ? 1 : 0;
    const_cast<uint8_t *>(a.nb_end)[(int64_t)i * 32 + lane] = (uint8_t)end;
    if (lane == 0) const_cast<int32_t *>(a.nb_count)[i] = cnt;
}

// after a build (or none): the lists hold every pair within the cut-off
__global__ void nb_validate_kernel(int32_t *invalid) { *invalid = 0; }

// ---------------------------------------------------------------------------
// Re-ordering by lattice row.
// ---------------------------------------------------------------------------
// Every particle's rank within its cell row, and its cell marked in the row's
// occupancy words.  The particles come mostly in row order (the
// order of the last re-ordering), so the valid lanes of a warp form runs of
// equal rows (and of equal occupancy words): each run takes its ranks with one
// atomic on the row's count, and ORs its cells into a word with one atomic.
// The order within a row is free: every later sum is order-independent.
// (All lanes of a warp come here; those with p < np are a prefix of it.)
template <typename T>
__device__ __forceinline__ void count_particle(const typename Prec<T>::real4 *pos4, int64_t p, int64_t np,
                                               const FastDiv &fnx, int32_t *row_count, int32_t *rank, uint32_t *ccw,
                                               int W) {
    const unsigned act = __ballot_sync(0xffffffffu, p < np);
    if (p >= np) return;
    const int lane = (int)(threadIdx.x & 31), nvalid = __popc(act);
    const unsigned upto = 0xffffffffu >> (31 - lane);  // lanes 0..lane
    const uint32_t cell = (uint32_t)Prec<T>::cell_of(pos4[p]);
    const uint32_t row = fdiv(cell, fnx);
    // runs of equal rows: the run's first lane takes the ranks
    const uint32_t row_prev = __shfl_up_sync(act, row, 1);
    const unsigned heads = __ballot_sync(act, lane == 0 || row_prev != row);
    const int head = 31 - __clz((int)(heads & upto));
    const unsigned after = heads & ~upto;
    const int next = after ? __ffs((int)after) - 1 : nvalid;
    int base = 0;
    if (lane == head) base = atomicAdd(&row_count[row], next - head);
    base = __shfl_sync(act, base, head);
    rank[p] = base + (lane - head);
    const uint32_t cx = cell - row * fnx.d;
    const unsigned long long key = (unsigned long long)row * (unsigned)W + (cx >> 5);
    const unsigned long long key_prev = __shfl_up_sync(act, key, 1);
    const unsigned kheads = __ballot_sync(act, lane == 0 || key_prev != key);
    const unsigned kafter = kheads & ~upto;
    const int knext = kafter ? __ffs((int)kafter) - 1 : nvalid;
    // the run's cells ORed towards its first lane (segmented, log steps)
    uint32_t bits = 1u << (cx & 31);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t o = __shfl_down_sync(act, bits, off);
        if (lane + off < knext) bits |= o;
    }
    if (kheads & (1u << lane)) atomicOr(&ccw[key], bits);
}

template <typename T>
__global__ void __launch_bounds__(256)
    sort_count_kernel(const typename Prec<T>::real4 *pos4, int64_t np, FastDiv fnx, int32_t *row_count, int32_t *rank,
                      uint32_t *ccw, int W) {
    count_particle<T>(pos4, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, np, fnx, row_count, rank, ccw, W);
}

// Block-wide exclusive scan of one value per thread (whole warps, up to 1024
// threads).
__device__ __forceinline__ int32_t block_exclusive_scan(int32_t v, int32_t *total) {
    __shared__ int32_t warp_sum[32];
    const int warps = (int)(blockDim.x >> 5);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t x = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) warp_sum[w] = x;
    __syncthreads();
    if (w == 0) {
        int32_t s = lane < warps ? warp_sum[lane] : 0;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, s, off);
            if (lane >= off) s += y;
        }
        warp_sum[lane] = s;  // inclusive prefix of warp sums (the total beyond the last)
    }
    __syncthreads();
    const int32_t before = w > 0 ? warp_sum[w - 1] : 0;
    if (total) *total = warp_sum[31];
    __syncthreads();
    return before + x - v;
}

// Level 1: each block of 1024 threads turns 1024 row counts into exclusive
// offsets within its chunk and records the chunk total.
__global__ void __launch_bounds__(1024) sort_chunk_scan_kernel(int32_t *row_count, int64_t n, int32_t *chunk_total) {
    const int64_t i = (int64_t)blockIdx.x * 1024 + threadIdx.x;
    const int32_t v = i < n ? row_count[i] : 0;
    int32_t tot;
    const int32_t ex = block_exclusive_scan(v, &tot);
    if (i < n) row_count[i] = ex;
    if (threadIdx.x == 0) chunk_total[blockIdx.x] = tot;
}

// Level 2: block c adds the totals of chunks 0..c-1 to its 1024 offsets,
// giving the first slot of every row; row_start[n] = np closes the table.
__global__ void __launch_bounds__(1024) sort_finalize_kernel(const int32_t *row_offset, const int32_t *chunk_total,
                                                             int64_t n, int32_t *row_start, int32_t np) {
    int32_t before;
    const int32_t v = (int)threadIdx.x < (int)blockIdx.x ? chunk_total[threadIdx.x] : 0;
    block_exclusive_scan(v, &before);  // total of the first blockIdx.x chunks
    const int64_t i = (int64_t)blockIdx.x * 1024 + threadIdx.x;
    if (i < n) row_start[i] = before + row_offset[i];
    if (i == n - 1) row_start[n] = np;
}

// Move every particle to row_start[row] + rank within the row, with its
// conservative force (if any) and its last coupling force (integrator
// HALF_STEP, where it carries over to the next MD step).
template <typename T>
struct ScatterArgs {
    using R4 = typename Prec<T>::real4;
    const R4 *pos_in, *vel_in, *fcons_in, *fc_in;
    const int32_t *pid_in;
    R4 *pos_out, *vel_out, *fcons_out, *fc_out;
    int32_t *pid_out, *slot_of, *slot_row;
    int32_t *rank;
    int64_t np;
    FastDiv fnx;
    int bonds, carry_fc;
};
template <typename T>
__device__ __forceinline__ void scatter_particle(const ScatterArgs<T> &a, int64_t p, uint32_t row, int32_t dst) {
    a.slot_row[dst] = (int32_t)row;
    a.vel_out[dst] = a.vel_in[p];
    if (a.bonds) a.fcons_out[dst] = a.fcons_in[p];
    if (a.carry_fc) a.fc_out[dst] = a.fc_in[p];
    const int32_t id = a.pid_in[p];
    a.pid_out[dst] = id;
    a.slot_of[id] = dst;
}
template <typename T>
__global__ void __launch_bounds__(256) sort_scatter_kernel(ScatterArgs<T> a, const int32_t *row_start) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.np) return;
    const typename Prec<T>::real4 R = a.pos_in[p];
    const uint32_t row = fdiv((uint32_t)Prec<T>::cell_of(R), a.fnx);
    const int32_t dst = row_start[row] + a.rank[p];
    a.pos_out[dst] = R;
    scatter_particle(a, p, row, dst);
}

// ---------------------------------------------------------------------------
// Active nodes, rebuilt after each re-ordering.
// ---------------------------------------------------------------------------
// Level 0: node x of row (y, z) is active when a particle's cell has it as a
// corner, i.e. when cell x or x - 1 (periodic) of one of the four cell rows
// (y - oy, z - oz), oy, oz in {0, 1}, holds a particle.  A group of L lanes
// (L = min(32, W rounded up to a power of two)) builds one row's words from
// the cell-occupancy words ccw, with the in-row slot of each word's first
// active node (a scan over the group), and the row's count.
// (All lanes of a warp come here; valid: nrow is a row.)  Returns the row's
// count, in every lane of the group.
template <bool L2 = false>
__device__ __forceinline__ int active_row(const uint32_t *ccw, int nx, const FastDiv &fny, int nz, int W, int L,
                                          uint2 *occw, int nrow, int sub, bool valid) {
    const int ny = (int)fny.d;
    int cr[4] = {0, 0, 0, 0};
    if (valid) {
        const int z = (int)fdiv((uint32_t)nrow, fny), y = nrow - z * ny;
        const int ym = y == 0 ? ny - 1 : y - 1, zm = z == 0 ? nz - 1 : z - 1;
        cr[0] = y + ny * z;
        cr[1] = ym + ny * z;
        cr[2] = y + ny * zm;
        cr[3] = ym + ny * zm;
    }
    const int last = nx - 1;
    const uint32_t tail_mask = (nx & 31) ? ((1u << (nx & 31)) - 1u) : 0xffffffffu;
    auto word = [&](const uint32_t *p) { return L2 ? __ldcg(p) : *p; };
    int carry = 0;
    for (int w0 = 0; w0 < W; w0 += L) {  // uniform over the warp
        const int w = w0 + sub;
        uint32_t a = 0u;
        if (valid && w < W) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t *cw = ccw + (size_t)cr[c] * W;
                const uint32_t b = word(cw + w);
                // cell x - 1 of bit x: the previous word's top bit, or (w = 0)
                // the periodic neighbour x = nx - 1
                const uint32_t in = w > 0 ? (word(cw + w - 1) >> 31) : ((word(cw + (last >> 5)) >> (last & 31)) & 1u);
                a |= b | (b << 1) | in;
            }
            if (w == W - 1) a &= tail_mask;
        }
        const int cnt = __popc(a);
        int incl = cnt;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, off, L);
            if (off < L && sub >= off) incl += v;
        }
        if (valid && w < W) occw[(size_t)nrow * W + w] = make_uint2(a, (uint32_t)(carry + incl - cnt));
        carry += __shfl_sync(0xffffffffu, incl, L - 1, L);
    }
    return carry;
}
__global__ void __launch_bounds__(256)
    active_rows_kernel(const uint32_t *ccw, int nx, FastDiv fny, int nz, int W, int L, uint2 *occw, int32_t *row_count,
                       int n_rows) {
    const int lane = (int)(threadIdx.x & 31);
    const int gwarp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int nrow = gwarp * (32 / L) + lane / L, sub = lane % L;
    const bool valid = nrow < n_rows;
    const int cnt = active_row(ccw, nx, fny, nz, W, L, occw, nrow, sub, valid);
    if (valid && sub == 0) row_count[nrow] = cnt;
}

// Level 2 (after sort_chunk_scan_kernel turned the row counts into offsets
// within chunks of 1024 rows): the first slot of every row added to the
// in-row slots of its words, one word per thread; block (c, s) takes slice s
// of chunk c's words.
constexpr int FINALIZE_SLICES = 4;
__global__ void __launch_bounds__(1024) active_finalize_kernel(const int32_t *row_offset, const int32_t *chunk_total,
                                                               int64_t n_rows, uint2 *occw, int W, int32_t *arow) {
    int32_t before;
    const int32_t v = (int)threadIdx.x < (int)blockIdx.x ? chunk_total[threadIdx.x] : 0;
    block_exclusive_scan(v, &before);  // total of the first blockIdx.x chunks
    const int64_t r0 = (int64_t)blockIdx.x * 1024, r1 = r0 + 1024 < n_rows ? r0 + 1024 : n_rows;
    const int64_t w_end = r1 * W;
    for (int64_t i = r0 * W + (int64_t)blockIdx.y * 1024 + threadIdx.x; i < w_end; i += FINALIZE_SLICES * 1024) {
        const int64_t row = i / W;
        const uint32_t b = (uint32_t)(before + row_offset[row]);
        uint2 wd = occw[i];
        wd.y += b;
        occw[i] = wd;
        if (i == row * W) arow[row] = (int32_t)b;  // the row's first compact slot
        if (row == n_rows - 1 && i == w_end - 1) arow[n_rows] = (int32_t)(wd.y + __popc(wd.x));  // closes the table
    }
}

// The re-ordering and the active set in one launch, for lattices of at most one
// row per thread of the grid: the counting of the particles, the scan of the
// rows with the marking of the active nodes, and the move of the particles with
// the numbering of the nodes, between two grid barriers.  Block b takes the
// rows [b per, (b + 1) per); for the scans it adds up the counts of all rows
// before its own (at most 38,912 values out of L2).  row_count and ccw are zero
// before and after -- unless the limit of a barrier ends the kernel: the counts
// then stay as they are, and no later launch gets past its first barrier to use
// them.  As seven launches and two memsets the same took 23 us at
// 64^3 nodes, where each of them is a launch's latency; this takes 9.
constexpr int REORDER_THREADS = 256;

// sum of v[0..n) over the block, read past L1, 16 values of a thread in flight
__device__ __forceinline__ int32_t block_sum_before(const int32_t *v, int n) {
    const int4 *v4 = reinterpret_cast<const int4 *>(v);
    int32_t s = 0;
    for (int i = (int)threadIdx.x; i < n / 4; i += 4 * REORDER_THREADS) {
        int4 q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            q[u] = i + u * REORDER_THREADS < n / 4 ? __ldcg(v4 + i + u * REORDER_THREADS) : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < 4; ++u) s += (q[u].x + q[u].y) + (q[u].z + q[u].w);
    }
    if ((int)threadIdx.x < n % 4) s += __ldcg(v + n / 4 * 4 + threadIdx.x);
    int32_t total;
    block_exclusive_scan(s, &total);
    return total;
}

template <typename T>
__global__ void __launch_bounds__(REORDER_THREADS)
    reorder_kernel(ScatterArgs<T> a, int32_t *row_count, int32_t *active_count, int32_t *row_start, uint32_t *ccw,
                   uint2 *occw, int32_t *arow, int32_t *lb_missed, FastDiv fny, int nz, int W, int L, int per,
                   GridBarrier words) {
    PhaseBarrier<false> bar{words};
    const int n_rows = (int)fny.d * nz, nx = (int)a.fnx.d;
    const int64_t stride = (int64_t)gridDim.x * REORDER_THREADS, start = (int64_t)blockIdx.x * REORDER_THREADS;
    const int tid = (int)threadIdx.x, lane = tid & 31;
    for (int64_t b = start; b < a.np; b += stride)
        count_particle<T>(a.pos_in, b + tid, a.np, a.fnx, row_count, a.rank, ccw, W);
    if (blockIdx.x == 0 && tid == 0) *lb_missed = 0;
    if (!bar.meet()) return;
    const int r0 = min(n_rows, (int)blockIdx.x * per), r1 = min(n_rows, r0 + per), r = r0 + tid;
    int32_t before = block_sum_before(row_count, r0);
    const int32_t first = before + block_exclusive_scan(r < r1 ? __ldcg(row_count + r) : 0, nullptr);
    if (r < r1) row_start[r] = first;
    if (blockIdx.x == 0 && tid == 0) row_start[n_rows] = (int32_t)a.np;
    const int rows_per_warp = 32 / L;
    for (int q = r0 + (tid >> 5) * rows_per_warp; q < r1; q += (REORDER_THREADS / 32) * rows_per_warp) {
        const int nrow = q + lane / L;
        const bool valid = nrow < r1;
        const int cnt = active_row<true>(ccw, nx, fny, nz, W, L, occw, nrow, lane % L, valid);
        if (valid && lane % L == 0) active_count[nrow] = cnt;
    }
    if (!bar.meet()) return;
    before = block_sum_before(active_count, r0);
    const int32_t mine = r < r1 ? __ldcg(active_count + r) : 0;
    __shared__ int32_t s_base[REORDER_THREADS];
    s_base[tid] = before + block_exclusive_scan(mine, nullptr);
    if (r < r1) {
        arow[r] = s_base[tid];
        if (r == n_rows - 1) arow[n_rows] = s_base[tid] + mine;
        row_count[r] = 0;
    }
    __syncthreads();
    for (int i = tid; i < (r1 - r0) * W; i += REORDER_THREADS) {
        const size_t w = (size_t)r0 * W + i;
        occw[w].y += (uint32_t)s_base[i / W];
        ccw[w] = 0u;
    }
    for (int64_t p = start + tid; p < a.np; p += stride) {
        const typename Prec<T>::real4 R = a.pos_in[p];
        const uint32_t row = fdiv((uint32_t)Prec<T>::cell_of(R), a.fnx);
        const int32_t dst = __ldcg(row_start + row) + a.rank[p];
        a.pos_out[dst] = R;
        scatter_particle(a, p, row, dst);
    }
    bar.finish();
}

// Node field entries of the active nodes brought up to date from their
// compact records (for the observables and the host accessors).
template <typename T>
__global__ void __launch_bounds__(256) active_sync_kernel(const uint2 *occw, const typename Prec<T>::node4 *cact,
                                                          typename Prec<T>::node4 *node, int64_t N, int nx, int W) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= N) return;
    const int64_t row = r / nx;
    const int x = (int)(r - row * nx);
    const int sl = active_slot(occw[(size_t)row * W + (x >> 5)], x);
    if (sl >= 0) node[r] = cact[sl];
}

// shared memory of the row gather with `warps` warps per block: the rows'
// active words and the sums of up to nx active nodes per row
template <typename T>
static size_t gather_smem_bytes(const lbmd_ctx *ctx, int warps) {
    using fix = typename Prec<T>::fix;
    return gather_occ_bytes(warps, active_words(ctx->p.nx)) + (size_t)warps * acc_words<fix>(ctx->p.nx) * sizeof(fix);
}

template <typename T, bool CLUSTER>
static const void *phase_kernel(bool half, int cons) {
    if (half)
        return cons == 2   ? (const void *)team_phase_kernel<T, true, 2, CLUSTER>
               : cons == 1 ? (const void *)team_phase_kernel<T, true, 1, CLUSTER>
                           : (const void *)team_phase_kernel<T, true, 0, CLUSTER>;
    return cons == 2   ? (const void *)team_phase_kernel<T, false, 2, CLUSTER>
           : cons == 1 ? (const void *)team_phase_kernel<T, false, 1, CLUSTER>
                       : (const void *)team_phase_kernel<T, false, 0, CLUSTER>;
}

// The row gather's shared memory grows with nx: as many warps per block (at
// most GATHER_WARPS) as fit in 200 KB, and the opt-in above the default
// 48 KB per block.
template <typename T>
static cudaError_t setup_t(lbmd_ctx *ctx) {
    int warps = GATHER_WARPS;
    while (warps > 1 && gather_smem_bytes<T>(ctx, warps) > (size_t)200 * 1024) --warps;
    const size_t smem = gather_smem_bytes<T>(ctx, warps);
    if (smem > (size_t)200 * 1024) return cudaErrorInvalidValue;
    ctx->gather_warps = warps;
    cudaError_t e = cudaFuncSetAttribute(spread_rows_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // threads of the team phase that are resident at once: the Lennard-Jones
    // forms take the most registers and shared memory
    int per_sm = 1 << 30;
    for (int k = 0; k < 6; ++k) {
        e = cudaFuncSetAttribute(phase_kernel<T, true>(k >= 3, k % 3), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        if (k % 3 != 2) continue;
        int n = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, phase_kernel<T, false>(k >= 3, 2), 2 * PHASE_THREADS, 0);
        if (e != cudaSuccess) return e;
        per_sm = std::min(per_sm, n);
    }
    ctx->phase_threads = (int64_t)per_sm * ctx->sm_count * 2 * PHASE_THREADS;
    // the largest cluster every form can run as
    ctx->phase_cluster = PHASE_CLUSTER;
    for (int half = 0; half < 2; ++half)
        if ((e = limit_cluster(phase_kernel<T, true>(half != 0, 2), PHASE_THREADS, ctx->phase_cluster)) != cudaSuccess)
            return e;
    return md_tile_setup_kernels(ctx);
}

template <typename T>
static PArgs<T> make_pargs(lbmd_ctx *ctx, int substep) {
    using P = Prec<T>;
    const int b = ctx->pcur;
    PArgs<T> a;
    a.pos4 = static_cast<typename P::real4 *>(pos_now(ctx));
    a.vel4 = static_cast<typename P::real4 *>(vel_now(ctx));
    a.fcons4 = static_cast<typename P::real4 *>(ctx->fcons4[b]);
    a.pid = ctx->pid[b];
    a.slot_of = ctx->slot_of;
    a.fc4 = static_cast<typename P::real4 *>(ctx->fc4[b]);
    a.old4 = static_cast<typename P::real4 *>(ctx->old4);
    a.node = static_cast<typename P::node4 *>(ctx->node);
    a.jacc = static_cast<typename P::node4 *>(ctx->jacc);
    a.bond_count = ctx->bond_count;
    a.bond_partner = ctx->bond_partner;
    a.bond_k = ctx->bond_k;
    a.bond_r0 = ctx->bond_r0;
    a.bond_kind = ctx->bond_kind;
    a.lj_eps24 = (T)(24.0 * ctx->lj_eps);
    a.lj_sig2 = (T)(ctx->lj_sigma * ctx->lj_sigma);
    a.lj_rc2 = (T)(ctx->lj_rc * ctx->lj_rc);
    {
        // |error| of an FP32 absolute coordinate <= max edge * 2^-24, of a
        // distance <= sqrt(3) * 2 of that (plus the float arithmetic); the
        // margin is a generous multiple of it
        const double edge = std::max(ctx->p.nx, std::max(ctx->p.ny, ctx->p.nz));
        const double margin = edge * std::ldexp(1.0, -18) + 1e-6;
        a.lj_filter2 = (float)((ctx->lj_rc + margin) * (ctx->lj_rc + margin));
    }
    const bool lists = ctx->lj_rc > 0.0 && ctx->nb_list;
    a.nb_list = lists ? ctx->nb_list : nullptr;
    a.nb_count = lists ? ctx->nb_count : nullptr;
    a.nb_end = lists ? ctx->nb_end : nullptr;
    a.nb_invalid = lists ? ctx->nb_invalid : nullptr;
    a.nb_ref4 = lists ? static_cast<const typename P::real4 *>(ctx->nb_ref4) : nullptr;
    a.nb_half_skin2 = (T)(0.25 * LBMD_NB_SKIN * LBMD_NB_SKIN);
    a.nx = ctx->p.nx;
    a.ny = ctx->p.ny;
    a.nz = ctx->p.nz;
    a.fd_nx = make_fastdiv((uint32_t)ctx->p.nx);
    a.fd_ny = make_fastdiv((uint32_t)ctx->p.ny);
    a.np = ctx->np;
    a.zeta = (T)ctx->p.zeta;
    a.dt = (T)ctx->dt;
    a.half_dt = (T)(0.5 * ctx->dt);
    a.amp = (T)sqrt(2.0 * ctx->p.zeta * ctx->p.kT / ctx->dt);
    a.neg_scale_dt = (T)ctx->dt * -(T)ctx->fix.scale;
    a.fis = (T)ctx->fix.inv_scale;
    a.key0 = (uint32_t)(ctx->p.seed & 0xffffffffu);
    a.key1 = (uint32_t)(ctx->p.seed >> 32);
    a.lb_step = ctx->d_lb_step;
    a.n_sub = ctx->p.n_sub;
    a.substep = substep;
    a.mig_par = (int)((ctx->lb_step * ctx->p.n_sub + substep) & 1);
    a.noisy = ctx->p.kT > 0.0 ? 1 : 0;
    a.gauss = ctx->p.noise == LBMD_NOISE_GAUSS ? 1 : 0;
    a.variant = ctx->p.variant;
    a.row_start = ctx->row_start;
    a.slot_row = ctx->slot_row;
    a.migrant_slot = ctx->migrant_slot;
    a.migrant_count = ctx->migrant_count;
    a.np_cap = ctx->p.max_particles > 0 ? ctx->p.max_particles : 1;
    a.b_atomic = 0;
    a.kick_spreads = 0;
    a.occw = active_words_now(ctx);
    a.cact = static_cast<typename P::node4 *>(active_records_now(ctx));
    a.cact_acc = static_cast<typename P::node4 *>(active_records_acc(ctx));
    a.interp_compact = ctx->p.variant != LBMD_VARIANT_A || a_copy(ctx) ? 1 : 0;
    a.inactive_acc = ctx->p.variant == LBMD_VARIANT_A ? a.jacc : a.node;
    a.occ_words = active_words(ctx->p.nx);
    return a;
}

// Whether the transfers go to the nodes with atomics (else the row gather).
static bool spreads_atomic(const lbmd_ctx *ctx) {
    return ctx->p.spread == LBMD_SPREAD_ATOMIC ||
           (ctx->p.spread == LBMD_SPREAD_AUTO &&
            // (FP64: the faster at every density; the figures stand at LBMD_SPREAD_AUTO)
            (ctx->p.precision == LBMD_FP64 || ctx->np < (int64_t)LBMD_SPREAD_ATOMIC_PER_ROW * ctx->p.ny * ctx->p.nz));
}

// `count` MD steps from `substep` on in one launch, where the system allows it.
// *done says whether it did.
template <typename T>
static cudaError_t md_phase_t(lbmd_ctx *ctx, int substep, int count, bool *done) {
    *done = true;
    if (ctx->np == 0) return cudaSuccess;
    const bool atomic = spreads_atomic(ctx);
    // Variant A without conservative forces, from two steps on; a single step
    // has nothing to keep in registers (139x146x135 nodes, 32,748 particles, m =
    // 1: 192 us a cycle against 189 with the separate kernels).  A few thousand
    // particles and less are left to the teams below: 48^3 nodes, 500
    // particles, m = 4, 30.8 us a cycle against 35.2 (FP64, 32^3, m = 5: 54.3
    // against 69.9); with 5000 particles the two are even, with 19,000 and m = 10
    // it is 49.2 against 40.2.
    const bool team_a = 8 * ctx->np <= (int64_t)128 * ctx->sm_count;
    if (ctx->p.variant == LBMD_VARIANT_A && !has_cons(ctx) && count > 1 && !team_a &&
        (atomic || ctx->p.spread == LBMD_SPREAD_AUTO)) {
        const PArgs<T> a = make_pargs<T>(ctx, substep);
        const unsigned blocks = (unsigned)((ctx->np + 127) / 128);
        if (ctx->p.integrator == LBMD_INTEGRATOR_HALF_STEP)
            frozen_phase_kernel<T, true><<<blocks, 128, 0, ctx->stream>>>(a, count);
        else
            frozen_phase_kernel<T, false><<<blocks, 128, 0, ctx->stream>>>(a, count);
        return cudaGetLastError();
    }
    // Variants B and C, conservative forces in any variant, and few particles of
    // variant A, while a team of lanes per particle fits the GPU at once.
    if ((ctx->p.spread == LBMD_SPREAD_AUTO || ctx->p.spread == LBMD_SPREAD_ATOMIC) &&
        (ctx->p.variant != LBMD_VARIANT_A || has_cons(ctx) || team_a)) {
        const bool half = ctx->p.integrator == LBMD_INTEGRATOR_HALF_STEP;
        const int cons = ctx->lj_rc > 0.0 ? 2 : has_cons(ctx) ? 1 : 0;
        const int64_t threads = ctx->np * (cons == 2 ? 32 : 8), one_block = (int64_t)PHASE_THREADS * ctx->sm_count;
        // Up to that many particles the teams are the faster, m = 10, us a cycle
        // with them / with the separate kernels: FP32 64^3 ideal 19,400 particles
        // 75.9 / 87.3, bonded 96.2 / 121.2; 4,800 Lennard-Jones beads 132 / 147;
        // FP64 ideal 9,600 204 / 245.  FP64 with conservative forces only up to one
        // block of the smaller size per SM (the larger ones put twice the FP64 work
        // on half as many SMs): bonded 4,864 particles 282 / 350, 4,900 443 / 350
        // (m = 2: 134 / 145, 166 / 146); 1,216 beads 342 / 390, 1,248 548 / 495,
        // 2,400 570 / 557.
        if (threads <= (sizeof(T) == 8 && cons ? std::min(one_block, ctx->phase_threads) : ctx->phase_threads)) {
            PArgs<T> a = make_pargs<T>(ctx, substep);
            GridBarrier words{ctx->phase_bar, ctx->dev_error, ctx->host_error, ctx->barrier_polls};
            void *args[] = {&a, &count, &words};
            // one block per SM if that takes at most twice the threads each
            const int per = threads > one_block ? 2 * PHASE_THREADS : PHASE_THREADS;
            return launch_phase(phase_kernel<T, true>(half, cons), phase_kernel<T, false>(half, cons),
                                (unsigned)((threads + per - 1) / per), per, ctx->phase_cluster, args, ctx->stream);
        }
    }
    *done = false;
    return cudaSuccess;
}

template <typename T>
static cudaError_t md_substep_t(lbmd_ctx *ctx, int substep) {
    if (ctx->np == 0) return cudaSuccess;
    PArgs<T> a = make_pargs<T>(ctx, substep);
    const unsigned blocks = (unsigned)((ctx->np + 255) / 256);
    const unsigned cblocks = (unsigned)((ctx->np + COUPLE_THREADS - 1) / COUPLE_THREADS);
    const bool cons = has_cons(ctx);
    const bool atomic = spreads_atomic(ctx);
    a.b_atomic = atomic ? 1 : 0;
    a.kick_spreads = atomic && cons ? 1 : 0;
    // the tiled step only on request: at the benchmark density it measured
    // slower than the separate particle pass and row gather
    const bool tiles = !atomic && md_tile_supported(ctx) && ctx->p.spread == LBMD_SPREAD_TILES;
    cudaError_t e;
    if (tiles) {
        // the whole MD step in one pass over tiles of rows (new positions,
        // velocities and records into the other buffers) and a short
        // follow-up (transfers across the periodic wrap, listed particles)
        if ((e = md_tile_step<T>(ctx, a)) != cudaSuccess) return e;
        ctx->pv ^= 1;
        ctx->rec ^= 1;
        return cudaSuccess;
    }
    if (ctx->p.integrator == LBMD_INTEGRATOR_HALF_STEP) {
        if (cons)
            couple_half_kernel<T, true><<<cblocks, COUPLE_THREADS, 0, ctx->stream>>>(a);
        else
            couple_half_kernel<T, false><<<cblocks, COUPLE_THREADS, 0, ctx->stream>>>(a);
    } else if (cons) {
        couple_kernel<T, true><<<cblocks, COUPLE_THREADS, 0, ctx->stream>>>(a);
    } else {
        couple_kernel<T, false><<<cblocks, COUPLE_THREADS, 0, ctx->stream>>>(a);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (cons) {
        if (ctx->lj_rc > 0.0)
            pair_kick_kernel<T, true><<<(unsigned)((ctx->np + 7) / 8), PAIR_THREADS, 0, ctx->stream>>>(a);
        else
            bond_kick_kernel<T, true><<<blocks, 256, 0, ctx->stream>>>(a);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (atomic && cons) {
        // spread by the bond / pair kernel above
    } else if (atomic) {
        if (sizeof(T) == 4)
            spread_all_kernel<T><<<(unsigned)((8 * ctx->np + 255) / 256), 256, 0, ctx->stream>>>(a);
        else
            migrant_spread_kernel<T><<<blocks, 256, 0, ctx->stream>>>(a, 1);
    } else {
        const int rows = (int)((int64_t)ctx->p.ny * ctx->p.nz);
        const int gw = ctx->gather_warps;
        const unsigned gblocks = (unsigned)((rows + gw - 1) / gw);
        spread_rows_kernel<T><<<gblocks, 32 * gw, gather_smem_bytes<T>(ctx, gw), ctx->stream>>>(a, rows);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        migrant_spread_kernel<T><<<2 * ctx->sm_count, 256, 0, ctx->stream>>>(a, 0);
    }
    return cudaGetLastError();
}

template <typename T>
static cudaError_t bond_forces_t(lbmd_ctx *ctx) {
    if (ctx->np == 0) return cudaSuccess;
    PArgs<T> a = make_pargs<T>(ctx, 0);
    const unsigned blocks = (unsigned)((ctx->np + 255) / 256);
    if (ctx->lj_rc > 0.0)
        pair_kick_kernel<T, false><<<(unsigned)((ctx->np + 7) / 8), PAIR_THREADS, 0, ctx->stream>>>(a);
    else
        bond_kick_kernel<T, false><<<blocks, 256, 0, ctx->stream>>>(a);
    return cudaGetLastError();
}

template <typename T>
static ScatterArgs<T> scatter_args(lbmd_ctx *ctx) {
    using R4 = typename Prec<T>::real4;
    const int b = ctx->pcur, o = b ^ 1;
    const int v = ctx->pv, vo = v ^ 1;  // position / velocity buffers
    ScatterArgs<T> a;
    a.pos_in = static_cast<const R4 *>(ctx->pos4[v]);
    a.vel_in = static_cast<const R4 *>(ctx->vel4[v]);
    a.fcons_in = static_cast<const R4 *>(ctx->fcons4[b]);
    a.fc_in = static_cast<const R4 *>(ctx->fc4[b]);
    a.pid_in = ctx->pid[b];
    a.pos_out = static_cast<R4 *>(ctx->pos4[vo]);
    a.vel_out = static_cast<R4 *>(ctx->vel4[vo]);
    a.fcons_out = static_cast<R4 *>(ctx->fcons4[o]);
    a.fc_out = static_cast<R4 *>(ctx->fc4[o]);
    a.pid_out = ctx->pid[o];
    a.slot_of = ctx->slot_of;
    a.slot_row = ctx->slot_row;
    a.rank = ctx->sort_rank;
    a.np = ctx->np;
    a.fnx = make_fastdiv((uint32_t)ctx->p.nx);
    a.bonds = has_cons(ctx) ? 1 : 0;
    a.carry_fc = ctx->p.integrator == LBMD_INTEGRATOR_HALF_STEP ? 1 : 0;
    return a;
}

template <typename T>
static cudaError_t sort_t(lbmd_ctx *ctx) {
    const int64_t rows = (int64_t)ctx->p.ny * ctx->p.nz;
    const int W = active_words(ctx->p.nx);
    cudaError_t e = cudaMemsetAsync(ctx->row_count, 0, (size_t)rows * sizeof(int32_t), ctx->stream);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ctx->ccw, 0, (size_t)rows * W * sizeof(uint32_t), ctx->stream)) != cudaSuccess) return e;
    const ScatterArgs<T> a = scatter_args<T>(ctx);
    const unsigned blocks = (unsigned)((ctx->np + 255) / 256);
    sort_count_kernel<T><<<blocks, 256, 0, ctx->stream>>>(a.pos_in, ctx->np, a.fnx, ctx->row_count, ctx->sort_rank,
                                                            ctx->ccw, W);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int n_chunks = (int)((rows + 1023) / 1024);
    sort_chunk_scan_kernel<<<n_chunks, 1024, 0, ctx->stream>>>(ctx->row_count, rows, ctx->chunk_total);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    sort_finalize_kernel<<<n_chunks, 1024, 0, ctx->stream>>>(ctx->row_count, ctx->chunk_total, rows, ctx->row_start,
                                                             (int32_t)ctx->np);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    sort_scatter_kernel<T><<<blocks, 256, 0, ctx->stream>>>(a, ctx->row_start);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    ctx->pcur ^= 1;
    ctx->pv ^= 1;
    return cudaSuccess;
}

template <typename T>
static cudaError_t active_set_t(lbmd_ctx *ctx) {
    const int64_t rows = (int64_t)ctx->p.ny * ctx->p.nz;
    const int W = active_words(ctx->p.nx);
    uint2 *occw = active_words_next(ctx);  // built for the coming LB cycle
    int32_t *arow = ctx->arow[(ctx->lb_step + 1) & 1];
    int L = 1;
    while (L < W && L < 32) L <<= 1;
    const int64_t warps = (rows + (32 / L) - 1) / (32 / L);
    const unsigned blocks = (unsigned)((warps + 7) / 8);
    active_rows_kernel<<<blocks, 256, 0, ctx->stream>>>(ctx->ccw, ctx->p.nx, make_fastdiv((uint32_t)ctx->p.ny),
                                                        ctx->p.nz, W, L, occw, ctx->row_count, (int)rows);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int n_chunks = (int)((rows + 1023) / 1024);
    sort_chunk_scan_kernel<<<n_chunks, 1024, 0, ctx->stream>>>(ctx->row_count, rows, ctx->chunk_total);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    active_finalize_kernel<<<dim3(n_chunks, FINALIZE_SLICES), 1024, 0, ctx->stream>>>(ctx->row_count,
                                                                                      ctx->chunk_total, rows, occw,
                                                                                      W, arow);
    return cudaGetLastError();
}

// Re-ordering and active set of the coming cycle in one launch (reorder_kernel),
// while a thread of the grid takes at most one row and 4 particles; larger
// systems take the separate kernels, which fill the GPU.  64 x 196 x 196 nodes (38,416
// rows), m = 2, us a cycle in one launch / separately, FP32: 1,000 particles
// 137 / 141, 100,000 161 / 163, 200,000 184 / 183, 300,000 204 / 200 (FP64 676 / 678,
// 745 / 746, 812 / 806, 879 / 873); 96 x 128 x 128, 150,000: 136 / 140 (575 / 578).
static bool reorder_fits(const lbmd_ctx *ctx) {
    const int64_t threads = (int64_t)ctx->sm_count * REORDER_THREADS;
    return (int64_t)ctx->p.ny * ctx->p.nz <= threads && ctx->np <= 4 * threads;
}
template <typename T>
static cudaError_t reorder_t(lbmd_ctx *ctx) {
    ScatterArgs<T> a = scatter_args<T>(ctx);
    const int rows = ctx->p.ny * ctx->p.nz;
    int W = active_words(ctx->p.nx), L = 1, nz = ctx->p.nz;
    while (L < W && L < 32) L <<= 1;
    const int64_t most = std::max<int64_t>(ctx->np, rows);
    const unsigned blocks =
        (unsigned)std::min<int64_t>(ctx->sm_count, (most + REORDER_THREADS - 1) / REORDER_THREADS);
    int per = (rows + (int)blocks - 1) / (int)blocks;
    uint2 *occw = active_words_next(ctx);
    int32_t *arow = ctx->arow[(ctx->lb_step + 1) & 1];
    FastDiv fny = make_fastdiv((uint32_t)ctx->p.ny);
    GridBarrier words{ctx->phase_bar, ctx->dev_error, ctx->host_error, ctx->barrier_polls};
    void *args[] = {&a,    &ctx->row_count, &ctx->active_count, &ctx->row_start, &ctx->ccw, &occw, &arow,
                    &ctx->lb_missed, &fny, &nz, &W, &L, &per, &words};
    const cudaError_t e = cudaLaunchCooperativeKernel((const void *)reorder_kernel<T>, dim3(blocks),
                                                      dim3(REORDER_THREADS), args, 0, ctx->stream);
    if (e != cudaSuccess) return e;
    ctx->pcur ^= 1;
    ctx->pv ^= 1;
    return cudaSuccess;
}

template <typename T>
static cudaError_t active_sync_t(lbmd_ctx *ctx) {
    using N4 = typename Prec<T>::node4;
    const unsigned blocks = (unsigned)((ctx->N + 255) / 256);
    active_sync_kernel<T><<<blocks, 256, 0, ctx->stream>>>(active_words_now(ctx),
                                                           static_cast<const N4 *>(active_records_now(ctx)),
                                                           static_cast<N4 *>(ctx->node), ctx->N, ctx->p.nx,
                                                           active_words(ctx->p.nx));
    return cudaGetLastError();
}

template <typename T>
static cudaError_t nb_build_t(lbmd_ctx *ctx) {
    if (ctx->np == 0 || !(ctx->lj_rc > 0.0) || !ctx->nb_list) return cudaSuccess;
    PArgs<T> a = make_pargs<T>(ctx, 0);
    const double rl = ctx->lj_rc + LBMD_NB_SKIN;
    nb_build_kernel<T><<<(unsigned)((ctx->np + NB_WARPS - 1) / NB_WARPS), 32 * NB_WARPS, 0, ctx->stream>>>(
        a, (T)(rl * rl), (int)std::ceil(rl));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    nb_validate_kernel<<<1, 1, 0, ctx->stream>>>(ctx->nb_invalid);
    return cudaGetLastError();
}

}  // namespace lbmd

static cudaError_t launch_sort_particles(lbmd_ctx *ctx);

// The particles in row order and the active nodes of the coming cycle; the list
// of rows the collide leaves to its follow-up emptied.
cudaError_t launch_reorder(lbmd_ctx *ctx) {
    const bool dbl = ctx->p.precision == LBMD_FP64;
    cudaError_t e;
    // without particles both sets are empty, as lbmd_create left them
    if (ctx->np == 0) return cudaMemsetAsync(ctx->lb_missed, 0, sizeof(int32_t), ctx->stream);
    if (lbmd::reorder_fits(ctx)) {
        ctx->in_buckets = true;
        if ((e = dbl ? lbmd::reorder_t<double>(ctx) : lbmd::reorder_t<float>(ctx)) != cudaSuccess) return e;
        return launch_nb_build(ctx);
    }
    if ((e = launch_sort_particles(ctx)) != cudaSuccess) return e;
    if ((e = launch_nb_build(ctx)) != cudaSuccess) return e;
    if ((e = dbl ? lbmd::active_set_t<double>(ctx) : lbmd::active_set_t<float>(ctx)) != cudaSuccess) return e;
    return cudaMemsetAsync(ctx->lb_missed, 0, sizeof(int32_t), ctx->stream);
}

cudaError_t launch_active_sync(lbmd_ctx *ctx) {
    if (ctx->p.variant == LBMD_VARIANT_A) return cudaSuccess;
    return ctx->p.precision == LBMD_FP64 ? lbmd::active_sync_t<double>(ctx) : lbmd::active_sync_t<float>(ctx);
}

cudaError_t launch_md_steps(lbmd_ctx *ctx, int substep, int count) {
    ctx->in_buckets = false;
    const bool dbl = ctx->p.precision == LBMD_FP64;
    bool done = false;
    cudaError_t e = dbl ? lbmd::md_phase_t<double>(ctx, substep, count, &done)
                        : lbmd::md_phase_t<float>(ctx, substep, count, &done);
    for (int s = 0; !done && s < count && e == cudaSuccess; ++s)
        e = dbl ? lbmd::md_substep_t<double>(ctx, substep + s) : lbmd::md_substep_t<float>(ctx, substep + s);
    return e;
}

// The conservative forces at the current positions; right after a re-ordering
// the Lennard-Jones lists are built first (they are otherwise void until the
// next LB step, and the pairs all pairs).
cudaError_t launch_bond_forces_only(lbmd_ctx *ctx) {
    if (ctx->in_buckets) {
        const cudaError_t e = launch_nb_build(ctx);
        if (e != cudaSuccess) return e;
    }
    return ctx->p.precision == LBMD_FP64 ? lbmd::bond_forces_t<double>(ctx) : lbmd::bond_forces_t<float>(ctx);
}

cudaError_t setup_particle_kernels(lbmd_ctx *ctx) {
    return ctx->p.precision == LBMD_FP64 ? lbmd::setup_t<double>(ctx) : lbmd::setup_t<float>(ctx);
}

cudaError_t launch_nb_build(lbmd_ctx *ctx) {
    return ctx->p.precision == LBMD_FP64 ? lbmd::nb_build_t<double>(ctx) : lbmd::nb_build_t<float>(ctx);
}

// The re-ordering alone; leaves the counting arrays dirty.
static cudaError_t launch_sort_particles(lbmd_ctx *ctx) {
    ctx->in_buckets = true;
    return ctx->p.precision == LBMD_FP64 ? lbmd::sort_t<double>(ctx) : lbmd::sort_t<float>(ctx);
}

// Outside the cycles (particles added, a state loaded): every particle into the
// row bucket of its cell, the counting arrays cleared for reorder_kernel.
cudaError_t launch_bucket_particles(lbmd_ctx *ctx) {
    cudaError_t e = launch_sort_particles(ctx);
    if (e != cudaSuccess) return e;
    const size_t rows = (size_t)ctx->p.ny * ctx->p.nz;
    if ((e = cudaMemsetAsync(ctx->row_count, 0, rows * sizeof(int32_t), ctx->stream)) != cudaSuccess) return e;
    return cudaMemsetAsync(ctx->ccw, 0, rows * lbmd::active_words(ctx->p.nx) * sizeof(uint32_t), ctx->stream);
}
