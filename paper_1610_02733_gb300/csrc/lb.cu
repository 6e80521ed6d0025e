// lb.cu -- the lattice Boltzmann update (Sec. 2, Eq. (3)) on the GPU.
//
// lb_collide_push: one thread per node.  Reads the 19 post-stream populations
// f*_i (coalesced structure-of-arrays loads), the momentum the particles
// handed over since the last LB step, and applies the MRT collision in moment
// space with thermal noise (Philox in registers) and the forcing term of the
// force density F = J_acc / tau_LB + g; the post-collision populations are
// pushed to the neighbours r + c_i in the other buffer.
//
// Variant C: the transfers of the MD steps enter the populations through the
// forcing part of the collision (apply_transfer), once per LB step.
//
// The post-stream moments rho* and j* of the freshly streamed populations
// (the node field the MD steps of the next LB cycle read and, in variants B and
// C, update, plus the compact record of every active node) are fused into
// lb_collide_push: a block computes them for the node row two planes back,
// once the 27 blocks around that row have pushed (per-block flags tagged with
// the LB step); moments_rest_kernel covers the rows the dataflow cannot
// reach.  node_moments_kernel computes them on their own (creation, replaced
// populations).
#include "lb_core.cuh"
#include "lb_fixed.cuh"
#include "lbmd_ctx.h"
#include "lbmd_device.cuh"

namespace lbmd {

template <typename T, typename S>
struct LbArgs {
    const S *__restrict__ fin;
    S *__restrict__ fout;
    T rho_base;  // deviation storage: sum_i of the stored rest values w_i rho0
    typename Prec<T>::node4 *node;
    typename Prec<T>::node4 *jacc;
    const uint2 *occw;                     // active nodes of this cycle
    const typename Prec<T>::node4 *cact;   // their compact records
    const uint2 *occw_new;                 // active nodes of the next cycle
    typename Prec<T>::node4 *cact_new;     // ... whose records the fused moments write
    typename Prec<T>::node4 *cact_new2;    // variant A with a frozen copy: the same records again
    int occ_words;
    // fused post-stream moments (dataflow between collide blocks)
    uint32_t *blk_done;
    int32_t *missed, *missed_list;
    int spin;  // polls of the wait for the neighbour blocks (0: every row to the fallback)
    int nx, ny, nz;
    int64_t N;
    T fs, fis;            // fixed-point scale of the momentum density and its inverse
    int32_t *range_flag;  // set when a written record reaches half the fixed-point range
    T gamma_bulk, gamma_shear, gamma_ghost;
    T amp16[Q];  // noise amplitude sqrt(mu b_k (1 - g_k^2)) times sqrt(12) 2^-16
    T ampg[Q];   // the amplitude itself (normal variates)
    T g[3];
    uint32_t key0, key1;
    const unsigned long long *lb_step;
    int noisy;
    int variant;
    FixedArgs fx;  // FP64: the integer form of the collision
};

// Range guard: a record whose momentum reaches half the fixed-point range
// raises the context's flag (the integer sums of later transfers could wrap).
template <typename T>
__device__ __forceinline__ typename Prec<T>::node4 guarded_record(const NodeSums<T> &s, int32_t *range_flag) {
    using P = Prec<T>;
    if (P::beyond_half(s.ix) | P::beyond_half(s.iy) | P::beyond_half(s.iz)) atomicOr(range_flag, 1);
    return P::pack(s.rho, s.ix, s.iy, s.iz);
}

// Post-stream moments rho*, j* (Eqs. (1), (2)) of node (x, y, t): the node
// record and, for an active node of the coming cycle, its compact record.  The populations are read through L2 (ld.global.cg): they
// were written by other blocks of the same kernel.
template <typename T, typename S>
__device__ __forceinline__ void node_moments_at(const S *f, typename Prec<T>::node4 *node, const uint2 *occw,
                                                typename Prec<T>::node4 *cact, typename Prec<T>::node4 *cact2,
                                                int occ_words, int64_t N, int nx, int ny, T rho_base, T fs, int e,
                                                int32_t *range_flag, int x, int y, int t) {
    using P = Prec<T>;
    using St = PopStore<S, T>;
    const uint32_t r = (uint32_t)x + (uint32_t)nx * ((uint32_t)y + (uint32_t)ny * (uint32_t)t);
    T fl[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) fl[i] = St::arith_cg(f + (size_t)i * N + r);
    const typename P::node4 rec = guarded_record(node_sums<St::deviation>(fl, rho_base, fs, e), range_flag);
    node[r] = rec;
    const int sl = active_slot(occw[((size_t)y + (size_t)ny * t) * occ_words + (x >> 5)], x);
    if (sl >= 0) {
        cact[sl] = rec;
        if (cact2) cact2[sl] = rec;
    }
}

// The moments of node row (block) b of the collide grid are computed, once
// its 27 neighbouring blocks (planes t - 1..t + 1) have pushed, by the block
// FUSE_LAG planes further on; rows of the first plane and of the last
// FUSE_LAG planes (whose neighbourhood wraps to later planes), and any row
// whose wait ran out, are left to moments_rest_kernel.
constexpr int FUSE_LAG = 2;
// The wait polls at most ctx->fuse_spin times (64 ns apart; default
// LBMD_DEFAULT_FUSE_SPIN, far above the few us the lag needs); a context can
// lower it (lbmd_set_moments_wait), down to 0, where every row goes to the
// fallback kernel.

// The transfer J_acc to node (x, y, z) since the last LB step.  A record's
// j = fix(j*) + sum of fixed-point transfers: the difference is exactly the
// accumulated transfer (an active node's record is its compact one -- variant
// A: the accumulating copy; B and C: an inactive node's is the node field).
// Variant A, inactive node: J_acc holds what was handed over there (rarely
// anything; cleared only where set).
//
// FP32 arithmetic, as the real force of a node with momentum (jx, jy, jz): the
// integers are converted at once (kept as integers beside the sums they cost
// the kernel 8 bytes more of spills and 1.6 % of the cycle).
template <typename T, typename S, bool C>
__device__ __forceinline__ void node_force(const LbArgs<T, S> &a, uint32_t r, int x, int y, int z, T jx, T jy, T jz,
                                           T &Fx, T &Fy, T &Fz) {
    using P = Prec<T>;
    const int sl = active_slot(a.occw[((size_t)y + (size_t)a.ny * z) * a.occ_words + (x >> 5)], x);
    if (C || sl >= 0 || a.variant == LBMD_VARIANT_B) {
        const typename P::node4 n = sl >= 0 ? a.cact[sl] : a.node[r];
        Fx = P::from_fix(P::jx_of(n) - P::to_fix(jx, a.fs), a.fis);
        Fy = P::from_fix(P::jy_of(n) - P::to_fix(jy, a.fs), a.fis);
        Fz = P::from_fix(P::jz_of(n) - P::to_fix(jz, a.fs), a.fis);
    } else {
        const typename P::node4 J = a.jacc[r];
        Fx = P::from_fix(P::jx_of(J), a.fis);
        Fy = P::from_fix(P::jy_of(J), a.fis);
        Fz = P::from_fix(P::jz_of(J), a.fis);
        if ((P::jx_of(J) | P::jy_of(J) | P::jz_of(J)) != 0) {
            typename P::node4 zero;
            zero.x = zero.y = zero.z = zero.w = 0;
            a.jacc[r] = zero;
        }
    }
}

// FP64: the integers themselves; ix, iy, iz are fix(j*).
template <bool C>
__device__ __forceinline__ void node_transfer(const LbArgs<double, double> &a, uint32_t r, int x, int y, int z,
                                              long long ix, long long iy, long long iz, long long J[3]) {
    const int sl = active_slot(a.occw[((size_t)y + (size_t)a.ny * z) * a.occ_words + (x >> 5)], x);
    if (C || sl >= 0 || a.variant == LBMD_VARIANT_B) {
        const L4 n = sl >= 0 ? a.cact[sl] : a.node[r];
        J[0] = n.y - ix;
        J[1] = n.z - iy;
        J[2] = n.w - iz;
    } else {
        const L4 n = a.jacc[r];
        J[0] = n.y;
        J[1] = n.z;
        J[2] = n.w;
        if ((J[0] | J[1] | J[2]) != 0) a.jacc[r] = L4{0, 0, 0, 0};
    }
}

// FP64 form: f -> the post-collision populations, for the transfer J.
template <bool RELAX_FULL, bool GAUSS, bool C>
__device__ __forceinline__ void collide_with_transfer(const LbArgs<double, double> &a, double f[Q], NodeSums<double> s,
                                                      const long long J[3], uint32_t r, uint32_t step) {
    using P = Prec<double>;
    double Fx = P::from_fix(J[0], a.fis), Fy = P::from_fix(J[1], a.fis), Fz = P::from_fix(J[2], a.fis);
    if (C && !(Fx == 0.0 && Fy == 0.0 && Fz == 0.0)) {
        apply_transfer(f, s.rho, s.jx, s.jy, s.jz, Fx, Fy, Fz, a.gamma_bulk, a.gamma_shear);
        pop_moments<false>(f, 0.0, s.rho, s.rho_m, s.jx, s.jy, s.jz);
        Fx = Fy = Fz = 0.0;
    }
    collide<double, RELAX_FULL, LbArgs<double, double>, GAUSS>(f, s.rho, s.rho_m, s.jx, s.jy, s.jz, Fx + a.g[0],
                                                               Fy + a.g[1], Fz + a.g[2], a, a.key0, a.key1, r, step);
}

// The FP64 form of the collision for a node outside the integer form's range
// (out of line: kept off the common path); out gets the new populations.
template <bool GAUSS, bool C>
__device__ __noinline__ void collide_fp64_out(const LbArgs<double, double> &a, uint32_t r, uint32_t step, long long Jx,
                                              long long Jy, long long Jz, double *out) {
    double f[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = a.fin[(size_t)i * a.N + r];
    NodeSums<double> s;
    pop_moments<false>(f, 0.0, s.rho, s.rho_m, s.jx, s.jy, s.jz);
    const long long J[3] = {Jx, Jy, Jz};
    collide_with_transfer<true, GAUSS, C>(a, f, s, J, r, step);
#pragma unroll
    for (int i = 0; i < Q; ++i) out[i] = f[i];
}
template <bool GAUSS, bool C>
__device__ __forceinline__ void collide_node_fp64(const LbArgs<double, double> &a, uint32_t r, uint32_t step,
                                                  const long long J[3], double f[Q]) {
    double out[Q];
    collide_fp64_out<GAUSS, C>(a, r, step, J[0], J[1], J[2], out);
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = out[i];
}

// The noise numbers of a node's 15 modes for collide_fixed, as collide() draws
// them.
template <bool GAUSS>
struct FluidNoise {
    uint32_t w[8];
    __device__ __forceinline__ FluidNoise(const LbArgs<double, double> &a, uint32_t node, uint32_t step) {
        if (!a.noisy) return;
#pragma unroll
        for (uint32_t q = 0; q < 2; ++q) {
            const U4 v = philox4x32_10(U4{node, step, 0u, q}, a.key0, a.key1);
            w[4 * q] = v.x;
            w[4 * q + 1] = v.y;
            w[4 * q + 2] = v.z;
            w[4 * q + 3] = v.w;
        }
    }
    __device__ __forceinline__ uint32_t bits(int k) const {
        const int t = k - 4;
        return (t & 1) ? w[t >> 1] >> 16 : w[t >> 1] & 0xffffu;
    }
    __device__ __forceinline__ double normal(int) const { return 0.0; }
};
template <>
struct FluidNoise<true> {
    double g[16];
    __device__ __forceinline__ FluidNoise(const LbArgs<double, double> &a, uint32_t node, uint32_t step) {
        if (!a.noisy) return;
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q) {
            const U4 v = philox4x32_10(U4{node, step, 0u, q}, a.key0, a.key1);
            box_muller(v.x, v.y, g[4 * q], g[4 * q + 1]);
            box_muller(v.z, v.w, g[4 * q + 2], g[4 * q + 3]);
        }
#pragma unroll
        for (int k = 4; k < Q; ++k) g[k - 4] *= a.ampg[k];
    }
    __device__ __forceinline__ uint32_t bits(int) const { return 0u; }
    __device__ __forceinline__ double normal(int k) const { return g[k - 4]; }
};

// One thread per node; grid (ceil(nx / blockDim.x), ny, nz).  The variant is
// a run-time (warp-uniform) flag rather than a template parameter: both
// variants then execute one compiled instruction sequence, so at m = 1 they
// agree bit for bit, as the paper's algorithmic equivalence requires.
// Collide node (x, y, z) and push its post-collision populations to the
// neighbours r + c_i in the other buffer.
// C (variant C, a kernel instance of its own): the cycle's transfers enter the
// populations first, then the collision sees the body force only.
template <typename T, typename S, bool RELAX_FULL, bool GAUSS, bool C>
__device__ __forceinline__ void collide_push_node(const LbArgs<T, S> &a, int x, int y, int z,
                                                  unsigned long long step) {
    using P = Prec<T>;
    using St = PopStore<S, T>;
    const uint32_t r = (uint32_t)x + (uint32_t)a.nx * ((uint32_t)y + (uint32_t)a.ny * (uint32_t)z);
    T f[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = St::arith(a.fin + (size_t)i * a.N + r);
    if constexpr (sizeof(T) == 8) {
        typename P::fix J[3];
        FixedMoments o;
        bool done = RELAX_FULL && a.fx.usable && fixed_moments_in_range(f, a.fx.e, o);
        if (RELAX_FULL && done) {
            node_transfer<C>(a, r, x, y, z, record_momentum(o.j[0]), record_momentum(o.j[1]), record_momentum(o.j[2]),
                             J);
            const FluidNoise<GAUSS> noise(a, r, (uint32_t)step);
            done = collide_fixed<C, GAUSS>(o, J, a.gamma_shear, a.g, a.fx, a.noisy != 0, noise, f);
            if (!done) collide_node_fp64<GAUSS, C>(a, r, (uint32_t)step, J, f);
        } else {
            const NodeSums<T> s = node_sums<false>(f, T(0), a.fs, a.fx.e);
            node_transfer<C>(a, r, x, y, z, s.ix, s.iy, s.iz, J);
            if (RELAX_FULL)
                collide_node_fp64<GAUSS, C>(a, r, (uint32_t)step, J, f);
            else
                collide_with_transfer<RELAX_FULL, GAUSS, C>(a, f, s, J, r, (uint32_t)step);
        }
    } else {
        T rho, rho_m, jx, jy, jz;
        pop_moments<St::deviation>(f, a.rho_base, rho, rho_m, jx, jy, jz);
        T Fx, Fy, Fz;
        node_force<T, S, C>(a, r, x, y, z, jx, jy, jz, Fx, Fy, Fz);
        if (C && !(Fx == T(0) && Fy == T(0) && Fz == T(0))) {
            apply_transfer(f, rho, jx, jy, jz, Fx, Fy, Fz, a.gamma_bulk, a.gamma_shear);
            pop_moments<St::deviation>(f, a.rho_base, rho, rho_m, jx, jy, jz);
            Fx = Fy = Fz = T(0);
        }
        Fx += a.g[0];
        Fy += a.g[1];
        Fz += a.g[2];
        collide<T, RELAX_FULL, LbArgs<T, S>, GAUSS>(f, rho, rho_m, jx, jy, jz, Fx, Fy, Fz, a, a.key0, a.key1, r,
                                                    (uint32_t)step);
    }

    const int xm = x == 0 ? a.nx - 1 : x - 1, xp = x == a.nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? a.ny - 1 : y - 1, yp = y == a.ny - 1 ? 0 : y + 1;
    const int zm = z == 0 ? a.nz - 1 : z - 1, zp = z == a.nz - 1 ? 0 : z + 1;
    const int X[3] = {xm, x, xp}, Y[3] = {ym, y, yp}, Z[3] = {zm, z, zp};
    if constexpr (St::stochastic) {
        // stochastic rounding of the stored deviations: 16 random bits per
        // population from Philox stream 2 of (node, LB step), population i
        // from call i / 8, word (i / 2) mod 4, low half for even i
        U4 rb{0u, 0u, 0u, 0u};
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            if ((i & 7) == 0) rb = philox4x32_10(U4{r, (uint32_t)step, 2u, (uint32_t)(i >> 3)}, a.key0, a.key1);
            const uint32_t w = ((i >> 1) & 3) == 0 ? rb.x : ((i >> 1) & 3) == 1 ? rb.y : ((i >> 1) & 3) == 2 ? rb.z : rb.w;
            const uint32_t t = (uint32_t)X[CX(i) + 1] +
                               (uint32_t)a.nx * ((uint32_t)Y[CY(i) + 1] + (uint32_t)a.ny * (uint32_t)Z[CZ(i) + 1]);
            St::store_arith_sr(a.fout + (size_t)i * a.N + t, f[i], (i & 1) ? w >> 16 : w & 0xffffu);
        }
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const uint32_t t = (uint32_t)X[CX(i) + 1] +
                               (uint32_t)a.nx * ((uint32_t)Y[CY(i) + 1] + (uint32_t)a.ny * (uint32_t)Z[CZ(i) + 1]);
            St::store_arith(a.fout + (size_t)i * a.N + t, f[i]);
        }
    }
}

// Resident blocks per SM the compiler plans registers for.  FP32 storage: 6 (40
// registers; two cycles at 256^3 with 10^6 particles 3341 us, 5 blocks 3406,
// 7 blocks, with spills, 3425).  Rounded-to-nearest 16-bit storage with full
// relaxation and uniform noise: 7 (3183 us, 6 blocks 3287); the stochastic
// rounding form measured slower at 7.  Variant C 5.  FP64: 2 with the
// collision in integers (128 registers), 3 in its FP64 form.
template <typename T, typename S, bool RELAX_FULL, bool GAUSS, bool C>
constexpr int collide_min_blocks() {
    return sizeof(T) == 8                                                              ? (RELAX_FULL ? 2 : 3)
           : C                                                                         ? 5
           : RELAX_FULL && PopStore<S, T>::deviation && !PopStore<S, T>::stochastic ? 7
                                                                                       : 6;
}

template <typename T, typename S, bool RELAX_FULL, bool GAUSS, bool C>
__global__ void __launch_bounds__(256, (collide_min_blocks<T, S, RELAX_FULL, GAUSS, C>()))
    lb_collide_push(const __grid_constant__ LbArgs<T, S> a) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y, z = blockIdx.z;
    // the step counter, read before the fallback kernel advances it; it also
    // tags the blocks that have pushed
    const unsigned long long step = *a.lb_step;
    if (x < a.nx) collide_push_node<T, S, RELAX_FULL, GAUSS, C>(a, x, y, z, step);

    // fused post-stream moments: publish this block, then compute the
    // moments of the block FUSE_LAG planes back once its neighbourhood is in
    const uint32_t gx = gridDim.x, gy = gridDim.y;
    const uint32_t epoch = (uint32_t)step + 1u;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicExch(&a.blk_done[blockIdx.x + gx * (blockIdx.y + gy * blockIdx.z)], epoch);
    }
    const int t = z - FUSE_LAG;
    if (t < 1) return;
    __shared__ int s_ok;
    if (threadIdx.x < 32) {
        bool ok = a.spin > 0;
        if (ok && threadIdx.x < 27) {
            const int dx = (int)threadIdx.x % 3 - 1, dy = ((int)threadIdx.x / 3) % 3 - 1;
            const int dz = (int)threadIdx.x / 9 - 1;
            const uint32_t xb = (blockIdx.x + gx + dx) % gx, yb = (uint32_t)((y + a.ny + dy) % a.ny);
            const volatile uint32_t *flag = a.blk_done + xb + gx * (yb + gy * (uint32_t)(t + dz));
            int polls = 0;
            while (*flag != epoch) {
                if (++polls > a.spin) {
                    ok = false;
                    break;
                }
                __nanosleep(64);
            }
        }
        ok = __all_sync(0xffffffffu, ok);
        if (threadIdx.x == 0) {
            __threadfence();
            s_ok = ok ? 1 : 0;
        }
    }
    __syncthreads();
    if (!s_ok) {
        if (threadIdx.x == 0) a.missed_list[atomicAdd(a.missed, 1)] = (int32_t)(blockIdx.x + gx * (y + gy * t));
        return;
    }
    if (x < a.nx)
        node_moments_at<T, S>(a.fout, a.node, a.occw_new, a.cact_new, a.cact_new2, a.occ_words, a.N, a.nx, a.ny,
                              a.rho_base, a.fs, a.fx.e, a.range_flag, x, y, t);
}

// The moments the collide kernel left: node rows of plane 0 and of the last
// FUSE_LAG planes, and the rows whose wait ran out (counted into
// missed_total, `pieces` for a block); then the LB step counter advances.
template <typename T, typename S>
__global__ void __launch_bounds__(256)
    moments_rest_kernel(const S *__restrict__ f, typename Prec<T>::node4 *node, const uint2 *occw,
                        typename Prec<T>::node4 *cact, typename Prec<T>::node4 *cact2, int occ_words, int64_t N,
                        int nx, int ny, int nz, T rho_base, T fs, int e, int32_t *range_flag, const int32_t *missed,
                        const int32_t *missed_list,
                        unsigned long long *missed_total, int pieces, unsigned long long *lb_step) {
    const int gx = (nx + (int)blockDim.x - 1) / (int)blockDim.x;
    const int rows = gx * ny;
    // boundary planes: 0 and max(1, nz - FUSE_LAG) .. nz - 1
    const int first_tail = nz - FUSE_LAG > 1 ? nz - FUSE_LAG : 1;
    const int n_planes = 1 + (nz - first_tail);
    const int n_boundary = n_planes * rows;
    const int total = n_boundary + *missed;
    for (int i = blockIdx.x; i < total; i += gridDim.x) {
        int b;
        if (i < n_boundary) {
            const int k = i / rows;
            const int plane = k == 0 ? 0 : first_tail + (k - 1);
            b = i - k * rows + plane * rows;
        } else {
            b = missed_list[i - n_boundary];
        }
        const int xb = b % gx, rest = b / gx, y = rest % ny, t = rest / ny;
        const int x = xb * (int)blockDim.x + (int)threadIdx.x;
        if (x < nx)
            node_moments_at<T, S>(f, node, occw, cact, cact2, occ_words, N, nx, ny, rho_base, fs, e, range_flag, x, y,
                                  t);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *missed_total += (unsigned long long)*missed * (unsigned)pieces;
        *lb_step += 1ull;
    }
}

template <typename T, typename S>
__global__ void __launch_bounds__(256)
    node_moments_kernel(const S *__restrict__ f, typename Prec<T>::node4 *node, const uint2 *occw,
                        typename Prec<T>::node4 *cact, typename Prec<T>::node4 *cact2, int occ_words, int64_t N,
                        int nx, int ny, T rho_base, T fs, int e, int32_t *range_flag) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= nx) return;
    node_moments_at<T, S>(f, node, occw, cact, cact2, occ_words, N, nx, ny, rho_base, fs, e, range_flag, x, blockIdx.y,
                          blockIdx.z);
}

template <typename T, typename S>
__global__ void init_equilibrium_kernel(S *f, int64_t N, T rho0) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= N) return;
#pragma unroll
    for (int i = 0; i < Q; ++i) PopStore<S, T>::store(f + (int64_t)i * N + r, T(WEIGHT(i)) * rho0, T(WEIGHT(i)) * rho0);
}

// Node kernels run one thread per node on a (x-blocks, ny, nz) grid: a row of up
// to 256 nodes is one block, rounded up to a power of two.  Two blocks of half
// that have as many threads, and twice the flags to set and to wait for: two
// cycles at 96 x 80 x 112 nodes (51,200 particles, variant C, m = 5) 249.6 us
// with blocks of 64, 239.6 with 128; 250 x 201 x 181 (545,000, variant A) 1153.6
// with 128, 1150.3 with 256.
static dim3 node_block(const lbmd_ctx *ctx) {
    const int bx = ctx->p.nx > 128 ? 256 : (ctx->p.nx > 64 ? 128 : (ctx->p.nx > 32 ? 64 : 32));
    return dim3(bx, 1, 1);
}
static dim3 node_grid(const lbmd_ctx *ctx, dim3 block) {
    return dim3((ctx->p.nx + block.x - 1) / block.x, ctx->p.ny, ctx->p.nz);
}

// Normal variates and variant C are kernel instances of their own, so that
// the default one keeps its registers; neither combines with the storage
// forms that lbmd_create refuses them for.
template <typename T, typename S, bool FULL>
static void launch_collide(lbmd_ctx *ctx, const LbArgs<T, S> &a, dim3 grid, dim3 block) {
    const bool gauss = ctx->p.noise == LBMD_NOISE_GAUSS, c = ctx->p.variant == LBMD_VARIANT_C;
    cudaStream_t st = ctx->stream;
    if constexpr (!PopStore<S, T>::deviation) {
        if (gauss && c) return lb_collide_push<T, S, FULL, true, true><<<grid, block, 0, st>>>(a);
        if (gauss) return lb_collide_push<T, S, FULL, true, false><<<grid, block, 0, st>>>(a);
    }
    if constexpr (!PopStore<S, T>::stochastic) {
        if (c) return lb_collide_push<T, S, FULL, false, true><<<grid, block, 0, st>>>(a);
    }
    lb_collide_push<T, S, FULL, false, false><<<grid, block, 0, st>>>(a);
}

template <typename T, typename S>
static cudaError_t lb_step_t(lbmd_ctx *ctx) {
    LbArgs<T, S> a;
    a.fin = static_cast<const S *>(ctx->f[ctx->cur]);
    a.fout = static_cast<S *>(ctx->f[ctx->cur ^ 1]);
    a.rho_base = rest_density<T, S>(ctx);
    a.node = static_cast<typename Prec<T>::node4 *>(ctx->node);
    a.jacc = static_cast<typename Prec<T>::node4 *>(ctx->jacc);
    a.occw = active_words_now(ctx);
    a.cact = static_cast<const typename Prec<T>::node4 *>(active_records_acc(ctx));
    a.occw_new = active_words_next(ctx);
    a.cact_new = static_cast<typename Prec<T>::node4 *>(active_records_next(ctx));
    a.cact_new2 = static_cast<typename Prec<T>::node4 *>(active_records_copy(ctx, (int)((ctx->lb_step + 1) & 1)));
    a.occ_words = active_words(ctx->p.nx);
    a.blk_done = ctx->blk_done;
    a.missed = ctx->lb_missed;
    a.missed_list = ctx->missed_list;
    a.spin = ctx->fuse_spin;
    a.fs = (T)ctx->fix.scale;
    a.fis = (T)ctx->fix.inv_scale;
    a.range_flag = ctx->range_flag;
    a.nx = ctx->p.nx;
    a.ny = ctx->p.ny;
    a.nz = ctx->p.nz;
    a.N = ctx->N;
    a.gamma_bulk = (T)ctx->co.gamma_bulk;
    a.gamma_shear = (T)ctx->co.gamma_shear;
    a.gamma_ghost = (T)ctx->co.gamma_ghost;
    for (int k = 0; k < Q; ++k) {
        a.amp16[k] = (T)(ctx->co.noise_amp[k] * 3.4641016151377544 * 1.52587890625e-05);
        a.ampg[k] = (T)ctx->co.noise_amp[k];
    }
    for (int d = 0; d < 3; ++d) a.g[d] = (T)ctx->co.body_force[d];
    a.key0 = (uint32_t)(ctx->p.seed & 0xffffffffu);
    a.key1 = (uint32_t)(ctx->p.seed >> 32);
    a.lb_step = ctx->d_lb_step;
    a.noisy = ctx->co.noisy;
    a.fx = fixed_constants(ctx->fix.e, ctx->co.noise_amp, ctx->co.body_force);
    a.variant = ctx->p.variant;
    const dim3 block = node_block(ctx), grid = node_grid(ctx, block);
    cudaError_t e;
    const bool full = ctx->co.gamma_bulk == 0.0 && ctx->co.gamma_ghost == 0.0;
    if (full)
        launch_collide<T, S, true>(ctx, a, grid, block);
    else
        launch_collide<T, S, false>(ctx, a, grid, block);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // the moments the collide kernel left, on the new populations (the count of
    // missed rows is in pieces of 256, 128, 64 or 32 nodes, the largest that nx fills)
    const int piece = ctx->p.nx >= 256 ? 256 : ctx->p.nx >= 128 ? 128 : ctx->p.nx >= 64 ? 64 : 32;
    const int pieces = (ctx->p.nx + piece - 1) / piece / (int)grid.x;
    moments_rest_kernel<T, S><<<2 * ctx->sm_count, block, 0, ctx->stream>>>(
        a.fout, a.node, a.occw_new, a.cact_new, a.cact_new2, a.occ_words, ctx->N, ctx->p.nx, ctx->p.ny, ctx->p.nz,
        a.rho_base,
        a.fs, ctx->fix.e, ctx->range_flag, ctx->lb_missed, ctx->missed_list, ctx->missed_total, pieces,
        ctx->d_lb_step);
    return cudaGetLastError();
}

// node field (and the current active nodes' records) of the current
// populations, outside the LB step (creation, replaced populations)
template <typename T, typename S>
static cudaError_t node_moments_t(lbmd_ctx *ctx) {
    const dim3 block = node_block(ctx), grid = node_grid(ctx, block);
    node_moments_kernel<T, S><<<grid, block, 0, ctx->stream>>>(
        static_cast<const S *>(ctx->f[ctx->cur]), static_cast<typename Prec<T>::node4 *>(ctx->node),
        active_words_now(ctx), static_cast<typename Prec<T>::node4 *>(active_records_now(ctx)),
        static_cast<typename Prec<T>::node4 *>(active_records_copy(ctx, (int)(ctx->lb_step & 1))),
        active_words(ctx->p.nx), ctx->N, ctx->p.nx, ctx->p.ny, rest_density<T, S>(ctx), (T)ctx->fix.scale,
        ctx->fix.e, ctx->range_flag);
    return cudaGetLastError();
}

template <typename T, typename S>
static cudaError_t init_equilibrium_t(lbmd_ctx *ctx) {
    const unsigned blocks = (unsigned)((ctx->N + 255) / 256);
    init_equilibrium_kernel<T, S><<<blocks, 256, 0, ctx->stream>>>(static_cast<S *>(ctx->f[ctx->cur]), ctx->N,
                                                                    (T)ctx->p.rho0);
    return cudaGetLastError();
}

}  // namespace lbmd

// population storage per precision: FP32 and FP64 plain, FP16 / BF16 as
// deviations with FP32 arithmetic
#define LBMD_DISPATCH_POPS(ctx, FN, ...)                                                      \
    ((ctx)->p.precision == LBMD_FP64          ? FN<double, double>(__VA_ARGS__)               \
     : (ctx)->p.precision == LBMD_FP16_DEV    ? FN<float, __half>(__VA_ARGS__)                \
     : (ctx)->p.precision == LBMD_BF16_DEV    ? FN<float, __nv_bfloat16>(__VA_ARGS__)         \
     : (ctx)->p.precision == LBMD_FP16_DEV_SR ? FN<float, lbmd::half_sr>(__VA_ARGS__)         \
     : (ctx)->p.precision == LBMD_BF16_DEV_SR ? FN<float, lbmd::bf16_sr>(__VA_ARGS__)         \
                                              : FN<float, float>(__VA_ARGS__))

// One LB update: re-order the particles by row and build the active nodes of
// the coming cycle (the particles do not move during the LB step), then collide and stream with the post-stream moments fused in
// (node field and the new active nodes' compact records).
cudaError_t launch_lb_step(lbmd_ctx *ctx) {
    cudaError_t e = launch_reorder(ctx);
    if (e != cudaSuccess) return e;
    if ((e = md_tile_build_table(ctx, (int)((ctx->lb_step + 1) & 1))) != cudaSuccess) return e;
    if ((e = LBMD_DISPATCH_POPS(ctx, lbmd::lb_step_t, ctx)) != cudaSuccess) return e;
    ctx->cur ^= 1;
    ctx->rec = 0;  // the moments wrote the next set's first record buffer
    return cudaSuccess;
}

cudaError_t launch_node_moments(lbmd_ctx *ctx, bool) { return LBMD_DISPATCH_POPS(ctx, lbmd::node_moments_t, ctx); }

cudaError_t launch_init_equilibrium(lbmd_ctx *ctx) { return LBMD_DISPATCH_POPS(ctx, lbmd::init_equilibrium_t, ctx); }
