// AA-pattern stream-collide: one lattice A updated in place.
//
// The fused update of Sec. 2 needs two grids when populations move to their
// neighbours in every step. The AA pattern (Bailey et al., 2009) alternates
// two kinds of step on one lattice instead, each moving the same bytes as a
// two-grid step. Two layouts of the pre-collision state f^n alternate:
//   natural (before an even step): slot i of cell x holds f^n_i(x);
//   swapped (before an odd step):  slot opp(i) of x holds P^{n-1}_i(x), the
//     post-collision value of the even step, so f^n_i(x) is slot opp(i) of
//     x - e_i if that cell is fluid, else slot i of x itself (halfway
//     bounce-back, plus the moving-wall term).
// Even step: cell x reads slot i of x, collides, and writes P_i(x) to slot
// opp(i) of x; no neighbour is touched. Odd step: cell x gathers from the
// swapped layout, collides, and writes P_i(x) to slot i of x + e_i (where the
// next even step reads f_i(x + e_i)); if x + e_i is solid, the bounced value
// goes to slot opp(i) of x instead. In both steps a fluid cell writes the
// slots it read, each read before it is written by the same thread, and (the
// odd step's mask-free scatter) solid slots that no one reads, so the
// in-place update has no races (and the read-only load path is safe: no
// fluid cell reads a slot after it is written within a launch).
//
// Halfway bounce-back needs only the odd step: where x - e_j is solid (bit
// opp(j) of the push mask, i.e. x + e_opp(j) is solid too) population j is
// read from slot j of x itself, and population opp(j) is written back there.
// Solid cells' values are never used; the even step stores their lanes with
// the rest of the pair (whole 32-byte sectors). The odd step (aa_odd_pair) lets
// every lane load values it discards (a solid lane slots that a neighbour may be
// rewriting) and lets fluid cells store into solid slots that no one reads.
#pragma once

#include "lbm_kernels.cuh"

namespace lbm {

// Live lanes of the pair (x0, x0 + 1): fluid and inside the row.
template <bool FLAGS>
__device__ __forceinline__ void pair_live(const Dev &d, int c, bool has1, bool &live0, bool &live1) {
    live0 = true;
    live1 = has1;
    if (FLAGS) {
        const uchar2 fl = __ldg(reinterpret_cast<const uchar2 *>(d.flags + c));
        live0 = !fl.x;
        live1 = has1 && !fl.y;
    }
}

template <class R, int FORCE, bool TFORM>
__device__ __forceinline__ void pair_force(const Dev &d, int c, typename Pair2<R>::V &Fx, typename Pair2<R>::V &Fy,
                                           typename Pair2<R>::V &Fz, Guo2<R> &G) {
    Fx = Fy = Fz = vsplat(R(0));
    if (FORCE == 1) {
        Fx = vsplat(DevR<R>::F(d, 0));
        Fy = vsplat(DevR<R>::F(d, 1));
        Fz = vsplat(DevR<R>::F(d, 2));
        if constexpr (sizeof(R) == 4) G = uniform_guo<R, TFORM>(d);
    } else if (FORCE == 2) {
        const R *F = static_cast<const R *>(d.Ffield);
        ld2_real(F + c, Fx.x, Fx.y);
        ld2_real(F + d.g.qs + c, Fy.x, Fy.y);
        ld2_real(F + 2 * d.g.qs + c, Fz.x, Fz.y);
        if constexpr (sizeof(R) == 4) G = guo2<R>(TFORM ? DevR<R>::cs(d) : R(1) - R(0.5) * DevR<R>::omega(d), Fx, Fy, Fz);
    }
}

template <class R, bool RECORD>
__device__ __forceinline__ void pair_check_record(const Dev &d, int c, bool live0, bool live1, const Mom2<R> &m,
                                                  R *tape) {
    const bool bad0 = live0 && !(m.rho.x > R(0) && m.rho.x < R(1e30));
    const bool bad1 = live1 && !(m.rho.y > R(0) && m.rho.y < R(1e30));
    if (bad0 || bad1) atomicOr(d.status, LBM_STATUS_DIVERGED);
    if (RECORD) {
        const long long qs = d.g.qs;
        st2_real(tape + c, m.rho.x, m.rho.y);
        st2_real(tape + qs + c, m.ux.x, m.ux.y);
        st2_real(tape + 2 * qs + c, m.uy.x, m.uy.y);
        st2_real(tape + 3 * qs + c, m.uz.x, m.uz.y);
    }
}

// The AA kernels are launched as programmatic dependents of the step before them
// (see k_step): wait for it to complete, then let the next one be scheduled.
__device__ __forceinline__ void aa_dependent() {
    if (STEP_PDL) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
}

// Even step (natural -> swapped): local, every access an aligned pair; the flat
// launch (whole rows: FP16 channel 76.9 us, mean with the odd step, against 75.6).
// RED: also hand out the pair's pre-collision totals.
template <int S, bool FLAGS, int FORCE, bool RECORD, bool RED>
__device__ __forceinline__ void aa_even_pair(const Dev &d, typename Stor<S>::T *__restrict__ A,
                                             typename Stor<S>::R *__restrict__ tape,
                                             PairTotals<typename Stor<S>::R> *tot) {
    typedef typename Stor<S>::R R;
    typedef typename Pair2<R>::V V;
    int x0, y, z;
    // alternating plane order (see k_step) on walled lattices only: without
    // flags the 16-bit forms spill 16 more bytes at 64 registers for it (the
    // 512^3 box lost 2.4%, and a lattice that size keeps no plane in L2)
    const int bz = FLAGS && d.zrev ? (int)gridDim.y - 1 - (int)blockIdx.y : (int)blockIdx.y;
    if (!pair_cell<true>(d.g, d.PF, blockDim.x, blockDim.y, blockIdx.x, bz, threadIdx.x, threadIdx.y, x0, y, z))
        return;
    const long long qs = d.g.qs;
    const int c = cell_index(d.g, x0, y, z);
    bool live0, live1;
    pair_live<FLAGS>(d, c, x0 + 1 < d.g.nx, live0, live1);
    // (solid cells load, collide and store like the others: an early exit on
    // the flags would put a dependent load before the gather)
    const R nan = quiet_nan<R>();
    V s[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) Stor<S>::ld2(A + (long long)i * qs + c, s[i].x, s[i].y);
    V Fx, Fy, Fz;
    Guo2<R> G;
    pair_force<R, FORCE, relax_about_t(S)>(d, c, Fx, Fy, Fz, G);
    Mom2<R> m;
    if constexpr (S == LBM_F64)
        m = pair64<FORCE != 0, true, RECORD || RED>(d, s, Fx, Fy, Fz, live0, live1);
    else
        m = moments2<R, FORCE != 0>(s, Fx, Fy, Fz, d.incomp);
    if (RED) tot->set(m, live0, live1);
    pair_check_record<R, RECORD>(d, c, live0, live1, m, tape);
    if constexpr (S != LBM_F64)
        collide2<R, FORCE != 0, relax_about_t(S)>(s, m, DevR<R>::omega(d), DevR<R>::cs(d), Fx, Fy, Fz, G, d.incomp);
    // a solid lane writes its NaN back (its slots stay marked). FP32: a
    // 32-byte sector whose 8 cells are all solid skips its stores instead (as
    // in the two-grid step: no reader takes a solid slot's value), found by
    // one ballot over the sector's four pairs on lanes 4k .. 4k + 3
    bool skip = false;
    if constexpr (FLAGS && S == LBM_F32) {
        if ((d.g.pitch & 7) == 0 && (((d.g.nx + 1) / 2) & 3) == 0) {
            const unsigned sb = __ballot_sync(__activemask(), !live0 && !live1);
            skip = ((sb >> ((threadIdx.x & 31) & ~3u)) & 0xFu) == 0xFu;
        }
    }
    if (!skip) {
#pragma unroll
        for (int i = 0; i < Q; ++i)
            Stor<S>::st2(A + (long long)opp(i) * qs + c, !FLAGS || live0 ? s[i].x : nan,
                         !FLAGS || live1 ? s[i].y : nan);
    }
}

template <int S, bool FLAGS, int FORCE, bool RECORD>
__global__ void __launch_bounds__(128, 2 * StepBlocks<S>::value)
    k_aa_even(const Dev d, typename Stor<S>::T *__restrict__ A, typename Stor<S>::R *__restrict__ tape) {
    aa_dependent();
    aa_even_pair<S, FLAGS, FORCE, RECORD, false>(d, A, tape, nullptr);
}

// The even step with the totals of its pre-collision state summed per block
// (every thread, in the lattice or not, reaches the block sum).
template <int S, bool FLAGS, int FORCE>
__global__ void __launch_bounds__(128, 2 * StepBlocks<S>::value)
    k_aa_even_reduce(const Dev d, typename Stor<S>::T *__restrict__ A, double *__restrict__ partials) {
    aa_dependent();
    PairTotals<typename Stor<S>::R> tot;
    tot.clear();
    aa_even_pair<S, FLAGS, FORCE, false, true>(d, A, nullptr, &tot);
    block_partials(tot, partials, blockIdx.y * gridDim.x + blockIdx.x);
}

// Odd step (swapped -> natural): gather from the neighbours, scatter to them.
// Halfway bounce-back (push mask bit j: x + e_j is solid):
//  - loads: every population from slot opp(i) of x - e_i without waiting for the
//    mask; a pair with a bounce bit then loads its bounced ones (bit opp(i)) from
//    slot i of x itself over them.
//  - stores: every population of a live cell to its neighbour's slot, a solid
//    neighbour's included (slot i of a solid x + e_i is written by x alone and
//    read by no one: x itself reads its own slot there), and the bounced ones
//    then to the cell's own slots.
// Always the flat launch, blocks of 128 threads, with 32-bit lattice offsets
// where they fit (I). Walled channel, mean of an even and an odd step, us, FP32 /
// FP16: 91.6 / 77.9 with 6 / 7 blocks per SM (80 / 72 registers; FP32 with a force
// per cell 5: 108.1 against 110.9); 64-bit offsets 99.4 / 88.3; loads that select
// their address by the mask instead 97.2 / 82.7, which with 64-bit offsets in 2
// blocks of 256 (128 registers) were the former 103.4 / 92.5. Without flags, FP16
// 256^3: 7 blocks 223.7, 8 226.4, 6 227.3 (a force per cell, 256x128x128: 73.2,
// 76.1, 71.6).
template <int S, bool FLAGS, int FORCE> constexpr int aa_odd_blocks() {
    if (S == LBM_F64) return 2;
    if (S == LBM_F32) return FLAGS && FORCE == 2 ? 5 : 6;
    return FORCE == 2 && !FLAGS ? 6 : 7;
}

template <int S, bool FLAGS, int FORCE, bool RECORD, bool RED, class I>
__device__ __forceinline__ void aa_odd_pair(const Dev &d, typename Stor<S>::T *__restrict__ A,
                                            typename Stor<S>::R *__restrict__ tape,
                                             PairTotals<typename Stor<S>::R> *tot) {
    typedef typename Stor<S>::T T;
    typedef typename Stor<S>::R R;
    typedef typename Pair2<R>::V V;
    int x0, y, z;
    // alternating plane order (see k_step) on walled lattices only: without
    // flags the 16-bit forms spill 16 more bytes at 64 registers for it (the
    // 512^3 box lost 2.4%, and a lattice that size keeps no plane in L2)
    const int bz = FLAGS && d.zrev ? (int)gridDim.y - 1 - (int)blockIdx.y : (int)blockIdx.y;
    if (!pair_cell<true>(d.g, d.PF, blockDim.x, blockDim.y, blockIdx.x, bz, threadIdx.x, threadIdx.y, x0, y, z))
        return;
    const Geom &g = d.g;
    const long long qs = g.qs;
    const bool has1 = x0 + 1 < g.nx;
    const int c = cell_index(g, x0, y, z);
    uint32_t m0 = 0u, m1 = has1 ? 0u : SOLID_BIT;
    if (FLAGS) {
        const uint2 mm = ld_resident2(d.mask + c);
        m0 = mm.x;
        m1 |= mm.y;
    }
    const bool live0 = !(m0 & SOLID_BIT), live1 = !(m1 & SOLID_BIT);
    // neighbour columns: x0 - 1, x0 + 1, x0 + 2 (the last only for a full pair)
    const int xa = wrap1(x0 - 1, g.nx);
    const int xb = wrap1(x0 + 1, g.nx);
    const int xc = has1 ? wrap1(x0 + 2, g.nx) : x0;
    V s[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const T *Pn = lat_at<I>(A, opp(i), qs, (wrap1(z - ez(i), g.nz) * g.ny + wrap1(y - ey(i), g.ny)) * g.pitch);
        if (ex(i) == 0) {
            Stor<S>::ld2(Pn + x0, s[i].x, s[i].y);
        } else {
            s[i].x = Stor<S>::ld(Pn + (ex(i) > 0 ? xa : xb));
            s[i].y = Stor<S>::ld(Pn + (ex(i) > 0 ? x0 : xc));
        }
    }
    const uint32_t r0 = live0 ? m0 : 0u, r1 = live1 ? m1 : 0u;
    const bool bounce = FLAGS && ((r0 | r1) & 0x7fffeu);
    if (bounce) {
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            const T *Po = lat_at<I>(A, i, qs, c);
            if ((r0 >> opp(i)) & 1u) s[i].x = Stor<S>::ld(Po);
            if ((r1 >> opp(i)) & 1u) s[i].y = Stor<S>::ld(Po + 1);
        }
    }
    if (FLAGS && !live0 && !live1) return;
    const uint2 mv = FLAGS && d.moving_on && ((r0 | r1) & MOVING_BIT)
                         ? moving_links(d, c, r0, r1)
                         : make_uint2(0u, 0u);
    if (mv.x | mv.y) {
        // bounced off a moving wall: plus 6 w_i (e_i . u_w)
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            if ((mv.x >> opp(i)) & 1u) s[i].x += wall_term<R>(d, i);
            if ((mv.y >> opp(i)) & 1u) s[i].y += wall_term<R>(d, i);
        }
    }
    V Fx, Fy, Fz;
    Guo2<R> G;
    pair_force<R, FORCE, relax_about_t(S)>(d, c, Fx, Fy, Fz, G);
    Mom2<R> m;
    if constexpr (S == LBM_F64)
        m = pair64<FORCE != 0, true, RECORD || RED>(d, s, Fx, Fy, Fz, live0, live1);
    else
        m = moments2<R, FORCE != 0>(s, Fx, Fy, Fz, d.incomp);
    if (RED) tot->set(m, live0, live1);
    pair_check_record<R, RECORD>(d, c, live0, live1, m, tape);
    if constexpr (S != LBM_F64)
        collide2<R, FORCE != 0, relax_about_t(S)>(s, m, DevR<R>::omega(d), DevR<R>::cs(d), Fx, Fy, Fz, G, d.incomp);
    // P_i(x) to slot i of x + e_i
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        T *Pn = lat_at<I>(A, i, qs, (wrap1(z + ez(i), g.nz) * g.ny + wrap1(y + ey(i), g.ny)) * g.pitch);
        if (ex(i) == 0 && live0 && live1) {
            Stor<S>::st2(Pn + x0, s[i].x, s[i].y);
        } else {
            if (live0) Stor<S>::st(Pn + (ex(i) > 0 ? xb : (ex(i) < 0 ? xa : x0)), s[i].x);
            if (live1) Stor<S>::st(Pn + (ex(i) > 0 ? xc : (ex(i) < 0 ? x0 : x0 + 1)), s[i].y);
        }
    }
    if (bounce) {
        // the bounced values, to the own slots
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            T *Po = lat_at<I>(A, opp(i), qs, c);
            if ((r0 >> i) & 1u) Stor<S>::st(Po, s[i].x);
            if ((r1 >> i) & 1u) Stor<S>::st(Po + 1, s[i].y);
        }
    }
    if (mv.x | mv.y) {
        // a population bounced back from a moving wall arrives as opp(i) and
        // carries 6 w_opp(i) (e_opp(i) . u_w) = -6 w_i (e_i . u_w): rewrite
        // the own slots just stored (same thread, so this store is the last)
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            T *Po = A + (long long)opp(i) * qs + c;
            if ((mv.x >> i) & 1u) Stor<S>::st(Po, s[i].x - wall_term<R>(d, i));
            if ((mv.y >> i) & 1u) Stor<S>::st(Po + 1, s[i].y - wall_term<R>(d, i));
        }
    }
}

template <int S, bool FLAGS, int FORCE, bool RECORD, class I>
__global__ void __launch_bounds__(128, aa_odd_blocks<S, FLAGS, FORCE>())
    k_aa_odd(const Dev d, typename Stor<S>::T *__restrict__ A, typename Stor<S>::R *__restrict__ tape) {
    aa_dependent();
    aa_odd_pair<S, FLAGS, FORCE, RECORD, false, I>(d, A, tape, nullptr);
}

// The odd step with the totals of its pre-collision state summed per block.
template <int S, bool FLAGS, int FORCE, class I>
__global__ void __launch_bounds__(128, S == LBM_F64 ? 2 : 5)
    k_aa_odd_reduce(const Dev d, typename Stor<S>::T *__restrict__ A, double *__restrict__ partials) {
    aa_dependent();
    PairTotals<typename Stor<S>::R> tot;
    tot.clear();
    aa_odd_pair<S, FLAGS, FORCE, false, true, I>(d, A, nullptr, &tot);
    block_partials(tot, partials, blockIdx.y * gridDim.x + blockIdx.x);
}

// Both steps run on the flat launch; the odd one with 32-bit offsets where all 19
// arrays fit them.
inline bool aa_narrow(const Dev &d) { return (long long)Q * d.g.qs < (1LL << 32); }
inline dim3 aa_grid(const Dev &d) { return dim3(d.PF.nyb, d.PF.nzr); }

template <int S, bool FLAGS, int FORCE, bool RECORD>
static cudaError_t launch_aa3(const Dev &d, void *A, int odd, void *tape) {
    auto k = !odd ? k_aa_even<S, FLAGS, FORCE, RECORD>
                  : (aa_narrow(d) ? k_aa_odd<S, FLAGS, FORCE, RECORD, unsigned>
                                  : k_aa_odd<S, FLAGS, FORCE, RECORD, long long>);
    return launch_dependent(k, aa_grid(d), dim3(d.PF.bx_threads), d.stream, d, static_cast<typename Stor<S>::T *>(A),
                            static_cast<typename Stor<S>::R *>(tape));
}

template <int S, bool FLAGS, int FORCE>
static cudaError_t launch_aa_tape(const Dev &d, void *A, int odd, void *tape) {
    return tape ? launch_aa3<S, FLAGS, FORCE, true>(d, A, odd, tape)
                : launch_aa3<S, FLAGS, FORCE, false>(d, A, odd, nullptr);
}

template <int S, bool FLAGS>
static cudaError_t launch_aa2(const Dev &d, void *A, int odd, void *tape) {
    if (d.Ffield) return launch_aa_tape<S, FLAGS, 2>(d, A, odd, tape);
    if (d.force_on) return launch_aa_tape<S, FLAGS, 1>(d, A, odd, tape);
    return launch_aa_tape<S, FLAGS, 0>(d, A, odd, tape);
}

template <int S, bool FLAGS, int FORCE>
static cudaError_t launch_aa_reduce3(const Dev &d, void *A, int odd, double *partials, double *out) {
    auto k = !odd ? k_aa_even_reduce<S, FLAGS, FORCE>
                  : (aa_narrow(d) ? k_aa_odd_reduce<S, FLAGS, FORCE, unsigned>
                                  : k_aa_odd_reduce<S, FLAGS, FORCE, long long>);
    const dim3 grid = aa_grid(d);
    const cudaError_t e = launch_dependent(k, grid, dim3(d.PF.bx_threads), d.stream, d,
                                           static_cast<typename Stor<S>::T *>(A), partials);
    if (e != cudaSuccess) return e;
    const int n = (int)(grid.x * grid.y);
    return sum_partials(partials, n, partials + 4 * (size_t)n, out, d.stream);
}

template <int S, bool FLAGS>
static cudaError_t launch_aa_reduce2(const Dev &d, void *A, int odd, double *partials, double *out) {
    if (d.Ffield) return launch_aa_reduce3<S, FLAGS, 2>(d, A, odd, partials, out);
    if (d.force_on) return launch_aa_reduce3<S, FLAGS, 1>(d, A, odd, partials, out);
    return launch_aa_reduce3<S, FLAGS, 0>(d, A, odd, partials, out);
}

template <int S>
cudaError_t AaOps<S>::step_reduce(const Dev &d, void *A, int odd, double *partials, double *out) {
    if (d.flags && !d.mask) return cudaErrorInvalidValue;
    return d.flags ? launch_aa_reduce2<S, true>(d, A, odd, partials, out)
                   : launch_aa_reduce2<S, false>(d, A, odd, partials, out);
}

template <int S>
cudaError_t AaOps<S>::step(const Dev &d, void *A, int odd, void *tape) {
    if (d.flags && !d.mask) return cudaErrorInvalidValue;  // the odd step selects with the push masks
    return d.flags ? launch_aa2<S, true>(d, A, odd, tape) : launch_aa2<S, false>(d, A, odd, tape);
}

}  // namespace lbm
