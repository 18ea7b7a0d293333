// Kernels of the D3Q19 BGK path, templated on the population storage format.
// Included by one translation unit per format (lbm_ops_*.cu), which
// instantiates Ops<S>.
//
// Data layout (HBM): two padded structure-of-arrays lattices of 19 arrays
// each, P[i][z][y][pitch]; the kernels keep the post-collision populations
// P^n at the cell where they were computed and gather them at the start of
// the next step (Sec. 6: loads from the neighbours, aligned coalesced stores
// to the local cell, two grids). With halfway bounce-back folded into the
// gather (Sec. 2: bounce-back combined with streaming):
//   f^{n+1}_i(x) = P^n_i(x - e_i)        if x - e_i is fluid
//                = P^n_{opp(i)}(x)        otherwise.
#pragma once

#include "lbm_launch.h"

namespace lbm {

// v rounded once, to nearest even, to an element of a canonical or stored
// array. Each is the direct conversion of the value's own type: GB300 runs
// conversions to and from double on its FP64 pipe (2 a clock and SM), and a
// detour over double kept that pipe 90% busy in the 16-bit state kernels.
template <class T> struct Rn;
template <> struct Rn<double> {
    static __device__ __forceinline__ double of(double v) { return v; }
    static __device__ __forceinline__ double of(float v) { return (double)v; }
};
template <> struct Rn<float> {
    static __device__ __forceinline__ float of(double v) { return __double2float_rn(v); }
    static __device__ __forceinline__ float of(float v) { return v; }
};
template <> struct Rn<__half> {
    static __device__ __forceinline__ __half of(double v) { return __double2half(v); }
    static __device__ __forceinline__ __half of(float v) { return __float2half_rn(v); }
};
template <> struct Rn<__nv_bfloat16> {
    static __device__ __forceinline__ __nv_bfloat16 of(double v) { return __double2bfloat16(v); }
    static __device__ __forceinline__ __nv_bfloat16 of(float v) { return __float2bfloat16_rn(v); }
};

// Element access of canonical arrays in a storage format: values are read in
// the narrowest arithmetic type that holds them exactly (V).
template <int D> struct IOFmt;
template <> struct IOFmt<LBM_F64> {
    typedef double T;
    typedef double V;
    static __device__ __forceinline__ V get(const T *p) { return __ldg(p); }
};
template <> struct IOFmt<LBM_F32> {
    typedef float T;
    typedef float V;
    static __device__ __forceinline__ V get(const T *p) { return __ldg(p); }
};
template <> struct IOFmt<LBM_F16S> {
    typedef __half T;
    typedef float V;
    static __device__ __forceinline__ V get(const T *p) { return Stor<LBM_F16S>::ld(p); }
};
template <> struct IOFmt<LBM_BF16S> {
    typedef __nv_bfloat16 T;
    typedef float V;
    static __device__ __forceinline__ V get(const T *p) { return Stor<LBM_BF16S>::ld(p); }
};

// Elements p[0], p[1] of a canonical array; whole pairs move at once where
// `pair` says that they are aligned (pair_aligned).
template <int D, class P>
__device__ __forceinline__ void get2(const P *p, bool pair, bool has1, typename IOFmt<D>::V &a,
                                     typename IOFmt<D>::V &b) {
    if (pair) {
        Stor<D>::ld2(p, a, b);
    } else {
        a = IOFmt<D>::get(p);
        b = IOFmt<D>::get(p + (has1 ? 1 : 0));  // (no branch between a thread's loads)
    }
}
template <class T> struct alignas(2 * sizeof(T)) Two {
    T a, b;
};
template <class T, class V> __device__ __forceinline__ void put2(T *p, bool pair, bool has1, V a, V b) {
    if (pair) {
        *reinterpret_cast<Two<T> *>(p) = Two<T>{Rn<T>::of(a), Rn<T>::of(b)};
    } else {
        p[0] = Rn<T>::of(a);
        if (has1) p[1] = Rn<T>::of(b);
    }
}

// Canonical state arrays of a moment-split context hold plain shifted
// deviations in the format's 16-bit element type.
template <> struct IOFmt<LBM_F16M> : IOFmt<LBM_F16S> {};
template <> struct IOFmt<LBM_BF16M> : IOFmt<LBM_BF16S> {};

// Whether every pair (x0, x0 + 1), x0 even, of every array [k][nz][ny][nx] at
// p starts on a whole-pair boundary (host side).
inline bool pair_aligned(const Geom &g, const void *p, size_t elem) {
    return (g.nx & 1) == 0 && reinterpret_cast<uintptr_t>(p) % (2 * elem) == 0;
}

// ---------------------------------------------------------------------------
// Moment-split storage (LBM_F16M, LBM_BF16M): a cell holds, for its 19
// post-collision values P_i, the momentum word J (SplitJ) and the remainders
// g_i = s_i - K_i (e_i . J) (s_i = P_i - w_i, J as stored), rebuilt as
// s_i = K_i (e_i . J) + g_i with one fused multiply-add. K_i = 3 w_i, taken as
// the momentum-exact pair of OddK (2 K_axis + 8 K_diag = 1 exactly, so the
// base parts carry J itself). Writing e_i = sigma e'_i with the first non-zero
// component of e'_i equal to +1, K_i (e_i . J) = (sigma K_i)(e'_i . J): e'_i . J
// is one component or one sum / difference (edot_first), the same value in the
// packed step kernel and the per-cell readers.
LBM_HD constexpr bool first_positive(int i) {
    return ex(i) > 0 || (ex(i) == 0 && (ey(i) > 0 || (ey(i) == 0 && ez(i) > 0)));
}
// e'_i: the member of the pair (i, opp(i)) whose first non-zero component is +1.
LBM_HD constexpr int split_first(int i) { return first_positive(i) ? i : opp(i); }
// sigma K_i (0 for the rest population).
LBM_HD constexpr float split_k(int i) {
    return i == 0 ? 0.0f : (first_positive(i) ? 1.0f : -1.0f) * (i <= 6 ? OddK<float>::AXIS : OddK<float>::DIAG);
}

// e'_i . J of one cell's momentum word (scalar; the association of edot_first).
template <int S> __device__ __forceinline__ float split_edot(int i, uint2 w) {
    const float jx = SplitJ<S>::lo(w.x), jy = SplitJ<S>::hi(w.x), jz = SplitJ<S>::lo(w.y);
    if (ex(i)) {
        if (ey(i)) return ey(i) > 0 ? __fadd_rn(jx, jy) : __fsub_rn(jx, jy);
        if (ez(i)) return ez(i) > 0 ? __fadd_rn(jx, jz) : __fsub_rn(jx, jz);
        return jx;
    }
    if (ey(i)) {
        if (ez(i)) return ez(i) > 0 ? __fadd_rn(jy, jz) : __fsub_rn(jy, jz);
        return jy;
    }
    return jz;
}

// Momentum words of a moment-split lattice P (one uint2 per padded cell).
template <class T> __device__ __forceinline__ const uint2 *split_words(const Dev &d, const T *P) {
    return reinterpret_cast<const uint2 *>(P + d.jo);
}
template <class T> __device__ __forceinline__ uint2 *split_words(const Dev &d, T *P) {
    return reinterpret_cast<uint2 *>(P + d.jo);
}

// In a row of odd length the padding cell after the last cell holds a copy of
// the momentum word of the row's first cell (x = 0): the lone last cell of the
// row, whose thread loads the word pair (nx - 1, nx), pulls its e_x = -1
// values from cell 0 (periodic in x). Every writer of cell 0's word keeps it.
__device__ __forceinline__ void split_ghost(const Dev &d, uint2 *J, int x, int c, uint2 w) {
    if ((d.g.nx & 1) && x == 0) J[c + d.g.nx] = w;
}

// Two values rounded to the 16-bit format (nearest even) from double.
template <int S> __device__ __forceinline__ unsigned split_pack(double a, double b) {
    union {
        unsigned short h[2];
        unsigned u;
    } v;
    if (S == LBM_F16M) {
        v.h[0] = __half_as_ushort(__double2half(a));
        v.h[1] = __half_as_ushort(__double2half(b));
    } else {
        v.h[0] = __bfloat16_as_ushort(__double2bfloat16(a));
        v.h[1] = __bfloat16_as_ushort(__double2bfloat16(b));
    }
    return v.u;
}

// Write one cell's 19 shifted values v at cell c of a
// moment-split lattice: J = sum_i v_i e_i rounded to the format, then the
// remainders g_i = v_i - K_i (e_i . J) rounded.
template <int S>
__device__ __forceinline__ void split_store(const Dev &d, typename Stor<S>::T *P, int x, int c, const double v[Q]) {
    double jx = 0.0, jy = 0.0, jz = 0.0;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        if (ex(i)) jx += ex(i) > 0 ? v[i] : -v[i];
        if (ey(i)) jy += ey(i) > 0 ? v[i] : -v[i];
        if (ez(i)) jz += ez(i) > 0 ? v[i] : -v[i];
    }
    const unsigned wx = split_pack<S>(jx, jy), wy = split_pack<S>(jz, 0.0);
    const uint2 w = make_uint2(wx, wy);
    P[c] = Rn<typename Stor<S>::T>::of(v[0]);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const double g = fma((double)-split_k(i), (double)split_edot<S>(split_first(i), w), v[i]);
        P[(long long)i * d.g.qs + c] = Rn<typename Stor<S>::T>::of(g);
    }
    split_words(d, P)[c] = w;
    split_ghost(d, split_words(d, P), x, c, w);
}

// The same values, as if newly read: what a rare branch computes from them is
// not computed ahead of it and kept in registers.
__device__ __forceinline__ void forget(int &a) { asm volatile("" : "+r"(a)); }

// The moving-wall bits of the pair at cell c among the bits of m0 and m1. One
// dependent load: a flag load per bounced link put a chain of them on the
// threads next to a lid, which the whole step of a small cavity waits for
// (65x67x63: 9.3 us a step, 6.3 with these words).
__device__ __forceinline__ uint2 moving_links(const Dev &d, int c, uint32_t m0, uint32_t m1) {
    uint2 v = ld_resident2(d.moving + c);
    v.x &= m0;
    v.y &= m1;
    return v;
}

// Moving-wall term of a population bounced into direction i: 6 w_i (e_i . u_w).
template <class R> __device__ __forceinline__ R wall_term(const Dev &d, int i);
template <> __device__ __forceinline__ float wall_term<float>(const Dev &d, int i) { return d.wcf[i]; }
template <> __device__ __forceinline__ double wall_term<double>(const Dev &d, int i) { return d.wc[i]; }

// NaN marks solid slots in the AA pattern. (It is hygiene only: the odd step's
// mask-free scatter stores into solid slots, and no reader takes a solid slot's value.)
__device__ __forceinline__ bool nan_marked(const Dev &d) { return d.layout != LAYOUT_PULL; }

// ---------------------------------------------------------------------------
// Fused stream-collide (Sec. 2 steps 1-3, Eq. 1; Sec. 6 pull-style update).
//
// Each thread updates the two x-adjacent cells x0, x0 + 1 of one row, so the
// populations with e_x = 0 (rest, +-y, +-z and the yz diagonals) move as one
// aligned pair per load and every population is stored as one aligned pair;
// populations with e_x = +-1 come from sources shifted by one cell and are
// loaded per cell. Every pair is stored whole, a solid cell included, so
// 32-byte sectors are written complete (FP32 leaves out the sectors whose
// cells are all solid, which no one reads). Halfway bounce-back takes one of
// these forms, chosen per storage format by measurement (Bounce<S>):
//
//  - mask-guided reload (FP32 and FP64): a 32-bit push mask per cell (bit j:
//    x + e_j is solid) is loaded first but the gather
//    does not wait for it (every load takes the neighbour's address); pairs
//    with a bounce bit then reload their bounced populations from the cell's
//    own opposite slots, over the gathered values, before the moments.
//    Solid slots are never read. 37.5 against 34.0 GFLUPS on the channel for
//    solid slots that hold NaN, each value tested and the moments taken twice.
//  - separate kernel (16-bit storage), the paper's arrangement (Sec. 7: the
//    non-fluid cells are treated in a separate kernel): a solid cell s keeps in
//    slot i the value that its fluid neighbour s + e_i pulls next step (that
//    neighbour's post-collision population opp(i)); after the step, k_bounce
//    copies those values along a precomputed list of boundary links. Fewest
//    instructions in the step kernel, which is what the 2-byte formats need.
// In every form the fluid cells' own slots hold the post-collision
// populations, which is what the flag-aware readers (macros, state, reduction,
// adjoint) gather.
//
// Resident blocks of 256 threads per SM (two of 128 for one of 256 in the flat
// launch): FP32 storage 3 (<= 80 registers), 16-bit storage 4 (<= 64: fewer bytes
// per thread, so more threads in flight); the FP64 AA steps, two cells a thread,
// 1 (<= 255). The FP64 two-grid step has its own (k_step64).
template <int S> struct StepBlocks {
    static constexpr int value = S == LBM_F64 ? 1 : ((S == LBM_F32 || is_split(S)) ? 3 : 4);
};
template <int S> struct Bounce {
    static constexpr int mode = bounce_mode(S);
};
template <int S> struct LinkBounce {
    static constexpr bool value = Bounce<S>::mode == BB_LINKS;
};

template <class R> __device__ __forceinline__ R quiet_nan();
template <> __device__ __forceinline__ float quiet_nan<float>() { return __int_as_float(0x7fffffff); }
template <> __device__ __forceinline__ double quiet_nan<double>() {
    return __longlong_as_double(0x7fffffffffffffffLL);
}

// The precomputed Guo constants of a uniform force, with c = 1 - omega/2, or
// over omega (c' = tau - 1/2) for the form of collide2 that relaxes about T.
template <class R, bool TFORM> __device__ __forceinline__ Guo2<R> uniform_guo(const Dev &d);
template <> __device__ __forceinline__ Guo2<float> uniform_guo<float, false>(const Dev &d) {
    Guo2<float> t;
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        t.A[p] = vsplat(d.gAf[p]);
        t.C[p] = vsplat(d.gCf[p]);
    }
    return t;
}
template <> __device__ __forceinline__ Guo2<float> uniform_guo<float, true>(const Dev &d) {
    Guo2<float> t;
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        t.A[p] = vsplat(d.gAtf[p]);
        t.C[p] = vsplat(d.gCtf[p]);
    }
    return t;
}
// Where the gather finds the row of population i that cell row (y, z) pulls
// from, (y - e_iy, z - e_iz): in the source lattice in global memory, or in
// a shared-memory copy of those 19 rows (see k_step_tma).
// Offset k qs + c of lattice P: in 64 bits, or (I = unsigned, where every
// offset of the lattice fits) as one 32-bit index, which costs fewer
// instructions per address.
template <class I, class T> __device__ __forceinline__ T *lat_at(T *P, int k, long long qs, int c) {
    if constexpr (sizeof(I) == 4)
        return P + ((unsigned)k * (unsigned)qs + (unsigned)c);
    else
        return P + (long long)k * qs + c;
}

template <int S, class I = long long> struct GlobalRows {
    typedef typename Stor<S>::T T;
    typedef typename Stor<S>::R R;
    const T *src;
    __device__ __forceinline__ const T *row(const Geom &g, int i, int y, int z) const {
        return lat_at<I>(src, i, g.qs, (wrap1(z - ez(i), g.nz) * g.ny + wrap1(y - ey(i), g.ny)) * g.pitch);
    }
    static __device__ __forceinline__ R ld(const T *p) { return Stor<S>::ld(p); }
    static __device__ __forceinline__ void ld2(const T *p, R &a, R &b) { Stor<S>::ld2(p, a, b); }
};
template <int S> struct SharedRows {
    typedef typename Stor<S>::T T;
    typedef typename Stor<S>::R R;
    const T *buf;  // [Q][pitch]
    __device__ __forceinline__ const T *row(const Geom &g, int i, int, int) const { return buf + i * g.pitch; }
    static __device__ __forceinline__ R ld(const T *p) { return Stor<S>::ls(p); }
    static __device__ __forceinline__ void ld2(const T *p, R &a, R &b) { Stor<S>::ls2(p, a, b); }
};

// A pair's contribution to the totals: rho - 1 and the momentum j + F/2 of its
// fluid cells (0 for the others), and how many fluid cells it has.
template <class R> struct PairTotals {
    typename Pair2<R>::V v[4];
    int cells;
    __device__ __forceinline__ void clear() {
        v[0] = v[1] = v[2] = v[3] = vsplat(R(0));
        cells = 0;
    }
    __device__ __forceinline__ void set(const Mom2<R> &m, bool live0, bool live1) {
        const typename Pair2<R>::V a[4] = {m.rho1, m.jx, m.jy, m.jz};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k].x = live0 ? a[k].x : R(0);
            v[k].y = live1 ? a[k].y : R(0);
        }
        cells = (int)live0 + (int)live1;
    }
};

// Totals of FP32 values without FP64 arithmetic, which GB300 executes at 2 a
// clock and SM (the block sums of a step took longer than the step itself:
// 256^3 box, BF16, 595 us against 212; 259 with integer sums). A value |v| < 1024 is cut exactly
// into whole multiples of 2^-12, 2^-35, 2^-58 and 2^-81 (adding and taking off
// 1.5 2^23 grid steps rounds to a grid), and the multiples are summed as
// integers: exactly, and in any order. What is dropped is below 2^-82 per
// value, so the sums carry less rounding than FP64 ones.
constexpr int TOT_LEVELS = 4;
__host__ __device__ constexpr int tot_grid(int l) { return -12 - 23 * l; }
__device__ __forceinline__ constexpr float pow2f(int e) {
    float r = 1.0f;
    for (; e < 0; ++e) r *= 0.5f;
    for (; e > 0; --e) r *= 2.0f;
    return r;
}
__device__ __forceinline__ constexpr double pow2d(int e) {
    double r = 1.0;
    for (; e < 0; ++e) r *= 0.5;
    return r;
}
__device__ __forceinline__ bool tot_fits(float v) { return fabsf(v) < 1024.0f; }  // (false for NaN)
__device__ __forceinline__ void tot_add(int h[TOT_LEVELS], float v) {
#pragma unroll
    for (int l = 0; l < TOT_LEVELS; ++l) {
        constexpr float one = 1.5f * 8388608.0f;
        const float M = one * pow2f(tot_grid(l));
        const float t = __fadd_rn(v, M);
        h[l] += __float_as_int(t) - __float_as_int(M);  // the multiple: |v| / 2^grid <= 2^22
        v = __fsub_rn(v, __fsub_rn(t, M));
    }
}

// The block's sum of every thread's red[4], in a fixed order, to out[k] of
// thread k < 4. Every thread of the block calls it (whole warps, <= 256 threads).
__device__ __forceinline__ double block_sum_d(const double red[4]) {
    __shared__ double sm[8][4];
    const int tid = threadIdx.y * blockDim.x + threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nwarps = (blockDim.x * blockDim.y) >> 5;
    // halves of the warp exchange two of the quantities, quarters one: 6 FP64
    // adds a thread instead of the 20 of four whole butterflies
    const bool up = lane & 16, up2 = lane & 8;
    const double a = (up ? red[2] : red[0]) + __shfl_xor_sync(0xffffffffu, up ? red[0] : red[2], 16);
    const double b = (up ? red[3] : red[1]) + __shfl_xor_sync(0xffffffffu, up ? red[1] : red[3], 16);
    double v = (up2 ? b : a) + __shfl_xor_sync(0xffffffffu, up2 ? a : b, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((lane & 7) == 0) sm[wid][lane >> 3] = v;
    __syncthreads();
    double t = 0.0;
    if (tid < 4)
        for (int w = 0; w < nwarps; ++w) t += sm[w][tid];
    return t;
}

// The block's totals (sum rho, sum j) to partials[4 b + k] of block b, from
// each thread's pair. FP32: integer sums (above); where a value of the block is
// too large for them (or NaN), FP64 sums in a fixed order.
__device__ __forceinline__ void block_partials(const PairTotals<double> &p, double *__restrict__ partials, int b) {
    double red[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) red[k] = p.v[k].x + p.v[k].y;
    red[0] += (double)p.cells;
    const double t = block_sum_d(red);
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    if (tid < 4) partials[4 * (long long)b + tid] = t;
}
__device__ __forceinline__ void block_partials(const PairTotals<float> &p, double *__restrict__ partials, int b) {
    __shared__ int smw[8][4 * TOT_LEVELS + 1];
    const int tid = threadIdx.y * blockDim.x + threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nwarps = (blockDim.x * blockDim.y) >> 5;
    bool fits = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) fits = fits && tot_fits(p.v[k].x) && tot_fits(p.v[k].y);
    if (__syncthreads_or(!fits)) {
        double red[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) red[k] = (double)p.v[k].x + (double)p.v[k].y;
        red[0] += (double)p.cells;
        const double t = block_sum_d(red);
        if (tid < 4) partials[4 * (long long)b + tid] = t;
        return;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        int h[TOT_LEVELS] = {0, 0, 0, 0};
        tot_add(h, p.v[k].x);
        tot_add(h, p.v[k].y);
#pragma unroll
        for (int l = 0; l < TOT_LEVELS; ++l) {
            const int r = __reduce_add_sync(0xffffffffu, h[l]);  // |r| <= 32 * 2 * 2^22
            if (lane == 0) smw[wid][k * TOT_LEVELS + l] = r;
        }
    }
    const int n = __reduce_add_sync(0xffffffffu, p.cells);
    if (lane == 0) smw[wid][4 * TOT_LEVELS] = n;
    __syncthreads();
    if (tid < 4) {
        double t = 0.0;
#pragma unroll
        for (int l = TOT_LEVELS - 1; l >= 0; --l) {
            long long h = 0;
            for (int w = 0; w < nwarps; ++w) h += smw[w][tid * TOT_LEVELS + l];
            t = fma((double)h, pow2d(tot_grid(l)), t);
        }
        if (tid == 0) {
            int n = 0;
            for (int w = 0; w < nwarps; ++w) n += smw[w][4 * TOT_LEVELS];
            t += (double)n;
        }
        partials[4 * (long long)b + tid] = t;
    }
}

// ---------------------------------------------------------------------------
// One cell in FP64: moments and collision in fixed point (lbm_fixed.cuh), in
// FP64 arithmetic where the cell is outside its range. Every FP64 kernel takes
// its cells through here, so they agree bit for bit.
struct Cell64 {
    double rho1, rho, jx, jy, jz, ux, uy, uz;  // (j = j + F/2)
};
// The FP64 form: s is replaced by its post-collision values if `collide`.
static __device__ __noinline__ void cell64_fp64(double *s, Cell64 *m, double Fx, double Fy, double Fz, double omega,
                                                bool incomp, bool collide) {
    double v[Q];
    for (int i = 0; i < Q; ++i) v[i] = s[i];
    const Mom<double> o = moments<double>(v, Fx, Fy, Fz, incomp);
    m->rho1 = o.rho1;
    m->rho = o.rho;
    m->ux = o.ux;
    m->uy = o.uy;
    m->uz = o.uz;
    m->jx = incomp ? o.ux : o.rho * o.ux;
    m->jy = incomp ? o.uy : o.rho * o.uy;
    m->jz = incomp ? o.uz : o.rho * o.uz;
    if (!collide) return;
    const double rho_e = incomp ? 1.0 : o.rho, c = 1.0 - 0.5 * omega;
    const double usq = o.ux * o.ux + o.uy * o.uy + o.uz * o.uz, uF = o.ux * Fx + o.uy * Fy + o.uz * Fz;
    for (int i = 0; i < Q; ++i) {
        const double w = weight(i), eu = ex(i) * o.ux + ey(i) * o.uy + ez(i) * o.uz;
        const double eF = ex(i) * Fx + ey(i) * Fy + ez(i) * Fz;
        s[i] = (1.0 - omega) * v[i] + omega * w * (o.rho1 + rho_e * (3.0 * eu + 4.5 * eu * eu - 1.5 * usq)) +
               c * w * (3.0 * (eF - uF) + 9.0 * eu * eF);
    }
}
// MOM: m is wanted (otherwise only m.rho, 1 or what a diverging cell has).
template <bool FORCE, bool COLLIDE, bool MOM>
__device__ __forceinline__ void cell64(const Dev &d, double s[Q], double Fx, double Fy, double Fz, Cell64 &m) {
    FixedMom f;
    m.rho = 1.0;
    if (fixed_moments<FORCE>(s, Fx, Fy, Fz, f)) {
        if (MOM) {
            m.rho1 = fx_out(f.r, f.E);
            m.rho = 1.0 + m.rho1;
            m.jx = fx_out(f.jx, f.E);
            m.jy = fx_out(f.jy, f.E);
            m.jz = fx_out(f.jz, f.E);
            const double inv = d.incomp ? 1.0 : rcp_rn(m.rho);
            m.ux = m.jx * inv;
            m.uy = m.jy * inv;
            m.uz = m.jz * inv;
        }
        if (COLLIDE) fixed_collide<FORCE>(s, f, d.fk, d.incomp);
    } else {
        double t[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) t[i] = s[i];
        Cell64 o;
        cell64_fp64(t, &o, Fx, Fy, Fz, d.omega, d.incomp, COLLIDE);
        m = o;
#pragma unroll
        for (int i = 0; COLLIDE && i < Q; ++i) s[i] = t[i];
    }
}

// The pair's moments, and its collision (COLLIDE), cell by cell; a cell that is
// not live is left alone, with rho = 1. (The solid slots of an AA lattice hold
// NaN, which is outside the fixed-point range: one such lane sent its whole warp
// through cell64_fp64, and 65% of the warps of the 256x128x128 channel hold one:
// mean AA step 1871 us, 418 without them; in FP64 arithmetic throughout 1383.)
template <bool FORCE, bool COLLIDE, bool MOM>
__device__ __forceinline__ Mom2<double> pair64(const Dev &d, double2 s[Q], double2 Fx, double2 Fy, double2 Fz,
                                               bool live0, bool live1) {
    Mom2<double> m;
    m.rho = vsplat(1.0);
    if (MOM) m.rho1 = m.jx = m.jy = m.jz = m.ux = m.uy = m.uz = vsplat(0.0);
    if (live0) {
        double t[Q];
        Cell64 o;
#pragma unroll
        for (int i = 0; i < Q; ++i) t[i] = s[i].x;
        cell64<FORCE, COLLIDE, MOM>(d, t, Fx.x, Fy.x, Fz.x, o);
#pragma unroll
        for (int i = 0; COLLIDE && i < Q; ++i) s[i].x = t[i];
        m.rho.x = o.rho;
        if (MOM)
            m.rho1.x = o.rho1, m.jx.x = o.jx, m.jy.x = o.jy, m.jz.x = o.jz, m.ux.x = o.ux, m.uy.x = o.uy, m.uz.x = o.uz;
    }
    if (live1) {
        double t[Q];
        Cell64 o;
#pragma unroll
        for (int i = 0; i < Q; ++i) t[i] = s[i].y;
        cell64<FORCE, COLLIDE, MOM>(d, t, Fx.y, Fy.y, Fz.y, o);
#pragma unroll
        for (int i = 0; COLLIDE && i < Q; ++i) s[i].y = t[i];
        m.rho.y = o.rho;
        if (MOM)
            m.rho1.y = o.rho1, m.jx.y = o.jx, m.jy.y = o.jy, m.jz.y = o.jz, m.ux.y = o.ux, m.uy.y = o.uy, m.uz.y = o.uz;
    }
    return m;
}

// The moments of a pair for the readers. FP64: the NaN of an AA lattice's solid cells
// is replaced first (see pair64; on two-grid lattices, which hold none, macros of the
// 256x128x128 channel take 175 us, 181 with a branch on each cell).
template <class R, bool FORCE>
__device__ __forceinline__ Mom2<R> pair_moments(const Dev &d, typename Pair2<R>::V s[Q], typename Pair2<R>::V Fx,
                                                typename Pair2<R>::V Fy, typename Pair2<R>::V Fz, bool live0,
                                                bool live1) {
    if constexpr (sizeof(R) == 8) {
        if (d.layout != LAYOUT_PULL) {
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                if (!live0) s[i].x = R(0);
                if (!live1) s[i].y = R(0);
            }
        }
        return pair64<FORCE, false, true>(d, s, Fx, Fy, Fz, true, true);
    } else {
        return moments2<R, FORCE>(s, Fx, Fy, Fz, d.incomp);
    }
}

// One fused step for the cell pair (x0, x0 + 1) of row (y, z): gather through
// `rows` (the cell's own opposite populations, for bounce-back, from src),
// collide, store to dst. RED: also hand out the pair's totals (of the
// pre-collision state); the pair then never returns early, so that its block
// can reduce.
template <int S, bool FLAGS, int FORCE, bool RECORD, class Rows, bool RED = false, class I = long long>
__device__ __forceinline__ void step_pair(const Dev &d, const Rows &rows, const typename Stor<S>::T *__restrict__ src,
                                          typename Stor<S>::T *__restrict__ dst, typename Stor<S>::R *__restrict__ tape,
                                          int x0, int y, int z, PairTotals<typename Stor<S>::R> *tot = nullptr) {
    typedef typename Stor<S>::T T;
    typedef typename Stor<S>::R R;
    typedef typename Pair2<R>::V V;  // lane x: cell x0, lane y: cell x0 + 1
    constexpr bool MFIX = Bounce<S>::mode == BB_MFIX;
    constexpr bool LINKS = !MFIX;  // flag-free gather
    const Geom &g = d.g;
    const bool has1 = x0 + 1 < g.nx;
    const int c = cell_index(g, x0, y, z);
    uint32_t m0 = 0u, m1 = 0u;
    bool live0 = true, live1 = has1;
    if (FLAGS && !LINKS) {
        const uint2 mm = ld_resident2(d.mask + c);
        m0 = mm.x;
        m1 = mm.y;
        live0 = !(m0 & SOLID_BIT);
        live1 = has1 && !(m1 & SOLID_BIT);
    } else if (FLAGS) {
        const uchar2 fl = __ldg(reinterpret_cast<const uchar2 *>(d.flags + c));
        // (no early exit for two solid cells: branching on this load would put
        // a dependent round trip in front of the gather, which measured ~12%
        // slower on the walled channel than loading and storing their pairs)
        live0 = !fl.x;
        live1 = has1 && !fl.y;
    }
    // source columns of the e_x = +-1 populations
    const int xa = wrap1(x0 - 1, g.nx);              // e_x = +1, cell x0
    const int xb = wrap1(x0 + 1, g.nx);              // e_x = -1, cell x0
    const int xc = has1 ? wrap1(x0 + 2, g.nx) : x0;  // e_x = -1, cell x0 + 1 (e_x = +1 pulls from x0)
    V s[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const T *Pi = rows.row(g, i, y, z);
        if (ex(i) == 0) {
            Rows::ld2(Pi + x0, s[i].x, s[i].y);
        } else {
            s[i].x = Rows::ld(Pi + (ex(i) > 0 ? xa : xb));
            s[i].y = Rows::ld(Pi + (ex(i) > 0 ? x0 : xc));
        }
    }
    // (a solid cell's mask has the bits of its solid neighbours, but its
    // values are never read: only fluid lanes reload, which spares the pairs
    // inside obstacles 36 loads; walled channel +1.5%)
    const uint32_t r0 = live0 ? m0 : 0u, r1 = live1 ? m1 : 0u;
    if (FLAGS && MFIX && ((r0 | r1) & 0x7fffeu)) {
        // a pair next to a solid: its bounced populations come from the
        // cell's own opposite slots, loaded over the gathered (unread) ones
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            const T *Po = lat_at<I>(src, opp(i), g.qs, c);
            if ((r0 >> opp(i)) & 1u) s[i].x = Stor<S>::ld(Po);
            if ((r1 >> opp(i)) & 1u) s[i].y = Stor<S>::ld(Po + 1);
        }
    }
    if (FLAGS && !LINKS && d.moving_on && ((m0 | m1) & MOVING_BIT)) {
        // next to a moving wall: add its term to the bounced values
        const uint2 mv = moving_links(d, c, m0, m1);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            if ((mv.x >> opp(i)) & 1u) s[i].x += wall_term<R>(d, i);
            if ((mv.y >> opp(i)) & 1u) s[i].y += wall_term<R>(d, i);
        }
    }
    V Fx = vsplat(R(0)), Fy = vsplat(R(0)), Fz = vsplat(R(0));
    Guo2<R> G;
    if (FORCE == 1) {
        Fx = vsplat(DevR<R>::F(d, 0));
        Fy = vsplat(DevR<R>::F(d, 1));
        Fz = vsplat(DevR<R>::F(d, 2));
        G = uniform_guo<R, relax_about_t(S)>(d);
    } else if (FORCE == 2) {
        const R *F = static_cast<const R *>(d.Ffield);
        ld2_real(F + c, Fx.x, Fx.y);
        ld2_real(F + g.qs + c, Fy.x, Fy.y);
        ld2_real(F + 2 * g.qs + c, Fz.x, Fz.y);
        G = guo2<R>(relax_about_t(S) ? DevR<R>::cs(d) : R(1) - R(0.5) * DevR<R>::omega(d), Fx, Fy, Fz);
    }
    const Mom2<R> m = moments2<R, FORCE != 0>(s, Fx, Fy, Fz, d.incomp);
    const bool bad0 = live0 && !(m.rho.x > R(0) && m.rho.x < R(1e30));
    const bool bad1 = live1 && !(m.rho.y > R(0) && m.rho.y < R(1e30));
    if (bad0 || bad1) atomicOr(d.status, LBM_STATUS_DIVERGED);
    if (RED) tot->set(m, live0, live1);
    if (RECORD) {
        const long long qs = g.qs;
        st2_real(tape + c, m.rho.x, m.rho.y);
        st2_real(tape + qs + c, m.ux.x, m.ux.y);
        st2_real(tape + 2 * qs + c, m.uy.x, m.uy.y);
        st2_real(tape + 3 * qs + c, m.uz.x, m.uz.y);
    }
    collide2<R, FORCE != 0, relax_about_t(S)>(s, m, DevR<R>::omega(d), DevR<R>::cs(d), Fx, Fy, Fz, G, d.incomp);
    // The pair is stored whole, a solid cell included, so 32-byte sectors are
    // written complete: a solid cell's values are never read (mask-guided
    // reload, where all-solid sectors are left out below), or its slots are
    // link targets that k_bounce rewrites (links). When moving-wall links are
    // written into solid slots by other threads of this launch, a pair with a
    // solid cell stores its fluid cell alone.
    if (FLAGS && LinkBounce<S>::value && d.has_moving && !(live0 && live1)) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            if (live0) Stor<S>::st(lat_at<I>(dst, i, g.qs, c), s[i].x);
            if (live1) Stor<S>::st(lat_at<I>(dst, i, g.qs, c + 1), s[i].y);
        }
    } else {
        // FP32 mask-guided reload: a 32-byte sector whose 8 cells are all solid
        // is read by no one (the gather replaces every value it loads from a
        // solid slot, and the readers output zeros for solid cells), so its
        // four pairs skip their stores. Where rows start on sector boundaries
        // and hold a multiple of 4 pairs, the sector's pairs are on the lanes
        // 4k .. 4k + 3 of a warp; a lane not in step here (or past the edge)
        // counts as fluid, so no store is skipped on its account. Walled
        // channel +1.4%.
        bool skip = false;
        if constexpr (FLAGS && MFIX && S == LBM_F32) {
            if ((g.pitch & 7) == 0 && (((g.nx + 1) / 2) & 3) == 0) {
                const unsigned sb = __ballot_sync(__activemask(), !live0 && !live1);
                skip = ((sb >> ((threadIdx.x & 31) & ~3u)) & 0xFu) == 0xFu;
            }
        }
        // write-back stores: the planes a step writes last stay in L2 for the
        // next step, which starts on them (FP32 channel 39.3 against 39.8
        // GFLUPS with streaming stores; the AA and reverse steps keep theirs)
        if (!skip) {
#pragma unroll
            for (int i = 0; i < Q; ++i) Stor<S>::st2_wb(lat_at<I>(dst, i, g.qs, c), s[i].x, s[i].y);
        }
    }
    if (FLAGS && LinkBounce<S>::value && d.has_moving) {
        // Links into a moving wall (not in the link list): slot opp(j) of the
        // wall cell x + e_j gets P_j(x) + 6 w_opp(j) (e_opp(j) . u_w), formed
        // from the unrounded P_j(x) so that it is rounded to storage once.
        const uint2 mm = moving_links(d, c, live0 ? ~0u : 0u, live1 ? ~0u : 0u);
        if (mm.x | mm.y) {
#pragma unroll
            for (int j = 1; j < Q; ++j) {
                if ((mm.x >> j) & 1u)
                    Stor<S>::st(lat_at<I>(dst, opp(j), g.qs, push_dst(g, x0, y, z, j)), s[j].x - wall_term<R>(d, j));
                if ((mm.y >> j) & 1u)
                    Stor<S>::st(lat_at<I>(dst, opp(j), g.qs, push_dst(g, x0 + 1, y, z, j)),
                                s[j].y - wall_term<R>(d, j));
            }
        }
    }
}

// The pre-collision values of the cell pair (x0, x0 + 1) of row (y, z) in a
// moment-split lattice, m0 and m1 the push masks of its cells.
template <int S, bool FLAGS>
__device__ __forceinline__ void gather_pair_split(const Dev &d, const typename Stor<S>::T *__restrict__ src, int x0,
                                                  int y, int z, int c, bool has1, uint32_t m0, uint32_t m1,
                                                  float2 s[Q]) {
    typedef typename Stor<S>::T T;
    typedef float R;
    typedef float2 V;  // lane x: cell x0, lane y: cell x0 + 1
    const Geom &g = d.g;
    const int xa = wrap1(x0 - 1, g.nx);              // e_x = +1, cell x0
    const int xb = wrap1(x0 + 1, g.nx);              // e_x = -1, cell x0
    const int xc = has1 ? wrap1(x0 + 2, g.nx) : x0;  // e_x = -1, cell x0 + 1 (e_x = +1 pulls from x0)
    // Momentum words of the nine source rows (y - e_y, z - e_z), r = 3 (e_y + 1)
    // + e_z + 1: the pair (x0, x0 + 1) of each, and cells xa and xc of the five
    // rows that directions with e_x = +-1 pull from (those with e_y e_z = 0).
    // The lone last cell of an odd row pulls its e_x = -1 values from the
    // row's first cell: its pair's second word is the copy of that cell's word
    // kept after the row's last cell (split_ghost), so no lane needs a select.
    const uint2 *Js = split_words(d, src);
    uint4 jq[9];
    uint2 ja[9], jc[9];
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        const int dy = r / 3 - 1, dz = r % 3 - 1;
        const int rb = (wrap1(z - dz, g.nz) * g.ny + wrap1(y - dy, g.ny)) * g.pitch;
        jq[r] = __ldg(reinterpret_cast<const uint4 *>(Js + rb + x0));
        if (dy == 0 || dz == 0) {
            ja[r] = __ldg(Js + rb + xa);
            jc[r] = __ldg(Js + rb + xc);
        }
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const T *Pi =
            lat_at<long long>(src, i, g.qs, (wrap1(z - ez(i), g.nz) * g.ny + wrap1(y - ey(i), g.ny)) * g.pitch);
        V gi;
        if (ex(i) == 0) {
            Stor<S>::ld2(Pi + x0, gi.x, gi.y);
        } else {
            gi.x = Stor<S>::ld(Pi + (ex(i) > 0 ? xa : xb));
            gi.y = Stor<S>::ld(Pi + (ex(i) > 0 ? x0 : xc));
        }
        if (i == 0) {
            s[0] = gi;
            continue;
        }
        const int r = (ey(i) + 1) * 3 + ez(i) + 1;
        uint2 wa, wb;  // the momentum words of the two source cells
        if (ex(i) == 0) {
            wa = make_uint2(jq[r].x, jq[r].y);
            wb = make_uint2(jq[r].z, jq[r].w);
        } else if (ex(i) > 0) {
            wa = ja[r];
            wb = make_uint2(jq[r].x, jq[r].y);
        } else {  // sources xb, xc: x0 + 1 (or its copy of cell 0 for a lone last cell) and x0 + 2
            wa = make_uint2(jq[r].z, jq[r].w);
            wb = jc[r];
        }
        const V jx = make_float2(SplitJ<S>::lo(wa.x), SplitJ<S>::lo(wb.x));
        const V jy = make_float2(SplitJ<S>::hi(wa.x), SplitJ<S>::hi(wb.x));
        const V jz = make_float2(SplitJ<S>::lo(wa.y), SplitJ<S>::lo(wb.y));
        s[i] = vfma(vsplat(split_k(i)), edot_first(split_first(i), jx, jy, jz), gi);
    }
    if (FLAGS && ((m0 | m1) & 0x7fffeu)) {
        // a pair next to a solid: its bounced values are the cell's own
        // opposite ones, rebuilt from its own momentum word (row r = 4) and
        // selected over the gathered (unread) ones. Per opposite pair (i, io)
        // one e'.J of the own word serves both directions, and the pair's own
        // remainders i and io load as two aligned pair words: branch-free, and
        // 14% faster on the walled channel than a predicated scalar load per
        // bounced value.
        const V ox = make_float2(SplitJ<S>::lo(jq[4].x), SplitJ<S>::lo(jq[4].z));
        const V oy = make_float2(SplitJ<S>::hi(jq[4].x), SplitJ<S>::hi(jq[4].z));
        const V oz = make_float2(SplitJ<S>::lo(jq[4].y), SplitJ<S>::lo(jq[4].w));
#pragma unroll
        for (int p = 0; p < NPAIR; ++p) {
            const int i = pair_first(p), io = opp(i);
            const V e = edot_first(i, ox, oy, oz);
            V gi, gio;
            Stor<S>::ld2(lat_at<long long>(src, i, g.qs, c), gi.x, gi.y);
            Stor<S>::ld2(lat_at<long long>(src, io, g.qs, c), gio.x, gio.y);
            const V ri = vfma(vsplat(split_k(io)), e, gio);
            const V rio = vfma(vsplat(split_k(i)), e, gi);
            s[i].x = ((m0 >> io) & 1u) ? ri.x : s[i].x;
            s[i].y = ((m1 >> io) & 1u) ? ri.y : s[i].y;
            s[io].x = ((m0 >> i) & 1u) ? rio.x : s[io].x;
            s[io].y = ((m1 >> i) & 1u) ? rio.y : s[io].y;
        }
    }
    if (FLAGS && d.moving_on && ((m0 | m1) & MOVING_BIT)) {
        const uint2 mv = moving_links(d, c, m0, m1);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            if ((mv.x >> opp(i)) & 1u) s[i].x += wall_term<R>(d, i);
            if ((mv.y >> opp(i)) & 1u) s[i].y += wall_term<R>(d, i);
        }
    }
}

// The fused step of step_pair for the moment-split formats: the gather
// rebuilds each value from its source cell's remainder and momentum word, the
// bounce-back reload (the mask-guided form) rebuilds the cell's own opposite
// values from its own word, and the store writes the pair's momentum word,
// J = j + F (the momentum of the post-collision values: the Guo collision
// adds F), rounded, then the remainders against it.
template <int S, bool FLAGS, int FORCE, bool RECORD, bool RED = false, bool ODD = false>
__device__ __forceinline__ void step_pair_split(const Dev &d, const typename Stor<S>::T *__restrict__ src,
                                                typename Stor<S>::T *__restrict__ dst, float *__restrict__ tape,
                                                int x0, int y, int z, PairTotals<typename Stor<S>::R> *tot = nullptr) {
    typedef typename Stor<S>::T T;
    typedef float R;
    typedef float2 V;  // lane x: cell x0, lane y: cell x0 + 1
    const Geom &g = d.g;
    const bool has1 = x0 + 1 < g.nx;
    const int c = cell_index(g, x0, y, z);
    uint32_t m0 = 0u, m1 = 0u;
    bool live0 = true, live1 = has1;
    if (FLAGS) {
        const uint2 mm = ld_resident2(d.mask + c);
        m0 = mm.x;
        m1 = mm.y;
        live0 = !(m0 & SOLID_BIT);
        live1 = has1 && !(m1 & SOLID_BIT);
    }
    V s[Q];
    gather_pair_split<S, FLAGS>(d, src, x0, y, z, c, has1, m0, m1, s);
    V Fx = vsplat(R(0)), Fy = vsplat(R(0)), Fz = vsplat(R(0));
    Guo2<R> G;
    if (FORCE == 1) {
        Fx = vsplat(DevR<R>::F(d, 0));
        Fy = vsplat(DevR<R>::F(d, 1));
        Fz = vsplat(DevR<R>::F(d, 2));
        G = uniform_guo<R, false>(d);
    } else if (FORCE == 2) {
        const R *F = static_cast<const R *>(d.Ffield);
        ld2_real(F + c, Fx.x, Fx.y);
        ld2_real(F + g.qs + c, Fy.x, Fy.y);
        ld2_real(F + 2 * g.qs + c, Fz.x, Fz.y);
        G = guo2<R>(R(1) - R(0.5) * DevR<R>::omega(d), Fx, Fy, Fz);
    }
    const Mom2<R> m = moments2<R, FORCE != 0>(s, Fx, Fy, Fz, d.incomp);
    const bool bad0 = live0 && !(m.rho.x > R(0) && m.rho.x < R(1e30));
    const bool bad1 = live1 && !(m.rho.y > R(0) && m.rho.y < R(1e30));
    if (bad0 || bad1) atomicOr(d.status, LBM_STATUS_DIVERGED);
    if (RED) tot->set(m, live0, live1);
    if (RECORD) {
        const long long qs = g.qs;
        st2_real(tape + c, m.rho.x, m.rho.y);
        st2_real(tape + qs + c, m.ux.x, m.ux.y);
        st2_real(tape + 2 * qs + c, m.uy.x, m.uy.y);
        st2_real(tape + 3 * qs + c, m.uz.x, m.uz.y);
    }
    collide2<R, FORCE != 0, false>(s, m, DevR<R>::omega(d), DevR<R>::cs(d), Fx, Fy, Fz, G, d.incomp);
    // the pair's momentum word, then the remainders against the rounded J
    V Jx = m.jx, Jy = m.jy, Jz = m.jz;
    if (FORCE) {
        const V h = vsplat(R(0.5));
        Jx = vfma(h, Fx, Jx);
        Jy = vfma(h, Fy, Jy);
        Jz = vfma(h, Fz, Jz);
    }
    const unsigned w0x = SplitJ<S>::pack(Jx.x, Jy.x), w0y = SplitJ<S>::pack(Jz.x, R(0));
    const unsigned w1x = SplitJ<S>::pack(Jx.y, Jy.y), w1y = SplitJ<S>::pack(Jz.y, R(0));
    const V tx = make_float2(SplitJ<S>::lo(w0x), SplitJ<S>::lo(w1x));
    const V ty = make_float2(SplitJ<S>::hi(w0x), SplitJ<S>::hi(w1x));
    const V tz = make_float2(SplitJ<S>::lo(w0y), SplitJ<S>::lo(w1y));
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        const int i = pair_first(p), io = opp(i);
        const V e = edot_first(i, tx, ty, tz);
        s[i] = vfma(vsplat(-split_k(i)), e, s[i]);
        s[io] = vfma(vsplat(-split_k(io)), e, s[io]);
    }
    // Pairs are stored whole, a solid cell included (its values are never
    // read: the mask-guided reload rebuilds bounced values from the fluid
    // cell's own slots), so 32-byte sectors are written complete.
#pragma unroll
    for (int i = 0; i < Q; ++i) Stor<S>::st2(lat_at<long long>(dst, i, g.qs, c), s[i].x, s[i].y);
    uint2 *Jd = split_words(d, dst);
    if (!ODD || has1)
        *reinterpret_cast<uint4 *>(Jd + c) = make_uint4(w0x, w0y, w1x, w1y);
    else  // the lone last cell of an odd row: the slot after it holds cell 0's copy
        Jd[c] = make_uint2(w0x, w0y);
    if (ODD) split_ghost(d, Jd, x0, c, make_uint2(w0x, w0y));
}

// Launch every step kernel as a programmatic dependent of the kernel before it
// on its stream (the previous step, or the link form's bounce kernel): its
// blocks are scheduled as that kernel drains, and wait for it to complete
// before their first load. Measured: the link form's chain +1%; FP32 steps
// +0.5% when launched one by one (short runs), +0.2% in replayed graphs.
constexpr int STEP_PDL = 1;

// Block shape of the step kernel: the flat launch's blocks hold 128 threads at
// most (256 where wide_blocks_fit), whole rows 256. Blocks of 128 per SM, and what was measured (us a step):
//  - FP32 with flags (32-bit offsets): 7 (72 registers, no spills: 28 warps)
//    +1.1% on the walled channel over 3 of 256 (80 registers); 4 of 256 (64)
//    spilled 48 bytes and lost 4%. A force per cell: 6 (80), channel 97.2 to 94.2.
//  - moment split with flags: 7, BF16 channel 90.4 against 100.7 with 6; without
//    flags 6, BF16 384^3 960 against 1030.
//  - 16-bit: 8 (64); with a force per cell 6 (80), 200^3 FP16 117.5 against 125.4,
//    porous channel (whole rows, 3 of 256), recorded, 430 against 484.
template <bool FLAT, int S, bool FLAGS> constexpr int step_threads() {
    return FLAT && !wide_blocks_fit(S, FLAGS) ? 128 : 256;
}
template <int S, bool FLAGS, int FORCE, bool FLAT, bool U32, bool RED = false> constexpr int step_min_blocks() {
    const int rows = FORCE == 2 && StepBlocks<S>::value == 4 ? 3 : StepBlocks<S>::value;
    if (!FLAT || wide_blocks_fit(S, FLAGS)) return rows;
    if (U32 || (is_split(S) && FLAGS && !RED)) return FORCE == 2 ? 6 : 7;
    return 2 * rows;
}

// FLAT: the launch of d.PF (pairs in plane order), else of d.P (whole rows).
// ODD (moment-split formats only): rows of odd length, whose last cell is
// alone in its pair (see split_ghost). U32: 32-bit lattice offsets (lat_at).
template <int S, bool FLAGS, int FORCE, bool RECORD, bool FLAT = false, bool ODD = false, bool U32 = false>
__global__ void __launch_bounds__(step_threads<FLAT, S, FLAGS>(), step_min_blocks<S, FLAGS, FORCE, FLAT, U32>())
    k_step(const Dev d, const typename Stor<S>::T *__restrict__ src, typename Stor<S>::T *__restrict__ dst,
           typename Stor<S>::R *__restrict__ tape) {
    // launched as a programmatic dependent: wait for the kernel before it (the
    // previous step, or a bounce kernel whose links land in src) to complete
    // (a no-op when launched normally)
    if (STEP_PDL) asm volatile("griddepcontrol.wait;" ::: "memory");
    // let the next kernel (the bounce kernel, or the next step) be scheduled
    // once every block of this grid is running; it still waits for this grid
    // to complete before it reads what this grid writes
    if (STEP_PDL) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // blocks are dispatched in index order: with d.zrev the planes run from
    // the last to the first. (The BF16 split step keeps ascending order: with
    // the reversal its code schedules worse, 35.5 against 36.8 GFLUPS on the
    // walled channel at the same spills, while the FP16 split one gains 1.3%.)
    constexpr bool REV = S != LBM_BF16M;
    const int bz = REV && d.zrev ? (int)gridDim.y - 1 - (int)blockIdx.y : (int)blockIdx.y;
    int x0, y, z;
    if (!pair_cell<FLAT>(d.g, FLAT ? d.PF : d.P, blockDim.x, blockDim.y, blockIdx.x, bz, threadIdx.x, threadIdx.y,
                         x0, y, z))
        return;
    if constexpr (is_split(S))
        step_pair_split<S, FLAGS, FORCE, RECORD, false, ODD>(d, src, dst, tape, x0, y, z);
    else if constexpr (U32)
        step_pair<S, FLAGS, FORCE, RECORD, GlobalRows<S, unsigned>, false, unsigned>(
            d, GlobalRows<S, unsigned>{src}, src, dst, tape, x0, y, z);
    else
        step_pair<S, FLAGS, FORCE, RECORD>(d, GlobalRows<S>{src}, src, dst, tape, x0, y, z);
}

// The step with the mass/momentum totals of its pre-collision state fused in
// (the reduction of lbm_reduce without a pass of its own): every thread, in
// the lattice or not, reaches the block reduction; partials[4 b + k] of block
// b = blockIdx.y * gridDim.x + blockIdx.x, summed in a fixed order.
template <int S, bool FLAGS, int FORCE, bool FLAT, bool ODD = false>
__global__ void __launch_bounds__(step_threads<FLAT, S, FLAGS>(), step_min_blocks<S, FLAGS, FORCE, FLAT, false, true>())
    k_step_reduce(const Dev d, const typename Stor<S>::T *__restrict__ src, typename Stor<S>::T *__restrict__ dst,
                  double *__restrict__ partials) {
    if (FLAGS && LinkBounce<S>::value) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    PairTotals<typename Stor<S>::R> tot;
    tot.clear();
    int x0, y, z;
    if (pair_cell<FLAT>(d.g, FLAT ? d.PF : d.P, blockDim.x, blockDim.y, blockIdx.x, blockIdx.y, threadIdx.x,
                        threadIdx.y, x0, y, z)) {
        if constexpr (is_split(S))
            step_pair_split<S, FLAGS, FORCE, false, true, ODD>(d, src, dst, nullptr, x0, y, z, &tot);
        else
            step_pair<S, FLAGS, FORCE, false, GlobalRows<S>, true>(d, GlobalRows<S>{src}, src, dst, nullptr, x0, y,
                                                                  z, &tot);
    }
    block_partials(tot, partials, blockIdx.y * gridDim.x + blockIdx.x);
}

// ---------------------------------------------------------------------------
// The fused step in FP64 storage, one cell a thread (a warp's 8-byte loads of
// 32 consecutive cells fill whole lines): gather with the mask-guided reload,
// moments and collision in fixed point (lbm_fixed.cuh), store whole sectors
// (a solid cell stores zeros nobody reads). Threads take the cells of the
// fluid box's rows in order, across row ends. I: 32-bit lattice offsets where
// they fit. RED: also the totals of the pre-collision state, per block. 5 blocks
// of 128 threads per SM (<= 102 registers): channel 312 us a step, against 332
// with 2 of 256 (125 registers) and 322 with 4 of 128 (280 now, with the integer
// instructions of lbm_fixed.cuh as they are).
template <bool FLAGS, int FORCE, bool RECORD, bool RED, class I>
__global__ void __launch_bounds__(128, 5)
    k_step64(const Dev d, const double *__restrict__ src, double *__restrict__ dst, double *__restrict__ out) {
    // (as k_step: a programmatic dependent of the kernel before it)
    if (STEP_PDL) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (STEP_PDL) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const Geom &g = d.g;
    const int bz = d.zrev ? (int)gridDim.y - 1 - (int)blockIdx.y : (int)blockIdx.y;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = k / g.nx;
    PairTotals<double> tot;
    if (RED) tot.clear();
    if (r < d.P.nyr) {
        const int x = k - r * g.nx, y = d.P.y0 + r, z = d.P.z0 + bz;
        const int c = cell_index(g, x, y, z);
        const uint32_t m = FLAGS ? __ldg(d.mask + c) : 0u;
        const bool live = !(m & SOLID_BIT);
        const int xa = wrap1(x - 1, g.nx), xb = wrap1(x + 1, g.nx);
        double s[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i)
            s[i] = __ldg(GlobalRows<LBM_F64, I>{src}.row(g, i, y, z) + (ex(i) == 0 ? x : (ex(i) > 0 ? xa : xb)));
        if (FLAGS && live && (m & 0x7fffeu)) {
            // bounced populations come from the cell's own opposite slots
#pragma unroll
            for (int i = 1; i < Q; ++i)
                if ((m >> opp(i)) & 1u) s[i] = __ldg(lat_at<I>(src, opp(i), g.qs, c));
            if (d.moving_on && (m & MOVING_BIT)) {
                const uint32_t mv = __ldg(d.moving + c);
#pragma unroll
                for (int i = 1; i < Q; ++i)
                    if ((mv >> opp(i)) & 1u) s[i] += d.wc[i];
            }
        }
        if (!FLAGS || live) {
            double Fx = 0.0, Fy = 0.0, Fz = 0.0;
            if (FORCE == 1) {
                Fx = d.F[0];
                Fy = d.F[1];
                Fz = d.F[2];
            } else if (FORCE == 2) {
                const double *F = static_cast<const double *>(d.Ffield);
                Fx = __ldg(F + c);
                Fy = __ldg(F + g.qs + c);
                Fz = __ldg(F + 2 * g.qs + c);
            }
            Cell64 mo;
            cell64<FORCE != 0, true, RECORD || RED>(d, s, Fx, Fy, Fz, mo);
            if (!(mo.rho > 0.0 && mo.rho < 1e30)) atomicOr(d.status, LBM_STATUS_DIVERGED);
            if (RECORD) {
                __stcs(out + c, mo.rho);
                __stcs(out + g.qs + c, mo.ux);
                __stcs(out + 2 * g.qs + c, mo.uy);
                __stcs(out + 3 * g.qs + c, mo.uz);
            }
            if (RED) {
                tot.v[0].x = mo.rho1;
                tot.v[1].x = mo.jx;
                tot.v[2].x = mo.jy;
                tot.v[3].x = mo.jz;
                tot.cells = 1;
            }
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) *lat_at<I>(dst, i, g.qs, c) = !FLAGS || live ? s[i] : 0.0;
    }
    if (RED) block_partials(tot, out, blockIdx.y * gridDim.x + blockIdx.x);
}

// ---------------------------------------------------------------------------
// The step with its source rows staged in shared memory by the Tensor Memory
// Accelerator (FP32 and 16-bit storage). A cell row (y, z) pulls population
// i from the one row (y - e_iy, z - e_iz) of array i, shifted by e_ix, so a
// block that updates whole cell rows needs exactly 19 source rows per row.
// One thread issues them as 1-D bulk asynchronous copies (cp.async.bulk,
// whole padded rows: 16-byte aligned, sizes a multiple of 16 bytes) that
// signal an mbarrier with their byte count; the block computes row k from one
// buffer while the copies of row k + 1 land in the other. The loads are thus
// in flight without holding registers. The gathered values, the arithmetic
// (step_pair) and the stores are the same as in k_step, so both give the
// same bits. Opt-in (lbm_options.stage_rows): measured against the direct
// kernel it gains 1-4% on 16-bit lattices without obstacles, and loses on
// walled ones, where the block barrier per row exposes the latency of the
// bounce-back reloads that the direct kernel hides behind other warps.
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
// Wait for the phase with the given parity to complete, for at most ~1 s.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > (1LL << 31)) return false;
    return true;
}
__device__ __forceinline__ void bulk_copy_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// Order this thread's earlier shared-memory accesses (and the block's, after
// a barrier) before later asynchronous-proxy writes to the same memory.
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// The 19 source rows of cell row r into buf [Q][pitch], counted on bar.
// Row r of the fluid box (see pair_launch) as (y, z).
__device__ __forceinline__ void box_row(const RowLaunch &P, int r, int &y, int &z) {
    y = P.y0 + r % P.nyr;
    z = P.z0 + r / P.nyr;
}

template <int S>
__device__ __forceinline__ void issue_source_rows(const Geom &g, const RowLaunch &P, const typename Stor<S>::T *src,
                                                  typename Stor<S>::T *buf, uint64_t *bar, int r, uint32_t rowbytes) {
    int y, z;
    box_row(P, r, y, z);
    mbar_arrive_expect_tx(bar, (uint32_t)Q * rowbytes);
#pragma unroll 1
    for (int i = 0; i < Q; ++i) {
        const long long row = (long long)(wrap1(z - ez(i), g.nz) * g.ny + wrap1(y - ey(i), g.ny)) * g.pitch;
        bulk_copy_g2s(buf + i * g.pitch, src + (long long)i * g.qs + row, rowbytes, bar);
    }
}

template <int S, bool FLAGS, int FORCE, bool RECORD>
__global__ void __launch_bounds__(512)
    k_step_tma(const Dev d, const typename Stor<S>::T *__restrict__ src, typename Stor<S>::T *__restrict__ dst,
               typename Stor<S>::R *__restrict__ tape) {
    typedef typename Stor<S>::T T;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const Geom &g = d.g;
    const uint32_t rowbytes = (uint32_t)g.pitch * (uint32_t)sizeof(T);
    T *buf = reinterpret_cast<T *>(smem_raw);  // [2][Q][pitch]
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw + 2 * Q * rowbytes);
    const int nrows = d.P.nyr * d.P.nzr;  // the rows of the fluid box
    const int t = threadIdx.x, stride = gridDim.x;
    if (t == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 1, 1);
        fence_mbar_init();
    }
    __syncthreads();
    int r = blockIdx.x;
    if (t == 0) {
        if (r < nrows) issue_source_rows<S>(g, d.P, src, buf, bar, r, rowbytes);
        if (r + stride < nrows) issue_source_rows<S>(g, d.P, src, buf + Q * g.pitch, bar + 1, r + stride, rowbytes);
    }
    const int pairs = (g.nx + 1) >> 1;
    for (int k = 0; r < nrows; ++k, r += stride) {
        const int b = k & 1;
        const bool ok = mbar_wait_bounded(bar + b, (k >> 1) & 1);
        if (__syncthreads_or(!ok)) {
            // copies that never completed: report, give the other buffer's
            // copies a bounded chance to land, and leave. If that second
            // wait runs out too, the block exits with bulk copies still
            // addressed to its shared memory; there is no way to cancel them,
            // and an SM that later reuses that shared memory for another
            // block could see it overwritten. This path has never been
            // observed (no test forces it, nor may one: forcing it means a
            // copy that never completes); the status word tells the caller to
            // discard the run. The kernel is opt-in (lbm_options.stage_rows).
            if (t == 0) {
                atomicOr(d.status, LBM_STATUS_TIMEOUT);
                mbar_wait_bounded(bar + (b ^ 1), ((k + 1) >> 1) & 1);
            }
            return;
        }
        int y, z;
        box_row(d.P, r, y, z);
        const SharedRows<S> rows{buf + b * Q * g.pitch};
        for (int p = t; p < pairs; p += blockDim.x) step_pair<S, FLAGS, FORCE, RECORD>(d, rows, src, dst, tape, 2 * p, y, z);
        __syncthreads();  // every read of buffer b is done
        if (t == 0 && r + 2 * stride < nrows) {
            fence_async_shared();
            issue_source_rows<S>(g, d.P, src, buf + b * Q * g.pitch, bar + b, r + 2 * stride, rowbytes);
        }
    }
}

// Bounce-back links (separate-kernel form): for each fluid cell x and
// direction j with x + e_j solid and at rest, slot opp(j) of the solid cell
// receives the post-collision population j of x, copied bit for bit (links
// into moving walls are written by the step kernel). Links are grouped by
// direction (blockIdx.x + 1) and ordered by cell within a direction. Every
// direction's links are cut into gridDim.y equal spans, block (j, b) taking
// span b of direction j: blocks are dispatched span by span across the 18
// directions, so the kernel sweeps the planes once, against the order of the
// step before it, and ends on the planes the next step starts with (FP16
// channel 45.9 GFLUPS; sweeping in the step's own order 44.2, and one sweep
// per direction 45.6).
// Each thread copies LINKS_PER_THREAD links (256 apart, so index loads stay
// coalesced); all index loads are issued before the value loads, and all value
// loads before the stores, so the two dependent round trips are shared.
constexpr int LINKS_PER_THREAD = 4;
static_assert(256 * LINKS_PER_THREAD == BOUNCE_LINKS_PER_BLOCK, "k_bounce block size");
constexpr int BOUNCE_SWEEP_OPPOSITE = 1;
// Launch k_bounce as a programmatic dependent of the step kernel.
constexpr int BOUNCE_PDL = 1;

template <int S>
__global__ void __launch_bounds__(256) k_bounce(const Dev d, typename Stor<S>::T *__restrict__ P) {
    typedef typename Stor<S>::T T;
    const int j = blockIdx.x + 1;
    const int base = d.link_off[j];
    const int nb = (int)gridDim.y;
    const int b = (d.zrev ^ BOUNCE_SWEEP_OPPOSITE) ? nb - 1 - (int)blockIdx.y : (int)blockIdx.y;
    const int nj = d.link_off[j + 1] - base;
    const int span = (nj + nb - 1) / nb;  // <= blockDim.x * LINKS_PER_THREAD: nb spans the largest direction
    const int k0 = b * span + threadIdx.x;
    const int n = min(nj, (b + 1) * span);  // end of this block's span
    const uint2 *L = reinterpret_cast<const uint2 *>(d.links) + base;
    const T *from = P + (long long)j * d.g.qs;
    T *to = P + (long long)opp(j) * d.g.qs;
    uint2 l[LINKS_PER_THREAD];
    T v[LINKS_PER_THREAD];
#pragma unroll
    for (int r = 0; r < LINKS_PER_THREAD; ++r) {
        const int k = k0 + r * blockDim.x;
        l[r] = k < n ? ld_resident2(reinterpret_cast<const uint32_t *>(L + k)) : make_uint2(0u, 0u);  // (fluid, solid)
    }
    // Launched as a programmatic dependent of the step kernel: the links above
    // do not depend on it, the values below do. Wait here for the step's grid
    // to complete (a no-op when launched normally).
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // the next step kernel may be scheduled from here on: no earlier, so that
    // it cannot start before the step this kernel waited for has completed
    if (STEP_PDL) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#pragma unroll
    for (int r = 0; r < LINKS_PER_THREAD; ++r)
        if (k0 + r * blockDim.x < n) v[r] = from[l[r].x];
#pragma unroll
    for (int r = 0; r < LINKS_PER_THREAD; ++r)
        if (k0 + r * blockDim.x < n) to[l[r].y] = v[r];
}

// ---------------------------------------------------------------------------
// Readers and writers of the whole lattice run on the flat paired launch over
// all rows (solid ones too): two x-adjacent cells per thread, d.PF.
inline RowLaunch all_pairs(const Geom &g) {
    const RowLaunch rows = pair_launch(g);
    return flat_launch(rows, flat_threads(rows));
}
inline dim3 pairs_grid(const RowLaunch &P) { return dim3(P.nyb, P.nzr); }

// The push masks of the pair at cell c, 0 for a cell that is solid or past the
// row's end, and which of the two cells are fluid.
template <bool FLAGS>
__device__ __forceinline__ void pair_masks(const Dev &d, int c, bool has1, uint32_t &m0, uint32_t &m1, bool &live0,
                                           bool &live1) {
    m0 = m1 = 0u;
    live0 = true;
    live1 = has1;
    if (FLAGS) {
        const uint2 mm = ld_resident2(d.mask + c);
        live0 = !(mm.x & SOLID_BIT);
        live1 = has1 && !(mm.y & SOLID_BIT);
        m0 = live0 ? mm.x : 0u;
        m1 = live1 ? mm.y : 0u;
    }
}

// The 19 pre-collision values of the fluid cells of the pair (x0, x0 + 1) of row
// (y, z), from P in the layout d.layout: every value is loaded from its source,
// and pairs next to a solid (m0, m1: their push masks) then load their bounced
// values over it. In the link form a solid source's slot already holds the
// bounced value (what the next step will read); the AA swapped layout is the
// pull layout with slot i and slot opp(i) exchanged. (One mask word a cell
// instead of 18 flag bytes, and loads that do not wait for them.)
template <int S, bool FLAGS>
__device__ __forceinline__ void gather_pair(const Dev &d, const typename Stor<S>::T *__restrict__ P, int x0, int y,
                                            int z, int c, bool has1, uint32_t m0, uint32_t m1,
                                            typename Pair2<typename Stor<S>::R>::V s[Q]) {
    typedef typename Stor<S>::T T;
    typedef typename Stor<S>::R R;
    const Geom &g = d.g;
    if constexpr (is_split(S)) {
        gather_pair_split<S, FLAGS>(d, P, x0, y, z, c, has1, m0, m1, s);
        return;
    } else {
        if (d.layout == LAYOUT_AA_NAT) {
#pragma unroll
            for (int i = 0; i < Q; ++i) Stor<S>::ld2(P + (long long)i * g.qs + c, s[i].x, s[i].y);
            return;
        }
        const bool mirror = d.layout == LAYOUT_AA_SWAP;
        const int xa = wrap1(x0 - 1, g.nx), xb = wrap1(x0 + 1, g.nx);
        const int xc = has1 ? wrap1(x0 + 2, g.nx) : x0;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const T *Pi = P + (mirror ? opp(i) : i) * g.qs +
                          (wrap1(z - ez(i), g.nz) * g.ny + wrap1(y - ey(i), g.ny)) * g.pitch;
            if (ex(i) == 0) {
                Stor<S>::ld2(Pi + x0, s[i].x, s[i].y);
            } else {
                s[i].x = Stor<S>::ld(Pi + (ex(i) > 0 ? xa : xb));
                s[i].y = Stor<S>::ld(Pi + (ex(i) > 0 ? x0 : xc));
            }
        }
        // (the link form's solid slots hold the bounced values already)
        if (FLAGS && !(bounce_in_solid(S) && !mirror) && ((m0 | m1) & 0x7fffeu)) {
            forget(c);
#pragma unroll
            for (int i = 1; i < Q; ++i) {
                const T *Po = P + (mirror ? i : opp(i)) * g.qs + c;
                if ((m0 >> opp(i)) & 1u) s[i].x = Stor<S>::ld(Po);
                if ((m1 >> opp(i)) & 1u) s[i].y = Stor<S>::ld(Po + 1);
            }
            if (d.moving_on && ((m0 | m1) & MOVING_BIT)) {
                const uint2 mv = moving_links(d, c, m0, m1);
#pragma unroll
                for (int i = 1; i < Q; ++i) {
                    if ((mv.x >> opp(i)) & 1u) s[i].x += wall_term<R>(d, i);
                    if ((mv.y >> opp(i)) & 1u) s[i].y += wall_term<R>(d, i);
                }
            }
        }
    }
}

// Resident pairs of 128-thread blocks per SM of the readers and writers, the
// measured best of 2 and 3: FP64 2 (3 spilled: get_state of the channel 210
// against 343 us), moment-split storage with flags 2 (macros 101 against 148
// us), else 3 (FP16 channel, macros 65 against 75 us, set_state 95 against
// 133); set_state with flags takes 7 single blocks (82.4 against 91).
template <int S, bool FLAGS> struct FieldBlocks {
    static constexpr int value = S == LBM_F64 ? 2 : (FLAGS && is_split(S) ? 2 : 3);
};

// ---------------------------------------------------------------------------
// Initial state: P^{-1}_i(y) = f_eq_i at y + e_i if that cell is fluid, else
// f_eq_{opp(i)}(y) (so that the gather yields f^0 = f_eq(rho0, u0)), stored
// shifted by -w_i. Each fluid cell x forms its own 19 values once and pushes
// them: f_eq_i(x) to slot i of x - e_i, and f_eq_opp(i)(x) to its own slot i
// where x + e_i is solid. A solid x - e_i takes its push too: in the link form
// that is the value its slot must hold, and in the others nobody reads it.
// Bound by HBM (4 reals read and 19 values written a cell); every cell forming
// the values of its 18 neighbours was bound by their 76 loads and by arithmetic
// (FP64: its pipe 85% busy). Whole call, channel: FP32 195 to 131 us (floor 57), FP16
// 197 to 94, FP64 2373 to 306; 256^3 box, FP32 440 to 248 us (floor 227).
// f_eq - w of the two cells of a pair: per direction one expression,
// w (rho1 + rho (3 e.u + 9/2 (e.u)^2 - 3/2 u.u)), its roundings in this order. (The even
// and odd parts of opposite directions formed once take 8 operations a pair of them
// instead of 11 and are as accurate, but differ in the last FP32 bit, which the 16-bit
// formats turn into a whole storage step of the initial state. On packed cells this
// order costs no time: 256^3 box FP32 260 to 250 us, FP16 219 to 216, channel FP16
// 99 to 94, FP32 127 to 132.)
__device__ __forceinline__ void feq2(float2 f[Q], float2 rho1, float2 ux, float2 uy, float2 uz, bool incomp) {
    const float2 rho = incomp ? vsplat(1.0f) : vadd(vsplat(1.0f), rho1);
    const float2 usq = vfma(uz, uz, vfma(ux, ux, vmul(uy, uy)));
    f[0] = vmul(vsplat((float)(1.0 / 3.0)), vfma(rho, vmul(vsplat(-1.5f), usq), rho1));
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        const int i = pair_first(p);
        const float2 w = vsplat(i <= 6 ? (float)(1.0 / 18.0) : (float)(1.0 / 36.0));
        const float2 eu = edot_first(i, ux, uy, uz), sq = vmul(vmul(vsplat(4.5f), eu), eu);
        f[i] = vmul(w, vfma(rho, vfma(vsplat(-1.5f), usq, vfma(vsplat(3.0f), eu, sq)), rho1));
        f[opp(i)] = vmul(w, vfma(rho, vfma(vsplat(-1.5f), usq, vfma(vsplat(-3.0f), eu, sq)), rho1));
    }
}

// The same of one cell in FP64.
__device__ __forceinline__ void feq64(double f[Q], double rho1, double ux, double uy, double uz, bool incomp) {
    const double rho = incomp ? 1.0 : 1.0 + rho1, usq = fma(uz, uz, fma(ux, ux, uy * uy));
    f[0] = (1.0 / 3.0) * fma(rho, -1.5 * usq, rho1);
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        const int i = pair_first(p);
        const double w = i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0, eu = ex(i) * ux + ey(i) * uy + ez(i) * uz, sq = 4.5 * eu * eu;
        f[i] = w * fma(rho, fma(-1.5, usq, fma(3.0, eu, sq)), rho1);
        f[opp(i)] = w * fma(rho, fma(-1.5, usq, fma(-3.0, eu, sq)), rho1);
    }
}

// Store the remainders g of a cell pair and its momentum words wa, wb.
template <int S>
__device__ __forceinline__ void split_put_pair(const Dev &d, typename Stor<S>::T *__restrict__ P, int x0, int c,
                                               bool has1, const float2 g[Q], uint2 wa, uint2 wb) {
#pragma unroll
    for (int i = 0; i < Q; ++i) Stor<S>::st2(P + i * d.g.qs + c, g[i].x, g[i].y);
    uint2 *J = split_words(d, P);
    if (has1)
        *reinterpret_cast<uint4 *>(J + c) = make_uint4(wa.x, wa.y, wb.x, wb.y);
    else  // the lone last cell of an odd row: the slot after it holds cell 0's copy
        J[c] = wa;
    split_ghost(d, J, x0, c, wa);
}

// Write the 19 shifted values v of a cell pair to a moment-split lattice:
// their momentum rounded to the format, then the remainders against it (the
// tail of step_pair_split, for values that are not a collision's).
template <int S>
__device__ __forceinline__ void split_store_pair(const Dev &d, typename Stor<S>::T *__restrict__ P, int x0, int c,
                                                 bool has1, float2 v[Q]) {
    const float2 jx = vadd(vadd(vadd(vsub(v[1], v[2]), vsub(v[7], v[10])), vadd(vsub(v[8], v[9]), vsub(v[11], v[14]))),
                           vsub(v[12], v[13]));
    const float2 jy = vadd(vadd(vadd(vsub(v[3], v[4]), vsub(v[7], v[10])), vadd(vsub(v[9], v[8]), vsub(v[15], v[18]))),
                           vsub(v[16], v[17]));
    const float2 jz = vadd(vadd(vadd(vsub(v[5], v[6]), vsub(v[11], v[14])), vadd(vsub(v[13], v[12]), vsub(v[15], v[18]))),
                           vsub(v[17], v[16]));
    const uint2 wa = make_uint2(SplitJ<S>::pack(jx.x, jy.x), SplitJ<S>::pack(jz.x, 0.0f));
    const uint2 wb = make_uint2(SplitJ<S>::pack(jx.y, jy.y), SplitJ<S>::pack(jz.y, 0.0f));
    const float2 tx = make_float2(SplitJ<S>::lo(wa.x), SplitJ<S>::lo(wb.x));
    const float2 ty = make_float2(SplitJ<S>::hi(wa.x), SplitJ<S>::hi(wb.x));
    const float2 tz = make_float2(SplitJ<S>::lo(wa.y), SplitJ<S>::lo(wb.y));
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        const int i = pair_first(p), io = opp(i);
        const float2 e = edot_first(i, tx, ty, tz);
        v[i] = vfma(vsplat(-split_k(i)), e, v[i]);
        v[io] = vfma(vsplat(-split_k(io)), e, v[io]);
    }
    split_put_pair<S>(d, P, x0, c, has1, v, wa, wb);
}

// a + b rounded to odd: exact if a float holds the sum, else the neighbour with an odd
// last bit. Rounding that to 16 bits gives the sum rounded once.
__device__ __forceinline__ float odd_of(float down, float up) { return __float_as_uint(down) & 1u ? down : up; }
__device__ __forceinline__ float2 odd_add(float2 a, float2 b) {
    return make_float2(odd_of(__fadd_rd(a.x, b.x), __fadd_ru(a.x, b.x)), odd_of(__fadd_rd(a.y, b.y), __fadd_ru(a.y, b.y)));
}
__device__ __forceinline__ float2 odd_fma(float k, float2 a, float2 b) {
    return make_float2(odd_of(__fmaf_rd(k, a.x, b.x), __fmaf_ru(k, a.x, b.x)),
                       odd_of(__fmaf_rd(k, a.y, b.y), __fmaf_ru(k, a.y, b.y)));
}
// A sum of floats and the sum of its roundings.
struct Sum2 {
    float2 s, e;
    // (Knuth's two-sum: b's part of the rounded sum, then what both lost)
    __device__ __forceinline__ void add(float2 b) {
        const float2 t = vadd(s, b), v = vsub(t, s);
        e = vadd(e, vadd(vsub(s, vsub(t, v)), vsub(b, v)));
        s = t;
    }
};
__device__ __forceinline__ Sum2 operator-(float2 a, float2 b) {
    Sum2 r = {a, vsplat(0.0f)};
    r.add(vmul(b, vsplat(-1.0f)));
    return r;
}
__device__ __forceinline__ Sum2 operator+(Sum2 a, Sum2 b) {
    a.add(b.s);
    a.e = vadd(a.e, b.e);
    return a;
}
__device__ __forceinline__ Sum2 operator-(Sum2 a) { return Sum2{vmul(a.s, vsplat(-1.0f)), vmul(a.e, vsplat(-1.0f))}; }

// The same from values of a canonical state, which is exchanged unrounded: the
// momentum and the remainders are each rounded once, to 16 bits, as split_store
// rounds them from double (in FP32, twice). FP64 adds would take 2.5 ms for a 256^3
// box, which moves in 0.3.
template <int S>
__device__ __forceinline__ void split_store_pair_once(const Dev &d, typename Stor<S>::T *__restrict__ P, int x0, int c,
                                                      bool has1, float2 v[Q]) {
    const Sum2 a = v[7] - v[10], b = v[8] - v[9], e = v[11] - v[14], f = v[12] - v[13], g = v[15] - v[18],
               h = v[16] - v[17];
    const Sum2 jx = (v[1] - v[2]) + a + b + e + f, jy = (v[3] - v[4]) + a + -b + g + h,
               jz = (v[5] - v[6]) + e + -f + g + -h;
    const float2 ox = odd_add(jx.s, jx.e), oy = odd_add(jy.s, jy.e), oz = odd_add(jz.s, jz.e);
    const uint2 wa = make_uint2(SplitJ<S>::pack(ox.x, oy.x), SplitJ<S>::pack(oz.x, 0.0f));
    const uint2 wb = make_uint2(SplitJ<S>::pack(ox.y, oy.y), SplitJ<S>::pack(oz.y, 0.0f));
    const float2 tx = make_float2(SplitJ<S>::lo(wa.x), SplitJ<S>::lo(wb.x));
    const float2 ty = make_float2(SplitJ<S>::hi(wa.x), SplitJ<S>::hi(wb.x));
    const float2 tz = make_float2(SplitJ<S>::lo(wa.y), SplitJ<S>::lo(wb.y));
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        const int i = pair_first(p), io = opp(i);
        const float2 w = edot_first(i, tx, ty, tz);
        v[i] = odd_fma(-split_k(i), w, v[i]);
        v[io] = odd_fma(-split_k(io), w, v[io]);
    }
    split_put_pair<S>(d, P, x0, c, has1, v, wa, wb);
}

// f_eq_i - w_i of two cells.
__device__ __forceinline__ float2 feq_pair(int i, float2 r1, float2 ux, float2 uy, float2 uz, bool incomp) {
    const float2 rho = incomp ? vsplat(1.0f) : vadd(vsplat(1.0f), r1);
    const float2 usq = vmul(vsplat(-1.5f), vfma(uz, uz, vfma(uy, uy, vmul(ux, ux))));
    const float w = i == 0 ? (float)(1.0 / 3.0) : (i <= 6 ? (float)(1.0 / 18.0) : (float)(1.0 / 36.0));
    if (i == 0) return vmul(vsplat(w), vfma(rho, usq, r1));
    // (the odd part joins in one rounding, with the momentum-exact 3 w of OddK)
    const float2 e = edot_first(split_first(i), ux, uy, uz);
    const float2 even = vmul(vsplat(w), vfma(rho, vfma(vmul(vsplat(4.5f), e), e, usq), r1));
    return vfma(vmul(vsplat(split_k(i)), rho), e, even);
}

// Moment-split storage: the 19 values that the cells of a pair hold, formed from
// their neighbours' fields (row by row: the pair and the cells left and right of
// it), written as J and remainders. 256^3 box 378 us (floor 152), 399 with 6
// blocks per SM; one cell a thread with 76 field loads took 511. Walled channel
// with 5 blocks 137 us, 155 with 4.
template <int S, bool FLAGS>
__global__ void __launch_bounds__(128, FLAGS ? 5 : 7)
    k_init_eq_split(const Dev d, typename Stor<S>::T *__restrict__ P, const float *__restrict__ rho0,
                    const float *__restrict__ u0, bool pair) {
    const Geom &g = d.g;
    int x0, y, z;
    if (!pair_cell<true>(g, d.PF, blockDim.x, blockDim.y, blockIdx.x, blockIdx.y, threadIdx.x, threadIdx.y, x0, y, z))
        return;
    const bool has1 = x0 + 1 < g.nx;
    const int c = cell_index(g, x0, y, z);
    uint32_t m0, m1;
    bool live0, live1;
    pair_masks<FLAGS>(d, c, has1, m0, m1, live0, live1);
    if (FLAGS && !live0 && !live1) return;
    const long long N = d.n_cells;
    const int xa = wrap1(x0 - 1, g.nx), xb = wrap1(x0 + 1, g.nx), xc = wrap1(xb + 1, g.nx);
    float2 v[Q];
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        const int dy = r / 3 - 1, dz = r % 3 - 1;
        const int row = (wrap1(z + dz, g.nz) * g.ny + wrap1(y + dy, g.ny)) * g.nx;
        float2 f[4];  // rho - 1, u of cells x0, x0 + 1
        float fa[4], fc[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            f[k] = vsplat(1.0f);
            fa[k] = fc[k] = 1.0f;
            if (k == 0 && !rho0) continue;
            const float *p = (k ? u0 + (k - 1) * N : rho0) + row;
            if (pair) {
                ld2_real(p + x0, f[k].x, f[k].y);
            } else {
                f[k].x = __ldg(p + x0);
                f[k].y = __ldg(p + xb);
            }
            if (dy == 0 || dz == 0) {
                fa[k] = __ldg(p + xa);
                fc[k] = __ldg(p + xc);
            }
        }
        f[0] = vadd(f[0], vsplat(-1.0f));
        fa[0] -= 1.0f;
        fc[0] -= 1.0f;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            if (ey(i) != dy || ez(i) != dz) continue;
            float2 q[4];  // the fields of x + e_i
#pragma unroll
            for (int k = 0; k < 4; ++k)
                q[k] = ex(i) == 0 ? f[k] : (ex(i) > 0 ? make_float2(f[k].y, fc[k]) : make_float2(fa[k], f[k].x));
            v[i] = feq_pair(i, q[0], q[1], q[2], q[3], d.incomp);
        }
    }
    if (FLAGS && ((m0 | m1) & 0x7fffeu)) {  // next to a solid: the cell's own opposite value
        const long long cc = canon_index(g, x0, y, z);
        float2 f[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            f[k] = vsplat(1.0f);
            if (k || rho0) get2<LBM_F32>((k ? u0 + (k - 1) * N : rho0) + cc, false, has1, f[k].x, f[k].y);
        }
        f[0] = vadd(f[0], vsplat(-1.0f));
        const uint2 mv = d.moving_on && ((m0 | m1) & MOVING_BIT) ? moving_links(d, c, m0, m1) : make_uint2(0u, 0u);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            float2 o = feq_pair(opp(i), f[0], f[1], f[2], f[3], d.incomp);
            if ((mv.x >> i) & 1u) o.x += d.wcf[i];
            if ((mv.y >> i) & 1u) o.y += d.wcf[i];
            if ((m0 >> i) & 1u) v[i].x = o.x;
            if ((m1 >> i) & 1u) v[i].y = o.y;
        }
    }
    split_store_pair<S>(d, P, x0, c, has1, v);
}

template <int S, bool FLAGS>
__global__ void __launch_bounds__(128, 2 * FieldBlocks<S, FLAGS>::value)
    k_init_eq(const Dev d, typename Stor<S>::T *__restrict__ P, const typename Stor<S>::R *__restrict__ rho0,
              const typename Stor<S>::R *__restrict__ u0, bool pair) {
    typedef typename Stor<S>::R R;
    typedef typename Stor<S>::T T;
    constexpr int RF = sizeof(R) == 8 ? LBM_F64 : LBM_F32;  // canonical format of R
    const Geom &g = d.g;
    // (whole warps stay to the end: neighbouring lanes exchange values)
    int x0, y, z;
    const bool in = pair_cell<true>(g, d.PF, blockDim.x, blockDim.y, blockIdx.x, blockIdx.y, threadIdx.x, threadIdx.y,
                                    x0, y, z);
    const bool has1 = x0 + 1 < g.nx;
    const int c = in ? cell_index(g, x0, y, z) : 0;
    const long long N = d.n_cells, cc = canon_index(g, x0, y, z);
    uint32_t m0 = 0u, m1 = 0u;
    bool live0 = false, live1 = false;
    R r[2] = {R(1), R(1)}, ux[2] = {R(0), R(0)}, uy[2] = {R(0), R(0)}, uz[2] = {R(0), R(0)};
    if (in) {
        pair_masks<FLAGS>(d, c, has1, m0, m1, live0, live1);
        if (!FLAGS || live0 || live1) {
            if (rho0) get2<RF>(rho0 + cc, pair, has1, r[0], r[1]);
            get2<RF>(u0 + cc, pair, has1, ux[0], ux[1]);
            get2<RF>(u0 + N + cc, pair, has1, uy[0], uy[1]);
            get2<RF>(u0 + 2 * N + cc, pair, has1, uz[0], uz[1]);
        }
    }
    typedef typename Pair2<R>::V V;
    V f[Q];
    if constexpr (S == LBM_F64) {
        double f0[Q], f1[Q];
        if (!fixed_equilibrium(f0, r[0] - 1.0, ux[0], uy[0], uz[0], d.incomp))
            feq64(f0, r[0] - 1.0, ux[0], uy[0], uz[0], d.incomp);
        if (!fixed_equilibrium(f1, r[1] - 1.0, ux[1], uy[1], uz[1], d.incomp))
            feq64(f1, r[1] - 1.0, ux[1], uy[1], uz[1], d.incomp);
#pragma unroll
        for (int i = 0; i < Q; ++i) f[i] = make_double2(f0[i], f1[i]);
    } else {
        feq2(f, make_float2(r[0] - 1.0f, r[1] - 1.0f), make_float2(ux[0], ux[1]), make_float2(uy[0], uy[1]),
             make_float2(uz[0], uz[1]), d.incomp);
    }
    if (d.layout == LAYOUT_AA_NAT) {  // AA natural layout: f^0_i(x) at the cell itself
        const R nan = quiet_nan<R>();
        if (!in) return;
#pragma unroll
        for (int i = 0; i < Q; ++i)
            put2(P + i * g.qs + c, true, true, !FLAGS || live0 ? f[i].x : nan, !FLAGS || live1 ? f[i].y : nan);
        return;
    }
    // Cells x0 and x0 + 1 to columns x0 - e_x and x0 + 1 - e_x. Where e_x = +-1
    // the column pair (x0, x0 + 1) takes one value of this lane and one of its
    // neighbour's, so that it is stored whole: `next` and `prev` say which
    // neighbour pairs up (same row, both cells fluid); other values go singly.
    // (Storing every value of these 10 populations singly: FP16 channel 86 us,
    // FP32 111.)
    const int lane = threadIdx.x & 31;
    const bool right0 = __shfl_down_sync(0xffffffffu, live0, 1);
    const bool next = in && lane < 31 && x0 + 2 < g.nx && live1 && right0;
    const bool left = __shfl_up_sync(0xffffffffu, next, 1);
    const bool prev = lane > 0 && left;
    // (to column x + 1 the lone last cell of an odd row goes alone, to column 0)
    const bool next1 = next && x0 + 3 < g.nx, prev1 = prev && has1;
    const int xa = wrap1(x0 - 1, g.nx), xb = wrap1(x0 + 1, g.nx);
    const int xc = has1 ? wrap1(x0 + 2, g.nx) : x0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        T *row = P + i * g.qs + (wrap1(z - ez(i), g.nz) * g.ny + wrap1(y - ey(i), g.ny)) * g.pitch;
        if (ex(i) == 0) {
            if (live0 && live1) {
                put2(row + x0, true, true, f[i].x, f[i].y);
            } else {
                if (live0) row[x0] = Rn<T>::of(f[i].x);
                if (live1) row[x0 + 1] = Rn<T>::of(f[i].y);
            }
        } else if (ex(i) > 0) {
            const R v = __shfl_down_sync(0xffffffffu, f[i].x, 1);
            if (next) put2(row + x0, true, true, f[i].y, v);
            else if (live1) row[x0] = Rn<T>::of(f[i].y);
            if (live0 && !prev) row[xa] = Rn<T>::of(f[i].x);
        } else {
            const R v = __shfl_up_sync(0xffffffffu, f[i].y, 1);
            if (prev1) put2(row + x0, true, true, v, f[i].x);
            else if (live0) row[xb] = Rn<T>::of(f[i].x);
            if (live1 && !next1) row[xc] = Rn<T>::of(f[i].y);
        }
    }
    if (FLAGS && ((m0 | m1) & 0x7fffeu)) {
        // (the gather adds the moving-wall term to a value bounced off a moving wall)
        const uint2 mv = !bounce_in_solid(S) && d.moving_on && ((m0 | m1) & MOVING_BIT) ? moving_links(d, c, m0, m1)
                                                                                       : make_uint2(0u, 0u);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (!(((k ? m1 : m0) >> i) & 1u)) continue;
                R v = k ? f[opp(i)].y : f[opp(i)].x;
                if (((k ? mv.y : mv.x) >> i) & 1u) v += wall_term<R>(d, i);
                P[i * g.qs + c + k] = Rn<T>::of(v);
            }
        }
    }
}

// The values v of a cell, each with its moving-wall term where bit i of mv is set, to
// a moment-split lattice.
template <int S>
static __device__ __noinline__ void split_store_moving(const Dev &d, typename Stor<S>::T *P, int x, int c, uint32_t mv,
                                                       const float *v) {
    double t[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) t[i] = (double)v[i] + ((mv >> i) & 1u ? d.wc[i] : 0.0);
    split_store<S>(d, P, x, c, t);
}

// ---------------------------------------------------------------------------
// get_state: canonical shifted f^n = gather(P), format D; solid cells 0.
// Bound by HBM (19 values read and 19 written a cell). One cell a thread with
// 18 flag loads and every value converted over double took 1622 us for the
// 384x256x256 porous channel (FP16 to BF16: 1.9 GB, 0.17 of copy bandwidth).
// Blocks of 128 per SM: FP64 storage to narrower states 5 (4 before: channel to BF16
// 185 to 165 us, AA 157 to 137), FP32 and 16-bit storage to FP64 states 8 and 7 (6:
// channel 191 to 178 us and 165 to 157).
template <int S, int D, bool FLAGS> constexpr int get_state_blocks() {
    if (is_split(S)) return 2 * FieldBlocks<S, FLAGS>::value;
    if (S == LBM_F64) return D == LBM_F64 ? 4 : 5;
    return D == LBM_F64 ? (S == LBM_F32 ? 8 : 7) : 2 * FieldBlocks<S, FLAGS>::value;
}

// ALT: rows of odd length to FP64 states, where a pair is aligned in every other row
// and population: each thread looks, and stores whole pairs where it can (cavity
// 127x129x125, FP16 104 to 80 us, FP32 110 to 91; on small lattices the look costs
// more than it gives, 95x61x53 18.4 to 22).
template <int S, int D, bool FLAGS, bool ALT = false>
__global__ void __launch_bounds__(128, get_state_blocks<S, D, FLAGS>())
    k_get_state(const Dev d, const typename Stor<S>::T *__restrict__ P, typename IOFmt<D>::T *__restrict__ out,
                bool pair) {
    typedef typename Stor<S>::R R;
    typedef typename IOFmt<D>::T TD;
    int x0, y, z;
    if (!pair_cell<true>(d.g, d.PF, blockDim.x, blockDim.y, blockIdx.x, blockIdx.y, threadIdx.x, threadIdx.y, x0, y,
                         z))
        return;
    const bool has1 = x0 + 1 < d.g.nx;
    const int c = cell_index(d.g, x0, y, z);
    const long long N = d.n_cells, cc = canon_index(d.g, x0, y, z);
    uint32_t m0, m1;
    bool live0, live1;
    pair_masks<FLAGS>(d, c, has1, m0, m1, live0, live1);
    if (FLAGS && !live0 && !live1) {
#pragma unroll
        for (int i = 0; i < Q; ++i) put2(out + i * N + cc, pair, has1, 0.0f, 0.0f);
        return;
    }
    typename Pair2<R>::V s[Q];
    gather_pair<S, FLAGS>(d, P, x0, y, z, c, has1, m0, m1, s);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        TD *p = out + i * N + cc;
        const bool whole = ALT ? has1 && (reinterpret_cast<uintptr_t>(p) & (2 * sizeof(TD) - 1)) == 0 : pair;
        put2(p, whole, has1, !FLAGS || live0 ? s[i].x : R(0), !FLAGS || live1 ? s[i].y : R(0));
    }
}

// Blocks of 128 per SM of set_state. Narrower storage from FP64 states, whose 38
// values are held as doubles, 5 (96 registers): with the 7 of the narrower states the
// kernels with flags spilled 312 to 416 bytes (AA channel FP32 163
// to 142 us, FP16 169 to 145; two-grid 206 to 156 and 232 to 208).
template <int S, int D, bool FLAGS> constexpr int set_state_blocks() {
    if (D == LBM_F64 && S != LBM_F64) return 5;
    return FLAGS && !is_split(S) && S != LBM_F64 ? 7 : 2 * FieldBlocks<S, FLAGS>::value;
}

// set_state: P_i(y) = s_i(y + e_i) if fluid there, else s_{opp(i)}(y). The
// loads follow the reverse step's gather (sources y + e_i, the pair's own
// values over them where a mask bit is set). Moment-split storage collects the
// 19 values its cells hold and rounds momentum and remainders once, whatever format
// they come in (256^3 box from FP32 301 us; in double 3017).
template <int S, int D, bool FLAGS>
__global__ void __launch_bounds__(128, set_state_blocks<S, D, FLAGS>())
    k_set_state(const Dev d, typename Stor<S>::T *__restrict__ P, const typename IOFmt<D>::T *__restrict__ in,
                bool pair) {
    typedef typename Stor<S>::T T;
    typedef typename IOFmt<D>::T TD;
    typedef typename IOFmt<D>::V V;
    const Geom &g = d.g;
    int x0, y, z;
    if (!pair_cell<true>(g, d.PF, blockDim.x, blockDim.y, blockIdx.x, blockIdx.y, threadIdx.x, threadIdx.y, x0, y, z))
        return;
    const bool has1 = x0 + 1 < g.nx;
    const int c = cell_index(g, x0, y, z);
    const long long N = d.n_cells, cc = canon_index(g, x0, y, z);
    uint32_t m0, m1;
    bool live0, live1;
    pair_masks<FLAGS>(d, c, has1, m0, m1, live0, live1);
    const bool mark = FLAGS && nan_marked(d);
    if (FLAGS && !mark && !live0 && !live1) return;
    V s0[Q], s1[Q];
    if (!is_split(S) && d.layout == LAYOUT_AA_NAT) {  // AA natural layout: s_i(x) at the cell itself
        if (pair) {
#pragma unroll
            for (int i = 0; i < Q; ++i) get2<D>(in + i * N + cc, true, true, s0[i], s1[i]);
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i) get2<D>(in + i * N + cc, false, has1, s0[i], s1[i]);
        }
    } else {
        const int xa = wrap1(x0 - 1, g.nx), xb = wrap1(x0 + 1, g.nx);
        const int xc = has1 ? wrap1(x0 + 2, g.nx) : x0;
        // (the loads of one kind together, so that `pair` is tested once and
        // all of them are in flight at the same time)
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            if (ex(i) == 0) continue;
            const TD *row = in + i * N + (long long)(wrap1(z + ez(i), g.nz) * g.ny + wrap1(y + ey(i), g.ny)) * g.nx;
            s0[i] = IOFmt<D>::get(row + (ex(i) > 0 ? xb : xa));
            s1[i] = IOFmt<D>::get(row + (ex(i) > 0 ? xc : x0));
        }
        if (pair) {
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if (ex(i) == 0)
                    get2<D>(in + i * N + x0 +
                                (long long)(wrap1(z + ez(i), g.nz) * g.ny + wrap1(y + ey(i), g.ny)) * g.nx,
                            true, true, s0[i], s1[i]);
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if (ex(i) == 0)
                    get2<D>(in + i * N + x0 +
                                (long long)(wrap1(z + ez(i), g.nz) * g.ny + wrap1(y + ey(i), g.ny)) * g.nx,
                            false, has1, s0[i], s1[i]);
        }
        if (FLAGS && ((m0 | m1) & 0x7fffeu)) {
#pragma unroll
            for (int i = 1; i < Q; ++i) {
                const TD *own = in + opp(i) * N + cc;
                if ((m0 >> i) & 1u) s0[i] = IOFmt<D>::get(own);
                if ((m1 >> i) & 1u) s1[i] = IOFmt<D>::get(own + 1);
            }
        }
    }
    const uint2 mv = FLAGS && d.has_moving && d.layout == LAYOUT_PULL && ((m0 | m1) & MOVING_BIT)
                         ? moving_links(d, c, m0, m1)
                         : make_uint2(0u, 0u);
    if constexpr (is_split(S) && sizeof(V) == 4) {
        if (FLAGS && !live0 && !live1) return;
        if (d.moving_on && (mv.x | mv.y)) {  // rare: with the walls' terms, in double
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (!(k ? live1 : live0)) continue;
                float t[Q];
#pragma unroll
                for (int i = 0; i < Q; ++i) t[i] = k ? s1[i] : s0[i];
                split_store_moving<S>(d, P, x0 + k, c + k, k ? mv.y : mv.x, t);
            }
            return;
        }
        float2 v[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) v[i] = make_float2(s0[i], s1[i]);
        split_store_pair_once<S>(d, P, x0, c, has1, v);
        return;
    } else if constexpr (is_split(S)) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (!(k ? live1 : live0)) continue;
            double v[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                v[i] = (double)(k ? s1[i] : s0[i]);
                if (d.moving_on && (((k ? mv.y : mv.x) >> i) & 1u)) v[i] += d.wc[i];
            }
            split_store<S>(d, P, x0 + k, c + k, v);
        }
        return;
    } else {
        if (FLAGS && bounce_in_solid(S) && d.has_moving && !mark && !(live0 && live1)) {
            // (other threads write a solid cell's moving-wall links, below)
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                if (live0) P[i * g.qs + c] = Rn<T>::of(s0[i]);
                if (live1) P[i * g.qs + c + 1] = Rn<T>::of(s1[i]);
            }
        } else {
            // a pair is stored whole, a solid cell as zeros (never read, or
            // filled by the link kernel after this one) or as the NaN that
            // marks it: storing the fluid cell alone took 870 us for the
            // porous channel (384x256x256, FP16 from BF16) against 634
            const V solid = mark ? V(quiet_nan<float>()) : V(0);
#pragma unroll
            for (int i = 0; i < Q; ++i)
                put2(P + i * g.qs + c, true, true, !FLAGS || live0 ? s0[i] : solid, !FLAGS || live1 ? s1[i] : solid);
        }
        // links into moving walls, which the link kernel leaves to their fluid
        // cell: the solid slot that the link form pulls f_opp(i)(x) from; in
        // the other forms the gather adds the moving-wall term, taken off here
        // (summed in double, rounded once)
        if (FLAGS && (mv.x | mv.y) && (d.moving_on || bounce_in_solid(S))) {
#pragma unroll
            for (int i = 1; i < Q; ++i) {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if (!(((k ? mv.y : mv.x) >> i) & 1u)) continue;
                    const V v = k ? s1[i] : s0[i];
                    if (bounce_in_solid(S))
                        P[(long long)opp(i) * g.qs + push_dst(g, x0 + k, y, z, i)] = Rn<T>::of(v);
                    else
                        P[i * g.qs + c + k] = Rn<T>::of((double)v + d.wc[i]);
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// The pair's body force: uniform, or the force field at cell c.
template <class R, bool FORCE>
__device__ __forceinline__ void pair_force_at(const Dev &d, int c, typename Pair2<R>::V &Fx,
                                              typename Pair2<R>::V &Fy, typename Pair2<R>::V &Fz) {
    Fx = Fy = Fz = vsplat(R(0));
    if (!FORCE) return;
    if (d.Ffield) {
        const R *F = static_cast<const R *>(d.Ffield);
        ld2_real(F + c, Fx.x, Fx.y);
        ld2_real(F + d.g.qs + c, Fy.x, Fy.y);
        ld2_real(F + 2 * d.g.qs + c, Fz.x, Fz.y);
    } else {
        Fx = vsplat(DevR<R>::F(d, 0));
        Fy = vsplat(DevR<R>::F(d, 1));
        Fz = vsplat(DevR<R>::F(d, 2));
    }
}

// Macroscopic fields (Sec. 2 step 1): rho and u = (j + F/2)/rho; solid 0.
// Bound by HBM (19 values read, 4 reals written a cell).
template <int S, bool FLAGS, bool FORCE>
__global__ void __launch_bounds__(128, 2 * FieldBlocks<S, FLAGS>::value)
    k_macros(const Dev d, const typename Stor<S>::T *__restrict__ P, typename Stor<S>::R *__restrict__ rho,
             typename Stor<S>::R *__restrict__ u, bool pair) {
    typedef typename Stor<S>::R R;
    typedef typename Pair2<R>::V V;
    int x0, y, z;
    if (!pair_cell<true>(d.g, d.PF, blockDim.x, blockDim.y, blockIdx.x, blockIdx.y, threadIdx.x, threadIdx.y, x0, y,
                         z))
        return;
    const bool has1 = x0 + 1 < d.g.nx;
    const int c = cell_index(d.g, x0, y, z);
    const long long N = d.n_cells, cc = canon_index(d.g, x0, y, z);
    uint32_t m0, m1;
    bool live0, live1;
    pair_masks<FLAGS>(d, c, has1, m0, m1, live0, live1);
    V o[4] = {vsplat(R(0)), vsplat(R(0)), vsplat(R(0)), vsplat(R(0))};
    if (!FLAGS || live0 || live1) {
        V s[Q], Fx, Fy, Fz;
        gather_pair<S, FLAGS>(d, P, x0, y, z, c, has1, m0, m1, s);
        pair_force_at<R, FORCE>(d, c, Fx, Fy, Fz);
        const Mom2<R> m = pair_moments<R, FORCE>(d, s, Fx, Fy, Fz, live0, live1);
        o[0] = m.rho;
        o[1] = m.ux;
        o[2] = m.uy;
        o[3] = m.uz;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        R *p = k ? u + (k - 1) * N : rho;
        if (k || rho)
            put2(p + cc, pair, has1, !FLAGS || live0 ? o[k].x : R(0), !FLAGS || live1 ? o[k].y : R(0));
    }
}

// ---------------------------------------------------------------------------
// Mass and momentum totals of planes z0 <= z < z1: each thread walks the pairs
// tid, tid + stride, ... in order; every warp adds the integer sums of its
// pairs (tot_add) to 64-bit ones, one (quantity, level) a lane; warps and
// blocks combine in a fixed order. Deterministic. Bound by HBM (19 values read
// a cell). FP64 values, and FP32 ones too large for the integer sums, are
// added in FP64.
template <int S, bool FLAGS, bool FORCE>
__global__ void __launch_bounds__(RED_THREADS, FLAGS || is_split(S) ? 2 : FieldBlocks<S, FLAGS>::value)
    k_reduce(const Dev d, const typename Stor<S>::T *__restrict__ P, int z0, int z1, double *__restrict__ partials) {
    typedef typename Stor<S>::R R;
    typedef typename Pair2<R>::V V;
    constexpr bool INT = sizeof(R) == 4;
    const int W = (d.g.nx + 1) / 2, per = W * d.g.ny, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long pairs = (long long)per * (z1 - z0);
    double red[4] = {0.0, 0.0, 0.0, 0.0};
    long long acc = 0, cells = 0;
    bool in_red = !INT;
    // (whole warps iterate together: their sums need every lane)
    for (long long q0 = (long long)blockIdx.x * RED_THREADS + 32 * wid; q0 < pairs;
         q0 += (long long)gridDim.x * RED_THREADS) {
        const long long q = q0 + lane;
        PairTotals<R> tot;
        tot.clear();
        if (q < pairs) {
            int x0, y, z;
            reduce_pair((int)q, W, per, z0, x0, y, z);  // (pairs < 2^31)
            const bool has1 = x0 + 1 < d.g.nx;
            const int c = cell_index(d.g, x0, y, z);
            uint32_t m0, m1;
            bool live0, live1;
            pair_masks<FLAGS>(d, c, has1, m0, m1, live0, live1);
            if (!FLAGS || live0 || live1) {
                V s[Q], Fx, Fy, Fz;
                gather_pair<S, FLAGS>(d, P, x0, y, z, c, has1, m0, m1, s);
                pair_force_at<R, FORCE>(d, c, Fx, Fy, Fz);
                tot.set(pair_moments<R, FORCE>(d, s, Fx, Fy, Fz, live0, live1), live0, live1);
            }
        }
        cells += tot.cells;
        bool fits = INT;
        if constexpr (INT) {
#pragma unroll
            for (int k = 0; k < 4; ++k) fits = fits && tot_fits(tot.v[k].x) && tot_fits(tot.v[k].y);
            fits = __all_sync(0xffffffffu, fits);
            if (fits) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    int h[TOT_LEVELS] = {0, 0, 0, 0};
                    tot_add(h, tot.v[k].x);
                    tot_add(h, tot.v[k].y);
#pragma unroll
                    for (int l = 0; l < TOT_LEVELS; ++l) {
                        const int sum = __reduce_add_sync(0xffffffffu, h[l]);
                        if (lane == k * TOT_LEVELS + l) acc += sum;
                    }
                }
            }
        }
        if (!fits) {
            in_red = true;
#pragma unroll
            for (int k = 0; k < 4; ++k) red[k] += (double)tot.v[k].x + (double)tot.v[k].y;
        }
    }
    __shared__ long long sm[RED_THREADS / 32][4 * TOT_LEVELS + 1];
    if (lane < 4 * TOT_LEVELS) sm[wid][lane] = acc;
    for (int o = 16; o > 0; o >>= 1) cells += __shfl_xor_sync(0xffffffffu, cells, o);
    if (lane == 0) sm[wid][4 * TOT_LEVELS] = cells;
    double t = 0.0;
    if (__syncthreads_or(in_red)) t = block_sum_d(red);
    if (threadIdx.x < 4) {
#pragma unroll
        for (int l = TOT_LEVELS - 1; INT && l >= 0; --l) {
            long long h = 0;
            for (int w = 0; w < RED_THREADS / 32; ++w) h += sm[w][threadIdx.x * TOT_LEVELS + l];
            t = fma((double)h, pow2d(tot_grid(l)), t);
        }
        if (threadIdx.x == 0) {
            long long n = 0;
            for (int w = 0; w < RED_THREADS / 32; ++w) n += sm[w][4 * TOT_LEVELS];
            t += (double)n;
        }
        partials[blockIdx.x * 4 + threadIdx.x] = t;
    }
}

// ---------------------------------------------------------------------------
// Adjoint seed (not in the paper): lambda^T_m = dL/drho + g.(e_m - u)/rho,
// g = dL/du, at the gathered state; grad_F += g / (2 rho) (u contains F/2).
// Incompressible model (u = j + F/2): lambda^T_m = dL/drho + g.e_m, grad_F += g/2.
template <int S, bool FLAGS, bool FORCE>
__global__ void __launch_bounds__(128, 2 * FieldBlocks<S, FLAGS>::value)
    k_adj_seed(const Dev d, const typename Stor<S>::T *__restrict__ P, const typename Stor<S>::R *__restrict__ dL_du,
               const typename Stor<S>::R *__restrict__ dL_drho, typename Stor<S>::R *__restrict__ lam,
               typename Stor<S>::R *__restrict__ grad_F, bool pair) {
    typedef typename Stor<S>::R R;
    typedef typename Pair2<R>::V V;
    constexpr int RF = sizeof(R) == 8 ? LBM_F64 : LBM_F32;  // canonical format of R
    int x0, y, z;
    if (!pair_cell<true>(d.g, d.PF, blockDim.x, blockDim.y, blockIdx.x, blockIdx.y, threadIdx.x, threadIdx.y, x0, y,
                         z))
        return;
    const bool has1 = x0 + 1 < d.g.nx;
    const int c = cell_index(d.g, x0, y, z);
    const long long qs = d.g.qs, N = d.n_cells, cc = canon_index(d.g, x0, y, z);
    uint32_t m0, m1;
    bool live0, live1;
    pair_masks<FLAGS>(d, c, has1, m0, m1, live0, live1);
    if (FLAGS && !live0 && !live1) return;  // solid cells' adjoint slots are never read
    V s[Q], Fx, Fy, Fz, gx, gy, gz, dr = vsplat(R(0));
    get2<RF>(dL_du + cc, pair, has1, gx.x, gx.y);
    get2<RF>(dL_du + N + cc, pair, has1, gy.x, gy.y);
    get2<RF>(dL_du + 2 * N + cc, pair, has1, gz.x, gz.y);
    if (dL_drho) get2<RF>(dL_drho + cc, pair, has1, dr.x, dr.y);
    gather_pair<S, FLAGS>(d, P, x0, y, z, c, has1, m0, m1, s);
    pair_force_at<R, FORCE>(d, c, Fx, Fy, Fz);
    const Mom2<R> m = pair_moments<R, FORCE>(d, s, Fx, Fy, Fz, live0, live1);
    const V inv = d.incomp ? vsplat(R(1)) : vrcp(m.rho);
    const V gu = vfma(gz, m.uz, vfma(gy, m.uy, vmul(gx, m.ux)));
    const V base = d.incomp ? dr : vsub(dr, vmul(gu, inv));
    const V hx = vmul(gx, inv), hy = vmul(gy, inv), hz = vmul(gz, inv);
    // (a solid cell of a mixed pair gets a value nobody reads)
    st2_real(lam + c, base.x, base.y);
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        const int i = pair_first(p), o = opp(i);
        const V e = edot_first(i, hx, hy, hz), a = vadd(base, e), b = vsub(base, e);
        st2_real(lam + i * qs + c, a.x, a.y);
        st2_real(lam + o * qs + c, b.x, b.y);
    }
    if (grad_F) {
        const V h[3] = {hx, hy, hz};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            R *G = grad_F + k * N + cc;
            if (live0) G[0] += R(0.5) * h[k].x;
            if (live1) G[1] += R(0.5) * h[k].y;
        }
    }
}

// ---------------------------------------------------------------------------
// Host launchers.
inline dim3 row_grid(const Dev &d) { return dim3(d.L.nxb * d.L.nyb, d.g.nz); }
inline dim3 row_block(const Dev &d) { return dim3(d.L.bx_threads, d.L.by_threads); }

// The step kernels run on the paired launch (two cells per thread).
inline dim3 step_grid(const Dev &d) { return dim3(d.P.nxb * d.P.nyb, d.P.nzr); }
inline dim3 step_block(const Dev &d) { return dim3(d.P.bx_threads, d.P.by_threads); }

// 32-bit lattice offsets: measured on the FP32 step with flags (walled
// channel +0.9%); the 16-bit and flag-free steps gained nothing (512^3 box
// FP16 -1.9%), so they keep 64-bit offsets.
template <int S, bool FLAGS> inline bool step_u32(const Dev &d) {
    return S == LBM_F32 && FLAGS && (long long)Q * d.g.qs < (1LL << 32);
}

// Launch k as a programmatic dependent of the kernel before it on the stream.
template <class... P, class... A>
static cudaError_t launch_dependent(void (*k)(P...), dim3 grid, dim3 block, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = STEP_PDL;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k, args...);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int S, bool FLAGS, int FORCE, bool FLAT, bool ODD = false, bool U32 = false>
static cudaError_t launch_step3f(const Dev &d, const void *src, void *dst, void *tape) {
    typedef typename Stor<S>::T T;
    typedef typename Stor<S>::R R;
    if constexpr (!U32 && S == LBM_F32 && FLAGS) {
        // (with flags the flat launch's blocks hold at most 128 threads, step_threads)
        if (step_u32<S, FLAGS>(d)) return launch_step3f<S, FLAGS, FORCE, FLAT, ODD, true>(d, src, dst, tape);
    }
    const RowLaunch &P = FLAT ? d.PF : d.P;
    const dim3 grid(P.nxb * P.nyb, P.nzr), block(P.bx_threads, P.by_threads);
    return launch_dependent(tape ? k_step<S, FLAGS, FORCE, true, FLAT, ODD, U32> : k_step<S, FLAGS, FORCE, false, FLAT, ODD, U32>,
                            grid, block, d.stream, d, static_cast<const T *>(src), static_cast<T *>(dst),
                            static_cast<R *>(tape));
}

// Always the flat launch where that measured faster with whole-warp rows too (its
// index code compiles to fewer spills): FP32 (walled channel +1%) and 16-bit storage
// without flags (512^3 box +3%). The 16-bit link form with flags takes it only where
// whole rows would leave lanes idle, or on small lattices (the flat form spilled
// more: -4.5%).
template <int S, bool FLAGS> constexpr bool always_flat() { return S == LBM_F32 || is_split(S) || !FLAGS; }

template <int S, bool FLAGS, int FORCE>
static cudaError_t launch_step3(const Dev &d, const void *src, void *dst, void *tape) {
    if constexpr (is_split(S))
        return (d.g.nx & 1) ? launch_step3f<S, FLAGS, FORCE, true, true>(d, src, dst, tape)
                            : launch_step3f<S, FLAGS, FORCE, true, false>(d, src, dst, tape);
    else if constexpr (always_flat<S, FLAGS>())
        return launch_step3f<S, FLAGS, FORCE, true>(d, src, dst, tape);
    else
        return d.flat_step ? launch_step3f<S, FLAGS, FORCE, true>(d, src, dst, tape)
                           : launch_step3f<S, FLAGS, FORCE, false>(d, src, dst, tape);
}

// Shared memory of the row-staged step: two buffers of 19 padded rows.
constexpr int TMA_SMEM_MAX = 200 * 1024;
template <int S> inline int tma_smem_bytes(const Dev &d) {
    return 2 * Q * d.g.pitch * (int)sizeof(typename Stor<S>::T) + 16;
}
// The row-staged step serves FP32 and 16-bit shifted storage when rows are
// whole 16-byte multiples and two buffers fit.
template <int S> inline bool tma_eligible(const Dev &d) {
    const long long rowbytes = (long long)d.g.pitch * sizeof(typename Stor<S>::T);
    return d.row_staging && rowbytes % 16 == 0 && tma_smem_bytes<S>(d) <= TMA_SMEM_MAX;
}

template <int S, bool FLAGS, int FORCE, bool RECORD>
static cudaError_t launch_step_tma4(const Dev &d, const void *src, void *dst, void *tape) {
    typedef typename Stor<S>::T T;
    typedef typename Stor<S>::R R;
    auto kern = k_step_tma<S, FLAGS, FORCE, RECORD>;
    // (set on every launch: the attribute belongs to the current device's context)
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, TMA_SMEM_MAX);
    if (e != cudaSuccess) return e;
    const int smem = tma_smem_bytes<S>(d);
    const int pairs = (d.g.nx + 1) / 2;
    const int threads = pairs >= 512 ? 512 : (pairs + 31) / 32 * 32;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem);
    if (e != cudaSuccess) return e;
    const long long nrows = (long long)d.P.nyr * d.P.nzr;
    const long long want = (long long)(occ > 0 ? occ : 1) * d.num_sms;
    const int grid = (int)(nrows < want ? nrows : want);
    kern<<<grid, threads, smem, d.stream>>>(d, static_cast<const T *>(src), static_cast<T *>(dst),
                                           static_cast<R *>(tape));
    return cudaGetLastError();
}

// FP64: one cell a thread over the box rows; 32-bit offsets where they fit.
// RED: out is the partials (4 doubles per block), else the tape or null.
inline int step64_threads(const Dev &d) { return small_lattice(d.P) ? 64 : 128; }
inline dim3 step64_grid(const Dev &d) {
    const int t = step64_threads(d);
    return dim3((unsigned)(((long long)d.P.nyr * d.g.nx + t - 1) / t), d.P.nzr);
}
template <bool FLAGS, int FORCE, bool RECORD, bool RED>
static cudaError_t launch_step64(const Dev &d, const void *src, void *dst, void *out) {
    const bool narrow = (long long)Q * d.g.qs < (1LL << 32);
    return launch_dependent(narrow ? k_step64<FLAGS, FORCE, RECORD, RED, unsigned> : k_step64<FLAGS, FORCE, RECORD, RED, long long>,
                            step64_grid(d), dim3(step64_threads(d)), d.stream, d, static_cast<const double *>(src),
                            static_cast<double *>(dst), static_cast<double *>(out));
}

template <int S, bool FLAGS, int FORCE>
static cudaError_t launch_step3_any(const Dev &d, const void *src, void *dst, void *tape) {
    if constexpr (S == LBM_F64) {
        return tape ? launch_step64<FLAGS, FORCE, true, false>(d, src, dst, tape)
                    : launch_step64<FLAGS, FORCE, false, false>(d, src, dst, nullptr);
    } else {
        if constexpr (!is_split(S)) {  // (the moment-split formats have no staged form)
            if (tma_eligible<S>(d))
                return tape ? launch_step_tma4<S, FLAGS, FORCE, true>(d, src, dst, tape)
                            : launch_step_tma4<S, FLAGS, FORCE, false>(d, src, dst, tape);
        }
        return launch_step3<S, FLAGS, FORCE>(d, src, dst, tape);
    }
}

template <int S, bool FLAGS>
static cudaError_t launch_step2(const Dev &d, const void *src, void *dst, void *tape) {
    if (d.Ffield) return launch_step3_any<S, FLAGS, 2>(d, src, dst, tape);
    if (d.force_on) return launch_step3_any<S, FLAGS, 1>(d, src, dst, tape);
    return launch_step3_any<S, FLAGS, 0>(d, src, dst, tape);
}

template <int S>
cudaError_t Ops<S>::step(const Dev &d, const void *src, void *dst, void *tape) {
    if (!d.flags) return launch_step2<S, false>(d, src, dst, tape);
    if (!d.mask) return cudaErrorInvalidValue;  // every two-grid form with flags may read the push masks
    cudaError_t e = launch_step2<S, true>(d, src, dst, tape);
    if (e != cudaSuccess || !LinkBounce<S>::value || d.link_max == 0) return e;
    const int per_block = 256 * LINKS_PER_THREAD;
    // programmatic dependent launch: the bounce kernel's blocks may start (and
    // load their links) while the step kernel drains; they wait for its grid
    // before reading the values (griddepcontrol.wait in k_bounce)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(Q - 1, (d.link_max + per_block - 1) / per_block);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = d.stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = BOUNCE_PDL;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_bounce<S>, d, static_cast<typename Stor<S>::T *>(dst));
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template <int S>
cudaError_t Ops<S>::bounce(const Dev &d, void *dst) {
    if (!d.flags || !LinkBounce<S>::value || d.link_max == 0) return cudaSuccess;
    const int per_block = 256 * LINKS_PER_THREAD;
    k_bounce<S><<<dim3(Q - 1, (d.link_max + per_block - 1) / per_block), 256, 0, d.stream>>>(
        d, static_cast<typename Stor<S>::T *>(dst));
    return cudaGetLastError();
}

// The fused step-reduce kernel, with the launch mapping of the plain step
// (launch_step3); grid: its blocks, one partial each.
template <int S, bool FLAGS, int FORCE>
static cudaError_t launch_step_reduce3(const Dev &d, const void *src, void *dst, double *partials, dim3 &grid) {
    typedef typename Stor<S>::T T;
    const bool flat = always_flat<S, FLAGS>() || d.flat_step;
    const RowLaunch &P = flat ? d.PF : d.P;
    const dim3 block(P.bx_threads, P.by_threads);
    grid = dim3(P.nxb * P.nyb, P.nzr);
    void (*k)(Dev, const T *, T *, double *) = k_step_reduce<S, FLAGS, FORCE, true>;
    if constexpr (is_split(S)) {
        if (d.g.nx & 1) k = k_step_reduce<S, FLAGS, FORCE, true, true>;
    } else if constexpr (!always_flat<S, FLAGS>()) {
        if (!flat) k = k_step_reduce<S, FLAGS, FORCE, false>;
    }
    k<<<grid, block, 0, d.stream>>>(d, static_cast<const T *>(src), static_cast<T *>(dst), partials);
    return cudaGetLastError();
}
template <int S, bool FLAGS>
static cudaError_t launch_step_reduce2(const Dev &d, const void *src, void *dst, double *partials, dim3 &grid) {
    if (d.Ffield) return launch_step_reduce3<S, FLAGS, 2>(d, src, dst, partials, grid);
    if (d.force_on) return launch_step_reduce3<S, FLAGS, 1>(d, src, dst, partials, grid);
    return launch_step_reduce3<S, FLAGS, 0>(d, src, dst, partials, grid);
}

template <int S>
cudaError_t Ops<S>::step_reduce(const Dev &d, const void *src, void *dst, double *partials, double *out) {
    typedef typename Stor<S>::T T;
    if (d.flags && !d.mask) return cudaErrorInvalidValue;
    if constexpr (S == LBM_F64) {
        cudaError_t e;
        if (d.flags)
            e = d.Ffield ? launch_step64<true, 2, false, true>(d, src, dst, partials)
                         : (d.force_on ? launch_step64<true, 1, false, true>(d, src, dst, partials)
                                       : launch_step64<true, 0, false, true>(d, src, dst, partials));
        else
            e = d.Ffield ? launch_step64<false, 2, false, true>(d, src, dst, partials)
                         : (d.force_on ? launch_step64<false, 1, false, true>(d, src, dst, partials)
                                       : launch_step64<false, 0, false, true>(d, src, dst, partials));
        if (e != cudaSuccess) return e;
        const dim3 grid = step64_grid(d);
        const int n = (int)(grid.x * grid.y);
        return sum_partials(partials, n, partials + 4 * (size_t)n, out, d.stream);
    } else {
        dim3 grid;
        cudaError_t e = d.flags ? launch_step_reduce2<S, true>(d, src, dst, partials, grid)
                                : launch_step_reduce2<S, false>(d, src, dst, partials, grid);
        if (e != cudaSuccess) return e;
        if (d.flags && LinkBounce<S>::value && d.link_max > 0) {
            const int per_block = 256 * LINKS_PER_THREAD;
            k_bounce<S><<<dim3(Q - 1, (d.link_max + per_block - 1) / per_block), 256, 0, d.stream>>>(
                d, static_cast<T *>(dst));
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        return sum_partials(partials, (int)(grid.x * grid.y), partials + 4 * (size_t)grid.x * grid.y, out, d.stream);
    }
}

// NaN marks on every slot of every solid cell (AA pattern; no-op otherwise).
template <int S>
__global__ void __launch_bounds__(256) k_fill_solid(const Dev d, typename Stor<S>::T *__restrict__ P) {
    int x, y, z;
    if (!row_cell(d.g, d.L.nxb, blockDim.x, blockDim.y, blockIdx.x, blockIdx.y, threadIdx.x, threadIdx.y, x, y, z))
        return;
    const int c = cell_index(d.g, x, y, z);
    if (!d.flags[c]) return;
#pragma unroll
    for (int i = 0; i < Q; ++i) P[(long long)i * d.g.qs + c] = Stor<S>::enc(quiet_nan<typename Stor<S>::R>());
}

template <int S>
cudaError_t Ops<S>::fill_solid(const Dev &d, void *lat) {
    if (!d.flags || d.layout == LAYOUT_PULL) return cudaSuccess;
    k_fill_solid<S><<<row_grid(d), row_block(d), 0, d.stream>>>(d, static_cast<typename Stor<S>::T *>(lat));
    return cudaGetLastError();
}

template <int S>
cudaError_t Ops<S>::init_eq(const Dev &d0, void *lat, const void *rho0, const void *u0) {
    typedef typename Stor<S>::T T;
    typedef typename Stor<S>::R R;
    if (d0.flags && !d0.mask) return cudaErrorInvalidValue;
    if constexpr (is_split(S)) {
        Dev d = d0;
        d.PF = all_pairs(d.g);
        const bool pair = pair_aligned(d.g, u0, sizeof(R)) && (!rho0 || pair_aligned(d.g, rho0, sizeof(R)));
        if (d.flags)
            k_init_eq_split<S, true><<<pairs_grid(d.PF), d.PF.bx_threads, 0, d.stream>>>(
                d, static_cast<T *>(lat), static_cast<const R *>(rho0), static_cast<const R *>(u0), pair);
        else
            k_init_eq_split<S, false><<<pairs_grid(d.PF), d.PF.bx_threads, 0, d.stream>>>(
                d, static_cast<T *>(lat), static_cast<const R *>(rho0), static_cast<const R *>(u0), pair);
    } else {
        Dev d = d0;
        d.PF = all_pairs(d.g);
        const bool pair = pair_aligned(d.g, u0, sizeof(R)) && (!rho0 || pair_aligned(d.g, rho0, sizeof(R)));
        if (d.flags)
            k_init_eq<S, true><<<pairs_grid(d.PF), d.PF.bx_threads, 0, d.stream>>>(
                d, static_cast<T *>(lat), static_cast<const R *>(rho0), static_cast<const R *>(u0), pair);
        else
            k_init_eq<S, false><<<pairs_grid(d.PF), d.PF.bx_threads, 0, d.stream>>>(
                d, static_cast<T *>(lat), static_cast<const R *>(rho0), static_cast<const R *>(u0), pair);
    }
    return cudaGetLastError();
}

template <int S, int D>
static cudaError_t launch_get(const Dev &d0, const void *lat, void *dst) {
    typedef typename Stor<S>::T T;
    typedef typename IOFmt<D>::T TD;
    if (d0.flags && !d0.mask) return cudaErrorInvalidValue;
    Dev d = d0;
    d.PF = all_pairs(d.g);
    const bool pair = pair_aligned(d.g, dst, sizeof(TD));
    void (*k)(Dev, const T *, TD *, bool) = d.flags ? k_get_state<S, D, true> : k_get_state<S, D, false>;
    if constexpr (D == LBM_F64 && S != LBM_F64 && !is_split(S)) {
        if ((d.g.nx & 1) && d.PF.bx_threads > 64) k = d.flags ? k_get_state<S, D, true, true> : k_get_state<S, D, false, true>;
    }
    k<<<pairs_grid(d.PF), d.PF.bx_threads, 0, d.stream>>>(d, static_cast<const T *>(lat), static_cast<TD *>(dst), pair);
    return cudaGetLastError();
}

template <int S, int D>
static cudaError_t launch_set(const Dev &d0, void *lat, const void *src) {
    typedef typename Stor<S>::T T;
    typedef typename IOFmt<D>::T TD;
    if (d0.flags && !d0.mask) return cudaErrorInvalidValue;
    Dev d = d0;
    d.PF = all_pairs(d.g);
    const bool pair = pair_aligned(d.g, src, sizeof(TD));
    if (d.flags)
        k_set_state<S, D, true><<<pairs_grid(d.PF), d.PF.bx_threads, 0, d.stream>>>(
            d, static_cast<T *>(lat), static_cast<const TD *>(src), pair);
    else
        k_set_state<S, D, false><<<pairs_grid(d.PF), d.PF.bx_threads, 0, d.stream>>>(
            d, static_cast<T *>(lat), static_cast<const TD *>(src), pair);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || d.layout != LAYOUT_PULL) return e;
    return Ops<S>::bounce(d, lat);  // the link form's solid slots, from their fluid cells' own (1343 us for the
                                    // porous channel with scattered stores from the kernel above)
}

template <int S>
cudaError_t Ops<S>::get_state(const Dev &d, const void *lat, void *dst, int fmt) {
    switch (fmt) {
    case LBM_F64: return launch_get<S, LBM_F64>(d, lat, dst);
    case LBM_F32: return launch_get<S, LBM_F32>(d, lat, dst);
    case LBM_F16S: case LBM_F16M: return launch_get<S, LBM_F16S>(d, lat, dst);
    case LBM_BF16S: case LBM_BF16M: return launch_get<S, LBM_BF16S>(d, lat, dst);
    }
    return cudaErrorInvalidValue;
}

template <int S>
cudaError_t Ops<S>::set_state(const Dev &d, void *lat, const void *src, int fmt) {
    switch (fmt) {
    case LBM_F64: return launch_set<S, LBM_F64>(d, lat, src);
    case LBM_F32: return launch_set<S, LBM_F32>(d, lat, src);
    case LBM_F16S: case LBM_F16M: return launch_set<S, LBM_F16S>(d, lat, src);
    case LBM_BF16S: case LBM_BF16M: return launch_set<S, LBM_BF16S>(d, lat, src);
    }
    return cudaErrorInvalidValue;
}

template <int S, bool FLAGS>
static cudaError_t launch_macros(const Dev &d0, const void *lat, void *rho, void *u) {
    typedef typename Stor<S>::T T;
    typedef typename Stor<S>::R R;
    if (d0.flags && !d0.mask) return cudaErrorInvalidValue;
    Dev d = d0;
    d.PF = all_pairs(d.g);
    const bool pair = pair_aligned(d.g, u, sizeof(R)) && (!rho || pair_aligned(d.g, rho, sizeof(R)));
    if (d.force_on)
        k_macros<S, FLAGS, true><<<pairs_grid(d.PF), d.PF.bx_threads, 0, d.stream>>>(
            d, static_cast<const T *>(lat), static_cast<R *>(rho), static_cast<R *>(u), pair);
    else
        k_macros<S, FLAGS, false><<<pairs_grid(d.PF), d.PF.bx_threads, 0, d.stream>>>(
            d, static_cast<const T *>(lat), static_cast<R *>(rho), static_cast<R *>(u), pair);
    return cudaGetLastError();
}

template <int S>
cudaError_t Ops<S>::macros(const Dev &d, const void *lat, void *rho, void *u) {
    return d.flags ? launch_macros<S, true>(d, lat, rho, u) : launch_macros<S, false>(d, lat, rho, u);
}

template <int S, bool FLAGS>
static cudaError_t launch_reduce(const Dev &d, const void *lat, int z0, int z1, double *partials, int blocks) {
    typedef typename Stor<S>::T T;
    if (d.flags && !d.mask) return cudaErrorInvalidValue;
    if (d.force_on)
        k_reduce<S, FLAGS, true><<<blocks, RED_THREADS, 0, d.stream>>>(d, static_cast<const T *>(lat), z0, z1,
                                                                      partials);
    else
        k_reduce<S, FLAGS, false><<<blocks, RED_THREADS, 0, d.stream>>>(d, static_cast<const T *>(lat), z0, z1,
                                                                       partials);
    return cudaGetLastError();
}

template <int S>
cudaError_t Ops<S>::reduce(const Dev &d, const void *lat, int z0, int z1, double *partials, double *out) {
    // one pair a thread, at most RED_BLOCKS blocks
    const long long want = ((long long)(d.g.nx + 1) / 2 * d.g.ny * (z1 - z0) + RED_THREADS - 1) / RED_THREADS;
    const int blocks = (int)(want < 1 ? 1 : (want < RED_BLOCKS ? want : RED_BLOCKS));
    cudaError_t e = d.flags ? launch_reduce<S, true>(d, lat, z0, z1, partials, blocks)
                            : launch_reduce<S, false>(d, lat, z0, z1, partials, blocks);
    if (e != cudaSuccess) return e;
    return sum_partials(partials, blocks, nullptr, out, d.stream);
}

template <int S, bool FLAGS>
static cudaError_t launch_seed(const Dev &d0, const void *lat, const void *dL_du, const void *dL_drho, void *lam,
                               void *grad_F) {
    typedef typename Stor<S>::T T;
    typedef typename Stor<S>::R R;
    if (d0.flags && !d0.mask) return cudaErrorInvalidValue;
    Dev d = d0;
    d.PF = all_pairs(d.g);
    const bool pair = pair_aligned(d.g, dL_du, sizeof(R)) && (!dL_drho || pair_aligned(d.g, dL_drho, sizeof(R)));
    if (d.force_on)
        k_adj_seed<S, FLAGS, true><<<pairs_grid(d.PF), d.PF.bx_threads, 0, d.stream>>>(
            d, static_cast<const T *>(lat), static_cast<const R *>(dL_du), static_cast<const R *>(dL_drho),
            static_cast<R *>(lam), static_cast<R *>(grad_F), pair);
    else
        k_adj_seed<S, FLAGS, false><<<pairs_grid(d.PF), d.PF.bx_threads, 0, d.stream>>>(
            d, static_cast<const T *>(lat), static_cast<const R *>(dL_du), static_cast<const R *>(dL_drho),
            static_cast<R *>(lam), static_cast<R *>(grad_F), pair);
    return cudaGetLastError();
}

template <int S>
cudaError_t Ops<S>::adj_seed(const Dev &d, const void *lat, const void *dL_du, const void *dL_drho, void *lam,
                             void *grad_F) {
    return d.flags ? launch_seed<S, true>(d, lat, dL_du, dL_drho, lam, grad_F)
                   : launch_seed<S, false>(d, lat, dL_du, dL_drho, lam, grad_F);
}

}  // namespace lbm
