// FP64 moments and collision of one cell in block fixed point.
//
// GB300 executes FP64 arithmetic at 2 operations a clock and SM, and integer
// arithmetic at 64 to 128: an update's 164 FP64 operations held the FP64 step
// at 0.12 of copy bandwidth (1383 us on the 256x128x128 channel; 280 us in this
// form). Here a cell's 19 deviations s_i (and half its force)
// are aligned to one exponent, that of the largest of them, as 64-bit integers
// with the largest in [2^57, 2^58): 5 bits finer than its FP64 spacing. Sums
// of them are exact. Products are rounded to nearest and keep 2 more bits. What is
// added to (1 - omega) s_i comes back as a double, correctly rounded, and one FP64
// multiply-add per population is left.
//
// Against extended precision, relative to the cell's largest value, the
// post-collision values are off (rms) by 0.2 to 1.0 times what the FP64 form is, the
// momentum they carry by 0.1 to 1.04 times, with no mean in it: for tau from 0.5005
// to 50, flows of 1e-9 to 0.2 with density deviations up to 0.2, noise, and forces
// from none to the largest value of the cell (tests/test_fixed64_cpu.py). Equilibria
// and moments are off by 0.4 to 0.7 times. (With inputs cut at 2^-56, products rounded
// to that unit and a fixed offset for their dropped low parts, the momentum was off
// by up to 2.8 times and had a mean of a few 1e-17 of either sign, by tau: a body
// force. The step took 272 us.)
//
// With j' = j + F/2, u = j'/rho (u = j' in the incompressible model) and
// c = 1 - omega/2, collide2's E and P (omega folded in) are, in
//   g = (omega j' + c F)/12,  h = g + c F/12,  v = 3/2 u,
//   X_a = v_a h_a,  X_ab = v_a h_b + v_b h_a,
//   B = omega (rho - 1)/36 - (X_x + X_y + X_z)/3:
//   rest 12 B;  axis a  E = 2 (B + X_a), P = 2 g_a;
//   diagonal (a, +-b)  E = B + X_a + X_b +- X_ab, P = g_a +- g_b.
#pragma once

#include <math.h>
#include <string.h>

#include "lbm_device.cuh"

namespace lbm {

// Constants of the collision as 62-bit fractions (value 2^62, rounded). omega is
// taken as 1 - (1 - omega), so that it and the rounded 1 - omega add up to 1: else
// every step would scale mass and momentum by the rounding (tau = 5: 1 + 5.6e-17).
struct FixedK {
    long long w9, w12, c6;  // omega/9, omega/12, (1 - omega/2)/6
    double omc;             // 1 - omega
};
inline FixedK fixed_k(double omega) {
    FixedK k;
    k.omc = 1.0 - omega;
    const long long w = (long long)ldexp(1.0 - k.omc, 61);  // omega < 2
    k.w9 = (w * 2 + 4) / 9;
    k.w12 = (w + 3) / 6;
    k.c6 = ((1LL << 62) - w + 3) / 6;  // (2^62 - omega 2^61) / 6
    return k;
}

LBM_HD uint32_t fx_hi(double a) {
#ifdef __CUDA_ARCH__
    return (uint32_t)__double2hiint(a);
#else
    uint64_t b;
    memcpy(&b, &a, 8);
    return (uint32_t)(b >> 32);
#endif
}
LBM_HD uint32_t fx_lo(double a) {
#ifdef __CUDA_ARCH__
    return (uint32_t)__double2loint(a);
#else
    uint64_t b;
    memcpy(&b, &a, 8);
    return (uint32_t)b;
#endif
}
LBM_HD double fx_double(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi, (int)lo);
#else
    const uint64_t b = ((uint64_t)hi << 32) | lo;
    double a;
    memcpy(&a, &b, 8);
    return a;
#endif
}
// The place of the leading one of a, -1 for 0.
LBM_HD int fx_top(uint64_t a) {
#ifdef __CUDA_ARCH__
    int p;
    asm("bfind.u64 %0, %1;" : "=r"(p) : "l"(a));
    return p;
#else
    return a ? 63 - __builtin_clzll(a) : -1;
#endif
}
// -q where sign is negative: a predicated negation, two instructions fewer than
// xor and subtract. (With it, the leading one found in one go and the rounding in
// one addition, the channel step went from 312 to 266 us.)
LBM_HD long long fx_neg_if(long long q, int sign) {
#ifdef __CUDA_ARCH__
    asm("{\n .reg .pred p;\n setp.lt.s32 p, %1, 0;\n @p neg.s64 %0, %0;\n}" : "+l"(q) : "r"(sign));
    return q;
#else
    return sign < 0 ? -q : q;
#endif
}
// a >> n, 0 from n = 64 on.
LBM_HD uint64_t fx_shr(uint64_t a, int n) {
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));
    return r;
#else
    return n < 64 ? a >> n : 0;
#endif
}

// a 2^(57 - (E - 1023)), E >= the exponent field of a; towards zero.
LBM_HD long long fx_in(double a, int E) {
    const uint32_t h = fx_hi(a);
    const int sh = E + 5 - (int)((h >> 20) & 0x7ffu);
    const uint64_t q = ((((uint64_t)((h & 0xfffffu) | 0x100000u)) << 32) | fx_lo(a)) << 10;
    return fx_neg_if((long long)fx_shr(q, sh), (int)h);
}

// q 2^((E - 1023) - 57), |q| < 2^63, rounded to nearest (ties away from zero).
LBM_HD double fx_out(long long q, int E) {
    const int qh = (int)(q >> 32);
    const uint64_t a = (uint64_t)fx_neg_if(q, qh);
    const int p = fx_top(a);
    // the leading one to bit 62, half a unit of the 53 bits kept added (the
    // leading bit adds the last 1 of the exponent field, a carry one more)
    const uint64_t r = ((a << (62 - p)) + (1u << 9)) >> 10;
    uint32_t hi = (uint32_t)(r >> 32) + ((uint32_t)(E + p - 58) << 20);
    hi = (hi & 0x7fffffffu) | ((uint32_t)qh & 0x80000000u);
    return fx_double(p < 0 ? 0u : hi, (uint32_t)r);
}

// Limbs of 31 bits: a = h 2^31 + l, |a| < 2^62; products of limbs fit signed
// 64 bits, two at a time.
struct L31 {
    int h, l;
};
LBM_HD L31 limbs(long long a) { return L31{(int)(a >> 31), (int)((uint32_t)a & 0x7fffffffu)}; }
LBM_HD uint32_t fx_mulhi(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
// a b / 2^(62 - K), rounded to nearest (to within 2^(K - 31)); |the result| < 2^63.
// (b, the factor that several products share or a constant, is the one shifted.)
template <int K> LBM_HD long long mulk(L31 a, L31 b) {
    const uint32_t ll = fx_mulhi((uint32_t)a.l, (uint32_t)b.l << 1);
    const long long mid = (long long)a.h * b.l + ((long long)a.l * b.h + (long long)(ll + (1u << (30 - K))));
    return (long long)((unsigned long long)((long long)a.h * b.h) << K) + (mid >> (31 - K));
}

// The moments of a cell: rho - 1, j' and F/2 in units of 2^((E - 1023) - 57).
struct FixedMom {
    int E;
    long long r, jx, jy, jz, fx, fy, fz;
};

// False where the cell is outside the range of the fixed-point collision
// (|s_i| or |F|, |rho - 1| or |j'| >= 1/4, or the latter 8 to 16 times the largest of
// the s_i and F, or not finite): the caller then takes FP64 arithmetic. (A flow near
// equilibrium has |rho - 1| < 4 and |j'| < 6 times its largest s_i. With these limits
// |u| <= 1/3, and every sum and product below stays within its 62 or 63 bits.)
template <bool FORCE>
LBM_HD bool fixed_moments(const double s[Q], double Fx, double Fy, double Fz, FixedMom &m) {
    uint32_t top = 128u << 20;  // (values below 2^-895 count as zero; keeps every result a normal number)
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const uint32_t a = fx_hi(s[i]) & 0x7fffffffu;
        top = a > top ? a : top;
    }
    if (FORCE) {
        const uint32_t a = fx_hi(Fx) & 0x7fffffffu, b = fx_hi(Fy) & 0x7fffffffu, c = fx_hi(Fz) & 0x7fffffffu;
        top = a > top ? a : top;
        top = b > top ? b : top;
        top = c > top ? c : top;
    }
    const int E = (int)(top >> 20);
    m.E = E;
    if (E > 1020) return false;
    long long q[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) q[i] = fx_in(s[i], E);
    long long r = q[0];
#pragma unroll
    for (int i = 1; i < Q; ++i) r += q[i];
    m.r = r;
    m.jx = (q[1] - q[2]) + (q[7] - q[10]) + (q[8] - q[9]) + (q[11] - q[14]) + (q[12] - q[13]);
    m.jy = (q[3] - q[4]) + (q[7] - q[10]) + (q[9] - q[8]) + (q[15] - q[18]) + (q[16] - q[17]);
    m.jz = (q[5] - q[6]) + (q[11] - q[14]) + (q[13] - q[12]) + (q[15] - q[18]) + (q[17] - q[16]);
    m.fx = m.fy = m.fz = 0;
    if (FORCE) {
        m.fx = fx_in(Fx, E + 1);
        m.fy = fx_in(Fy, E + 1);
        m.fz = fx_in(Fz, E + 1);
        m.jx += m.fx;
        m.jy += m.fy;
        m.jz += m.fz;
    }
    // |r|, |j| < 2^61 units and 1/4 (compared in the high halves)
    const int n = 1023 - E;  // >= 3: the unit is 2^-(57 + n)
    const int rh = (int)(m.r >> 32), xh = (int)(m.jx >> 32), yh = (int)(m.jy >> 32), zh = (int)(m.jz >> 32);
    const int o = (rh ^ (rh >> 31)) | (xh ^ (xh >> 31)) | (yh ^ (yh >> 31)) | (zh ^ (zh >> 31));
    return (o >> (n < 6 ? 23 + n : 29)) == 0;
}
// s <- (1 - omega) s + E +- P (see the head of this file), or with EQ
// s <- E +- P: at omega = 1 and no force that is the equilibrium. g, h, X and B are
// held in quarters of m's unit, so that 2 (B + X) +- 2 g is whole in halves of it and
// 12 B in units.
template <bool FORCE, bool EQ = false>
LBM_HD void fixed_collide(double s[Q], const FixedMom &m, const FixedK &k, bool incomp) {
    const int n = 1023 - m.E;  // >= 3
    const int n2 = n - 1 < 63 ? n - 1 : 63, n0 = n + 1 < 63 ? n + 1 : 63;
    // j' and 3/2 / rho as 58- and 60-bit fractions
    const L31 j58x = limbs(m.jx >> n2), j58y = limbs(m.jy >> n2), j58z = limbs(m.jz >> n2);
    long long inv15 = 3LL << 59;
    if (!incomp) {
        // 1/rho, rho = R / 2^56 in [1/2, 3/2]: y = 2^30 (1 + e) / rho to 22 bits
        // from a float reciprocal, then y (1 + t), t = d + d^2, d = 1 - rho y
        const uint64_t R = (uint64_t)((1LL << 56) + (m.r >> n0));
        const uint32_t Rh = (uint32_t)((R + (1u << 31)) >> 32);
#ifdef __CUDA_ARCH__
        const uint32_t y = (uint32_t)__float2uint_rn(__fdividef(18014398509481984.0f, (float)Rh));
#else
        const uint32_t y = (uint32_t)(18014398509481984.0f / (float)Rh + 0.5f);
#endif
        const uint64_t p = (((R >> 32) * y) << 8) + (((R & 0xffffffffu) * y) >> 24);  // rho y, 62 bits
        const long long d = (long long)((1ULL << 62) - p);                             // |d| < 2^41
        const int dh = (int)(d >> 11);
        const long long t = d + (((long long)dh * dh) >> 40);
        // y t / 2^32
        const long long yt = (long long)y * (int)(t >> 32) + (long long)(((uint64_t)y * (uint32_t)t) >> 32);
        const long long inv = ((long long)y << 30) + yt;
        inv15 = inv + (inv >> 1);
    }
    const L31 iv = limbs(inv15);
    const L31 w12 = limbs(k.w12);
    long long gx = mulk<2>(limbs(m.jx), w12), gy = mulk<2>(limbs(m.jy), w12), gz = mulk<2>(limbs(m.jz), w12);
    long long hx = gx, hy = gy, hz = gz;
    if (FORCE) {
        const L31 c6 = limbs(k.c6);
        const long long cx = mulk<2>(limbs(m.fx), c6), cy = mulk<2>(limbs(m.fy), c6), cz = mulk<2>(limbs(m.fz), c6);
        gx += cx;
        gy += cy;
        gz += cz;
        hx = gx + cx;
        hy = gy + cy;
        hz = gz + cz;
    }
    // v as 60-bit fractions (|v| < 3/2)
    const L31 vx = limbs(mulk<4>(j58x, iv)), vy = limbs(mulk<4>(j58y, iv)), vz = limbs(mulk<4>(j58z, iv));
    const L31 lx = limbs(hx), ly = limbs(hy), lz = limbs(hz);
    const long long X = mulk<2>(vx, lx), Y = mulk<2>(vy, ly), Z = mulk<2>(vz, lz);
    const long long XY = FORCE ? mulk<2>(vx, ly) + mulk<2>(vy, lx) : mulk<2>(vx, ly) << 1;
    const long long XZ = FORCE ? mulk<2>(vx, lz) + mulk<2>(vz, lx) : mulk<2>(vx, lz) << 1;
    const long long YZ = FORCE ? mulk<2>(vy, lz) + mulk<2>(vz, ly) : mulk<2>(vy, lz) << 1;
    constexpr long long third = 1537228672809129301LL;  // 2^62 / 3
    const long long B = mulk<0>(limbs(m.r), limbs(k.w9)) - mulk<0>(limbs(X + Y + Z), limbs(third));
    const int E = m.E;
    s[0] = EQ ? fx_out(3 * B, E) : fma(k.omc, s[0], fx_out(3 * B, E));
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        const int i = pair_first(p);
        const int Ep = p < 3 ? E - 1 : E - 2;
        long long e, o;
        if (p == 0) { e = B + X; o = gx; }
        else if (p == 1) { e = B + Y; o = gy; }
        else if (p == 2) { e = B + Z; o = gz; }
        else if (ez(i) == 0) { e = B + X + Y + (ey(i) > 0 ? XY : -XY); o = ey(i) > 0 ? gx + gy : gx - gy; }
        else if (ey(i) == 0) { e = B + X + Z + (ez(i) > 0 ? XZ : -XZ); o = ez(i) > 0 ? gx + gz : gx - gz; }
        else { e = B + Y + Z + (ez(i) > 0 ? YZ : -YZ); o = ez(i) > 0 ? gy + gz : gy - gz; }
        s[i] = EQ ? fx_out(e + o, Ep) : fma(k.omc, s[i], fx_out(e + o, Ep));
        s[opp(i)] = EQ ? fx_out(e - o, Ep) : fma(k.omc, s[opp(i)], fx_out(e - o, Ep));
    }
}

// f_eq(1 + rho1, u) - w of one cell; false (f untouched) outside the range above.
LBM_HD bool fixed_equilibrium(double f[Q], double rho1, double ux, double uy, double uz, bool incomp) {
    uint32_t top = 128u << 20;
    const double v[4] = {rho1, ux, uy, uz};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t a = fx_hi(v[i]) & 0x7fffffffu;
        top = a > top ? a : top;
    }
    if ((top >> 20) > 1020u) return false;  // |rho1|, |u| < 1/4
    const int E = (int)(top >> 20) - 3;     // (the results are a sixth of u: 3 more bits)
    FixedMom m;
    m.E = E;
    m.r = fx_in(rho1, E);
    m.jx = fx_in(ux, E);
    m.jy = fx_in(uy, E);
    m.jz = fx_in(uz, E);
    m.fx = m.fy = m.fz = 0;
    if (!incomp) {  // j = u + rho1 u (rho1 as a 61-bit fraction)
        const int n = 1023 - E - 4;  // >= 2
        const L31 r = limbs(m.r >> (n < 63 ? n : 63));
        m.jx += mulk<1>(r, limbs(m.jx));
        m.jy += mulk<1>(r, limbs(m.jy));
        m.jz += mulk<1>(r, limbs(m.jz));
    }
    fixed_collide<false, true>(f, m, FixedK{0x071c71c71c71c71cLL, 0x0555555555555555LL, 0, 0.0}, incomp);
    return true;
}

}  // namespace lbm
