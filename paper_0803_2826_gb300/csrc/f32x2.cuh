// f32x2.cuh -- the collision of two neighbouring nodes at once in Blackwell's
// packed FP32 arithmetic (add / sub / mul / fma .rn.f32x2: one instruction
// computes the same IEEE operation on the two 32-bit halves of a 64-bit
// register pair).
//
// The paired stream-collide kernels hold nodes x0 and x0 + 1 of a row in
// every thread and do the same arithmetic on both; here the two values of a
// quantity travel as one F2 (low half: node x0, high half: node x0 + 1), so
// the moment transform (Table 1, Eq. forward), the relaxation and forcing
// (Eq. lco_update, Sec. 3.7 Sigma), the Box-Muller scaling of the noise
// (Sec. 3.5) and the back transform (Eq. back_transformation) issue one
// instruction per operation for the pair instead of two.  Operations without
// a packed form (reciprocal, log2, rsqrt, sine / cosine, the Philox integer
// rounds, compares) run per half.  Every packed operation rounds each half
// exactly as the scalar operation would, so the results are those of
// collide_node (stream_collide.cuh) up to which multiplications the assembler
// joins with an addition behind them: with noise to the bit, without it but for
// the last bit of some values where gamma_odd or gamma_even is not 0.
#pragma once

#include <cstdint>

#include "d3q19.cuh"
#include "step_args.h"

namespace lbp {

struct F2 {
    unsigned long long v;
};

__device__ __forceinline__ F2 f2(float lo, float hi)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ F2 f2s(float c) { return f2(c, c); }
__device__ __forceinline__ void split(F2 a, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ float lo(F2 a)
{
    float l, h;
    split(a, l, h);
    return l;
}
__device__ __forceinline__ float hi(F2 a)
{
    float l, h;
    split(a, l, h);
    return h;
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b)
{
    F2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b)
{
    F2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b)
{
    F2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
// a * b + c, rounded once per half
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c)
{
    F2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return d;
}
__device__ __forceinline__ F2 fma2(F2 a, float b, F2 c) { return fma2(a, f2s(b), c); }
__device__ __forceinline__ F2 operator*(F2 a, float b) { return a * f2s(b); }

// Forward transform m_k = sum_i e_ki n_i (Eq. forward, Table 1) of both nodes:
// the even / odd factorisation of lbd::forward.
__device__ __forceinline__ void forward2(const F2 n[19], F2 m[19])
{
    const F2 sx = n[1] + n[2], sy = n[3] + n[4], sz = n[5] + n[6];
    const F2 sa = n[7] + n[10], sb = n[8] + n[9];
    const F2 sc = n[11] + n[14], sd = n[12] + n[13];
    const F2 se = n[15] + n[18], sg = n[16] + n[17];
    const F2 dx = n[1] - n[2], dy = n[3] - n[4], dz = n[5] - n[6];
    const F2 pa = n[7] - n[10], pb = n[8] - n[9];
    const F2 pc = n[11] - n[14], pd = n[12] - n[13];
    const F2 pe = n[15] - n[18], pg = n[16] - n[17];

    const F2 A = sx + sy + sz;
    const F2 Dxy = sa + sb, Dyz = sc + sd, Dxz = se + sg;
    const F2 D = Dxy + Dyz + Dxz;
    const F2 t5 = (Dxy + Dxz) - (Dyz + Dyz);
    const F2 t6 = Dxy - Dxz;
    const F2 syz = sy + sz;
    const F2 sx2 = sx + sx;
    m[0] = n[0] + A + D;
    m[4] = D - n[0];
    m[5] = sx2 - syz + t5;
    m[6] = sy - sz + t6;
    m[7] = sa - sb;
    m[8] = sc - sd;
    m[9] = se - sg;
    m[16] = n[0] - (A + A) + D;
    m[17] = syz - sx2 + t5;
    m[18] = sz - sy + t6;

    const F2 Px = pa + pb, Qx = pe + pg;
    const F2 Py = pa - pb, Qy = pc + pd;
    const F2 Pz = pc - pd, Qz = pe - pg;
    const F2 hx = Px + Qx, hy = Py + Qy, hz = Pz + Qz;
    m[1] = dx + hx;
    m[2] = dy + hy;
    m[3] = dz + hz;
    m[10] = hx - (dx + dx);
    m[11] = hy - (dy + dy);
    m[12] = hz - (dz + dz);
    m[13] = Px - Qx;
    m[14] = Qy - Py;
    m[15] = Qz - Pz;
}

// The conserved moments m_0 .. m_3 alone (mass and momentum).
__device__ __forceinline__ void forward2_conserved(const F2 n[19], F2 m[4])
{
    const F2 sa = n[7] + n[10], sb = n[8] + n[9], sc = n[11] + n[14], sd = n[12] + n[13];
    const F2 se = n[15] + n[18], sg = n[16] + n[17];
    const F2 pa = n[7] - n[10], pb = n[8] - n[9], pc = n[11] - n[14], pd = n[12] - n[13];
    const F2 pe = n[15] - n[18], pg = n[16] - n[17];
    const F2 A = (n[1] + n[2]) + (n[3] + n[4]) + (n[5] + n[6]);
    m[0] = n[0] + A + ((sa + sb) + (sc + sd) + (se + sg));
    m[1] = (n[1] - n[2]) + ((pa + pb) + (pe + pg));
    m[2] = (n[3] - n[4]) + ((pa - pb) + (pc + pd));
    m[3] = (n[5] - n[6]) + ((pc - pd) + (pe - pg));
}

// Back transform n_i = a_i sum_k e_ki M_k (M_k = m_k / w_k, but m_k itself for
// k = 1..3) of both nodes: lbd::backward in packed form.  WEIGHTED false leaves
// the a_i and that factor out, which is the transpose of forward2 (the reverse
// mode's dL/dn_i = sum_k e_ki mu_k).
template <bool WEIGHTED>
__device__ __forceinline__ F2 weigh(float a, F2 v) { return WEIGHTED ? f2s(a) * v : v; }

// M_k + v for k = 1..3.  WEIGHTED: M holds m_k, not yet over its norm 1/3, and
// the momentum, the largest of the moments, is multiplied and added in one rounding.
template <bool WEIGHTED>
__device__ __forceinline__ F2 plus3(F2 j, F2 v) { return WEIGHTED ? fma2(j, f2s(3.0f), v) : j + v; }

template <bool WEIGHTED = true>
__device__ __forceinline__ void backward2(const F2 M[19], F2 n[19])
{
    const F2 M5x2 = M[5] + M[5], M16x2 = M[16] + M[16], M17x2 = M[17] + M[17];
    n[0] = weigh<WEIGHTED>(lbd::kA0, M[0] - M[4] + M[16]);
    {
        const F2 base = M[0] - M16x2;
        const F2 Ex = base + M5x2 - M17x2;
        const F2 Ox = plus3<WEIGHTED>(M[1], f2s(-2.0f) * M[10]);
        const F2 Eyz = base - M[5] + M[17];
        const F2 Ey = Eyz + M[6] - M[18];
        const F2 Ez = Eyz - M[6] + M[18];
        const F2 Oy = plus3<WEIGHTED>(M[2], f2s(-2.0f) * M[11]);
        const F2 Oz = plus3<WEIGHTED>(M[3], f2s(-2.0f) * M[12]);
        n[1] = weigh<WEIGHTED>(lbd::kA1, Ex + Ox);
        n[2] = weigh<WEIGHTED>(lbd::kA1, Ex - Ox);
        n[3] = weigh<WEIGHTED>(lbd::kA1, Ey + Oy);
        n[4] = weigh<WEIGHTED>(lbd::kA1, Ey - Oy);
        n[5] = weigh<WEIGHTED>(lbd::kA1, Ez + Oz);
        n[6] = weigh<WEIGHTED>(lbd::kA1, Ez - Oz);
    }
    {
        const F2 base = M[0] + M[4] + M[16];
        const F2 Exy = base + M[5] + M[6] + M[17] + M[18];
        const F2 E7 = Exy + M[7], E8 = Exy - M[7];
        const F2 oxy1 = plus3<WEIGHTED>(M[1], M[10]) + M[13];
        const F2 oxy2 = plus3<WEIGHTED>(M[2], M[11]) - M[14];
        const F2 O7 = oxy1 + oxy2, O8 = oxy1 - oxy2;
        n[7] = weigh<WEIGHTED>(lbd::kA2, E7 + O7);
        n[10] = weigh<WEIGHTED>(lbd::kA2, E7 - O7);
        n[8] = weigh<WEIGHTED>(lbd::kA2, E8 + O8);
        n[9] = weigh<WEIGHTED>(lbd::kA2, E8 - O8);
        const F2 Eyz = base - M5x2 - M17x2;
        const F2 E11 = Eyz + M[8], E12 = Eyz - M[8];
        const F2 oyz2 = plus3<WEIGHTED>(M[2], M[11]) + M[14];
        const F2 oyz3 = plus3<WEIGHTED>(M[3], M[12]) - M[15];
        const F2 O11 = oyz2 + oyz3, O12 = oyz2 - oyz3;
        n[11] = weigh<WEIGHTED>(lbd::kA2, E11 + O11);
        n[14] = weigh<WEIGHTED>(lbd::kA2, E11 - O11);
        n[12] = weigh<WEIGHTED>(lbd::kA2, E12 + O12);
        n[13] = weigh<WEIGHTED>(lbd::kA2, E12 - O12);
        const F2 Exz = base + M[5] - M[6] + M[17] - M[18];
        const F2 E15 = Exz + M[9], E16 = Exz - M[9];
        const F2 oxz1 = plus3<WEIGHTED>(M[1], M[10]) - M[13];
        const F2 oxz3 = plus3<WEIGHTED>(M[3], M[12]) + M[15];
        const F2 O15 = oxz1 + oxz3, O16 = oxz1 - oxz3;
        n[15] = weigh<WEIGHTED>(lbd::kA2, E15 + O15);
        n[18] = weigh<WEIGHTED>(lbd::kA2, E15 - O15);
        n[16] = weigh<WEIGHTED>(lbd::kA2, E16 + O16);
        n[17] = weigh<WEIGHTED>(lbd::kA2, E16 - O16);
    }
}

// -2 ln(1 - d) = 2 d + d^2 + kLog3 d^3 + kLog4 d^4 + kLog5 d^5 for d in [0, 2^-5]:
// the three coefficients are fitted for the least relative error there, 2.2e-11
// (the Taylor coefficients 2/3, 1/2, 2/5 leave 5.0e-9, one term more 1.3e-10).
constexpr float kLog3 = 0.666670024f, kLog4 = 0.499496400f, kLog5 = 0.423335731f;

// Box-Muller pairs of the two nodes (words (a0, b0) of node x0, (a1, b1) of
// node x0 + 1): the map of lbd::box_muller -- uniforms (2 (w >> 9) + 1) 2^-24
// from the mantissa bits, -2 ln v1 from the hardware log2 or the series near
// 1, the radius sqrt(-2 ln v1) as L rsqrt(L), the centred angle -- to FP32
// rounding, with the arithmetic packed and the special functions per half.
// nsd is minus the standard deviation (a factor of the radius: -2 ln v1 alone
// goes through the reciprocal square root, so the amplitude of a node is one
// square root however small it is; the sign of the centred angle's sine and
// cosine costs nothing there, and a negation per half elsewhere).
__device__ __forceinline__ void box_muller2(uint32_t a0, uint32_t b0, uint32_t a1, uint32_t b1, F2 &g0, F2 &g1,
                                            F2 nsd)
{
    const F2 v1 = f2(lbd::one_to_two(a0), lbd::one_to_two(a1)) - f2s(0.99999994039535522f);
    const F2 d1 = f2s(1.0f) - v1;
    // 2 pi (v2 - 1/2) = 2 pi (m - 3/2) + 2 pi 2^-24, m the float in [1, 2) of the word
    const F2 ang = fma2(f2(lbd::one_to_two(b0), lbd::one_to_two(b1)) - f2s(1.5f), f2s(6.283185307179586f),
                        f2s(3.7450704e-07f));
    float v1l, v1h, d1l, d1h;
    split(v1, v1l, v1h);
    split(d1, d1l, d1h);
    const F2 lg = f2(lbd::log2_normal(v1l), lbd::log2_normal(v1h)) * f2s(-1.3862943611198906f);
    F2 t = fma2(d1, f2s(kLog5), f2s(kLog4));
    t = fma2(d1, t, f2s(kLog3));
    t = fma2(d1, t, f2s(1.0f));
    t = fma2(d1, t, f2s(2.0f));
    const F2 ser = d1 * t;
    float sl, sh, ll, lh;
    split(ser, sl, sh);
    split(lg, ll, lh);
    const float Ll = d1l < 0.03125f ? sl : ll, Lh = d1h < 0.03125f ? sh : lh;
    const F2 nr = f2(Ll, Lh) * f2(lbd::rsqrt_normal(Ll), lbd::rsqrt_normal(Lh)) * nsd;  // -sqrt(L) sd
    float al, ah, s0, c0, s1, c1;
    split(ang, al, ah);
    __sincosf(al, &s0, &c0);
    __sincosf(ah, &s1, &c1);
    g0 = nr * f2(c0, c1);
    g1 = nr * f2(s0, s1);
}

// The same for one node.
__device__ __forceinline__ void box_muller1(uint32_t a, uint32_t b, float &g0, float &g1, float nsd)
{
    const float v1 = lbd::one_to_two(a) - 0.99999994039535522f;
    const float d1 = 1.0f - v1;
    const float ang = fmaf(lbd::one_to_two(b) - 1.5f, 6.283185307179586f, 3.7450704e-07f);
    const float lg = __fmul_rn(lbd::log2_normal(v1), -1.3862943611198906f);
    float t = fmaf(d1, kLog5, kLog4);
    t = fmaf(d1, t, kLog3);
    t = fmaf(d1, t, 1.0f);
    t = fmaf(d1, t, 2.0f);
    const float L = d1 < 0.03125f ? __fmul_rn(d1, t) : lg;
    const float nr = __fmul_rn(__fmul_rn(L, lbd::rsqrt_normal(L)), nsd);
    float s, c;
    __sincosf(ang, &s, &c);
    g0 = __fmul_rn(nr, c);
    g1 = __fmul_rn(nr, s);
}

// -sqrt(mu rho) of both nodes (mu rho0 where the amplitude is the reference's).
__device__ __forceinline__ F2 noise_nsd(const lbi::StepArgs &a, F2 rho)
{
    if (a.noise_rho0) return f2s(-sqrtf(a.mu * a.rho0));
    float l, h;
    split(rho * a.mu, l, h);
    return f2(-sqrtf(l), -sqrtf(h));
}

// Where add_noise2 takes its Philox round keys: ParamKeys reads the
// precomputed keys of one seed (kernel parameters: constant-bank operands);
// RunningKeys forms round r's keys as key + r W from the two key words (two
// adds a round, but only two registers: for kernels whose key is data, e.g.
// one per replica, and which would otherwise hold all twenty).  pair() runs
// the two nodes' counter blocks.
struct ParamKeys {
    const lbd::RoundKeys &rk;
    __device__ __forceinline__ void pair(const lbd::U4 &c0, const lbd::U4 &c1, lbd::U4 &r0, lbd::U4 &r1) const
    {
        r0 = lbd::philox10(c0, rk);
        r1 = lbd::philox10(c1, rk);
    }
};
struct RunningKeys {
    uint32_t k0, k1;
    __device__ __forceinline__ void pair(const lbd::U4 &c0, const lbd::U4 &c1, lbd::U4 &r0, lbd::U4 &r1) const
    {
        r0 = c0;
        r1 = c1;
#pragma unroll
        for (int r = 0; r < 10; ++r) {
            const uint32_t q0 = k0 + (uint32_t)r * lbd::kPhiloxW0, q1 = k1 + (uint32_t)r * lbd::kPhiloxW1;
            lbd::philox_round(r0, q0, q1);
            lbd::philox_round(r1, q0, q1);
        }
    }
};

// The deterministic part of the collision of two nodes (Sec. 3.4, 3.7): from
// their moments m and force densities (fx, fy, fz) to the post-collision
// moments over w_k, M, and the densities.  The noisy update is bound by
// instruction issue, so constants are multiplied on the host where that costs
// no accuracy and the forcing is passed over where nothing forces; with the
// Box-Muller map above, 256^3 FP16 376 us a step (396 before), 512 replicas
// 1.26 ms (1.29), 200^3 FP32 180 us (188), 256^3 FP32 365 us (382).
__device__ __forceinline__ void relax2(const F2 m[19], F2 fx, F2 fy, F2 fz, const lbi::StepArgs &a, F2 M[19], F2 &rho)
{
    const F2 half = f2s(0.5f), three = f2s(3.0f);
    rho = f2s(a.rho0) + m[0];
    float rl, rh;
    split(rho, rl, rh);
    const F2 inv_rho = f2(__frcp_rn(rl), __frcp_rn(rh));
    const F2 ux = fma2(half, fx, m[1]) * inv_rho;
    const F2 uy = fma2(half, fy, m[2]) * inv_rho;
    const F2 uz = fma2(half, fz, m[3]) * inv_rho;

    const F2 uxx = ux * ux, uyy = uy * uy, uzz = uz * uz;
    const F2 u2 = uxx + uyy + uzz;
    // M_k = (gamma_k (m_k - m^eq_k) + m^eq_k + F_k) / w_k: the rounding of gamma_k
    // only meets the difference, nothing cancels however small gamma_k is, and
    // 1 / w_k is exact.  (gamma_k / w_k and (1 - gamma_k) / w_k from the host save
    // a quarter of these operations: 2 to 3% of a step of a box in the L2, 148 x 23
    // x 271 24.1 against 24.8 us, 1.2% of a batched step, 0.4% or less of larger
    // boxes; but they round to a factor of up to 1 + 1e-7 on a moment at equilibrium.)
    const F2 ruy = rho * uy, nrho = f2s(-a.rho0) - m[0], nruy = nrho * uy;
    const F2 t5 = uxx * three - u2, t6 = uyy - uzz;
    F2 S[6] = {rho * u2, rho * t5, rho * t6, ruy * ux, ruy * uz, rho * uz * ux};  // m^eq
    const F2 d[6] = {fma2(nrho, u2, m[4]), fma2(nrho, t5, m[5]),  fma2(nrho, t6, m[6]),
                     fma2(nruy, ux, m[7]), fma2(nruy, uz, m[8]), fma2(nrho * uz, ux, m[9])};
    F2 jx = m[1], jy = m[2], jz = m[3];
    M[0] = m[0];
    if (a.forced) {  // the same for the whole launch
        const F2 uf = ux * fx + uy * fy + uz * fz;
        S[0] = fma2(uf, a.frc[0], S[0]);
        S[1] = fma2(ux * fx * three - uf, a.frc[1], S[1]);
        S[2] = fma2(uy * fy - uz * fz, a.frc[1], S[2]);
        S[3] = fma2(ux * fy + uy * fx, a.frc[2], S[3]);
        S[4] = fma2(uy * fz + uz * fy, a.frc[2], S[4]);
        S[5] = fma2(uz * fx + ux * fz, a.frc[2], S[5]);
        jx = jx + fx;
        jy = jy + fy;
        jz = jz + fz;
    }
    M[1] = jx;  // (backward2 multiplies by 1 / w = 3)
    M[2] = jy;
    M[3] = jz;
#pragma unroll
    for (int k = 4; k < 10; ++k)
        M[k] = fma2(d[k - 4], k == 4 ? a.g_bulk : a.g_shear, S[k - 4]) * lbd::inv_w(k);
#pragma unroll
    for (int k = 10; k < 19; ++k) M[k] = m[k] * a.rel[k - 10];
}

// The noise of nodes node0, node0 + 1 (Sec. 3.5) added to M:
// sqrt(mu rho w_k) phi_k r_k / w_k is (phi_k / sqrt(w_k)) times a Gaussian of
// variance mu rho; the four Gaussians of each Philox block go into their
// modes at once (r_4 .. r_18 = Gaussians 0 .. 14).
template <class Keys>
__device__ __forceinline__ void add_noise2(F2 M[19], F2 rho, const lbi::StepArgs &a, const Keys &keys, uint32_t node0,
                                           uint32_t step, uint32_t replica)
{
    const F2 nsd = noise_nsd(a, rho);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        lbd::U4 r0, r1;
        keys.pair(lbd::U4{node0, step, (uint32_t)b, replica}, lbd::U4{node0 + 1u, step, (uint32_t)b, replica}, r0, r1);
        F2 g[4];
        box_muller2(r0.x, r0.y, r1.x, r1.y, g[0], g[1], nsd);
        box_muller2(r0.z, r0.w, r1.z, r1.w, g[2], g[3], nsd);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int k = 4 + 4 * b + j;
            if (k < 19) M[k] = fma2(g[j], a.amp[k - 4], M[k]);
        }
    }
}

// Collision of nodes node0, node0 + 1 from their moments m and force densities
// to the post-collision deviations out: lbi::collide_node of each node, paired.
template <bool NOISE>
__device__ __forceinline__ void collide_moments2(const F2 m[19], F2 fx, F2 fy, F2 fz, const lbi::StepArgs &a,
                                                 const lbd::RoundKeys &rk, uint32_t node0, uint32_t replica,
                                                 F2 out[19])
{
    F2 M[19], rho;
    relax2(m, fx, fy, fz, a, M, rho);
    if (NOISE) add_noise2(M, rho, a, ParamKeys{rk}, node0, a.step, replica);
    backward2(M, out);
}

}  // namespace lbp
