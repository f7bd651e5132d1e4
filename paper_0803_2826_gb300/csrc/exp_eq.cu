// exp_eq.cu -- the stream-collide update with the exponential equilibrium of
// Sec. 3.6, Eq. (equildist_lagrange): the populations that maximise the
// entropy of Eq. (boltzmann_entropy_function) at given mass and momentum,
// n^eq_i = rho a_i exp(lambda.c_i) / Z, Z = sum_i a_i exp(lambda.c_i), with
// lambda the root of sum_i a_i c_i exp(lambda.c_i) / Z = u.  The standard
// equilibrium of Eq. (original_equil_distrib) is its expansion to O(u^2);
// this one also has parts on the kinetic modes (O(u^3)), which the
// relaxation keeps.  Everything else is the collision of
// stream_collide.cuh: the same moments, eigenvalues, forcing and noise.
// Two nodes per thread with the arithmetic in packed FP32 (f32x2.cuh), as in
// the quadratic update.
//
// lambda comes from Newton's method in FP32 from the first-order value
// lambda = 3u: one step with the Jacobian of rest for |u| below 0.1, two with
// the full Jacobian above (kSlowFlow).  With
// x_i = exp(lambda.c_i) - 1 and s = sum_i a_i x_i the deviation from the
// reference state is n^eq_i - a_i rho0 = a_i (delta rho + rho (x_i - s) /
// (1 + s)): no difference of nearly equal numbers.
#include "stream_collide.cuh"

namespace lbi {

namespace {

using lbp::F2;

__device__ __forceinline__ F2 rcp2(F2 v)
{
    float l, h;
    lbp::split(v, l, h);
    return lbp::f2(__frcp_rn(l), __frcp_rn(h));
}

// x_i = exp(lambda.c_i) - 1 for the 18 moving directions of both nodes from
// ep_d = exp(lambda_d) - 1 and em_d = exp(-lambda_d) - 1:
// (1 + x)(1 + e) - 1 = x + e + x e over the (one or two) non-zero components
// of c_i.
__device__ __forceinline__ void exp_dirs2(const F2 ep[3], const F2 em[3], F2 x[19])
{
    x[0] = lbp::f2s(0.0f);
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        const int c3[3] = {lbd::cx(i), lbd::cy(i), lbd::cz(i)};
        F2 xi = lbp::f2s(0.0f);
        bool first = true;
#pragma unroll
        for (int d = 0; d < 3; ++d)
            if (c3[d] != 0) {
                const F2 e = c3[d] > 0 ? ep[d] : em[d];
                xi = first ? e : lbp::fma2(xi, e, xi + e);  // (1 + x)(1 + e) - 1
                first = false;
            }
        x[i] = xi;
    }
}

// exp(+-l) - 1: the expm1 per half, and exp(-a) - 1 = -x / (1 + x) for
// x = exp(a) - 1.
__device__ __forceinline__ void exp_axes2(const F2 l[3], F2 ep[3], F2 em[3])
{
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        float lo, hi;
        lbp::split(l[d], lo, hi);
        ep[d] = lbp::f2(expm1f(lo), expm1f(hi));
        em[d] = (lbp::f2s(0.0f) - ep[d]) * rcp2(lbp::f2s(1.0f) + ep[d]);
    }
}

// The same for |l| <= 0.3, from the power series of sinh and cosh - 1 up to
// l^7 and l^8 (remainder 6e-11).
__device__ __forceinline__ void exp_axes_small2(const F2 l[3], F2 ep[3], F2 em[3])
{
    const F2 one = lbp::f2s(1.0f);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const F2 q = l[d] * l[d];
        F2 s = lbp::fma2(q, 1.0f / 42.0f, one);
        s = lbp::fma2(q * s, 1.0f / 20.0f, one);
        s = lbp::fma2(q * s, 1.0f / 6.0f, one) * l[d];
        F2 c = lbp::fma2(q, 1.0f / 56.0f, one);
        c = lbp::fma2(q * c, 1.0f / 30.0f, one);
        c = lbp::fma2(q * c, 1.0f / 12.0f, one) * (q * 0.5f);
        ep[d] = c + s;
        em[d] = c - s;
    }
}

// sum_i a_i x_i and sum_i a_i c_i x_i of the moving directions.
__device__ __forceinline__ void exp_sums2(const F2 x[19], F2 &sm, F2 m[3])
{
    const F2 a1 = lbp::f2s(lbd::kA1), a2 = lbp::f2s(lbd::kA2);
    const F2 pa = x[7] - x[10], pb = x[8] - x[9], pc = x[11] - x[14], pd = x[12] - x[13];
    const F2 pe = x[15] - x[18], pg = x[16] - x[17];
    sm = lbp::fma2(a2, ((x[7] + x[10]) + (x[8] + x[9])) + ((x[11] + x[14]) + (x[12] + x[13])) +
                           ((x[15] + x[18]) + (x[16] + x[17])),
                   a1 * ((x[1] + x[2]) + (x[3] + x[4]) + (x[5] + x[6])));
    m[0] = lbp::fma2(a2, (pa + pb) + (pe + pg), a1 * (x[1] - x[2]));
    m[1] = lbp::fma2(a2, (pa - pb) + (pc + pd), a1 * (x[3] - x[4]));
    m[2] = lbp::fma2(a2, (pc - pd) + (pe - pg), a1 * (x[5] - x[6]));
}

// Two full Newton steps on lambda from 3u (|u| above kSlowFlow): the Jacobian
// is the covariance of c under the weights.
__device__ __forceinline__ void exp_newton2(const F2 u[3], F2 l[3])
{
    const F2 third = lbp::f2s(1.0f / 3.0f);
#pragma unroll 1
    for (int it = 0; it < 2; ++it) {
        F2 sm = lbp::f2s(0.0f), m[3], C[6], ep[3], em[3], x[19];
#pragma unroll
        for (int k = 0; k < 3; ++k) m[k] = lbp::f2s(0.0f);
#pragma unroll
        for (int k = 0; k < 6; ++k) C[k] = lbp::f2s(0.0f);
        exp_axes2(l, ep, em);
        exp_dirs2(ep, em, x);
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            const int cx = lbd::cx(i), cy = lbd::cy(i), cz = lbd::cz(i);
            const F2 w = x[i] * lbd::weight(i);
            sm = sm + w;
            if (cx) m[0] = cx > 0 ? m[0] + w : m[0] - w;
            if (cy) m[1] = cy > 0 ? m[1] + w : m[1] - w;
            if (cz) m[2] = cz > 0 ? m[2] + w : m[2] - w;
            if (cx) C[0] = C[0] + w;
            if (cy) C[1] = C[1] + w;
            if (cz) C[2] = C[2] + w;
            if (cx && cy) C[3] = cx * cy > 0 ? C[3] + w : C[3] - w;
            if (cy && cz) C[4] = cy * cz > 0 ? C[4] + w : C[4] - w;
            if (cz && cx) C[5] = cz * cx > 0 ? C[5] + w : C[5] - w;
        }
        const F2 iz = rcp2(lbp::f2s(1.0f) + sm);
#pragma unroll
        for (int d = 0; d < 3; ++d) m[d] = m[d] * iz;
        // covariance (1/3 I + sum a c c x) / Z - m m^T
        const F2 axx = (third + C[0]) * iz - m[0] * m[0], ayy = (third + C[1]) * iz - m[1] * m[1];
        const F2 azz = (third + C[2]) * iz - m[2] * m[2], axy = C[3] * iz - m[0] * m[1];
        const F2 ayz = C[4] * iz - m[1] * m[2], azx = C[5] * iz - m[2] * m[0];
        const F2 r[3] = {u[0] - m[0], u[1] - m[1], u[2] - m[2]};
        // Cramer's rule on the symmetric 3x3 system
        const F2 c00 = ayy * azz - ayz * ayz, c01 = azx * ayz - axy * azz, c02 = axy * ayz - azx * ayy;
        const F2 det = axx * c00 + axy * c01 + azx * c02;
        const F2 c11 = axx * azz - azx * azx, c12 = axy * azx - axx * ayz, c22 = axx * ayy - axy * axy;
        const F2 id = rcp2(det);
        l[0] = lbp::fma2(id, c00 * r[0] + c01 * r[1] + c02 * r[2], l[0]);
        l[1] = lbp::fma2(id, c01 * r[0] + c11 * r[1] + c12 * r[2], l[1]);
        l[2] = lbp::fma2(id, c02 * r[0] + c12 * r[1] + c22 * r[2], l[2]);
    }
}

// Up to this |u|^2 one step of Newton's method with the Jacobian of rest, 1/3,
// reaches FP32 rounding.  D3Q19's weights have no fourth cumulants, so 3u is
// off by O(u^5) only and the Jacobian by O(u^4): at |u| = 0.1 the start is
// 4.5e-5 of lambda off and the step leaves 1e-8 of it, 2e-10 in a population
// (evaluated in 64 bits over 4000 directions).
constexpr float kSlowFlow = 0.01f;

// Deviation moments meq of n^eq - a rho0 for both nodes.
__device__ __forceinline__ void exp_eq_moments2(F2 drho, F2 rho, F2 ux, F2 uy, F2 uz, F2 meq[19])
{
    const F2 three = lbp::f2s(3.0f);
    const F2 u[3] = {ux, uy, uz};
    F2 l[3] = {ux * three, uy * three, uz * three};
    F2 x[19], ep[3], em[3], sm, m[3];
    float q0, q1;
    lbp::split(ux * ux + uy * uy + uz * uz, q0, q1);
    if (fmaxf(q0, q1) < kSlowFlow) {
        exp_axes_small2(l, ep, em);
        exp_dirs2(ep, em, x);
        exp_sums2(x, sm, m);
        const F2 iz = rcp2(lbp::f2s(1.0f) + sm);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            // d lambda = 3 (u - <c>), below 2e-5: exp(+-d lambda) - 1 to second order
            const F2 dl = (u[d] - m[d] * iz) * three;
            const F2 h = dl * dl * 0.5f;
            const F2 p = h + dl, q = h - dl;
            ep[d] = lbp::fma2(ep[d], p, ep[d] + p);
            em[d] = lbp::fma2(em[d], q, em[d] + q);
        }
    } else {
        exp_newton2(u, l);
        exp_axes2(l, ep, em);
    }
    exp_dirs2(ep, em, x);
    exp_sums2(x, sm, m);
    const F2 g = rho * rcp2(lbp::f2s(1.0f) + sm);
    F2 d[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) d[i] = lbp::fma2(g, x[i] - sm, drho) * lbd::weight(i);
    lbp::forward2(d, meq);
}

// The collision of collide_moments2() with the moments of the exponential
// equilibrium in place of the quadratic ones (all non-conserved modes).
template <bool NOISE>
__device__ __forceinline__ void collide_exp2(const F2 m[19], F2 fx, F2 fy, F2 fz, const StepArgs &a, uint32_t node0,
                                             F2 out[19])
{
    const F2 half = lbp::f2s(0.5f), three = lbp::f2s(3.0f);
    const F2 rho = lbp::f2s(a.rho0) + m[0];
    const F2 inv_rho = rcp2(rho);
    const F2 ux = lbp::fma2(half, fx, m[1]) * inv_rho;
    const F2 uy = lbp::fma2(half, fy, m[2]) * inv_rho;
    const F2 uz = lbp::fma2(half, fz, m[3]) * inv_rho;
    F2 meq[19];
    exp_eq_moments2(m[0], rho, ux, uy, uz, meq);
    const F2 uf = ux * fx + uy * fy + uz * fz;
    const F2 gs1 = lbp::f2s(1.0f + a.g_shear), hgs1 = lbp::f2s(0.5f * (1.0f + a.g_shear));
    const F2 F[6] = {lbp::f2s(1.0f + a.g_bulk) * uf, gs1 * (ux * fx * three - uf), gs1 * (uy * fy - uz * fz),
                     hgs1 * (ux * fy + uy * fx),      hgs1 * (uy * fz + uz * fy),   hgs1 * (uz * fx + ux * fz)};
    F2 M[19];
    M[0] = m[0];
    M[1] = m[1] + fx;  // (backward2 multiplies by 1 / w = 3)
    M[2] = m[2] + fy;
    M[3] = m[3] + fz;
    M[4] = lbp::fma2(lbp::f2s(a.g_bulk), m[4] - meq[4], meq[4] + F[0]) * lbd::inv_w(4);
#pragma unroll
    for (int k = 5; k < 10; ++k) M[k] = lbp::fma2(lbp::f2s(a.g_shear), m[k] - meq[k], meq[k] + F[k - 4]) * lbd::inv_w(k);
#pragma unroll
    for (int k = 10; k < 16; ++k) M[k] = lbp::fma2(lbp::f2s(a.g_odd), m[k] - meq[k], meq[k]) * lbd::inv_w(k);
#pragma unroll
    for (int k = 16; k < 19; ++k) M[k] = lbp::fma2(lbp::f2s(a.g_even), m[k] - meq[k], meq[k]) * lbd::inv_w(k);
    if (NOISE) lbp::add_noise2(M, rho, a, lbp::ParamKeys{a.rk}, node0, a.step, a.replica);
    lbp::backward2(M, out);
}

// The pull and store of k_stream_collide_linear, the exponential collision.
// Bound by instruction issue: 128^3 with noise 70 us a step, against 129 us
// with two full Newton steps on every node and expm1f for each exponential
// (quadratic equilibrium: 52 us).
template <int DT, bool NOISE, bool WALLS, bool ODD>
__global__ void __launch_bounds__(kLinBX) k_stream_collide_exp2(const typename lbd::Store<DT>::T *src,
                                                                typename lbd::Store<DT>::T *dst, const float *ffield,
                                                                float *facc, const StepArgs a)
{
    PairAt at;
    const bool mine = locate_pair<WALLS>(a, at);
    wait_for_previous();
    if (!mine) return;
    F2 n[19], m[19], out[19];
    float f0[3], f1[3];
    load_linear<DT, true, WALLS, ODD>(src, ffield, facc, a, at, n, f0, f1);
    lbp::forward2(n, m);
    collide_exp2<NOISE>(m, lbp::f2(f0[0], f1[0]), lbp::f2(f0[1], f1[1]), lbp::f2(f0[2], f1[2]), a, at.s, out);
    if (ODD)
        store_pair_any<DT>(dst, a, at, out);
    else
        store_pair<DT>(dst, a, at.s, out);
}

template <int DT>
cudaError_t launch_exp_dt(const lb_handle *h, const void *src, void *dst, float *facc)
{
    using T = typename lbd::Store<DT>::T;
    StepArgs a = make_args(h);
    a.consume = facc && facc == h->facc;
    const T *s = static_cast<const T *>(src);
    T *d = static_cast<T *>(dst);
    const bool noise = a.kT > 0.0f, walls = h->p.walls != 0;
    const bool odd = !sc_paired(h) || !pair_aligned(src, 2 * sizeof(T)) || !pair_aligned(dst, 2 * sizeof(T)) ||
                     !pair_aligned(facc, 8);
#define LBI_EXP2(NZ, WL) (odd ? k_stream_collide_exp2<DT, NZ, WL, true> : k_stream_collide_exp2<DT, NZ, WL, false>)
    return launch_chained(noise ? (walls ? LBI_EXP2(true, true) : LBI_EXP2(true, false))
                                : (walls ? LBI_EXP2(false, true) : LBI_EXP2(false, false)),
                          linear_grid(a), kLinBX, h->stream, s, d, h->force, facc, a);
#undef LBI_EXP2
}

}  // namespace

// One stream-collide launch of a handle whose lb_params.equilibrium selects
// the exponential form.
cudaError_t launch_stream_collide_exp(const lb_handle *h, const void *src, void *dst, float *facc)
{
    switch (h->p.dtype) {
    case LB_F32: return launch_exp_dt<0>(h, src, dst, facc);
    case LB_F16: return launch_exp_dt<1>(h, src, dst, facc);
    default: return launch_exp_dt<2>(h, src, dst, facc);
    }
}

}  // namespace lbi
