// adjoint.cu -- reverse mode of the deterministic (kT = 0) stream-collide
// step, the kinetic-energy loss seed, and a checkpointed driver.
//
// One forward step maps the stored state S_t to S_{t+1} = C(pull(S_t), f).
// Its adjoint, derived here in moment space (Table 1 basis, q = a):
//   back transform  n* = B m*,  B = diag(a) E^T diag(1/w)
//                   -> mu*_k = (1/w_k) sum_i e_ki a_i lambda_i
//   relaxation      m*_0 = m_0, m*_a = m_a + f_a (a = 1..3),
//                   m*_k = (1 - g_k) rho P_k(u) + g_k m_k + F_k(u, f) (k = 4..9),
//                   m*_k = g_k m_k (k >= 10), with rho = rho0 + m_0,
//                   u = (m_1..3 + f/2) / rho   (Sec. 3.4 Eq. (lco_update),
//                   Sec. 3.7 Eqs. (special_choice_momentum_density),
//                   (moment_two_external_force))
//   forward         m = E n -> dL/dn_i = sum_k e_ki mu_k
//   pull            n_i(r) = S_i(r - c_i) (or S_opp(i)(r) at a wall)
//                   -> lambda_t is the push of dL/dn back to those entries;
//                   every fluid entry receives exactly one value, so the
//                   push is a plain store.
// P_k are the equilibrium stress polynomials (u^2, 3ux^2 - u^2, uy^2 - uz^2,
// ux uy, uy uz, uz ux) and F_k the force moments of Sigma.
#include <cmath>
#include <vector>

#include "stream_collide.cuh"

namespace lbi {

extern template cudaError_t launch_stream_collide_dt<0>(const lb_handle *, const void *, void *, float *, float *);
extern template cudaError_t launch_stream_collide_dt<1>(const lb_handle *, const void *, void *, float *, float *);
extern template cudaError_t launch_stream_collide_dt<2>(const lb_handle *, const void *, void *, float *, float *);

namespace {

constexpr int kAdjBX = 128;

template <bool WALLS>
__device__ __forceinline__ void neighbours(int x, int y, int z, const StepArgs &a, int &xm, int &xp, int &ym, int &yp,
                                           int &zm, int &zp)
{
    xm = (x == 0) ? a.nx - 1 : x - 1;
    xp = (x == a.nx - 1) ? 0 : x + 1;
    ym = (y == 0) ? a.ny - 1 : y - 1;
    yp = (y == a.ny - 1) ? 0 : y + 1;
    if (WALLS) {
        zm = z - 1;
        zp = z + 1;
    } else {
        zm = (z == 0) ? a.nz - 1 : z - 1;
        zp = (z == a.nz - 1) ? 0 : z + 1;
    }
}

// Source entry of the pull for direction i at node (x, y, z): returns the
// plane and the node index; at a wall the link bounces back to the node itself.
template <bool WALLS>
__device__ __forceinline__ void pull_source(int i, int x, int y, int z, int xm, int xp, int ym, int yp, int zm, int zp,
                                            const StepArgs &a, int &plane, uint32_t &node)
{
    const int sx = lbd::cx(i) == 1 ? xm : (lbd::cx(i) == -1 ? xp : x);
    const int sy = lbd::cy(i) == 1 ? ym : (lbd::cy(i) == -1 ? yp : y);
    const int sz = lbd::cz(i) == 1 ? zm : (lbd::cz(i) == -1 ? zp : z);
    const bool bounce = WALLS && lbd::cz(i) != 0 && (sz == 0 || sz == a.nz - 1);
    if (bounce) {
        plane = lbd::opposite(i);
        node = (uint32_t)((z * a.ny + y) * a.nx + x);
    } else {
        plane = i;
        node = (uint32_t)((sz * a.ny + sy) * a.nx + sx);
    }
}

// Store of the pushed pair dn to the entries the pair pulls from: nodes x0,
// x0 + 1 of one row (even nx), the mirror of load_pair.
template <bool WALLS>
__device__ __forceinline__ void push_pair(float *lam_out, const StepArgs &a, const PairAt &at, const lbp::F2 dn[19])
{
    const int xm = at.x == 0 ? a.nx - 1 : at.x - 1, xp = at.x + 2 == a.nx ? 0 : at.x + 2;
    const PullAt p = pull_at<WALLS>(a, at.x, at.y, at.z);
    const size_t P = a.pitch;
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        float v0, v1;
        lbp::split(dn[i], v0, v1);
        const bool bounce = WALLS && ((lbd::cz(i) == 1 && p.lo) || (lbd::cz(i) == -1 && p.hi));
        if (bounce || lbd::cx(i) == 0) {
            const size_t k = bounce ? (size_t)lbd::opposite(i) * P + at.s
                                    : (size_t)i * P + p.z[1 - lbd::cz(i)] + p.y[1 - lbd::cy(i)] + (uint32_t)at.x;
            if (in_bounds(k + 1, 19 * P, a.err)) Pair<0>::store(lam_out + k, v0, v1, 1.0f);
            continue;
        }
        const size_t row = (size_t)i * P + p.z[1 - lbd::cz(i)] + p.y[1 - lbd::cy(i)];
        const size_t k0 = row + (uint32_t)(lbd::cx(i) == 1 ? xm : at.x + 1);
        const size_t k1 = row + (uint32_t)(lbd::cx(i) == 1 ? at.x : xp);
        if (in_bounds(k0, 19 * P, a.err)) lam_out[k0] = v0;
        if (in_bounds(k1, 19 * P, a.err)) lam_out[k1] = v1;
    }
}

// The reverse of one step for two consecutive nodes per thread, in packed
// FP32 over the linear node index (the mapping and the addresses of
// k_stream_collide_linear).  Of the state only rho and u enter, so only the
// conserved moments of the pulled populations are formed.  With the quadratic
// forms P_k = u^T Q_k u (Q_4 = 1, Q_5 = diag(2, -1, -1), Q_6 = diag(0, 1, -1),
// Q_7..9 = 1/2 off the diagonal) and F_k = (1 + g_k) u^T Q_k f, the adjoint of
// the equilibrium and the forcing is that of T = sum_5..9 mu*_k Q_k and mu*_4:
// two matrix-vector products T u, T f instead of the rows of six Jacobians.
// Bound by memory (264 bytes a node); at 64^3, where part of it stays in the
// L2, about 12 us a step against 19 us with one node a thread in scalar arithmetic
// (802 instructions a node, half the threads of a 64-node row's block idle).
template <int DT, bool WALLS, bool ODD>
__global__ void __launch_bounds__(kLinBX)
    k_adjoint_step(const typename lbd::Store<DT>::T *state, const float *lam_in, float *lam_out, const float *ffield,
                   const float *impulse, float *grad_f, const StepArgs a)
{
    using lbp::F2;
    using lbp::f2s;
    using lbp::fma2;
    PairAt at;
    const bool mine = locate_pair<WALLS>(a, at);
    wait_for_previous();
    if (!mine) return;
    const size_t P = a.pitch;

    // rho and u of the forward step; al_i = a_i lambda_i
    F2 n[19], m[4], al[19];
    float f0[3], f1[3];
    load_linear<DT, true, WALLS, ODD>(state, ffield, const_cast<float *>(impulse), a, at, n, f0, f1);  // (only read)
#pragma unroll
    for (int i = 0; i < 19; ++i) {  // s is even, and s + 1 lies in the plane's padding at most
        const float *p = lam_in + (size_t)i * P + at.s;
        const float2 v = ODD ? make_float2(ld_f32(p), ld_f32(p + 1)) : ld_f32x2(p);
        al[i] = lbp::f2(v.x, v.y) * lbd::weight(i);
    }
    lbp::forward2_conserved(n, m);
    const F2 rho = f2s(a.rho0) + m[0];
    float rl, rh;
    lbp::split(rho, rl, rh);
    const F2 ir = lbp::f2(__frcp_rn(rl), __frcp_rn(rh));
    F2 f[3], u[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        f[d] = lbp::f2(f0[d], f1[d]);
        u[d] = fma2(f2s(0.5f), f[d], m[1 + d]) * ir;
    }

    // adjoint of the back transform
    F2 mu[19];
    lbp::forward2(al, mu);
#pragma unroll
    for (int k = 1; k < 19; ++k) mu[k] = mu[k] * lbd::inv_w(k);

    // adjoint of the relaxation, the equilibrium and the force moments
    const F2 txx = mu[5] + mu[5], tyy = mu[6] - mu[5], tzz = f2s(0.0f) - mu[5] - mu[6];
    const F2 txy = mu[7] * 0.5f, tyz = mu[8] * 0.5f, tzx = mu[9] * 0.5f;
    const F2 Tu[3] = {fma2(txx, u[0], fma2(txy, u[1], tzx * u[2])), fma2(txy, u[0], fma2(tyy, u[1], tyz * u[2])),
                      fma2(tzx, u[0], fma2(tyz, u[1], tzz * u[2]))};
    const F2 Tf[3] = {fma2(txx, f[0], fma2(txy, f[1], tzx * f[2])), fma2(txy, f[0], fma2(tyy, f[1], tyz * f[2])),
                      fma2(tzx, f[0], fma2(tyz, f[1], tzz * f[2]))};
    const F2 a4 = mu[4] * (1.0f - a.g_bulk), b4 = mu[4] * (1.0f + a.g_bulk);
    F2 rbar = f2s(0.0f), udot = f2s(0.0f), ubar[3], fbar[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const F2 Au = fma2(a4, u[d], Tu[d] * (1.0f - a.g_shear));
        const F2 Bu = fma2(b4, u[d], Tu[d] * (1.0f + a.g_shear));
        const F2 Bf = fma2(b4, f[d], Tf[d] * (1.0f + a.g_shear));
        rbar = fma2(u[d], Au, rbar);
        ubar[d] = fma2(rho, Au + Au, Bf);
        udot = fma2(ubar[d], u[d], udot);
        fbar[d] = mu[1 + d] + Bu;
    }
    mu[0] = mu[0] + rbar - udot * ir;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const F2 w = ubar[d] * ir;
        mu[1 + d] = mu[1 + d] + w;
        fbar[d] = fma2(w, 0.5f, fbar[d]);
    }
    mu[4] = mu[4] * a.g_bulk;
#pragma unroll
    for (int k = 5; k < 10; ++k) mu[k] = mu[k] * a.g_shear;
#pragma unroll
    for (int k = 10; k < 16; ++k) mu[k] = mu[k] * a.g_odd;
#pragma unroll
    for (int k = 16; k < 19; ++k) mu[k] = mu[k] * a.g_even;

    // dL/dn_i = sum_k e_ki mu_k, pushed to the pull sources
    F2 dn[19];
    lbp::backward2<false>(mu, dn);
    if (ODD) {
        int xb, yb, zb;
        second_node(a, at, xb, yb, zb);
        const PullAt pa = pull_at<WALLS>(a, at.x, at.y, at.z), pb = pull_at<WALLS>(a, xb, yb, zb);
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            float v0, v1;
            lbp::split(dn[i], v0, v1);
            const size_t ka = pull_index<WALLS>(a, pa, i), kb = pull_index<WALLS>(a, pb, i);
            if (at.va && in_bounds(ka, 19 * P, a.err)) lam_out[ka] = v0;
            if (at.vb && in_bounds(kb, 19 * P, a.err)) lam_out[kb] = v1;
        }
    } else {
        push_pair<WALLS>(lam_out, a, at, dn);
    }
    if (grad_f) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {  // component stride N: no 8-byte alignment in general
            float v0, v1;
            lbp::split(fbar[d], v0, v1);
            float *g = grad_f + d * a.nn + at.s;
            if (at.va) g[0] += v0;
            if (at.vb) g[1] += v1;
        }
    }
}

// lambda_T for L = 1/2 sum_{box} |j|^2 / rho: dL/dn_i = u.c_i - u^2/2 inside
// the box, 0 elsewhere (every fluid entry is written); dL/df += u/2.
template <int DT, bool WALLS>
__global__ void __launch_bounds__(kAdjBX)
    k_adjoint_seed(const typename lbd::Store<DT>::T *__restrict__ state, float *__restrict__ lam_out,
                   const float *__restrict__ ffield, float *grad_f, double *loss, int3 lo, int3 hi, const StepArgs a)
{
    using S = lbd::Store<DT>;
    const int x = blockIdx.x * kAdjBX + threadIdx.x;
    const int y = blockIdx.y;
    const int z = blockIdx.z + a.z0;
    float Lloc = 0.0f;
    if (x < a.nx) {
        int xm, xp, ym, yp, zm, zp;
        neighbours<WALLS>(x, y, z, a, xm, xp, ym, yp, zm, zp);
        const size_t P = a.pitch;
        const uint32_t self = (uint32_t)((z * a.ny + y) * a.nx + x);
        const bool inside = x >= lo.x && x < hi.x && y >= lo.y && y < hi.y && z >= lo.z && z < hi.z;
        float n[19];
        int plane[19];
        uint32_t src[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            pull_source<WALLS>(i, x, y, z, xm, xp, ym, yp, zm, zp, a, plane[i], src[i]);
            n[i] = inside ? S::load(state + (size_t)plane[i] * P + src[i], a.inv_scale) : 0.0f;
        }
        float dn[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) dn[i] = 0.0f;
        if (inside) {
            float m[19];
            lbd::forward(n, m);
            float f[3] = {a.fx, a.fy, a.fz};
            if (ffield) {
                f[0] += ffield[self];
                f[1] += ffield[a.nn + self];
                f[2] += ffield[2 * a.nn + self];
            }
            const float rho = a.rho0 + m[0];
            const float j[3] = {m[1] + 0.5f * f[0], m[2] + 0.5f * f[1], m[3] + 0.5f * f[2]};
            const float u[3] = {j[0] / rho, j[1] / rho, j[2] / rho};
            const float u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
            Lloc = 0.5f * (j[0] * j[0] + j[1] * j[1] + j[2] * j[2]) / rho;
#pragma unroll
            for (int i = 0; i < 19; ++i) dn[i] = u[0] * lbd::cx(i) + u[1] * lbd::cy(i) + u[2] * lbd::cz(i) - 0.5f * u2;
            if (grad_f) {
                grad_f[self] += 0.5f * u[0];
                grad_f[a.nn + self] += 0.5f * u[1];
                grad_f[2 * a.nn + self] += 0.5f * u[2];
            }
        }
#pragma unroll
        for (int i = 0; i < 19; ++i) lam_out[(size_t)plane[i] * P + src[i]] = dn[i];
    }
    // loss: warp reduction, one double atomic per warp
    double v = (double)Lloc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(loss, v);
}

template <int DT>
cudaError_t launch_adjoint_dt(const lb_handle *h, const void *state, const float *lam_in, float *lam_out,
                              float *grad_f, const float *impulse)
{
    using T = typename lbd::Store<DT>::T;
    const StepArgs a = make_args(h);
    const T *s = static_cast<const T *>(state);
    const bool odd = !sc_paired(h) || !pair_aligned(state, 2 * sizeof(T)) || !pair_aligned(lam_in, 8) ||
                     !pair_aligned(lam_out, 8) || !pair_aligned(impulse, 8);
    return launch_chained(h->p.walls ? (odd ? k_adjoint_step<DT, true, true> : k_adjoint_step<DT, true, false>)
                                     : (odd ? k_adjoint_step<DT, false, true> : k_adjoint_step<DT, false, false>),
                          linear_grid(a), kLinBX, h->stream, s, lam_in, lam_out, h->force, impulse, grad_f, a);
}

// dL/du at the nodes (lam_u, [3][pitch], set by the coupling reverse pass)
// into dL/dstate through u = (sum n c + f/2) / rho of the pulled populations:
// d u_d / d n_i = (c_id - u_d) / rho, added at the stored entry each n_i is
// pulled from; d u_d / d f_d = 1 / (2 rho) into grad_f ([3][N]).  lam_u is
// zeroed on the way, so it is clean for the next call.
template <int DT, bool WALLS>
__global__ void __launch_bounds__(kAdjBX)
    k_lambda_u_to_pops(const typename lbd::Store<DT>::T *__restrict__ state, float *lam_u, float *lam_out,
                       const float *__restrict__ ffield, const float *__restrict__ impulse, float *grad_f,
                       const StepArgs a)
{
    using S = lbd::Store<DT>;
    const int x = blockIdx.x * kAdjBX + threadIdx.x;
    if (x >= a.nx) return;
    const int y = blockIdx.y;
    const int z = blockIdx.z + a.z0;
    const size_t P = a.pitch;
    const uint32_t self = (uint32_t)((z * a.ny + y) * a.nx + x);
    const float lu[3] = {lam_u[self], lam_u[P + self], lam_u[2 * P + self]};
    if (lu[0] == 0.0f && lu[1] == 0.0f && lu[2] == 0.0f) return;
    lam_u[self] = lam_u[P + self] = lam_u[2 * P + self] = 0.0f;
    int xm, xp, ym, yp, zm, zp;
    neighbours<WALLS>(x, y, z, a, xm, xp, ym, yp, zm, zp);
    float n[19];
    int plane[19];
    uint32_t src[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        pull_source<WALLS>(i, x, y, z, xm, xp, ym, yp, zm, zp, a, plane[i], src[i]);
        n[i] = S::load(state + (size_t)plane[i] * P + src[i], a.inv_scale);
    }
    float m[19];
    lbd::forward(n, m);
    // the velocity the forward coupling interpolated: f = body force + field
    // (the particle impulses of the step are not part of it)
    float f[3] = {a.fx, a.fy, a.fz};
    if (ffield) {
        f[0] += ffield[self];
        f[1] += ffield[a.nn + self];
        f[2] += ffield[2 * a.nn + self];
    }
    (void)impulse;
    const float rho = a.rho0 + m[0];
    const float ir = 1.0f / rho;
    const float u[3] = {(m[1] + 0.5f * f[0]) * ir, (m[2] + 0.5f * f[1]) * ir, (m[3] + 0.5f * f[2]) * ir};
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        const float v = lu[0] * ((float)lbd::cx(i) - u[0]) + lu[1] * ((float)lbd::cy(i) - u[1]) +
                        lu[2] * ((float)lbd::cz(i) - u[2]);
        atomicAdd(lam_out + (size_t)plane[i] * P + src[i], v * ir);
    }
    if (grad_f) {
#pragma unroll
        for (int d = 0; d < 3; ++d) grad_f[d * a.nn + self] += 0.5f * lu[d] * ir;
    }
}

template <int DT>
cudaError_t launch_lambda_u_dt(const lb_handle *h, const void *state, float *lam_u, float *lam_out, float *grad_f)
{
    using T = typename lbd::Store<DT>::T;
    const StepArgs a = make_args(h);
    dim3 grid((a.nx + kAdjBX - 1) / kAdjBX, a.ny, a.z1 - a.z0);
    const T *s = static_cast<const T *>(state);
    if (h->p.walls)
        k_lambda_u_to_pops<DT, true><<<grid, kAdjBX, 0, h->stream>>>(s, lam_u, lam_out, h->force, nullptr, grad_f, a);
    else
        k_lambda_u_to_pops<DT, false><<<grid, kAdjBX, 0, h->stream>>>(s, lam_u, lam_out, h->force, nullptr, grad_f, a);
    return cudaGetLastError();
}

template <int DT>
cudaError_t launch_seed_dt(const lb_handle *h, const void *state, float *lam_out, float *grad_f, double *loss,
                           int3 lo, int3 hi)
{
    using T = typename lbd::Store<DT>::T;
    const StepArgs a = make_args(h);
    dim3 grid((a.nx + kAdjBX - 1) / kAdjBX, a.ny, a.z1 - a.z0);
    const T *s = static_cast<const T *>(state);
    if (h->p.walls)
        k_adjoint_seed<DT, true><<<grid, kAdjBX, 0, h->stream>>>(s, lam_out, h->force, grad_f, loss, lo, hi, a);
    else
        k_adjoint_seed<DT, false><<<grid, kAdjBX, 0, h->stream>>>(s, lam_out, h->force, grad_f, loss, lo, hi, a);
    return cudaGetLastError();
}

cudaError_t launch_adjoint(const lb_handle *h, const void *state, const float *lam_in, float *lam_out, float *grad_f,
                           const float *impulse = nullptr)
{
    switch (h->p.dtype) {
    case LB_F32: return launch_adjoint_dt<0>(h, state, lam_in, lam_out, grad_f, impulse);
    case LB_F16: return launch_adjoint_dt<1>(h, state, lam_in, lam_out, grad_f, impulse);
    default: return launch_adjoint_dt<2>(h, state, lam_in, lam_out, grad_f, impulse);
    }
}

cudaError_t launch_lambda_u(const lb_handle *h, const void *state, float *lam_u, float *lam_out, float *grad_f)
{
    switch (h->p.dtype) {
    case LB_F32: return launch_lambda_u_dt<0>(h, state, lam_u, lam_out, grad_f);
    case LB_F16: return launch_lambda_u_dt<1>(h, state, lam_u, lam_out, grad_f);
    default: return launch_lambda_u_dt<2>(h, state, lam_u, lam_out, grad_f);
    }
}

// a += b over n floats
__global__ void k_axpy1(float *a, const float *b, size_t n)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        a[i] += b[i];
}

cudaError_t launch_seed(const lb_handle *h, const void *state, float *lam_out, float *grad_f, double *loss, int3 lo,
                        int3 hi)
{
    switch (h->p.dtype) {
    case LB_F32: return launch_seed_dt<0>(h, state, lam_out, grad_f, loss, lo, hi);
    case LB_F16: return launch_seed_dt<1>(h, state, lam_out, grad_f, loss, lo, hi);
    default: return launch_seed_dt<2>(h, state, lam_out, grad_f, loss, lo, hi);
    }
}

cudaError_t step_from(lb_handle *h, const void *src, void *dst, uint32_t step, float *impulse = nullptr)
{
    const uint32_t saved = h->step;
    h->step = step;
    cudaError_t e;
    switch (h->p.dtype) {
    case LB_F32:
        e = h->p.equilibrium ? launch_stream_collide_exp(h, src, dst, impulse)
                             : launch_stream_collide_dt<0>(h, src, dst, impulse, nullptr);
        break;
    case LB_F16:
        e = h->p.equilibrium ? launch_stream_collide_exp(h, src, dst, impulse)
                             : launch_stream_collide_dt<1>(h, src, dst, impulse, nullptr);
        break;
    default:
        e = h->p.equilibrium ? launch_stream_collide_exp(h, src, dst, impulse)
                             : launch_stream_collide_dt<2>(h, src, dst, impulse, nullptr);
        break;
    }
    h->step = saved;
    return e;
}

bool check_adjoint_handle(const lb_handle *h, const char *who)
{
    if (!h) {
        set_error("%s: handle is NULL", who);
        return false;
    }
    if (h->p.kT != 0.0) {
        set_error("%s: the adjoint is defined for deterministic runs (kT = 0)", who);
        return false;
    }
    if (h->p.equilibrium) {
        set_error("%s: the adjoint is derived for the quadratic equilibrium", who);
        return false;
    }
    return true;
}

bool box_ok(const lb_handle *h, const int lo[3], const int hi[3])
{
    const int L[3] = {h->p.nx, h->p.ny, h->p.nz};
    for (int d = 0; d < 3; ++d)
        if (lo[d] < 0 || hi[d] > L[d] || lo[d] > hi[d]) return false;
    return true;
}

// Carve `count` blocks of `bytes` each (256-byte aligned) from the handle's
// arena, growing it first if needed (the only allocation of the reverse-mode
// drivers; a grown arena replaces the old one, whose contents are dropped).
struct Carver {
    size_t need = 0;
    std::vector<std::pair<void **, size_t>> req;
    void add(void **p, size_t bytes)
    {
        req.push_back({p, need});
        need += (bytes + 255) & ~(size_t)255;
    }
    cudaError_t place(lb_handle *h)
    {
        if (h->arena_bytes < need) {
            cudaError_t e = cudaStreamSynchronize(h->stream);  // the old arena may still be in use
            if (e != cudaSuccess) return e;
            cudaFree(h->arena);
            h->arena = nullptr;
            h->arena_bytes = 0;
            e = cudaMalloc((void **)&h->arena, need);
            if (e != cudaSuccess) {
                h->arena = nullptr;
                return e;
            }
            h->arena_bytes = need;
        }
        for (auto &r : req) *r.first = h->arena + r.second;
        return cudaSuccess;
    }
};

}  // namespace
}  // namespace lbi

using namespace lbi;

extern "C" {

lb_status lb_step_from(lb_handle *h, const void *src, void *dst, uint32_t step)
{
    if (!h || !src || !dst || src == dst) {
        set_error("lb_step_from: need a handle and two distinct buffers");
        return LB_EINVAL;
    }
    join_overlap(h);
    cudaError_t e = step_from(h, src, dst, step);
    h->launches += 1;
    return e == cudaSuccess ? LB_OK : cuda_fail("lb_step_from", e);
}

lb_status lb_adjoint_step(lb_handle *h, const void *state, const float *lambda_in, float *lambda_out,
                          float *grad_force)
{
    if (!check_adjoint_handle(h, "lb_adjoint_step")) return h ? LB_EUNSUPPORTED : LB_EINVAL;
    if (!state || !lambda_in || !lambda_out || lambda_in == lambda_out) {
        set_error("lb_adjoint_step: need a state and two distinct adjoint buffers");
        return LB_EINVAL;
    }
    join_overlap(h);
    cudaError_t e = launch_adjoint(h, state, lambda_in, lambda_out, grad_force);
    h->launches += 1;
    return e == cudaSuccess ? LB_OK : cuda_fail("lb_adjoint_step", e);
}

lb_status lb_adjoint_seed_kinetic(lb_handle *h, const void *state, const int lo[3], const int hi[3], float *lambda_out,
                                  float *grad_force, double *loss)
{
    if (!h || !state || !lo || !hi || !lambda_out || !loss) {
        set_error("lb_adjoint_seed_kinetic: NULL argument");
        return LB_EINVAL;
    }
    join_overlap(h);
    if (!box_ok(h, lo, hi)) {
        set_error("lb_adjoint_seed_kinetic: sub-box outside the lattice");
        return LB_EINVAL;
    }
    cudaError_t e = cudaMemsetAsync(loss, 0, sizeof(double), h->stream);
    if (e == cudaSuccess)
        e = launch_seed(h, state, lambda_out, grad_force, loss, make_int3(lo[0], lo[1], lo[2]),
                        make_int3(hi[0], hi[1], hi[2]));
    h->launches += 1;
    return e == cudaSuccess ? LB_OK : cuda_fail("lb_adjoint_seed_kinetic", e);
}

// Arena layout of the uncoupled reverse pass: nseg checkpoints, K - 1
// segment states, two adjoint buffers.
struct KineticBuffers {
    std::vector<void *> ckpt, seg;
    float *lam[2] = {nullptr, nullptr};
    float *gseed = nullptr;  // dL/df of the loss itself (j = sum n c + f/2), [3][N]
};

static cudaError_t kinetic_buffers(lb_handle *h, int nsteps, int K, KineticBuffers &b)
{
    const int nseg = (nsteps + K - 1) / K;
    const size_t pop_bytes = 19 * h->pitch * h->elem;
    const size_t lam_bytes = 19 * h->pitch * sizeof(float);
    b.ckpt.assign(nseg, nullptr);
    b.seg.assign(K, nullptr);
    Carver c;
    for (int s = 0; s < nseg; ++s) c.add(&b.ckpt[s], pop_bytes);
    for (int k = 1; k < K; ++k) c.add(&b.seg[k], pop_bytes);
    for (int q = 0; q < 2; ++q) c.add((void **)&b.lam[q], lam_bytes);
    c.add((void **)&b.gseed, 3 * h->n_nodes * sizeof(float));
    return c.place(h);
}

lb_status lb_adjoint_forward(lb_handle *h, int nsteps, int checkpoint_every, const int lo[3], const int hi[3],
                             double *loss)
{
    const NvtxRange range("lb_adjoint_forward");
    if (!check_adjoint_handle(h, "lb_adjoint_forward")) return h ? LB_EUNSUPPORTED : LB_EINVAL;
    if (nsteps < 1 || checkpoint_every < 1 || !lo || !hi || !loss || !box_ok(h, lo, hi)) {
        set_error("lb_adjoint_forward: need nsteps >= 1, checkpoint_every >= 1, a valid sub-box and a loss");
        return LB_EINVAL;
    }
    join_overlap(h);
    if (h->facc_dirty) {
        set_error("lb_adjoint_forward: pending particle impulses are not differentiated");
        return LB_EUNSUPPORTED;
    }
    const int K = std::min(checkpoint_every, nsteps);
    KineticBuffers b;
    cudaError_t e = kinetic_buffers(h, nsteps, K, b);
    if (e != cudaSuccess) {
        set_error("lb_adjoint_forward: checkpoint allocation failed (%s)", cudaGetErrorString(e));
        return LB_ENOMEM;
    }
    h->adj_ready = 0;
    const uint32_t step0 = h->step;
    // Each step writes its result where it is needed: a checkpoint at the end
    // of a segment, the segment states themselves in the last segment (the
    // reverse pass then has nothing to recompute there), the handle's buffers
    // otherwise and at the end: the one lb_step would have ended in, so that a
    // captured call with an even number of steps can be replayed on its result.
    const int last0 = (nsteps - 1) / K * K;  // first step of the last segment
    void *const end = h->pops[(h->cur + nsteps) & 1];
    void *src = h->pops[h->cur];
    e = cudaMemcpyAsync(b.ckpt[0], src, 19 * h->pitch * h->elem, cudaMemcpyDeviceToDevice, h->stream);
    for (int t = 0; t < nsteps && e == cudaSuccess; ++t) {
        const int other = src == h->pops[0] ? 1 : 0;
        void *dst = h->pops[other];
        if (t + 1 < nsteps && (t + 1) % K == 0) dst = b.ckpt[(t + 1) / K];
        else if (t + 1 < nsteps && t >= last0) dst = b.seg[t + 1 - last0];
        else if (t + 1 == nsteps) dst = end;  // (src is a checkpoint or a segment state, or nsteps is 1)
        timer_mark(h, 0, 0, h->stream);
        e = step_from(h, src, dst, step0 + (uint32_t)t);
        timer_mark(h, 0, 1, h->stream);
        h->launches += 1;
        src = dst;
    }
    if (e != cudaSuccess) return cuda_fail("lb_adjoint_forward", e);
    h->cur = (h->cur + nsteps) & 1;
    h->step = step0 + (uint32_t)nsteps;
    // the loss and its seed lambda_T = dL/dstate at the final state (first
    // adjoint buffer) with its own dL/df (gseed), for lb_adjoint_backward.
    // The adjoint buffers are not cleared: every fluid entry is written before
    // it is read, and the others only reach results that are not stored.
    e = cudaMemsetAsync(loss, 0, sizeof(double), h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(b.gseed, 0, 3 * h->n_nodes * sizeof(float), h->stream);
    if (e == cudaSuccess)
        e = launch_seed(h, h->pops[h->cur], b.lam[0], b.gseed, loss, make_int3(lo[0], lo[1], lo[2]),
                        make_int3(hi[0], hi[1], hi[2]));
    h->launches += 1;
    if (e != cudaSuccess) return cuda_fail("lb_adjoint_forward", e);
    h->adj_ready = 1;
    h->adj_nsteps = nsteps;
    h->adj_K = K;
    h->adj_step0 = step0;
    return LB_OK;
}

lb_status lb_adjoint_backward(lb_handle *h, float *grad_force)
{
    const NvtxRange range("lb_adjoint_backward");
    if (!check_adjoint_handle(h, "lb_adjoint_backward")) return h ? LB_EUNSUPPORTED : LB_EINVAL;
    if (!grad_force) {
        set_error("lb_adjoint_backward: grad_force is NULL");
        return LB_EINVAL;
    }
    join_overlap(h);
    if (!h->adj_ready) {
        set_error("lb_adjoint_backward: no lb_adjoint_forward run to reverse");
        return LB_EINVAL;
    }
    const int nsteps = h->adj_nsteps, K = h->adj_K;
    const int nseg = (nsteps + K - 1) / K;
    KineticBuffers b;
    cudaError_t e = kinetic_buffers(h, nsteps, K, b);  // the forward's layout: no allocation
    if (e != cudaSuccess) return cuda_fail("lb_adjoint_backward", e);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(grad_force, b.gseed, 3 * h->n_nodes * sizeof(float), cudaMemcpyDeviceToDevice,
                            h->stream);
    int cur = 0;
    for (int s = nseg - 1; s >= 0 && e == cudaSuccess; --s) {
        const int t0 = s * K, t1 = std::min(nsteps, t0 + K);
        b.seg[0] = b.ckpt[s];
        for (int t = t0; s < nseg - 1 && t < t1 - 1 && e == cudaSuccess; ++t) {
            e = step_from(h, b.seg[t - t0], b.seg[t - t0 + 1], h->adj_step0 + (uint32_t)t);
            h->launches += 1;
        }
        for (int t = t1 - 1; t >= t0 && e == cudaSuccess; --t) {
            e = launch_adjoint(h, b.seg[t - t0], b.lam[cur], b.lam[1 - cur], grad_force);
            h->launches += 1;
            cur = 1 - cur;
        }
    }
    h->adj_ready = 0;  // the adjoint buffers were consumed
    return e == cudaSuccess ? LB_OK : cuda_fail("lb_adjoint_backward", e);
}

lb_status lb_adjoint_kinetic(lb_handle *h, int nsteps, int checkpoint_every, const int lo[3], const int hi[3],
                             float *grad_force, double *loss)
{
    if (!grad_force) {
        set_error("lb_adjoint_kinetic: grad_force is NULL");
        return LB_EINVAL;
    }
    lb_status st = lb_adjoint_forward(h, nsteps, checkpoint_every, lo, hi, loss);
    if (st != LB_OK) return st;
    return lb_adjoint_backward(h, grad_force);
}


lb_status lb_adjoint_step_impulse(lb_handle *h, const void *state, const float *impulse, const float *lambda_in,
                                  float *lambda_out, float *grad_force)
{
    if (!check_adjoint_handle(h, "lb_adjoint_step_impulse")) return h ? LB_EUNSUPPORTED : LB_EINVAL;
    if (!state || !lambda_in || !lambda_out || lambda_in == lambda_out) {
        set_error("lb_adjoint_step_impulse: need a state and two distinct adjoint buffers");
        return LB_EINVAL;
    }
    join_overlap(h);
    cudaError_t e = launch_adjoint(h, state, lambda_in, lambda_out, grad_force, impulse);
    h->launches += 1;
    return e == cudaSuccess ? LB_OK : cuda_fail("lb_adjoint_step_impulse", e);
}

lb_status lb_adjoint_couple(lb_handle *h, const void *state, const lb_particles *start, const lb_couple_params *cp,
                            const float *lambda_facc, float *lambda_pos, float *lambda_mom, float *lambda_pops,
                            float *grad_force)
{
    if (!check_adjoint_handle(h, "lb_adjoint_couple")) return h ? LB_EUNSUPPORTED : LB_EINVAL;
    if (!state || !start || !cp || !lambda_facc || !lambda_pops ||
        (start->n > 0 && (!lambda_pos || !lambda_mom))) {
        set_error("lb_adjoint_couple: NULL argument");
        return LB_EINVAL;
    }
    join_overlap(h);
    if (!h->lam_u) {
        cudaError_t e = cudaMalloc((void **)&h->lam_u, 3 * h->pitch * sizeof(float));
        if (e == cudaSuccess) e = cudaMemsetAsync(h->lam_u, 0, 3 * h->pitch * sizeof(float), h->stream);
        if (e != cudaSuccess) {
            set_error("lb_adjoint_couple: scratch allocation failed (%s)", cudaGetErrorString(e));
            return LB_ENOMEM;
        }
    }
    lb_status st = couple_adjoint(h, state, start, cp, lambda_facc, lambda_pos, lambda_mom, h->lam_u);
    if (st != LB_OK || start->n == 0) return st;
    cudaError_t e = launch_lambda_u(h, state, h->lam_u, lambda_pops, grad_force);
    h->launches += 1;
    return e == cudaSuccess ? LB_OK : cuda_fail("lb_adjoint_couple", e);
}

lb_status lb_adjoint_kinetic_coupled(lb_handle *h, const lb_particles *parts, const lb_couple_params *cp, int nsteps,
                                     int checkpoint_every, const int lo[3], const int hi[3], float *grad_force,
                                     float *grad_pos, float *grad_mom, double *loss)
{
    const NvtxRange range("lb_adjoint_kinetic_coupled");
    if (!check_adjoint_handle(h, "lb_adjoint_kinetic_coupled")) return h ? LB_EUNSUPPORTED : LB_EINVAL;
    if (!parts || !cp || nsteps < 1 || checkpoint_every < 1 || !lo || !hi || !grad_force || !loss ||
        !box_ok(h, lo, hi) || (parts->n > 0 && (!grad_pos || !grad_mom))) {
        set_error("lb_adjoint_kinetic_coupled: need particles, nsteps >= 1, checkpoint_every >= 1, a valid "
                  "sub-box and outputs");
        return LB_EINVAL;
    }
    if (!adjoint_couple_ok(h, parts, cp, "lb_adjoint_kinetic_coupled")) return LB_EUNSUPPORTED;
    join_overlap(h);
    if (h->facc_dirty) {
        set_error("lb_adjoint_kinetic_coupled: pending particle impulses (call lb_step first)");
        return LB_EUNSUPPORTED;
    }
    lb_couple_params c1 = *cp;
    c1.flags &= ~LB_COUPLE_OVERLAP;
    const int n = parts->n;
    const int K = std::min(checkpoint_every, nsteps);
    const int nseg = (nsteps + K - 1) / K;
    const size_t pop_bytes = 19 * h->pitch * h->elem;
    const size_t lam_bytes = 19 * h->pitch * sizeof(float);
    const size_t facc_bytes = 3 * h->pitch * sizeof(float);
    const size_t grad_bytes = 3 * h->n_nodes * sizeof(float);
    const size_t pos_bytes = (size_t)n * 3 * sizeof(double), mom_bytes = (size_t)n * 3 * sizeof(float);
    std::vector<void *> ckpt(nseg, nullptr), seg(K, nullptr);
    std::vector<double *> cpos(nseg, nullptr), spos(K + 1, nullptr);  // particles before step k of a segment
    std::vector<float *> cmom(nseg, nullptr), smom(K + 1, nullptr), sfacc(K, nullptr);
    float *lam[2] = {nullptr, nullptr};
    float *gstep = nullptr;
    cudaError_t e = cudaSuccess;
    {
        // all temporaries from the handle's arena (allocated once, reused)
        Carver c;
        for (int s = 0; s < nseg; ++s) {
            c.add(&ckpt[s], pop_bytes);
            if (n) c.add((void **)&cpos[s], pos_bytes);
            if (n) c.add((void **)&cmom[s], mom_bytes);
        }
        for (int k = 0; k <= K; ++k) {
            if (k > 0 && k < K) c.add(&seg[k], pop_bytes);
            if (n) c.add((void **)&spos[k], pos_bytes);
            if (n) c.add((void **)&smom[k], mom_bytes);
            if (k < K) c.add((void **)&sfacc[k], facc_bytes);
        }
        for (int b = 0; b < 2; ++b) c.add((void **)&lam[b], lam_bytes);
        c.add((void **)&gstep, grad_bytes);
        e = c.place(h);
    }
    h->adj_ready = 0;  // the arena now holds this call's buffers
    if (e != cudaSuccess) {
        set_error("lb_adjoint_kinetic_coupled: checkpoint allocation failed (%s)", cudaGetErrorString(e));
        return LB_ENOMEM;
    }
    const uint32_t step0 = h->step;
    // forward pass: populations and particle state checkpointed every K steps
    for (int t = 0; t < nsteps && e == cudaSuccess; ++t) {
        if (t % K == 0) {
            e = cudaMemcpyAsync(ckpt[t / K], h->pops[h->cur], pop_bytes, cudaMemcpyDeviceToDevice, h->stream);
            if (e == cudaSuccess && n)
                e = cudaMemcpyAsync(cpos[t / K], parts->pos, pos_bytes, cudaMemcpyDeviceToDevice, h->stream);
            if (e == cudaSuccess && n)
                e = cudaMemcpyAsync(cmom[t / K], parts->mom, mom_bytes, cudaMemcpyDeviceToDevice, h->stream);
        }
        lb_status st = (e == cudaSuccess) ? couple_particles(h, parts, &c1) : LB_ECUDA;
        if (st == LB_OK) st = lb_step(h, 1);
        if (st != LB_OK) {
            return st;
        }
    }
    int cur = 0;
    if (e == cudaSuccess) e = cudaMemsetAsync(lam[0], 0, lam_bytes, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(lam[1], 0, lam_bytes, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(grad_force, 0, grad_bytes, h->stream);
    if (e == cudaSuccess && n) e = cudaMemsetAsync(grad_pos, 0, (size_t)n * 3 * sizeof(float), h->stream);
    if (e == cudaSuccess && n) e = cudaMemsetAsync(grad_mom, 0, (size_t)n * 3 * sizeof(float), h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(loss, 0, sizeof(double), h->stream);
    if (e == cudaSuccess)
        e = launch_seed(h, h->pops[h->cur], lam[cur], grad_force, loss, make_int3(lo[0], lo[1], lo[2]),
                        make_int3(hi[0], hi[1], hi[2]));
    h->launches += 1;
    for (int sgi = nseg - 1; sgi >= 0 && e == cudaSuccess; --sgi) {
        const int t0 = sgi * K, t1 = std::min(nsteps, t0 + K);
        seg[0] = ckpt[sgi];
        // recompute the segment: populations, the particle state before each
        // step and each step's impulses
        if (n) e = cudaMemcpyAsync(spos[0], cpos[sgi], pos_bytes, cudaMemcpyDeviceToDevice, h->stream);
        if (e == cudaSuccess && n) e = cudaMemcpyAsync(smom[0], cmom[sgi], mom_bytes, cudaMemcpyDeviceToDevice, h->stream);
        for (int t = t0; t < t1 && e == cudaSuccess; ++t) {
            const int k = t - t0;
            if (n) {  // the coupling updates in place: run it on a copy in slot k + 1
                e = cudaMemcpyAsync(spos[k + 1], spos[k], pos_bytes, cudaMemcpyDeviceToDevice, h->stream);
                if (e == cudaSuccess)
                    e = cudaMemcpyAsync(smom[k + 1], smom[k], mom_bytes, cudaMemcpyDeviceToDevice, h->stream);
                lb_particles pk = *parts;
                pk.pos = spos[k + 1];
                pk.mom = smom[k + 1];
                if (e == cudaSuccess && couple_on(h, seg[k], &pk, &c1, sfacc[k]) != LB_OK) e = cudaErrorLaunchFailure;
            } else {
                e = cudaMemsetAsync(sfacc[k], 0, facc_bytes, h->stream);
            }
            if (e == cudaSuccess && t + 1 < t1) {
                e = step_from(h, seg[k], seg[k + 1], step0 + (uint32_t)t, sfacc[k]);
                h->launches += 1;
            }
        }
        // reverse through the segment
        for (int t = t1 - 1; t >= t0 && e == cudaSuccess; --t) {
            const int k = t - t0;
            e = cudaMemsetAsync(gstep, 0, grad_bytes, h->stream);
            if (e == cudaSuccess) e = launch_adjoint(h, seg[k], lam[cur], lam[1 - cur], gstep, sfacc[k]);
            if (e == cudaSuccess) {
                const size_t cnt = 3 * h->n_nodes;
                k_axpy1<<<(unsigned int)std::min<size_t>((cnt + 255) / 256, 4096), 256, 0, h->stream>>>(grad_force,
                                                                                                      gstep, cnt);
                e = cudaGetLastError();
            }
            if (e == cudaSuccess && n) {
                lb_particles pk = *parts;
                pk.pos = spos[k];
                pk.mom = smom[k];
                if (lb_adjoint_couple(h, seg[k], &pk, &c1, gstep, grad_pos, grad_mom, lam[1 - cur], grad_force) !=
                    LB_OK)
                    e = cudaErrorLaunchFailure;
            }
            h->launches += 2;
            cur = 1 - cur;
        }
    }
    return e == cudaSuccess ? LB_OK : cuda_fail("lb_adjoint_kinetic_coupled", e);
}

}  // extern "C"
