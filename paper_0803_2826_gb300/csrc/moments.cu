// moments.cu -- state initialisation / conversion and the hydrodynamic
// moments of the pre-collision state.
//
//   init        n^eq(rho, u) of Eq. (original_equil_distrib), in FP64, stored
//               as deviations n - a rho0 in the storage format
//   moments     rho = m_0, j = m_1..3 + f/2, pi from m_0, m_4..m_9
//               (Sec. 3.4 Eqs. (hmodes_beg)-(hmodes_end); Sec. 3.7 for j)
//   sums        sum over fluid nodes of dm_k and dm_k^2 with a deterministic
//               two-pass reduction (block partials in scratch, then one
//               block adds the partials in block order)
#include <cstdio>

#include "stream_collide.cuh"

namespace lbi {

namespace {

__device__ __forceinline__ void node_xyz(size_t s, int nx, int ny, int &x, int &y, int &z)
{
    const size_t row = s / (size_t)nx;
    x = (int)(s - row * (size_t)nx);
    z = (int)(row / (size_t)ny);
    y = (int)(row - (size_t)z * (size_t)ny);
}

template <int DT>
__global__ void k_init_equilibrium(typename lbd::Store<DT>::T *dst, const double *rho, const double *u,
                                   const StepArgs a)
{
    using S = lbd::Store<DT>;
    const size_t N = a.nn;
    for (size_t s = blockIdx.x * (size_t)blockDim.x + threadIdx.x; s < N;
         s += (size_t)gridDim.x * blockDim.x) {
        const double r = rho ? rho[s] : (double)a.rho0;
        const double ux = u ? u[s] : 0.0, uy = u ? u[N + s] : 0.0, uz = u ? u[2 * N + s] : 0.0;
        const double u2 = ux * ux + uy * uy + uz * uz;
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            const double ai = (i == 0) ? 1.0 / 3.0 : (i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
            const double cu = ux * lbd::cx(i) + uy * lbd::cy(i) + uz * lbd::cz(i);
            const double dev = ai * (r - (double)a.rho0) + ai * r * (3.0 * cu + 4.5 * cu * cu - 1.5 * u2);
            dst[(size_t)i * a.pitch + s] = S::pack((float)dev, a.scale);
        }
    }
}

template <int DT>
__global__ void k_set_populations(typename lbd::Store<DT>::T *dst, const double *n, const StepArgs a)
{
    using S = lbd::Store<DT>;
    const size_t N = a.nn;
    for (size_t s = blockIdx.x * (size_t)blockDim.x + threadIdx.x; s < N;
         s += (size_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            const double ai = (i == 0) ? 1.0 / 3.0 : (i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
            const double dev = n[(size_t)i * N + s] - ai * (double)a.rho0;
            dst[(size_t)i * a.pitch + s] = S::pack((float)dev, a.scale);
        }
    }
}

template <int DT>
__global__ void k_get_populations(const typename lbd::Store<DT>::T *src, double *n, const StepArgs a)
{
    using S = lbd::Store<DT>;
    const size_t N = a.nn;
    const size_t plane = (size_t)a.nx * a.ny;
    for (size_t s = blockIdx.x * (size_t)blockDim.x + threadIdx.x; s < N;
         s += (size_t)gridDim.x * blockDim.x) {
        const int z = (int)(s / plane);
        const bool solid = z < a.z0 || z >= a.z1;  // wall nodes hold no state: the rest state
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            const double ai = (i == 0) ? 1.0 / 3.0 : (i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
            const float dev = solid ? 0.0f : S::cvt(src[(size_t)i * a.pitch + s], a.inv_scale);
            n[(size_t)i * N + s] = ai * (double)a.rho0 + (double)dev;
        }
    }
}

constexpr int kRedThreads = 256;

template <int DT>
__global__ void __launch_bounds__(kRedThreads)
    k_moments(const typename lbd::Store<DT>::T *__restrict__ src, const float *__restrict__ ffield, float *rho_out,
              float *j_out, float *pi_out, double *partials, const StepArgs a)
{
    using S = lbd::Store<DT>;
    const size_t N = a.nn;
    const bool walls = a.z0 > 0;
    // per-thread partial sums in FP32 (a thread sees ~N / grid nodes); the
    // block and grid levels add in FP64
    float acc[2 * 19];
#pragma unroll
    for (int k = 0; k < 38; ++k) acc[k] = 0.0f;

    for (size_t s = blockIdx.x * (size_t)blockDim.x + threadIdx.x; s < N;
         s += (size_t)gridDim.x * blockDim.x) {
        int x, y, z;
        node_xyz(s, a.nx, a.ny, x, y, z);
        if (z < a.z0 || z >= a.z1) {  // solid wall plane
            if (rho_out) rho_out[s] = a.rho0;
            if (j_out) for (int d = 0; d < 3; ++d) j_out[d * N + s] = 0.0f;
            if (pi_out) for (int c = 0; c < 6; ++c) pi_out[c * N + s] = 0.0f;
            continue;
        }
        const int xm = (x == 0) ? a.nx - 1 : x - 1, xp = (x == a.nx - 1) ? 0 : x + 1;
        const int ym = (y == 0) ? a.ny - 1 : y - 1, yp = (y == a.ny - 1) ? 0 : y + 1;
        int zm, zp;
        if (walls) {
            zm = z - 1;
            zp = z + 1;
        } else {
            zm = (z == 0) ? a.nz - 1 : z - 1;
            zp = (z == a.nz - 1) ? 0 : z + 1;
        }
        float n[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            const int sx = lbd::cx(i) == 1 ? xm : (lbd::cx(i) == -1 ? xp : x);
            const int sy = lbd::cy(i) == 1 ? ym : (lbd::cy(i) == -1 ? yp : y);
            const int sz = lbd::cz(i) == 1 ? zm : (lbd::cz(i) == -1 ? zp : z);
            const bool bounce = walls && lbd::cz(i) != 0 && (sz == 0 || sz == a.nz - 1);
            const size_t off = bounce ? ((size_t)lbd::opposite(i) * a.pitch + s)
                                      : ((size_t)i * a.pitch + ((size_t)sz * a.ny + sy) * a.nx + sx);
            n[i] = S::cvt(src[off], a.inv_scale);
        }
        float m[19];
        lbd::forward(n, m);
        const float rho = a.rho0 + m[0];
        if (rho_out) rho_out[s] = rho;
        if (j_out) {
            float fx = a.fx, fy = a.fy, fz = a.fz;
            if (ffield) {
                fx += ffield[s];
                fy += ffield[N + s];
                fz += ffield[2 * N + s];
            }
            j_out[s] = m[1] + 0.5f * fx;
            j_out[N + s] = m[2] + 0.5f * fy;
            j_out[2 * N + s] = m[3] + 0.5f * fz;
        }
        if (pi_out) {
            pi_out[s] = (rho + m[4] + m[5]) * (1.0f / 3.0f);
            pi_out[N + s] = (2.0f * rho + 2.0f * m[4] - m[5] + 3.0f * m[6]) * (1.0f / 6.0f);
            pi_out[2 * N + s] = (2.0f * rho + 2.0f * m[4] - m[5] - 3.0f * m[6]) * (1.0f / 6.0f);
            pi_out[3 * N + s] = m[7];
            pi_out[4 * N + s] = m[8];
            pi_out[5 * N + s] = m[9];
        }
#pragma unroll
        for (int k = 0; k < 19; ++k) {
            acc[k] += m[k];
            acc[19 + k] = fmaf(m[k], m[k], acc[19 + k]);
        }
    }

    // block reduction in a fixed order: warp shuffles, then warps in order
    __shared__ double red[kRedThreads / 32][38];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 38; ++k) {
        double v = (double)acc[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[warp][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < 38) {
        double v = 0.0;
        for (int w = 0; w < kRedThreads / 32; ++w) v += red[w][threadIdx.x];
        partials[(size_t)blockIdx.x * 38 + threadIdx.x] = v;
    }
}

// Component stores of a pair: one access where pair says the address allows.
__device__ __forceinline__ void put_pair(float *out, size_t k, lbp::F2 v, bool pair, bool second)
{
    float v0, v1;
    lbp::split(v, v0, v1);
    if (pair) {
        *reinterpret_cast<float2 *>(out + k) = make_float2(v0, v1);
        return;
    }
    out[k] = v0;
    if (second) out[k + 1] = v1;
}

// The fields alone (no sums): two consecutive nodes per thread over the
// linear index of all nodes, the loads of k_stream_collide_linear, solid
// nodes rho0 and zeros.  wide: component stride and outputs allow 8-byte
// stores.  Bound by memory (76 bytes a node read, 40 written).  256^3:
// 272 us, against 428 us with the 38 unused sums of k_moments in registers
// (96 of them, a quarter of the warps) and one node a thread.
template <int DT, bool WALLS, bool ODD>
__global__ void __launch_bounds__(kLinBX)
    k_fields(const typename lbd::Store<DT>::T *src, const float *ffield, float *rho_out, float *j_out, float *pi_out,
             const StepArgs a, bool wide)
{
    using lbp::F2;
    using lbp::f2s;
    const uint32_t N = (uint32_t)a.nn;
    PairAt at;
    at.s = 2u * (blockIdx.x * (uint32_t)kLinBX + threadIdx.x);
    wait_for_previous();
    if (at.s >= N) return;
    const bool second = at.s + 1u < N;
    const uint32_t row = divide(at.s, a.dnx), z = divide(row, a.dny);
    at.x = (int)(at.s - row * (uint32_t)a.nx);
    at.y = (int)(row - z * (uint32_t)a.ny);
    at.z = (int)z;
    at.va = true;
    at.vb = second;
    bool solid0 = false, solid1 = false;
    if (WALLS) {
        int xb, yb, zb;
        second_node(a, at, xb, yb, zb);
        solid0 = at.z < a.z0 || at.z >= a.z1;
        solid1 = zb < a.z0 || zb >= a.z1;
        at.va = !solid0;
        at.vb = second && !solid1;
        if (solid0) {  // the pulls are those of the fluid node of the pair
            at.x = xb;
            at.y = yb;
            at.z = zb;
        }
    }
    F2 n[19], m[19];
    float f0[3], f1[3];
    if (!WALLS || at.va || at.vb) {
        load_linear<DT, true, WALLS, ODD>(src, ffield, nullptr, a, at, n, f0, f1);
    } else {
#pragma unroll
        for (int i = 0; i < 19; ++i) n[i] = f2s(0.0f);
        f0[0] = f0[1] = f0[2] = f1[0] = f1[1] = f1[2] = 0.0f;
    }
    lbp::forward2(n, m);
    const bool pair = wide && second;
    // solid nodes: rho0, and zeros
    const auto fluid = [&](F2 v) {
        return WALLS ? lbp::f2(solid0 ? 0.0f : lbp::lo(v), solid1 ? 0.0f : lbp::hi(v)) : v;
    };
    const F2 rho = f2s(a.rho0) + fluid(m[0]);
    if (rho_out) put_pair(rho_out, at.s, rho, pair, second);
    if (j_out) {
#pragma unroll
        for (int d = 0; d < 3; ++d)
            put_pair(j_out, d * a.nn + at.s, fluid(lbp::fma2(f2s(0.5f), lbp::f2(f0[d], f1[d]), m[1 + d])), pair, second);
    }
    if (pi_out) {
        const F2 third = f2s(1.0f / 3.0f), sixth = f2s(1.0f / 6.0f);
        const F2 b = (rho + rho) + (m[4] + m[4]) - m[5];
        const F2 t6 = m[6] * 3.0f;
        put_pair(pi_out, at.s, fluid((rho + m[4] + m[5]) * third), pair, second);
        put_pair(pi_out, a.nn + at.s, fluid((b + t6) * sixth), pair, second);
        put_pair(pi_out, 2 * a.nn + at.s, fluid((b - t6) * sixth), pair, second);
#pragma unroll
        for (int c = 3; c < 6; ++c) put_pair(pi_out, c * a.nn + at.s, fluid(m[4 + c]), pair, second);
    }
}

__global__ void k_sum_partials(const double *partials, int nblocks, double *sums, unsigned int *err)
{
    const int k = threadIdx.x;
    if (k >= 38) return;
    double v = 0.0;
    for (int b = 0; b < nblocks; ++b) v += partials[(size_t)b * 38 + k];
    sums[k] = v;
    if (!isfinite(v)) atomicOr(err, LB_DERR_NONFINITE);
}

int grid_for(size_t N, int cap)
{
    size_t g = (N + kRedThreads - 1) / kRedThreads;
    if (g > (size_t)cap) g = (size_t)cap;
    if (g < 1) g = 1;
    return (int)g;
}

}  // namespace

#define LBI_DT_SWITCH(DTV, CALL)                  \
    switch (DTV) {                                \
    case LB_F32: { constexpr int DT = 0; CALL; } break;  \
    case LB_F16: { constexpr int DT = 1; CALL; } break;  \
    default: { constexpr int DT = 2; CALL; } break;      \
    }

cudaError_t launch_init_equilibrium(const lb_handle *h, void *dst, const double *rho, const double *u)
{
    const StepArgs a = make_args(h);
    const int g = grid_for(a.nn, 8 * device_sm_count());
    LBI_DT_SWITCH(h->p.dtype,
                  (k_init_equilibrium<DT><<<g, kRedThreads, 0, h->stream>>>(
                      static_cast<typename lbd::Store<DT>::T *>(dst), rho, u, a)));
    return cudaGetLastError();
}

cudaError_t launch_set_populations(const lb_handle *h, void *dst, const double *n)
{
    const StepArgs a = make_args(h);
    const int g = grid_for(a.nn, 8 * device_sm_count());
    LBI_DT_SWITCH(h->p.dtype, (k_set_populations<DT><<<g, kRedThreads, 0, h->stream>>>(
                                  static_cast<typename lbd::Store<DT>::T *>(dst), n, a)));
    return cudaGetLastError();
}

cudaError_t launch_get_populations(const lb_handle *h, const void *src, double *n)
{
    const StepArgs a = make_args(h);
    const int g = grid_for(a.nn, 8 * device_sm_count());
    LBI_DT_SWITCH(h->p.dtype, (k_get_populations<DT><<<g, kRedThreads, 0, h->stream>>>(
                                  static_cast<const typename lbd::Store<DT>::T *>(src), n, a)));
    return cudaGetLastError();
}

cudaError_t launch_moments(const lb_handle *h, const void *src, float *rho, float *j, float *pi, double *sums)
{
    const StepArgs a = make_args(h);
    if (!sums) {
        const bool wide = a.nn % 2 == 0 && pair_aligned(rho, 8) && pair_aligned(j, 8) && pair_aligned(pi, 8);
        const dim3 grid((unsigned)(((a.nn + 1) / 2 + kLinBX - 1) / kLinBX));
        const bool odd = !sc_paired(h), walls = h->p.walls != 0;
        LBI_DT_SWITCH(h->p.dtype, return launch_chained(walls ? (odd ? k_fields<DT, true, true> : k_fields<DT, true, false>)
                                                              : (odd ? k_fields<DT, false, true> : k_fields<DT, false, false>),
                                                        grid, kLinBX, h->stream,
                                                        static_cast<const typename lbd::Store<DT>::T *>(src), h->force,
                                                        rho, j, pi, a, wide));
    }
    const int g = grid_for(a.nn, h->red_blocks);
    double *partials = h->d_partials;
    LBI_DT_SWITCH(h->p.dtype, (k_moments<DT><<<g, kRedThreads, 0, h->stream>>>(
                                  static_cast<const typename lbd::Store<DT>::T *>(src), h->force, rho, j,
                                  pi, partials, a)));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_sum_partials<<<1, 64, 0, h->stream>>>(h->d_partials, g, sums, h->d_err);
    return cudaGetLastError();
}

}  // namespace lbi
