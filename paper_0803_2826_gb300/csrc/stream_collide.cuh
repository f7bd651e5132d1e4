// stream_collide.cuh -- fused pull-stream + MRT collision + noise + forcing.
//
// Two consecutive nodes per thread in packed FP32 (f32x2.cuh); the 19 plane
// loads and 19 plane stores of a warp are coalesced (the +-x neighbours of a
// row are the same 32-byte sectors shifted by one element).  Threads map to
// the nodes in one of two ways.  Rows whose pairs fill whole blocks (nx a
// multiple of 256) keep one row per block: no division, y and z from the
// block index (k_stream_collide2; 256^3 FP32 with noise 383 us a step against
// 389 us in the linear mapping when the two were compared).  All other boxes run over the linear node
// index (k_stream_collide_linear), so no lane is idle however short or odd the
// rows are: 64^3 10.3 us against 12.3 us with a block per row, 200^3 189 us
// against 248 us, and rows of odd length, which went one node a thread in
// scalar arithmetic before, 257 x 131 x 129 BF16 between walls 121 us against
// 170 us.  Everything between the loads and the stores stays in registers:
//   pull       n_i(r) = n*_i(r - c_i)                       Eq. (LBE)
//              (link bounce-back at solid z-planes,          Sec. 4.1 Eq. (MBB), u_b = 0)
//   moments    m_k = sum_i e_ki n_i                          Sec. 3.4 Eq. (forward), Table 1
//   velocity   j = m_1..3 + f/2, u = j / rho                 Sec. 3.7 Eq. (special_choice_momentum_density)
//   relax      m*_k = m^eq_k + gamma_k (m_k - m^eq_k) + F_k  Eq. (lco_update); Sec. 3.7 Sigma
//   noise      + sqrt(mu rho w_k) (1 - gamma_k^2)^1/2 r_k    Eqs. (stochupdaterule1), (detailedbalance1)
//   back       n*_i = a_i sum_k e_ki m*_k / w_k              Eq. (back_transformation), q = a
//   store      deviation n*_i - a_i rho0 (scaled for FP16 / BF16)
#pragma once

#include "d3q19.cuh"
#include "f32x2.cuh"
#include "lbf_internal.h"

namespace lbi {

constexpr int kBX = 128;  // threads per block along x
// Threads per block of the linear mapping: small boxes then still spread over
// the SMs (16^3: 4.1 us a step with 64, 5.6 us with 128; no difference from
// 64^3 on).
constexpr int kLinBX = 64;


// Collision of one node (Sec. 3.4, 3.5, 3.7) from its pulled populations n
// (deviations n_i - a_i rho0) and the force density (fx, fy, fz) to the
// post-collision deviations out: lbp::relax2, add_noise2 and backward2 for one
// node, operation by operation, so that a node that is updated again by itself
// (impulse nodes, nodes next to spheres) rounds as its neighbours in the packed
// update do.  (What multiplications the assembler joins with an addition behind
// them can still differ.)  The noise stream is Philox with round keys rk and
// counter (node, a.step, b, replica).
template <bool NOISE>
__device__ __forceinline__ void collide_node(const float n[19], float fx, float fy, float fz, const StepArgs &a,
                                             const lbd::RoundKeys &rk, uint32_t node, uint32_t replica,
                                             float out[19])
{
    float m[19];
    lbd::forward<true>(n, m);
    const float rho = a.rho0 + m[0];
    const float inv_rho = __frcp_rn(rho);
    const float ux = __fmul_rn(fmaf(0.5f, fx, m[1]), inv_rho);
    const float uy = __fmul_rn(fmaf(0.5f, fy, m[2]), inv_rho);
    const float uz = __fmul_rn(fmaf(0.5f, fz, m[3]), inv_rho);
    const float uxx = __fmul_rn(ux, ux), uyy = __fmul_rn(uy, uy), uzz = __fmul_rn(uz, uz);
    const float u2 = uxx + uyy + uzz;
    const float ruy = __fmul_rn(rho, uy), nrho = -a.rho0 - m[0], nruy = __fmul_rn(nrho, uy);
    const float t5 = __fmul_rn(uxx, 3.0f) - u2, t6 = uyy - uzz;
    float S[6] = {__fmul_rn(rho, u2), __fmul_rn(rho, t5), __fmul_rn(rho, t6),
                  __fmul_rn(ruy, ux), __fmul_rn(ruy, uz), __fmul_rn(__fmul_rn(rho, uz), ux)};
    const float d[6] = {fmaf(nrho, u2, m[4]), fmaf(nrho, t5, m[5]), fmaf(nrho, t6, m[6]),
                        fmaf(nruy, ux, m[7]), fmaf(nruy, uz, m[8]), fmaf(__fmul_rn(nrho, uz), ux, m[9])};
    float M[19];
    M[0] = m[0];
    M[1] = m[1];
    M[2] = m[2];
    M[3] = m[3];
    if (a.forced) {
        const float xx = __fmul_rn(ux, fx), yy = __fmul_rn(uy, fy), zz = __fmul_rn(uz, fz);
        const float uf = xx + yy + zz;
        S[0] = fmaf(uf, a.frc[0], S[0]);
        S[1] = fmaf(__fmul_rn(xx, 3.0f) - uf, a.frc[1], S[1]);
        S[2] = fmaf(yy - zz, a.frc[1], S[2]);
        S[3] = fmaf(__fmul_rn(ux, fy) + __fmul_rn(uy, fx), a.frc[2], S[3]);
        S[4] = fmaf(__fmul_rn(uy, fz) + __fmul_rn(uz, fy), a.frc[2], S[4]);
        S[5] = fmaf(__fmul_rn(uz, fx) + __fmul_rn(ux, fz), a.frc[2], S[5]);
        M[1] += fx;
        M[2] += fy;
        M[3] += fz;
    }
#pragma unroll
    for (int k = 4; k < 10; ++k)
        M[k] = __fmul_rn(fmaf(d[k - 4], k == 4 ? a.g_bulk : a.g_shear, S[k - 4]), lbd::inv_w(k));
#pragma unroll
    for (int k = 10; k < 19; ++k) M[k] = __fmul_rn(m[k], a.rel[k - 10]);
    if (NOISE) {
        const float nsd = -sqrtf(a.noise_rho0 ? a.mu * a.rho0 : __fmul_rn(rho, a.mu));
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const lbd::U4 r = lbd::philox10(lbd::U4{node, a.step, (uint32_t)b, replica}, rk);
            float g[4];
            lbp::box_muller1(r.x, r.y, g[0], g[1], nsd);
            lbp::box_muller1(r.z, r.w, g[2], g[3], nsd);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int k = 4 + 4 * b + j;
                if (k < 19) M[k] = fmaf(g[j], a.amp[k - 4], M[k]);
            }
        }
    }
    lbd::backward<true>(M, out);
}

// One step of a butterfly reduce-scatter over the warp: each lane keeps one
// half of its N values (the upper half if `hi`), receives the other lane's
// copy of that half and adds it, so the lanes now hold disjoint halves.
template <int N>
__device__ __forceinline__ void butterfly_half(const float *in, float *out, int offset, bool hi)
{
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const float keep = hi ? in[i + N / 2] : in[i];
        const float send = hi ? in[i] : in[i + N / 2];
        out[i] = keep + __shfl_xor_sync(0xffffffffu, send, offset);
    }
}

// Moment sums of a warp: lane l holds 38 values (m0_k + m1_k, then
// m0_k^2 + m1_k^2; zeros where valid is false), the warp needs their 38 sums.
// Five butterfly steps halve the values per lane (40 -> 20 -> 10 -> 5, padded
// to 6 -> 3, padded to 4 -> 2), each sum is formed in a fixed order, and the
// lane that ends with sum k writes it to part[warp][k].  After a
// __syncthreads the block's sums are part[0] + ... + part[kBX/32 - 1]
// (block_moment_sums_out).  Every lane of the warp calls it.
__device__ __forceinline__ void warp_moment_sums(const float m0[19], const float m1[19], bool valid,
                                                 float (*part)[38])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float a[40];
#pragma unroll
    for (int k = 0; k < 19; ++k) {
        a[k] = m0[k] + m1[k];
        a[19 + k] = fmaf(m0[k], m0[k], m1[k] * m1[k]);
    }
    a[38] = a[39] = 0.0f;
    if (!__all_sync(0xffffffffu, valid)) {  // a warp at the end of a row
#pragma unroll
        for (int k = 0; k < 38; ++k) a[k] = valid ? a[k] : 0.0f;
    }
    float b[20], c[10], d[6], e[4], f[2];
    butterfly_half<40>(a, b, 16, lane & 16);
    butterfly_half<20>(b, c, 8, lane & 8);
    butterfly_half<10>(c, d, 4, lane & 4);
    d[5] = 0.0f;
    butterfly_half<6>(d, e, 2, lane & 2);
    e[3] = 0.0f;
    butterfly_half<4>(e, f, 1, lane & 1);
    // lane l holds, for j = 0, 1, the sum of entry k = base + b1 3 + pos of
    // the 5-entry block base = 20 b4 + 10 b3 + 5 b2, pos = 2 b0 + j (b_i the
    // bits of l); pos 3 and block entries 5 and beyond are padding
    const int base = 20 * ((lane >> 4) & 1) + 10 * ((lane >> 3) & 1) + 5 * ((lane >> 2) & 1);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int pos = 2 * (lane & 1) + j;
        const int idx = 3 * ((lane >> 1) & 1) + pos;
        const int k = base + idx;
        if (pos < 3 && idx < 5 && k < 38) part[warp][k] = f[j];
    }
}

// FP32 throughout: FP64 arithmetic is slow on this part, and a block that
// ends in a chain of FP64 adds holds its SM slot meanwhile.
__device__ __forceinline__ void block_moment_sums_out(const float (*part)[38], float *out)
{
    __syncthreads();
    if (threadIdx.x < 38) {
        float t = 0.0f;
#pragma unroll
        for (int w = 0; w < kBX / 32; ++w) t += part[w][threadIdx.x];
        out[threadIdx.x] = t;
    }
}

// The whole update of fluid node (x, y, z): pull, force, collision, store.
template <int DT, bool NOISE, bool FIELD, bool WALLS>
__device__ __forceinline__ void update_node(const typename lbd::Store<DT>::T *__restrict__ src,
                                            typename lbd::Store<DT>::T *__restrict__ dst,
                                            const float *__restrict__ ffield, const float *__restrict__ facc,
                                            const StepArgs &a, int x, int y, int z)
{
    using S = lbd::Store<DT>;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int xm = (x == 0) ? nx - 1 : x - 1;
    const int xp = (x == nx - 1) ? 0 : x + 1;
    const int ym = (y == 0) ? ny - 1 : y - 1;
    const int yp = (y == ny - 1) ? 0 : y + 1;
    int zm, zp;
    if (WALLS) {
        zm = z - 1;
        zp = z + 1;
    } else {
        zm = (z == 0) ? nz - 1 : z - 1;
        zp = (z == nz - 1) ? 0 : z + 1;
    }
    const size_t P = a.pitch;
    const uint32_t self = (uint32_t)((z * ny + y) * nx + x);

    // ---- pull streaming --------------------------------------------------
    float n[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        const int sx = lbd::cx(i) == 1 ? xm : (lbd::cx(i) == -1 ? xp : x);
        const int sy = lbd::cy(i) == 1 ? ym : (lbd::cy(i) == -1 ? yp : y);
        const int sz = lbd::cz(i) == 1 ? zm : (lbd::cz(i) == -1 ? zp : z);
        bool bounce = false;
        if (WALLS && lbd::cz(i) != 0) bounce = (sz == 0) || (sz == nz - 1);
        const size_t k = bounce ? (size_t)lbd::opposite(i) * P + self
                                : (size_t)i * P + (uint32_t)((sz * ny + sy) * nx + sx);
        n[i] = in_bounds(k, 19 * P, a.err) ? S::load(src + k, a.inv_scale) : 0.0f;
    }

    // ---- force and collision -----------------------------------------------
    float fx = a.fx, fy = a.fy, fz = a.fz;
    if (FIELD) {
        if (ffield) {  // caller's field, component stride N
            fx += ld_f32(ffield + self);
            fy += ld_f32(ffield + a.nn + self);
            fz += ld_f32(ffield + 2 * a.nn + self);
        }
        if (facc) {  // library accumulator, component stride = plane pitch
            fx += ld_f32(facc + self);
            fy += ld_f32(facc + P + self);
            fz += ld_f32(facc + 2 * P + self);
        }
    }
    float out[19];
    collide_node<NOISE>(n, fx, fy, fz, a, a.rk, self, a.replica, out);
#pragma unroll
    for (int i = 0; i < 19; ++i)
        if (in_bounds((size_t)i * P + self, 19 * P, a.err)) dst[(size_t)i * P + self] = S::pack(out[i], a.scale);
}

// Node k (0 .. span^3 - 1, x fastest) of the block of nodes that an impulse
// stencil can touch around the recorded cell (bx, by, bz): [b, b + 1] per
// axis for span 2 (phi_2), [b - 1, b + 2] for span 4 (phi_3 and phi_4).
// Returns false for a node outside the fluid.
template <bool WALLS>
__device__ __forceinline__ bool patch_node(int bx, int by, int bz, int k, int span, const StepArgs &a, int &x,
                                           int &y, int &z)
{
    if (span == 3) {  // a phi_3 stencil origin: the 27 nodes of the stencil
        x = bx + k % 3;
        y = by + (k / 3) % 3;
        z = bz + k / 9;
    } else {  // a cell: its corners (span 2) or one node further on each side (span 4)
        const int sh = span == 4 ? 2 : 1, lo = span == 4 ? -1 : 0, m = span - 1;
        x = bx + lo + (k & m);
        y = by + lo + ((k >> sh) & m);
        z = bz + lo + (k >> (2 * sh));
    }
    x = x < 0 ? x + a.nx : (x >= a.nx ? x - a.nx : x);
    y = y < 0 ? y + a.ny : (y >= a.ny ? y - a.ny : y);
    if ((unsigned)x >= (unsigned)a.nx) x = ((x % a.nx) + a.nx) % a.nx;  // boxes narrower than the stencil
    if ((unsigned)y >= (unsigned)a.ny) y = ((y % a.ny) + a.ny) % a.ny;
    if (!WALLS) {
        z = z < 0 ? z + a.nz : (z >= a.nz ? z - a.nz : z);
        if ((unsigned)z >= (unsigned)a.nz) z = ((z % a.nz) + a.nz) % a.nz;
    }
    return z >= a.z0 && z < a.z1;
}

// Clears the impulses of a node patch_node refuses, where it is a solid one
// (clear_solid; any number of threads may).
__device__ __forceinline__ void clear_outside(float *facc, const StepArgs &a, int x, int y, int z)
{
    if (z < 0 || z >= a.nz) return;
    const size_t node = ((size_t)z * a.ny + y) * a.nx + x;
    facc[node] = facc[a.pitch + node] = facc[2 * a.pitch + node] = 0.0f;
}

// Re-update of the nodes that received particle impulses, after an update of
// all nodes that left the impulses out (the coupling ran meanwhile): the
// span^3 nodes of each record of particle p, records[s][p] (the linear index
// of its cell at sub-step s, or of its phi_3 stencil origin: span 3), are
// updated again from the same pre-step state
// with the impulses added.  The update of a node depends only on that state, the
// forces at the node and the counter-based noise, so the result is the one a
// single update with the impulses would give (collide_node).  Thread (p, q) walks p's
// distinct cells and takes nodes q, q + 8, ... of each; a node shared by several
// particles is updated once, by the thread that raises its tag to `tag`
// first (tags grow by one per patch, so the array is never cleared).
template <int DT, bool NOISE, bool WALLS>
__global__ void __launch_bounds__(kBX) k_patch_impulse_nodes(const typename lbd::Store<DT>::T *__restrict__ src,
                                                             typename lbd::Store<DT>::T *__restrict__ dst,
                                                             const float *ffield, float *facc, const int *records,
                                                             int n, int nsub, int span, unsigned int *claim,
                                                             unsigned int tag, const StepArgs a)
{
    const int t = blockIdx.x * kBX + threadIdx.x;
    wait_for_previous();
    if (t >= n * 8) return;
    const int p = t >> 3, q = t & 7;
    const int nk = span * span * span;
    const unsigned group = 0xFFu << (threadIdx.x & 24);
    int prev = -1, mine = 0;
    for (int s = 0; s < nsub; ++s) {
        // eight sub-steps' records at a time, one in a lane: one load's latency for all
        if ((s & 7) == 0) mine = s + q < nsub ? records[(size_t)(s + q) * n + p] : -1;
        const int base = __shfl_sync(group, mine, s & 7, 8);
        if (base == prev) continue;  // same cell as the sub-step before
        prev = base;
        const uint32_t row = divide((uint32_t)base, a.dnx), plane = divide(row, a.dny);
        const int bx = base - (int)(row * (uint32_t)a.nx), by = (int)(row - plane * (uint32_t)a.ny), bz = (int)plane;
        for (int e = q; e < nk; e += 8) {
            int x, y, z;
            if (!patch_node<WALLS>(bx, by, bz, e, span, a, x, y, z)) {
                clear_outside(facc, a, x, y, z);
                continue;
            }
            const size_t node = ((size_t)z * a.ny + y) * a.nx + x;
            if (atomicMax(claim + node, tag) == tag) continue;  // another thread has it
            update_node<DT, NOISE, true, WALLS>(src, dst, ffield, facc, a, x, y, z);
            // the impulses are applied: clear them for the next coupling call
            loads_done();
            facc[node] = 0.0f;
            facc[a.pitch + node] = 0.0f;
            facc[2 * a.pitch + node] = 0.0f;
        }
    }
}

// The same for FP32 storage, by a correction of the stored result instead of
// a second update: the forces enter the collision only through u and the
// force moments of modes 1..9, and rho and the pre-collision j are
// recovered from the stored n* (mass is conserved, the stored momentum is
// j + f).  With f_b the force of the first update and f_n = f_b + the
// impulse, the stored moments change by dM_1..3 = 3 (f_n - f_b) and, for
// k = 4..9, dM_k = ((1 - gamma_k) (m^eq_k(u_n) - m^eq_k(u_b)) + F_k(u_n, f_n)
// - F_k(u_b, f_b)) / w_k; n* += backward(dM).  No pull and no noise; the
// claim makes sure each node is corrected once.  Eight blocks per SM (64 registers, no
// spills): the launch for the workload's ~1.3e5 threads fits in one wave.
template <bool WALLS>
__global__ void __launch_bounds__(kBX, 8) k_patch_impulse_nodes_f32(float *dst, const float *ffield, float *facc,
                                                                 const int *records, int n,
                                                                 int nsub, int span, unsigned int *claim,
                                                                 unsigned int tag, const StepArgs a)
{
    const int t = blockIdx.x * kBX + threadIdx.x;
    wait_for_previous();
    if (t >= n * 8) return;
    const int p = t >> 3, q = t & 7;
    const size_t P = a.pitch;
    const int nk = span * span * span;
    const unsigned group = 0xFFu << (threadIdx.x & 24);
    int prev = -1, mine = 0;
    for (int s = 0; s < nsub; ++s) {
        // eight sub-steps' records at a time, one in a lane: one load's latency for all
        if ((s & 7) == 0) mine = s + q < nsub ? records[(size_t)(s + q) * n + p] : -1;
        const int base = __shfl_sync(group, mine, s & 7, 8);
        if (base == prev) continue;  // same cell as the sub-step before
        prev = base;
        const uint32_t row = divide((uint32_t)base, a.dnx), plane = divide(row, a.dny);
        const int bx = base - (int)(row * (uint32_t)a.nx), by = (int)(row - plane * (uint32_t)a.ny), bz = (int)plane;
        for (int e = q; e < nk; e += 8) {
            int x, y, z;
            if (!patch_node<WALLS>(bx, by, bz, e, span, a, x, y, z)) {
                clear_outside(facc, a, x, y, z);
                continue;
            }
            const size_t node = ((size_t)z * a.ny + y) * a.nx + x;
            // the claim, the impulse and the stored values are requested
            // together (one memory round trip instead of three); the values
            // are used only by the thread that wins the claim, and nothing
            // else writes this node during the kernel
            const unsigned int had = atomicMax(claim + node, tag);
            const float df[3] = {facc[node], facc[P + node], facc[2 * P + node]};
            float ns[19], m[19];
#pragma unroll
            for (int i = 0; i < 19; ++i) ns[i] = dst[(size_t)i * P + node];
            if (had == tag) continue;  // another thread has it
            if (df[0] == 0.0f && df[1] == 0.0f && df[2] == 0.0f) continue;
            lbd::forward(ns, m);
            float fb[3] = {a.fx, a.fy, a.fz};
            if (ffield) {
                fb[0] += ffield[node];
                fb[1] += ffield[a.nn + node];
                fb[2] += ffield[2 * a.nn + node];
            }
            const float fn[3] = {fb[0] + df[0], fb[1] + df[1], fb[2] + df[2]};
            const float rho = a.rho0 + m[0];
            const float ir = 1.0f / rho;
            const float j[3] = {m[1] - fb[0], m[2] - fb[1], m[3] - fb[2]};
            float dM[19];
#pragma unroll
            for (int k = 0; k < 19; ++k) dM[k] = 0.0f;
            dM[1] = 3.0f * df[0];
            dM[2] = 3.0f * df[1];
            dM[3] = 3.0f * df[2];
            const float gs1 = 1.0f + a.g_shear;
#pragma unroll
            for (int side = 0; side < 2; ++side) {  // + (u_n, f_n), - (u_b, f_b)
                const float *f = side ? fb : fn;
                const float sg = side ? -1.0f : 1.0f;
                const float ux = (j[0] + 0.5f * f[0]) * ir, uy = (j[1] + 0.5f * f[1]) * ir, uz = (j[2] + 0.5f * f[2]) * ir;
                const float uxx = ux * ux, uyy = uy * uy, uzz = uz * uz, u2 = uxx + uyy + uzz;
                const float uf = ux * f[0] + uy * f[1] + uz * f[2];
                dM[4] += sg * ((1.0f - a.g_bulk) * rho * u2 + (1.0f + a.g_bulk) * uf);
                dM[5] += sg * ((1.0f - a.g_shear) * rho * (3.0f * uxx - u2) + gs1 * (3.0f * ux * f[0] - uf));
                dM[6] += sg * ((1.0f - a.g_shear) * rho * (uyy - uzz) + gs1 * (uy * f[1] - uz * f[2]));
                dM[7] += sg * ((1.0f - a.g_shear) * rho * ux * uy + 0.5f * gs1 * (ux * f[1] + uy * f[0]));
                dM[8] += sg * ((1.0f - a.g_shear) * rho * uy * uz + 0.5f * gs1 * (uy * f[2] + uz * f[1]));
                dM[9] += sg * ((1.0f - a.g_shear) * rho * uz * ux + 0.5f * gs1 * (uz * f[0] + ux * f[2]));
            }
#pragma unroll
            for (int k = 4; k < 10; ++k) dM[k] *= lbd::inv_w(k);
            float dn[19];
            lbd::backward(dM, dn);
#pragma unroll
            for (int i = 0; i < 19; ++i) dst[(size_t)i * P + node] = ns[i] + dn[i];
            // the impulses are applied: clear them for the next coupling call
            facc[node] = 0.0f;
            facc[P + node] = 0.0f;
            facc[2 * P + node] = 0.0f;
        }
    }
}

// Two neighbouring nodes x0 = 2t, x0 + 1 per thread (even nx).  Both pull
// their populations from the same rows of each plane, so one address per
// plane serves both (the second is an immediate offset); planes with c_x = 0
// and all stores move the pair as one 8-byte (FP32) or 4-byte (FP16 / BF16)
// access.  Collision and noise are those of collide_node, computed for the
// two nodes at once in packed FP32 (f32x2.cuh).
template <int DT>
struct Pair;
template <>
struct Pair<0> {
    static __device__ __forceinline__ void load(const float *p, float inv, float &a, float &b)
    {
        const float2 v = ld_f32x2(p);
        a = v.x;
        b = v.y;
    }
    static __device__ __forceinline__ void store(float *p, float a, float b, float)
    {
        *reinterpret_cast<float2 *>(p) = make_float2(a, b);
    }
};
template <>
struct Pair<1> {
    static __device__ __forceinline__ void load(const __half *p, float inv, float &a, float &b)
    {
        const unsigned int w = ld_u32(p);
        const __half2 v = *reinterpret_cast<const __half2 *>(&w);
        a = __low2float(v) * inv;
        b = __high2float(v) * inv;
    }
    static __device__ __forceinline__ void store(__half *p, float a, float b, float sc)
    {
        *reinterpret_cast<__half2 *>(p) = __floats2half2_rn(a * sc, b * sc);
    }
};
template <>
struct Pair<2> {
    static __device__ __forceinline__ void load(const __nv_bfloat16 *p, float inv, float &a, float &b)
    {
        const unsigned int w = ld_u32(p);
        const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162 *>(&w);
        a = __low2float(v) * inv;
        b = __high2float(v) * inv;
    }
    static __device__ __forceinline__ void store(__nv_bfloat16 *p, float a, float b, float sc)
    {
        *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(a * sc, b * sc);
    }
};

// Pull streaming of nodes x0, x0 + 1 of row (y, z) (link bounce-back at solid
// z-planes) into packed pairs n (node x0 in the low halves, FP16 / BF16
// unscaled), and their force densities f0, f1 (body force + caller's field +
// library accumulator).  Impulses that are applied for good (a.consume) are
// cleared here, by the thread that owns their nodes (take), so no other pass
// has to find them again: few nodes carry any, and the test is three ORs and a
// branch (512^3 FP16 with 1e5 particles: 50 us of clearing less a step).
template <int DT, bool WALLS>
__device__ __forceinline__ void pull_pair(const typename lbd::Store<DT>::T *__restrict__ src, const StepArgs &a, int x0,
                                          int y, int z, uint32_t self, lbp::F2 n[19])
{
    using S = lbd::Store<DT>;
    using PR = Pair<DT>;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int xm = (x0 == 0) ? nx - 1 : x0 - 1;       // source of node x0 for c_x = +1
    const int xp = (x0 + 2 == nx) ? 0 : x0 + 2;       // source of node x0 + 1 for c_x = -1
    const int ym = (y == 0) ? ny - 1 : y - 1;
    const int yp = (y == ny - 1) ? 0 : y + 1;
    int zm, zp;
    if (WALLS) {
        zm = z - 1;
        zp = z + 1;
    } else {
        zm = (z == 0) ? nz - 1 : z - 1;
        zp = (z == nz - 1) ? 0 : z + 1;
    }
    const uint32_t P = (uint32_t)a.pitch;
    const size_t lim = 19 * (size_t)P;  // elements of a population buffer (index checks)
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        const int sy = lbd::cy(i) == 1 ? ym : (lbd::cy(i) == -1 ? yp : y);
        const int sz = lbd::cz(i) == 1 ? zm : (lbd::cz(i) == -1 ? zp : z);
        bool bounce = false;
        if (WALLS && lbd::cz(i) != 0) bounce = (sz == 0) || (sz == nz - 1);
        // stored values as loaded (FP16 / BF16: still scaled; the pair is
        // unscaled below by one packed multiply)
        float v0 = 0.0f, v1 = 0.0f;
        if (bounce) {
            const uint32_t k = (uint32_t)lbd::opposite(i) * P + self;
            if (in_bounds(k + 1, lim, a.err)) PR::load(src + k, 1.0f, v0, v1);
        } else {
            const uint32_t row = (uint32_t)i * P + (uint32_t)((sz * ny + sy) * nx);
            if (lbd::cx(i) == 0) {
                if (in_bounds(row + x0 + 1, lim, a.err)) PR::load(src + row + x0, 1.0f, v0, v1);
            } else if (lbd::cx(i) == 1) {
                if (in_bounds(row + xm, lim, a.err) && in_bounds(row + x0, lim, a.err)) {
                    v0 = S::load(src + row + xm, 1.0f);
                    v1 = S::load(src + row + x0, 1.0f);
                }
            } else {
                if (in_bounds(row + x0 + 1, lim, a.err) && in_bounds(row + xp, lim, a.err)) {
                    v0 = S::load(src + row + x0 + 1, 1.0f);
                    v1 = S::load(src + row + xp, 1.0f);
                }
            }
        }
        n[i] = DT == 0 ? lbp::f2(v0, v1) : lbp::f2(v0, v1) * lbp::f2s(a.inv_scale);
    }
}

// A particle that a narrow channel cannot keep inside its band spreads to the
// solid planes too.  No update reads that; it is cleared, with the impulses
// that are applied, by the threads of the fluid nodes next to it.
__device__ __forceinline__ void clear_solid(float *facc, const StepArgs &a, int z, uint32_t self)
{
    const uint32_t plane = (uint32_t)a.nx * (uint32_t)a.ny;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (z == a.z0) facc[d * a.pitch + (self - plane)] = 0.0f;
        if (z == a.z1 - 1) facc[d * a.pitch + (self + plane)] = 0.0f;
    }
}
__device__ __forceinline__ void clear_solid_pair(float *facc, const StepArgs &a, int z, uint32_t self)  // even nx
{
    const uint32_t plane = (uint32_t)a.nx * (uint32_t)a.ny;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (z == a.z0) Pair<0>::store(facc + d * a.pitch + (self - plane), 0.0f, 0.0f, 1.0f);
        if (z == a.z1 - 1) Pair<0>::store(facc + d * a.pitch + (self + plane), 0.0f, 0.0f, 1.0f);
    }
}

template <int DT, bool FIELD, bool WALLS>
__device__ __forceinline__ void load_pair(const typename lbd::Store<DT>::T *__restrict__ src,
                                          const float *__restrict__ ffield, float *facc,
                                          const StepArgs &a, int x0, int y, int z, lbp::F2 n[19], float f0[3],
                                          float f1[3], bool take = true)
{
    const uint32_t P = (uint32_t)a.pitch;
    const uint32_t self = (uint32_t)((z * a.ny + y) * a.nx + x0);
    // only the planes next to a wall look at their links (z is the same for
    // a whole row, so a warp rarely takes both ways)
    if (WALLS && (z == a.z0 || z == a.z1 - 1)) {
        if (FIELD && facc && a.consume && take) clear_solid_pair(facc, a, z, self);
        pull_pair<DT, true>(src, a, x0, y, z, self, n);
    } else {
        pull_pair<DT, false>(src, a, x0, y, z, self, n);
    }
    f0[0] = f1[0] = a.fx;
    f0[1] = f1[1] = a.fy;
    f0[2] = f1[2] = a.fz;
    if (FIELD) {
        if (ffield) {  // caller's field, component stride N
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                f0[d] += ld_f32(ffield + d * a.nn + self);
                f1[d] += ld_f32(ffield + d * a.nn + self + 1);
            }
        }
        if (facc) {  // library accumulator, component stride = plane pitch
            unsigned int bits = 0u;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                float u, v;
                Pair<0>::load(facc + d * (size_t)P + self, 1.0f, u, v);
                f0[d] += u;
                f1[d] += v;
                bits |= __float_as_uint(u) | __float_as_uint(v);
            }
            if (bits && a.consume && take) {
#pragma unroll
                for (int d = 0; d < 3; ++d) Pair<0>::store(facc + d * (size_t)P + self, 0.0f, 0.0f, 1.0f);
            }
        }
    }
}

// Store of the packed post-collision pair (FP16 / BF16: scaled by one packed
// multiply, then rounded to nearest even).
template <int DT>
__device__ __forceinline__ void store_pair(typename lbd::Store<DT>::T *__restrict__ dst, const StepArgs &a,
                                           uint32_t self, const lbp::F2 out[19])
{
    const size_t P = a.pitch;
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        float o0, o1;
        lbp::split(DT == 0 ? out[i] : out[i] * lbp::f2s(a.scale), o0, o1);
        if (in_bounds((size_t)i * P + self + 1, 19 * P, a.err)) Pair<DT>::store(dst + (size_t)i * P + self, o0, o1, 1.0f);
    }
}

template <int DT, bool NOISE, bool FIELD, bool WALLS, bool SUMS = false>
__device__ __forceinline__ void update_pair(const typename lbd::Store<DT>::T *__restrict__ src,
                                            typename lbd::Store<DT>::T *__restrict__ dst,
                                            const float *__restrict__ ffield, float *facc,
                                            const StepArgs &a, int x0, int y, int z, bool valid = true,
                                            float (*part)[38] = nullptr)
{
    const uint32_t self = (uint32_t)((z * a.ny + y) * a.nx + x0);
    lbp::F2 n[19];
    float f0[3], f1[3];
    load_pair<DT, FIELD, WALLS>(src, ffield, facc, a, x0, y, z, n, f0, f1, valid);
    // both nodes' moments, collision, noise and back transform in packed
    // FP32 (f32x2.cuh), node x0 in the low halves
    lbp::F2 m[19], out[19];
    lbp::forward2(n, m);
    if (SUMS) {  // both nodes' moments summed before the collisions
        float m0[19], m1[19];
#pragma unroll
        for (int k = 0; k < 19; ++k) lbp::split(m[k], m0[k], m1[k]);
        warp_moment_sums(m0, m1, valid, part);
        if (!valid) return;
    }
    lbp::collide_moments2<NOISE>(m, lbp::f2(f0[0], f1[0]), lbp::f2(f0[1], f1[1]), lbp::f2(f0[2], f1[2]), a, a.rk,
                                 self, a.replica, out);
    store_pair<DT>(dst, a, self, out);
}

// Rows mapped to blocks: block (x, y, z) takes 2 kBX consecutive nodes of row
// (y, z).  SUMS: the block also writes the moment sums of its nodes
// (pre-collision, as lb_moments defines them) to partials[block][38].
__device__ __forceinline__ size_t block_linear()
{
    return blockIdx.x + (size_t)gridDim.x * (blockIdx.y + (size_t)gridDim.y * blockIdx.z);
}

template <int DT, bool NOISE, bool FIELD, bool WALLS, bool SUMS>
__device__ __forceinline__ void rows_update(const typename lbd::Store<DT>::T *__restrict__ src,
                                            typename lbd::Store<DT>::T *__restrict__ dst,
                                            const float *__restrict__ ffield, float *facc, const StepArgs &a,
                                            float *partials)
{
    const int x0 = 2 * (blockIdx.x * kBX + threadIdx.x);
    wait_for_previous();
    if (SUMS) {
        __shared__ float part[kBX / 32][38];
        const bool valid = x0 < a.nx;  // lanes past the row load nodes 0, 1 of it and store nothing
        update_pair<DT, NOISE, FIELD, WALLS, true>(src, dst, ffield, facc, a, valid ? x0 : 0, blockIdx.y,
                                                   blockIdx.z + a.z0, valid, part);
        block_moment_sums_out(part, partials + 38 * block_linear());
    } else {
        if (x0 >= a.nx) return;
        update_pair<DT, NOISE, FIELD, WALLS>(src, dst, ffield, facc, a, x0, blockIdx.y, blockIdx.z + a.z0);
    }
}

template <int DT, bool NOISE, bool FIELD, bool WALLS, bool SUMS>
__global__ void __launch_bounds__(kBX)
    k_stream_collide2(const typename lbd::Store<DT>::T *__restrict__ src, typename lbd::Store<DT>::T *__restrict__ dst,
                      const float *__restrict__ ffield, float *facc, const StepArgs a, float *partials)
{
    rows_update<DT, NOISE, FIELD, WALLS, SUMS>(src, dst, ffield, facc, a, partials);
}

// The same where a force field is read: room for seven blocks of 128 threads
// per SM in FP32 (72 registers, no spills) and for eight in FP16 / BF16 (64
// registers, 24 to 72 bytes of spills), where the update wants warps more than
// registers: 512^3 FP16 between walls with the impulses of 1e5 tracers 3.43 ms a
// step against 3.49 ms with the compiler's own 72 to 74 registers.  Elsewhere
// the two are close: 512 x 512 x 256 FP16 1597 against 1590 us, 256^3 FP32
// between walls 407 against 412 us, 200^3 FP32 204 against 201 us.  Without a
// field the compiler's own choice, 72 registers, is the best (256^3 FP32 365 us;
// 371 us with room for six or seven blocks, 383 us for eight).
template <int DT>
constexpr int field_blocks() { return DT == 0 ? 7 : 8; }

template <int DT, bool NOISE, bool WALLS>
__global__ void __launch_bounds__(kBX, field_blocks<DT>())
    k_stream_collide2_field(const typename lbd::Store<DT>::T *__restrict__ src,
                            typename lbd::Store<DT>::T *__restrict__ dst, const float *__restrict__ ffield, float *facc,
                            const StepArgs a, float *partials)
{
    rows_update<DT, NOISE, true, WALLS, false>(src, dst, ffield, facc, a, partials);
}

// Two consecutive nodes s, s + 1 (s even) per thread over the fluid's linear
// index range, for boxes whose rows do not fill whole blocks of pairs: every
// lane of every warp but the last has its two nodes, whatever nx.  In a row
// of even length both nodes lie in the same row (load_pair); in one of odd
// length the pair may straddle two rows, or the wall and the fluid, so each
// node takes its own addresses and only the store moves the pair as one
// access.  va / vb: the node lies in the fluid (the first pair of a channel
// with an odd plane, the last of an odd number of nodes).
struct PairAt {
    uint32_t s;
    int x, y, z;    // node s, or s + 1 where only that one is fluid
    bool va, vb;
};

// Blocks of bx threads that cover the fluid nodes of a box of nn nodes, or
// those between its first and last plane (locate_pair).
inline dim3 linear_grid(size_t nn, size_t plane, bool walls, int bx)
{
    const size_t first = walls ? plane : 0;
    const size_t pairs = (nn - first - (first & ~(size_t)1) + 1) / 2;
    return dim3((unsigned)((pairs + bx - 1) / bx));
}
inline dim3 linear_grid(const StepArgs &a) { return linear_grid(a.nn, (size_t)a.nx * a.ny, a.z0 > 0, kLinBX); }

template <bool WALLS, int BX = kLinBX>
__device__ __forceinline__ bool locate_pair(const StepArgs &a, PairAt &p)
{
    const uint32_t plane = (uint32_t)a.nx * (uint32_t)a.ny;
    const uint32_t first = WALLS ? plane : 0u;
    const uint32_t end = (uint32_t)a.nn - first;
    p.s = (first & ~1u) + 2u * (blockIdx.x * (uint32_t)BX + threadIdx.x);
    if (p.s >= end) return false;
    p.va = !WALLS || p.s >= first;
    p.vb = p.s + 1u < end;
    const uint32_t s = p.va ? p.s : p.s + 1u;
    const uint32_t row = divide(s, a.dnx);
    const uint32_t z = divide(row, a.dny);
    p.x = (int)(s - row * (uint32_t)a.nx);
    p.y = (int)(row - z * (uint32_t)a.ny);
    p.z = (int)z;
    return true;
}

// Pull addresses of one node: row offsets of its neighbours and their x.  The
// box (nx, ny, nz, z0, z1, pitch) comes from any struct that has them.
struct PullAt {
    int x[3];          // x - 1, x, x + 1 (wrapped)
    uint32_t y[3], z[3];  // row offsets y nx and plane offsets z nx ny, the same way
    uint32_t self;
    bool lo, hi;       // next to the lower / upper wall: c_z = +1 / -1 bounce back
};

template <bool WALLS, class Geo>
__device__ __forceinline__ PullAt pull_at(const Geo &a, int x, int y, int z)
{
    PullAt p;
    p.x[0] = x == 0 ? a.nx - 1 : x - 1;
    p.x[1] = x;
    p.x[2] = x == a.nx - 1 ? 0 : x + 1;
    const uint32_t nx = (uint32_t)a.nx, pl = nx * (uint32_t)a.ny;
    p.y[0] = (uint32_t)(y == 0 ? a.ny - 1 : y - 1) * nx;
    p.y[1] = (uint32_t)y * nx;
    p.y[2] = (uint32_t)(y == a.ny - 1 ? 0 : y + 1) * nx;
    if (WALLS) {
        p.lo = z == a.z0;
        p.hi = z == a.z1 - 1;
        p.z[0] = (uint32_t)(z - 1) * pl;
        p.z[2] = (uint32_t)(z + 1) * pl;
    } else {
        p.lo = p.hi = false;
        p.z[0] = (uint32_t)(z == 0 ? a.nz - 1 : z - 1) * pl;
        p.z[2] = (uint32_t)(z == a.nz - 1 ? 0 : z + 1) * pl;
    }
    p.z[1] = (uint32_t)z * pl;
    p.self = p.z[1] + p.y[1] + (uint32_t)x;
    return p;
}

// Index of the stored entry that population i of the node is pulled from.
template <bool WALLS, class Geo>
__device__ __forceinline__ size_t pull_index(const Geo &a, const PullAt &p, int i)
{
    const uint32_t off = p.z[1 - lbd::cz(i)] + p.y[1 - lbd::cy(i)] + (uint32_t)p.x[1 - lbd::cx(i)];
    const bool bounce = WALLS && ((lbd::cz(i) == 1 && p.lo) || (lbd::cz(i) == -1 && p.hi));
    return WALLS && bounce ? (size_t)lbd::opposite(i) * a.pitch + p.self : (size_t)i * a.pitch + off;
}

// Population i as pulled by the node (stored value, FP16 / BF16 still scaled).
template <int DT, bool WALLS>
__device__ __forceinline__ float pull_one(const typename lbd::Store<DT>::T *__restrict__ src, const StepArgs &a,
                                          const PullAt &p, int i)
{
    const size_t k = pull_index<WALLS>(a, p, i);
    return in_bounds(k, 19 * a.pitch, a.err) ? lbd::Store<DT>::load(src + k, 1.0f) : 0.0f;
}

// Node s + 1 of a located pair; the located node itself where there is only one.
template <class Geo>
__device__ __forceinline__ void second_node(const Geo &a, const PairAt &at, int &xb, int &yb, int &zb)
{
    xb = at.x;
    yb = at.y;
    zb = at.z;
    if (!(at.va && at.vb)) return;
    if (++xb < a.nx) return;
    xb = 0;
    if (++yb < a.ny) return;
    yb = 0;
    zb += 1;
}

template <int DT, bool FIELD, bool WALLS>
__device__ __forceinline__ void load_pair_any(const typename lbd::Store<DT>::T *__restrict__ src,
                                              const float *__restrict__ ffield, float *facc,
                                              const StepArgs &a, const PairAt &at, lbp::F2 n[19], float f0[3],
                                              float f1[3], bool take = true)
{
    int xb, yb, zb;
    second_node(a, at, xb, yb, zb);
    const PullAt pa = pull_at<WALLS>(a, at.x, at.y, at.z), pb = pull_at<WALLS>(a, xb, yb, zb);
    if (WALLS && (pa.lo || pa.hi || pb.lo || pb.hi)) {  // next to a wall (load_pair)
        if (FIELD && facc && a.consume && take) {
            clear_solid(facc, a, at.z, pa.self);
            clear_solid(facc, a, zb, pb.self);
        }
#pragma unroll
        for (int i = 0; i < 19; ++i)
            n[i] = lbp::f2(pull_one<DT, true>(src, a, pa, i), pull_one<DT, true>(src, a, pb, i));
    } else {
#pragma unroll
        for (int i = 0; i < 19; ++i)
            n[i] = lbp::f2(pull_one<DT, false>(src, a, pa, i), pull_one<DT, false>(src, a, pb, i));
    }
    if (DT != 0) {
#pragma unroll
        for (int i = 0; i < 19; ++i) n[i] = n[i] * lbp::f2s(a.inv_scale);
    }
    f0[0] = f1[0] = a.fx;
    f0[1] = f1[1] = a.fy;
    f0[2] = f1[2] = a.fz;
    if (FIELD) {
        unsigned int bits = 0u;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (ffield) {  // caller's field, component stride N
                f0[d] += ld_f32(ffield + d * a.nn + pa.self);
                f1[d] += ld_f32(ffield + d * a.nn + pb.self);
            }
            if (facc) {  // library accumulator, component stride = plane pitch
                const float u = ld_f32(facc + d * a.pitch + pa.self), v = ld_f32(facc + d * a.pitch + pb.self);
                f0[d] += u;
                f1[d] += v;
                bits |= __float_as_uint(u) | __float_as_uint(v);
            }
        }
        if (bits && a.consume && take) {
#pragma unroll
            for (int d = 0; d < 3; ++d) facc[d * a.pitch + pa.self] = facc[d * a.pitch + pb.self] = 0.0f;
        }
    }
}

// The store of one node of the pair.
template <int DT>
__device__ __forceinline__ void store_one(typename lbd::Store<DT>::T *__restrict__ dst, const StepArgs &a, uint32_t s,
                                          const lbp::F2 out[19], bool second)
{
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        const float o = second ? lbp::hi(out[i]) : lbp::lo(out[i]);
        const size_t k = (size_t)i * a.pitch + s;
        if (in_bounds(k, 19 * a.pitch, a.err)) dst[k] = lbd::Store<DT>::pack(o, a.scale);
    }
}

// The pair's store, node by node where only one is fluid (va or vb false) or
// the buffer does not start on a pair.
template <int DT>
__device__ __forceinline__ void store_pair_any(typename lbd::Store<DT>::T *__restrict__ dst, const StepArgs &a,
                                               const PairAt &at, const lbp::F2 out[19])
{
    if (at.va && at.vb && ((uintptr_t)dst & (2 * sizeof(*dst) - 1)) == 0) {
        store_pair<DT>(dst, a, at.s, out);
        return;
    }
    if (at.va) store_one<DT>(dst, a, at.s, out, false);
    if (at.vb) store_one<DT>(dst, a, at.s + 1u, out, true);
}

template <int DT, bool FIELD, bool WALLS, bool ODD>
__device__ __forceinline__ void load_linear(const typename lbd::Store<DT>::T *__restrict__ src,
                                            const float *__restrict__ ffield, float *facc,
                                            const StepArgs &a, const PairAt &at, lbp::F2 n[19], float f0[3],
                                            float f1[3])
{
    if (ODD)
        load_pair_any<DT, FIELD, WALLS>(src, ffield, facc, a, at, n, f0, f1);
    else
        load_pair<DT, FIELD, WALLS>(src, ffield, facc, a, at.x, at.y, at.z, n, f0, f1);
}

template <int DT, bool NOISE, bool FIELD, bool WALLS, bool ODD>
__device__ __forceinline__ void linear_update(const typename lbd::Store<DT>::T *__restrict__ src,
                                              typename lbd::Store<DT>::T *__restrict__ dst,
                                              const float *__restrict__ ffield, float *facc, const StepArgs &a)
{
    PairAt at;
    const bool mine = locate_pair<WALLS>(a, at);
    wait_for_previous();
    if (!mine) return;
    lbp::F2 n[19], m[19], out[19];
    float f0[3], f1[3];
    load_linear<DT, FIELD, WALLS, ODD>(src, ffield, facc, a, at, n, f0, f1);
    lbp::forward2(n, m);
    lbp::collide_moments2<NOISE>(m, lbp::f2(f0[0], f1[0]), lbp::f2(f0[1], f1[1]), lbp::f2(f0[2], f1[2]), a, a.rk, at.s,
                                 a.replica, out);
    if (ODD)
        store_pair_any<DT>(dst, a, at, out);
    else
        store_pair<DT>(dst, a, at.s, out);
}

template <int DT, bool NOISE, bool FIELD, bool WALLS, bool ODD>
__global__ void __launch_bounds__(kLinBX)
    k_stream_collide_linear(const typename lbd::Store<DT>::T *__restrict__ src,
                            typename lbd::Store<DT>::T *__restrict__ dst, const float *__restrict__ ffield, float *facc,
                            const StepArgs a)
{
    linear_update<DT, NOISE, FIELD, WALLS, ODD>(src, dst, ffield, facc, a);
}

// With a force field (k_stream_collide2_field); rows of odd length spill too
// much for that and leave the count open (257 x 131 x 129 FP32 between walls
// with a field 119 us a step, 133 us with room for seven blocks).
template <int DT, bool NOISE, bool WALLS, bool ODD>
__global__ void __launch_bounds__(kLinBX, ODD ? 0 : field_blocks<DT>() * kBX / kLinBX)
    k_stream_collide_linear_field(const typename lbd::Store<DT>::T *__restrict__ src,
                                  typename lbd::Store<DT>::T *__restrict__ dst, const float *__restrict__ ffield,
                                  float *facc, const StepArgs a)
{
    linear_update<DT, NOISE, true, WALLS, ODD>(src, dst, ffield, facc, a);
}

// The step's kernel of either mapping.
template <int DT, bool NOISE, bool FIELD, bool WALLS>
auto rows_kernel()
{
    if constexpr (FIELD) return k_stream_collide2_field<DT, NOISE, WALLS>;
    else return k_stream_collide2<DT, NOISE, false, WALLS, false>;
}
template <int DT, bool NOISE, bool FIELD, bool WALLS, bool ODD>
auto linear_kernel()
{
    if constexpr (FIELD) return k_stream_collide_linear_field<DT, NOISE, WALLS, ODD>;
    else return k_stream_collide_linear<DT, NOISE, false, WALLS, ODD>;
}

// The step with moment sums on boxes whose pairs cannot move as one access
// (rows of odd length, or more elements than 32-bit indices reach): pairs over
// the linear index as in the ODD form of k_stream_collide_linear, whose
// arithmetic and so whose populations these are bit for bit.  3 x 200 x 200
// takes 15 us and 65^3 19 us a step; with a row to a block, which leaves most
// of it idle, 199 and 34 us, and one node a thread 126 and 29 us.
template <int DT, bool NOISE, bool FIELD, bool WALLS>
__global__ void __launch_bounds__(kBX) k_stream_collide_sums_any(const typename lbd::Store<DT>::T *__restrict__ src,
                                                                 typename lbd::Store<DT>::T *__restrict__ dst,
                                                                 const float *__restrict__ ffield,
                                                                 float *facc, const StepArgs a, float *partials)
{
    __shared__ float part[kBX / 32][38];
    PairAt at;
    const bool mine = locate_pair<WALLS, kBX>(a, at);
    if (!mine) {  // lanes past the last pair load the first fluid node and store nothing
        at.s = 0u;
        at.x = at.y = 0;
        at.z = a.z0;
        at.va = at.vb = false;
    }
    wait_for_previous();
    lbp::F2 n[19], m[19], out[19];
    float f0[3], f1[3];
    load_pair_any<DT, FIELD, WALLS>(src, ffield, facc, a, at, n, f0, f1, mine);
    lbp::forward2(n, m);
    float m0[19], m1[19];
#pragma unroll
    for (int k = 0; k < 19; ++k) {
        lbp::split(m[k], m0[k], m1[k]);
        if (!at.va) m0[k] = 0.0f;
        if (!at.vb) m1[k] = 0.0f;
    }
    warp_moment_sums(m0, m1, mine, part);
    if (mine) {
        lbp::collide_moments2<NOISE>(m, lbp::f2(f0[0], f1[0]), lbp::f2(f0[1], f1[1]), lbp::f2(f0[2], f1[2]), a, a.rk,
                                     at.s, a.replica, out);
        store_pair_any<DT>(dst, a, at, out);
    }
    block_moment_sums_out(part, partials + 38 * block_linear());
}

// Launch geometry of the stream-collide kernels: two nodes per thread when
// rows pair up and element indices fit 32 bits.
inline bool sc_paired(const lb_handle *h)
{
    return (h->p.nx % 2 == 0) && (19.0 * (double)h->pitch < 4294967296.0);
}

// A caller's buffer may start at any element; pairs that move as one access
// need an address that is a multiple of the pair.
inline bool pair_aligned(const void *p, size_t bytes) { return ((uintptr_t)p & (bytes - 1)) == 0; }

inline dim3 sc_grid(const lb_handle *h)
{
    const int nzf = h->p.walls ? h->p.nz - 2 : h->p.nz;
    return dim3(((h->p.nx + 1) / 2 + kBX - 1) / kBX, h->p.ny, nzf);
}

// Grid of the launch with moment sums (a row of partial sums a block).
inline dim3 sums_grid(const lb_handle *h)
{
    return sc_paired(h) ? sc_grid(h) : linear_grid(h->n_nodes, (size_t)h->p.nx * h->p.ny, h->p.walls != 0, kBX);
}

// partials != NULL: the launch also writes per-block moment sums
// (partials[block][38], block = blockIdx.x + gridDim.x (blockIdx.y + gridDim.y blockIdx.z)),
// and src, dst are the handle's own buffers (256-byte aligned, so sc_paired decides).
template <int DT>
cudaError_t launch_stream_collide_dt(const lb_handle *h, const void *src, void *dst, float *facc,
                                     float *partials)
{
    using T = typename lbd::Store<DT>::T;
    StepArgs a = make_args(h);
    a.forced |= facc != nullptr;
    a.consume = facc && facc == h->facc;  // (the reverse pass keeps its impulse buffers)
    const dim3 grid = sc_grid(h);
    const dim3 block(kBX);
    const bool noise = a.kT > 0.0f;
    const bool field = (h->force != nullptr) || (facc != nullptr);
    const bool walls = h->p.walls != 0;
    const bool aligned = pair_aligned(src, 2 * sizeof(T)) && pair_aligned(dst, 2 * sizeof(T)) && pair_aligned(facc, 8);
    const bool paired = sc_paired(h) && aligned;
    const T *s = static_cast<const T *>(src);
    T *d = static_cast<T *>(dst);
    const bool rows = !partials && paired && (h->p.nx / 2) % kBX == 0;
    const bool odd = !paired;
    const dim3 linear = linear_grid(a);
#define LBI_SC(NZ, FL, WL)                                                                                        \
    (partials ? (sc_paired(h)                                                                                     \
                     ? launch_chained(k_stream_collide2<DT, NZ, FL, WL, true>, grid, block, h->stream, s, d,        \
                                      h->force, facc, a, partials)                                                \
                     : launch_chained(k_stream_collide_sums_any<DT, NZ, FL, WL>, sums_grid(h), block, h->stream, s, \
                                      d, h->force, facc, a, partials))                                            \
     : rows   ? launch_chained(rows_kernel<DT, NZ, FL, WL>(), grid, block, h->stream, s, d, h->force,    \
                               facc, a, nullptr)                                                                  \
     : odd    ? launch_chained(linear_kernel<DT, NZ, FL, WL, true>(), linear, dim3(kLinBX), h->stream, s, d, \
                               h->force, facc, a)                                                                 \
              : launch_chained(linear_kernel<DT, NZ, FL, WL, false>(), linear, dim3(kLinBX), h->stream, s,  \
                               d, h->force, facc, a))
    if (noise) {
        if (field) return walls ? LBI_SC(true, true, true) : LBI_SC(true, true, false);
        return walls ? LBI_SC(true, false, true) : LBI_SC(true, false, false);
    }
    if (field) return walls ? LBI_SC(false, true, true) : LBI_SC(false, true, false);
    return walls ? LBI_SC(false, false, true) : LBI_SC(false, false, false);
#undef LBI_SC
}

template <int DT>
cudaError_t launch_patch_dt(const lb_handle *h, const void *src, void *dst, float *facc, const int *records,
                            int n, int nsub, int span, unsigned int *claim, unsigned int tag)
{
    using T = typename lbd::Store<DT>::T;
    StepArgs a = make_args(h);
    a.forced = 1;
    if (n <= 0 || nsub <= 0) return cudaSuccess;
    const unsigned int blocks = (unsigned int)(((size_t)n * 8 + kBX - 1) / kBX);
    const T *s = static_cast<const T *>(src);
    T *d = static_cast<T *>(dst);
    const bool noise = a.kT > 0.0f, walls = h->p.walls != 0;
    if (DT == 0) {  // FP32: correct the stored result in place
        float *d32 = reinterpret_cast<float *>(dst);
        return walls ? launch_chained(k_patch_impulse_nodes_f32<true>, blocks, kBX, h->stream, d32, h->force, facc,
                                      records, n, nsub, span, claim, tag, a)
                     : launch_chained(k_patch_impulse_nodes_f32<false>, blocks, kBX, h->stream, d32, h->force, facc,
                                      records, n, nsub, span, claim, tag, a);
    }
#define LBI_PATCH(NZ, WL)                                                                                             \
    launch_chained(k_patch_impulse_nodes<DT, NZ, WL>, blocks, kBX, h->stream, s, d, h->force, facc, records, n, nsub,   \
                   span, claim, tag, a)
    if (noise) return walls ? LBI_PATCH(true, true) : LBI_PATCH(true, false);
    return walls ? LBI_PATCH(false, true) : LBI_PATCH(false, false);
#undef LBI_PATCH
}

}  // namespace lbi
