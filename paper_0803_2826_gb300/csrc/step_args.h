// step_args.h -- the constants every update kernel receives by value (a
// kernel's view of the handle: geometry, relaxation, noise and force).
#pragma once

#include <cstddef>
#include <cstdint>

#include "d3q19.cuh"
#include "lbfluct.h"

namespace lbi {

// Unsigned division by a run-time constant (round-up method of Granlund and
// Montgomery, "Division by invariant integers using multiplication", 1994).
struct Div {
    uint32_t m, s, d;  // d <= 1: identity
};

inline Div make_div(uint32_t d)
{
    Div v{0, 0, d};
    if (d <= 1) return v;
    uint32_t l = 0;
    while ((1ull << l) < d) ++l;
    v.m = (uint32_t)((((1ull << l) - d) << 32) / d + 1);
    v.s = l - 1;
    return v;
}

__device__ __forceinline__ uint32_t divide(uint32_t n, const Div &v)
{
    if (v.d <= 1) return n;
    const uint32_t t = __umulhi(v.m, n);
    return (t + ((n - t) >> 1)) >> v.s;
}

// Geometry and physics constants a kernel launch needs, in FP32 where the
// kernels compute in FP32.
struct StepArgs {
    int nx, ny, nz;
    int z0, z1;            // fluid z-range [z0, z1)
    size_t pitch;          // elements per population plane
    size_t nn;             // nodes nx*ny*nz (component stride of caller fields)
    Div dnx, dny;          // division by nx and ny (node index -> coordinates)
    float rho0;
    float kT;
    float mu;              // kT / c_s^2
    float g_shear, g_bulk, g_odd, g_even;
    float phi_shear, phi_bulk, phi_odd, phi_even;  // sqrt(1 - gamma^2)
    float amp[15];         // noise of mode k = 4..18 per unit sqrt(mu rho): phi_k / sqrt(w_k)
    float rel[9];          // gamma_k / w_k of mode k = 10..18
    float frc[3];          // 1 + gamma_bulk, 1 + gamma_shear, half of that
    float reserved[3];     // 0 (keeps the members below where they are read in fours)
    float fx, fy, fz;      // uniform body force
    int forced;            // a body force, a force field or particle impulses act
    float scale, inv_scale;  // storage scale of FP16/BF16 deviations
    int noise_rho0;
    uint32_t key0, key1;   // Philox key (seed)
    uint32_t replica;
    uint32_t step;
    lbd::RoundKeys rk;     // Philox round keys of (key0, key1)
    unsigned int *err;     // device error word (index checks of LB_DEBUG_BOUNDS builds)
    // (last: one word before the noise constants shifts the pairs they are read
    // in, and the 256^3 FP32 update goes from 72 registers and 365 us to 76 and 376)
    int consume;           // the impulses read are applied for good: clear them
};
static_assert(offsetof(StepArgs, amp) % 8 == 4 && offsetof(StepArgs, rk) % 16 == 0,
              "the noise constants or the round keys moved against the groups they are read in");

// Index checks of a library built with -DLB_DEBUG_BOUNDS: the element index i
// of an access to an array of n elements is tested first; outside, the error
// word gets LB_DERR_BOUNDS and the caller skips the access.  In ordinary
// builds the test is the constant true and costs nothing.
#ifdef LB_DEBUG_BOUNDS
__device__ __forceinline__ bool in_bounds(size_t i, size_t n, unsigned int *err)
{
    if (i < n) return true;
    if (err) atomicOr(err, LB_DERR_BOUNDS);
    return false;
}
#else
__device__ __forceinline__ constexpr bool in_bounds(size_t, size_t, unsigned int *) { return true; }
#endif

}  // namespace lbi
