// Per-vertex bodies of the damped steps between plates and of their adjoint,
// and the per-cell moduli gradient: shared by the general path
// (csrc/adjoint.cu) and the on-chip one (csrc/relax.cu).
#pragma once

#include "mr.cuh"

namespace cf {

struct PlateZ {
    float lo, hi;  // plate heights relative to the cell's integer origin
};

__device__ __forceinline__ PlateZ plates_of(const MeshView &m, int c, const float *zlo, const float *zhi) {
    const float oz = (float)__ldg(m.origin + 3 * c + 2);
    return {__ldg(zlo + c) - oz, __ldg(zhi + c) - oz};
}

// v <- c v + dt (f_el + f_plate), y <- y + dt v of a vertex at displacement uu,
// velocity vv, with elastic force f and reference height zr; the roundings
// written out, so that every path takes the same step bit for bit.
__device__ __forceinline__ void plate_move(float4 uu, float4 vv, float4 f, float zr, PlateZ pz, float dt, float c,
                                           float kp, float4 &un, float4 &vn) {
    const float z = __fadd_rn(zr, uu.z);
    const float fz = __fmaf_rn(-kp, fmaxf(z - pz.hi, 0.f), __fmaf_rn(kp, fmaxf(pz.lo - z, 0.f), f.z));
    vn = make_float4(__fmaf_rn(c, vv.x, __fmul_rn(dt, f.x)), __fmaf_rn(c, vv.y, __fmul_rn(dt, f.y)),
                     __fmaf_rn(c, vv.z, __fmul_rn(dt, fz)), 0.f);
    un = make_float4(__fmaf_rn(dt, vn.x, uu.x), __fmaf_rn(dt, vn.y, uu.y), __fmaf_rn(dt, vn.z, uu.z), 0.f);
}

// lambda_y <- lambda_y + dt (J_el m + J_plate m), lambda_v <- c m of a vertex at
// height z, with J_el m = j and J_plate = diag(0, 0, -kp) in a plate; mn = m of
// the step before.
__device__ __forceinline__ void adjoint_move(float4 l, float4 j, float4 m, float z, PlateZ pz, float dt, float c,
                                             float kp, float4 &a, float4 &b, float4 &mn) {
    const float jz = (z < pz.lo || z > pz.hi) ? -kp * m.z : 0.f;
    a = make_float4(l.x + dt * j.x, l.y + dt * j.y, l.z + dt * (j.z + jz), 0.f);
    b = make_float4(c * m.x, c * m.y, c * m.z, 0.f);
    mn = make_float4(fmaf(dt, a.x, b.x), fmaf(dt, a.y, b.y), fmaf(dt, a.z, b.z), 0.f);
}

// From the sums G = lambda . df/d(mu1, mu2, kappa) of a cell, with
// mu1 = w mu and mu2 = (1 - w) mu: add its derivative with respect to mu
// (k = 0), w (k = 1) or kappa (k = 2), times scale, to grad[0], grad[2] or
// grad[1].
__device__ __forceinline__ void add_moduli_rate(int k, double G0, double G1, double Gk, float4 mat, double scale,
                                                double *grad) {
    const double mu = (double)mat.x + (double)mat.y, w = (double)mat.w;
    const double d = scale * (k == 0 ? w * G0 + (1.0 - w) * G1 : k == 1 ? mu * (G0 - G1) : Gk);
    atomicAdd(grad + (k == 0 ? 0 : k == 1 ? 2 : 1), d);
}

}  // namespace cf
