// Compression between plates and its adjoint (differentiation of the elastic
// forces with respect to positions and to the moduli).
//
// The paper compresses a cell between a resting plate and a moving one, with
// a repulsive force keeping vertices out of the plates (Sec. 4.2; the form of
// that force is in the supplement): here a one-sided harmonic penalty per
// vertex, f_z = k (z_lo - z)_+ - k (z - z_hi)_+, and quasi-static relaxation
// by damped steps of unit-mass vertices,
//   v <- c v + dt (f_el(y) + f_plate(y)),  y <- y + dt v   (0 <= c < 1;
// c = 0 is the first-order gradient flow y <- y + dt^2 f). The measured force
// is the top plate's, F = sum_v k (z_v - z_hi)_+.
//
// Adjoint of one step with (lambda_y, lambda_v) = dL/d(y, v) after it and
// m = dt lambda_y + lambda_v (the sensitivity to the new velocity):
//   lambda_y <- lambda_y + dt (J_el + J_plate) m,  lambda_v <- c m,
//   dL/dtheta += dt m . df/dtheta.
// J_el = -Hessian of the elastic energy is symmetric, so J_el m is the
// directional derivative of the forces along m: k_tet_jvp evaluates the stress
// on dual numbers (mr_stress in mr.cuh, the expressions of the force kernels'
// mr_stress_inv in fused multiply-adds; the two are separate sources). The
// forces are linear in (mu_1, mu_2, kappa), so m . df/d(mu, kappa, w) comes from
// the rates of the unit-modulus energies along m (mr_energy_rates): FP32 per
// tet, as the stress, summed as float pairs of about 48 bits over a warp (on
// chip, over a thread's tets and steps and the block), FP64 from there.
#include "plate_ops.cuh"

namespace cf {

// ---------------------------------------------------------------- parameters
// Sum of `val` over the lanes of a warp that share cell c, added into
// dst[stride * c] once per warp when the whole warp has one cell (elements
// of a cell are contiguous, so that is the common case). Every lane calls;
// c < 0 marks lanes without an element.
__device__ __forceinline__ void warp_cell_add(int c, double val, double *dst, int stride) {
    const unsigned full = 0xffffffffu;
    const int c0 = __shfl_sync(full, c, 0);
    if (__all_sync(full, c == c0)) {
        for (int o = 16; o > 0; o >>= 1) val += __shfl_xor_sync(full, val, o);
        if ((threadIdx.x & 31) == 0 && c >= 0) atomicAdd(dst + stride * c, val);
    } else if (c >= 0) {
        atomicAdd(dst + stride * c, val);
    }
}

// Add one tet per thread, g = lambda . df/d(mu1, mu2, kappa) of cell c (c < 0:
// none), times 2^(127 - b) (see direction_exponent), to its cell's gradient.
// Every thread of the block calls. Where the block has one cell (the common
// case: a cell's tets are contiguous) the lanes of a warp are summed as float
// pairs (Sum2), on the warp's largest b, and one thread goes on in FP64: one
// addition per warp to a single cell's three sums took 35 us for 201 k tets
// (6 k additions to the same address).
constexpr int kVjpBlock = 128;

__device__ __forceinline__ void block_add_moduli(const MeshView &m, int c, const float (&g)[3], int b, double scale,
                                                 double *grad) {
    constexpr int kWarps = kVjpBlock / 32;
    __shared__ Sum2 part[3][kWarps];
    __shared__ int exponent[kWarps], c0;
    if (threadIdx.x == 0) c0 = c;  // the block's first tet: no later one has an element if it has none
    __syncthreads();
    if (__syncthreads_and(c == c0 || c < 0)) {
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        const int top = __reduce_max_sync(0xffffffffu, c < 0 ? 1 : b), less = 127 + b - top;
        const float f = less > 0 ? power_of_two(less) : 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            Sum2 a;
            a.hi = c < 0 ? 0.f : f * g[k];
            warp_sum(a);
            if (lane == 0) part[k][w] = a;
        }
        if (lane == 0) exponent[w] = top;
        __syncthreads();
        if (threadIdx.x >= 32 || c0 < 0) return;
        double G = 0.0;  // lane k: sum k over the warps
        if (lane < 3)
            for (int q = 0; q < kWarps; ++q) G += part[lane][q].value() * power_of_two_64(exponent[q]);
        const double G0 = __shfl_sync(0xffffffffu, G, 0), G1 = __shfl_sync(0xffffffffu, G, 1);
        if (lane < 3) add_moduli_rate(lane, G0, G1, G, __ldg(m.mat + c0), scale, grad + 3 * c0);
    } else if (c >= 0) {
        const float4 mat = __ldg(m.mat + c);
        const double s = scale * power_of_two_64(b);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            add_moduli_rate(k, (double)g[0], (double)g[1], (double)g[2], mat, s, grad + 3 * c);
    }
}

// Gradient dH of a direction on tet a4, times 2^(127 - b); returns b.
__device__ __forceinline__ int scaled_grad(const float4 *__restrict__ v, int4 a4, const float (&Bm)[3][3],
                                           float (&dH)[3][3]) {
    const float4 l0 = __ldg(v + a4.x), l1 = __ldg(v + a4.y), l2 = __ldg(v + a4.z), l3 = __ldg(v + a4.w);
    const int b = direction_exponent(largest(l0, largest(l1, largest(l2, largest(l3, 0.f)))));
    const float f = power_of_two(254 - b);
    tet_grad(times(l0, f), times(l1, f), times(l2, f), times(l3, f), Bm, dH);
    return b;
}

// lambda . df/d(mu, kappa, w) per cell, times `scale`, added into grad[3 c + .]:
// the rates of the unit-modulus energies along lambda's gradient
// (mr_energy_rates). Three stresses and 36 FP64 products per tet in its place
// were bound by FP64: 201 k tets 52 us, now 10.9 (9.7 without the
// directions' scaling); 20 k tets 12.0 us, now 7.0.
__global__ void __launch_bounds__(kVjpBlock) k_param_vjp(MeshView m, const float4 *__restrict__ u,
                                                   const float4 *__restrict__ lam, double scale, double *grad) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    int c = -1, b = 1;
    float g[3] = {0.f, 0.f, 0.f};
    if (t < m.T) {
        const int4 a4 = __ldg(m.tet + t);
        float Bm[3][3];
        load_B(m, t, Bm);
        float H[3][3], dH[3][3];
        tet_grad(__ldg(u + a4.x), __ldg(u + a4.y), __ldg(u + a4.z), __ldg(u + a4.w), Bm, H);
        b = scaled_grad(lam, a4, Bm, dH);
        InvT<float> inv;
        invariants_t(H, inv);
        mr_energy_rates(H, dH, inv, g);
        const float V0 = __ldg(m.V0 + t);
#pragma unroll
        for (int k = 0; k < 3; ++k) g[k] *= -V0;
        c = __ldg(m.tcell + t);
    }
    block_add_moduli(m, c, g, b, scale, grad);
}

cudaError_t launch_param_vjp(const MeshView &m, const float4 *u, const float4 *lam, double scale, double *grad,
                             cudaStream_t s) {
    if (m.T == 0) return cudaSuccess;
    k_param_vjp<<<(m.T + kVjpBlock - 1) / kVjpBlock, kVjpBlock, 0, s>>>(m, u, lam, scale, grad);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- JVP
// Corner tangents d f / d eps of f(u + eps v) into m.fc. GRAD: the same
// evaluation also adds v . df/d(mu, kappa, w), times `scale`, to grad: the
// reverse step needs both along the same direction (528 k tets: 31 us, where
// two launches took 20 + 126 us). Bound by its ~900 FP32 operations a tet;
// held to 72 registers (20 bytes of spills): a recomputed and reversed step of
// 872 k tets 111 us, 115 at 80 registers and 121 at the 96 it would take.
template <bool GRAD>
__global__ void __launch_bounds__(GRAD ? kVjpBlock : 128, GRAD ? 7 : 0) k_tet_jvp(MeshView m, const float4 *__restrict__ u,
                                                 const float4 *__restrict__ v, double scale, double *grad) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (!GRAD && t >= m.T) return;
    int c = -1, b = 1;
    float g[3] = {0.f, 0.f, 0.f};
    if (t < m.T) {
        const int4 a4 = __ldg(m.tet + t);
        float Bm[3][3];
        load_B(m, t, Bm);
        float H[3][3], dH[3][3];
        tet_grad(__ldg(u + a4.x), __ldg(u + a4.y), __ldg(u + a4.z), __ldg(u + a4.w), Bm, H);
        if (GRAD)
            b = scaled_grad(v, a4, Bm, dH);
        else
            tet_grad(__ldg(v + a4.x), __ldg(v + a4.y), __ldg(v + a4.z), __ldg(v + a4.w), Bm, dH);
        const float4 mat = __ldg(m.mat + mat_slot(m, t));
        const float V0 = __ldg(m.V0 + t);
        float f[4][3];
        InvT<float> inv;
        tet_tangent(H, dH, mat, Bm, V0, inv, f);
        if (GRAD) {
            mr_energy_rates(H, dH, inv, g);
#pragma unroll
            for (int k = 0; k < 3; ++k) g[k] *= -V0;
            c = __ldg(m.tcell + t);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const float4 fa = make_float4(f[a][0], f[a][1], f[a][2], 0.f);
            m.fc[a * m.T + t] = GRAD ? times(fa, power_of_two(b)) : fa;
        }
    }
    if (GRAD) block_add_moduli(m, c, g, b, scale, grad);
}

cudaError_t launch_force_jvp(const MeshView &m, const float4 *u, const float4 *v, float4 *out, unsigned *err,
                             cudaStream_t s, double scale, double *grad) {
    if (m.T == 0) return cudaSuccess;
    if (grad)
        k_tet_jvp<true><<<(m.T + kVjpBlock - 1) / kVjpBlock, kVjpBlock, 0, s>>>(m, u, v, scale, grad);
    else
        k_tet_jvp<false><<<(m.T + 127) / 128, 128, 0, s>>>(m, u, v, 0.0, nullptr);
    MeshView g = m;
    g.fv = out;
    return launch_gather_spread(g, u, nullptr, nullptr, err, s);
}

// ---------------------------------------------------------------- plates
// v <- c v + dt (f_el + f_plate), y <- y + dt v from (u_in, v_in) into
// (u_out, v_out); outputs may alias inputs.
__global__ void k_plate_step(MeshView m, const float4 *u_in, const float4 *v_in, const float4 *__restrict__ fel,
                             float4 *u_out, float4 *v_out, float dt, float c, float kp, const float *__restrict__ zlo,
                             const float *__restrict__ zhi, unsigned *err) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= m.V) return;
    const float4 xr = __ldg(m.xr + v);
    const PlateZ pz = plates_of(m, __float_as_int(xr.w), zlo, zhi);
    float4 un, vn;
    plate_move(u_in[v], v_in[v], fel[v], xr.z, pz, dt, c, kp, un, vn);
    if (!isfinite(un.x + un.y + un.z)) atomicOr(err, ERR_NONFINITE);
    u_out[v] = un;
    v_out[v] = vn;
}

cudaError_t launch_plate_step(const MeshView &m, const float4 *u_in, const float4 *v_in, const float4 *fel,
                              float4 *u_out, float4 *v_out, float dt, float c, float kp, const float *zlo,
                              const float *zhi, unsigned *err, cudaStream_t s) {
    if (m.V == 0) return cudaSuccess;
    k_plate_step<<<(m.V + 255) / 256, 256, 0, s>>>(m, u_in, v_in, fel, u_out, v_out, dt, c, kp, zlo, zhi, err);
    return cudaGetLastError();
}

// F_c = sum over the cell's vertices of k (z - z_hi)_+ (added into out[c]).
__global__ void k_plate_force(MeshView m, const float4 *__restrict__ u, float kp, const float *__restrict__ zlo,
                              const float *__restrict__ zhi, double *out) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    int c = -1;
    double f = 0.0;
    if (v < m.V) {
        const float4 xr = __ldg(m.xr + v);
        c = __float_as_int(xr.w);
        const PlateZ pz = plates_of(m, c, zlo, zhi);
        f = (double)kp * (double)fmaxf(xr.z + __ldg(u + v).z - pz.hi, 0.f);
    }
    warp_cell_add(c, f, out, 1);
}

cudaError_t launch_plate_force(const MeshView &m, const float4 *u, float kp, const float *zlo, const float *zhi,
                               double *out, cudaStream_t s) {
    if (m.V == 0) return cudaSuccess;
    k_plate_force<<<(m.V + 255) / 256, 256, 0, s>>>(m, u, kp, zlo, zhi, out);
    return cudaGetLastError();
}

// lambda_z += dL/dF_c * dF_c/dz_v = dF[c] k [z_v > z_hi].
__global__ void k_adj_seed(MeshView m, const float4 *__restrict__ u, float kp, const float *__restrict__ zlo,
                           const float *__restrict__ zhi, const double *__restrict__ dF, float4 *lam) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= m.V) return;
    const float4 xr = __ldg(m.xr + v);
    const int c = __float_as_int(xr.w);
    const PlateZ pz = plates_of(m, c, zlo, zhi);
    if (xr.z + __ldg(u + v).z > pz.hi) lam[v].z += (float)(__ldg(dF + c) * (double)kp);
}

// m = dt lambda_y + lambda_v
__global__ void k_adj_m(int n, const float4 *__restrict__ ly, const float4 *__restrict__ lv, float dt, float4 *mvec) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const float4 a = __ldg(ly + v), b = __ldg(lv + v);
    mvec[v] = make_float4(fmaf(dt, a.x, b.x), fmaf(dt, a.y, b.y), fmaf(dt, a.z, b.z), 0.f);
}

// lambda_y <- lambda_y + dt (J_el m + J_plate m), lambda_v <- c m at positions
// u, and m = dt lambda_y + lambda_v of the step before, with J_el m given (jv) and J_plate = diag(0, 0, -k) on penetrating
// vertices.
__global__ void k_adj_step(MeshView m, const float4 *__restrict__ u, const float4 *__restrict__ jv,
                           float4 *mvec, float4 *ly, float4 *lv, float dt, float c, float kp,
                           const float *__restrict__ zlo, const float *__restrict__ zhi) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= m.V) return;
    const float4 xr = __ldg(m.xr + v);
    const PlateZ pz = plates_of(m, __float_as_int(xr.w), zlo, zhi);
    const float z = xr.z + __ldg(u + v).z;
    float4 a, b, mn;
    adjoint_move(ly[v], __ldg(jv + v), mvec[v], z, pz, dt, c, kp, a, b, mn);
    ly[v] = a;
    lv[v] = b;
    mvec[v] = mn;
}

cudaError_t launch_adj_seed(const MeshView &m, const float4 *u, float kp, const float *zlo, const float *zhi,
                            const double *dF, float4 *lam, cudaStream_t s) {
    if (m.V == 0) return cudaSuccess;
    k_adj_seed<<<(m.V + 255) / 256, 256, 0, s>>>(m, u, kp, zlo, zhi, dF, lam);
    return cudaGetLastError();
}

cudaError_t launch_adj_m(int n, const float4 *ly, const float4 *lv, float dt, float4 *mvec, cudaStream_t s) {
    if (n > 0) k_adj_m<<<(n + 255) / 256, 256, 0, s>>>(n, ly, lv, dt, mvec);
    return cudaGetLastError();
}

cudaError_t launch_adj_step(const MeshView &m, const float4 *u, const float4 *jv, float4 *mvec, float4 *ly,
                            float4 *lv, float dt, float c, float kp, const float *zlo, const float *zhi,
                            cudaStream_t s) {
    if (m.V == 0) return cudaSuccess;
    k_adj_step<<<(m.V + 255) / 256, 256, 0, s>>>(m, u, jv, mvec, ly, lv, dt, c, kp, zlo, zhi);
    return cudaGetLastError();
}

// double [n][3] (host layout) -> float4 [n]
__global__ void k_pack3(const double *__restrict__ in, int n, float4 *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = make_float4((float)in[3 * i], (float)in[3 * i + 1], (float)in[3 * i + 2], 0.f);
}

cudaError_t launch_pack3(const double *in, int n, float4 *out, cudaStream_t s) {
    if (n > 0) k_pack3<<<(n + 255) / 256, 256, 0, s>>>(in, n, out);
    return cudaGetLastError();
}

}  // namespace cf
