// Mooney-Rivlin first Piola stress P = dU/dF of one tet (Sec. 2, Sec. 3.1-3.2):
// in FP32 for the force kernels, and on dual numbers (value and directional
// derivative), which the adjoint uses for Hessian-vector products.
//
// With H = A B (F = I + H), the chain rule of Sec. 3.1 over the derivative
// table of Sec. 3.2 sums to P = alpha F + beta cof(F) + gamma F C with
//   alpha = mu1 J^-2/3 + mu2 T_C J^-4/3,
//   beta  = -(mu1/3) T_C J^-5/3 - (mu2/3)(T_C^2 - T_C2) J^-7/3 + kappa (J-1),
//   gamma = -mu2 J^-4/3,  cof(F) = J F^-T.
// FP32 without cancellation: at small strain the three terms are O(mu) each
// and cancel to O(mu |H|). Writing C = I + E (E = H + H^T + H^T H),
// cof(F) = (1 + tr H) I - H^T + cof(H) and F C = I + H + E + H E, the O(mu)
// parts collect into sigma I with
//   sigma = alpha + beta + gamma
//         = mu1 s (3j - e)/(3J) + mu2 s^2 (6j - e + 3je - e^2 + q)/(3J) + kappa j,
// where j = J - 1 = tr H + ((tr H)^2 - tr H^2)/2 + det H, e = tr E, q = tr E^2
// and s = J^-2/3 = exp(-2/3 log1p(j)). Every remaining term is O(|H|).
#pragma once

#include "internal.cuh"

namespace cf {

// ---------------------------------------------------------------- dual numbers
struct Dual {
    float v, d;
    Dual() = default;
    __device__ __forceinline__ Dual(float a) : v(a), d(0.f) {}
    __device__ __forceinline__ Dual(float a, float b) : v(a), d(b) {}
};

__device__ __forceinline__ Dual m_add(Dual a, Dual b) { return {a.v + b.v, a.d + b.d}; }
__device__ __forceinline__ Dual m_add(float a, Dual b) { return {a + b.v, b.d}; }
__device__ __forceinline__ Dual m_sub(Dual a, Dual b) { return {a.v - b.v, a.d - b.d}; }
__device__ __forceinline__ Dual m_mul(Dual a, Dual b) { return {a.v * b.v, fmaf(a.d, b.v, a.v * b.d)}; }
__device__ __forceinline__ Dual m_mul(float a, Dual b) { return {a * b.v, a * b.d}; }
__device__ __forceinline__ Dual m_fma(Dual a, Dual b, Dual c) {  // a b + c: three operations
    return {fmaf(a.v, b.v, c.v), fmaf(a.d, b.v, fmaf(a.v, b.d, c.d))};
}
__device__ __forceinline__ Dual m_fma(float a, Dual b, Dual c) { return {fmaf(a, b.v, c.v), fmaf(a, b.d, c.d)}; }
__device__ __forceinline__ Dual m_neg(Dual a) { return {-a.v, -a.d}; }
__device__ __forceinline__ Dual m_exp(Dual a) {
    const float e = expf(a.v);
    return {e, e * a.d};
}
__device__ __forceinline__ Dual m_rcp(Dual a) {
    const float r = 1.f / a.v;
    return {r, -a.d * r * r};
}

// Sums of products with their roundings written out, so that every kernel
// that evaluates a tet gets the same bits whatever surrounds it (left to the
// compiler, which product of a sum is contracted depends on the context).
__device__ __forceinline__ float m_dot3(float a, float b, float c, float d, float e, float f) {
    return __fmaf_rn(e, f, __fmaf_rn(a, b, __fmul_rn(c, d)));
}
__device__ __forceinline__ float m_cross(float a, float b, float c, float d) {  // a b - c d
    return __fmaf_rn(a, b, -__fmul_rn(c, d));
}
// tr H^2 in row order; (1,2)(2,1) is rounded before it is added
__device__ __forceinline__ float m_trace_sq(const float (&h)[3][3]) {
    float s = __fmul_rn(h[0][0], h[0][0]);
    s = __fmaf_rn(h[0][1], h[1][0], s);
    s = __fmaf_rn(h[0][2], h[2][0], s);
    s = __fmaf_rn(h[1][0], h[0][1], s);
    s = __fmaf_rn(h[1][1], h[1][1], s);
    const float q = __fmul_rn(h[1][2], h[2][1]);
    s = __fadd_rn(s, q);
    s = __fmaf_rn(h[2][0], h[0][2], s);
    s = __fadd_rn(s, q);
    return __fmaf_rn(h[2][2], h[2][2], s);
}

// ---------------------------------------------------------------- stress
template <class S>
struct InvT {
    S t, e, q, j, J, L;  // tr H, tr E, tr E^2, J-1, J, log J
    S E[3][3];
};

__device__ __forceinline__ float det3t(const float (&h)[3][3]) {
    const float A = m_cross(h[1][1], h[2][2], h[1][2], h[2][1]), B = m_cross(h[1][0], h[2][2], h[1][2], h[2][0]),
                C = m_cross(h[1][0], h[2][1], h[1][1], h[2][0]);
    return __fmaf_rn(h[0][2], C, m_cross(h[0][0], A, h[0][1], B));
}

__device__ __forceinline__ void invariants_t(const float (&H)[3][3], InvT<float> &v) {
    v.t = H[0][0] + H[1][1] + H[2][2];
    const float trH2 = m_trace_sq(H);
    float hh = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) hh = hh + H[i][k] * H[i][k];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int l = 0; l < 3; ++l)
            v.E[k][l] = H[k][l] + H[l][k] + H[0][k] * H[0][l] + H[1][k] * H[1][l] + H[2][k] * H[2][l];
    v.e = 2.f * v.t + hh;
    float q = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int l = 0; l < 3; ++l) q = q + v.E[k][l] * v.E[k][l];
    v.q = q;
    v.j = v.t + 0.5f * (v.t * v.t - trH2) + det3t(H);
    v.J = 1.f + v.j;
    v.L = log1pf(v.j);
}

// a b - c d, a cofactor of H. KEEP: those that are also cofactors of the
// determinant stay in registers since the invariants, as suits the on-chip
// steps (64 registers; 1 % faster) and the fused chain (40 -> 32 bytes of
// spills). Otherwise the factors come in the other order, which rounds the
// same but leaves the compiler two evaluations: the force kernel, held to 40
// registers, spills less (36 -> 28 bytes stored, 32 -> 16 read; forces of the
// 400-cell suspension 160 -> 157 us, a relaxation step of 50 k to 270 k tets
// 1 us shorter).
template <bool KEEP>
__device__ __forceinline__ float mr_cofactor(float a, float b, float c, float d) {
    return KEEP ? m_cross(a, b, c, d) : m_cross(b, a, d, c);
}

// P = dU/dF for F = I + H, moduli (mu1, mu2, kappa) and the invariants v of
// H (invariants_t; the caller may replace j, J and L by a more accurate J - 1).
template <bool KEEP = false>
__device__ __forceinline__ void mr_stress_inv(const float (&H)[3][3], float mu1, float mu2, float kappa,
                                              const InvT<float> &v, float (&P)[3][3]) {
    const float s = expf(-(2.f / 3.f) * v.L);  // J^-2/3
    const float s2 = s * s;                    // J^-4/3
    const float TC = 3.f + v.e;
    const float TC2 = 3.f + 2.f * v.e + v.q;
    const float iJ3 = 1.f / (3.f * v.J);
    const float alpha = mu1 * s + mu2 * TC * s2;
    const float beta = kappa * v.j - (mu1 * TC * s + mu2 * (TC * TC - TC2) * s2) * iJ3;
    const float gamma = -mu2 * s2;
    const float sigma = mu1 * s * (3.f * v.j - v.e) * iJ3 +
                        mu2 * s2 * (6.f * v.j - v.e + 3.f * v.j * v.e - v.e * v.e + v.q) * iJ3 + kappa * v.j;
    float cofH[3][3];
    cofH[0][0] = mr_cofactor<KEEP>(H[1][1], H[2][2], H[1][2], H[2][1]);
    cofH[0][1] = mr_cofactor<KEEP>(H[1][2], H[2][0], H[1][0], H[2][2]);
    cofH[0][2] = mr_cofactor<KEEP>(H[1][0], H[2][1], H[1][1], H[2][0]);
    cofH[1][0] = mr_cofactor<KEEP>(H[0][2], H[2][1], H[0][1], H[2][2]);
    cofH[1][1] = mr_cofactor<KEEP>(H[0][0], H[2][2], H[0][2], H[2][0]);
    cofH[1][2] = mr_cofactor<KEEP>(H[0][1], H[2][0], H[0][0], H[2][1]);
    cofH[2][0] = mr_cofactor<KEEP>(H[0][1], H[1][2], H[0][2], H[1][1]);
    cofH[2][1] = mr_cofactor<KEEP>(H[0][2], H[1][0], H[0][0], H[1][2]);
    cofH[2][2] = mr_cofactor<KEEP>(H[0][0], H[1][1], H[0][1], H[1][0]);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const float HE = m_dot3(H[i][0], v.E[0][l], H[i][1], v.E[1][l], H[i][2], v.E[2][l]);
            float p = alpha * H[i][l] + beta * (cofH[i][l] - H[l][i]) + gamma * (H[i][l] + v.E[i][l] + HE);
            if (i == l) p = p + sigma + beta * v.t;
            P[i][l] = p;
        }
}

// P and the invariants for dual numbers, the same expressions in fused
// multiply-adds: a product that is added costs three operations instead of
// four, E is evaluated once per symmetric pair (which the compiler cannot see:
// the tangents of a b and b a round differently), and one reciprocal of J
// serves the logarithm's tangent too. A reverse step of 64 cells of 8.3 k tets,
// bound by instruction issue: 36 -> 30 us.
__device__ __forceinline__ void mr_stress(const Dual (&H)[3][3], float mu1, float mu2, float kappa, InvT<Dual> &v,
                                          Dual (&P)[3][3]) {
    v.t = m_add(m_add(H[0][0], H[1][1]), H[2][2]);
    Dual hh = m_mul(H[0][0], H[0][0]), off = Dual(0.f);
#pragma unroll
    for (int k = 1; k < 9; ++k) hh = m_fma(H[k / 3][k % 3], H[k / 3][k % 3], hh);
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int l = k; l < 3; ++l) {
            Dual e = m_add(H[k][l], H[l][k]);
#pragma unroll
            for (int i = 0; i < 3; ++i) e = m_fma(H[i][k], H[i][l], e);
            v.E[k][l] = v.E[l][k] = e;
            if (l != k) off = m_fma(e, e, off);
        }
    v.e = m_fma(2.f, v.t, hh);
    v.q = m_mul(v.E[0][0], v.E[0][0]);
    v.q = m_fma(2.f, off, m_fma(v.E[2][2], v.E[2][2], m_fma(v.E[1][1], v.E[1][1], v.q)));
    Dual cof[3][3];  // cof(H)
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, l1 = (l + 1) % 3, l2 = (l + 2) % 3;
            cof[i][l] = m_fma(H[i1][l1], H[i2][l2], m_neg(m_mul(H[i1][l2], H[i2][l1])));
        }
    const Dual det = m_fma(H[0][2], cof[0][2], m_fma(H[0][1], cof[0][1], m_mul(H[0][0], cof[0][0])));
    v.j = m_add(m_add(v.t, m_add(m_add(cof[0][0], cof[1][1]), cof[2][2])), det);
    v.J = m_add(1.f, v.j);
    const Dual iJ = m_rcp(v.J), iJ3 = m_mul(1.f / 3.f, iJ);
    v.L = {log1pf(v.j.v), v.j.d * iJ.v};
    const Dual s = m_exp(m_mul(-(2.f / 3.f), v.L));  // J^-2/3
    const Dual a1 = m_mul(mu1, s), a2 = m_mul(mu2, m_mul(s, s)), kj = m_mul(kappa, v.j);
    const Dual TC = m_add(3.f, v.e), TC2 = m_fma(2.f, v.e, m_add(3.f, v.q));
    const Dual alpha = m_fma(a2, TC, a1), gamma = m_neg(a2);
    const Dual x = m_fma(a2, m_fma(TC, TC, m_neg(TC2)), m_mul(a1, TC));
    const Dual beta = m_fma(m_neg(x), iJ3, kj);
    const Dual j3 = m_fma(3.f, v.j, m_neg(v.e));  // 3 j - e
    const Dual y = m_fma(v.e, j3, m_fma(6.f, v.j, m_sub(v.q, v.e)));
    const Dual sigma = m_fma(m_fma(a1, j3, m_mul(a2, y)), iJ3, kj);
    const Dual diag = m_fma(beta, v.t, sigma);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            Dual w = m_add(H[i][l], v.E[i][l]);  // H + E + H E
#pragma unroll
            for (int k = 0; k < 3; ++k) w = m_fma(H[i][k], v.E[k][l], w);
            const Dual p = i == l ? m_fma(gamma, w, diag) : m_mul(gamma, w);
            P[i][l] = m_fma(alpha, H[i][l], m_fma(beta, m_sub(cof[i][l], H[l][i]), p));
        }
}

// x / 3, to within an ulp: a factor 1.f / 3.f would be off by the same 3e-8 in
// every tet.
__device__ __forceinline__ float third(float x) {
    const float c = 1.f / 3.f, y = x * c;
    return fmaf(fmaf(-3.f, y, x), c, y);
}

// Rates of the three unit-modulus energies of one tet along dH: g = d/d eps of
// (I - 3)/2, (K - 3)/2 and (J - 1)^2/2 at H + eps dH, so that a direction
// lambda of the vertices with dH its gradient has lambda . f = -V0 g . (mu1,
// mu2, kappa). One contraction per modulus takes the place of a stress and
// twelve force components per modulus. With hd = H:dH and
// r = (H + H^T - t I - cof(H)):dH, de = 2 (tr dH + hd) and
// dj = tr dH + hd - r, and the O(|dH|) parts of de - 2 dj cancel by hand
// (J de - 2 dj = 2 r + j de, and twice that for K), so every term left is
// O(|H| |dH|), as in the stress; r is summed from the differences, which
// vanish under a rotation, not as the difference of two sums:
//   d(I) = s/J [J de - 2/3 (3 + e) dj],  s = J^-2/3,
//   d(K) = s^2/J [J dK' - 4/3 K' dj],    K' = 3 + 2e + (e^2 - q)/2.
// Sums over a cell against 64 bits, beside FP64 products of lambda with the
// forces of three unit-modulus stresses in its place: 0.9 of their error over
// random directions (noise, stretched, squashed and rotated cells of 1.7 k to
// 20 k tets; 0.8 to 1.25 for smooth directions).
__device__ __forceinline__ void mr_energy_rates(const float (&H)[3][3], const float (&dH)[3][3], const InvT<float> &v,
                                                float (&g)[3]) {
    const float dt = dH[0][0] + dH[1][1] + dH[2][2];
    float hd = 0.f, r = 0.f, eg = 0.f;  // eg = E:(F^T dH)
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, k1 = (k + 1) % 3, k2 = (k + 2) % 3;
            const float sym = i == k ? H[i][k] + H[k][i] - v.t : H[i][k] + H[k][i];
            r += (sym - fmaf(H[i1][k1], H[i2][k2], -(H[i1][k2] * H[i2][k1]))) * dH[i][k];
            hd += H[i][k] * dH[i][k];
            eg += v.E[i][k] * (dH[i][k] + H[0][i] * dH[0][k] + H[1][i] * dH[1][k] + H[2][i] * dH[2][k]);
        }
    const float dj = dt + (hd - r), de = 2.f * (dt + hd);
    const float dk = v.e * de - 2.f * eg;  // dK' - 2 de, with dq = 4 E:(F^T dH)
    const float k3 = 2.f * v.e + 0.5f * (v.e * v.e - v.q);
    const float s = expf(-(2.f / 3.f) * v.L), iJ = 1.f / v.J;
    g[0] = third(s * iJ * (3.f * r + 1.5f * v.j * de - v.e * dj));
    g[1] = third(s * s * iJ * (6.f * r + 1.5f * (dk + v.j * (2.f * de + dk)) - 2.f * k3 * dj));
    g[2] = v.j * dj;
}

// The rates are linear in dH. Directions are taken times a power of two that
// brings their largest component x (>= 0) near 1, 2^(127 - b) with b its biased
// exponent, and the sums back in FP64, so that neither leaves FP32's range
// where the direction itself does not. Infinities and NaN: factor 1.
__device__ __forceinline__ int direction_exponent(float x) {
    const int b = __float_as_int(x) >> 23;
    return b == 255 ? 127 : min(max(b, 1), 253);
}
__device__ __forceinline__ float power_of_two(int b) { return __int_as_float(b << 23); }  // 2^(b - 127), 0 < b < 255
__device__ __forceinline__ double power_of_two_64(int b) { return __hiloint2double((b - 127 + 1023) << 20, 0); }
__device__ __forceinline__ float largest(float4 a, float x) {
    return fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(a.z), x));
}
__device__ __forceinline__ float4 times(float4 a, float x) { return make_float4(a.x * x, a.y * x, a.z * x, 0.f); }

// A sum of floats kept as an unevaluated pair hi + lo: every addition is the
// exact two-sum (D. E. Knuth, The Art of Computer Programming vol. 2, 4.2.2),
// its error collected in lo, so the pair carries about 48 bits. FP64 units
// are few on this GPU (about two additions per clock and SM); six FP32
// additions per term are several times cheaper and as exact here.
struct Sum2 {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float t = __fadd_rn(hi, x), b = __fsub_rn(t, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, b)), __fsub_rn(x, b)));
        hi = t;
    }
    // an infinite or NaN sum: lo is NaN by then
    __device__ __forceinline__ double value() const { return isfinite(hi) ? (double)hi + (double)lo : (double)hi; }
};

// Sum of a pair over the lanes of a full warp (every lane ends with it).
__device__ __forceinline__ void warp_sum(Sum2 &a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h = __shfl_xor_sync(0xffffffffu, a.hi, o), l = __shfl_xor_sync(0xffffffffu, a.lo, o);
        a.add(h);
        a.lo = __fadd_rn(a.lo, l);
    }
}

// Nearly incompressible tets (kappa >= kStiffVolume (mu1 + mu2), Poisson
// ratio 0.495 and above) take J - 1 in FP64. The volume term kappa (J - 1)
// multiplies any rounding of J - 1 by kappa: under a nearly isochoric
// deformation J - 1 is small against |H|, and J - 1 from the FP32 B and
// FP32 products carries errors of ~1e-7 |H|, which reach the forces
// amplified by kappa / mu (measured: 7e-5 relative at kappa = 2,000 mu in
// simple shear). In FP64, from the FP32 displacements (exact in FP64) and the
// FP64 B of the precompute, J - 1 is exact to ~1e-16 |H|; the rest of the
// stress stays FP32.
constexpr float kStiffVolume = 100.f;

__device__ __forceinline__ bool needs_fp64_volume(const MeshView &m, float4 mat) {
    return m.B64 != nullptr && mat.z >= kStiffVolume * (mat.x + mat.y);
}

// J - 1 = tr H + ((tr H)^2 - tr H^2) / 2 + det H in FP64 with H = A B, A from
// the column differences a_k = w_k - w_4 (k = 1..3, exact in FP64), B from
// B64 ([9][T]).
__device__ __forceinline__ double volume_change64_body(const double *__restrict__ B64, int T, int t, float4 w0,
                                                       float4 w1, float4 w2, float4 w3) {
    const double A[3][3] = {{(double)w0.x - w3.x, (double)w1.x - w3.x, (double)w2.x - w3.x},
                            {(double)w0.y - w3.y, (double)w1.y - w3.y, (double)w2.y - w3.y},
                            {(double)w0.z - w3.z, (double)w1.z - w3.z, (double)w2.z - w3.z}};
    double Bm[3][3], H[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j) Bm[k][j] = __ldg(B64 + (size_t)(3 * k + j) * T + t);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) H[i][j] = A[i][0] * Bm[0][j] + A[i][1] * Bm[1][j] + A[i][2] * Bm[2][j];
    const double tr = H[0][0] + H[1][1] + H[2][2];
    double tr2 = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) tr2 += H[i][k] * H[k][i];
    const double det = H[0][0] * (H[1][1] * H[2][2] - H[1][2] * H[2][1]) -
                       H[0][1] * (H[1][0] * H[2][2] - H[1][2] * H[2][0]) +
                       H[0][2] * (H[1][0] * H[2][1] - H[1][1] * H[2][0]);
    return tr + 0.5 * (tr * tr - tr2) + det;
}

// The same as a called function, for kernels whose FP32 path the FP64
// registers would otherwise crowd (one thread per tet).
static __device__ __noinline__ double volume_change64(const double *__restrict__ B64, int T, int t, float4 w0, float4 w1,
                                               float4 w2, float4 w3) {
    return volume_change64_body(B64, T, t, w0, w1, w2, w3);
}

// Replace J - 1 (and J, log J) of v by j.
__device__ __forceinline__ void set_volume_change(InvT<float> &v, float j) {
    v.j = j;
    v.J = 1.f + j;
    v.L = log1pf(j);
}

// Corner forces f^a_i = -V_0 sum_l P_il B_al (a = 1..3), f^4 = -(f^1 + f^2 + f^3)
// (Sec. 3.1 with dF_kl/du_i^a = delta_ki B_ml (delta_ma - delta_4a)).
__device__ __forceinline__ void corner_forces(const float (&P)[3][3], const float (&Bm)[3][3], float V0,
                                              float (&f)[4][3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int i = 0; i < 3; ++i) f[a][i] = -V0 * (P[i][0] * Bm[a][0] + P[i][1] * Bm[a][1] + P[i][2] * Bm[a][2]);
#pragma unroll
    for (int i = 0; i < 3; ++i) f[3][i] = -(f[0][i] + f[1][i] + f[2][i]);
}

// A B for a tet: A_ik = w_i^k - w_i^4 from four per-vertex vectors.
__device__ __forceinline__ void tet_grad(const float4 &w0, const float4 &w1, const float4 &w2, const float4 &w3,
                                         const float (&Bm)[3][3], float (&H)[3][3]) {
    const float A[3][3] = {{w0.x - w3.x, w1.x - w3.x, w2.x - w3.x},
                           {w0.y - w3.y, w1.y - w3.y, w2.y - w3.y},
                           {w0.z - w3.z, w1.z - w3.z, w2.z - w3.z}};
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) H[i][j] = A[i][0] * Bm[0][j] + A[i][1] * Bm[1][j] + A[i][2] * Bm[2][j];
}

// Corner tangents along dH of a tet at H (the stress on dual numbers), and the
// invariants at H.
__device__ __forceinline__ void tet_tangent(const float (&H)[3][3], const float (&dH)[3][3], float4 mat,
                                            const float (&Bm)[3][3], float V0, InvT<float> &inv, float (&f)[4][3]) {
    Dual Hd[3][3], P[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) Hd[i][j] = Dual(H[i][j], dH[i][j]);
    InvT<Dual> v;
    mr_stress(Hd, mat.x, mat.y, mat.z, v, P);
    float dP[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            dP[i][j] = P[i][j].d;
            inv.E[i][j] = v.E[i][j].v;
        }
    corner_forces(dP, Bm, V0, f);
    inv.t = v.t.v;
    inv.e = v.e.v;
    inv.q = v.q.v;
    inv.j = v.j.v;
    inv.J = v.J.v;
    inv.L = v.L.v;
}

// Material slot of tet t.
__device__ __forceinline__ int mat_slot(const MeshView &m, int t) { return __ldg((m.tmat ? m.tmat : m.tcell) + t); }

// B, V0 and the tet's material slot: three 16-byte loads from the packed
// rows when the view has them, else eleven 4-byte loads from the separate
// arrays.
__device__ __forceinline__ void load_tet_params(const MeshView &m, int t, float (&Bm)[3][3], float &V0, int &slot) {
    if (m.Bp) {
        const float4 r0 = __ldg(m.Bp + t), r1 = __ldg(m.Bp + m.T + t), r2 = __ldg(m.Bp + 2 * m.T + t);
        Bm[0][0] = r0.x; Bm[0][1] = r0.y; Bm[0][2] = r0.z;
        Bm[1][0] = r1.x; Bm[1][1] = r1.y; Bm[1][2] = r1.z;
        Bm[2][0] = r2.x; Bm[2][1] = r2.y; Bm[2][2] = r2.z;
        V0 = r0.w;
        slot = __float_as_int(r1.w);
        return;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j) Bm[k][j] = __ldg(m.B + (3 * k + j) * m.T + t);
    V0 = __ldg(m.V0 + t);
    slot = mat_slot(m, t);
}

__device__ __forceinline__ void load_B(const MeshView &m, int t, float (&Bm)[3][3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j) Bm[k][j] = __ldg(m.B + (3 * k + j) * m.T + t);
}

}  // namespace cf
