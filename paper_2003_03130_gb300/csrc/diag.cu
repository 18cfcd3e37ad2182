// K8: Taylor deformation parameter of a cell on the device (Sec. 3.3).
//
// Inertia tensor of the tet mesh at the current positions,
//   Theta_ij = sum_l V_l (r^l.r^l delta_ij - r^l_i r^l_j),
// with r^l the centroid of tet l relative to the volume-weighted centroid of
// the cell and V_l its current volume. One pass accumulates, in double and in
// a fixed order (per-block tree, then the blocks in index order), the moments
// M = sum V, m = sum V c, S = sum V c c^T of the tet centroids c; then
// Theta = (tr S' ) I - S' with S' = S - m m^T / M. A single thread finishes:
// eigenvalues theta_1 >= theta_2 >= theta_3 by cyclic Jacobi rotations,
// semi-axes a_i = sqrt((5 / 2M)(...)) (the printed expression has units of
// length squared, so a_i is its square root), D = (a3 - a1)/(a3 + a1), and the
// inclination of the major axis (eigenvector of theta_3) to x in the x-y
// plane, in (-90, 90] degrees. Positions enter relative to the cell's integer
// origin (translation does not change Theta).
#include <cooperative_groups.h>

#include "internal.cuh"

namespace cf {

constexpr int kTaylorBlock = 256;
constexpr int kMoments = 10;  // M, m (3), S (6: xx yy zz xy xz yz)

__global__ void __launch_bounds__(kTaylorBlock) k_taylor_partial(MeshView m, const float4 *__restrict__ u, int t0,
                                                                 int t1, double *partial) {
    __shared__ double red[kMoments][kTaylorBlock];
    const int t = t0 + blockIdx.x * blockDim.x + threadIdx.x;
    double v[kMoments] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    if (t < t1) {
        const int4 a = __ldg(m.tet + t);
        const int idx[4] = {a.x, a.y, a.z, a.w};
        double p[4][3];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float4 xr = __ldg(m.xr + idx[c]), du = __ldg(u + idx[c]);
            p[c][0] = (double)(xr.x + du.x);
            p[c][1] = (double)(xr.y + du.y);
            p[c][2] = (double)(xr.z + du.z);
        }
        double e[3][3];
        for (int k = 0; k < 3; ++k)
            for (int i = 0; i < 3; ++i) e[k][i] = p[k][i] - p[3][i];
        const double det = e[0][0] * (e[1][1] * e[2][2] - e[1][2] * e[2][1]) -
                           e[0][1] * (e[1][0] * e[2][2] - e[1][2] * e[2][0]) +
                           e[0][2] * (e[1][0] * e[2][1] - e[1][1] * e[2][0]);
        const double V = fabs(det) / 6.0;
        double c[3];
        for (int i = 0; i < 3; ++i) c[i] = 0.25 * (p[0][i] + p[1][i] + p[2][i] + p[3][i]);
        v[0] = V;
        v[1] = V * c[0];
        v[2] = V * c[1];
        v[3] = V * c[2];
        v[4] = V * c[0] * c[0];
        v[5] = V * c[1] * c[1];
        v[6] = V * c[2] * c[2];
        v[7] = V * c[0] * c[1];
        v[8] = V * c[0] * c[2];
        v[9] = V * c[1] * c[2];
    }
#pragma unroll
    for (int k = 0; k < kMoments; ++k) red[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int w = kTaylorBlock / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
#pragma unroll
            for (int k = 0; k < kMoments; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < kMoments) partial[blockIdx.x * kMoments + threadIdx.x] = red[threadIdx.x][0];
}

// Symmetric 3x3 eigen-decomposition by cyclic Jacobi rotations; columns of
// V are the eigenvectors. One warp's FP64 issue bounds it (an FP64
// instruction holds its pipe for 64 cycles), so a rotation takes one square
// root, one division and one reciprocal square root, and updates only the
// entries that it changes. Angles from FP32, made rotations in FP64, took
// more FP64 instructions and 3 us longer.
__device__ __forceinline__ void rotate3(double &app, double &aqq, double &apq, double &arp, double &arq,
                                        double (&V)[3][3], int p, int q) {
    if (apq * apq == 0.0) return;  // also where its square underflows
    const double d = aqq - app, b = 2.0 * apq;
    const double t = (d >= 0.0 ? b : -b) / (fabs(d) + sqrt(fma(d, d, b * b)));
    const double c = rsqrt(fma(t, t, 1.0)), s = t * c;
    app -= t * apq;
    aqq += t * apq;
    apq = 0.0;
    const double rp = arp, rq = arq;
    arp = c * rp - s * rq;
    arq = s * rp + c * rq;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double vp = V[k][p], vq = V[k][q];
        V[k][p] = c * vp - s * vq;
        V[k][q] = s * vp + c * vq;
    }
}

// lam: the eigenvalues of the symmetric matrix (xx, yy, zz, xy, xz, yz).
__device__ __forceinline__ void jacobi3(double xx, double yy, double zz, double xy, double xz, double yz,
                                        double (&lam)[3], double (&V)[3][3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) V[i][j] = i == j ? 1.0 : 0.0;
    for (int sweep = 0; sweep < 50; ++sweep) {
        const double off = xy * xy + xz * xz + yz * yz;
        const double dia = xx * xx + yy * yy + zz * zz;
        if (off <= 1e-30 * (dia > 1.0 ? dia : 1.0)) break;
        rotate3(xx, yy, xy, xz, yz, V, 0, 1);
        rotate3(xx, zz, xz, xy, yz, V, 0, 2);
        rotate3(yy, zz, yz, xy, xz, V, 1, 2);
    }
    lam[0] = xx;
    lam[1] = yy;
    lam[2] = zz;
}

// out[10]: D, D from the printed (squared) expression, inclination (deg),
// a1 <= a2 <= a3, theta1 >= theta2 >= theta3, volume.
// Warp k sums moment k over the blocks (lanes strided, then a fixed shuffle
// tree), thread 0 finishes: 30 us for 787 blocks and 26 us for 78, most of it
// the eigenvalues. One thread that summed all of them, a chain of dependent
// FP64 additions, took 376 and 66 us.
__global__ void __launch_bounds__(32 * kMoments) k_taylor_final(const double *__restrict__ partial, int nblocks,
                                                                double *out) {
    __shared__ double s[kMoments];
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double sum = 0.0;
#pragma unroll 4
    for (int b = lane; b < nblocks; b += 32) sum += partial[(size_t)b * kMoments + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) s[k] = sum;
    __syncthreads();
    if (threadIdx.x != 0) return;
    const double M = s[0];
    const double c0[3] = {s[1] / M, s[2] / M, s[3] / M};
    // second moments about the centroid
    double S[3][3];
    S[0][0] = s[4] - M * c0[0] * c0[0];
    S[1][1] = s[5] - M * c0[1] * c0[1];
    S[2][2] = s[6] - M * c0[2] * c0[2];
    S[0][1] = S[1][0] = s[7] - M * c0[0] * c0[1];
    S[0][2] = S[2][0] = s[8] - M * c0[0] * c0[2];
    S[1][2] = S[2][1] = s[9] - M * c0[1] * c0[2];
    const double tr = S[0][0] + S[1][1] + S[2][2];
    double lam[3], V[3][3];
    jacobi3(tr - S[0][0], tr - S[1][1], tr - S[2][2], -S[0][1], -S[0][2], -S[1][2], lam, V);
    int ord[3] = {0, 1, 2};  // descending eigenvalues
    for (int i = 0; i < 3; ++i)
        for (int j = i + 1; j < 3; ++j)
            if (lam[ord[j]] > lam[ord[i]]) {
                const int tmp = ord[i];
                ord[i] = ord[j];
                ord[j] = tmp;
            }
    const double t1 = lam[ord[0]], t2 = lam[ord[1]], t3 = lam[ord[2]];
    const double pre = 5.0 / (2.0 * M);
    const double a1s = pre * (-t1 + t2 + t3), a2s = pre * (t1 - t2 + t3), a3s = pre * (t1 + t2 - t3);
    const double a1 = sqrt(a1s > 0 ? a1s : 0), a2 = sqrt(a2s > 0 ? a2s : 0), a3 = sqrt(a3s > 0 ? a3s : 0);
    const int k3 = ord[2];
    double ang = atan2(V[1][k3], V[0][k3]) * (180.0 / 3.14159265358979323846);
    if (ang <= -90.0) ang += 180.0;
    if (ang > 90.0) ang -= 180.0;
    out[0] = (a3 - a1) / (a3 + a1);
    out[1] = (a3s - a1s) / (a3s + a1s);
    out[2] = ang;
    out[3] = a1;
    out[4] = a2;
    out[5] = a3;
    out[6] = t1;
    out[7] = t2;
    out[8] = t3;
    out[9] = M;
}

cudaError_t launch_taylor(const MeshView &m, const float4 *u, int t0, int t1, double *partial, double *out,
                          cudaStream_t s) {
    const int nb = (t1 - t0 + kTaylorBlock - 1) / kTaylorBlock;
    if (nb > 0) k_taylor_partial<<<nb, kTaylorBlock, 0, s>>>(m, u, t0, t1, partial);
    k_taylor_final<<<1, 32 * kMoments, 0, s>>>(partial, nb, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- cell strain
// Largest distance between two vertices of a cell (the elongation d_max of
// the cell strain, Sec. 6.1), exact over all pairs. With r_i the distance of
// vertex i from any centre c, |y_i - y_j| <= r_i + r_j, so once some pair at
// distance L is known only vertices with r_i + r_max >= L can belong to a
// longer one: k_extent_select takes c the middle of the bounding box and L
// from the vertex farthest from c and the one farthest from that, and keeps
// those vertices (the surface, for a cell: 6 k of 37 k), k_extent_pairs
// sweeps the pairs of the kept ones, tile against tile. The maximum does not
// depend on the order; the bound is widened by 1e-4, far more than the
// rounding of the FP32 distances. All pairs of all vertices in one block per
// tile took 52 us for 4.2 k vertices and 428 us for 37 k; selection and pairs
// together take 18 and 23 us. Cells whose pairs of tiles fill at most one
// round of blocks (8.7 k vertices) take them all without a selection, those of
// one tile in one block that writes to the host: the whole call for 81 vertices
// 22 us with the old kernel, 33 with a selection, 15 now; for 365 29, 34
// and 27, for 4.2 k 68, 41 and 28. Positions enter relative to the cell's
// integer origin.
constexpr int kExtentBlock = kExtentOne;
constexpr int kSelectBlock = 1024;

__device__ __forceinline__ float dist2(float3 a, float3 b) {
    const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
    return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

__device__ __forceinline__ float3 rel_pos(const MeshView &m, const float4 *__restrict__ u, int v) {
    const float4 xr = __ldg(m.xr + v), du = __ldg(u + v);
    return make_float3(xr.x + du.x, xr.y + du.y, xr.z + du.z);
}

// x[k] = maximum over the cluster's threads: over the warp, the block, then
// the blocks through their shared memory; every thread ends with it. Each
// call of a kernel has its own `sc`, so no block overwrites what another
// still reads.
constexpr int kSelectCluster = 8, kSelectWarps = kSelectBlock / 32;

template <int N>
struct SelectScratch {
    float warp[N][kSelectWarps], block[N];
};

template <int N>
__device__ __forceinline__ void cluster_max(float (&x)[N], SelectScratch<N> &sc) {
    namespace cg = cooperative_groups;
    const cg::cluster_group cl = cg::this_cluster();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < N; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x[k] = fmaxf(x[k], __shfl_xor_sync(0xffffffffu, x[k], o));
        if (lane == 0) sc.warp[k][w] = x[k];
    }
    __syncthreads();
    if (w < N) {  // warp k finishes value k
        float y = sc.warp[w][lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) y = fmaxf(y, __shfl_xor_sync(0xffffffffu, y, o));
        if (lane == 0) sc.block[w] = y;
    }
    cl.sync();
#pragma unroll
    for (int k = 0; k < N; ++k) {
        x[k] = *cl.map_shared_rank(&sc.block[k], lane % kSelectCluster);
#pragma unroll
        for (int o = kSelectCluster / 2; o > 0; o >>= 1) x[k] = fmaxf(x[k], __shfl_xor_sync(0xffffffffu, x[k], o));
    }
}

// One cluster of eight blocks: every pass over the vertices waits for the one
// before, so it is bound by latency: 12 us for 4.2 k vertices and 17 us for
// 37 k (one block: 9 and 34 us).
__global__ void __cluster_dims__(kSelectCluster, 1, 1) __launch_bounds__(kSelectBlock)
    k_extent_select(MeshView m, const float4 *__restrict__ u, int v0, int nv, float4 *keep, int *nkeep, unsigned *out) {
    namespace cg = cooperative_groups;
    __shared__ SelectScratch<6> box;
    __shared__ SelectScratch<1> red[3];
    const int lane = threadIdx.x & 31, first = blockIdx.x * kSelectBlock + threadIdx.x;
    constexpr int kStride = kSelectCluster * kSelectBlock;
    if (first == 0) {  // before the first cluster barrier
        *nkeep = 0;
        *out = 0u;
        __threadfence();
    }
    float b[6] = {-3e38f, -3e38f, -3e38f, -3e38f, -3e38f, -3e38f};  // upper ends, negated lower ends
    for (int k = first; k < nv; k += kStride) {
        const float3 y = rel_pos(m, u, v0 + k);
        b[0] = fmaxf(b[0], y.x), b[1] = fmaxf(b[1], y.y), b[2] = fmaxf(b[2], y.z);
        b[3] = fmaxf(b[3], -y.x), b[4] = fmaxf(b[4], -y.y), b[5] = fmaxf(b[5], -y.z);
    }
    cluster_max(b, box);
    const float3 c = make_float3(0.5f * (b[0] - b[3]), 0.5f * (b[1] - b[4]), 0.5f * (b[2] - b[5]));
    float rmax[1] = {-1.f}, at[1] = {0.f}, far[1] = {-1.f};
    for (int k = first; k < nv; k += kStride) rmax[0] = fmaxf(rmax[0], dist2(rel_pos(m, u, v0 + k), c));
    cluster_max(rmax, red[0]);
    // one vertex at rmax (the same operations give the same bits); any will
    // do, and none (NaN, or an index beyond FP32's integers) leaves another
    for (int k = first; k < nv; k += kStride)
        if (dist2(rel_pos(m, u, v0 + k), c) == rmax[0]) at[0] = (float)min(k, 1 << 24);
    cluster_max(at, red[1]);
    const float3 ya = rel_pos(m, u, v0 + min((int)at[0], nv - 1));
    for (int k = first; k < nv; k += kStride) far[0] = fmaxf(far[0], dist2(rel_pos(m, u, v0 + k), ya));
    cluster_max(far, red[2]);
    const float need = sqrtf(far[0]) * (1.f - 1e-4f) - sqrtf(rmax[0]);  // kept if r_i >= need
    for (int k0 = blockIdx.x * kSelectBlock; k0 < nv; k0 += kStride) {
        const int k = k0 + threadIdx.x;
        float3 y = make_float3(0.f, 0.f, 0.f);
        bool take = false;
        if (k < nv) {
            y = rel_pos(m, u, v0 + k);
            take = !(sqrtf(dist2(y, c)) * (1.f + 1e-4f) < need);
        }
        const unsigned mask = __ballot_sync(0xffffffffu, take);
        int base = 0;
        if (lane == 0 && mask) base = atomicAdd(nkeep, __popc(mask));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (take) keep[base + __popc(mask & ((1u << lane) - 1u))] = make_float4(y.x, y.y, y.z, 0.f);
    }
    cg::this_cluster().sync();  // no block leaves while another reads its shared memory
}

// Pairs of kept vertices (KEPT; else of all of the cell's), one pair of tiles
// (row <= column) per block and round; non-negative floats order like their
// bits.
template <bool KEPT>
__global__ void __launch_bounds__(kExtentBlock) k_extent_pairs(const float4 *__restrict__ keep,
                                                               const int *__restrict__ nkeep, MeshView m,
                                                               const float4 *__restrict__ u, int v0, int nv,
                                                               unsigned *out) {
    __shared__ float4 tile[kExtentBlock];
    const int n = KEPT ? *nkeep : nv, nt = (n + kExtentBlock - 1) / kExtentBlock;
    auto at = [&](int k) {  // padding takes vertex 0: real pairs
        k = k < n ? k : 0;
        if (KEPT) return keep[k];
        const float3 y = rel_pos(m, u, v0 + k);
        return make_float4(y.x, y.y, y.z, 0.f);
    };
    float best = 0.f;
    int row = 0;
    long long first = 0;  // index of the pair (row, row)
    for (long long p = blockIdx.x; p < (long long)nt * (nt + 1) / 2; p += gridDim.x) {
        while (p >= first + nt - row) first += nt - row++;
        const int i = row * kExtentBlock + threadIdx.x, j = (row + (int)(p - first)) * kExtentBlock + threadIdx.x;
        __syncthreads();
        tile[threadIdx.x] = at(j);
        __syncthreads();
        const float4 q = at(i);
        const float3 y = make_float3(q.x, q.y, q.z);
#pragma unroll 8
        for (int k = 0; k < kExtentBlock; ++k) {
            const float4 o = tile[k];
            best = fmaxf(best, dist2(make_float3(o.x, o.y, o.z), y));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(best));
}

// A cell of one tile: one block, its maximum stored without an atomic, so that
// *out can be mapped host memory.
__global__ void __launch_bounds__(kExtentBlock) k_extent_one(MeshView m, const float4 *__restrict__ u, int v0, int nv,
                                                             unsigned *out) {
    __shared__ float3 tile[kExtentBlock];
    __shared__ float most[kExtentBlock / 32];
    const float3 y = rel_pos(m, u, v0 + min((int)threadIdx.x, nv - 1));
    tile[threadIdx.x] = y;
    __syncthreads();
    float best = 0.f;
    for (int k = 0; k < nv; ++k) best = fmaxf(best, dist2(tile[k], y));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0) most[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x > 0) return;
    for (int w = 1; w < kExtentBlock / 32; ++w) best = fmaxf(best, most[w]);
    *out = __float_as_uint(best);
}

cudaError_t launch_extent_one(const MeshView &m, const float4 *u, int v0, int nv, unsigned *out, cudaStream_t s) {
    k_extent_one<<<1, kExtentBlock, 0, s>>>(m, u, v0, nv, out);
    return cudaGetLastError();
}

cudaError_t launch_max_extent(const MeshView &m, const float4 *u, int v0, int nv, float4 *keep, unsigned *out,
                              int blocks, cudaStream_t s) {
    const long long nt = (nv + kExtentBlock - 1) / kExtentBlock;
    if (nt * (nt + 1) / 2 <= blocks) {
        const cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned), s);
        if (e != cudaSuccess || nv <= 0) return e;
        k_extent_pairs<false><<<(int)(nt * (nt + 1) / 2), kExtentBlock, 0, s>>>(nullptr, nullptr, m, u, v0, nv, out);
        return cudaGetLastError();
    }
    int *nkeep = reinterpret_cast<int *>(out + 1);
    k_extent_select<<<kSelectCluster, kSelectBlock, 0, s>>>(m, u, v0, nv, keep, nkeep, out);
    k_extent_pairs<true><<<blocks, kExtentBlock, 0, s>>>(keep, nkeep, m, u, v0, nv, out);
    return cudaGetLastError();
}

}  // namespace cf
