// Relaxation between plates with a cell's state kept on chip: one thread-block
// cluster per cell takes n damped steps (or n reverse steps of the adjoint) in
// one launch.
//
// Cells between plates do not touch one another, so a step needs no barrier
// wider than a cell. A cell's vertices are cut into `cs` contiguous ranges, one
// per block of the cluster; a block evaluates every tet that touches its
// vertices (tets on a cut are evaluated by both sides: 11 % more tets for two
// blocks of an 8 k-tet cell), so corner forces stay in its shared memory and
// the only data that blocks exchange are the new displacements of their own
// vertices, written into every block's copy of the cell through distributed
// shared memory. Per step: tets -> corner forces (shared memory) -> sums over
// the incidence rows, the damped step, the exchange. Two cluster barriers
// order it: one after the tets (nobody reads the old displacements any more;
// its wait hides under the sums) and one after the exchange.
//
// The order of every sum is that of k_gather_spread (four strided partial sums
// per vertex, a fixed tree), and the tets run the same code, so the positions
// are those of the general path (three launches a step, k_tet_force,
// k_gather_spread, k_plate_step), bit for bit. That path stays for cells
// that do not fit (shared memory holds 16 bytes per vertex of the cell, 16 more
// per vertex and 36 per tet of a block, the reverse step 32 and 36; up to eight
// blocks a cluster, 65,535 vertices a cell and 32 incidences a vertex) and
// where it is expected to be faster (csrc/plates.cu, make_plan).
//
// Bound by instruction issue and the two barriers of a step: 655 warp
// instructions per 32 tets, incidences included, in 0.71 of the slots of the SMs
// that have a block (reverse steps 1,040 in 0.62). 64 cells of 8.3 k tets (1,863
// vertices) on 128 SMs: 16.2 us a step, where three launches take 29 (the corner
// forces cross L2 there, 64 bytes written and read per tet); a reverse step
// 30.5 us, 40 in launches. A cell of 1.2 k tets: 3.2 us a step and 4.6 a reverse
// one, 12.4 and 14 in launches. Velocities stay in shared memory and the trail is
// stored a step late, since a barrier's release waits for every store still on
// its way (19 -> 17.5 us). Measured and not taken: every tet in one block only,
// corner forces read from the neighbour through distributed shared memory (20.5
// us).
#include <climits>

#include "cell_ops.cuh"
#include "plate_ops.cuh"

namespace cf {

namespace cg = cooperative_groups;

// Threads per block. The steps hide shared-memory and L2 latency better with
// 1,024 threads of 64 registers than with 512 of 128 (64 cells of 8 k tets:
// 19 us a step against 22; 768 threads: 20); the reverse step's dual numbers
// need the 128.
constexpr int kStepBlock = 1024;
constexpr int kReverseBlock = 512;

// Own vertex range of block r of `cs` of a cell with vertices [v0, v0 + nv).
__host__ __device__ __forceinline__ int part_begin(int v0, int nv, int r, int cs) {
    return v0 + (int)((long long)nv * r / cs);
}

__device__ __forceinline__ bool touches(int4 a, int lo, int hi) {
    return (a.x >= lo && a.x < hi) || (a.y >= lo && a.y < hi) || (a.z >= lo && a.z < hi) || (a.w >= lo && a.w < hi);
}

// ---------------------------------------------------------------- plan
// Tets per block for clusters of 1, 2, 4 and 8 blocks: block 15 c + k of the
// grid counts block k of cell c (k = 0; 1, 2; 3..6; 7..14). cells[c] = (first
// vertex, vertices, first tet, tets). counts[15 c + k]; *degree = the largest
// number of incidences of a vertex.
__global__ void __launch_bounds__(256) k_relax_count(MeshView m, const int4 *__restrict__ cells, int *counts,
                                                     int *degree) {
    const int c = blockIdx.x / 15, k = blockIdx.x % 15;
    const int cs = k >= 7 ? 8 : k >= 3 ? 4 : k >= 1 ? 2 : 1, r = k - (cs - 1);
    const int4 cell = cells[c];
    const int lo = part_begin(cell.x, cell.y, r, cs), hi = part_begin(cell.x, cell.y, r + 1, cs);
    __shared__ int total;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    int n = 0;
    for (int t = threadIdx.x; t < cell.w; t += blockDim.x) n += touches(__ldg(m.tet + cell.z + t), lo, hi);
    atomicAdd(&total, n);
    if (cs == 1)
        for (int v = lo + threadIdx.x; v < hi; v += blockDim.x) atomicMax(degree, m.csr_ptr[v + 1] - m.csr_ptr[v]);
    __syncthreads();
    if (threadIdx.x == 0) counts[blockIdx.x] = total;
}

// The tets of every part in ascending order, packed for the step kernels:
// rows[k * NT + i] = row k of B with .w = V0, vertex indices 0 and 1, indices 2
// and 3 (16 bits each, within the cell); list[i] = the tet, its sign bit set
// unless this part owns its first corner (an owner counts its gradient).
// slot[r * T + t] = the place of tet t in block r's part.
__global__ void __launch_bounds__(1024) k_relax_fill(MeshView m, const RelaxPart *__restrict__ parts, int cs,
                                                     const int4 *__restrict__ cells, float4 *rows, int NT, int *list,
                                                     int *slot) {
    __shared__ int warp_count[32], before[32], base;
    const RelaxPart p = parts[blockIdx.x];
    const int r = blockIdx.x % cs, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int4 cell = cells[p.cell];
    if (threadIdx.x == 0) base = 0;
    for (int t0 = 0; t0 < cell.w; t0 += 1024) {
        const int t = cell.z + t0 + threadIdx.x;
        int4 a = make_int4(-1, -1, -1, -1);
        if (t0 + (int)threadIdx.x < cell.w) a = __ldg(m.tet + t);
        const bool mine = touches(a, p.v0, p.v0 + p.nv);
        const unsigned mask = __ballot_sync(0xffffffffu, mine);
        if (lane == 0) warp_count[w] = __popc(mask);
        __syncthreads();
        if (w == 0) {
            int n = warp_count[lane], x = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            before[lane] = base + x - n;
            __syncwarp();
            if (lane == 31) base += x;
        }
        __syncthreads();
        if (mine) {
            const int s = before[w] + __popc(mask & ((1u << lane) - 1u)), i = p.t0 + s;
            float4 b0 = __ldg(m.Bp + t), b1 = __ldg(m.Bp + m.T + t), b2 = __ldg(m.Bp + 2 * (size_t)m.T + t);
            b1.w = __int_as_float((a.x - cell.x) | (a.y - cell.x) << 16);
            b2.w = __int_as_float((a.z - cell.x) | (a.w - cell.x) << 16);
            rows[i] = b0;
            rows[NT + i] = b1;
            rows[2 * (size_t)NT + i] = b2;
            list[i] = a.x >= p.v0 && a.x < p.v0 + p.nv ? t : t | INT_MIN;
            slot[(size_t)r * m.T + t] = s;
        }
        __syncthreads();
    }
}

// Incidences of vertex v for its four lanes, eight 16-bit entries each, as in
// gather_vertex: lane k holds entries k, k + 4, ... of the row, 4 s + corner
// with s the tet's place in the part that owns v, 0xffff beyond the end.
__global__ void __launch_bounds__(256) k_relax_inc(MeshView m, const int4 *__restrict__ cells, int cs,
                                                   const int *__restrict__ slot, uint4 *inc) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    const int v = g >> 2, lane = g & 3;
    if (v >= m.V) return;
    const int4 cell = cells[__float_as_int(__ldg(m.xr + v).w)];
    int r = 0;
    while (v >= part_begin(cell.x, cell.y, r + 1, cs)) ++r;
    const int e0 = m.csr_ptr[v] + lane, e1 = m.csr_ptr[v + 1];
    unsigned q[8];
    for (int k = 0; k < 8; ++k) {
        const int e = e0 + 4 * k, id = e < e1 ? m.csr_idx[e] : 0;
        q[k] = e < e1 ? (unsigned)(slot[(size_t)r * m.T + (id >> 2)] << 2 | (id & 3)) : 0xffffu;
    }
    inc[g] = make_uint4(q[0] | q[1] << 16, q[2] | q[3] << 16, q[4] | q[5] << 16, q[6] | q[7] << 16);
}

cudaError_t launch_relax_count(const MeshView &m, const int4 *cells, int ncells, int *counts, int *degree,
                               cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(degree, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    k_relax_count<<<15 * ncells, 256, 0, s>>>(m, cells, counts, degree);
    return cudaGetLastError();
}

cudaError_t launch_relax_fill(const MeshView &m, const RelaxPart *parts, int nparts, int cs, const int4 *cells,
                              float4 *rows, int NT, int *list, int *slot, uint4 *inc, cudaStream_t s) {
    k_relax_fill<<<nparts, 1024, 0, s>>>(m, parts, cs, cells, rows, NT, list, slot);
    k_relax_inc<<<(int)((4LL * m.V + 255) / 256), 256, 0, s>>>(m, cells, cs, slot, inc);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- steps
// The displacements of a tet's corners and its B, V0 from the packed rows.
struct PackedTet {
    float4 b0, b1, b2;
};

__device__ __forceinline__ PackedTet load_packed(const RelaxPlan &pl, int i) {
    return {__ldg(pl.rows + i), __ldg(pl.rows + pl.NT + i), __ldg(pl.rows + 2 * (size_t)pl.NT + i)};
}

__device__ __forceinline__ void unpack_rows(const PackedTet &q, float (&Bm)[3][3], float &V0, int (&c)[4]) {
    Bm[0][0] = q.b0.x; Bm[0][1] = q.b0.y; Bm[0][2] = q.b0.z;
    Bm[1][0] = q.b1.x; Bm[1][1] = q.b1.y; Bm[1][2] = q.b1.z;
    Bm[2][0] = q.b2.x; Bm[2][1] = q.b2.y; Bm[2][2] = q.b2.z;
    V0 = q.b0.w;
    const unsigned a = __float_as_uint(q.b1.w), b = __float_as_uint(q.b2.w);
    c[0] = a & 0xffffu;
    c[1] = a >> 16;
    c[2] = b & 0xffffu;
    c[3] = b >> 16;
}

// Sum of the corner values of a vertex over the four lanes (every lane ends
// with it), in the order of gather_vertex. fc[9 s + 3 a + i] holds component i
// at corner a of the part's tet s; corner 3 is -((f0 + f1) + f2).
__device__ __forceinline__ void sum_incidences(const uint4 &e, const float *fc, float &fx, float &fy, float &fz) {
    fx = fy = fz = 0.f;
    const unsigned w[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const unsigned id = (w[k >> 1] >> (16 * (k & 1))) & 0xffffu;
        if (id == 0xffffu) break;
        const int a = id & 3;
        const float *f = fc + 9 * (id >> 2) + 3 * (a < 3 ? a : 0);
        float x = f[0], y = f[1], z = f[2];
        if (a == 3) {
            x = -__fadd_rn(__fadd_rn(x, f[3]), f[6]);
            y = -__fadd_rn(__fadd_rn(y, f[4]), f[7]);
            z = -__fadd_rn(__fadd_rn(z, f[5]), f[8]);
        }
        fx += x;
        fy += y;
        fz += z;
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        fx += __shfl_xor_sync(0xffffffffu, fx, o);
        fy += __shfl_xor_sync(0xffffffffu, fy, o);
        fz += __shfl_xor_sync(0xffffffffu, fz, o);
    }
}

// n damped steps of all cells from (u_in, v_in) to (u_out, v_out), which may be
// the same arrays. ckpt (may be null) receives the state before the first step
// (displacements, then velocities); trail (may be null) the displacements
// after every step but the last, step i at trail + (i + 1) V; fv (may be null) the elastic
// forces of the last step. The last step's displacements go to u_out alone.
__global__ void __launch_bounds__(kStepBlock, 1)
    k_relax_cells(RelaxPlan pl, MeshView m, const float4 *u_in, const float4 *v_in, float4 *u_out, float4 *v_out,
                  float4 *ckpt, float4 *trail, float4 *fv, int n, float dt, float c, float kp,
                  const float *__restrict__ zlo, const float *__restrict__ zhi, unsigned *err) {
    // [vertices of the cell] displacements, [own] velocities, the corner forces
    extern __shared__ float4 su[];
    const cg::cluster_group cluster = cg::this_cluster();
    const RelaxPart p = pl.parts[blockIdx.x];
    float4 *sv = su + p.cell_nv;
    float *fc = reinterpret_cast<float *>(sv + p.nv);
    const int lane = threadIdx.x & 3;
    const float4 cell_mat = __ldg(m.mat + p.cell);
    const bool by_index = pl.per_tet || needs_fp64_volume(m, cell_mat);
    const PlateZ pz = plates_of(m, p.cell, zlo, zhi);
    for (int j = threadIdx.x; j < p.cell_nv; j += kStepBlock) su[j] = u_in[p.cell_v0 + j];
    for (int j = threadIdx.x; j < p.nv; j += kStepBlock) {
        const int v = p.v0 + j;
        const float4 vel = v_in[v];
        sv[j] = vel;
        if (ckpt) {
            ckpt[v] = u_in[v];
            ckpt[m.V + v] = vel;
        }
    }
    __syncthreads();
    for (int step = 0; step < n; ++step) {
        // the displacements of the step before, here rather than where they
        // are made: a store that is still on its way holds up a barrier's release
        if (trail && step > 0)
            for (int j = threadIdx.x; j < p.nv; j += kStepBlock)
                trail[(size_t)step * m.V + p.v0 + j] = su[p.v0 - p.cell_v0 + j];
#pragma unroll 1
        for (int i = threadIdx.x; i < p.nt; i += kStepBlock) {
            TetIn in;
            int a[4];
            unpack_rows(load_packed(pl, p.t0 + i), in.Bm, in.V0, a);
#pragma unroll
            for (int k = 0; k < 4; ++k) in.w[k] = su[a[k]];
            int t = 0;  // only per-tet materials and the FP64 volume need the tet's index
            if (by_index) t = __ldg(pl.list + p.t0 + i) & INT_MAX;
            in.mat = pl.per_tet ? __ldg(m.mat + __ldg(m.tmat + t)) : cell_mat;
            float f[4][3];
            tet_corners<true>(m, in, err, t, f);
#pragma unroll
            for (int k = 0; k < 9; ++k) fc[9 * i + k] = f[k / 3][k % 3];
        }
        // first rows before the barrier, so that their latency hides under it
        uint4 e = make_uint4(~0u, ~0u, ~0u, ~0u);
        float z0 = 0.f;
        auto fetch = [&](int j) {
            if (j < p.nv) {
                e = __ldg(pl.inc + 4 * (size_t)(p.v0 + j) + lane);
                z0 = __ldg(m.xr + p.v0 + j).z;
            } else {
                e = make_uint4(~0u, ~0u, ~0u, ~0u);
            }
        };
        fetch(threadIdx.x >> 2);
        cluster.barrier_arrive();
        __syncthreads();
        for (int j0 = 0; j0 == 0 || j0 < p.nv; j0 += kStepBlock / 4) {
            const int j = j0 + (threadIdx.x >> 2), v = p.v0 + j, local = v - p.cell_v0;
            const uint4 ee = e;
            const float zr = z0;
            if (j0 + kStepBlock / 4 < p.nv) fetch(j + kStepBlock / 4);
            float fx, fy, fz;
            sum_incidences(ee, fc, fx, fy, fz);
            const bool live = j < p.nv;
            float4 un = make_float4(0.f, 0.f, 0.f, 0.f), vn = un;
            if (live) plate_move(su[local], sv[j], make_float4(fx, fy, fz, 0.f), zr, pz, dt, c, kp, un, vn);
            if (j0 == 0) cluster.barrier_wait();  // every block is done with the old displacements
            __syncwarp();                         // the four lanes have read theirs
            if (!live) continue;
            for (int r = lane; r < pl.cs; r += 4) *cluster.map_shared_rank(su + local, r) = un;
            if (lane == 0) {
                if (!isfinite(fx + fy + fz) || !isfinite(un.x + un.y + un.z)) atomicOr(err, ERR_NONFINITE);
                sv[j] = vn;
            } else if (step == n - 1) {
                if (lane == 1) u_out[v] = un;
                if (lane == 2) v_out[v] = vn;
                if (lane == 3 && fv) fv[v] = make_float4(fx, fy, fz, 0.f);
            }
        }
        cluster.sync();  // the new displacements are everywhere
    }
}

// The n reverse steps of a segment, last first, from the displacements y at
// the start of each (y + i V), on the adjoint state (ly, lv) in place:
// m = dt ly + lv, ly += dt (J_el + J_plate) m, lv = c m; and the cells'
// gradients += dt m . df/d(mu, kappa, w).
__global__ void __launch_bounds__(kReverseBlock, 1)
    k_relax_reverse(RelaxPlan pl, MeshView m, const float4 *__restrict__ y, float4 *ly, float4 *lv, int n, float dt,
                    float c, float kp, const float *__restrict__ zlo, const float *__restrict__ zhi, double *grad,
                    unsigned *err) {
    extern __shared__ float4 su[];  // [vertices of the cell] displacements, then m, then the corner tangents
    __shared__ Sum2 part[3][kReverseBlock / 32];
    __shared__ float warp_top[kReverseBlock / 32];
    const cg::cluster_group cluster = cg::this_cluster();
    const RelaxPart p = pl.parts[blockIdx.x];
    float4 *sm = su + p.cell_nv;
    float *fc = reinterpret_cast<float *>(sm + p.cell_nv);
    const int lane = threadIdx.x & 3;
    const float4 mat = __ldg(m.mat + p.cell);
    const PlateZ pz = plates_of(m, p.cell, zlo, zhi);
    float top = 0.f;
    for (int j = threadIdx.x; j < p.cell_nv; j += kReverseBlock) {
        const int v = p.cell_v0 + j;
        su[j] = __ldg(y + (size_t)(n - 1) * m.V + v);
        const float4 a = ly[v], b = lv[v];
        sm[j] = make_float4(fmaf(dt, a.x, b.x), fmaf(dt, a.y, b.y), fmaf(dt, a.z, b.z), 0.f);
        top = largest(sm[j], top);
    }
    // m and the tangents are held times 2^(127 - b), see direction_exponent;
    // every block of the cluster has read the whole cell, so they agree on b
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    if ((threadIdx.x & 31) == 0) warp_top[threadIdx.x >> 5] = top;
    __syncthreads();
    for (int w = 0; w < kReverseBlock / 32; ++w) top = fmaxf(top, warp_top[w]);
    const int b2 = direction_exponent(top);
    const float down = power_of_two(254 - b2), up = power_of_two(b2);
    for (int j = threadIdx.x; j < p.cell_nv; j += kReverseBlock) sm[j] = times(sm[j], down);
    cluster.sync();  // ly, lv are read before any block changes them
    Sum2 g[3];
    for (int step = n - 1; step >= 0; --step) {
        if ((int)threadIdx.x < p.nt) {
            PackedTet q = load_packed(pl, p.t0 + threadIdx.x);
#pragma unroll 1
            for (int i = threadIdx.x; i < p.nt; i += kReverseBlock) {
                const PackedTet now = q;
                if (i + kReverseBlock < p.nt) q = load_packed(pl, p.t0 + i + kReverseBlock);
                float Bm[3][3], V0, H[3][3], dH[3][3], f[4][3], gt[3];
                int a[4];
                unpack_rows(now, Bm, V0, a);
                tet_grad(su[a[0]], su[a[1]], su[a[2]], su[a[3]], Bm, H);
                tet_grad(sm[a[0]], sm[a[1]], sm[a[2]], sm[a[3]], Bm, dH);
                InvT<float> inv;
                tet_tangent(H, dH, mat, Bm, V0, inv, f);
                if (pl.list[p.t0 + i] >= 0) {
                    mr_energy_rates(H, dH, inv, gt);
#pragma unroll
                    for (int k = 0; k < 3; ++k) g[k].add(-V0 * gt[k]);
                }
#pragma unroll
                for (int k = 0; k < 9; ++k) fc[9 * i + k] = f[k / 3][k % 3];
            }
        }
        cluster.barrier_arrive();
        __syncthreads();
        const float4 *now = y + (size_t)step * m.V;
        if (step > 0)  // the next displacements (this block's copy; its tets are done)
            for (int j = threadIdx.x; j < p.cell_nv; j += kReverseBlock) su[j] = __ldg(now - m.V + p.cell_v0 + j);
        for (int j0 = 0; j0 == 0 || j0 < p.nv; j0 += kReverseBlock / 4) {
            const int j = j0 + (threadIdx.x >> 2), v = p.v0 + j, local = v - p.cell_v0;
            const bool live = j < p.nv;
            const uint4 e = live ? __ldg(pl.inc + 4 * (size_t)v + lane) : make_uint4(~0u, ~0u, ~0u, ~0u);
            float jx, jy, jz;
            sum_incidences(e, fc, jx, jy, jz);
            jx *= up, jy *= up, jz *= up;
            float4 a, b, mn = make_float4(0.f, 0.f, 0.f, 0.f);
            if (live) {
                const float z = __ldg(m.xr + v).z + __ldg(now + v).z;
                adjoint_move(ly[v], make_float4(jx, jy, jz, 0.f), times(sm[local], up), z, pz, dt, c, kp, a, b, mn);
                mn = times(mn, down);
            }
            if (j0 == 0) cluster.barrier_wait();  // every block is done with the old m
            __syncwarp();                         // the four lanes have read ly
            if (!live) continue;
            for (int r = lane; r < pl.cs; r += 4) *cluster.map_shared_rank(sm + local, r) = mn;
            if (lane == 0) {
                ly[v] = a;
                if (!isfinite(jx + jy + jz)) atomicOr(err, ERR_NONFINITE);  // as the general path's vertex sums
            }
            if (lane == 1) lv[v] = b;
        }
        cluster.sync();
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        warp_sum(g[k]);
        if ((threadIdx.x & 31) == 0) part[k][threadIdx.x >> 5] = g[k];
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    double G = 0.0;
    if (threadIdx.x < 3)
        for (int w = 0; w < kReverseBlock / 32; ++w) G += part[threadIdx.x][w].value();
    G *= power_of_two_64(b2);
    const double G0 = __shfl_sync(0xffffffffu, G, 0), G1 = __shfl_sync(0xffffffffu, G, 1);
    if (threadIdx.x < 3) add_moduli_rate(threadIdx.x, G0, G1, G, mat, (double)dt, grad + 3 * p.cell);
}

// ---------------------------------------------------------------- launchers
size_t relax_smem(int cell_nv, int nv, int nt, bool reverse) {
    return sizeof(float4) * ((size_t)cell_nv * (reverse ? 2 : 1) + (reverse ? 0 : nv)) + sizeof(float) * 9 * (size_t)nt;
}

cudaError_t prepare_relax(int smem_max) {
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute(k_relax_cells, a, smem_max);
    return e == cudaSuccess ? cudaFuncSetAttribute(k_relax_reverse, a, smem_max - kRelaxStatic) : e;
}

static cudaLaunchConfig_t relax_config(const RelaxPlan &pl, int block, size_t smem, cudaLaunchAttribute *attr, cudaStream_t s) {
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = pl.cs;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(pl.nparts);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

cudaError_t launch_relax_cells(const RelaxPlan &pl, const MeshView &m, const float4 *u_in, const float4 *v_in,
                               float4 *u_out, float4 *v_out, float4 *ckpt, float4 *trail, float4 *fv, int n, float dt,
                               float c, float kp, const float *zlo, const float *zhi, unsigned *err, cudaStream_t s) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = relax_config(pl, kStepBlock, pl.smem_step, &attr, s);
    return cudaLaunchKernelEx(&cfg, k_relax_cells, pl, m, u_in, v_in, u_out, v_out, ckpt, trail, fv, n, dt, c, kp, zlo,
                              zhi, err);
}

cudaError_t launch_relax_reverse(const RelaxPlan &pl, const MeshView &m, const float4 *y, float4 *ly, float4 *lv, int n,
                                 float dt, float c, float kp, const float *zlo, const float *zhi, double *grad,
                                 unsigned *err, cudaStream_t s) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = relax_config(pl, kReverseBlock, pl.smem_reverse, &attr, s);
    return cudaLaunchKernelEx(&cfg, k_relax_reverse, pl, m, y, ly, lv, n, dt, c, kp, zlo, zhi, grad, err);
}

// Clusters of the plan that can be resident at a time (a cluster's blocks must
// be at once); 0: none.
int relax_clusters(const RelaxPlan &pl) {
    cudaLaunchAttribute attr;
    int a = 0, b = 0;
    const cudaLaunchConfig_t f = relax_config(pl, kStepBlock, pl.smem_step, &attr, nullptr);
    if (cudaOccupancyMaxActiveClusters(&a, k_relax_cells, &f) != cudaSuccess) a = 0;
    const cudaLaunchConfig_t r = relax_config(pl, kReverseBlock, pl.smem_reverse, &attr, nullptr);
    if (cudaOccupancyMaxActiveClusters(&b, k_relax_reverse, &r) != cudaSuccess) b = 0;
    cudaGetLastError();
    return a < b ? a : b;
}

}  // namespace cf
