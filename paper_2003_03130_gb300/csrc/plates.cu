// C ABI of the compression set-up (cells between two plates, no fluid) and
// of its adjoint: cf_plates_set, cf_relax, cf_plate_force, cf_tape_clear,
// cf_relax_adjoint, cf_adjoint_gradients, cf_force_jvp, cf_force_param_vjp.
//
// Relaxation steps (unit-mass vertices): v <- c v + dt (f_el + f_plate),
// y <- y + dt v. A recorded cf_relax call appends a tape entry and keeps
// device checkpoints of (y, v) every kTapeStride steps and at its end.
// cf_relax_adjoint reverses the last entry: it adds dL/dF * dF/dy to lambda_y
// (F = top-plate force at the end of that call), then, segment by segment from
// the last, restores the checkpoint, recomputes the segment's states, and
// walks it backwards with m = dt lambda_y + lambda_v:
//   lambda_y <- lambda_y + dt (J_el + J_plate) m, lambda_v <- c m,
// accumulating dt m . df/d(mu, kappa, w) per cell in double.
#include <algorithm>
#include <cmath>
#include <functional>
#include <new>
#include <queue>

#include "ctx.h"

namespace {

constexpr int kTapeStride = 50;
constexpr int kRelaxSteps = 1000;  // steps of one launch, at most (3 to 20 ms a wave of cells)
// Steps in launches of their own before the on-chip plan is made, which takes
// 60 us (a cell of 192 tets) to 350 (64 of 8.3 k) once per mesh: a mesh that is
// relaxed by a few steps need not pay it (a first call of one step 24 to 82 us,
// with the plan 80 to 440). A first call of 32 steps is at worst 8 % longer than
// in launches (200 cells of 1.2 k tets: 705 and 655 us), one of 64 never.
constexpr int kPlanSteps = 32;

void free_adjoint(cf_ctx *c) {
    for (auto *p : c->ckpt) cudaFree(p);
    c->ckpt.clear();
    c->ck_used = 0;
    c->tape.clear();
    ++c->tape_gen;
    dfree(c->vel_r);
    dfree(c->lam);
    dfree(c->lamv);
    dfree(c->mvec);
    dfree(c->jv);
    dfree(c->vtmp);
    dfree(c->seg);
    dfree(c->segv);
    dfree(c->grad);
    dfree(c->gtmp);
    dfree(c->pforce);
    dfree(c->dF);
    dfree(c->zlo);
    dfree(c->zhi);
    cf_free_plan(c);
    c->plan_steps = 0;
    c->adj_V = c->adj_C = 0;
}

// Buffers sized for the current mesh (reallocated, and the tape dropped, when
// cells were added since).
cf_status ensure_adjoint(cf_ctx *c) {
    const int C = (int)c->cells.size();
    if (c->adj_V == c->V && c->adj_C == C) return CF_OK;
    std::vector<float> zlo = c->zlo_h, zhi = c->zhi_h;
    free_adjoint(c);
    CUDA_TRY(c, dalloc(&c->vel_r, c->V));
    CUDA_TRY(c, dalloc(&c->lam, c->V));
    CUDA_TRY(c, dalloc(&c->lamv, c->V));
    CUDA_TRY(c, dalloc(&c->mvec, c->V));
    CUDA_TRY(c, dalloc(&c->jv, c->V));
    CUDA_TRY(c, dalloc(&c->vtmp, c->V));
    CUDA_TRY(c, dalloc(&c->seg, (size_t)(kTapeStride + 1) * c->V));
    CUDA_TRY(c, dalloc(&c->segv, (size_t)(kTapeStride + 1) * c->V));
    CUDA_TRY(c, dalloc(&c->grad, 3 * (size_t)C));
    CUDA_TRY(c, dalloc(&c->gtmp, 3 * (size_t)C));
    CUDA_TRY(c, dalloc(&c->pforce, C));
    CUDA_TRY(c, dalloc(&c->dF, C));
    CUDA_TRY(c, dalloc(&c->zlo, C));
    CUDA_TRY(c, dalloc(&c->zhi, C));
    CUDA_TRY(c, cudaMemsetAsync(c->vel_r, 0, sizeof(float4) * c->V, c->stream));
    CUDA_TRY(c, cudaMemsetAsync(c->lam, 0, sizeof(float4) * c->V, c->stream));
    CUDA_TRY(c, cudaMemsetAsync(c->lamv, 0, sizeof(float4) * c->V, c->stream));
    CUDA_TRY(c, cudaMemsetAsync(c->grad, 0, sizeof(double) * 3 * C, c->stream));
    c->adj_V = c->V;
    c->adj_C = C;
    if ((int)zlo.size() == C) {
        c->zlo_h = zlo;
        c->zhi_h = zhi;
        CUDA_TRY(c, cudaMemcpyAsync(c->zlo, zlo.data(), sizeof(float) * C, cudaMemcpyHostToDevice, c->stream));
        CUDA_TRY(c, cudaMemcpyAsync(c->zhi, zhi.data(), sizeof(float) * C, cudaMemcpyHostToDevice, c->stream));
    } else {
        c->zlo_h.clear();
        c->zhi_h.clear();
    }
    return CF_OK;
}

// Time of a step on chip and of a step in launches of their own, microseconds:
// a + tet t + vertex v, for the tets of a cell's largest block (a cluster's
// step) or for all tets and vertices (the launches of a step, bound by their
// latency up to some 50 k tets: `least`). Fitted to 110 sets of cells on GB300
// (1 to 2,000 cells of 192 to 13.6 k tets, equal ones and one large cell among
// small ones), which they meet within 19 %; a reverse step includes the
// recomputed forward one.
struct StepTime {
    double least, a, tet, vertex;
};
constexpr StepTime kChipStep{0.0, 2.15, 2.92e-3, 0.0}, kChipReverse{0.0, 4.9, 8.6e-3, 0.0};
constexpr StepTime kLaunchStep{12.4, 10.9, 3.4e-5, 1.8e-5}, kLaunchReverse{25.0, 25.8, 5.9e-5, 1.47e-4};
// A launch on chip takes 2 us more than its steps, and each wave of cells 4 (the
// state of a cell, read and written): a call of one step of 8.3 k tets 20.9 us,
// in launches 19.8.
constexpr double kChipCall = 2.0, kChipWave = 4.0;

double step_time(const StepTime &q, double nt, double nv) {
    return std::max(q.least, q.a + q.tet * nt + q.vertex * nv);
}

// Time of a step on chip of cells whose largest blocks hold nt tets, `slots`
// clusters at a time, the next cell on the slot that is free first.
double on_chip_time(const StepTime &q, const std::vector<int> &nt, int slots) {
    std::priority_queue<double, std::vector<double>, std::greater<double>> busy;
    double end = 0.0;
    for (const int n : nt) {
        double t = step_time(q, n, 0);
        if ((int)busy.size() == slots) {
            t += busy.top();
            busy.pop();
        }
        busy.push(t);
        end = std::max(end, t);
    }
    return end;
}

struct PlanScratch {
    int4 *cells = nullptr;
    int *counts = nullptr, *slot = nullptr;
    ~PlanScratch() {
        dfree(cells);
        dfree(counts);
        dfree(slot);
    }
};

// The on-chip relaxation's plan for the current mesh, if it fits and is
// expected to be faster: cells cut into `cs` blocks, the fewest that hold a
// part in shared memory; more, up to eight, while every block still gets an SM
// of its own and a part has more than kRelaxRound tets. The cells of a mesh
// share cs, and a block has its SM to itself, so many small cells run in
// waves, and one large cell cuts the small ones beside it too. Steps and
// reverse steps go on chip each where the estimates above say so. Measured,
// on chip against three launches a step: 64 cells of 8.3 k tets 16.3 and 28.9
// us, reverse steps 47 and 70; 2,000 cells of 192 tets 36.9 and 25.8, reverse
// 88 and 66; 300 of 192 beside one of 13.6 k 50 and 14.5, reverse 121 and 35.
// plan_state: 1 with the plan, 2 if the mesh takes the launches.
cudaError_t build_plan(cf_ctx *c) {
    const int C = (int)c->cells.size();
    std::vector<int4> cells(C);
    c->plan_state = 2;
    for (int k = 0; k < C; ++k) {
        const CellInfo &ci = c->cells[k];
        if (ci.nv > 0xffff) return cudaSuccess;
        cells[k] = make_int4(ci.v_off, ci.nv, ci.t_off, ci.nt);
    }
    if (C > INT_MAX / 15) return cudaSuccess;
    int smem = 0;
    cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device);
    if (smem <= kRelaxStatic || prepare_relax(smem) != cudaSuccess) {
        cudaGetLastError();
        return cudaSuccess;
    }
    for (const int4 &q : cells)  // some block of eight holds an eighth of a cell's tets or more
        if (relax_smem(q.y, q.y, (q.w + 7) / 8, true) > (size_t)(smem - kRelaxStatic)) return cudaSuccess;
    const MeshView m = view(c);
    PlanScratch d;
#define TRY_P(expr)                                \
    do {                                           \
        const cudaError_t e_ = (expr);             \
        if (e_ != cudaSuccess) return e_;          \
    } while (0)
    TRY_P(dalloc(&d.cells, C));
    TRY_P(dalloc(&d.counts, 15 * (size_t)C + 1));
    TRY_P(cudaMemcpyAsync(d.cells, cells.data(), sizeof(int4) * C, cudaMemcpyHostToDevice, c->stream));
    TRY_P(launch_relax_count(m, d.cells, C, d.counts, d.counts + 15 * (size_t)C, c->stream));
    std::vector<int> counts(15 * (size_t)C + 1);
    TRY_P(cudaMemcpyAsync(counts.data(), d.counts, sizeof(int) * counts.size(), cudaMemcpyDeviceToHost, c->stream));
    TRY_P(cudaStreamSynchronize(c->stream));
    if (counts.back() > kRelaxDegree) return cudaSuccess;
    std::vector<int> most_of(C);  // tets of a cell's largest block
    auto largest = [&](int cs, bool &fits) {
        fits = true;
        for (int k = 0; k < C; ++k) {
            const int *n = counts.data() + 15 * (size_t)k + cs - 1;
            most_of[k] = *std::max_element(n, n + cs);
            if (relax_smem(cells[k].y, cells[k].y, most_of[k], true) > (size_t)(smem - kRelaxStatic)) fits = false;
        }
        return *std::max_element(most_of.begin(), most_of.end());
    };
    int cs = 1;
    bool fits = false;
    while (largest(cs, fits), !fits && cs < 8) cs *= 2;
    if (!fits) return cudaSuccess;
    while (cs < 8 && 2LL * cs * C <= c->sms && largest(cs, fits) > kRelaxRound) cs *= 2;
    RelaxPlan pl{};
    pl.cs = cs;
    pl.nparts = cs * C;
    std::vector<RelaxPart> parts(pl.nparts);
    long long nt_all = 0;
    for (int k = 0; k < C; ++k)
        for (int r = 0; r < cs; ++r) {
            RelaxPart &q = parts[(size_t)cs * k + r];
            q.cell = k;
            q.cell_v0 = cells[k].x;
            q.cell_nv = cells[k].y;
            q.v0 = cells[k].x + (int)((long long)cells[k].y * r / cs);
            q.nv = cells[k].x + (int)((long long)cells[k].y * (r + 1) / cs) - q.v0;
            q.t0 = (int)nt_all;
            q.nt = counts[15 * (size_t)k + cs - 1 + r];
            nt_all += q.nt;
            pl.smem_step = std::max(pl.smem_step, relax_smem(q.cell_nv, q.nv, q.nt, false));
            pl.smem_reverse = std::max(pl.smem_reverse, relax_smem(q.cell_nv, q.nv, q.nt, true));
        }
    if (nt_all > INT_MAX) return cudaSuccess;
    pl.NT = (int)nt_all;
    const int slots = relax_clusters(pl);
    if (slots == 0) return cudaSuccess;
    largest(cs, fits);
    const double gain = step_time(kLaunchStep, c->T, c->V) - on_chip_time(kChipStep, most_of, slots);
    const double call = kChipCall + kChipWave * ((C + slots - 1) / slots);
    pl.from = gain > 0.0 ? (int)std::min(1e9, 1.0 + std::floor(call / gain)) : INT_MAX;
    pl.reverse = on_chip_time(kChipReverse, most_of, slots) < step_time(kLaunchReverse, c->T, c->V);
    if (pl.from == INT_MAX && !pl.reverse) return cudaSuccess;
    TRY_P(dalloc(&c->plan_parts, parts.size()));
    TRY_P(dalloc(&c->plan_rows, 3 * (size_t)pl.NT));
    TRY_P(dalloc(&c->plan_list, pl.NT));
    TRY_P(dalloc(&c->plan_inc, 4 * (size_t)c->V));
    TRY_P(dalloc(&d.slot, (size_t)cs * c->T));
    TRY_P(cudaMemcpyAsync(c->plan_parts, parts.data(), sizeof(RelaxPart) * parts.size(), cudaMemcpyHostToDevice,
                          c->stream));
    TRY_P(launch_relax_fill(m, c->plan_parts, pl.nparts, cs, d.cells, c->plan_rows, pl.NT, c->plan_list, d.slot,
                            c->plan_inc, c->stream));
    TRY_P(cudaStreamSynchronize(c->stream));  // the host vectors and the scratch go
#undef TRY_P
    pl.parts = c->plan_parts;
    pl.rows = c->plan_rows;
    pl.list = c->plan_list;
    pl.inc = c->plan_inc;
    c->plan = pl;
    c->plan_state = 1;
    return cudaSuccess;
}

// Without memory for a plan the launches are taken, and the next call tries
// again.
cf_status make_plan(cf_ctx *c) {
    if (c->plan_state) return CF_OK;
    cudaError_t e;
    try {
        e = build_plan(c);
    } catch (const std::bad_alloc &) {
        e = cudaErrorMemoryAllocation;
    }
    if (c->plan_state == 1) return CF_OK;
    const int state = e == cudaSuccess ? c->plan_state : 0;
    cf_free_plan(c);
    c->plan_state = state;
    if (e == cudaErrorMemoryAllocation) cudaGetLastError();
    return e == cudaSuccess || e == cudaErrorMemoryAllocation
               ? CF_OK
               : fail(c, CF_ECUDA, "relaxation plan: %s", cudaGetErrorString(e));
}

// The plan before n more steps are taken, once enough of them are.
cf_status plan_before(cf_ctx *c, long long n) {
    if (c->plan_state) return CF_OK;
    c->plan_steps = std::min(c->plan_steps + n, (long long)kPlanSteps);
    return c->plan_steps < kPlanSteps ? CF_OK : make_plan(c);
}

// The plan if the mesh has one that takes n steps (reverse: n reverse steps) on
// chip, with the materials' present form.
const RelaxPlan *plan_of(cf_ctx *c, bool reverse, int n) {
    if (c->plan_state != 1 || !(reverse ? c->plan.reverse : n >= c->plan.from)) return nullptr;
    c->plan.per_tet = 0;
    for (const CellInfo &ci : c->cells) c->plan.per_tet |= ci.per_tet;
    return &c->plan;
}

cf_status upload_plates(cf_ctx *c, const std::vector<float> &zlo, const std::vector<float> &zhi) {
    CUDA_TRY(c, cudaMemcpyAsync(c->zlo, zlo.data(), sizeof(float) * zlo.size(), cudaMemcpyHostToDevice, c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(c->zhi, zhi.data(), sizeof(float) * zhi.size(), cudaMemcpyHostToDevice, c->stream));
    return CF_OK;
}

// forces at u into c->fv, then one damped step (u_in, v_in) -> (u_out, v_out)
cf_status relax_step(cf_ctx *c, const MeshView &m, const float4 *u_in, const float4 *v_in, float4 *u_out,
                     float4 *v_out, float dt, float cd, float kp) {
    CUDA_TRY(c, launch_tet_force(m, u_in, c->d_err, c->stream));
    CUDA_TRY(c, launch_gather_spread(m, u_in, nullptr, nullptr, c->d_err, c->stream));
    CUDA_TRY(c, launch_plate_step(m, u_in, v_in, c->fv, u_out, v_out, dt, cd, kp, c->zlo, c->zhi, c->d_err,
                                  c->stream));
    return CF_OK;
}

cf_status save_state(cf_ctx *c, float4 *dst, const float4 *u, const float4 *v) {
    CUDA_TRY(c, cudaMemcpyAsync(dst, u, sizeof(float4) * c->V, cudaMemcpyDeviceToDevice, c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(dst + c->V, v, sizeof(float4) * c->V, cudaMemcpyDeviceToDevice, c->stream));
    return CF_OK;
}

cf_status need_cells(cf_ctx *c) {
    if (!c) return CF_EINVAL;
    if (c->T == 0) return fail(c, CF_ESTATE, "no cells");
    return ensure_adjoint(c);
}

// The parameter gradients are per cell: a cell whose tets carry their own
// materials has no single (mu, kappa, w) to differentiate.
cf_status need_uniform_materials(cf_ctx *c) {
    for (size_t i = 0; i < c->cells.size(); ++i)
        if (c->cells[i].per_tet)
            return fail(c, CF_ESTATE, "cell %zu has per-tet materials: parameter gradients are per cell", i);
    return CF_OK;
}

}  // namespace

extern "C" {

cf_status cf_plates_set(cf_ctx *c, double k_plate, const double *z_lo, const double *z_hi) {
    cf_status st = need_cells(c);
    if (st != CF_OK) return st;
    DeviceGuard dg(c->device);
    const int C = (int)c->cells.size();
    if (!z_lo || !z_hi || !(k_plate >= 0.0) || !std::isfinite(k_plate)) return fail(c, CF_EINVAL, "bad plates");
    std::vector<float> lo(C), hi(C);
    for (int i = 0; i < C; ++i) {
        if (!(std::isfinite(z_lo[i]) && std::isfinite(z_hi[i]) && z_lo[i] < z_hi[i]))
            return fail(c, CF_EINVAL, "cell %d: need finite plates with z_lo < z_hi", i);
        lo[i] = (float)z_lo[i];
        hi[i] = (float)z_hi[i];
    }
    c->k_plate = (float)k_plate;
    c->zlo_h = lo;
    c->zhi_h = hi;
    st = upload_plates(c, lo, hi);
    return st != CF_OK ? st : wait_stream(c);
}

cf_status cf_relax(cf_ctx *c, int32_t n, double dt, double damping, int32_t record) {
    cf_status st = need_cells(c);
    if (st != CF_OK) return st;
    DeviceGuard dg(c->device);
    if ((int)c->zlo_h.size() != (int)c->cells.size()) return fail(c, CF_ESTATE, "call cf_plates_set first");
    if (n < 1 || !(dt > 0.0) || !std::isfinite(dt)) return fail(c, CF_EINVAL, "need n >= 1 and dt > 0");
    if (!(damping >= 0.0 && damping < 1.0)) return fail(c, CF_EINVAL, "need 0 <= damping < 1");
    const MeshView m = view(c);
    float4 *u = c->u[c->cur];
    const float cd = (float)damping;
    cf_ctx::TapeEntry e{};
    if (record) {
        e.n = n;
        e.dt = (float)dt;
        e.c = cd;
        e.kp = c->k_plate;
        e.zlo = c->zlo_h;
        e.zhi = c->zhi_h;
        e.ck0 = c->ck_used;
        e.nck = (n - 1) / kTapeStride + 2;
        for (const CellInfo &ci : c->cells) e.mats.push_back(ci.mat);
        while ((int)c->ckpt.size() < e.ck0 + e.nck) {
            float4 *p = nullptr;
            CUDA_TRY(c, dalloc_spare(c, &p, 2 * (size_t)c->V));
            c->ckpt.push_back(p);
        }
    }
    st = plan_before(c, n);
    if (st != CF_OK) return st;
    const RelaxPlan *pl = plan_of(c, false, n);
    for (int k = 0; pl && k < n;) {  // on chip: a launch per checkpoint, or per kRelaxSteps
        const int b = std::min(record ? kTapeStride : kRelaxSteps, n - k);
        CUDA_TRY(c, launch_relax_cells(*pl, m, u, c->vel_r, u, c->vel_r,
                                       record ? c->ckpt[e.ck0 + k / kTapeStride] : nullptr, nullptr,
                                       k + b == n ? c->fv : nullptr, b, (float)dt, cd, c->k_plate, c->zlo, c->zhi,
                                       c->d_err, c->stream));
        k += b;
    }
    for (int k = 0; !pl && k < n; ++k) {
        if (record && k % kTapeStride == 0) {
            st = save_state(c, c->ckpt[e.ck0 + k / kTapeStride], u, c->vel_r);
            if (st != CF_OK) return st;
        }
        st = relax_step(c, m, u, c->vel_r, u, c->vel_r, (float)dt, cd, c->k_plate);
        if (st != CF_OK) return st;
    }
    if (record) {
        st = save_state(c, c->ckpt[e.ck0 + e.nck - 1], u, c->vel_r);
        if (st != CF_OK) return st;
        c->ck_used = e.ck0 + e.nck;
        c->tape.push_back(e);
    }
    return consume_errors(c);
}

cf_status cf_get_relax_path(cf_ctx *c, int32_t *path) {
    cf_status st = need_cells(c);
    if (st != CF_OK) return st;
    DeviceGuard dg(c->device);
    if (!path) return fail(c, CF_EINVAL, "null output");
    st = make_plan(c);
    if (st != CF_OK) return st;
    path[0] = plan_of(c, false, kRelaxSteps) ? c->plan.cs : 0;
    path[1] = plan_of(c, true, kRelaxSteps) ? c->plan.cs : 0;
    path[2] = kRelaxSteps;
    return CF_OK;
}

cf_status cf_plate_force(cf_ctx *c, double *out) {
    cf_status st = need_cells(c);
    if (st != CF_OK) return st;
    DeviceGuard dg(c->device);
    if (!out) return fail(c, CF_EINVAL, "null output");
    if ((int)c->zlo_h.size() != (int)c->cells.size()) return fail(c, CF_ESTATE, "call cf_plates_set first");
    const int C = (int)c->cells.size();
    CUDA_TRY(c, cudaMemsetAsync(c->pforce, 0, sizeof(double) * C, c->stream));
    CUDA_TRY(c, launch_plate_force(view(c), c->u[c->cur], c->k_plate, c->zlo, c->zhi, c->pforce, c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(out, c->pforce, sizeof(double) * C, cudaMemcpyDeviceToHost, c->stream));
    return wait_stream(c);
}

cf_status cf_tape_clear(cf_ctx *c) {
    cf_status st = need_cells(c);
    if (st != CF_OK) return st;
    DeviceGuard dg(c->device);
    c->tape.clear();
    ++c->tape_gen;
    c->ck_used = 0;
    CUDA_TRY(c, cudaMemsetAsync(c->vel_r, 0, sizeof(float4) * c->V, c->stream));
    CUDA_TRY(c, cudaMemsetAsync(c->lam, 0, sizeof(float4) * c->V, c->stream));
    CUDA_TRY(c, cudaMemsetAsync(c->lamv, 0, sizeof(float4) * c->V, c->stream));
    CUDA_TRY(c, cudaMemsetAsync(c->grad, 0, sizeof(double) * 3 * c->cells.size(), c->stream));
    return wait_stream(c);
}

cf_status cf_relax_adjoint(cf_ctx *c, const double *dF) {
    cf_status st = need_cells(c);
    if (st == CF_OK) st = need_uniform_materials(c);
    if (st != CF_OK) return st;
    DeviceGuard dg(c->device);
    if (c->tape.empty()) return fail(c, CF_ESTATE, "no recorded cf_relax call left to reverse");
    if (!dF) return fail(c, CF_EINVAL, "null dF");
    const cf_ctx::TapeEntry e = c->tape.back();
    const int C = (int)c->cells.size();
    for (int k = 0; k < C; ++k) {
        const float4 a = e.mats[k], b = c->cells[k].mat;
        if (a.x != b.x || a.y != b.y || a.z != b.z || a.w != b.w)
            return fail(c, CF_ESTATE, "cell %d: materials changed since the recorded cf_relax call", k);
    }
    const MeshView m = view(c);
    st = upload_plates(c, e.zlo, e.zhi);
    if (st != CF_OK) return st;
    CUDA_TRY(c, cudaMemcpyAsync(c->dF, dF, sizeof(double) * C, cudaMemcpyHostToDevice, c->stream));
    CUDA_TRY(c, launch_adj_seed(m, c->ckpt[e.ck0 + e.nck - 1], e.kp, c->zlo, c->zhi, c->dF, c->lam, c->stream));
    st = plan_before(c, 3LL * e.n);  // a step again and its reverse, which takes two
    if (st != CF_OK) return st;
    const RelaxPlan *pl = plan_of(c, true, e.n);
    if (!pl) CUDA_TRY(c, launch_adj_m(c->V, c->lam, c->lamv, e.dt, c->mvec, c->stream));
    for (int j = e.nck - 2; j >= 0; --j) {
        const int s0 = j * kTapeStride, len = std::min(kTapeStride, e.n - s0);
        const size_t V = (size_t)c->V;
        const float4 *ck = c->ckpt[e.ck0 + j];
        CUDA_TRY(c, cudaMemcpyAsync(c->seg, ck, sizeof(float4) * V, cudaMemcpyDeviceToDevice, c->stream));
        if (pl) {
            if (len > 1)
                CUDA_TRY(c, launch_relax_cells(*pl, m, ck, ck + V, c->seg + (size_t)(len - 1) * V, c->segv, nullptr,
                                               c->seg, nullptr, len - 1, e.dt, e.c, e.kp, c->zlo, c->zhi, c->d_err,
                                               c->stream));
            CUDA_TRY(c, launch_relax_reverse(*pl, m, c->seg, c->lam, c->lamv, len, e.dt, e.c, e.kp, c->zlo, c->zhi,
                                             c->grad, c->d_err, c->stream));
            continue;
        }
        CUDA_TRY(c, cudaMemcpyAsync(c->segv, ck + V, sizeof(float4) * V, cudaMemcpyDeviceToDevice, c->stream));
        for (int i = 0; i + 1 < len; ++i) {  // states of the segment's steps
            st = relax_step(c, m, c->seg + i * V, c->segv + i * V, c->seg + (i + 1) * V, c->segv + (i + 1) * V, e.dt,
                            e.c, e.kp);
            if (st != CF_OK) return st;
        }
        for (int i = len - 1; i >= 0; --i) {
            const float4 *y = c->seg + i * V;
            CUDA_TRY(c, launch_force_jvp(m, y, c->mvec, c->jv, c->d_err, c->stream, (double)e.dt, c->grad));
            CUDA_TRY(c, launch_adj_step(m, y, c->jv, c->mvec, c->lam, c->lamv, e.dt, e.c, e.kp, c->zlo, c->zhi,
                                        c->stream));
        }
    }
    c->tape.pop_back();
    c->ck_used = e.ck0;
    st = upload_plates(c, c->zlo_h, c->zhi_h);
    if (st != CF_OK) return st;
    return consume_errors(c);
}

cf_status cf_tape_generation(cf_ctx *c, int64_t *out) {
    if (!c || !out) return CF_EINVAL;
    *out = c->tape_gen;
    return CF_OK;
}

cf_status cf_adjoint_gradients(cf_ctx *c, double *out) {
    cf_status st = need_cells(c);
    if (st == CF_OK) st = need_uniform_materials(c);
    if (st != CF_OK) return st;
    DeviceGuard dg(c->device);
    if (!out) return fail(c, CF_EINVAL, "null output");
    CUDA_TRY(c, cudaMemcpyAsync(out, c->grad, sizeof(double) * 3 * c->cells.size(), cudaMemcpyDeviceToHost,
                                c->stream));
    return wait_stream(c);
}

cf_status cf_force_jvp(cf_ctx *c, const double *v, double *out) {
    cf_status st = need_cells(c);
    if (st != CF_OK) return st;
    DeviceGuard dg(c->device);
    if (!v || !out) return fail(c, CF_EINVAL, "null array");
    CUDA_TRY(c, cudaMemcpyAsync(c->stage, v, sizeof(double) * 3 * c->V, cudaMemcpyHostToDevice, c->stream));
    CUDA_TRY(c, launch_pack3(c->stage, c->V, c->vtmp, c->stream));
    CUDA_TRY(c, launch_force_jvp(view(c), c->u[c->cur], c->vtmp, c->jv, c->d_err, c->stream));
    CUDA_TRY(c, launch_get_forces(c->jv, 0, c->V, c->stage, c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(out, c->stage, sizeof(double) * 3 * c->V, cudaMemcpyDeviceToHost, c->stream));
    return consume_errors(c);
}

cf_status cf_force_param_vjp(cf_ctx *c, const double *lam, double *out) {
    cf_status st = need_cells(c);
    if (st == CF_OK) st = need_uniform_materials(c);
    if (st != CF_OK) return st;
    DeviceGuard dg(c->device);
    if (!lam || !out) return fail(c, CF_EINVAL, "null array");
    const int C = (int)c->cells.size();
    CUDA_TRY(c, cudaMemcpyAsync(c->stage, lam, sizeof(double) * 3 * c->V, cudaMemcpyHostToDevice, c->stream));
    CUDA_TRY(c, launch_pack3(c->stage, c->V, c->vtmp, c->stream));
    CUDA_TRY(c, cudaMemsetAsync(c->gtmp, 0, sizeof(double) * 3 * C, c->stream));
    CUDA_TRY(c, launch_param_vjp(view(c), c->u[c->cur], c->vtmp, 1.0, c->gtmp, c->stream));
    CUDA_TRY(c, cudaMemcpyAsync(out, c->gtmp, sizeof(double) * 3 * C, cudaMemcpyDeviceToHost, c->stream));
    return wait_stream(c);
}

}  // extern "C"

void cf_free_adjoint(cf_ctx *c) { free_adjoint(c); }

void cf_free_plan(cf_ctx *c) {
    dfree(c->plan_parts);
    dfree(c->plan_rows);
    dfree(c->plan_list);
    dfree(c->plan_inc);
    c->plan_state = 0;
}
