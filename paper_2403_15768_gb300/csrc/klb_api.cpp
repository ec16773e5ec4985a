// C ABI of the KLB library (declared in include/klb.h): lattice creation in
// a caller-provided device buffer, couplings, initial state, time stepping,
// FP64 observables and host access to fields and state.

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "klb.h"
#include "klb_host.h"
#include "klb_internal.h"

#ifndef KLB_BOUNDS
#define KLB_BOUNDS 0
#endif

using namespace klb;

// Host view of the time level of a lattice: steps taken, buffer holding the
// current state, and (reduced-precision storage) the reference generation of
// each buffer and whether the next step switches to refreshed references.
struct HostState {
    int64_t step = 0;
    int64_t since_reset = 0;  // steps since creation / init / set_state
    int cur = 0;              // state buffer holding g*(n-1)
    int gen_buf[2] = {0, 0};
    bool refresh_pending = false;
};

struct klb_lattice {
    klb_desc desc;
    std::vector<uint8_t> mask;
    Geometry geo;
    MemoryPlan plan;
    cudaStream_t stream = nullptr;
    char *base = nullptr;
    klb_couplings cp{0, 0, 0, 0, 0};
    double kT = 0.0;          // thermal fluctuations of the water (0: off)
    uint64_t seed = 0;
    HostState st;
    std::string err;
};

namespace {

thread_local std::string g_create_error;

klb_status fail(klb_lattice *L, klb_status st, const std::string &msg)
{
    if (L)
        L->err = msg;
    else
        g_create_error = msg;
    return st;
}

klb_status cuda_fail(klb_lattice *L, cudaError_t e, const char *what)
{
    return fail(L, KLB_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define KLB_CUDA(L, call)                                         \
    do {                                                          \
        cudaError_t e_ = (call);                                  \
        if (e_ != cudaSuccess) return cuda_fail((L), e_, #call);  \
    } while (0)

size_t arith_size(const klb_lattice *L) { return L->desc.storage == KLB_FP64 ? 8 : 4; }
bool reduced(const klb_lattice *L) { return reduced_storage(L->desc.storage); }

void *dev(const klb_lattice *L, size_t off) { return L->base + off; }

// Lagged-velocity slot of step m (slots rotate with period 3).
int slot_of(int64_t m) { return (int)(((m % 3) + 3) % 3); }

// Bytes of a lattice's two state buffers.
size_t state_bytes(const klb_lattice *L)
{
    return 2 * (L->plan.pop_bytes[0] + L->plan.pop_bytes[1] + L->plan.pop_bytes[2]);
}

// Kernel arguments that follow the time level `st` (the step about to run, or
// the one observed).
template <typename T>
void fill_level(const klb_lattice *L, const HostState &st, StepArgs<T> &a)
{
    const MemoryPlan &p = L->plan;
    const int64_t n = st.step;
    for (int s = 0; s < 3; ++s) {
        a.in[s] = dev(L, p.pop[st.cur][s]);
        a.out[s] = dev(L, p.pop[1 - st.cur][s]);
        a.in_prev[s] = dev(L, p.pop[1 - st.cur][s]);
    }
    if (reduced(L))
        for (int s = 0; s < 3; ++s) {
            a.dec_in[s] = (const float *)dev(L, p.ref_dec[st.gen_buf[st.cur]][s]);
            a.dec_prev[s] = (const float *)dev(L, p.ref_dec[st.gen_buf[1 - st.cur]][s]);
            a.enc_out[s] = (const float *)dev(L, p.ref_enc[st.gen_buf[st.cur]][s]);
        }
    for (int c = 0; c < 2; ++c) {
        a.U0[c] = (T *)dev(L, p.U[slot_of(n)][c]);
        a.U1[c] = (const T *)dev(L, p.U[slot_of(n - 1)][c]);
        a.U2[c] = (const T *)dev(L, p.U[slot_of(n - 2)][c]);
        a.U3[c] = (const T *)dev(L, p.U[slot_of(n - 3)][c]);
    }
    a.residual_valid = st.since_reset >= 2;
    a.step_lo = (uint32_t)((uint64_t)n & 0xffffffffu);
    a.step_hi = (uint32_t)((uint64_t)n >> 32);
}

// All kernel arguments for the time level `st`; the step kernel runs blocks
// of sbx threads, with the small-lattice form of the solid rows or not, and
// touches all_bytes of state buffers per launch.
template <typename T>
void fill_args_at(const klb_lattice *L, const HostState &st, int sbx, bool fine, size_t all_bytes, StepArgs<T> &a)
{
    const Geometry &g = L->geo;
    const MemoryPlan &p = L->plan;
    std::memset((void *)&a, 0, sizeof a);
    fill_level(L, st, a);
    if (reduced(L)) {
        a.scale = L->desc.storage == KLB_FP16_DEV ? kFp16Scale : 1.0f;
        a.inv_scale = 1.0f / a.scale;
        a.acc = (float *)dev(L, p.acc);
    } else {
        a.scale = a.inv_scale = 1.0f;
    }
    for (int c = 0; c < 2; ++c) {
        a.rows[c] = (const RowInfo *)dev(L, p.rows[c]);
        a.n_rows[c] = (int)g.rows[c].size();
        a.n_slots[c] = (int)g.slot_row[c].size();
    }
    a.nx = g.nx;
    a.nxp = g.nxp;
    a.nchunk = p.nchunk;
    a.nbw = (int)g.rows[kFluid].size() * a.nchunk;
    a.snchunk = (g.nx + sbx - 1) / sbx;
    a.split = L->desc.storage == KLB_FP64 && fine;
    // divisions by multiplication: the kernel's first instructions wait for them
    auto divider = [](int d, uint32_t &mul, uint32_t &shift) {
        uint32_t sh = 0;
        while ((1u << sh) < (uint32_t)d) ++sh;
        shift = 31 + sh;
        mul = (uint32_t)((1ull << (31 + sh)) / (uint32_t)d + 1);
    };
    a.nseg64 = (g.nx + 63) / 64;
    a.sseg = fine ? (g.nx + 31) / 32 : a.nseg64;
    divider(a.nseg64, a.seg_mul, a.seg_shift);
    divider(a.sseg, a.sseg_mul, a.sseg_shift);
    a.nch32 = (g.nx + 31) / 32;
    a.nseg_w = (int)g.rows[kFluid].size() * a.nch32;
    const klb_desc &d = L->desc;
    a.rho0 = (T)d.rho0;
    a.om[0] = (T)(1.0 / d.tau_w);
    a.om[1] = (T)(1.0 / d.tau_e);
    a.om[2] = (T)(1.0 / d.tau_p);
    for (int k = 0; k < 3; ++k) a.G[k] = (T)d.G[k];
    a.g_we = (T)L->cp.g_we;
    a.g_wp = (T)L->cp.g_wp;
    a.g_ep = (T)L->cp.g_ep;
    a.g_ec = (T)L->cp.g_ec;
    a.g_pc = (T)L->cp.g_pc;
    a.q_p = (T)(d.phonon_eq == KLB_PHONON_WAVE ? 0.0 : 1.0);
    a.partials = (double *)dev(L, p.partials);
    a.field = (T *)dev(L, p.field);
    const double om = 1.0 / d.tau_w;
    a.noise_amp = (T)(L->kT > 0.0 ? std::sqrt(3.0 * d.rho0 * L->kT * om * (2.0 - om)) : 0.0);
    a.key[0] = (uint32_t)(L->seed & 0xffffffffu);
    a.key[1] = (uint32_t)(L->seed >> 32);
    a.bounds_err = (unsigned *)dev(L, p.bounds);
    for (int s = 0; s < 3; ++s) a.ck.s[s] = collide_k(g.Q, (float)a.om[s]);
    a.ahead = step_ahead(g.Q, d.storage, g.nxp, all_bytes);
}

// Form of the solid rows, threads per block and blocks of a lattice's step:
// those of its plan, but for thermal noise in FP32, which has its own rule.
struct StepForm {
    bool fine;
    int sbx, blocks;
};

StepForm step_form(const klb_lattice *L)
{
    const Geometry &g = L->geo;
    const long long nw = (long long)g.rows[kFluid].size(), ns = (long long)g.rows[kSolid].size();
    StepForm f{L->plan.fine, L->plan.sbx, L->plan.snblocks};
    if (L->kT > 0.0 && f.fine && L->desc.storage == KLB_FP32 && !noise_ep(g.Q, step_items(g.nx, nw, ns, true))) {
        f.fine = false;
        f.sbx = step_width(step_items(g.nx, nw, ns, false));
        f.blocks = step_blocks(g.nx, (int)nw, (int)ns, f.sbx, KLB_FP32, false);
    }
    return f;
}

template <typename T>
void fill_args(const klb_lattice *L, StepArgs<T> &a)
{
    const StepForm f = step_form(L);
    fill_args_at(L, L->st, f.sbx, f.fine, state_bytes(L), a);
}

// The host side of one step: encode generation of the output, whether the
// step accumulates x-sums for a reference refresh, and whether a refresh
// into that generation must run before it.
struct StepPlan {
    int outgen;
    bool acc;
    bool refresh;
};

StepPlan plan_step(const HostState &st, bool red)
{
    StepPlan sp;
    sp.outgen = st.gen_buf[st.cur];
    sp.refresh = red && st.refresh_pending;
    if (sp.refresh) sp.outgen = 1 - st.gen_buf[st.cur];
    sp.acc = red && (st.step + 1) % kRefEvery == 0;
    return sp;
}

void advance(HostState &st, const StepPlan &sp)
{
    st.gen_buf[1 - st.cur] = sp.outgen;
    st.cur = 1 - st.cur;
    ++st.step;
    ++st.since_reset;
    st.refresh_pending = sp.acc;
}

// Runs `body(args)` with arguments of the lattice's arithmetic type.
template <typename F>
cudaError_t with_args(const klb_lattice *L, F body)
{
    if (L->desc.storage == KLB_FP64) {
        StepArgs<double> a;
        fill_args(L, a);
        return body(&a);
    }
    StepArgs<float> a;
    fill_args(L, a);
    return body(&a);
}

// Sets the encode references of the next output buffer (generation gen).
void set_enc(const klb_lattice *L, void *args, int gen)
{
    if (!reduced(L)) return;
    StepArgs<float> *a = static_cast<StepArgs<float> *>(args);
    for (int s = 0; s < 3; ++s) a->enc_out[s] = (const float *)dev(L, L->plan.ref_enc[gen][s]);
}

// Reference refresh into generation gen from the x-sums of the last
// accumulating pass.
cudaError_t refresh_refs(const klb_lattice *L, int gen)
{
    float *enc[3], *dec[3];
    for (int s = 0; s < 3; ++s) {
        enc[s] = (float *)dev(L, L->plan.ref_enc[gen][s]);
        dec[s] = (float *)dev(L, L->plan.ref_dec[gen][s]);
    }
    return with_args(L, [&](void *a) { return launch_ref(L->geo.Q, L->desc.storage, a, enc, dec, L->stream); });
}

int nblocks(const klb_lattice *L) { return L->plan.nblocks_w + L->plan.nblocks_s; }

// Observation pass enqueued on the lattice's stream: the pass and the
// reduction of its blocks' partial sums to the kNumSums sums.
cudaError_t launch_observe(const klb_lattice *L, double *partials, double *sums)
{
    const bool f64 = L->desc.storage == KLB_FP64;
    const int blocks = f64 ? nblocks(L) : L->plan.oblocks;
    const cudaError_t e = with_args(L, [&](void *a) {
        if (f64) {
            static_cast<StepArgs<double> *>(a)->partials = partials;
        } else {
            static_cast<StepArgs<float> *>(a)->partials = partials;
            static_cast<StepArgs<float> *>(a)->obs_solid = L->plan.oblocks_s;
        }
        return launch(L->geo.Q, L->desc.storage, a, kModeObserve, blocks, f64 ? L->plan.bx : kBlockX, L->stream);
    });
    return e != cudaSuccess ? e : launch_finalize(partials, blocks, sums, L->stream);
}

cudaError_t launch_observe(const klb_lattice *L)
{
    return launch_observe(L, (double *)dev(L, L->plan.partials), (double *)dev(L, L->plan.sums));
}

// Blocks that bound the lattices klb_observables_static takes.
int static_blocks(const klb_lattice *L) { return L->desc.storage == KLB_FP64 ? nblocks(L) : L->plan.static_blocks; }

// Species field index helpers: row class and row count of species s.
int cls_of(int s) { return s == 0 ? kFluid : kSolid; }

// Offset (elements) of species s in the field scratch [s][4][n_rows][nxp].
size_t field_offset(const klb_lattice *L, int s)
{
    const size_t nxp = L->geo.nxp, nrw = L->geo.rows[kFluid].size(),
                 nrs = L->geo.rows[kSolid].size();
    return s == 0 ? 0 : 4 * nrw * nxp + (s == 2 ? 4 * nrs * nxp : 0);
}

// Uninitialised host memory for downloads and uploads.
struct HostBuf {
    std::unique_ptr<char[]> p;
    size_t bytes = 0;
    bool alloc(size_t n)
    {
        p.reset(new (std::nothrow) char[n ? n : 1]);
        bytes = n;
        return p != nullptr;
    }
    template <typename T> T *as() const { return reinterpret_cast<T *>(p.get()); }
};

// Waits for the stream before the host buffers declared ahead of it are
// freed, if a call returns before its own synchronisation.
struct StreamGuard {
    cudaStream_t s;
    bool done = false;
    ~StreamGuard()
    {
        if (!done) cudaStreamSynchronize(s);
    }
};

klb_status no_host_memory(klb_lattice *L) { return fail(L, KLB_ENOMEM, "host allocation failed"); }

// n rows of nx elements padded to nxp: fill(k, o) writes row k's elements, the
// padding is zeroed here.  Where padding is a fifth of a row or more, all rows
// at once beforehand: lines of memory that the device has read are slow to
// write in parts, and a call per row takes longer than a narrow row's elements
// (150x150 pipe, nx 5: klb_init_equilibrium FP32 1.9 to 3.7 -> 0.56 ms, FP64 4.0
// to 7.5 -> 1.15; pipe R8, nx 8: klb_set_state FP64 0.26 to 0.42 -> 0.19 ms).
template <typename V, typename F>
void fill_rows(V *rows, size_t n, size_t nx, size_t nxp, F fill)
{
    const bool narrow = nx < 4 * (nxp - nx);
    if (narrow) std::memset((void *)rows, 0, n * nxp * sizeof(V));
    for (size_t k = 0; k < n; ++k) {
        V *o = rows + k * nxp;
        fill(k, o);
        if (!narrow)
            for (size_t x = nx; x < nxp; ++x) o[x] = V(0);
    }
}

// Rows of host box fields (either may be null) in the layout of the field
// scratch.
template <typename T>
void host_to_field(const klb_lattice *L, const double *drho, const double *u, T *f)
{
    const Geometry &g = L->geo;
    const size_t ncell = (size_t)g.nx * g.ny * g.nz, nxp = g.nxp, nx = g.nx;
    for (int s = 0; s < 3; ++s) {
        const int c = cls_of(s);
        const size_t nr = g.rows[c].size();
        T *fs = f + field_offset(L, s);
        host_parallel(nr, nr * nx * 4 * sizeof(double), [&, s, c, nr, fs](size_t r0, size_t r1) {
            for (int a = 0; a < 4; ++a) {
                const double *in = a == 0 ? (drho ? drho + s * ncell : nullptr) : (u ? u + (s * 3 + a - 1) * ncell : nullptr);
                T *o = fs + (a * nr + r0) * nxp;
                if (!in) {
                    std::memset((void *)o, 0, (r1 - r0) * nxp * sizeof(T));
                    continue;
                }
                const int *cs = g.rows[c].data() + r0;
                fill_rows(o, r1 - r0, nx, nxp, [=](size_t k, T *o) {
                    const double *q = in + nx * cs[k];
                    for (size_t x = 0; x < nx; ++x) o[x] = (T)q[x];
                });
            }
        });
    }
}

// Box arrays from rows: plane k of `planes` holds the values row(k, r) -> x
// of a row class at its cells and 0 elsewhere.
template <typename F>
void rows_to_box(const klb_lattice *L, int cls, size_t planes, double *box, F row)
{
    const Geometry &g = L->geo;
    const size_t ncs = (size_t)g.ny * g.nz, nx = g.nx, n = planes * ncs;
    host_parallel(n, n * nx * sizeof(double), [&, cls, ncs, nx, box](size_t i0, size_t i1) {
        const int *row_of = g.row_of_cs[cls].data();
        size_t k = i0 / ncs, cs = i0 - k * ncs;
        const bool narrow = nx < 32;  // zeroed together first, as in fill_rows
        if (narrow) std::memset(box + i0 * nx, 0, (i1 - i0) * nx * sizeof(double));
        for (size_t i = i0; i < i1;) {
            double *o = box + i * nx;
            if (row_of[cs] >= 0) {
                row(k, (size_t)row_of[cs], o);
                ++i;
                ++cs;
            } else {  // a run of cells without the class
                const size_t most = std::min(ncs - cs, i1 - i);
                size_t m = 1;
                while (m < most && row_of[cs + m] < 0) ++m;
                if (!narrow) std::memset(o, 0, m * nx * sizeof(double));
                i += m;
                cs += m;
            }
            if (cs == ncs) {
                cs = 0;
                ++k;
            }
        }
    });
}

klb_status sync(klb_lattice *L)
{
    KLB_CUDA(L, cudaStreamSynchronize(L->stream));
    return KLB_OK;
}

// A state buffer's three species lie one after the other in it, as do the two
// classes of a lagged-velocity slot (which goes in one copy).  Up to 1 MB the
// species go in one copy, beyond one after the other through the same host
// memory, whose first touch costs more than the copy (128x64x64 FP32: 76 MB
// in one, 25 in three).
struct PopsCopy {
    bool one;
    size_t bytes;  // of host memory
};

PopsCopy pops_copy(const klb_lattice *L)
{
    const MemoryPlan &p = L->plan;
    const size_t all = p.pop[0][2] - p.pop[0][0] + p.pop_bytes[2];
    if (all <= (1u << 20)) return {true, all};
    return {false, std::max(p.pop_bytes[0], std::max(p.pop_bytes[1], p.pop_bytes[2]))};
}

// Start from rest: every population, lagged velocity and reference is 0.  The
// first two lie one after the other in the lattice's buffer up to the row
// tables, as do the references of a generation: two fills at most (one per
// region, 12 or 18, took longer than k_init of a tiny lattice).
klb_status init_from_rest(klb_lattice *L)
{
    const MemoryPlan &p = L->plan;
    KLB_CUDA(L, cudaMemsetAsync(dev(L, p.pop[0][0]), 0, p.rows[kFluid] - p.pop[0][0], L->stream));
    if (reduced(L))
        KLB_CUDA(L, cudaMemsetAsync(dev(L, p.ref_enc[0][0]), 0, p.ref_enc[1][0] - p.ref_enc[0][0], L->stream));
    return KLB_OK;
}

void reset_state(klb_lattice *L, int64_t step)
{
    L->st.cur = 0;
    L->st.step = step;
    L->st.since_reset = 0;
    L->st.gen_buf[0] = L->st.gen_buf[1] = 0;
    L->st.refresh_pending = false;
}

template <typename T>
klb_status init_from_fields(klb_lattice *L, const double *drho, const double *u)
{
    if (!drho && !u) {
        reset_state(L, 0);
        klb_status st = init_from_rest(L);
        return st != KLB_OK ? st : sync(L);
    }
    HostBuf f;
    StreamGuard guard{L->stream};
    if (!f.alloc(L->plan.field_bytes)) return no_host_memory(L);
    host_to_field<T>(L, drho, u, f.as<T>());
    KLB_CUDA(L, cudaMemcpyAsync(dev(L, L->plan.field), f.p.get(), L->plan.field_bytes,
                                cudaMemcpyHostToDevice, L->stream));
    reset_state(L, 0);
    const int slot0 = slot_of(0);
    auto init_pass = [&](int mode) {
        return with_args(L, [&](void *a) {
            StepArgs<T> *A = (StepArgs<T> *)a;
            for (int s = 0; s < 3; ++s) A->out[s] = dev(L, L->plan.pop[0][s]);
            for (int c = 0; c < 2; ++c) A->U0[c] = (T *)dev(L, L->plan.U[slot0][c]);
            set_enc(L, a, 0);
            return launch(L->geo.Q, L->desc.storage, a, mode, nblocks(L), L->plan.bx, L->stream);
        });
    };
    if (reduced(L)) {
        // References first: the x-averages of the initial equilibria.
        KLB_CUDA(L, init_pass(kModeInitAcc));
        KLB_CUDA(L, refresh_refs(L, 0));
    }
    KLB_CUDA(L, init_pass(kModeInit));
    for (int s = 0; s < 3; ++s)
        KLB_CUDA(L, cudaMemcpyAsync(dev(L, L->plan.pop[1][s]), dev(L, L->plan.pop[0][s]),
                                    L->plan.pop_bytes[s], cudaMemcpyDeviceToDevice, L->stream));
    for (int t = 0; t < 3; ++t)
        for (int c = 0; c < 2; ++c)
            if (t != slot0 && L->plan.U_bytes[c])
                KLB_CUDA(L, cudaMemcpyAsync(dev(L, L->plan.U[t][c]), dev(L, L->plan.U[slot0][c]),
                                            L->plan.U_bytes[c], cudaMemcpyDeviceToDevice, L->stream));
    guard.done = true;
    return sync(L);
}

// Observables from the final sums (least squares u = A + B d^2 from its
// normal equations, means, residual, non-finite count); the one definition
// behind klb_observables and klb_observables_static.
klb_status finish_observables(klb_lattice *L, const double *S, klb_obs *out)
{
    const Geometry &g = L->geo;
    const double nan = std::numeric_limits<double>::quiet_NaN();
    std::memset(out, 0, sizeof *out);
    out->step = L->st.step;
    out->flow_rate = S[kSumUxFluid] / g.nx;
    out->d_wall = g.has_fit ? g.d_wall : nan;
    const double n = g.fit_n, s2 = g.fit_d2, s4 = g.fit_d4;
    const double su = S[kSumFitU], su2 = S[kSumFitUD2];
    const double det = n * s4 - s2 * s2;
    if (g.has_fit && n >= 2 && det != 0.0) {
        out->fit_B = (n * su2 - s2 * su) / det;
        out->fit_A = (su - out->fit_B * s2) / n;
        out->u_slip = out->fit_A + out->fit_B * g.d_wall * g.d_wall;
        out->dudn_wall = std::fabs(2.0 * out->fit_B * g.d_wall);
        out->slip_length = out->dudn_wall != 0.0 ? out->u_slip / out->dudn_wall
                                                 : std::numeric_limits<double>::infinity();
    } else {
        out->fit_A = out->fit_B = out->u_slip = out->dudn_wall = out->slip_length = nan;
    }
    out->u_wallrow_mean = g.wall_n > 0 ? S[kSumWallU] / g.wall_n : nan;
    const double ncells[3] = {(double)g.rows[kFluid].size() * g.nx,
                              (double)g.rows[kSolid].size() * g.nx,
                              (double)g.rows[kSolid].size() * g.nx};
    const double usum[3] = {S[kSumUxFluid], S[kSumUxE], S[kSumUxP]};
    for (int s = 0; s < 3; ++s) {
        out->mean_u[s] = usum[s] / ncells[s];
        out->momentum[s] = S[kSumMomW + s];
        out->mass[s] = S[kSumMassW + s];
    }
    out->residual = L->st.since_reset >= 2 ? S[kSumResidual] : nan;
    out->nonfinite = (int64_t)S[kSumNonfinite];
    out->clipped = (int64_t)S[kSumClipped];
    if (out->nonfinite > 0) return fail(L, KLB_EUNSTABLE, "non-finite density or velocity");
    if (out->clipped > 0)
        return fail(L, KLB_ERANGE,
                    std::to_string(out->clipped) +
                        " species-cells hold a population saturated at the 16-bit range (a difference "
                        "from the row's x-average beyond the representable range)");
    return KLB_OK;
}

bool finite5(const klb_couplings &c)
{
    return std::isfinite(c.g_we) && std::isfinite(c.g_wp) && std::isfinite(c.g_ep) &&
           std::isfinite(c.g_ec) && std::isfinite(c.g_pc);
}

}  // namespace

extern "C" {

size_t klb_lattice_bytes(const klb_desc *desc)
{
    if (!desc) return 0;
    Geometry g;
    std::string err;
    if (!build_geometry(*desc, g, err)) return 0;
    return plan_memory(g, desc->storage).total;
}

klb_status klb_lattice_info(const klb_desc *desc, klb_info *info)
{
    if (!desc || !info) return fail(nullptr, KLB_EINVAL, "null argument");
    Geometry g;
    std::string err;
    if (!build_geometry(*desc, g, err)) return fail(nullptr, KLB_EINVAL, err);
    std::memset(info, 0, sizeof *info);
    info->fluid_cs = (int64_t)g.rows[kFluid].size();
    info->solid_cs = (int64_t)g.rows[kSolid].size();
    info->species_cells[0] = info->fluid_cs * g.nx;
    info->species_cells[1] = info->species_cells[2] = info->solid_cs * g.nx;
    info->active_sites = (info->fluid_cs + info->solid_cs) * g.nx;
    for (int c = 0; c < 2; ++c) {
        info->iface_cs[c] = (int64_t)g.slot_row[c].size();
        info->max_faces[c] = g.max_faces[c];
    }
    info->d_wall = g.has_fit ? g.d_wall : std::numeric_limits<double>::quiet_NaN();
    info->bytes = plan_memory(g, desc->storage).total;
    return KLB_OK;
}

klb_status klb_create_lattice(const klb_desc *desc, void *dev_buf, size_t bytes, void *cuda_stream,
                              klb_lattice **out)
{
    if (!desc || !out) return fail(nullptr, KLB_EINVAL, "null argument");
    *out = nullptr;
    klb_lattice *L = new (std::nothrow) klb_lattice();
    if (!L) return fail(nullptr, KLB_ENOMEM, "host allocation failed");
    L->desc = *desc;
    if (desc->geom == KLB_GEOM_MASK && desc->mask && desc->ny > 0 && desc->nz > 0) {
        L->mask.assign(desc->mask, desc->mask + (size_t)desc->ny * desc->nz);
        L->desc.mask = L->mask.data();
    }
    std::string err;
    if (!build_geometry(L->desc, L->geo, err)) {
        delete L;
        return fail(nullptr, KLB_EINVAL, err);
    }
    L->plan = plan_memory(L->geo, L->desc.storage);
    if (!dev_buf || ((uintptr_t)dev_buf & 255u)) {
        delete L;
        return fail(nullptr, KLB_EINVAL, "dev_buf must be a 256-byte aligned device pointer");
    }
    if (bytes < L->plan.total) {
        delete L;
        return fail(nullptr, KLB_ENOMEM, "device buffer smaller than klb_lattice_bytes()");
    }
    L->base = (char *)dev_buf;
    L->stream = (cudaStream_t)cuda_stream;
    // Row tables, then a zero state.
    cudaError_t e = cudaSuccess;
    for (int c = 0; c < 2 && e == cudaSuccess; ++c)
        e = cudaMemcpyAsync(dev(L, L->plan.rows[c]), L->geo.info[c].data(),
                            sizeof(RowInfo) * L->geo.info[c].size(), cudaMemcpyHostToDevice,
                            L->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(dev(L, L->plan.bounds), 0, sizeof(unsigned), L->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(L->stream);
    if (e != cudaSuccess) {
        std::string m = std::string("uploading row tables: ") + cudaGetErrorString(e);
        delete L;
        return fail(nullptr, KLB_ECUDA, m);
    }
    klb_status st = klb_init_equilibrium(L, nullptr, nullptr);
    if (st != KLB_OK) {
        std::string m = L->err;
        delete L;
        return fail(nullptr, st, m);
    }
    *out = L;
    return KLB_OK;
}

klb_status klb_bounds_status(klb_lattice *L, uint32_t *site)
{
    if (!L || !site) return fail(L, KLB_EINVAL, "null argument");
    unsigned w = 0;
    KLB_CUDA(L, cudaMemcpyAsync(&w, dev(L, L->plan.bounds), sizeof w, cudaMemcpyDeviceToHost, L->stream));
    KLB_CUDA(L, cudaMemsetAsync(dev(L, L->plan.bounds), 0, sizeof w, L->stream));
    klb_status st = sync(L);
    if (st != KLB_OK) return st;
    *site = w;
    return KLB_OK;
}

int klb_bounds_checked(void) { return KLB_BOUNDS; }

klb_status klb_set_fluctuations(klb_lattice *L, double kT, uint64_t seed)
{
    if (!L) return fail(L, KLB_EINVAL, "null handle");
    if (!(kT >= 0.0) || !std::isfinite(kT)) return fail(L, KLB_EINVAL, "kT must be finite and >= 0");
    if (kT > 0.0 && reduced(L))
        return fail(L, KLB_EINVAL, "thermal fluctuations need FP32 or FP64 storage");
    L->kT = kT;
    L->seed = seed;
    return KLB_OK;
}

klb_status klb_set_couplings(klb_lattice *L, const klb_couplings *c)
{
    if (!L || !c) return fail(L, KLB_EINVAL, "null argument");
    if (!finite5(*c)) return fail(L, KLB_EINVAL, "non-finite coupling");
    // Stability of the lagged interface exchange (pair relaxation rate below
    // 4/3, Gershgorin over the cells): face-summed |gamma| below 0.6 rho0.
    const double sw = L->geo.max_faces[kFluid] * (std::fabs(c->g_we) + std::fabs(c->g_wp));
    const double ss = L->geo.max_faces[kSolid] * std::fmax(std::fabs(c->g_we), std::fabs(c->g_wp));
    if (std::fmax(sw, ss) >= 0.6 * L->desc.rho0)
        return fail(L, KLB_EINVAL, "interface couplings beyond the stability bound 0.6 rho0");
    // The co-located electron-phonon pair is implicit; only its matrix must stay regular.
    const double k = 0.5 * c->g_ep, a = L->desc.rho0 + k + 0.5 * c->g_ec,
                 b = L->desc.rho0 + k + 0.5 * c->g_pc;
    if (!(a > 0 && b > 0 && a * b - k * k > 0))
        return fail(L, KLB_EINVAL, "electron-phonon couplings make the implicit pair singular");
    L->cp = *c;
    return KLB_OK;
}

klb_status klb_init_equilibrium(klb_lattice *L, const double *drho, const double *u)
{
    if (!L) return fail(L, KLB_EINVAL, "null handle");
    return L->desc.storage == KLB_FP64 ? init_from_fields<double>(L, drho, u)
                                       : init_from_fields<float>(L, drho, u);
}

klb_status klb_step(klb_lattice *L, int64_t nsteps)
{
    if (!L) return fail(L, KLB_EINVAL, "null handle");
    if (nsteps < 0) return fail(L, KLB_EINVAL, "nsteps must be >= 0");
    for (int64_t n = 0; n < nsteps; ++n) {
        const StepPlan sp = plan_step(L->st, reduced(L));
        if (sp.refresh) {
            // Decode this step with the current references, encode its output
            // with references refreshed from the last step's x-averages.
            cudaError_t e = refresh_refs(L, sp.outgen);
            if (e != cudaSuccess) return cuda_fail(L, e, "reference refresh");
        }
        cudaError_t e = with_args(L, [&](void *a) {
            set_enc(L, a, sp.outgen);
            const int mode = sp.acc ? kModeStepAcc : (L->kT > 0.0 ? kModeStepNoise : kModeStep);
            const StepForm f = step_form(L);
            const bool ep = f.fine && L->desc.storage != KLB_FP64;
            return launch(L->geo.Q, L->desc.storage, a, ep ? mode | kModeEp : mode, f.blocks, f.sbx, L->stream);
        });
        if (e != cudaSuccess) return cuda_fail(L, e, "step kernel launch");
        advance(L->st, sp);
    }
    return KLB_OK;
}

}  // extern "C"

// Observation of many lattices with one synchronisation (the request loop):
// enqueue each lattice's pass and the copy of its sums to pinned host memory,
// synchronise the shared stream once, then finish each from its sums.
cudaError_t klb::observe_enqueue(klb_lattice *L, double *host_sums)
{
    cudaError_t e = launch_observe(L);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(host_sums, dev(L, L->plan.sums), sizeof(double) * kNumSums, cudaMemcpyDeviceToHost,
                            L->stream);
    return e;
}

klb_status klb::observe_finish(klb_lattice *L, const double *host_sums, klb_obs *out)
{
    return finish_observables(L, host_sums, out);
}

extern "C" {

klb_status klb_observables(klb_lattice *L, klb_obs *out)
{
    if (!L || !out) return fail(L, KLB_EINVAL, "null argument");
    KLB_CUDA(L, launch_observe(L));
    double S[kNumSums];
    KLB_CUDA(L, cudaMemcpyAsync(S, dev(L, L->plan.sums), sizeof S, cudaMemcpyDeviceToHost,
                                L->stream));
    klb_status st = sync(L);
    if (st != KLB_OK) return st;
    return finish_observables(L, S, out);
}

klb_status klb_observables_static(klb_lattice *L, klb_obs *out)
{
    if (!L || !out) return fail(L, KLB_EINVAL, "null argument");
    double *partials = nullptr, *sums = nullptr;
    size_t max_blocks = 0;
    KLB_CUDA(L, static_scratch(&partials, &sums, &max_blocks));
    if ((size_t)static_blocks(L) > max_blocks)
        return fail(L, KLB_EINVAL,
                    std::to_string(static_blocks(L)) +
                        " row chunks, more than the static observation takes (KLB_STATIC_MAX_BLOCKS = " +
                        std::to_string(max_blocks) + ")");
    KLB_CUDA(L, launch_observe(L, partials, sums));
    double S[kNumSums];
    KLB_CUDA(L, cudaMemcpyAsync(S, sums, sizeof S, cudaMemcpyDeviceToHost, L->stream));
    klb_status st = sync(L);
    if (st != KLB_OK) return st;
    return finish_observables(L, S, out);
}

klb_status klb_get_field(klb_lattice *L, double *drho, double *u)
{
    if (!L) return fail(L, KLB_EINVAL, "null handle");
    KLB_CUDA(L, with_args(L, [&](void *a) {
                 return launch(L->geo.Q, L->desc.storage, a, kModeField, nblocks(L),
                                    L->plan.bx, L->stream);
             }));
    HostBuf raw;
    StreamGuard guard{L->stream};
    if (!raw.alloc(L->plan.field_bytes)) return no_host_memory(L);
    KLB_CUDA(L, cudaMemcpyAsync(raw.p.get(), dev(L, L->plan.field), L->plan.field_bytes,
                                cudaMemcpyDeviceToHost, L->stream));
    klb_status st = sync(L);
    guard.done = true;
    if (st != KLB_OK) return st;
    const Geometry &g = L->geo;
    const size_t ncell = (size_t)g.nx * g.ny * g.nz, nxp = g.nxp, nx = g.nx;
    auto put = [&](auto *f) {
        for (int s = 0; s < 3; ++s) {
            const int c = cls_of(s);
            const size_t nr = g.rows[c].size();
            const auto *fs = f + field_offset(L, s);
            auto row = [&, fs, nr](size_t a, size_t r, double *o) {
                const auto *q = fs + (a * nr + r) * nxp;
                for (size_t x = 0; x < nx; ++x) o[x] = (double)q[x];
            };
            if (drho) rows_to_box(L, c, 1, drho + s * ncell, row);
            if (u) rows_to_box(L, c, 3, u + s * 3 * ncell, [&](size_t a, size_t r, double *o) { row(a + 1, r, o); });
        }
    };
    if (arith_size(L) == 8)
        put(raw.as<const double>());
    else
        put(raw.as<const float>());
    return KLB_OK;
}

klb_status klb_get_state(klb_lattice *L, double *gout, double *U1, double *U2)
{
    if (!L) return fail(L, KLB_EINVAL, "null handle");
    const Geometry &g = L->geo;
    const size_t ncell = (size_t)g.nx * g.ny * g.nz, nxp = g.nxp, nx = g.nx;
    const int Q = g.Q, storage = L->desc.storage;
    const bool red = reduced(L);
    const double inv = storage == KLB_FP16_DEV ? 1.0 / kFp16Scale : 1.0;
    if (gout) {
        HostBuf pops, refs[3];
        StreamGuard guard{L->stream};
        const size_t *at = L->plan.pop[L->st.cur];
        const PopsCopy pc = pops_copy(L);
        if (!pops.alloc(pc.bytes)) return no_host_memory(L);
        for (int s = 0; s < 3; ++s) {
            if (!refs[s].alloc(L->plan.ref_bytes[s])) return no_host_memory(L);
            if (red)
                KLB_CUDA(L, cudaMemcpyAsync(refs[s].p.get(), dev(L, L->plan.ref_enc[L->st.gen_buf[L->st.cur]][s]),
                                            refs[s].bytes, cudaMemcpyDeviceToHost, L->stream));
        }
        for (int s = 0; s < 3; ++s) {
            if (s == 0 || !pc.one) {
                guard.done = false;
                KLB_CUDA(L, cudaMemcpyAsync(pops.p.get(), dev(L, at[s]), pc.one ? pc.bytes : L->plan.pop_bytes[s],
                                            cudaMemcpyDeviceToHost, L->stream));
                klb_status st = sync(L);
                guard.done = true;
                if (st != KLB_OK) return st;
            }
            const int c = cls_of(s);
            const size_t nr = g.rows[c].size();
            // Population values of a row (reduced storage: the stored
            // difference, still to be scaled and shifted by its row reference).
            auto put = [&](auto *pop) {
                rows_to_box(L, c, Q, gout + (size_t)s * Q * ncell, [&, pop, nr, s](size_t i, size_t r, double *o) {
                    const auto *q = pop + (i * nr + r) * nxp;
                    using V = std::decay_t<decltype(*q)>;
                    if constexpr (std::is_same_v<V, __half> || std::is_same_v<V, __nv_bfloat16>) {
                        const double shift = refs[s].as<const float>()[r * kRefStride + i];
                        for (size_t x = 0; x < nx; ++x) {
                            float v;
                            if constexpr (std::is_same_v<V, __half>)
                                v = __half2float(q[x]);
                            else
                                v = __bfloat162float(q[x]);
                            o[x] = (double)(float)((double)v * inv + shift);
                        }
                    } else {
                        for (size_t x = 0; x < nx; ++x) o[x] = (double)q[x];
                    }
                });
            };
            const char *pop = pops.p.get() + (pc.one ? at[s] - at[0] : 0);
            switch (storage) {
            case KLB_FP64:
                put(reinterpret_cast<const double *>(pop));
                break;
            case KLB_FP32:
                put(reinterpret_cast<const float *>(pop));
                break;
            case KLB_FP16_DEV:
                put(reinterpret_cast<const __half *>(pop));
                break;
            default:
                put(reinterpret_cast<const __nv_bfloat16 *>(pop));
                break;
            }
        }
    }
    double *Uo[2] = {U1, U2};
    for (int t = 0; t < 2; ++t) {
        if (!Uo[t]) continue;
        const int slot = slot_of(L->st.step - 1 - t);
        HostBuf raw;
        StreamGuard guard{L->stream};
        const size_t *at = L->plan.U[slot];
        if (!raw.alloc(at[1] - at[0] + L->plan.U_bytes[kSolid])) return no_host_memory(L);
        if (raw.bytes)
            KLB_CUDA(L, cudaMemcpyAsync(raw.p.get(), dev(L, at[0]), raw.bytes, cudaMemcpyDeviceToHost, L->stream));
        klb_status st = sync(L);
        guard.done = true;
        if (st != KLB_OK) return st;
        for (int s = 0; s < 3; ++s) {
            const int c = cls_of(s);
            const size_t ns = g.slot_row[c].size(), a0 = s == 2 ? 3 : 0;
            auto put = [&](auto *U) {
                rows_to_box(L, c, 3, Uo[t] + s * 3 * ncell, [&, U, ns, a0, c](size_t a, size_t r, double *o) {
                    const int q = g.info[c][r].slot;
                    if (q < 0) {
                        std::memset(o, 0, nx * sizeof(double));
                        return;
                    }
                    const auto *v = U + ((a0 + a) * ns + (size_t)q) * nxp;
                    for (size_t x = 0; x < nx; ++x) o[x] = (double)v[x];
                });
            };
            const char *U = raw.p.get() + (at[c] - at[0]);
            if (arith_size(L) == 8)
                put(reinterpret_cast<const double *>(U));
            else
                put(reinterpret_cast<const float *>(U));
        }
    }
    return KLB_OK;
}

klb_status klb_set_state(klb_lattice *L, const double *gin, const double *U1, const double *U2,
                         int64_t step)
{
    if (!L || !gin || !U1 || !U2) return fail(L, KLB_EINVAL, "null argument");
    if (step < 0) return fail(L, KLB_EINVAL, "step must be >= 0");
    const Geometry &g = L->geo;
    const size_t ncell = (size_t)g.nx * g.ny * g.nz, nxp = g.nxp, nx = g.nx;
    const int Q = g.Q, storage = L->desc.storage;
    const bool red = reduced(L);
    const float scale = storage == KLB_FP16_DEV ? kFp16Scale : 1.0f;
    auto sat = [](float v, float m) { return v > m ? m : (v < -m ? -m : v); };  // NaN passes
    KLB_CUDA(L, cudaStreamSynchronize(L->stream));
    // All host memory first: without it the state and its time level stay as they are.
    HostBuf encs[3], decs[3], pops, Us[2];
    StreamGuard guard{L->stream};
    const MemoryPlan &p = L->plan;
    const PopsCopy pc = pops_copy(L);
    bool have = pops.alloc(pc.bytes);
    for (int t = 0; t < 2; ++t) have = have && Us[t].alloc(p.U[0][1] - p.U[0][0] + p.U_bytes[kSolid]);
    for (int s = 0; red && s < 3; ++s) have = have && encs[s].alloc(p.ref_bytes[s]) && decs[s].alloc(p.ref_bytes[s]);
    if (!have) return no_host_memory(L);
    reset_state(L, step);
    float *enc[3] = {}, *dec[3] = {};
    for (int s = 0; red && s < 3; ++s) {
        enc[s] = encs[s].as<float>();
        dec[s] = decs[s].as<float>();
        std::memset(enc[s], 0, p.ref_bytes[s]);
        std::memset(dec[s], 0, p.ref_bytes[s]);
    }
    for (int s = 0; s < 3; ++s) {
        const int c = cls_of(s);
        const size_t nr = g.rows[c].size();
        auto take = [&](auto *pop) {
            using V = std::decay_t<decltype(*pop)>;
            host_parallel((size_t)Q * nr, (size_t)Q * nr * nx * sizeof(double), [&, pop, nr, s, c](size_t k0, size_t k1) {
                const int *cs = g.rows[c].data();
                size_t i = k0 / nr, r = k0 - i * nr;
                fill_rows(pop + k0 * nxp, k1 - k0, nx, nxp, [&](size_t, V *o) {
                    const double *in = gin + ((size_t)s * Q + i) * ncell + nx * cs[r];
                    if constexpr (std::is_same_v<V, __half> || std::is_same_v<V, __nv_bfloat16>) {
                        // Reference of each (row, direction): the x-average of the state.
                        double sum = 0.0;
                        for (size_t x = 0; x < nx; ++x) sum += in[x];
                        const float ref = (float)(sum / g.nx);
                        enc[s][r * kRefStride + i] = ref;
                        for (size_t x = 0; x < nx; ++x) {
                            const float v = ((float)in[x] - ref) * scale;  // saturating, as the device encode
                            if constexpr (std::is_same_v<V, __half>)
                                o[x] = __float2half_rn(sat(v, 65504.0f));
                            else
                                o[x] = __float2bfloat16_rn(sat(v, 3.38953139e38f));
                        }
                    } else {
                        for (size_t x = 0; x < nx; ++x) o[x] = (V)in[x];
                    }
                    if (++r == nr) {
                        r = 0;
                        ++i;
                    }
                });
            });
        };
        char *pop = pops.p.get() + (pc.one ? p.pop[0][s] - p.pop[0][0] : 0);
        switch (storage) {
        case KLB_FP64:
            take(reinterpret_cast<double *>(pop));
            break;
        case KLB_FP32:
            take(reinterpret_cast<float *>(pop));
            break;
        case KLB_FP16_DEV:
            take(reinterpret_cast<__half *>(pop));
            break;
        default:
            take(reinterpret_cast<__nv_bfloat16 *>(pop));
            break;
        }
        if (!pc.one) {
            KLB_CUDA(L, cudaMemcpyAsync(dev(L, p.pop[0][s]), pop, p.pop_bytes[s], cudaMemcpyHostToDevice, L->stream));
            KLB_CUDA(L, cudaMemcpyAsync(dev(L, p.pop[1][s]), dev(L, p.pop[0][s]), p.pop_bytes[s],
                                        cudaMemcpyDeviceToDevice, L->stream));
            if (s < 2) KLB_CUDA(L, cudaStreamSynchronize(L->stream));  // the next species takes this memory
        }
    }
    if (pc.one) {
        KLB_CUDA(L, cudaMemcpyAsync(dev(L, p.pop[0][0]), pops.p.get(), pc.bytes, cudaMemcpyHostToDevice, L->stream));
        KLB_CUDA(L, cudaMemcpyAsync(dev(L, p.pop[1][0]), dev(L, p.pop[0][0]), pc.bytes, cudaMemcpyDeviceToDevice, L->stream));
    }
    if (red) {
        for (int s = 0; s < 3; ++s) {
            const int c = cls_of(s);
            const size_t nr = g.rows[c].size();
            for (size_t r = 0; r < nr; ++r)
                for (int i = 0; i < Q; ++i) {
                    const long q = g.info[c][r].src[i] / (g.nxp / kRowAlign);  // sdir * nr + srow
                    const long sdir = q / (long)nr, srow = q - sdir * (long)nr;
                    dec[s][r * kRefStride + i] = enc[s][srow * kRefStride + sdir];
                }
            KLB_CUDA(L, cudaMemcpyAsync(dev(L, L->plan.ref_enc[0][s]), enc[s], L->plan.ref_bytes[s],
                                        cudaMemcpyHostToDevice, L->stream));
            KLB_CUDA(L, cudaMemcpyAsync(dev(L, L->plan.ref_dec[0][s]), dec[s], L->plan.ref_bytes[s],
                                        cudaMemcpyHostToDevice, L->stream));
        }
    }
    const double *Ui[2] = {U1, U2};  // u(n-1), u(n-2)
    for (int t = 0; t < 2; ++t) {
        const size_t *at = p.U[slot_of(step - 1 - t)], n = Us[t].bytes;
        for (int c = 0; c < 2; ++c) {
            const size_t ns = g.slot_row[c].size();
            if (!ns) continue;
            auto take = [&](auto *U) {
                using V = std::decay_t<decltype(*U)>;
                const size_t na = c == kFluid ? 3 : 6, b0 = c == kFluid ? 0 : 3;  // component planes, first box plane
                host_parallel(na * ns, na * ns * nx * sizeof(double), [&, U, ns, b0, c, t](size_t k0, size_t k1) {
                    fill_rows(U + k0 * nxp, k1 - k0, nx, nxp, [&](size_t k, V *o) {
                        const size_t a = (k0 + k) / ns, q = k0 + k - a * ns;
                        const double *in = Ui[t] + (b0 + a) * ncell + nx * g.rows[c][g.slot_row[c][q]];
                        for (size_t x = 0; x < nx; ++x) o[x] = (V)in[x];
                    });
                });
            };
            char *U = Us[t].p.get() + (at[c] - at[0]);
            if (arith_size(L) == 8)
                take(reinterpret_cast<double *>(U));
            else
                take(reinterpret_cast<float *>(U));
        }
        if (n) KLB_CUDA(L, cudaMemcpyAsync(dev(L, at[0]), Us[t].p.get(), n, cudaMemcpyHostToDevice, L->stream));
        // u(n-3) unknown: reuse u(n-2)
        if (n && t == 1)
            KLB_CUDA(L, cudaMemcpyAsync(dev(L, p.U[slot_of(step - 3)][0]), dev(L, at[0]), n, cudaMemcpyDeviceToDevice,
                                        L->stream));
    }
    guard.done = true;
    return sync(L);
}

int64_t klb_get_step(const klb_lattice *L) { return L ? L->st.step : -1; }

int64_t klb_species_cells(const klb_lattice *L, int species)
{
    if (!L || species < 0 || species > 2) return -1;
    return (int64_t)L->geo.rows[cls_of(species)].size() * L->geo.nx;
}

klb_status klb_destroy(klb_lattice *L)
{
    if (!L) return KLB_OK;
    cudaError_t e = cudaStreamSynchronize(L->stream);
    delete L;
    if (e != cudaSuccess) {
        g_create_error = std::string("klb_destroy: ") + cudaGetErrorString(e);
        return KLB_ECUDA;
    }
    return KLB_OK;
}

const char *klb_last_error(const klb_lattice *L)
{
    return L ? L->err.c_str() : g_create_error.c_str();
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Batches

struct klb_batch {
    std::vector<klb_lattice *> mem;
    cudaStream_t user = nullptr;  // the members' stream
    cudaStream_t stream = nullptr;  // the batch's own stream (graph capture)
    cudaEvent_t ev_in = nullptr, ev_out = nullptr;
    char *base = nullptr;
    size_t bytes = 0;
    int Q = 19, storage = KLB_FP32;
    int period = 6;
    int width = kBlockX;
    int nblocks = 0;
    bool fine = false, by_table = false;  // small-lattice form of the solid rows; launched over device copies
    size_t rec_size = 0, table_off = 0, prefix_off = 0, ck_off = 0, reps_off = 0;
    std::vector<char> table;      // argument records [phase][member], the block prefix
    std::vector<int> prefix;
    std::vector<CollideSet> ck;   // and the members' collision constants
    std::vector<StepPlan> plans;  // per (phase, member)
    std::vector<char> acc;        // per phase: some member accumulates x-sums
    std::vector<int64_t> base_step;  // members' steps at phase 0
    std::vector<HostState> base_state;  // members' time levels at phase 0
    std::vector<HostState> now_state;   // and after the batch's last step
    std::vector<klb_couplings> cp;      // members' couplings in the tables
    int64_t phase = 0;               // steps taken since phase 0
    cudaGraphExec_t graph = nullptr;
    std::string err;
};

namespace {

klb_status bfail(klb_batch *B, klb_status st, const std::string &msg)
{
    B->err = msg;
    return st;
}

#define KLB_BCUDA(B, call)                                                                  \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess) return bfail((B), KLB_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

int batch_period(int storage) { return reduced_storage(storage) ? 6 * 2 * kRefEvery : 6; }

size_t rec_size(int storage) { return storage == KLB_FP64 ? sizeof(StepRecord<double>) : sizeof(StepRecord<float>); }

// Batch buffer: period count, and for batches that may be launched over
// device copies (batch_by_table) the block prefix, the collision constants
// (FP32 arithmetic) and the argument records [phase][member].
size_t batch_layout(int n, int storage, size_t *table_off, size_t *prefix_off, size_t *ck_off, size_t *reps_off)
{
    auto round_up = [](size_t b) { return (b + 255) / 256 * 256; };
    *reps_off = 0;
    *prefix_off = *ck_off = *table_off = 256;
    if (n <= kBatchParams) return 256;
    *ck_off = *prefix_off + round_up((size_t)(n + 1) * sizeof(int));
    *table_off = *ck_off + (storage == KLB_FP64 ? 0 : round_up((size_t)n * sizeof(CollideSet)));
    return *table_off + round_up((size_t)batch_period(storage) * n * rec_size(storage));
}

void destroy_graph(klb_batch *B)
{
    if (B->graph) cudaGraphExecDestroy(B->graph);
    B->graph = nullptr;
}

// Whether the solid rows of a member take the small-lattice form: with FP32
// arithmetic one form for the launch, with FP64 the members that take it alone.
bool fine_member(const klb_batch *B, const klb_lattice *L)
{
    return B->fine && (B->storage != KLB_FP64 || L->plan.fine);
}

// A member's argument records of every phase, from its time level now: the
// arguments once, then what follows the time level.
template <typename T>
void fill_records(klb_batch *B, int m, int width, size_t all_bytes)
{
    const klb_lattice *L = B->mem[m];
    const int n = (int)B->mem.size(), P = B->period;
    StepArgs<T> a;
    fill_args_at(L, L->st, width, fine_member(B, L), all_bytes, a);
    a.step_reps = (const uint32_t *)(B->base + B->reps_off);
    a.step_period = P;
    B->ck[m] = a.ck;
    HostState st = L->st;
    for (int k = 0; k < P; ++k) {
        const StepPlan sp = plan_step(st, reduced(L));
        B->plans[(size_t)k * n + m] = sp;
        B->acc[k] |= (char)sp.acc;
        fill_level(L, st, a);
        set_enc(L, &a, sp.outgen);
        reinterpret_cast<StepRecord<T> *>(B->table.data())[(size_t)k * n + m] = a;
        advance(st, sp);
    }
}

// Argument records for block width `width`, from each member's own time level
// now (phase 0), the block prefix, and the phase plans.  Every member's step
// pattern repeats after the batch period whatever its step count, so members
// may stand at different time levels.  A launch accumulates reference x-sums
// when any member needs them; the x-sums are stored, not added, so an extra
// pass leaves the other members' refreshes unchanged.
klb_status build_tables(klb_batch *B, int width)
{
    const int n = (int)B->mem.size(), P = B->period;
    std::vector<int> &prefix = B->prefix;
    B->table.resize((size_t)P * n * B->rec_size);
    B->ck.resize(n);
    prefix.assign(n + 1, 0);
    B->plans.resize((size_t)P * n);
    B->acc.assign(P, 0);
    size_t all_bytes = 0;
    for (const klb_lattice *L : B->mem) all_bytes += state_bytes(L);
    for (int m = 0; m < n; ++m) {
        if (B->storage == KLB_FP64)
            fill_records<double>(B, m, width, all_bytes);
        else
            fill_records<float>(B, m, width, all_bytes);
        const Geometry &g = B->mem[m]->geo;
        prefix[m + 1] = prefix[m] + step_blocks(g.nx, (int)g.rows[kFluid].size(), (int)g.rows[kSolid].size(), width,
                                                B->storage, fine_member(B, B->mem[m]));
    }
    KLB_BCUDA(B, cudaStreamSynchronize(B->stream));
    if (B->by_table) {
        KLB_BCUDA(B, cudaMemcpy(B->base + B->table_off, B->table.data(), B->table.size(), cudaMemcpyHostToDevice));
        KLB_BCUDA(B, cudaMemcpy(B->base + B->prefix_off, prefix.data(), prefix.size() * sizeof(int),
                                cudaMemcpyHostToDevice));
        if (B->storage != KLB_FP64)
            KLB_BCUDA(B, cudaMemcpy(B->base + B->ck_off, B->ck.data(), B->ck.size() * sizeof(CollideSet),
                                    cudaMemcpyHostToDevice));
    }
    KLB_BCUDA(B, cudaMemset(B->base + B->reps_off, 0, sizeof(uint32_t)));
    B->width = width;
    B->nblocks = prefix[n];
    B->phase = 0;
    B->base_step.resize(n);
    B->base_state.resize(n);
    B->now_state.resize(n);
    B->cp.resize(n);
    for (int m = 0; m < n; ++m) {
        B->base_step[m] = B->mem[m]->st.step;
        B->base_state[m] = B->now_state[m] = B->mem[m]->st;
        B->cp[m] = B->mem[m]->cp;
    }
    destroy_graph(B);
    return KLB_OK;
}

// One phase of the batch on its stream: reference refreshes due before the
// step, then the batched step kernel.
cudaError_t launch_phase(klb_batch *B, int k)
{
    const size_t n = B->mem.size();
    for (size_t m = 0; m < n; ++m) {
        const StepPlan &sp = B->plans[k * n + m];
        if (!sp.refresh) continue;
        klb_lattice *L = B->mem[m];
        cudaStream_t keep = L->stream;
        L->stream = B->stream;
        cudaError_t e = refresh_refs(L, sp.outgen);
        L->stream = keep;
        if (e != cudaSuccess) return e;
    }
    const size_t at = (size_t)k * n * B->rec_size;
    const BatchLaunch b{B->table.data() + at, B->base + B->table_off + at, B->prefix.data(),
                        (const int *)(B->base + B->prefix_off), B->ck.data(),
                        (const CollideSet *)(B->base + B->ck_off), (int)n, B->width, B->acc[k] != 0,
                        B->fine && B->storage != KLB_FP64, B->by_table};
    cudaError_t e = launch_batch(B->Q, B->storage, b, B->stream);
    if (e == cudaSuccess && k == B->period - 1) e = launch_count_period((uint32_t *)(B->base + B->reps_off), B->stream);
    return e;
}

klb_status capture_graph(klb_batch *B)
{
    destroy_graph(B);
    cudaGraph_t g = nullptr;
    KLB_BCUDA(B, cudaStreamBeginCapture(B->stream, cudaStreamCaptureModeThreadLocal));
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < B->period && e == cudaSuccess; ++k) e = launch_phase(B, k);
    cudaError_t e2 = cudaStreamEndCapture(B->stream, &g);
    if (e != cudaSuccess || e2 != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return bfail(B, KLB_ECUDA, std::string("graph capture: ") +
                                       cudaGetErrorString(e != cudaSuccess ? e : e2));
    }
    e = cudaGraphInstantiate(&B->graph, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        B->graph = nullptr;
        return bfail(B, KLB_ECUDA, std::string("graph instantiate: ") + cudaGetErrorString(e));
    }
    return KLB_OK;
}

bool in_phase(const klb_batch *B)
{
    for (size_t m = 0; m < B->mem.size(); ++m)
        if (B->mem[m]->st.step != B->base_step[m] + B->phase) return false;
    return true;
}

// Whether two time levels at the same step read and write the same buffers.
bool same_level(const HostState &a, const HostState &b)
{
    return a.cur == b.cur && a.gen_buf[0] == b.gen_buf[0] && a.gen_buf[1] == b.gen_buf[1] &&
           a.refresh_pending == b.refresh_pending;
}

// Whether every member stands where the tables' phase 0 assumed.  The step
// pattern repeats after a period from any time level but one: right after
// an initialisation of 16-bit storage no reference refresh is pending at a
// multiple of the refresh interval, where one is pending in every later
// period.
bool tables_repeat(const klb_batch *B)
{
    for (size_t m = 0; m < B->mem.size(); ++m)
        if (!same_level(B->mem[m]->st, B->base_state[m])) return false;
    return true;
}

// Whether the members are as the batch left them: klb_set_state at the same
// step resets a member's buffer and reference generation, and couplings are
// part of the argument records.
bool untouched(const klb_batch *B)
{
    for (size_t m = 0; m < B->mem.size(); ++m) {
        const klb_couplings &a = B->mem[m]->cp, &b = B->cp[m];
        if (!same_level(B->mem[m]->st, B->now_state[m]) || a.g_we != b.g_we || a.g_wp != b.g_wp ||
            a.g_ep != b.g_ep || a.g_ec != b.g_ec || a.g_pc != b.g_pc)
            return false;
    }
    return true;
}

// Advances the members' time levels by steps that the batch has enqueued.
void advance_members(klb_batch *B, int steps)
{
    for (size_t m = 0; m < B->mem.size(); ++m) {
        HostState &h = B->mem[m]->st;
        for (int j = 0; j < steps; ++j) advance(h, plan_step(h, reduced(B->mem[m])));
        B->now_state[m] = h;
    }
    B->phase += steps;
}

// Runs nsteps phases on the batch stream, replaying the graph for whole
// periods; advances every member's host state.  At the start of each later
// period the tables are checked against the members' time levels and built
// again if they no longer describe it.
klb_status run_steps(klb_batch *B, int64_t nsteps, bool use_graph)
{
    while (nsteps > 0) {
        if (B->phase > 0 && B->phase % B->period == 0 && !tables_repeat(B)) {
            klb_status st = build_tables(B, B->width);
            if (st != KLB_OK) return st;
        }
        const int k = (int)(B->phase % B->period);
        if (use_graph && k == 0 && nsteps >= B->period) {
            if (!B->graph) {
                klb_status st = capture_graph(B);
                if (st != KLB_OK) return st;
            }
            KLB_BCUDA(B, cudaGraphLaunch(B->graph, B->stream));
            advance_members(B, B->period);
            nsteps -= B->period;
            continue;
        }
        KLB_BCUDA(B, launch_phase(B, k));
        advance_members(B, 1);
        --nsteps;
    }
    return KLB_OK;
}

}  // namespace

size_t klb::batch_table_bytes(int storage, int n)
{
    size_t t, p, c, r;
    return n < 1 ? 0 : batch_layout(n, storage, &t, &p, &c, &r);
}

extern "C" {

size_t klb_batch_bytes(klb_lattice *const *members, int n)
{
    if (!members || n < 1 || !members[0]) return 0;
    size_t t, p, c, r;
    return batch_layout(n, members[0]->desc.storage, &t, &p, &c, &r);
}

klb_status klb_batch_create(klb_lattice *const *members, int n, void *dev_buf, size_t bytes,
                            klb_batch **out)
{
    if (!out) return fail(nullptr, KLB_EINVAL, "null argument");
    *out = nullptr;
    if (!members || n < 1) return fail(nullptr, KLB_EINVAL, "a batch needs at least one member");
    for (int m = 0; m < n; ++m) {
        const klb_lattice *L = members[m];
        if (!L) return fail(nullptr, KLB_EINVAL, "null member");
        if (L->geo.Q != members[0]->geo.Q || L->desc.storage != members[0]->desc.storage)
            return fail(nullptr, KLB_EINVAL, "batch members must share lattice kind and storage");
        if (L->stream != members[0]->stream)
            return fail(nullptr, KLB_EINVAL, "batch members must share one CUDA stream");
        for (int k = 0; k < m; ++k)
            if (members[k] == L) return fail(nullptr, KLB_EINVAL, "a lattice appears twice in the batch");
        if (L->kT > 0.0)
            return fail(nullptr, KLB_EINVAL, "lattices with thermal fluctuations cannot be batched");
    }
    klb_batch *B = new (std::nothrow) klb_batch();
    if (!B) return fail(nullptr, KLB_ENOMEM, "host allocation failed");
    B->mem.assign(members, members + n);
    B->Q = members[0]->geo.Q;
    B->storage = members[0]->desc.storage;
    B->period = batch_period(B->storage);
    B->rec_size = rec_size(B->storage);
    const size_t need = batch_layout(n, B->storage, &B->table_off, &B->prefix_off, &B->ck_off, &B->reps_off);
    if (!dev_buf || ((uintptr_t)dev_buf & 255u)) {
        delete B;
        return fail(nullptr, KLB_EINVAL, "dev_buf must be a 256-byte aligned device pointer");
    }
    if (bytes < need) {
        delete B;
        return fail(nullptr, KLB_ENOMEM, "device buffer smaller than klb_batch_bytes()");
    }
    B->base = (char *)dev_buf;
    B->bytes = bytes;
    B->user = members[0]->stream;
    cudaError_t e = cudaStreamCreateWithFlags(&B->stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&B->ev_in, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&B->ev_out, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaStreamSynchronize(B->user);
    if (e != cudaSuccess) {
        std::string m = std::string("batch setup: ") + cudaGetErrorString(e);
        klb_batch_destroy(B);
        return fail(nullptr, KLB_ECUDA, m);
    }
    int w = kBlockX;
    long long items[2] = {0, 0}, warps64 = 0;
    for (klb_lattice *L : B->mem) {
        const Geometry &g = L->geo;
        const long long nw = (long long)g.rows[kFluid].size(), ns = (long long)g.rows[kSolid].size();
        for (int e = 0; e < 2; ++e) items[e] += step_items(g.nx, nw, ns, e != 0);
        warps64 += fp64_warps(g.nx, nw, ns);
    }
    if (B->storage == KLB_FP64) {
        B->fine = fp64_batch_split(warps64);
        for (klb_lattice *L : B->mem) w = std::min(w, B->fine ? L->plan.sbx : L->plan.bx);
    } else {
        B->fine = step_ep(items[1]);
        w = step_width(items[B->fine]);
    }
    B->by_table = batch_by_table(n, B->storage, items[B->fine]);
    klb_status st = build_tables(B, w);
    if (st != KLB_OK) {
        std::string m = B->err;
        klb_batch_destroy(B);
        return fail(nullptr, st, m);
    }
    *out = B;
    return KLB_OK;
}

klb_status klb_batch_step(klb_batch *B, int64_t nsteps)
{
    if (!B) return KLB_EINVAL;
    if (nsteps < 0) return bfail(B, KLB_EINVAL, "nsteps must be >= 0");
    if (!in_phase(B))
        return bfail(B, KLB_ESTATE, "a member was stepped outside the batch; form the batch again");
    if (nsteps > 0 && !untouched(B)) {
        const klb_status st = build_tables(B, B->width);
        if (st != KLB_OK) return st;
    }
    KLB_BCUDA(B, cudaEventRecord(B->ev_in, B->user));
    KLB_BCUDA(B, cudaStreamWaitEvent(B->stream, B->ev_in, 0));
    klb_status st = run_steps(B, nsteps, true);
    KLB_BCUDA(B, cudaEventRecord(B->ev_out, B->stream));
    KLB_BCUDA(B, cudaStreamWaitEvent(B->user, B->ev_out, 0));
    return st;
}

klb_status klb_batch_autotune(klb_batch *B, int steps_per_candidate, int *width)
{
    if (!B) return KLB_EINVAL;
    if (steps_per_candidate < 1) return bfail(B, KLB_EINVAL, "steps_per_candidate must be >= 1");
    if (!in_phase(B))
        return bfail(B, KLB_ESTATE, "a member was stepped outside the batch; form the batch again");
    KLB_BCUDA(B, cudaStreamSynchronize(B->user));
    cudaEvent_t t0 = nullptr, t1 = nullptr;
    cudaError_t ce = cudaEventCreate(&t0);
    if (ce == cudaSuccess) ce = cudaEventCreate(&t1);
    if (ce != cudaSuccess) {
        if (t0) cudaEventDestroy(t0);
        return bfail(B, KLB_ECUDA, std::string("autotune events: ") + cudaGetErrorString(ce));
    }
    const int cand[3] = {32, 64, 128};
    int best = B->width;
    float best_ms = 1e30f;
    klb_status st = KLB_OK;
    for (int c = 0; c < 3 && st == KLB_OK; ++c) {
        st = build_tables(B, cand[c]);
        if (st != KLB_OK) break;
        st = run_steps(B, 1, false);  // warm-up
        if (st != KLB_OK) break;
        if (cudaEventRecord(t0, B->stream) != cudaSuccess) {
            st = bfail(B, KLB_ECUDA, "autotune timing");
            break;
        }
        st = run_steps(B, steps_per_candidate, false);
        if (st != KLB_OK) break;
        float ms = 0.f;
        if (cudaEventRecord(t1, B->stream) != cudaSuccess || cudaEventSynchronize(t1) != cudaSuccess ||
            cudaEventElapsedTime(&ms, t0, t1) != cudaSuccess)
            st = bfail(B, KLB_ECUDA, "autotune timing");
        if (st == KLB_OK && ms < best_ms) {
            best_ms = ms;
            best = cand[c];
        }
    }
    cudaEventDestroy(t0);
    cudaEventDestroy(t1);
    if (st != KLB_OK) return st;
    st = build_tables(B, best);
    if (width) *width = best;
    return st;
}

int klb_batch_width(const klb_batch *B) { return B ? B->width : 0; }
int64_t klb_batch_blocks(const klb_batch *B) { return B ? B->nblocks : 0; }

klb_status klb_batch_destroy(klb_batch *B)
{
    if (!B) return KLB_OK;
    if (B->stream) cudaStreamSynchronize(B->stream);
    destroy_graph(B);
    if (B->ev_in) cudaEventDestroy(B->ev_in);
    if (B->ev_out) cudaEventDestroy(B->ev_out);
    if (B->stream) cudaStreamDestroy(B->stream);
    delete B;
    return KLB_OK;
}

const char *klb_batch_last_error(const klb_batch *B) { return B ? B->err.c_str() : ""; }

}  // extern "C"
