// Test harness (host only): api.cu compiled by the host compiler against stand-ins for the
// CUDA runtime (device memory is the heap) and for the kernel launches (no pairs).  What a call is
// refused for, what it leaves in the plan and what it hands to the kernels is decided in api.cu and
// plan.cpp, which are the real ones.  Reads a script on standard input, prints one JSON value per line:
//   plan <9 lattice> <3 n> r_pe r_me frozen precision precond   create the plan: its status
//   step <9 lattice>   solve one orbital in this cell: status, and whether the solver was launched on a
//                      layout that is the one of the stencil it was given
//   oom <k>            the k-th device allocation from now on fails (0: none)
//   scans              how often mg_definite was asked since the last time
//   get | set <precond> <omega> | auto   exx_plan_get_schedule, _set_schedule, exx_plan_autotune
//   seen               [V-cycle, its Jacobi weight] of the last launch
//   layout <9 lattice> <3 n> <9 lattice> r_pe r_me   offsets of the first cell, stencil of the second:
//                      make_layout's status (larger of the two cells' errors)
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "plan.h"
static int g_scans = 0;   // questions whether a stencil's second-order operator is definite
static bool counted_mg_definite(const exx::Stencil &st)
{
    ++g_scans;
    return exx::mg_definite(st);
}
#define mg_definite counted_mg_definite
#include "api.cu"
#undef mg_definite

static long long g_alloc = 0, g_fail_at = 0;
static bool g_launched = false, g_match = false;
static int g_precond = 0;
static float g_omega = 0.f;
static exx_plan *g_plan = nullptr;
static char g_event;

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n)
{
    *p = nullptr;
    if (++g_alloc == g_fail_at) return cudaErrorMemoryAllocation;
    *p = std::calloc(n ? n : 1, 1);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { *p = std::calloc(n, 1); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { std::memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    std::memmove(d, s, n);
    return cudaSuccess;
}
// the solver slots are never read here and are large: left as calloc gives them
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 1; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorName(cudaError_t) { return "error"; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)&g_event; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *t, cudaEvent_t, cudaEvent_t) { *t = 1.f; return cudaSuccess; }
}

namespace exx {
cudaError_t launch_tables(const CellDev *, int, int, double *, float *, double *, float *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_gather_rows(const float *, const int32_t *, int, float *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_guess_info(const int32_t *, const uint8_t *, const int32_t *, const int32_t *, int, int4 *, cudaStream_t)
{
    return cudaSuccess;
}
cudaError_t launch_pair_list(const CellDev *, int, int, const ListDev &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_clamp_total(const ListDev &, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_finalize(const CellDev *, int, const ListDev &, CellResult *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_warm_map(const PairRec *, int, int, int *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_solve_cluster(const CellDev *, const ListDev &, const SolveSlots &, int, int, int, int, int *, cudaStream_t)
{
    return cudaSuccess;
}
int solve_blocks_per_sm(bool) { return 1; }
int cluster_capacity_bytes() { return 0; }
cudaError_t launch_solve(const CellDev *cells, const ListDev &, const SolveSlots &, bool, int, cudaStream_t)
{
    // the layout that belongs to the directions that the kernels are given
    g_launched = g_match = true;
    const CellDev &C = cells[0];
    g_precond = C.precond && C.set[1].mg;
    g_omega = C.mg_omega;
    for (int s = 0; s < 2; ++s) {
        Stencil st = g_plan->stencil;
        for (int d = 0; d < C.ndir; ++d)
            for (int k = 0; k < 3; ++k) st.dir[d][k] = C.dir[d][k];
        SetLayout L;
        const SetDev &S = C.set[s];
        if (make_layout(g_plan->off[s], st, C.fd_n, L) || !S.pe_off || !S.halo_off || !S.groups || !S.gs_perm || !S.S32 ||
            S.box != L.box || S.n_pe != L.n_pe || S.n_halo != L.n_halo ||
            std::memcmp(S.halo_off, L.halo_off.data(), 4 * (size_t)L.n_halo) ||
            std::memcmp(S.pe_off, L.pe_off.data(), 4 * (size_t)L.n_pe)) {
            g_match = false;
            continue;
        }
        for (int d = 0; d < 6; ++d) g_match = g_match && S.dstride[d] == L.dstride[d] && S.rstride[d] == L.rstride[d];
    }
    return cudaSuccess;
}
}  // namespace exx

static void show(int e, const exx_schedule &sc)
{
    std::printf("[%d, %d, %.4f, %d, %.1f]\n", e, sc.precond, sc.omega, sc.inner_shift, sc.ms);
}

static bool lattice(exx_cell &c)
{
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b)
            if (std::scanf("%lf", &c.lattice[a][b]) != 1) return false;
    return true;
}

int main()
{
    exx_ctx *ctx = nullptr;
    if (exx_ctx_create(&ctx, 0)) return 3;
    exx_cell c{};
    char cmd[32];
    while (std::scanf("%31s", cmd) == 1) {
        if (!std::strcmp(cmd, "plan")) {
            exx_params p{};
            double rpe, rme;
            if (!lattice(c) || std::scanf("%d %d %d %lf %lf %d %d %d", &c.n[0], &c.n[1], &c.n[2], &rpe, &rme, &p.frozen,
                                          &p.precision, &p.precond) != 8)
                return 4;
            p.r_pair = 6.0;
            p.r_pe_self = p.r_pe_pair = rpe;
            p.r_me_self = p.r_me_pair = rme;
            p.fd_order = 3;
            p.lmax = 6;
            p.cg_tol = 1e-9;
            p.cg_max_iter = 100;
            p.nq = 15;
            p.guess = 1;
            exx_plan_destroy(g_plan);
            const int box[3] = {4, 4, 4};
            std::printf("%d\n", exx_plan_create(ctx, &c, &p, 1, box, &g_plan));
        } else if (!std::strcmp(cmd, "step")) {
            if (!lattice(c) || !g_plan) return 4;
            const double centre[3] = {}, phi[64] = {};
            const int lo[3] = {};
            exx_orbitals o{};
            o.n_orb = 1;
            o.mem = EXX_MEM_DEVICE;
            o.centres = centre;
            o.box_lo = lo;
            o.phi = phi;
            for (int a = 0; a < 3; ++a) o.box[a] = 4;
            exx_result r{};
            g_launched = g_match = false;
            const int e = exx_pairs_solve(ctx, g_plan, &c, &o, &r, nullptr);
            std::printf("[%d, %s]\n", e, !g_launched ? "null" : g_match ? "true" : "false");
        } else if (!std::strcmp(cmd, "oom")) {
            int k;
            if (std::scanf("%d", &k) != 1) return 4;
            g_fail_at = k ? g_alloc + k : 0;
        } else if (!std::strcmp(cmd, "get")) {
            exx_schedule sc{};
            const int e = exx_plan_get_schedule(g_plan, &sc);
            show(e, sc);
        } else if (!std::strcmp(cmd, "set")) {
            exx_schedule sc{};
            sc.inner_shift = 14;
            if (std::scanf("%d %f", &sc.precond, &sc.omega) != 2) return 4;
            std::printf("%d\n", exx_plan_set_schedule(g_plan, &sc));
        } else if (!std::strcmp(cmd, "auto")) {   // (FP64 plans: nothing is launched)
            exx_schedule sc{};
            exx_orbitals o{};
            const int e = exx_plan_autotune(ctx, g_plan, &c, &o, 1, &sc, nullptr);
            show(e, sc);
        } else if (!std::strcmp(cmd, "seen")) {
            std::printf("[%d, %.4f]\n", g_precond, g_omega);
        } else if (!std::strcmp(cmd, "scans")) {
            std::printf("%d\n", g_scans);
            g_scans = 0;
        } else if (!std::strcmp(cmd, "layout")) {
            exx_cell a{}, b{};
            double rpe, rme;
            if (!lattice(a) || std::scanf("%d %d %d", &a.n[0], &a.n[1], &a.n[2]) != 3 || !lattice(b) ||
                std::scanf("%lf %lf", &rpe, &rme) != 2)
                return 4;
            Metric ma, mb;
            Stencil st;
            OffsetSet o;
            SetLayout L;
            int e = make_metric(a.lattice, a.n, ma);
            if (!e) e = make_metric(b.lattice, a.n, mb);
            if (!e) e = make_stencil(mb, 3, 15, nullptr, 0, st);
            if (!e) e = make_offsets(ma, rpe, rme, o);
            if (!e) e = make_layout(o, st, 3, L);
            std::printf("[%d", e);
            for (int d = 3; d < st.ndir; ++d) std::printf(", [%d, %d, %d]", st.dir[d][0], st.dir[d][1], st.dir[d][2]);
            std::printf("]\n");
        } else
            return 4;
    }
    exx_plan_destroy(g_plan);
    exx_ctx_destroy(ctx);
    return 0;
}
