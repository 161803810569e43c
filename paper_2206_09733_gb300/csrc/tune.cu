// Autotuner for the element kernels' launch shape.
//
// The BR1-gradient and element (volume) kernels run one thread per node with
// `epb` elements per CTA.  hs3d_autotune times every epb that gives a launch of
// its own (up to the kernel's largest CTA, max_cta_threads) on scratch copies of a
// smooth state (the element kernel as a middle RK stage, with its own clock and a
// tiny dt, so that the timed launches move the bytes of a real step), and keeps
// the fastest per (N, precision, kernel slot): the default, unless another is
// faster by more than kMargin.
// A mesh of fewer than kSMs elements per element of the largest CTA is spread over
// the SMs whatever epb is (spread_elems): there every epb would be the same launch
// and the choice noise, so the shapes are timed on a cube of the same degree that
// is large enough; the choice is for such meshes, and a small mesh's launches
// stay spread.
// Choices persist across processes in a small JSON file when HS3D_TUNE_CACHE names
// one: it is read on first use and rewritten after each tuning.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>
#include <vector>

#include "api_internal.h"

namespace hs3d {

static std::mutex g_tune_mu;
static bool g_cache_loaded = false;

static std::string cache_path()
{
    const char *p = getenv("HS3D_TUNE_CACHE");
    return p ? std::string(p) : std::string();
}

// Cache format: {"N<N>_p<prec>_k<slot>": epb, ...} (shape_slot)
static void load_cache_locked()
{
    if (g_cache_loaded) return;
    g_cache_loaded = true;
    std::string path = cache_path();
    if (path.empty()) return;
    FILE *f = fopen(path.c_str(), "r");
    if (!f) return;
    char buf[8192];
    size_t len = fread(buf, 1, sizeof buf - 1, f);
    fclose(f);
    buf[len] = 0;
    const char *s = buf;
    while ((s = strchr(s, '"')) != nullptr) {
        int N = 0, prec = 0, slot = 0, epb = 0;
        if (sscanf(s, "\"N%d_p%d_k%d\": %d", &N, &prec, &slot, &epb) == 4 && N >= 1 && N <= kMaxN && epb >= 1 &&
            epb <= 64 && prec >= 0 && prec <= 2 && slot >= 0 && slot < kShapeSlots)
            set_tuned_elems(N, prec, slot, epb);
        s = strchr(s + 1, '"');
        if (s) ++s;
    }
}

static void save_cache_locked()
{
    std::string path = cache_path();
    if (path.empty()) return;
    std::string tmp = path + ".tmp";
    FILE *f = fopen(tmp.c_str(), "w");
    if (!f) return;
    fprintf(f, "{");
    bool first = true;
    for (int N = 1; N <= kMaxN; ++N)
        for (int prec = 0; prec < 2; ++prec)
            for (int slot = 0; slot < kShapeSlots; ++slot) {
                int v = tuned_elems(N, prec, slot);
                if (v <= 0) continue;
                fprintf(f, "%s\"N%d_p%d_k%d\": %d", first ? "" : ", ", N, prec, slot, v);
                first = false;
            }
    fprintf(f, "}\n");
    fclose(f);
    rename(tmp.c_str(), path.c_str());
}

void tune_cache_load()
{
    std::lock_guard<std::mutex> g(g_tune_mu);
    load_cache_locked();
}

// Time per launch (the least of three runs of `reps`) of the gradient kernel, or
// of the element kernel as RK stage 1 (reads and writes u and g).
static float time_kernels(const hs3d_mesh *m, const hs3d_solver_cfg *c, const Batch &b, ShapeKernel k, int reps,
                          cudaStream_t s, cudaError_t &err)
{
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    auto launch = [&] {
        return k == kShapeGrad ? launch_grad(m->N, c->precision, b, s)
                               : launch_volume(m->N, c->precision, c->physics, c->volume_form, c->time_scheme, b, 1, -1, s);
    };
    err = launch();   // untimed (also surfaces launch errors for this shape)
    float best = 1e30f;
    for (int run = 0; run < 3 && err == cudaSuccess; ++run) {
        err = cudaEventRecord(e0, s);
        for (int r = 0; r < reps && err == cudaSuccess; ++r) err = launch();
        if (err == cudaSuccess) err = cudaEventRecord(e1, s);
        if (err == cudaSuccess) err = cudaEventSynchronize(e1);
        float ms = 0.f;
        if (err == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
        best = ms < best ? ms : best;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return best / reps;
}

// A shape replaces the default only where it is faster by more than this (the runs
// of one shape differ by about 1%).
constexpr float kMargin = 0.98f;

// Time the shapes of cfg's kernels on mesh m and set the choices.
static hs3d_status tune_on(hs3d_mesh *m, const hs3d_solver_cfg *c, cudaStream_t s)
{
    size_t sz = sizeof(double) * (size_t)m->E * 5 * m->n3;
    double *u = nullptr, *g = nullptr;
    Clock *clk = nullptr;
    cudaError_t e = cudaMalloc(&u, sz);
    if (e == cudaSuccess) e = cudaMalloc(&g, sz);
    if (e == cudaSuccess) e = cudaMalloc(&clk, sizeof(Clock));
    if (e != cudaSuccess) {
        if (u) cudaFree(u);
        if (g) cudaFree(g);
        cudaGetLastError();
        return cuda_fail(e, "autotune scratch");
    }
    // the stages advance the scratch state by dt = 1e-12 (|A_1| < 1 keeps g bounded)
    Clock hclk{};
    hclk.dt = 1e-12;
    e = cudaMemsetAsync(g, 0, sz, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(clk, &hclk, sizeof(Clock), cudaMemcpyHostToDevice, s);
    // a smooth state on this mesh: the Taylor-Green field (any positive state would do)
    hs3d_ic ic{HS3D_IC_TGV, c->gamma, 0.3, 0.0, 0.0, 0.0, 0.0};
    if (e == cudaSuccess) e = launch_init_state(m->N, m->E, m->X, ic, m->lo, m->hi, u, s);
    Item it = make_item(m, c, u, g, nullptr);
    it.clk = clk;
    Batch b = single_batch(it);
    // the face fluxes the volume kernel reads: one face pass
    cont_forget(m, nullptr);   // the trial launches rewrite the mesh's FP32 shadow
    if (e == cudaSuccess && c->precision != HS3D_FP64) e = launch_shadow(m->N, b, s);
    if (e == cudaSuccess && c->physics == HS3D_NS) e = launch_grad(m->N, c->precision, b, s);
    if (e == cudaSuccess) e = launch_face(m->N, c->precision, c->physics, c->surface_flux, b, s);
    const int n3 = m->n3;
    const bool gauss = m->nodes == HS3D_NODES_GAUSS;
    const int reps = m->E >= 4096 ? 5 : 20;
    for (const ShapeKernel k : {kShapeGrad, kShapeElem}) {
        if (e != cudaSuccess || (k == kShapeGrad && c->physics != HS3D_NS)) continue;
        const int slot = shape_slot(k, c->volume_form), keep = tuned_elems(m->N, c->precision, slot);
        const int most = max_cta_threads(m->N, c->precision, k, c->volume_form, gauss) / n3;
        int deflt = cta_target(m->N, c->precision, k, c->volume_form, gauss, m->E) / n3;
        deflt = deflt < 1 ? 1 : deflt > most ? most : deflt;
        std::vector<int> shapes;   // the default first, then the powers of two; one shape only: nothing to time
        if (most > 1) {
            shapes.push_back(deflt);
            for (int t = 1; t <= most; t *= 2)
                if (t != deflt) shapes.push_back(t);
        }
        int best = most > 1 ? 0 : 1;
        float best_ms = 0.f;
        for (const int t : shapes) {
            set_tuned_elems(m->N, c->precision, slot, t);
            const float ms = time_kernels(m, c, b, k, reps, s, e);
            if (e == cudaErrorInvalidValue || e == cudaErrorInvalidConfiguration) {
                // a shape the device cannot launch (shared memory): not a candidate
                cudaGetLastError();
                e = cudaSuccess;
            } else if (e != cudaSuccess) {
                break;
            } else if (best == 0 || ms < best_ms * (best == deflt ? kMargin : 1.0f)) {
                best_ms = ms;
                best = t;
            }
        }
        set_tuned_elems(m->N, c->precision, slot, best ? best : keep);
    }
    cudaStreamSynchronize(s);
    cudaFree(u);
    cudaFree(g);
    cudaFree(clk);
    return e == cudaSuccess ? HS3D_OK : cuda_fail(e, "autotune");
}

}  // namespace hs3d

using namespace hs3d;

extern "C" hs3d_status hs3d_autotune(const hs3d_mesh *mc, const hs3d_solver_cfg *c, int *choice_out, void *stream)
{
    hs3d_mesh *m = const_cast<hs3d_mesh *>(mc);
    if (!m) return fail(HS3D_ERR_INVALID, "mesh is NULL");
    hs3d_status st = validate_cfg(c);
    if (st == HS3D_OK) st = check_mesh_cfg(m, c);
    if (st != HS3D_OK) return st;
    const bool gauss = m->nodes == HS3D_NODES_GAUSS;
    int most = max_cta_threads(m->N, c->precision, kShapeElem, c->volume_form, gauss);
    if (c->physics == HS3D_NS) most = std::max(most, max_cta_threads(m->N, c->precision, kShapeGrad, c->volume_form, gauss));
    most /= m->n3;
    hs3d_mesh *big = nullptr;
    if (most > 1 && m->E < (long long)kSMs * most) {
        // a cube of the same degree with four of the largest CTAs per SM (built before
        // the lock is taken: creating a mesh reads the cache under it)
        hs3d_mesh_desc d{};
        d.N = m->N;
        d.nodes = m->nodes;
        d.perturb_amp = 0.05;
        for (int k = 0; k < 3; ++k) {
            d.lo[k] = -M_PI;
            d.hi[k] = M_PI;
            d.periodic[k] = 1;
        }
        d.ex = d.ey = d.ez = (int)std::ceil(std::cbrt(4.0 * kSMs * most));
        st = mesh_build(&d, &big);
    }
    {
        std::lock_guard<std::mutex> lock(g_tune_mu);
        load_cache_locked();
        if (st == HS3D_OK) st = tune_on(big ? big : m, c, (cudaStream_t)stream);
        if (st == HS3D_OK) save_cache_locked();
    }
    // no memory for the larger mesh: nothing is timed, the choices stay as they were
    if (st == HS3D_ERR_NOMEM && most > 1 && m->E < (long long)kSMs * most) st = HS3D_OK;
    mesh_free(big);
    if (st != HS3D_OK) return st;
    if (choice_out) {
        // what this mesh's launches use
        choice_out[0] = elems_per_cta(m->N, c->precision, kShapeGrad, c->volume_form, gauss, m->E);
        choice_out[1] = elems_per_cta(m->N, c->precision, kShapeElem, c->volume_form, gauss, m->E);
    }
    return HS3D_OK;
}
