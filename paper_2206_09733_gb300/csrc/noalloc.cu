// Quadrature diagnostics that allocate nothing.
//
// Some callers cannot call cudaMalloc: code that runs while a CUDA stream
// capture is active (allocation is prohibited there), code inside a host
// framework that owns every byte of device memory through its own pool, or
// real-time loops where an allocation and its implicit synchronisation are
// not allowed.  hs3d_diagnostics keeps its per-block partial sums in scratch
// owned by the mesh; this variant takes every input from the caller and keeps
// the partial sums in a fixed file-scope device array instead.
//
// The array lives in every device that loads the library, until the process
// exits.  Host code may not pass the array's name to a kernel (on the host it
// is only a stand-in symbol): its device address is looked up once per device
// with cudaGetSymbolAddress and that pointer is passed.
#include <mutex>

#include "api_internal.h"

namespace hs3d {

// Capacity stated in the interface.  (The grid stops growing at kDiagMaxBlocks, so
// the array holds the sums of any number of nodes; what was refused stays refused.)
constexpr long long kStaticMaxNodes = 8388608;

static __device__ __align__(256) double g_static_partials[7 * kDiagMaxBlocks];

// Device address of g_static_partials, looked up once per device.
static double *static_partials_ptr(int dev, cudaError_t &err)
{
    static std::mutex mu;
    static double *ptrs[64] = {};
    err = cudaSuccess;
    if (dev < 0 || dev >= 64) {
        err = cudaErrorInvalidDevice;
        return nullptr;
    }
    std::lock_guard<std::mutex> g(mu);
    if (!ptrs[dev]) {
        void *p = nullptr;
        err = cudaGetSymbolAddress(&p, g_static_partials);
        if (err != cudaSuccess) return nullptr;
        ptrs[dev] = (double *)p;
    }
    return ptrs[dev];
}

}  // namespace hs3d

using namespace hs3d;

extern "C" hs3d_status hs3d_diagnostics_noalloc(int N, int64_t E, double gamma, int nodes, const double *J,
                                                const double *u, const double *dudt, double *out, void *stream)
{
    if (N < 1 || N > kMaxN) return fail(HS3D_ERR_INVALID, "N=%d outside 1..%d", N, kMaxN);
    if (nodes != HS3D_NODES_LOBATTO && nodes != HS3D_NODES_GAUSS) return fail(HS3D_ERR_INVALID, "bad nodes %d", nodes);
    if (E < 1) return fail(HS3D_ERR_INVALID, "E must be >= 1");
    if (!(gamma > 1.0)) return fail(HS3D_ERR_INVALID, "gamma must be > 1");
    if (!J || !u || !out) return fail(HS3D_ERR_INVALID, "J, u and out must not be NULL");
    const long long n3 = (long long)(N + 1) * (N + 1) * (N + 1);
    const long long total = (long long)E * n3;
    if (total > kStaticMaxNodes)
        return fail(HS3D_ERR_INVALID,
                    "E*(N+1)^3 = %lld nodes exceeds this entry point's capacity of %lld nodes; use hs3d_diagnostics",
                    total, kStaticMaxNodes);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "no CUDA device");
    double *partials = static_partials_ptr(dev, e);
    if (!partials) return cuda_fail(e, "cudaGetSymbolAddress of the static scratch");
    // the kernels of hs3d_diagnostics (same partition and order of the sums)
    e = launch_diagnostics(N, nodes, E, gamma, J, u, dudt, partials, out, (cudaStream_t)stream);
    return e == cudaSuccess ? HS3D_OK : cuda_fail(e, "static diagnostics launch");
}
