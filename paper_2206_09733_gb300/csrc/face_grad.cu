// Face Riemann solve and BR1 gradients of the FP64 path (the mixed path:
// face_dev.cu, grad_dev.cu).
//
// k_face: one thread per face node.  Gathers the two traces (Gauss-Lobatto
// nodes include the element boundary, so the trace is the boundary node
// itself), computes the inviscid numerical flux (LF, Roe, central EC,
// Rusanov, low-dissipation Roe or entropy-stable matrix dissipation,
// Sec. 3.3) times the face scale and, for Navier-Stokes, subtracts the BR1
// viscous flux (F_v(L) + F_v(R)).Sn/2.  Each face is solved once; both
// elements read the result (with opposite sign on the -d side).
//
// k_grad: BR1 gradients of q = (v1, v2, v3, T), T = p/rho (Bassi & Rebay 1997):
//   J grad q_c = sum_d D_d (Ja^d_c q) + sum_faces (1/w_end) (q* - q_in) (+-Ja^d_c),
//   q* = (q_in + q_out)/2, stored as viscous stress and heat flux (kVisc
//   values per node).  Element per thread group, node per thread.
//
// Both are bound by the FP64 pipe, so they are written for few FP64
// instructions per warp: one reciprocal per state (rcp_fast, shared by
// velocities, enthalpy and temperature), one reciprocal square root for a
// norm and its inverse, and one instruction sequence for the two faces of a
// direction (a lane is on at most one of them).  16^3 elements of N = 3 (NS,
// Roe), one launch: k_face 122 -> 85 us, k_grad 177 -> 106 us.
#include "internal.cuh"
#include "physics.cuh"

namespace hs3d {

// Index of the node with index `end` along direction d and tangential (ta, tb).
template <int n>
__device__ __forceinline__ int face_node(int d, int end, int ta, int tb)
{
    if (d == 0) return end + n * (ta + n * tb);
    if (d == 1) return ta + n * (end + n * tb);
    return ta + n * (tb + n * end);
}

// Small CTAs: with its 142 registers a 256-thread CTA leaves one CTA (8 warps)
// per SM, 64-thread CTAs 12 warps, and a small mesh reaches more SMs (16^3,
// N = 3, two steps of three stages: 3175 -> 3071 us).
constexpr int kFaceThreads = 64;

template <int N, bool NS>
__global__ void __launch_bounds__(kFaceThreads) k_face(const __grid_constant__ Batch b, int flux)
{
    constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
    pdl_wait();
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= b.total_faces * n2) return;
    const long long gf = t / n2;
    const int ab = (int)(t - gf * n2);
    const Item &it = find_item_face(b, gf);
    if (it.clk && it.clk->done) return;
    const int E = it.E;
    // threads walk the faces element-major (the three +d faces of element 0,
    // then of element 1, ...), so that the state sectors an element's faces
    // share (every xi and eta trace sector holds nodes of both ends) are
    // fetched from DRAM once and then hit in L2; storage stays f = d*E + eL
    const int lf = (int)(gf - it.face_begin);
    const int eL = lf / 3;
    const int d = lf - 3 * eL;
    const int f = d * E + eL;
    const int eR = nbr_plus(eL, d, it.ex, it.ey, it.ez);
    const int ta = ab % n, tb = ab / n;
    const int pL = face_node<n>(d, N, ta, tb), pR = face_node<n>(d, 0, ta, tb);

    const Phys<double> P = phys_of<double>(it);
    double uL[5], uR[5];
    const double *UL = it.u + (size_t)eL * 5 * n3 + pL, *UR = it.u + (size_t)eR * 5 * n3 + pR;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        uL[v] = UL[v * n3];
        uR[v] = UR[v * n3];
    }
    const double *Fn = it.fn + (size_t)f * 3 * n2 + ab;
    const double s1 = Fn[0], s2 = Fn[n2], s3 = Fn[2 * n2];
    double gl[kVisc], gr[kVisc];
    if (NS) {
        const double *GL = (const double *)it.grad + (size_t)eL * kVisc * n3 + pL;
        const double *GR = (const double *)it.grad + (size_t)eR * kVisc * n3 + pR;
#pragma unroll
        for (int k = 0; k < kVisc; ++k) {
            gl[k] = GL[k * n3];
            gr[k] = GR[k * n3];
        }
    }
    const Prim<double> qL = prim_from_u<double>(uL, P.gm1), qR = prim_from_u<double>(uR, P.gm1);
    double fs[5];
    if (flux == HS3D_FLUX_EC) flux_ec(ec_node(qL), ec_node(qR), P.hg, s1, s2, s3, fs);
    else if (flux == HS3D_FLUX_LF) flux_lf(qL, uL, qR, uR, P.gamma, s1, s2, s3, fs);
    else if (flux == HS3D_FLUX_RUSANOV) flux_rusanov(qL, uL, qR, uR, P.gamma, s1, s2, s3, fs);
    else if (flux == HS3D_FLUX_MATRIX) flux_matrix(qL, qR, P.gamma, P.hg, s1, s2, s3, fs);
    else if (flux == HS3D_FLUX_LDROE) flux_ldroe(qL, uL, qR, uR, P.gamma, s1, s2, s3, fs);
    else flux_roe(qL, uL, qR, uR, P.gamma, s1, s2, s3, fs);
    if (NS) {
        double fl[5], fr[5];
        visc_flux(qL, gl, s1, s2, s3, fl);
        visc_flux(qR, gr, s1, s2, s3, fr);
#pragma unroll
        for (int v = 1; v < 5; ++v) fs[v] -= 0.5 * (fl[v] + fr[v]);
    }
    double *out = (double *)it.fstar + (size_t)f * 5 * n2 + ab;
#pragma unroll
    for (int v = 0; v < 5; ++v) out[v * n2] = fs[v];
}

// ------------------------------------------------------------------ BR1 gradients

template <int N>
constexpr int grad_threads()
{
    return max_cta_threads(N, HS3D_FP64, kShapeGrad, HS3D_VOL_STANDARD, false);
}

// (v, T) of a conserved state.
__device__ __forceinline__ void grad_vars(const double u[5], double gm1, double out[4])
{
    const Prim<double> q = prim_from_u<double>(u, gm1);
    out[0] = q.v1;
    out[1] = q.v2;
    out[2] = q.v3;
    out[3] = q.p * q.ir;
}

// Shared memory per element (doubles): the nine stress products of one
// direction, or of all three where they fit beside enough CTAs (n^3 <= 125: one
// barrier per direction less), [1 or 3][9][n3], and the neighbour traces of q
// [6 faces][4][n2] (slot 2d: the -d face, slot 2d+1: the +d face).  The products
// Ja^d_c q_v are combined once per node and direction (12 FP64 instructions),
// so that the contraction takes 9 multiply-adds per pair of nodes instead of 15
// instructions (with the Roe flux's summed Euler part: 16^3, N = 3, two steps
// 2.53 -> 2.45 ms; 11x12x13, N = 4, KG, RK4 1.65 -> 1.56).
template <int N>
constexpr int grad_buffers()
{
    return (N + 1) * (N + 1) * (N + 1) <= 125 ? 3 : 1;
}
template <int N>
constexpr int grad_per_elem()
{
    return grad_buffers<N>() * kVisc * (N + 1) * (N + 1) * (N + 1) + 24 * (N + 1) * (N + 1);
}

template <int N>
__global__ void __launch_bounds__(grad_threads<N>()) k_grad(const __grid_constant__ Batch b, const Ops *__restrict__ ops)
{
    constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
    constexpr int PER_ELEM = grad_per_elem<N>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *sD = (double *)smem_raw;                 // n*n
    double *sE = sD + ((n * n + 1) & ~1);            // [epb][PER_ELEM]
    pdl_wait();
    const int epb = blockDim.x / n3;
    for (int t = threadIdx.x; t < n * n; t += blockDim.x) sD[t] = ops->D[t];
    const int le = threadIdx.x / n3, p = threadIdx.x - le * n3;
    const long long ge = blockIdx.x * (long long)epb + le;
    bool valid = ge < b.total_elems;
    const Item *itp = nullptr;
    int e = 0;
    if (valid) {
        itp = &find_item_elem(b, ge);
        e = (int)(ge - itp->elem_begin);
        if (itp->clk && itp->clk->done) valid = false;
    }
    constexpr int NB = grad_buffers<N>();
    double *W = sE + (size_t)le * PER_ELEM;
    double *qn = W + NB * kVisc * n3;
    double ja[9] = {}, qin[4] = {};
    if (valid) {
        const Item &it = *itp;
        const double gm1 = it.gm1;
        // neighbour traces of q: all loads of this thread's face points first
        // (the loop is unrolled to its fixed trip count), then the conversions
        constexpr int IT = (6 * n2 + n3 - 1) / n3;
        const Nbrs nbs = elem_nbrs(e, it.ex, it.ey, it.ez);
        double raw[IT][5];
#pragma unroll
        for (int k = 0; k < IT; ++k) {
            const int t = p + k * n3;
            if (t < 6 * n2) {
                const int slot = t / n2, ab = t - slot * n2;
                if (it.face6) {
                    // mesh with per-element degrees: the mortar kernel left 2 q*_e - q_in
                    const double *src = (const double *)it.qhat6 + ((size_t)slot * it.E + e) * 4 * n2 + ab;
#pragma unroll
                    for (int v = 0; v < 4; ++v) raw[k][v] = src[v * n2];
                } else {
                    const int d = slot >> 1, plus = slot & 1;
                    const int pn = face_node<n>(d, plus ? 0 : N, ab % n, ab / n);
                    const double *src = it.u + (size_t)nbr_of_slot(nbs, slot) * 5 * n3 + pn;
#pragma unroll
                    for (int v = 0; v < 5; ++v) raw[k][v] = src[v * n3];
                }
            }
        }
        double uo[5];
        const double *U = it.u + (size_t)e * 5 * n3 + p;
        const double *JA = it.Ja + (size_t)e * 9 * n3 + p;
#pragma unroll
        for (int v = 0; v < 5; ++v) uo[v] = U[v * n3];
#pragma unroll
        for (int k = 0; k < 9; ++k) ja[k] = JA[k * n3];
#pragma unroll
        for (int k = 0; k < IT; ++k) {
            const int t = p + k * n3;
            if (t < 6 * n2) {
                const int slot = t / n2, ab = t - slot * n2;
                double g4[4];
                if (it.face6) {
#pragma unroll
                    for (int v = 0; v < 4; ++v) g4[v] = raw[k][v];
                } else {
                    grad_vars(raw[k], gm1, g4);
                }
#pragma unroll
                for (int v = 0; v < 4; ++v) qn[(slot * 4 + v) * n2 + ab] = g4[v];
            }
        }
        grad_vars(uo, gm1, qin);
    }
    const int ijk[3] = {p % n, (p / n) % n, p / n2};
    double acc[kVisc];
#pragma unroll
    for (int k = 0; k < kVisc; ++k) acc[k] = 0.0;
    // the other nodes of the line through this one
    auto contract = [&](const double *Wd, const double *Drow, int base, int stride, int i) {
#pragma unroll
        for (int k = 1; k < n; ++k) {
            const int m = (i + k < n) ? i + k : i + k - n;
            const double Dm = Drow[m];
#pragma unroll
            for (int c = 0; c < kVisc; ++c) acc[c] += Dm * Wd[c * n3 + base + m * stride];
        }
    };
    // D_ii is zero inside and -+1/(2w) at the two ends, where the BR1 lift
    // +-(1/w)(q_out - q_in)/2 Ja turns the diagonal term D_ii Ja q_in into
    // D_ii Ja q_out: no separate lift
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int i = ijk[d];
        const int stride = (d == 0) ? 1 : (d == 1) ? n : n2;
        const int base = p - i * stride;
        const double *Drow = sD + i * n;
        double *Wd = W + (NB == 3 ? d * kVisc * n3 : 0);
        if (NB == 1 && d > 0) __syncthreads();   // the previous direction's products are consumed
        if (valid) {
            double w[kVisc] = {};
            stress_add(w, ja[d * 3], ja[d * 3 + 1], ja[d * 3 + 2], qin[0], qin[1], qin[2], qin[3]);
#pragma unroll
            for (int c = 0; c < kVisc; ++c) Wd[c * n3 + p] = w[c];
        }
        if (NB == 1 || d == 2) __syncthreads();
        if (NB == 1 && valid) contract(Wd, Drow, base, stride, i);
    }
    if (!valid) return;
    if constexpr (NB == 3) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int stride = (d == 0) ? 1 : (d == 1) ? n : n2;
            contract(W + d * kVisc * n3, sD + ijk[d] * n, p - ijk[d] * stride, stride, ijk[d]);
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int i = ijk[d];
        if (i != 0 && i != N) continue;
        const int ta = (d == 0) ? ijk[1] : ijk[0];
        const int tb = (d == 2) ? ijk[1] : ijk[2];
        const double *Q = qn + (2 * d + (i == N ? 1 : 0)) * 4 * n2 + ta + n * tb;
        const double Dm = sD[i * n + i];
        stress_add(acc, Dm * ja[d * 3], Dm * ja[d * 3 + 1], Dm * ja[d * 3 + 2], Q[0], Q[n2], Q[2 * n2], Q[3 * n2]);
    }
    const Item &it = *itp;
    double t[kVisc];
    stress_of(acc, it.invJ[(size_t)e * n3 + p], it.mu, it.kappa, t);
    double *G = (double *)it.grad + (size_t)e * kVisc * n3 + p;
#pragma unroll
    for (int k = 0; k < kVisc; ++k) G[k * n3] = t[k];
}

// ------------------------------------------------------------------ launchers

template <int N>
static cudaError_t face_launch(int physics, int flux, const Batch &b, cudaStream_t s)
{
    constexpr int n2 = (N + 1) * (N + 1);
    long long total = b.total_faces * n2;
    if (total == 0) return cudaSuccess;
    const unsigned blocks = (unsigned)((total + kFaceThreads - 1) / kFaceThreads);
    cudaError_t e = physics == HS3D_NS ? launch_pdl(k_face<N, true>, blocks, kFaceThreads, 0, s, b, flux)
                                       : launch_pdl(k_face<N, false>, blocks, kFaceThreads, 0, s, b, flux);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int N>
static cudaError_t grad_launch(const Batch &b, cudaStream_t s)
{
    constexpr int n = N + 1, n3 = n * n * n;
    if (b.total_elems == 0) return cudaSuccess;
    const int epb = elems_per_cta(N, HS3D_FP64, kShapeGrad, HS3D_VOL_STANDARD, false, b.total_elems, b.beside);
    int threads = epb * n3;
    size_t smem = sizeof(double) * (((n * n + 1) & ~1) + (size_t)epb * grad_per_elem<N>());
    unsigned blocks = (unsigned)((b.total_elems + epb - 1) / epb);
    const Ops *ops = device_ops(N);
    if (!ops) return cudaErrorMemoryAllocation;
    cudaError_t e = launch_pdl(k_grad<N>, blocks, threads, smem, s, b, ops);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int N>
static cudaError_t prep_grad()
{
    cudaError_t e = cudaFuncSetAttribute(k_grad<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_grad<N>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) e = prepare_grad_dev(N);
    return e;
}

#define HS3D_SWITCH_N(CALL_N)                 \
    switch (N) {                              \
        case 1: return CALL_N(1);             \
        case 2: return CALL_N(2);             \
        case 3: return CALL_N(3);             \
        case 4: return CALL_N(4);             \
        case 5: return CALL_N(5);             \
        case 6: return CALL_N(6);             \
        case 7: return CALL_N(7);             \
        default: return cudaErrorInvalidValue; \
    }

cudaError_t prepare_grad(int N)
{
#define P(K) prep_grad<K>()
    HS3D_SWITCH_N(P)
#undef P
}

cudaError_t launch_face(int N, int prec, int physics, int flux, const Batch &b, cudaStream_t s)
{
    if (b.gauss) return launch_face_gauss(N, prec, physics, flux, b, s);
    if (prec != HS3D_FP64) return launch_face_dev(N, physics, flux, b, s);
#define F64(K) face_launch<K>(physics, flux, b, s)
    HS3D_SWITCH_N(F64)
#undef F64
}

cudaError_t launch_grad(int N, int prec, const Batch &b, cudaStream_t s)
{
    if (b.gauss) return launch_grad_gauss(N, prec, b, s);
    if (prec != HS3D_FP64) return launch_grad_dev(N, b, s);
#define G64(K) grad_launch<K>(b, s)
    HS3D_SWITCH_N(G64)
#undef G64
}

}  // namespace hs3d
