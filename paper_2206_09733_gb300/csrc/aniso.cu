// Anisotropic per-element degrees (Sec. 3.6: the order may differ per
// element and per reference direction, P_x, P_y, P_z), FP64.
//
// Element e has n_d = P_d + 1 Gauss-Lobatto nodes along d; node (i, j, k) is
// i + n_x (j + n_y k) and its state block [5][n_x n_y n_z] starts at off[e]
// (elements in mesh order).  Geometry: the element map is the degree-Ngeo
// interpolant (Ngeo = max(1, floor(Pmin/2)), Pmin over elements and
// directions) of the box map at the element's own nodes (built on the host,
// the free-stream rule of p-non-conforming faces), and the curl-form metric
// terms use each direction's own derivative matrix (k_ageo).
//
// A stage is
//   [k_amortar<0> -> k_agrad]   (Navier-Stokes: BR1 interface values, gradients)
//   k_amortar<1> -> k_avol      (face fluxes; volume + surface + 1/J + RK stage)
// The face between L (its +d face, tangential degrees (P_L[d0], P_L[d1]))
// and R (its -d face) carries a mortar of degree M_k = max(P_L[dk], P_R[dk])
// in each tangential direction k: both sides' traces (and gradients) are
// interpolated to the mortar points, the flux (or the BR1 value) is formed
// there with the face metric of a side whose tangential degrees are the
// mortar's (L first, then R; when neither is, L's face metric interpolated,
// exact since it has degree <= Pmin per direction), and each side receives
// its L2 projection, direction by direction (Kopriva et al. 2002, the method
// Sec. 3.6 names).  Each element face's result goes to its own block of the
// face arrays (fstar, qhat), at the face-node offset fnoff[6e + slot].
//
// The kernels are bound by the FP64 pipe (one warp instruction per 16 cycles
// and SM, however many lanes are active), so the stage kernels pack: elements
// are binned into CTAs of 256 (or 512) thread slots at mesh set-up, one slot
// per node (k_agrad, k_avol), and the faces of equal mortar degrees share CTAs
// of 128 threads, sorted by their sides' degrees so that a CTA's faces need
// the same passes (k_amortar).  Interpolation and projection go direction by
// direction and are skipped where the side has the mortar's degree; each pair
// of a line is evaluated once.  The set-up, initial-state and diagnostics
// kernels take one element per CTA, launched in classes by node count
// (kAnisoClass).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <new>
#include <tuple>
#include <vector>

#include "aniso.cuh"
#include "api_internal.h"
#include "ic.cuh"
#include "mortar.cuh"
#include "mortar_phys.cuh"
#include "physics.cuh"

namespace hs3d {

namespace {

// ------------------------------------------------------------------ device helpers

struct AShape {
    int n[3];
    int n3;
};

__device__ __forceinline__ AShape ashape(const int *P3, int e)
{
    AShape s;
    s.n[0] = P3[3 * e] + 1;
    s.n[1] = P3[3 * e + 1] + 1;
    s.n[2] = P3[3 * e + 2] + 1;
    s.n3 = s.n[0] * s.n[1] * s.n[2];
    return s;
}

__device__ __forceinline__ int astride(const AShape &s, int d) { return d == 0 ? 1 : d == 1 ? s.n[0] : s.n[0] * s.n[1]; }

// tangential directions of face direction d, in increasing order
__device__ __forceinline__ void aface_dirs(int d, int &d0, int &d1)
{
    d0 = (d == 0) ? 1 : 0;
    d1 = (d == 2) ? 1 : 2;
}

// node of an element with index `end` along d and tangential indices (ta, tb)
__device__ __forceinline__ int aface_node(const AShape &s, int d, int end, int ta, int tb)
{
    int idx[3];
    int d0, d1;
    aface_dirs(d, d0, d1);
    idx[d] = end;
    idx[d0] = ta;
    idx[d1] = tb;
    return idx[0] + s.n[0] * (idx[1] + s.n[1] * idx[2]);
}

// sum_m D_d[i_d][m] f[node with index m along d] (f in shared memory)
__device__ __forceinline__ double aderiv(const AOps *ops, const AShape &s, const double *f, int p, const int ijk[3],
                                         int d)
{
    const int nd = s.n[d], st = astride(s, d);
    const double *Drow = ops->D[nd - 1] + ijk[d] * nd;
    const int base = p - ijk[d] * st;
    double acc = 0.0;
    for (int m = 0; m < nd; ++m) acc += Drow[m] * f[base + m * st];
    return acc;
}

struct APhys {
    double gamma, gm1, hg, mu, kappa;
    int physics, flux, form;
};

APhys aphys(const hs3d_solver_cfg *c)
{
    APhys P;
    P.gamma = c->gamma;
    P.gm1 = c->gamma - 1.0;
    P.hg = 0.5 / P.gm1;
    P.mu = c->physics == HS3D_NS ? 1.0 / c->Re : 0.0;
    P.kappa = c->physics == HS3D_NS ? P.mu * c->gamma / ((c->gamma - 1.0) * c->Pr) : 0.0;
    P.physics = c->physics;
    P.flux = c->surface_flux;
    P.form = c->volume_form;
    return P;
}

// ------------------------------------------------------------------ geometry

// J, 1/J and the curl-form metric terms (Kopriva 2006) of every element from
// its node coordinates X (already in place), each derivative along d with the
// derivative matrix of the element's degree in d.
__global__ void __launch_bounds__(512) k_ageo(const int *__restrict__ elems, const int *__restrict__ P3, const long long *__restrict__ noff,
                       const AOps *__restrict__ ops, const double *__restrict__ Xall, double *__restrict__ Jaall,
                       double *__restrict__ Jall, double *__restrict__ invJall)
{
    extern __shared__ double sm[];
    const int e = elems[blockIdx.x];
    const AShape s = ashape(P3, e);
    const int n3 = s.n3, p = threadIdx.x;
    const bool live = p < n3;
    double *sX = sm;             // [3][n3]
    double *sT = sm + 3 * n3;    // [2][n3]
    const long long nb = noff[e];
    const double *X = Xall + 3 * nb;
    int ijk[3] = {0, 0, 0};
    double x[3] = {0, 0, 0};
    if (live) {
        ijk[0] = p % s.n[0];
        ijk[1] = (p / s.n[0]) % s.n[1];
        ijk[2] = p / (s.n[0] * s.n[1]);
        for (int c = 0; c < 3; ++c) x[c] = sX[c * n3 + p] = X[(size_t)c * n3 + p];
    }
    __syncthreads();
    double a[3][3] = {};   // a[d][c] = dX_c / dxi_d
    if (live)
        for (int d = 0; d < 3; ++d)
            for (int c = 0; c < 3; ++c) a[d][c] = aderiv(ops, s, sX + c * n3, p, ijk, d);
    if (live) {
        const double Jp = a[0][0] * (a[1][1] * a[2][2] - a[1][2] * a[2][1]) +
                          a[0][1] * (a[1][2] * a[2][0] - a[1][0] * a[2][2]) +
                          a[0][2] * (a[1][0] * a[2][1] - a[1][1] * a[2][0]);
        Jall[nb + p] = Jp;
        invJall[nb + p] = 1.0 / Jp;
    }
    double *Ja = Jaall + 9 * nb;
    for (int i = 0; i < 3; ++i) {
        const int i1 = (i + 1) % 3, i2 = (i + 2) % 3;
        for (int c = 0; c < 3; ++c) {
            const int m = (c + 1) % 3, l = (c + 2) % 3;
            __syncthreads();
            if (live) {
                sT[p] = x[l] * a[i1][m];
                sT[n3 + p] = x[l] * a[i2][m];
            }
            __syncthreads();
            if (live) Ja[(size_t)(i * 3 + c) * n3 + p] = aderiv(ops, s, sT, p, ijk, i2) - aderiv(ops, s, sT + n3, p, ijk, i1);
        }
    }
}

// ------------------------------------------------------------------ initial state

__global__ void __launch_bounds__(512) k_ainit(const int *__restrict__ elems, const int *__restrict__ P3, const long long *__restrict__ noff,
                        const double *__restrict__ Xall, hs3d_ic ic, double Lx, double Ly, double *__restrict__ u)
{
    const int e = elems[blockIdx.x];
    const AShape s = ashape(P3, e);
    const int p = threadIdx.x;
    if (p >= s.n3) return;
    const long long nb = noff[e];
    const double *X = Xall + 3 * nb;
    double w[5];
    ic_point(ic, Lx, Ly, X[p], X[s.n3 + p], X[2 * s.n3 + p], w);
    double *ue = u + 5 * nb;
    for (int v = 0; v < 5; ++v) ue[(size_t)v * s.n3 + p] = w[v];
}

// ------------------------------------------------------------------ dt maxima

// Per node: lam_c = sum_d n_d^2 (|Ja^d.v| + c |Ja^d|)/J and
// lam_v = (mu/rho) sum_d n_d^4 (|Ja^d|/J)^2 (each direction's resolution
// inside the sum), reduced to the clock's slot as bit patterns.
__device__ __forceinline__ void alam_node(const AShape &s, const double *Ja, int p, double iJ, const Prim<double> &q,
                                          const APhys &P, double &lc, double &lv)
{
    const double c = sound_speed(q, P.gamma);
    double sc = 0.0, sv = 0.0;
    for (int d = 0; d < 3; ++d) {
        const double a1 = Ja[(size_t)(d * 3) * s.n3 + p], a2 = Ja[(size_t)(d * 3 + 1) * s.n3 + p],
                     a3 = Ja[(size_t)(d * 3 + 2) * s.n3 + p];
        const double s2 = a1 * a1 + a2 * a2 + a3 * a3;
        const double n2 = (double)(s.n[d] * s.n[d]);
        sc += n2 * (fabs(a1 * q.v1 + a2 * q.v2 + a3 * q.v3) + c * sqrt_(s2));
        sv += n2 * n2 * s2;
    }
    lc = sc * iJ;
    lv = P.physics == HS3D_NS ? P.mu * sv * (iJ * iJ) * q.ir : 0.0;
}

// The element, its shape and this thread's node of a packed launch: slot
// blockIdx.x T + threadIdx.x; origin is the element's first thread.
struct ASlot {
    int e, p, origin;
    AShape s;
};
__device__ __forceinline__ bool aslot(const int *__restrict__ slot_elem, const int *__restrict__ slot0,
                                      const int *__restrict__ P3, ASlot &a)
{
    a.e = slot_elem[(size_t)blockIdx.x * blockDim.x + threadIdx.x];
    if (a.e < 0) return false;
    a.origin = slot0[a.e];
    a.p = (int)threadIdx.x - a.origin;
    a.s = ashape(P3, a.e);
    return true;
}

__global__ void __launch_bounds__(512) k_alambda(const int *__restrict__ slot_elem, const int *__restrict__ slot0,
                                                 const int *__restrict__ P3, const long long *__restrict__ noff,
                                                 const double *__restrict__ Jaall, const double *__restrict__ invJall,
                                                 const double *__restrict__ u, APhys P, Clock *clk, int slot)
{
    ASlot S{};
    const bool live = aslot(slot_elem, slot0, P3, S);
    double lc = 0.0, lv = 0.0;
    if (live) {
        const long long nb = noff[S.e];
        double w[5];
        for (int v = 0; v < 5; ++v) w[v] = u[5 * nb + (size_t)v * S.s.n3 + S.p];
        const Prim<double> q = prim_from_u<double>(w, P.gm1);
        if (!(q.rho > 0.0) || !(q.p > 0.0)) clk->bad = 1;
        else alam_node(S.s, Jaall + 9 * nb, S.p, invJall[nb + S.p], q, P, lc, lv);
    }
    cta_max_to_clock<double>(clk->lam[slot], P.physics == HS3D_NS, lc, lv);
}

// ------------------------------------------------------------------ mortar faces

// The faces of one CTA: `count` faces from `face0` of the table sorted by
// mortar degrees (nm0 x nm1 points each); passes: bit 0 / 1, some face's L / R
// side needs the first-direction interpolation and projection.
//   MODE 0: q* = (q(u_L) + q(u_R))/2 at the mortar points -> qhat of both sides (4 values);
//   MODE 1: s F*(u_L, u_R; n) - (F_v(L) + F_v(R)).Sn/2 -> fstar of both sides (5 values,
//           oriented along +d).
// 16^3 elements of degrees 2..5 (NS, Roe): flux launch 1331 -> 247 us, interface
// values 491 -> 74 us against one face per 64-thread CTA with both directions
// interpolated at once for every side.
constexpr int kAFaceThreads = 128;

template <int MODE, bool NS>
__global__ void __launch_bounds__(kAFaceThreads) k_amortar(const AFace *__restrict__ faces,
                                                           const AFaceCta *__restrict__ ctas,
                                                           const int *__restrict__ P3,
                                                           const long long *__restrict__ noff,
                                                           const long long *__restrict__ fnoff,
                                                           const double *__restrict__ u,
                                                           const double *__restrict__ grad,
                                                           const double *__restrict__ Jaall,
                                                           const MortarOps *__restrict__ mo, APhys P,
                                                           double *__restrict__ out)
{
    constexpr int T = kAFaceThreads;
    constexpr int NV = (MODE == 1 && NS) ? 5 + kVisc : 5;   // conservative state (+ viscous stress) per trace point
    constexpr int NO = MODE == 0 ? 4 : 5;
    constexpr int NM = MODE == 1 ? 3 : 0;                   // face metric
    __shared__ double tr[2][NV][T];
    __shared__ double sn[NM > 0 ? NM : 1][T];
    __shared__ double fm[NO][T];
    __shared__ double gk[2][NO][T];
    pdl_wait();
    const AFaceCta C = ctas[blockIdx.x];
    const int nm0 = C.nm0, nm1 = C.nm1, nM2 = nm0 * nm1;
    const int fi = threadIdx.x / nM2, p = threadIdx.x - fi * nM2, o = fi * nM2;
    const bool live = fi < C.count;
    AFace F{0, 0, 0};
    if (live) F = faces[C.face0 + fi];
    const int d = F.d;
    int d0, d1;
    aface_dirs(d, d0, d1);
    const int eS[2] = {F.eL, F.eR};
    AShape sh[2];
    int n0[2], n1[2];   // the sides' points per tangential direction
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        sh[k] = ashape(P3, eS[k]);
        n0[k] = d0 == 0 ? sh[k].n[0] : sh[k].n[1];
        n1[k] = d1 == 2 ? sh[k].n[2] : sh[k].n[1];
    }
    // the face metric of a side whose tangential degrees are the mortar's (L
    // first), else L's, interpolated (hk < 0)
    const int hk = (n0[0] == nm0 && n1[0] == nm1) ? 0 : (n0[1] == nm0 && n1[1] == nm1) ? 1 : -1;

    // 1. both sides' traces on their own face points
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (live && p < n0[k] * n1[k]) {
            const int node = aface_node(sh[k], d, k == 0 ? sh[k].n[d] - 1 : 0, p % n0[k], p / n0[k]);
            const long long nb = noff[eS[k]];
            const int n3 = sh[k].n3;
#pragma unroll
            for (int v = 0; v < 5; ++v) tr[k][v][o + p] = u[5 * nb + (size_t)v * n3 + node];
            if constexpr (MODE == 1 && NS) {
#pragma unroll
                for (int q = 0; q < kVisc; ++q) tr[k][5 + q][o + p] = grad[kVisc * nb + (size_t)q * n3 + node];
            }
            if constexpr (MODE == 1) {
                if (k == (hk > 0 ? 1 : 0)) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) sn[c][o + p] = Jaall[9 * nb + (size_t)(d * 3 + c) * n3 + node];
                }
            }
        }
    }
    __syncthreads();

    // 2. first tangential direction, in place: (n0 x n1) -> (nm0 x n1) points
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (!(C.passes & (1 << k))) continue;   // (uniform over the CTA)
        double r[NV], rs[3] = {0.0, 0.0, 0.0};
        const bool mine = live && n0[k] < nm0 && p < nm0 * n1[k];
        if (mine) {
            const int a = p % nm0, j = p / nm0;
            const double *I = mo->Pi[n0[k] - 1][nm0 - 1] + a * n0[k];
            const int src = o + n0[k] * j;
#pragma unroll
            for (int v = 0; v < NV; ++v) r[v] = 0.0;
            for (int i = 0; i < n0[k]; ++i) {
                const double w = I[i];
#pragma unroll
                for (int v = 0; v < NV; ++v) r[v] += w * tr[k][v][src + i];
                if constexpr (MODE == 1) {
                    if (k == 0 && hk < 0) {
#pragma unroll
                        for (int c = 0; c < 3; ++c) rs[c] += w * sn[c][src + i];
                    }
                }
            }
        }
        __syncthreads();
        if (mine) {
#pragma unroll
            for (int v = 0; v < NV; ++v) tr[k][v][o + p] = r[v];
            if constexpr (MODE == 1) {
                if (k == 0 && hk < 0) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) sn[c][o + p] = rs[c];
                }
            }
        }
    }
    if (C.passes) __syncthreads();

    // 3. second direction into registers, and the mortar function at this point
    if (live) {
        const int a = p % nm0, b = p / nm0;
        double w[2][NV];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (n1[k] < nm1) {
                const double *I = mo->Pi[n1[k] - 1][nm1 - 1] + b * n1[k];
#pragma unroll
                for (int v = 0; v < NV; ++v) w[k][v] = 0.0;
                for (int j = 0; j < n1[k]; ++j) {
                    const double c = I[j];
#pragma unroll
                    for (int v = 0; v < NV; ++v) w[k][v] += c * tr[k][v][o + a + nm0 * j];
                }
            } else {
#pragma unroll
                for (int v = 0; v < NV; ++v) w[k][v] = tr[k][v][o + p];
            }
        }
        if constexpr (MODE == 0) {
            double qL[4], qR[4];
            mortar_q(w[0], P.gm1, qL);
            mortar_q(w[1], P.gm1, qR);
#pragma unroll
            for (int v = 0; v < 4; ++v) fm[v][o + p] = 0.5 * (qL[v] + qR[v]);
        } else {
            double s3[3];
            if (hk < 0 && n1[0] < nm1) {
                const double *I = mo->Pi[n1[0] - 1][nm1 - 1] + b * n1[0];
                s3[0] = s3[1] = s3[2] = 0.0;
                for (int j = 0; j < n1[0]; ++j)
#pragma unroll
                    for (int c = 0; c < 3; ++c) s3[c] += I[j] * sn[c][o + a + nm0 * j];
            } else {
#pragma unroll
                for (int c = 0; c < 3; ++c) s3[c] = sn[c][o + p];
            }
            const MortarPhys<double> mp{P.gamma, P.gm1, P.hg, P.mu, P.kappa};
            double fs[5];
            mortar_riemann<double>(P.flux, w[0], w[1], mp, s3[0], s3[1], s3[2], fs);
            if constexpr (NS) {
                double fl[5], fr[5];
                const Prim<double> pL = mortar_prim(w[0], P.gm1), pR = mortar_prim(w[1], P.gm1);
                visc_flux(pL, &w[0][5], s3[0], s3[1], s3[2], fl);
                visc_flux(pR, &w[1][5], s3[0], s3[1], s3[2], fr);
#pragma unroll
                for (int v = 1; v < 5; ++v) fs[v] -= 0.5 * (fl[v] + fr[v]);
            }
#pragma unroll
            for (int v = 0; v < 5; ++v) fm[v][o + p] = fs[v];
        }
    }
    __syncthreads();

    // 4. each side's L2 projection onto its own face points, first direction ...
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (live && n0[k] < nm0 && p < n0[k] * nm1) {
            const int a = p % n0[k], j = p / n0[k];
            const double *P0 = mo->P[n0[k] - 1][nm0 - 1] + a * nm0;
            double r[NO];
#pragma unroll
            for (int v = 0; v < NO; ++v) r[v] = 0.0;
            for (int i = 0; i < nm0; ++i) {
                const double w = P0[i];
#pragma unroll
                for (int v = 0; v < NO; ++v) r[v] += w * fm[v][o + i + nm0 * j];
            }
#pragma unroll
            for (int v = 0; v < NO; ++v) gk[k][v][o + p] = r[v];
        }
    }
    if (C.passes) __syncthreads();

    // ... then the second, into the side's face block
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int f2 = n0[k] * n1[k];
        if (live && p < f2) {
            const int a = p % n0[k], b = p / n0[k];
            const double *src = (n0[k] < nm0 ? &gk[k][0][0] : &fm[0][0]) + o;
            const int slot = 2 * d + (k == 0 ? 1 : 0);
            double *dst = out + (size_t)NO * fnoff[6 * eS[k] + slot] + p;
            double r[NO];
            if (n1[k] < nm1) {
                const double *P1 = mo->P[n1[k] - 1][nm1 - 1] + b * nm1;
#pragma unroll
                for (int v = 0; v < NO; ++v) r[v] = 0.0;
                for (int j = 0; j < nm1; ++j) {
                    const double w = P1[j];
#pragma unroll
                    for (int v = 0; v < NO; ++v) r[v] += w * src[v * T + a + n0[k] * j];
                }
            } else {
#pragma unroll
                for (int v = 0; v < NO; ++v) r[v] = src[v * T + p];
            }
#pragma unroll
            for (int v = 0; v < NO; ++v) dst[(size_t)v * f2] = r[v];
        }
    }
}

// ------------------------------------------------------------------ BR1 gradients

// J grad q_c = sum_d D_d (Ja^d_c q) + sum_faces (q*_e - q_in) (+-Ja^d_c)/w_end,
// q = (v1, v2, v3, T), q*_e from the mortar kernel, stored as viscous stress and
// heat flux [kVisc][n3] at kVisc noff[e].  D_ii is zero inside and -+1/(2w) at
// the two ends, where the lift turns the diagonal term D_ii Ja q_in into
// D_ii Ja (2 q* - q_in); the nine stress products are formed once per node and
// direction.  16^3 elements of degrees 2..5: 484 -> 174 us per stage.
template <int T>
__global__ void __launch_bounds__(T) k_agrad(const int *__restrict__ slot_elem, const int *__restrict__ slot0,
                                             const int *__restrict__ P3, const long long *__restrict__ noff,
                                             const long long *__restrict__ fnoff, const AOps *__restrict__ ops,
                                             const double *__restrict__ u, const double *__restrict__ Jaall,
                                             const double *__restrict__ invJall, const double *__restrict__ qhat,
                                             APhys P, double *__restrict__ gradall)
{
    extern __shared__ double sm[];   // the stress products of one direction [kVisc][T]
    pdl_wait();
    ASlot S{};
    const bool live = aslot(slot_elem, slot0, P3, S);
    const int t = threadIdx.x;
    double qp[4] = {0, 0, 0, 0};
    long long nb = 0;
    int ijk[3] = {0, 0, 0}, n3 = 1;
    if (live) {
        nb = noff[S.e];
        n3 = S.s.n3;
        mortar_q(u + 5 * nb + S.p, P.gm1, qp, n3);
        ijk[0] = S.p % S.s.n[0];
        ijk[1] = (S.p / S.s.n[0]) % S.s.n[1];
        ijk[2] = S.p / (S.s.n[0] * S.s.n[1]);
    }
    const double *Ja = Jaall + 9 * nb + S.p;
    double G[kVisc] = {};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int nd = live ? S.s.n[d] : 1, st = live ? astride(S.s, d) : 0, i = ijk[d];
        double a1 = 0.0, a2 = 0.0, a3 = 0.0;
        if (d > 0) __syncthreads();   // the previous direction's products are consumed
        if (live) {
            a1 = Ja[(size_t)(d * 3) * n3];
            a2 = Ja[(size_t)(d * 3 + 1) * n3];
            a3 = Ja[(size_t)(d * 3 + 2) * n3];
            double w[kVisc] = {};
            stress_add(w, a1, a2, a3, qp[0], qp[1], qp[2], qp[3]);
#pragma unroll
            for (int c = 0; c < kVisc; ++c) sm[c * T + t] = w[c];
        }
        __syncthreads();
        if (live) {
            const double *Drow = ops->D[nd - 1] + i * nd;
            for (int k = 1; k < nd; ++k) {
                const int m = (i + k < nd) ? i + k : i + k - nd, pm = t + (m - i) * st;
                const double Dm = Drow[m];
#pragma unroll
                for (int c = 0; c < kVisc; ++c) G[c] += Dm * sm[c * T + pm];
            }
            if (i == 0 || i == nd - 1) {
                int d0, d1;
                aface_dirs(d, d0, d1);
                const int f2 = S.s.n[d0] * S.s.n[d1];
                const int slot = 2 * d + (i != 0 ? 1 : 0);
                const double *qs = qhat + (size_t)4 * fnoff[6 * S.e + slot] + ijk[d0] + S.s.n[d0] * ijk[d1];
                const double Dm = Drow[i];
                stress_add(G, Dm * a1, Dm * a2, Dm * a3, 2.0 * qs[0] - qp[0], 2.0 * qs[f2] - qp[1],
                           2.0 * qs[2 * f2] - qp[2], 2.0 * qs[3 * f2] - qp[3]);
            }
        }
    }
    if (!live) return;
    double tau[kVisc];
    stress_of(G, invJall[nb + S.p], P.mu, P.kappa, tau);
    double *Gout = gradall + kVisc * nb + S.p;
#pragma unroll
    for (int k = 0; k < kVisc; ++k) Gout[(size_t)k * S.s.n3] = tau[k];
}

// ------------------------------------------------------------------ volume + surface + RK

// du/dt = -(V + S)/J at every node; V the standard or split-form volume term
// (each direction with its own D), S = sum_faces (+-F*_e - (F_e - F_v)(in).(+-Ja^d))/w_end
// (split forms without the diagonal pair, as volume_kernel.cuh explains).
// stage < 0: du/dt into out; else the low-storage RK stage with coefficients
// (A, B) and the clock's dt, and (lam_slot >= 0) the new state's dt maxima.
// The pairs of an element's lines are spread over its threads by position
// first: thread q of the element takes position x = q / (n3/n_d) of line
// q mod (n3/n_d) and evaluates (x, x + k mod n_d), k = 1 .. n_d/2 (the half-way
// pair of an even n_d for x < n_d/2 only, the element's lower threads).
// 16^3 elements of degrees 2..5, NS, Chandrashekar form: 1266 -> 391 us per stage.
// Dynamic shared memory per thread slot (doubles): standard form the
// directional flux 5; split forms the pair inputs, Ja^d 3, F_v.Ja^d 4 (NS) and
// the pair fluxes [kp][5], kp = floor(n_max/2).
template <int FORM, bool NS>
constexpr int avol_smem_per(int kp)
{
    return FORM == HS3D_VOL_STANDARD ? 5 : split_slots64<FORM>() + 3 + (NS ? 4 : 0) + 5 * kp;
}

template <int T, bool NS, int FORM>
__global__ void __launch_bounds__(T, 512 / T) k_avol(const int *__restrict__ slot_elem, const int *__restrict__ slot0,
                                            const int *__restrict__ P3, const long long *__restrict__ noff,
                                            const long long *__restrict__ fnoff, const AOps *__restrict__ ops,
                                            double *__restrict__ u, double *__restrict__ g, double *__restrict__ out,
                                            const double *__restrict__ Jaall, const double *__restrict__ invJall,
                                            const double *__restrict__ gradall, const double *__restrict__ fstar,
                                            APhys P, Clock *clk, int stage, double rkA, double rkB, int lam_slot)
{
    constexpr bool STD = FORM == HS3D_VOL_STANDARD;
    constexpr int ZS = split_slots64<FORM>();
    extern __shared__ double sm[];
    pdl_wait();
    ASlot S{};
    // (a finished or failed run's clock stops its stages, not a residual evaluation)
    const bool live = aslot(slot_elem, slot0, P3, S) && (stage < 0 || !(clk->done));
    const int t = threadIdx.x;
    double *sF = sm;                              // standard: directional flux [5][T]
    double *sZ = sm;                              // split: pair inputs [ZS][T]
    double *sA = sm + ZS * T;                     // Ja^d [3][T]
    double *sV = sA + 3 * T;                      // F_v.Ja^d [4][T] (NS)
    double *PB = sV + (NS ? 4 : 0) * T;           // pair fluxes [kp][5][T]
    long long nb = 0;
    const double *Ja = nullptr;
    int ijk[3] = {0, 0, 0}, n3 = 1;
    double w[5] = {0, 0, 0, 0, 0}, G[kVisc] = {};
    Prim<double> q{};
    if (live) {
        nb = noff[S.e];
        Ja = Jaall + 9 * nb + S.p;
        n3 = S.s.n3;
        ijk[0] = S.p % S.s.n[0];
        ijk[1] = (S.p / S.s.n[0]) % S.s.n[1];
        ijk[2] = S.p / (S.s.n[0] * S.s.n[1]);
#pragma unroll
        for (int v = 0; v < 5; ++v) w[v] = u[5 * nb + (size_t)v * n3 + S.p];
        q = prim_from_u<double>(w, P.gm1);
        if (NS) {
#pragma unroll
            for (int k = 0; k < kVisc; ++k) G[k] = gradall[kVisc * nb + (size_t)k * n3 + S.p];
        }
        if constexpr (!STD) {
            double z[ZS];
            split_node64<FORM>(q, z);
#pragma unroll
            for (int k = 0; k < ZS; ++k) sZ[k * T + t] = z[k];
        }
    }
    double R[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int nd = live ? S.s.n[d] : 1, st = live ? astride(S.s, d) : 0, i = ijk[d];
        int d0, d1;
        aface_dirs(d, d0, d1);
        double own[5] = {0, 0, 0, 0, 0};   // standard: (F_e - F_v).Ja^d; split: F_v.Ja^d
        if (d > 0) __syncthreads();        // the previous direction's shared values are consumed
        if (live) {
            const double a1 = Ja[(size_t)(d * 3) * n3], a2 = Ja[(size_t)(d * 3 + 1) * n3],
                         a3 = Ja[(size_t)(d * 3 + 2) * n3];
            double fv[5] = {0, 0, 0, 0, 0};
            if (NS) visc_flux(q, G, a1, a2, a3, fv);
            if constexpr (STD) {
                euler_flux(q, q.E, a1, a2, a3, own);
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                    if (NS && v > 0) own[v] -= fv[v];
                    sF[v * T + t] = own[v];
                }
            } else {
                sA[t] = a1;
                sA[T + t] = a2;
                sA[2 * T + t] = a3;
                if (NS) {
#pragma unroll
                    for (int v = 1; v < 5; ++v) sV[(v - 1) * T + t] = own[v] = fv[v];
                }
            }
        }
        __syncthreads();
        if constexpr (!STD) {
            if (live) {
                const int lines = n3 / nd;
                const int x = S.p / lines, l = S.p - x * lines;
                const int tb = l / S.s.n[d0], ta = l - tb * S.s.n[d0];
                const int a = S.origin + x * st + ta * astride(S.s, d0) + tb * astride(S.s, d1);
                double za[ZS];
#pragma unroll
                for (int k = 0; k < ZS; ++k) za[k] = sZ[k * T + a];
                const double j1 = sA[a], j2 = sA[T + a], j3 = sA[2 * T + a];
                for (int k = 1; 2 * k <= nd; ++k) {
                    if (2 * k == nd && x >= k) break;
                    const int c = a + ((x + k < nd) ? k : k - nd) * st;
                    double zc[ZS], fs[5];
#pragma unroll
                    for (int m = 0; m < ZS; ++m) zc[m] = sZ[m * T + c];
                    split_pair64<FORM>(za, zc, P.gamma, P.hg, j1 + sA[c], j2 + sA[T + c], j3 + sA[2 * T + c], fs);
#pragma unroll
                    for (int v = 0; v < 5; ++v) PB[((k - 1) * 5 + v) * T + t] = fs[v];
                }
            }
            __syncthreads();
        }
        if (live) {
            const double *Drow = ops->D[nd - 1] + i * nd;
            const int base = t - i * st;
            if constexpr (STD) {
                for (int m = 0; m < nd; ++m) {
                    const double Dm = Drow[m];
#pragma unroll
                    for (int v = 0; v < 5; ++v) R[v] += Dm * sF[v * T + base + m * st];
                }
            } else {
                const int lines = n3 / nd;
                const int lq = S.origin + ijk[d0] + S.s.n[d0] * ijk[d1];   // + x lines: the pair thread of (x, this line)
                for (int k = 1; k < nd; ++k) {
                    const int m = (i + k < nd) ? i + k : i + k - nd;
                    const int x = (2 * k < nd || (2 * k == nd && i < k)) ? i : m;
                    const int slot = 2 * k <= nd ? k : nd - k;
                    const double Dm = Drow[m];
                    const double *F = PB + (slot - 1) * 5 * T + lq + x * lines;
#pragma unroll
                    for (int v = 0; v < 5; ++v) R[v] += Dm * F[v * T];
                    if (NS) {
#pragma unroll
                        for (int v = 1; v < 5; ++v) R[v] -= Dm * sV[(v - 1) * T + base + m * st];
                    }
                }
            }
            // surface term
            if (i == 0 || i == nd - 1) {
                const int f2 = S.s.n[d0] * S.s.n[d1];
                const double *fs = fstar + (size_t)5 * fnoff[6 * S.e + 2 * d + (i != 0 ? 1 : 0)] + ijk[d0] +
                                   S.s.n[d0] * ijk[d1];
                const double sw = i != 0 ? ops->iw0[nd - 1] : -ops->iw0[nd - 1];
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                    const double F = fs[(size_t)v * f2];
                    if constexpr (STD) {
                        R[v] = fma(sw, F - own[v], R[v]);
                    } else {
                        R[v] = fma(sw, F, R[v]);
                        if (NS && v > 0) R[v] = fma(0.5 * sw, own[v], R[v]);
                    }
                }
            }
        }
    }
    double lc = 0.0, lv = 0.0;
    if (live) {
        const double iJ = invJall[nb + S.p];
        if (stage < 0) {
#pragma unroll
            for (int v = 0; v < 5; ++v) out[5 * nb + (size_t)v * n3 + S.p] = -R[v] * iJ;
        } else {
            const double sd = -(clk->dt * iJ);
            double *gp = g + 5 * nb + S.p, *up = u + 5 * nb + S.p;
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                const double inc = R[v] * sd;
                const double gv = (stage == 0) ? inc : fma(rkA, gp[(size_t)v * n3], inc);
                gp[(size_t)v * n3] = gv;
                w[v] = fma(rkB, gv, w[v]);
                up[(size_t)v * n3] = w[v];
            }
            if (lam_slot >= 0) {
                const Prim<double> qn = prim_from_u<double>(w, P.gm1);
                if (!(qn.rho > 0.0) || !(qn.p > 0.0)) clk->bad = 1;
                else alam_node(S.s, Jaall + 9 * nb, S.p, iJ, qn, P, lc, lv);
            }
        }
    }
    if (lam_slot >= 0 && stage >= 0) cta_max_to_clock<double>(clk->lam[lam_slot], P.physics == HS3D_NS, lc, lv);
}

// ------------------------------------------------------------------ diagnostics

// part[e][0..4] = sum_nodes J w_i w_j w_k f_v (f = dudt, else u), part[e][5]
// = sum J www (w . dudt), part[e][6] = sum |J www w_v dudt_v| (entropy
// variables w = dS/du, S = -rho s); a fixed-order tree over the nodes.
__global__ void __launch_bounds__(512) k_adiag(const int *__restrict__ elems, const int *__restrict__ P3, const long long *__restrict__ noff,
                        const double *__restrict__ wts, const double *__restrict__ Jall, const double *__restrict__ u,
                        const double *__restrict__ dudt, double gamma, double *__restrict__ part)
{
    extern __shared__ double sm[];   // [7][blockDim]
    const int e = elems[blockIdx.x];
    const AShape s = ashape(P3, e);
    const int p = threadIdx.x, T = blockDim.x;
    double val[7] = {0, 0, 0, 0, 0, 0, 0};
    if (p < s.n3) {
        const int i = p % s.n[0], j = (p / s.n[0]) % s.n[1], k = p / (s.n[0] * s.n[1]);
        const long long nb = noff[e];
        const double wq = Jall[nb + p] * wts[(s.n[0] - 1) * kMaxn + i] * wts[(s.n[1] - 1) * kMaxn + j] *
                          wts[(s.n[2] - 1) * kMaxn + k];
        const double *f = (dudt ? dudt : u) + 5 * nb + p;
        for (int v = 0; v < 5; ++v) val[v] = wq * f[(size_t)v * s.n3];
        if (dudt) {
            double w[5];
            for (int v = 0; v < 5; ++v) w[v] = u[5 * nb + (size_t)v * s.n3 + p];
            const Prim<double> q = prim_from_u<double>(w, gamma - 1.0);
            // entropy variables w = dS/du of S = -rho s, s = ln p - gamma ln rho
            const double sent = log(q.p) - gamma * log(q.rho);
            const double rp = (gamma - 1.0) * q.rho / q.p;
            const double ev[5] = {gamma - sent - 0.5 * rp * (q.v1 * q.v1 + q.v2 * q.v2 + q.v3 * q.v3), rp * q.v1,
                                  rp * q.v2, rp * q.v3, -rp};
            for (int v = 0; v < 5; ++v) {
                const double t = wq * ev[v] * f[(size_t)v * s.n3];
                val[5] += t;
                val[6] += fabs(t);
            }
        }
    }
    for (int k = 0; k < 7; ++k) sm[k * T + p] = val[k];
    __syncthreads();
    for (int h = T / 2; h > 0; h >>= 1) {
        if (p < h)
            for (int k = 0; k < 7; ++k) sm[k * T + p] += sm[k * T + p + h];
        __syncthreads();
    }
    if (p < 7) part[(size_t)e * 7 + p] = sm[p * T];
}

// out[k] = sum_e part[e][k] in a fixed order (256 strided partial sums, then a tree)
__global__ void k_adiag_final(const double *__restrict__ part, int E, double *__restrict__ out)
{
    __shared__ double sm[7][256];
    const int p = threadIdx.x;
    for (int k = 0; k < 7; ++k) {
        double acc = 0.0;
        for (int e = p; e < E; e += 256) acc += part[(size_t)e * 7 + k];
        sm[k][p] = acc;
    }
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (p < h)
            for (int k = 0; k < 7; ++k) sm[k][p] += sm[k][p + h];
        __syncthreads();
    }
    if (p < 7) out[p] = sm[p][0];
}

// ------------------------------------------------------------------ host tables

const AOps *device_aops()
{
    static std::mutex mu;
    static std::vector<AOps *> per_device;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if ((int)per_device.size() <= dev) per_device.resize(dev + 1, nullptr);
    if (per_device[dev]) return per_device[dev];
    AOps h;
    memset(&h, 0, sizeof h);
    for (int N = 1; N <= kMaxN; ++N) {
        const Ops &o = host_ops(N);
        const int n = N + 1;
        for (int t = 0; t < n * n; ++t) h.D[N][t] = o.D[t];
        h.iw0[N] = 1.0 / o.w[0];
    }
    AOps *d = nullptr;
    if (cudaMalloc(&d, sizeof(AOps)) != cudaSuccess) return nullptr;
    if (cudaMemcpy(d, &h, sizeof(AOps), cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaFree(d);
        return nullptr;
    }
    per_device[dev] = d;
    return d;
}

// Gauss-Lobatto weights of every degree [kMaxn][kMaxn] (device copy; row N-1... indexed by n - 1).
const double *device_aweights()
{
    static std::mutex mu;
    static std::vector<double *> per_device;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if ((int)per_device.size() <= dev) per_device.resize(dev + 1, nullptr);
    if (per_device[dev]) return per_device[dev];
    double h[kMaxn * kMaxn] = {0};
    for (int N = 1; N <= kMaxN; ++N) {
        const Ops &o = host_ops(N);
        for (int i = 0; i <= N; ++i) h[N * kMaxn + i] = o.w[i];
    }
    double *d = nullptr;
    if (cudaMalloc(&d, sizeof h) != cudaSuccess) return nullptr;
    if (cudaMemcpy(d, h, sizeof h, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaFree(d);
        return nullptr;
    }
    per_device[dev] = d;
    return d;
}

void lagrange_at(int n, const double *x, double y, double *l)
{
    for (int j = 0; j < n; ++j) {
        double v = 1.0;
        for (int k = 0; k < n; ++k)
            if (k != j) v *= (y - x[k]) / (x[j] - x[k]);
        l[j] = v;
    }
}

// The box map (affine position plus amp (L_c/2pi) sin sin sin of it, angles
// over [-pi, pi]) at reference point r of element e.
void abox_point(const AnisoMesh *a, int e, const double r[3], double X[3])
{
    const int Ed[3] = {a->ex, a->ey, a->ez};
    const int ab[3] = {e % a->ex, (e / a->ex) % a->ey, e / (a->ex * a->ey)};
    double x0[3], th[3];
    for (int c = 0; c < 3; ++c) {
        const double L = a->hi[c] - a->lo[c];
        x0[c] = a->lo[c] + (L / Ed[c]) * (ab[c] + 0.5 * (r[c] + 1.0));
        th[c] = -M_PI + 2.0 * M_PI * (x0[c] - a->lo[c]) / L;
    }
    const double sn = sin(th[0]) * sin(th[1]) * sin(th[2]);
    for (int c = 0; c < 3; ++c) X[c] = x0[c] + a->amp * ((a->hi[c] - a->lo[c]) / (2.0 * M_PI)) * sn;
}

// Node coordinates [3][n3] of element e: the degree-Ngeo interpolant of the
// box map at the element's own nodes, direction by direction.
void anodes(const AnisoMesh *a, int e, double *X)
{
    const int G = a->Ngeo, ng = G + 1;
    const Ops &og = host_ops(G);
    int n[3];
    for (int d = 0; d < 3; ++d) n[d] = a->P3[3 * e + d] + 1;
    const int n3 = n[0] * n[1] * n[2];
    std::vector<double> Xg(3 * ng * ng * ng);
    for (int k = 0; k < ng; ++k)
        for (int j = 0; j < ng; ++j)
            for (int i = 0; i < ng; ++i) {
                const double r[3] = {og.xi[i], og.xi[j], og.xi[k]};
                double x[3];
                abox_point(a, e, r, x);
                for (int c = 0; c < 3; ++c) Xg[(size_t)c * ng * ng * ng + i + ng * (j + ng * k)] = x[c];
            }
    double L[3][kMaxn][kMaxn];
    for (int d = 0; d < 3; ++d) {
        const Ops &on = host_ops(n[d] - 1);
        for (int t = 0; t < n[d]; ++t) lagrange_at(ng, og.xi, on.xi[t], L[d][t]);
    }
    for (int c = 0; c < 3; ++c)
        for (int k = 0; k < n[2]; ++k)
            for (int j = 0; j < n[1]; ++j)
                for (int i = 0; i < n[0]; ++i) {
                    double acc = 0.0;
                    for (int kk = 0; kk < ng; ++kk)
                        for (int jj = 0; jj < ng; ++jj)
                            for (int ii = 0; ii < ng; ++ii)
                                acc += L[2][k][kk] * L[1][j][jj] * L[0][i][ii] *
                                       Xg[(size_t)c * ng * ng * ng + ii + ng * (jj + ng * kk)];
                    X[(size_t)c * n3 + i + n[0] * (j + n[1] * k)] = acc;
                }
}

// fn(class threads, number of elements, element list) for every non-empty class
template <class F>
cudaError_t for_classes(const AnisoMesh *a, F fn)
{
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < kAnisoClasses && e == cudaSuccess; ++k) {
        const int cnt = a->cls_begin[k + 1] - a->cls_begin[k];
        if (cnt > 0) e = fn(kAnisoClass[k], cnt, a->cls_elems + a->cls_begin[k]);
    }
    return e;
}

constexpr size_t kAGradSmemPer = kVisc;   // doubles per thread slot of k_agrad

template <class K>
cudaError_t allow_smem(K kernel, size_t bytes)
{
    // (the kernels' own static shared memory counts toward the 48 KB too)
    return bytes > 40 * 1024 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes)
                             : cudaSuccess;
}

template <int T, bool NS>
cudaError_t allow_avol_smem()
{
    constexpr int kp = kMaxn / 2;
    cudaError_t e = cudaSuccess;
#define HS3D_ALLOW(FORM) \
    if (e == cudaSuccess) e = allow_smem(k_avol<T, NS, FORM>, sizeof(double) * avol_smem_per<FORM, NS>(kp) * T);
    HS3D_ALLOW(HS3D_VOL_STANDARD)
    HS3D_ALLOW(HS3D_VOL_EC)
    HS3D_ALLOW(HS3D_VOL_KG)
    HS3D_ALLOW(HS3D_VOL_PIROZZOLI)
    HS3D_ALLOW(HS3D_VOL_DUCROS)
    HS3D_ALLOW(HS3D_VOL_MORINISHI)
    HS3D_ALLOW(HS3D_VOL_IR)
#undef HS3D_ALLOW
    return e;
}

// The stage kernels' shared-memory limits, for the largest degree whatever the
// mesh's: a limit belongs to the function, so one set from a mesh's own degrees
// would lower it under every live mesh of higher ones.  Once per device, at the
// set-up of its first mesh with packs of T slots (not a stream operation, but
// kept out of captured launches).
template <int T>
cudaError_t allow_stage_smem()
{
    static std::mutex mu;
    static std::vector<char> done;   // per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    if ((int)done.size() <= dev) done.resize(dev + 1, 0);
    if (done[dev]) return cudaSuccess;
    e = allow_avol_smem<T, false>();
    if (e == cudaSuccess) e = allow_avol_smem<T, true>();
    if (e == cudaSuccess) e = allow_smem(k_agrad<T>, sizeof(double) * kAGradSmemPer * T);
    if (e == cudaSuccess) done[dev] = 1;
    return e;
}

template <int T, bool NS>
cudaError_t launch_avol(const AnisoMesh *a, const APhys &P, double *u, double *g, double *out, int stage, double A,
                        double B, int lam_slot, cudaStream_t s)
{
    const AOps *ops = device_aops();
    if (!ops) return cudaErrorMemoryAllocation;
    const int kp = (a->Pmax + 1) / 2;
    switch (P.form) {
#define HS3D_AVOL(FORM)                                                                                               \
    case FORM:                                                                                                        \
        return launch_pdl(k_avol<T, NS, FORM>, a->npacks, T, sizeof(double) * avol_smem_per<FORM, NS>(kp) * T, s,      \
                          a->slot_elem, a->slot0, a->dP3, a->dnoff, a->dfnoff, ops, u, g, out, a->Ja, a->invJ,         \
                          a->grad, a->fstar, P, a->clk, stage, A, B, lam_slot);
        HS3D_AVOL(HS3D_VOL_STANDARD)
        HS3D_AVOL(HS3D_VOL_EC)
        HS3D_AVOL(HS3D_VOL_KG)
        HS3D_AVOL(HS3D_VOL_PIROZZOLI)
        HS3D_AVOL(HS3D_VOL_DUCROS)
        HS3D_AVOL(HS3D_VOL_MORINISHI)
        HS3D_AVOL(HS3D_VOL_IR)
#undef HS3D_AVOL
    }
    return cudaErrorInvalidValue;
}

// The stage kernels of a mesh whose packs have T thread slots.
template <int T>
cudaError_t launch_stage(const AnisoMesh *a, const APhys &P, double *u, double *g, double *out, int stage, double A,
                         double B, int lam_slot, cudaStream_t s)
{
    const MortarOps *mo = device_mortar_ops();
    const AOps *ops = device_aops();
    if (!mo || !ops) return cudaErrorMemoryAllocation;
    const bool ns = P.physics == HS3D_NS;
    cudaError_t e = cudaSuccess;
    if (ns) {
        e = launch_pdl(k_amortar<0, true>, a->nfctas, kAFaceThreads, 0, s, a->faces, a->fctas, a->dP3, a->dnoff,
                       a->dfnoff, u, a->grad, a->Ja, mo, P, a->qhat);
        if (e == cudaSuccess)
            e = launch_pdl(k_agrad<T>, a->npacks, T, sizeof(double) * kAGradSmemPer * T, s, a->slot_elem, a->slot0,
                           a->dP3, a->dnoff, a->dfnoff, ops, u, a->Ja, a->invJ, a->qhat, P, a->grad);
    }
    if (e == cudaSuccess)
        e = launch_pdl(ns ? k_amortar<1, true> : k_amortar<1, false>, a->nfctas, kAFaceThreads, 0, s, a->faces,
                       a->fctas, a->dP3, a->dnoff, a->dfnoff, u, a->grad, a->Ja, mo, P, a->fstar);
    if (e == cudaSuccess)
        e = ns ? launch_avol<T, true>(a, P, u, g, out, stage, A, B, lam_slot, s)
               : launch_avol<T, false>(a, P, u, g, out, stage, A, B, lam_slot, s);
    return e;
}

// Elements into packs of T thread slots, largest first, each into the fullest
// pack that still has room (packs kept by free slots).
void pack_elements(const AnisoMesh *a, int T, std::vector<int> &slot_elem, std::vector<int> &slot0)
{
    std::vector<std::vector<int>> by_n3(T + 1), open(T + 1);   // elements by node count, packs by free slots
    for (int e = 0; e < a->E; ++e) by_n3[a->noff[e + 1] - a->noff[e]].push_back(e);
    slot0.assign(a->E, 0);
    slot_elem.reserve((size_t)a->noff[a->E] * 9 / 8 + T);
    int packs = 0;
    for (int n3 = T; n3 > 0; --n3)
        for (int e : by_n3[n3]) {
            int room = n3;
            while (room <= T && open[room].empty()) ++room;
            int pk;
            if (room <= T) {
                pk = open[room].back();
                open[room].pop_back();
            } else {
                pk = packs++;
                room = T;
                slot_elem.resize((size_t)packs * T, -1);
            }
            slot0[e] = T - room;
            for (int k = 0; k < n3; ++k) slot_elem[(size_t)pk * T + slot0[e] + k] = e;
            open[room - n3].push_back(pk);
        }
}

// The face table sorted by mortar degrees, then by the sides' degrees, and its CTAs.
// A face's kind is the two sides' points (2 .. 8) in both tangential directions:
// 7^4 kinds, ranked once, and one counting pass (a comparison sort was a tenth of
// the set-up of 4352 elements).
void pack_faces(const AnisoMesh *a, std::vector<AFace> &faces, std::vector<AFaceCta> &ctas)
{
    constexpr int kKinds = kMaxN * kMaxN * kMaxN * kMaxN;
    struct Kind {
        int l0, r0, l1, r1, m0, m1;
    };
    static const std::vector<Kind> kinds = [] {   // in the order of the table
        std::vector<Kind> k;
        for (int l0 = 2; l0 <= kMaxn; ++l0)
            for (int r0 = 2; r0 <= kMaxn; ++r0)
                for (int l1 = 2; l1 <= kMaxn; ++l1)
                    for (int r1 = 2; r1 <= kMaxn; ++r1)
                        k.push_back(Kind{l0, r0, l1, r1, std::max(l0, r0), std::max(l1, r1)});
        std::sort(k.begin(), k.end(), [](const Kind &x, const Kind &y) {
            return std::tie(x.m0, x.m1, x.l0, x.r0, x.l1, x.r1) < std::tie(y.m0, y.m1, y.l0, y.r0, y.l1, y.r1);
        });
        return k;
    }();
    auto index = [](int l0, int r0, int l1, int r1) { return (((l0 - 2) * kMaxN + r0 - 2) * kMaxN + l1 - 2) * kMaxN + r1 - 2; };
    static const std::vector<int> rank = [&] {
        std::vector<int> r(kKinds);
        for (int k = 0; k < kKinds; ++k) r[index(kinds[k].l0, kinds[k].r0, kinds[k].l1, kinds[k].r1)] = k;
        return r;
    }();
    std::vector<int> kind(faces.size()), at(kKinds + 1, 0);
    for (size_t i = 0; i < faces.size(); ++i) {
        const AFace &f = faces[i];
        const int *L = &a->P3[3 * (size_t)f.eL], *R = &a->P3[3 * (size_t)f.eR];
        const int d0 = f.d == 0 ? 1 : 0, d1 = f.d == 2 ? 1 : 2;
        kind[i] = rank[index(L[d0] + 1, R[d0] + 1, L[d1] + 1, R[d1] + 1)];
        ++at[kind[i] + 1];
    }
    for (int k = 0; k < kKinds; ++k) at[k + 1] += at[k];
    std::vector<AFace> sorted(faces.size());
    {
        std::vector<int> next(at.begin(), at.end() - 1);
        for (size_t i = 0; i < faces.size(); ++i) sorted[next[kind[i]]++] = faces[i];
    }
    faces.swap(sorted);
    // CTAs of faces of equal mortar degrees, kind by kind
    AFaceCta c{0, 0, 0, 0, 0};
    for (int k = 0; k < kKinds; ++k) {
        const Kind &K = kinds[k];
        const int most = kAFaceThreads / (K.m0 * K.m1);
        for (int i = at[k]; i < at[k + 1];) {
            if (c.count > 0 && (c.nm0 != K.m0 || c.nm1 != K.m1 || c.count == most)) {
                ctas.push_back(c);
                c.count = 0;
            }
            if (c.count == 0) c = AFaceCta{i, 0, K.m0, K.m1, 0};
            const int take = std::min(most - c.count, at[k + 1] - i);
            c.count += take;
            c.passes |= (K.l0 < K.m0 ? 1 : 0) | (K.r0 < K.m0 ? 2 : 0);
            i += take;
        }
    }
    if (c.count > 0) ctas.push_back(c);
}

}  // namespace

// ------------------------------------------------------------------ host API

void aniso_free(AnisoMesh *a)
{
    if (!a) return;
    if (a->slab) cudaFree(a->slab);
    delete a;
}

hs3d_status aniso_build(const hs3d_mesh_desc *desc, const int *degree3, AnisoMesh **out)
{
    *out = nullptr;
    const long long E = (long long)desc->ex * desc->ey * desc->ez;
    AnisoMesh *a = new (std::nothrow) AnisoMesh();
    if (!a) return fail(HS3D_ERR_NOMEM, "host allocation failed");
    a->ex = desc->ex;
    a->ey = desc->ey;
    a->ez = desc->ez;
    a->E = (int)E;
    for (int c = 0; c < 3; ++c) {
        a->lo[c] = desc->lo[c];
        a->hi[c] = desc->hi[c];
    }
    a->amp = desc->perturb_amp;
    a->P3.assign(degree3, degree3 + 3 * E);
    a->Pmin = 99;
    a->Pmax = 0;
    for (int v : a->P3) {
        a->Pmin = v < a->Pmin ? v : a->Pmin;
        a->Pmax = v > a->Pmax ? v : a->Pmax;
    }
    a->Ngeo = a->Pmin / 2 >= 1 ? a->Pmin / 2 : 1;
    a->off.assign(E + 1, 0);
    a->noff.assign(E + 1, 0);
    a->fnoff.assign(6 * E + 1, 0);
    std::vector<int> cls[kAnisoClasses];
    for (long long e = 0; e < E; ++e) {
        const int n[3] = {a->P3[3 * e] + 1, a->P3[3 * e + 1] + 1, a->P3[3 * e + 2] + 1};
        const int n3 = n[0] * n[1] * n[2];
        a->noff[e + 1] = a->noff[e] + n3;
        a->off[e + 1] = 5 * a->noff[e + 1];
        for (int d = 0; d < 3; ++d) {
            const int d0 = d == 0 ? 1 : 0, d1 = d == 2 ? 1 : 2;
            for (int side = 0; side < 2; ++side)
                a->fnoff[6 * e + 2 * d + side + 1] = a->fnoff[6 * e + 2 * d + side] + n[d0] * n[d1];
        }
        int k = 0;
        while (kAnisoClass[k] < n3) ++k;
        cls[k].push_back((int)e);
    }
    std::vector<int> elems;
    for (int k = 0; k < kAnisoClasses; ++k) {
        a->cls_begin[k] = (int)elems.size();
        elems.insert(elems.end(), cls[k].begin(), cls[k].end());
    }
    a->cls_begin[kAnisoClasses] = (int)elems.size();
    std::vector<AFace> faces;
    faces.reserve(3 * E);
    for (long long e = 0; e < E; ++e) {
        const int ab[3] = {(int)(e % a->ex), (int)((e / a->ex) % a->ey), (int)(e / ((long long)a->ex * a->ey))};
        const int Ed[3] = {a->ex, a->ey, a->ez};
        for (int d = 0; d < 3; ++d) {
            int c[3] = {ab[0], ab[1], ab[2]};
            c[d] = (c[d] + 1) % Ed[d];
            faces.push_back(AFace{(int)e, c[0] + a->ex * (c[1] + a->ey * c[2]), d});
        }
    }
    long long n3max = 0;
    for (long long e = 0; e < E; ++e) n3max = std::max<long long>(n3max, a->noff[e + 1] - a->noff[e]);
    a->T = n3max <= 256 ? 256 : 512;
    std::vector<int> slot_elem, slot0;
    pack_elements(a, a->T, slot_elem, slot0);
    a->npacks = (unsigned)(slot_elem.size() / a->T);
    std::vector<AFaceCta> fctas;
    pack_faces(a, faces, fctas);
    a->nfctas = (unsigned)fctas.size();
    const long long nodes = a->noff[E], fnodes = a->fnoff[6 * E];
    std::vector<double> X(3 * (size_t)nodes);
    for (long long e = 0; e < E; ++e) anodes(a, (int)e, X.data() + 3 * a->noff[e]);
    struct {
        void **p;
        size_t bytes;
    } allocs[] = {
        {(void **)&a->dP3, sizeof(int) * 3 * E},
        {(void **)&a->dnoff, sizeof(long long) * (E + 1)},
        {(void **)&a->doff, sizeof(long long) * (E + 1)},
        {(void **)&a->dfnoff, sizeof(long long) * (6 * E + 1)},
        {(void **)&a->cls_elems, sizeof(int) * E},
        {(void **)&a->slot_elem, sizeof(int) * slot_elem.size()},
        {(void **)&a->slot0, sizeof(int) * E},
        {(void **)&a->faces, sizeof(AFace) * 3 * E},
        {(void **)&a->fctas, sizeof(AFaceCta) * fctas.size()},
        {(void **)&a->X, sizeof(double) * 3 * nodes},
        {(void **)&a->Ja, sizeof(double) * 9 * nodes},
        {(void **)&a->J, sizeof(double) * nodes},
        {(void **)&a->invJ, sizeof(double) * nodes},
        {(void **)&a->grad, sizeof(double) * kVisc * nodes},
        {(void **)&a->fstar, sizeof(double) * 5 * fnodes},
        {(void **)&a->qhat, sizeof(double) * 4 * fnodes},
        {(void **)&a->diag_part, sizeof(double) * 7 * E},
        {(void **)&a->clk, sizeof(Clock)},
        {(void **)&a->clkp, sizeof(Clock *)},
        {(void **)&a->one, sizeof(int)},
    };
    // one allocation for all of them (as api.cu's mesh_alloc), every array on a
    // 256-byte boundary
    for (auto &al : allocs) a->bytes += (al.bytes + 255) & ~(size_t)255;
    cudaError_t e = cudaMalloc(&a->slab, a->bytes);
    if (e != cudaSuccess) a->slab = nullptr;
    char *at = (char *)a->slab;
    for (auto &al : allocs) {
        *al.p = a->slab ? at : nullptr;
        at += (al.bytes + 255) & ~(size_t)255;
    }
    const int one = 1;
    static_assert(sizeof(long long) == sizeof(int64_t), "offset layout");
    if (e == cudaSuccess) e = cudaMemcpy(a->dP3, a->P3.data(), sizeof(int) * 3 * E, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(a->dnoff, a->noff.data(), sizeof(long long) * (E + 1), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(a->doff, a->off.data(), sizeof(long long) * (E + 1), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(a->dfnoff, a->fnoff.data(), sizeof(long long) * (6 * E + 1), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(a->cls_elems, elems.data(), sizeof(int) * E, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(a->slot_elem, slot_elem.data(), sizeof(int) * slot_elem.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(a->slot0, slot0.data(), sizeof(int) * E, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(a->fctas, fctas.data(), sizeof(AFaceCta) * fctas.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(a->faces, faces.data(), sizeof(AFace) * 3 * E, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(a->X, X.data(), sizeof(double) * 3 * nodes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(a->clk, 0, sizeof(Clock));
    if (e == cudaSuccess) e = cudaMemcpy(a->clkp, &a->clk, sizeof(Clock *), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(a->one, &one, sizeof(int), cudaMemcpyHostToDevice);
    const AOps *ops = device_aops();
    if (e == cudaSuccess && (!ops || !device_aweights() || !device_mortar_ops())) e = cudaErrorMemoryAllocation;
    if (e == cudaSuccess)
        e = for_classes(a, [&](int T, int cnt, const int *els) {
            k_ageo<<<cnt, T, sizeof(double) * 5 * T>>>(els, a->dP3, a->dnoff, ops, a->X, a->Ja, a->J, a->invJ);
            return cudaGetLastError();
        });
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = a->T == 256 ? allow_stage_smem<256>() : allow_stage_smem<512>();
    if (e != cudaSuccess) {
        cudaGetLastError();
        aniso_free(a);
        return cuda_fail(e, "anisotropic mesh set-up");
    }
    *out = a;
    return HS3D_OK;
}

cudaError_t aniso_stage(const AnisoMesh *a, const hs3d_solver_cfg *c, double *u, double *g, double *out, int stage,
                        int lam_slot, cudaStream_t s)
{
    const APhys P = aphys(c);
    double A = 0.0, B = 0.0;
    if (stage >= 0) rk_coeffs(c->time_scheme, stage, &A, &B);
    const cudaError_t e = a->T == 256 ? launch_stage<256>(a, P, u, g, out, stage, A, B, lam_slot, s)
                                      : launch_stage<512>(a, P, u, g, out, stage, A, B, lam_slot, s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t aniso_step(const AnisoMesh *a, const hs3d_solver_cfg *c, double *u, double *g, double dt, bool fresh,
                       cudaStream_t s)
{
    const APhys P = aphys(c);
    cudaError_t e = cudaSuccess;
    if (fresh && !(dt > 0.0)) {
        k_alambda<<<a->npacks, a->T, 0, s>>>(a->slot_elem, a->slot0, a->dP3, a->dnoff, a->Ja, a->invJ, u, P, a->clk, 0);
        e = cudaGetLastError();
    }
    // the maxima already carry n_d^2 (n_d^4): the p-mesh finalize with n = 1
    if (e == cudaSuccess)
        e = launch_pdt_finalize(a->clkp, a->one, 1, c->cfl, 8.0, 12.0, fresh ? 0 : 1, dt > 0.0 ? dt : 0.0, s);
    const int ns = rk_stages(c->time_scheme);
    for (int k = 0; k < ns && e == cudaSuccess; ++k) e = aniso_stage(a, c, u, g, nullptr, k, k == ns - 1 ? 1 : -1, s);
    return e;
}

cudaError_t aniso_init_state(const AnisoMesh *a, const hs3d_ic &ic, double *u, cudaStream_t s)
{
    return for_classes(a, [&](int T, int cnt, const int *els) {
        k_ainit<<<cnt, T, 0, s>>>(els, a->dP3, a->dnoff, a->X, ic, a->hi[0] - a->lo[0], a->hi[1] - a->lo[1], u);
        return cudaGetLastError();
    });
}

cudaError_t aniso_diagnostics(const AnisoMesh *a, const hs3d_solver_cfg *c, const double *u, const double *dudt,
                              double *out, cudaStream_t s)
{
    const double *wts = device_aweights();
    if (!wts) return cudaErrorMemoryAllocation;
    cudaError_t e = for_classes(a, [&](int T, int cnt, const int *els) {
        k_adiag<<<cnt, T, sizeof(double) * 7 * T, s>>>(els, a->dP3, a->dnoff, wts, a->J, u, dudt, c->gamma,
                                                       a->diag_part);
        return cudaGetLastError();
    });
    if (e == cudaSuccess) {
        k_adiag_final<<<1, 256, 0, s>>>(a->diag_part, a->E, out);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace hs3d
