// Element kernel: volume term + surface lifting + Jacobian scaling + RK stage.
// (Template shared by the per-volume-form translation units volume_*.cu.)
//
// Strong form of Eq. NS5 (Sec. 3.3) on Gauss-Lobatto nodes, per element:
//   du/dt = -(V + S)/J
//   standard form   V = sum_d D_d F~^d,   F~^d = Ja^d . (F_e - F_v)
//   split form      V = sum_d sum_m D_im F#(u_i, u_m).(Ja^d_i + Ja^d_m) - sum_d D_d (Ja^d . F_v)
//                   with a symmetric two-point flux F# (Sec. 3.5): Chandrashekar,
//                   Kennedy-Gruber, Pirozzoli, Ducros, Morinishi or Ismail-Roe
//   surface         S = (1/w_end) (F^* - F~^d_in) on the +d face, (1/w_0)(-F^* + F~^d_in) on the -d face
//                   F^* the face flux computed once per face by k_face
// followed either by the residual store or by one low-storage RK stage
// (Sec. 3.7) g <- A_k g + dt R, u <- u + B_k g in FP64, with the stage's A_k,
// B_k passed by the host (Williamson RK3 or Carpenter-Kennedy RK4).  After
// the last stage the kernel also reduces the dt maxima of the updated state (the time
// step rule's input for the next step) so that no separate pass over the
// state is needed between steps.
//
// FP64 arithmetic (the mixed path has its own element kernel, volume_dev.cuh).
// The kernel is bound by the FP64 pipe (one warp instruction per 16 cycles and
// SM), so what is counted is FP64 instructions per warp, partly filled warps
// included:
//   - the pair inputs are staged so that the means of a pair are plain sums
//     (split_node64), reciprocals and roots take one third-order step
//     (rcp_fast), and no logarithm is computed per node;
//   - split forms leave out the diagonal pair: D_ii is zero inside and
//     2 D_ii = +-1/w at the two ends, where F#(u_i, u_i).(2 Ja_i) D_ii is
//     exactly the own Euler flux that the surface term (1/w)(F* - F~_in)
//     takes off again, so neither is formed; of the viscous part the
//     diagonal takes half of the surface term's, and +-(1/w)(F* + F~_v/2)
//     remains;
//   - the two faces of a direction share one instruction sequence (a lane is
//     on at most one of them).
// 16^3 elements of N = 3, NS, Chandrashekar form, one launch: 365 -> 260 us.
//
// One thread per node, `epb` elements per CTA (a kernel argument).  The
// element's contravariant fluxes (standard form) or its per-node two-point-flux
// inputs (split form) are staged in shared memory; the six face-flux blocks of
// the element (contiguous 5n^2 chunks) are copied there by cp.async.
#pragma once

#include "internal.cuh"
#include "physics.cuh"

namespace hs3d {

// Largest CTA of the element kernel: 256 threads, or one element when it has
// more nodes, in whole warps.
template <int N>
constexpr int vol_threads()
{
    return (max_cta_threads(N, HS3D_FP64, kShapeElem, HS3D_VOL_STANDARD, false) + 31) & ~31;
}

// Minimum resident CTAs per SM asked of the compiler (Gauss-Legendre element
// kernel): the mixed path is latency bound, so its register budget is capped (64
// per thread with 256- or 512-thread CTAs) to keep more warps resident; the FP64
// path is bound by the FP64 pipe and keeps its registers.
template <int N, typename R>
constexpr int vol_min_blocks()
{
    return sizeof(R) == 4 ? (((N + 1) * (N + 1) * (N + 1) <= 256) ? 4 : 2) : 1;
}

// Index of the 5 n^2 face-flux block of face `slot` of element e: the +d
// face's own block d E + e or the -d neighbour's d E + owner (conforming
// mesh), or the element's own per-face block slot E + e (face6).
__device__ __forceinline__ size_t face_block(const Item &it, int slot, int d, int owner, int e)
{
    return it.face6 ? (size_t)slot * it.E + e : (size_t)d * it.E + owner;
}

template <typename R>
__device__ __forceinline__ const R *metric_ptr(const Item &it);
template <>
__device__ __forceinline__ const double *metric_ptr<double>(const Item &it) { return it.Ja; }
template <>
__device__ __forceinline__ const float *metric_ptr<float>(const Item &it) { return it.Jaf; }

// Residual store or RK stage of one node from V (volume + surface sum), then,
// after the last stage (lam_slot >= 0), the dt maxima of the updated state.
// u holds the FP64 state on the FP64 path (loaded here on the mixed path).
template <typename R, bool NS>
__device__ __forceinline__ void node_update(const Item &it, int e, int p, int n3, const R V[5], double u[5],
                                            int stage, double rkA, double rkB, int lam_slot, double &lc, double &lv,
                                            bool &lam_active)
{
    if constexpr (sizeof(R) == 4) {
        // the FP64 state is needed only for the RK accumulation
        if (stage >= 0) {
#pragma unroll
            for (int v = 0; v < 5; ++v) u[v] = it.u[(size_t)e * 5 * n3 + p + v * n3];
        }
    }

    float nf[5];   // mixed path: FP32 shadow of the updated state
    if constexpr (sizeof(R) == 8) {
        const double ij = it.invJ[(size_t)e * n3 + p];
        if (stage < 0) {
            double *O = it.out + (size_t)e * 5 * n3 + p;
#pragma unroll
            for (int v = 0; v < 5; ++v) O[v * n3] = -(double)V[v] * ij;
        } else {
            const double s = -(it.clk->dt * ij);
            double *Gp = it.g + (size_t)e * 5 * n3 + p;
            double *Up = it.u + (size_t)e * 5 * n3 + p;
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                const double inc = V[v] * s;
                const double gv = (stage == 0) ? inc : fma(rkA, Gp[v * n3], inc);
                Gp[v * n3] = gv;
                u[v] = fma(rkB, gv, u[v]);
                Up[v * n3] = u[v];
            }
        }
    } else {
        // mixed path: the increment dt R = -dt V / J is formed in FP32; the
        // register g holds FP32 increments ([E][5][n3] floats in the first half
        // of the caller's buffer) and the state accumulates in FP64 (one FP64
        // FMA per variable).
        const float ijf = it.invJf[(size_t)e * n3 + p];
        if (stage < 0) {
            double *O = it.out + (size_t)e * 5 * n3 + p;
#pragma unroll
            for (int v = 0; v < 5; ++v) O[v * n3] = f2d_exact(-(float)V[v] * ijf);
        } else {
            const float sdt = d2f_rn(it.clk->dt) * ijf;
            const float A = d2f_rn(rkA);
            const double B = rkB;
            float *Gp = (float *)it.g + (size_t)e * 5 * n3 + p;
            double *Up = it.u + (size_t)e * 5 * n3 + p;
            float *Sp = it.uf + (size_t)e * 5 * n3 + p;
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                const float inc = -(float)V[v] * sdt;
                const float gv = (stage == 0) ? inc : fmaf(A, Gp[v * n3], inc);
                Gp[v * n3] = gv;
                u[v] = fma(B, f2d_exact(gv), u[v]);
                Up[v * n3] = u[v];
                nf[v] = d2f_rn(u[v]);
                Sp[v * n3] = nf[v];
            }
        }
    }
    if (stage >= 0) {
        if (lam_slot >= 0) {
            // dt maxima of the updated state (same rule as k_lambda, in R)
            const Phys<R> P = phys_of<R>(it);
            Prim<R> qn;
            if constexpr (sizeof(R) == 8) qn = prim_from_u<R>(u, P.gm1);
            else qn = prim_from_f(nf, P.gm1);
            if (!(qn.rho > (R)0) || !(qn.p > (R)0)) {
                it.clk->bad = 1;
            } else {
                const R c = sound_speed(qn, P.gamma);
                R iJ;
                if constexpr (sizeof(R) == 8) iJ = it.invJ[(size_t)e * n3 + p];
                else iJ = it.invJf[(size_t)e * n3 + p];
                R sc = (R)0, sv = (R)0;
                const R *JA = metric_ptr<R>(it) + (size_t)e * 9 * n3 + p;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const R a1 = JA[(d * 3) * n3], a2 = JA[(d * 3 + 1) * n3], a3 = JA[(d * 3 + 2) * n3];
                    const R s2 = a1 * a1 + a2 * a2 + a3 * a3, an = sqrt_(s2);
                    if constexpr (sizeof(R) == 8) {
                        sc += fabs(a1 * qn.v1 + a2 * qn.v2 + a3 * qn.v3) + c * an;
                        sv += s2;
                    } else {
                        sc += (fabs(a1 * qn.v1 + a2 * qn.v2 + a3 * qn.v3) + c * an) * iJ;
                        sv += (an * iJ) * (an * iJ);
                    }
                }
                if constexpr (sizeof(R) == 8) {
                    lc = sc * iJ;
                    lv = NS ? P.mu * sv * (iJ * iJ) * qn.ir : 0.0;
                } else {
                    lc = widen<R>(sc);
                    lv = NS ? widen<R>(P.mu * sv / qn.rho) : 0.0;
                }
                lam_active = true;
            }
        }
    }
}

// Doubles staged per node: the three contravariant fluxes (standard form), or
// the pair inputs, the metric terms and (NS) the viscous fluxes without their
// zero mass component (split forms).
template <int FORM, bool NS>
constexpr int vol_smem_per_node()
{
    return is_standard(FORM) ? 15 : (split_slots64<FORM>() + 9 + (NS ? 12 : 0));
}

// Dynamic shared memory: D, the per-node staging of epb elements, their
// face-flux blocks, the split form's pair buffers [5][n/2][n3].
template <int N, bool NS, int FORM>
__host__ __device__ constexpr size_t vol_smem_bytes(int epb)
{
    constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
    constexpr size_t pairs = !is_standard(FORM) ? (size_t)5 * (n / 2) * n3 : 0;
    return sizeof(double) * (((n * n + 1) & ~1) + (size_t)epb * (vol_smem_per_node<FORM, NS>() * n3 + 30 * n2 + pairs));
}

template <int N, bool NS, int FORM>
__global__ void __launch_bounds__(vol_threads<N>(), 1)
k_volume(const __grid_constant__ Batch b, const Ops *__restrict__ ops, int stage, double rkA, double rkB, int lam_slot,
         int epb)
{
    constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
    constexpr bool STD = is_standard(FORM);
    constexpr int PER = vol_smem_per_node<FORM, NS>();
    constexpr int ZS = split_slots64<FORM>();   // split forms: slots of the pair inputs, then Ja, then the viscous fluxes
    constexpr int FACEVALS = 6 * 5 * n2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *sD = (double *)smem_raw;
    double *sbuf = sD + ((n * n + 1) & ~1);
    double *sface = sbuf + (size_t)epb * PER * n3;
    pdl_wait();
    for (int t = threadIdx.x; t < n * n; t += blockDim.x) sD[t] = ops->D[t];
    const int le = threadIdx.x / n3, p = threadIdx.x - le * n3;
    const long long ge = blockIdx.x * (long long)epb + le;
    bool valid = le < epb && ge < b.total_elems;
    const Item *itp = nullptr;
    int e = 0;
    if (valid) {
        itp = &find_item_elem(b, ge);
        e = (int)(ge - itp->elem_begin);
        if (itp->clk && itp->clk->done) valid = false;
    }
    double *S = sbuf + (size_t)le * PER * n3;
    double *F6 = sface + (size_t)le * FACEVALS;
    const int ijk[3] = {p % n, (p / n) % n, p / n2};

    double u[5];
    double V[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const double iw = ops->iw0;
    if (valid) {
        const Item &it = *itp;
        const Nbrs nb = elem_nbrs(e, it.ex, it.ey, it.ez);
        // the six face-flux blocks of this element (slot 2d+1: the +d face,
        // own index; slot 2d: the -d face, owned by the -d neighbour)
        const double *FS = (const double *)it.fstar;
#pragma unroll
        for (int slot = 0; slot < 6; ++slot) {
            const int d = slot >> 1;
            const int owner = (slot & 1) ? e : nb.m[d];
            cp_async_block<double>(F6 + slot * 5 * n2, FS + face_block(it, slot, d, owner, e) * 5 * n2, 5 * n2, p, n3);
        }
        const size_t node = (size_t)e * 5 * n3 + p;
        const Phys<double> P = phys_of<double>(it);
        double ja[9];
        const double *JA = it.Ja + (size_t)e * 9 * n3 + p;
#pragma unroll
        for (int k = 0; k < 9; ++k) ja[k] = JA[k * n3];
#pragma unroll
        for (int v = 0; v < 5; ++v) u[v] = it.u[node + v * n3];
        const Prim<double> q = prim_from_u<double>(u, P.gm1);
        double G[kVisc];
        if (NS) {
            const double *Gp = (const double *)it.grad + (size_t)e * kVisc * n3 + p;
#pragma unroll
            for (int k = 0; k < kVisc; ++k) G[k] = Gp[k * n3];
        }
        if constexpr (STD || NS) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                double fe[5], fv[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
                if (NS) visc_flux(q, G, ja[d * 3], ja[d * 3 + 1], ja[d * 3 + 2], fv);
                if constexpr (STD) {
                    euler_flux(q, q.E, ja[d * 3], ja[d * 3 + 1], ja[d * 3 + 2], fe);
#pragma unroll
                    for (int v = 0; v < 5; ++v) S[(d * 5 + v) * n3 + p] = (NS && v > 0) ? fe[v] - fv[v] : fe[v];
                } else {
#pragma unroll
                    for (int v = 1; v < 5; ++v) S[(ZS + 9 + d * 4 + v - 1) * n3 + p] = fv[v];
                }
            }
        }
        if constexpr (!STD) {
            double z[ZS];
            split_node64<FORM>(q, z);
#pragma unroll
            for (int k = 0; k < ZS; ++k) S[k * n3 + p] = z[k];
#pragma unroll
            for (int k = 0; k < 9; ++k) S[(ZS + k) * n3 + p] = ja[k];
        }
    }
    cp_async_wait_all();
    __syncthreads();

    double lc = 0.0, lv = 0.0;
    bool lam_active = false;
    if constexpr (STD) {
        if (valid) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int stride = (d == 0) ? 1 : (d == 1) ? n : n2;
                const int base = p - ijk[d] * stride;
                const double *Drow = sD + ijk[d] * n;
#pragma unroll
                for (int m = 0; m < n; ++m) {
                    const double Dm = Drow[m];
#pragma unroll
                    for (int v = 0; v < 5; ++v) V[v] += Dm * S[(d * 5 + v) * n3 + base + m * stride];
                }
            }
        }
    } else {
        // F#(u_i,u_m).(Ja_i + Ja_m) is symmetric in (i, m), so each pair of
        // nodes on a line is evaluated once and shared through shared memory.
        // Pair thread t = x n^2 + l (x a position along the line, l = ta + n tb
        // the line) evaluates the pairs (x, x + k mod n) for k = 1 .. n/2, the
        // half-way pair k = n/2 of an even n only for x < n/2: every pair of the
        // line exactly once, with no index search, and the threads with the
        // extra pair grouped in the lower warps.  Then every node sums D_im
        // times the fluxes of its line.
        constexpr int KP = n / 2;
        double *PB = sface + (size_t)epb * FACEVALS + (size_t)le * 5 * KP * n3;
        const double hg = valid ? itp->hg : 0.0;
        const double gam = valid ? itp->gamma : 0.0;
#pragma unroll 1
        for (int d = 0; d < 3; ++d) {
            const int sd = (d == 0) ? 1 : (d == 1) ? n : n2;   // node stride along d
            if (valid) {
                const int x = p / n2, l = p - x * n2;
                const int ta = l % n, tb = l / n;
                const int a = x * sd + ta * ((d == 0) ? n : 1) + tb * ((d == 2) ? n : n2);
                double za[ZS];
#pragma unroll
                for (int k = 0; k < ZS; ++k) za[k] = S[k * n3 + a];
                const double *SJ = S + (ZS + d * 3) * n3;
                const double j1 = SJ[a], j2 = SJ[n3 + a], j3 = SJ[2 * n3 + a];
#pragma unroll
                for (int k = 1; k <= KP; ++k) {
                    if (2 * k == n && x >= KP) break;
                    const int xm = (x + k < n) ? x + k : x + k - n;
                    const int c = a + (xm - x) * sd;
                    double zc[ZS];
#pragma unroll
                    for (int q = 0; q < ZS; ++q) zc[q] = S[q * n3 + c];
                    double fs[5];
                    split_pair64<FORM>(za, zc, gam, hg, j1 + SJ[c], j2 + SJ[n3 + c], j3 + SJ[2 * n3 + c], fs);
#pragma unroll
                    for (int v = 0; v < 5; ++v) PB[(v * KP + k - 1) * n3 + p] = fs[v];
                }
            }
            __syncthreads();
            if (valid) {
                const int i = ijk[d];
                const int ta = (d == 0) ? ijk[1] : ijk[0];
                const int tb = (d == 2) ? ijk[1] : ijk[2];
                const int l = ta + n * tb;
                const int base = p - i * sd;   // (viscous fluxes)
                const double *Drow = sD + i * n;
                // the other n - 1 nodes of the line, the pair (i, i + k mod n) with
                // pair thread x n^2 + l in slot k - 1 (x = i) or n - k - 1 (x = m)
#pragma unroll
                for (int k = 1; k < n; ++k) {
                    const int m = (i + k < n) ? i + k : i + k - n;
                    const double Dm = Drow[m];
                    int slot, x;
                    if (2 * k < n) {
                        slot = k;
                        x = i;
                    } else if (2 * k > n) {
                        slot = n - k;
                        x = m;
                    } else {
                        slot = KP;
                        x = (i < KP) ? i : m;
                    }
                    const double *F = PB + (slot - 1) * n3 + x * n2 + l;
#pragma unroll
                    for (int v = 0; v < 5; ++v) V[v] += Dm * F[v * KP * n3];
                    if (NS) {
#pragma unroll
                        for (int v = 1; v < 5; ++v) V[v] -= Dm * S[(ZS + 9 + d * 4 + v - 1) * n3 + base + m * sd];
                    }
                }
            }
            __syncthreads();
        }
    }
    if (valid) {
        const Item &it = *itp;
        // surface term: +-(1/w)(F* - F~) on the +-d face (standard form: the
        // difference is formed first, it is small where the large fluxes nearly
        // cancel; split forms: +-(1/w)(F* + F~_v/2), see the top)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (ijk[d] != N && ijk[d] != 0) continue;
            const int ta = (d == 0) ? ijk[1] : ijk[0];
            const int tb = (d == 2) ? ijk[1] : ijk[2];
            const bool plus = ijk[d] == N;
            const double sw = plus ? iw : -iw;
            const double *F = F6 + (2 * d + (plus ? 1 : 0)) * 5 * n2 + ta + n * tb;
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                if constexpr (STD) {
                    V[v] = fma(sw, F[v * n2] - S[(d * 5 + v) * n3 + p], V[v]);
                } else {
                    V[v] = fma(sw, F[v * n2], V[v]);
                    if (NS && v > 0) V[v] = fma(0.5 * sw, S[(ZS + 9 + d * 4 + v - 1) * n3 + p], V[v]);
                }
            }
        }
        node_update<double, NS>(it, e, p, n3, V, u, stage, rkA, rkB, lam_slot, lc, lv, lam_active);
    }
    if (lam_slot >= 0 && stage >= 0) rates_to_clock<double>(b, itp, lam_slot, NS, lc, lv, lam_active);
}

// ------------------------------------------------------------------ launch (one volume form)

template <int N, bool NS, int FORM>
static cudaError_t vol_launch2(const Batch &b, int stage, double rkA, double rkB, int lam_slot, cudaStream_t s)
{
    constexpr int n3 = (N + 1) * (N + 1) * (N + 1);
    const int epb = elems_per_cta(N, HS3D_FP64, kShapeElem, FORM, false, b.total_elems, b.beside);
    const int threads = epb * n3;
    const size_t smem = vol_smem_bytes<N, NS, FORM>(epb);
    unsigned blocks = (unsigned)((b.total_elems + epb - 1) / epb);
    const Ops *ops = device_ops(N);
    if (!ops) return cudaErrorMemoryAllocation;
    cudaError_t e = launch_pdl(k_volume<N, NS, FORM>, blocks, threads, smem, s, b, ops, stage, rkA, rkB,
                               stage >= 0 ? lam_slot : -1, epb);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int FORM>
cudaError_t launch_volume_form(int N, int prec, int physics, const Batch &b, int stage, double rkA, double rkB,
                               int lam_slot, cudaStream_t s)
{
    if (b.total_elems == 0) return cudaSuccess;
    if (prec != HS3D_FP64) return cudaErrorInvalidValue;
#define HS3D_VOLN(K)                                                                                  \
    case K:                                                                                           \
        return physics == HS3D_NS ? vol_launch2<K, true, FORM>(b, stage, rkA, rkB, lam_slot, s)       \
                                  : vol_launch2<K, false, FORM>(b, stage, rkA, rkB, lam_slot, s);
    switch (N) {
        HS3D_VOLN(1) HS3D_VOLN(2) HS3D_VOLN(3) HS3D_VOLN(4) HS3D_VOLN(5) HS3D_VOLN(6) HS3D_VOLN(7)
    }
#undef HS3D_VOLN
    return cudaErrorInvalidValue;
}

template <int N, int FORM>
static cudaError_t prep_vol_n()
{
    const int big = 220 * 1024;
    cudaError_t e = cudaSuccess;
#define HS3D_ATTR(NS)                                                                                      \
    if (e == cudaSuccess)                                                                                  \
        e = cudaFuncSetAttribute(k_volume<N, NS, FORM>, cudaFuncAttributeMaxDynamicSharedMemorySize, big); \
    if (e == cudaSuccess)                                                                                  \
        e = cudaFuncSetAttribute(k_volume<N, NS, FORM>, cudaFuncAttributePreferredSharedMemoryCarveout,    \
                                 cudaSharedmemCarveoutMaxShared);
    HS3D_ATTR(false)
    HS3D_ATTR(true)
#undef HS3D_ATTR
    return e;
}

template <int FORM>
cudaError_t prepare_volume_form(int N)
{
    switch (N) {
        case 1: return prep_vol_n<1, FORM>();
        case 2: return prep_vol_n<2, FORM>();
        case 3: return prep_vol_n<3, FORM>();
        case 4: return prep_vol_n<4, FORM>();
        case 5: return prep_vol_n<5, FORM>();
        case 6: return prep_vol_n<6, FORM>();
        case 7: return prep_vol_n<7, FORM>();
    }
    return cudaErrorInvalidValue;
}

// Each volume_<form>.cu instantiates the two entry points for its form.
#define HS3D_VOLUME_FORM_TU(FORM)                                                                               \
    template cudaError_t launch_volume_form<FORM>(int, int, int, const Batch &, int, double, double, int,        \
                                                  cudaStream_t);                                                 \
    template cudaError_t prepare_volume_form<FORM>(int);

}  // namespace hs3d
