// BR1 gradients of the mixed path (FP32 arithmetic on deviations).
//
//   J grad q_c = sum_d D_d (Ja^d_c q) + sum_faces (1/w_end) (q* - q_in) (+-Ja^d_c),
//   q = (v1, v2, v3, T), T = p/rho, q* = (q_in + q_out)/2           (Bassi & Rebay 1997)
//
// The element's reference state ubar (its centre node, lowmach.cuh) turns the
// FP64 state into deviations, and q into q - qbar: the constant qbar drops
// out of the volume term by the discrete metric identity and out of every
// jump, so T' = T - Tbar = (p' - Tbar rho' + rT)/rho (rT = pbar - Tbar rhobar)
// keeps its accuracy relative to the temperature fluctuation instead of to
// T ~ 1/(gamma Ma^2).  The neighbours' traces are read in FP64 and made
// deviations from the same reference, so the lifted jumps are accurate.
// On a mesh with per-element degrees (Item::face6) the mortar kernel supplies
// 2 q*_e - q_in in full FP32 values; it is made a deviation by subtracting qbar.
//
// One thread per node, epb elements per CTA; the element's FP32 metric terms
// arrive in shared memory by one bulk copy (TMA engine) per element when the
// block is a multiple of 16 bytes (an even number of nodes per direction),
// else by per-thread loads.
#include "internal.cuh"
#include "lowmach.cuh"
#include "physics.cuh"

namespace hs3d {

template <int N>
constexpr int grad_dev_threads()
{
    return max_cta_threads(N, HS3D_MIXED32, kShapeGrad, HS3D_VOL_STANDARD, false);
}

// Shared-memory floats per element: q' [n3] and neighbour-trace deviations [6][n2]
// in groups of four (one 16-byte load each), metric terms [9][n3].
template <int N>
constexpr int grad_dev_per_elem()
{
    return (13 * (N + 1) * (N + 1) * (N + 1) + 24 * (N + 1) * (N + 1) + 3) & ~3;
}

template <int n>
__device__ __forceinline__ int gd_face_node(int d, int end, int ta, int tb)
{
    if (d == 0) return end + n * (ta + n * tb);
    if (d == 1) return ta + n * (end + n * tb);
    return ta + n * (tb + n * end);
}

// Velocity and temperature deviations of a node.
__device__ __forceinline__ void grad_dev_vars(const Dev &d, const Anchor &A, float Tb, float rT, float q[4])
{
    q[0] = d.dv1;
    q[1] = d.dv2;
    q[2] = d.dv3;
    q[3] = (d.dp - Tb * d.dr + rT) * __fdividef(1.0f, d.rho);
}

// One tile (epb elements) of the gradient kernel; returns true on the thread
// that initialised its element's bulk-copy barrier.
template <int N, bool MORT>
__device__ __forceinline__ bool grad_dev_tile(const Batch &b, const Ops *__restrict__ ops, long long tile,
                                              unsigned long long *bulk_bar)
{
    constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
    constexpr bool BULK = (n % 2 == 0);
    constexpr int PER = grad_dev_per_elem<N>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *sD = (float *)smem_raw;
    float *sE = sD + ((n * n + 3) & ~3);
    const int epb = blockDim.x / n3;
    for (int t = threadIdx.x; t < n * n; t += blockDim.x) sD[t] = (!MORT && t % (n + 1) == 0) ? 0.0f : ops->Df[t];
    const float dend = ops->Df[n * n - 1];
    const int le = threadIdx.x / n3, p = threadIdx.x - le * n3;
    const long long ge = tile * epb + le;
    bool valid = ge < b.total_elems;
    const Item *itp = nullptr;
    int e = 0;
    if (valid) {
        itp = &find_item_elem(b, ge);
        e = (int)(ge - itp->elem_begin);
        if (itp->clk && itp->clk->done) valid = false;
    }
    const bool armed = BULK && valid && p == 0;
    float4 *q = (float4 *)(sE + (size_t)le * PER);
    float4 *qn = q + n3;
    float *ja = (float *)(qn + 6 * n2);
    float qin[4];
    if (valid) {
        const Item &it = *itp;
        double uo[5];
        const double *U = it.u + (size_t)e * 5 * n3;
#pragma unroll
        for (int v = 0; v < 5; ++v) uo[v] = U[v * n3 + p];
        // the element's reference state, left by the pass before
        const AnchorRec R = load_anchor(it.anc, e);
        if constexpr (BULK) {
            // one thread initialises, arms and fills the element's barrier; the
            // others poll it only after the block barrier below
            if (p == 0) {
                unsigned long long *bar = bulk_bar + le;
                mbar_init(bar, 1);
                mbar_arrive_expect_tx(bar, 9 * n3 * 4);
                bulk_g2s(ja, it.Jaf + (size_t)e * 9 * n3, 9 * n3 * 4, bar);
            }
        }
        const float gm1 = it.gm1f;
        const Anchor A = R.a;
        const float Tb = A.p * __fdividef(1.0f, A.rho);
        const float rT = fmaf(-Tb, A.rho, A.p);
        constexpr int IT = (6 * n2 + n3 - 1) / n3;
        if constexpr (MORT) {
            // 2 q*_e - q_in from the mortar kernel, full FP32 values -> deviations
#pragma unroll
            for (int k = 0; k < IT; ++k) {
                const int t = p + k * n3;
                if (t < 6 * n2) {
                    const int slot = t / n2, ab = t - slot * n2;
                    const float *src = (const float *)it.qhat6 + ((size_t)slot * it.E + e) * 4 * n2 + ab;
                    qn[t] = make_float4(src[0] - A.v1, src[n2] - A.v2, src[2 * n2] - A.v3, src[3 * n2] - Tb);
                }
            }
        } else {
            // neighbour traces in FP64: all loads first, then the deviations
            const Nbrs nbs = elem_nbrs(e, it.ex, it.ey, it.ez);
            double raw[IT][5];
#pragma unroll
            for (int k = 0; k < IT; ++k) {
                const int t = p + k * n3;
                if (t < 6 * n2) {
                    const int slot = t / n2, ab = t - slot * n2;
                    const int d = slot >> 1, plus = slot & 1;
                    const int pn = gd_face_node<n>(d, plus ? 0 : N, ab % n, ab / n);
                    const double *src = it.u + (size_t)nbr_of_slot(nbs, slot) * 5 * n3 + pn;
#pragma unroll
                    for (int v = 0; v < 5; ++v) raw[k][v] = src[v * n3];
                }
            }
#pragma unroll
            for (int k = 0; k < IT; ++k) {
                const int t = p + k * n3;
                if (t < 6 * n2) {
                    float g4[4];
                    grad_dev_vars(make_dev_rec(raw[k], A, R.Elo, gm1), A, Tb, rT, g4);
                    qn[t] = make_float4(g4[0], g4[1], g4[2], g4[3]);
                }
            }
        }
        grad_dev_vars(make_dev_rec(uo, A, R.Elo, gm1), A, Tb, rT, qin);
        q[p] = make_float4(qin[0], qin[1], qin[2], qin[3]);
        if constexpr (!BULK) {
            const float *JA = it.Jaf + (size_t)e * 9 * n3 + p;
#pragma unroll
            for (int k = 0; k < 9; ++k) ja[k * n3 + p] = JA[k * n3];
        }
    }
    __syncthreads();
    if (!valid) return armed;
    bool landed = true;
    if constexpr (BULK) {
        if (!mbar_wait(bulk_bar + le, 0, kBulkWaitPolls)) {
            // a wait that ran out of polls poisons the gradients and flags the solve
            landed = false;
            if (itp->clk) itp->clk->bad = 2;
        }
    }
    const int ijk[3] = {p % n, (p / n) % n, p / n2};
    const Item &it = *itp;
    if (MORT && !landed) qin[0] = qin[1] = qin[2] = qin[3] = NAN;
    // the twelve sums d q_v / dx_c, as packed pairs of v: (v1, v2) and (v3, T) share
    // the metric factor, one 16-byte load brings q (against single values, the run:
    // NS standard form, 24^3 N = 5 4.63 -> 4.47 ms, 24^3 N = 6 10.10 -> 9.89, 30^3 N = 4
    // 6.61 -> 6.53, 40^3 N = 3 6.04 -> 6.01)
    float2 a01[3], a23[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) a01[c] = a23[c] = pair(0.0f);
    auto add = [&](float s1, float s2, float s3, const float4 &Q) {
        const float s[3] = {s1, s2, s3};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            a01[c] = __ffma2_rn(pair(s[c]), make_float2(Q.x, Q.y), a01[c]);
            a23[c] = __ffma2_rn(pair(s[c]), make_float2(Q.z, Q.w), a23[c]);
        }
    };
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int i = ijk[d];
        const int stride = (d == 0) ? 1 : (d == 1) ? n : n2;
        const int base = p - i * stride;
        const float *Drow = sD + i * n;
        const float *J1 = ja + d * 3 * n3, *J2 = J1 + n3, *J3 = J2 + n3;
#pragma unroll
        for (int m = 0; m < n; ++m) {
            const int pm = base + m * stride;
            const float Dm = Drow[m];
            add(Dm * J1[pm], Dm * J2[pm], Dm * J3[pm], q[pm]);
        }
        if constexpr (!MORT) {
            // the two ends: D_ii Ja q_in + (+-1/w)(q_out - q_in)/2 Ja = D_ii Ja q_out,
            // D_ii = +-1/(2w) (sD holds zero on the diagonal)
            if (i == 0 || i == N) {
                const int ta = (d == 0) ? ijk[1] : ijk[0];
                const int tb = (d == 2) ? ijk[1] : ijk[2];
                const float Dm = i == N ? dend : -dend;
                add(Dm * J1[p], Dm * J2[p], Dm * J3[p], qn[(2 * d + (i == N ? 1 : 0)) * n2 + ta + n * tb]);
            }
        }
    }
    if constexpr (MORT) {
        // surface lifting of the BR1 jumps (q* - q_in) = (q_out - q_in)/2; the twelve
        // gradients stay, every rounding as the mortar path's FP32 fluxes expect it
        // (visc_flux_grad)
        const float iw = ops->iw0f;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int ta = (d == 0) ? ijk[1] : ijk[0];
            const int tb = (d == 2) ? ijk[1] : ijk[2];
            const int ab = ta + n * tb;
#pragma unroll
            for (int plus = 0; plus < 2; ++plus) {
                if (ijk[d] != (plus ? N : 0)) continue;
                const float sg = plus ? 1.0f : -1.0f;
                const float4 Q = qn[(2 * d + plus) * n2 + ab];
                add(sg * ja[(d * 3 + 0) * n3 + p], sg * ja[(d * 3 + 1) * n3 + p], sg * ja[(d * 3 + 2) * n3 + p],
                    make_float4(0.5f * (Q.x - qin[0]) * iw, 0.5f * (Q.y - qin[1]) * iw, 0.5f * (Q.z - qin[2]) * iw,
                                0.5f * (Q.w - qin[3]) * iw));
            }
        }
        const float ij = it.invJf[(size_t)e * n3 + p];
        float *G = (float *)it.grad + (size_t)e * 12 * n3 + p;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            G[c * n3] = a01[c].x * ij;
            G[(3 + c) * n3] = a01[c].y * ij;
            G[(6 + c) * n3] = a23[c].x * ij;
            G[(9 + c) * n3] = a23[c].y * ij;
        }
    } else {
        const float acc[kVisc] = {a01[0].x, a01[1].y, a23[2].x, a01[0].y + a01[1].x, a23[0].x + a01[2].x,
                                  a23[1].x + a01[2].y, a23[0].y, a23[1].y, a23[2].y};
        float tau[kVisc];
        stress_of(acc, landed ? it.invJf[(size_t)e * n3 + p] : NAN, it.muf, it.kappaf, tau);
        float *G = (float *)it.grad + (size_t)e * kVisc * n3 + p;
#pragma unroll
        for (int k = 0; k < kVisc; ++k) G[k * n3] = tau[k];
    }
    return armed;
}

template <int N>
__device__ __noinline__ bool grad_dev_tile_call(const Batch &b, const Ops *__restrict__ ops, long long tile,
                                                unsigned long long *bulk_bar)
{
    return grad_dev_tile<N, false>(b, ops, tile, bulk_bar);
}

// The gradient kernel: a CTA per tile, or (PERSIST, Batch::persistent) a
// persistent grid walking the tiles (as k_volume_dev).
template <int N, bool PERSIST, bool MORT = false>
__global__ void __launch_bounds__(grad_dev_threads<N>()) k_grad_dev(const __grid_constant__ Batch b,
                                                                    const Ops *__restrict__ ops, long long ntiles)
{
    pdl_wait();
    constexpr int n3 = (N + 1) * (N + 1) * (N + 1);
    constexpr bool BULK = ((N + 1) % 2 == 0);
    __shared__ unsigned long long bulk_bar[BULK ? 256 / (n3 < 256 ? n3 : 256) : 1];
    if constexpr (!PERSIST) {
        grad_dev_tile<N, MORT>(b, ops, blockIdx.x, bulk_bar);
    } else {
        for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            const bool armed = grad_dev_tile_call<N>(b, ops, tile, bulk_bar);
            if (tile + gridDim.x >= ntiles) break;   // (uniform across the CTA)
            __syncthreads();
            if (armed) mbar_inval(bulk_bar + threadIdx.x / n3);
        }
    }
}

// ------------------------------------------------------------------ four nodes per thread

// Row kernel, N = 7: a thread owns four consecutive nodes along xi, an element
// is one CTA of 128 threads instead of 512 (whose barriers stall half an SM).
// Per node the contraction needs 27 (n-1) multiply-adds of the nine stress
// products, formed once per node and direction, instead of 45 n instructions
// and 24 n shared-memory loads: xi-lines are contracted in registers (the two
// halves of a line swap their products by shuffles), eta- and zeta-lines read the
// products of four nodes with one 16-byte load, and every global array is read
// and written 16 bytes per thread.  32^3 elements, per launch: 787 -> 648 us.  (At
// N = 3, 16 lanes an element, it measured 1% slower than one node per thread.)
// FEW, up to kFewElems elements: at most two CTAs come to an SM anyway, so the
// register budget is theirs (152 instead of 96), which lets the metric terms'
// loads start ahead of the traces' arithmetic: 150 elements 11.9 -> 10.5 us a
// launch, 216 14.0 -> 12.7; the same results bit for bit.
template <int N>
struct GradRow {
    static constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
    static constexpr int RPL = n / 4;              // threads per xi-line
    static constexpr int TPE = n2 * RPL;           // threads per element (one CTA)
    static constexpr int DW = 2 * n2;              // D (zero diagonal) and its transpose
    // floats: products [9][n3], neighbour traces [6][4][n2]
    static constexpr size_t SMEM = sizeof(float) * (DW + 9 * n3 + 24 * n2);
    static_assert(TPE == 128, "one element per CTA of 128 threads");
};
template <int N>
constexpr bool has_grad_row()
{
    return N == 7;
}

__device__ __forceinline__ float4 ld4(const float *p) { return *(const float4 *)p; }
// Sums of four nodes as packed pairs (0, 1), (2, 3) (two FP32 operations per issue slot).
__device__ __forceinline__ void fma4(float2 acc[2][kVisc], int k, float d, const float4 &w)
{
    acc[0][k] = __ffma2_rn(make_float2(d, d), make_float2(w.x, w.y), acc[0][k]);
    acc[1][k] = __ffma2_rn(make_float2(d, d), make_float2(w.z, w.w), acc[1][k]);
}
__device__ __forceinline__ float at4(const float4 &v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

// Stress product k (stress_add's order) of the metric a and q = (v, T).
__device__ __forceinline__ float stress_term(int k, float a1, float a2, float a3, const float q[4])
{
    switch (k) {
        case 0: return a1 * q[0];
        case 1: return a2 * q[1];
        case 2: return a3 * q[2];
        case 3: return fmaf(a1, q[1], a2 * q[0]);
        case 4: return fmaf(a1, q[2], a3 * q[0]);
        case 5: return fmaf(a2, q[2], a3 * q[1]);
        case 6: return a1 * q[3];
        case 7: return a2 * q[3];
        default: return a3 * q[3];
    }
}

template <int N, bool PERSIST, bool FEW = false>
__global__ void __launch_bounds__(128, FEW ? 2 : 5) k_grad_row(const __grid_constant__ Batch b,
                                                               const Ops *__restrict__ ops, long long ntiles)
{
    using S = GradRow<N>;
    constexpr int n = S::n, n2 = S::n2, n3 = S::n3, RPL = S::RPL, TPE = S::TPE;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *sD = (float *)smem_raw, *sT = sD + n2;
    pdl_wait();
    for (int t = threadIdx.x; t < n2; t += TPE) {
        const float v = (t % (n + 1) == 0) ? 0.0f : ops->Df[t];
        sD[t] = v;
        sT[(t % n) * n + t / n] = v;
    }
    const float dend = ops->Df[n2 - 1];
    const int r = threadIdx.x, h = r % RPL, j = (r / RPL) % n, k = r / (RPL * n), p0 = 4 * r;
    float *W = sD + S::DW;                         // [9][n3]
    float *qn = W + 9 * n3;                        // [6][4][n2]
    __syncthreads();
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const long long ge = tile;
        bool valid = ge < b.total_elems;
        const Item *itp = &b.single;
        int e = 0;
        if (valid) {
            itp = &find_item_elem(b, ge);
            e = (int)(ge - itp->elem_begin);
            if (itp->clk && itp->clk->done) valid = false;
        }
        const Item &it = *itp;
        float q[4][4];
        if (valid) {
            // the metric terms, needed after the traces, toward L2 (the run -1%)
            prefetch_l2_block(it.Jaf + (size_t)e * 9 * n3, sizeof(float) * 9 * n3, r, TPE);
            double uo[5][4];
            const double *U = it.u + (size_t)e * 5 * n3 + p0;
#pragma unroll
            for (int v = 0; v < 5; ++v) {
                const double2 lo = *(const double2 *)(U + v * n3), hi = *(const double2 *)(U + v * n3 + 2);
                uo[v][0] = lo.x;
                uo[v][1] = lo.y;
                uo[v][2] = hi.x;
                uo[v][3] = hi.y;
            }
            const AnchorRec R = load_anchor(it.anc, e);
            const float gm1 = it.gm1f;
            const Anchor A = R.a;
            const float Tb = A.p * __fdividef(1.0f, A.rho);
            const float rT = fmaf(-Tb, A.rho, A.p);
            // neighbour traces: 6 n^2 face points over the element's threads
            const Nbrs nbs = elem_nbrs(e, it.ex, it.ey, it.ez);
            constexpr int IT = 6 * n2 / TPE;
            constexpr int BATCH = 3;   // face points loaded ahead of their conversion
#pragma unroll
            for (int c = 0; c < IT; c += BATCH) {
                double raw[BATCH][5];
#pragma unroll
                for (int s = 0; s < BATCH; ++s) {
                    const int t = r + (c + s) * TPE;
                    const int slot = t / n2, ab = t - slot * n2;
                    const int d = slot >> 1, plus = slot & 1;
                    const double *src = it.u + (size_t)nbr_of_slot(nbs, slot) * 5 * n3 +
                                        gd_face_node<n>(d, plus ? 0 : N, ab % n, ab / n);
#pragma unroll
                    for (int v = 0; v < 5; ++v) raw[s][v] = src[v * n3];
                }
#pragma unroll
                for (int s = 0; s < BATCH; ++s) {
                    const int t = r + (c + s) * TPE;
                    const int slot = t / n2, ab = t - slot * n2;
                    float g4[4];
                    grad_dev_vars(make_dev_rec(raw[s], A, R.Elo, gm1), A, Tb, rT, g4);
#pragma unroll
                    for (int v = 0; v < 4; ++v) qn[(slot * 4 + v) * n2 + ab] = g4[v];
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const double ui[5] = {uo[0][i], uo[1][i], uo[2][i], uo[3][i], uo[4][i]};
                grad_dev_vars(make_dev_rec(ui, A, R.Elo, gm1), A, Tb, rT, q[i]);
            }
        }
        __syncthreads();
        float2 acc[2][kVisc];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int c = 0; c < kVisc; ++c) acc[i][c] = make_float2(0.0f, 0.0f);
        // one node's stress products onto its sums
        auto add_node = [&](int i, float a1, float a2, float a3, float q1, float q2, float q3, float T) {
            float t[kVisc];
#pragma unroll
            for (int c = 0; c < kVisc; ++c) t[c] = i & 1 ? acc[i >> 1][c].y : acc[i >> 1][c].x;
            stress_add(t, a1, a2, a3, q1, q2, q3, T);
#pragma unroll
            for (int c = 0; c < kVisc; ++c) (i & 1 ? acc[i >> 1][c].y : acc[i >> 1][c].x) = t[c];
        };
        const float *JA = it.Jaf + (size_t)e * 9 * n3 + p0;
        // the diagonal term at the two ends of a line: D_ii Ja q_out (see k_grad_dev)
        auto end_row = [&](const float4 J[3], const float *Q, float dn) {
            const float4 Q0 = ld4(Q), Q1 = ld4(Q + n2), Q2 = ld4(Q + 2 * n2), Q3 = ld4(Q + 3 * n2);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                add_node(i, dn * at4(J[0], i), dn * at4(J[1], i), dn * at4(J[2], i), at4(Q0, i), at4(Q1, i), at4(Q2, i),
                         at4(Q3, i));
        };
        float4 J[3];
        if (valid) {
            // xi: in registers
#pragma unroll
            for (int c = 0; c < 3; ++c) J[c] = ld4(JA + c * n3);
            float4 Dm[4];   // column m of D for this thread's four nodes
#pragma unroll
            for (int m = 0; m < 4; ++m) Dm[m] = ld4(sT + (4 * h + m) * n + 4 * h);
#pragma unroll
            for (int c = 0; c < kVisc; ++c)
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float s = stress_term(c, at4(J[0], m), at4(J[1], m), at4(J[2], m), q[m]);
                    fma4(acc, c, s, Dm[m]);
                }
            {
                if (h == 0) {
                    const float *Q = qn + j + n * k;
                    add_node(0, -dend * J[0].x, -dend * J[1].x, -dend * J[2].x, Q[0], Q[n2], Q[2 * n2], Q[3 * n2]);
                }
                if (h == RPL - 1) {
                    const float *Q = qn + 4 * n2 + j + n * k;
                    add_node(3, dend * J[0].w, dend * J[1].w, dend * J[2].w, Q[0], Q[n2], Q[2 * n2], Q[3 * n2]);
                }
            }
        }
        {
            // the other half of the line: its products by shuffles (its J and q
            // instead would be 28 values against 36, but every product twice)
            float4 Dm[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) Dm[m] = ld4(sT + (4 * (h ^ 1) + m) * n + 4 * h);
#pragma unroll
            for (int c = 0; c < kVisc; ++c)
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float mine = valid ? stress_term(c, at4(J[0], m), at4(J[1], m), at4(J[2], m), q[m]) : 0.0f;
                    fma4(acc, c, __shfl_xor_sync(0xffffffffu, mine, 1), Dm[m]);
                }
        }
        // eta, then zeta: products through shared memory
#pragma unroll
        for (int d = 1; d < 3; ++d) {
            const int i = d == 1 ? j : k;
            if (valid) {
#pragma unroll
                for (int c = 0; c < 3; ++c) J[c] = ld4(JA + (d * 3 + c) * n3);
#pragma unroll
                for (int c = 0; c < kVisc; ++c) {
                    float4 s;
                    s.x = stress_term(c, J[0].x, J[1].x, J[2].x, q[0]);
                    s.y = stress_term(c, J[0].y, J[1].y, J[2].y, q[1]);
                    s.z = stress_term(c, J[0].z, J[1].z, J[2].z, q[2]);
                    s.w = stress_term(c, J[0].w, J[1].w, J[2].w, q[3]);
                    *(float4 *)(W + c * n3 + p0) = s;
                }
                if (i == 0 || i == N)
                    end_row(J, qn + (2 * d + (i == N ? 1 : 0)) * 4 * n2 + 4 * h + n * (d == 1 ? k : j),
                            i == N ? dend : -dend);
            }
            __syncthreads();
            if (valid) {
                const float *row = W + 4 * h + (d == 1 ? n2 * k : n * j);
                const int step = d == 1 ? n : n2;
#pragma unroll
                for (int m = 0; m < n; ++m) {
                    const float Dm = sD[i * n + m];
#pragma unroll
                    for (int c = 0; c < kVisc; ++c) fma4(acc, c, Dm, ld4(row + c * n3 + m * step));
                }
            }
            if (d == 1 || PERSIST) __syncthreads();   // W is written again
        }
        if (valid) {
            const float4 ij = ld4(it.invJf + (size_t)e * n3 + p0);
            float *G = (float *)it.grad + (size_t)e * kVisc * n3 + p0;
            float tau[4][kVisc];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float t[kVisc];
#pragma unroll
                for (int c = 0; c < kVisc; ++c) t[c] = i & 1 ? acc[i >> 1][c].y : acc[i >> 1][c].x;
                stress_of(t, at4(ij, i), it.muf, it.kappaf, tau[i]);
            }
#pragma unroll
            for (int c = 0; c < kVisc; ++c)
                *(float4 *)(G + c * n3) = make_float4(tau[0][c], tau[1][c], tau[2][c], tau[3][c]);
        }
        if (!PERSIST) break;
    }
}

template <int N>
static cudaError_t grad_dev_launch(const Batch &b, cudaStream_t s)
{
    constexpr int n = N + 1, n3 = n * n * n;
    if (b.total_elems == 0) return cudaSuccess;
    if constexpr (has_grad_row<N>()) {
        if (!b.mortar) {
            using S = GradRow<N>;
            const unsigned tiles = (unsigned)b.total_elems;
            const Ops *ops = device_ops(N);
            if (!ops) return cudaErrorMemoryAllocation;
            const cudaError_t e =
                b.persistent ? launch_pdl(k_grad_row<N, true>,
                                          persistent_grid(k_grad_row<N, true>, S::TPE, S::SMEM, tiles), S::TPE, S::SMEM,
                                          s, b, ops, (long long)tiles)
                             : launch_pdl(b.total_elems <= kFewElems ? k_grad_row<N, false, true> : k_grad_row<N, false>,
                                          tiles, S::TPE, S::SMEM, s, b, ops, (long long)tiles);
            return e != cudaSuccess ? e : cudaGetLastError();
        }
    }
    const int epb = elems_per_cta(N, HS3D_MIXED32, kShapeGrad, HS3D_VOL_STANDARD, false, b.total_elems, b.beside);
    const int threads = epb * n3;
    const size_t smem = sizeof(float) * (((n * n + 3) & ~3) + (size_t)epb * grad_dev_per_elem<N>());
    const unsigned blocks = (unsigned)((b.total_elems + epb - 1) / epb);
    const Ops *ops = device_ops(N);
    if (!ops) return cudaErrorMemoryAllocation;
    cudaError_t e = cudaSuccess;
    if (b.mortar || has_grad_row<N>()) {
        e = launch_pdl(k_grad_dev<N, false, true>, blocks, threads, smem, s, b, ops, (long long)blocks);
    } else {
        if constexpr (!has_grad_row<N>()) {
            if (b.persistent) {
                const unsigned grid = persistent_grid(k_grad_dev<N, true>, threads, smem, blocks);
                e = launch_pdl(k_grad_dev<N, true>, grid, threads, smem, s, b, ops, (long long)blocks);
            } else {
                e = launch_pdl(k_grad_dev<N, false>, blocks, threads, smem, s, b, ops, (long long)blocks);
            }
        }
    }
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template <typename K>
static cudaError_t grad_dev_prep_one(K kernel)
{
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    return e;
}

template <int N>
static cudaError_t grad_dev_prep()
{
    cudaError_t e = grad_dev_prep_one(k_grad_dev<N, false, true>);
    if constexpr (has_grad_row<N>()) {
        if (e == cudaSuccess) e = grad_dev_prep_one(k_grad_row<N, false>);
        if (e == cudaSuccess) e = grad_dev_prep_one(k_grad_row<N, false, true>);
        if (e == cudaSuccess) e = grad_dev_prep_one(k_grad_row<N, true>);
    } else {
        if (e == cudaSuccess) e = grad_dev_prep_one(k_grad_dev<N, false>);
        if (e == cudaSuccess) e = grad_dev_prep_one(k_grad_dev<N, true>);
    }
    return e;
}

cudaError_t launch_grad_dev(int N, const Batch &b, cudaStream_t s)
{
    switch (N) {
        case 1: return grad_dev_launch<1>(b, s);
        case 2: return grad_dev_launch<2>(b, s);
        case 3: return grad_dev_launch<3>(b, s);
        case 4: return grad_dev_launch<4>(b, s);
        case 5: return grad_dev_launch<5>(b, s);
        case 6: return grad_dev_launch<6>(b, s);
        case 7: return grad_dev_launch<7>(b, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t prepare_grad_dev(int N)
{
    switch (N) {
        case 1: return grad_dev_prep<1>();
        case 2: return grad_dev_prep<2>();
        case 3: return grad_dev_prep<3>();
        case 4: return grad_dev_prep<4>();
        case 5: return grad_dev_prep<5>();
        case 6: return grad_dev_prep<6>();
        case 7: return grad_dev_prep<7>();
    }
    return cudaErrorInvalidValue;
}

}  // namespace hs3d
