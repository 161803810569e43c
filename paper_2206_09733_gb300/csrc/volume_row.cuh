// Element kernel of the mixed path's standard form at N = 7 for launches over more
// than kFewElems elements (volume_dev.cuh states the method and why the line lies
// there): four consecutive nodes along xi per thread in the contraction.
//
// With one thread per node an element is a CTA of 512 threads, two of which
// fill an SM's registers: each of its barriers stalls half the SM, and every
// contracted value costs its own 4-byte shared-memory load (144 a node).  Here an
// element is a CTA of 128 threads, five to an SM.  A thread first forms the
// staged fluxes of four nodes a quarter of the element apart (coalesced loads,
// conflict-free stores, few registers), then takes the nodes 4r .. 4r + 3 of a
// xi-line: rows of eta- and zeta-lines and the line itself come as 16-byte loads,
// the RK update reads and writes global memory 16 bytes at a time.
// 20^3 elements, 4 steps: Euler 4.12 -> 3.40 ms; 32^3 elements, NS, per launch: 1157 -> 1020 us.
// Contractions two nodes to a packed instruction: the run of 32^3, NS, 23.3 -> 22.6 ms
// per 4 steps, Euler 20^3 3.40 -> 3.29.
// (At N = 3, 16 lanes an element, the same kernel measured 20% slower than one
// node per thread: too few warps to cover the loads.)
#pragma once

#include "volume_dev.cuh"

namespace hs3d {

template <int N>
struct VolRow {
    static constexpr int n = N + 1, n2 = n * n, n3 = n2 * n;
    static constexpr int RPL = n / 4;              // threads per xi-line
    static constexpr int TPE = n2 * RPL;           // threads per element (one CTA)
    static constexpr int DW = 4 * n2;              // D and its low part, row-major and transposed
    // floats: per direction four rest fluxes, then per direction the float-float
    // mass flux (hi, lo)
    static constexpr size_t SMEM = sizeof(float) * (DW + 18 * n3);
    static_assert(TPE == 128, "one element per CTA of 128 threads");
};

template <int N, bool NS, bool PERSIST>
__global__ void __launch_bounds__(128, 5) k_volume_row(const __grid_constant__ Batch b, const Ops *__restrict__ ops,
                                                       int stage, float rkA, double rkB, int lam_slot,
                                                       long long ntiles)
{
    using S = VolRow<N>;
    constexpr int n = S::n, n2 = S::n2, n3 = S::n3, RPL = S::RPL, TPE = S::TPE;
    constexpr int pc = anchor_node(n);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *sD = (float *)smem_raw, *sDl = sD + n2, *sT = sDl + n2, *sTl = sT + n2;
    pdl_wait();
    for (int t = threadIdx.x; t < n2; t += TPE) {
        const int tt = (t % n) * n + t / n;
        sD[t] = sT[tt] = ops->Df[t];
        sDl[t] = sTl[tt] = ops->Dlo[t];
    }
    const int r = threadIdx.x, h = r % RPL, j = (r / RPL) % n, k = r / (RPL * n), p0 = 4 * r;
    float *W = sD + S::DW;
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
        float Hb = 0.0f;
        // this element's side of its six faces; toward L2 while the fluxes are formed
        const float *face[6] = {};
        if (valid) {
            const Nbrs nb = elem_nbrs(e, it.ex, it.ey, it.ez);
            const float *FS = (const float *)it.fstar;
#pragma unroll
            for (int slot = 0; slot < 6; ++slot) {
                const int d = slot >> 1;
                face[slot] = FS + ((slot & 1) ? (((size_t)d * it.E + e) * 2) * 5 * n2
                                              : (((size_t)d * it.E + nb.m[d]) * 2 + 1) * 5 * n2);
                prefetch_l2_block(face[slot], sizeof(float) * 5 * n2, r, TPE);
            }
            // all the element's inputs toward L2: the loop below loads a quarter of them
            // per round, and 20 warps on an SM cannot cover DRAM four times over (32^3,
            // NS, 4 steps 22.6 -> 21.6 ms; 20^3, Euler 3.29 -> 3.06; the RK register as
            // well: +0.5%)
            prefetch_l2_block(it.u + (size_t)e * 5 * n3, sizeof(double) * 5 * n3, r, TPE);
            prefetch_l2_block(it.Jaf + (size_t)e * 9 * n3, sizeof(float) * 9 * n3, r, TPE);
            prefetch_l2_block(it.Jalo + (size_t)e * 9 * n3, sizeof(float) * 9 * n3, r, TPE);
            if (NS) prefetch_l2_block((const float *)it.grad + (size_t)e * kVisc * n3, sizeof(float) * kVisc * n3, r, TPE);
            const AnchorRec R = load_anchor(it.anc, e);
            const Anchor A = R.a;
            Hb = A.H;
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
                const int p = r + c * TPE;
                const double *U = it.u + (size_t)e * 5 * n3 + p;
                double u[5];
#pragma unroll
                for (int v = 0; v < 5; ++v) u[v] = U[v * n3];
                const float *JA = it.Jaf + (size_t)e * 9 * n3 + p, *JL = it.Jalo + (size_t)e * 9 * n3 + p;
                float ja[9], jl[9];
#pragma unroll
                for (int m = 0; m < 9; ++m) ja[m] = JA[m * n3];
#pragma unroll
                for (int m = 0; m < 9; ++m) jl[m] = JL[m * n3];
                float G[kVisc];
                if (NS) {
                    const float *Gp = (const float *)it.grad + (size_t)e * kVisc * n3 + p;
#pragma unroll
                    for (int m = 0; m < kVisc; ++m) G[m] = Gp[m * n3];
                }
                // momentum deviations as FP32 pairs (hi: the deviation rounded once; lo: the rest)
                float mh[3], ml[3];
#pragma unroll
                for (int m = 0; m < 3; ++m) ff_split(u[1 + m] - R.ad[1 + m], mh[m], ml[m]);
                const Dev dv = make_dev_f(dev_round(u[0] - R.ad[0]), mh[0], mh[1], mh[2], dev_round(u[4] - R.ad[4]), A,
                                          it.gm1f);
                const float dH = dev_dH(dv, A);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    float wh = 0.0f, wl = 0.0f;
                    ff_mul(wh, wl, ja[d * 3], jl[d * 3], mh[0], ml[0]);
                    ff_fma(wh, wl, ja[d * 3 + 1], jl[d * 3 + 1], mh[1], ml[1]);
                    ff_fma(wh, wl, ja[d * 3 + 2], jl[d * 3 + 2], mh[2], ml[2]);
                    W[(12 + 2 * d) * n3 + p] = wh;
                    W[(13 + 2 * d) * n3 + p] = wl;
                    float f[4];
                    dflux_euler_rest(dv, A, dH, ja[d * 3], ja[d * 3 + 1], ja[d * 3 + 2], f);
                    if (NS) {
                        float fv[5];
                        visc_flux(dev_prim(dv, A), G, ja[d * 3], ja[d * 3 + 1], ja[d * 3 + 2], fv);
#pragma unroll
                        for (int v = 0; v < 4; ++v) f[v] -= fv[v + 1];
                    }
#pragma unroll
                    for (int v = 0; v < 4; ++v) W[(d * 4 + v) * n3 + p] = f[v];
                }
            }
        }
        __syncthreads();
        float lc = 0.0f, lv = 0.0f;
        bool lam_active = false;
        if (valid) {
            // the RK update's inputs, ahead of the contraction
            float *Gp = (float *)it.g + (size_t)e * 5 * n3 + p0;
            const float4 ij = *(const float4 *)(it.invJf + (size_t)e * n3 + p0);
            float4 g4[5];
            double dtv = 0.0;
            if (stage >= 0) {
                dtv = it.clk->dt;
                if (stage > 0) {
#pragma unroll
                    for (int v = 0; v < 5; ++v) g4[v] = *(const float4 *)(Gp + v * n3);
                }
            }
            // packed pairs of nodes (0, 1), (2, 3): rows of rest fluxes, mass (hi, lo)
            float2 P[2][4], Ch[2], Cl[2];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int v = 0; v < 4; ++v) P[i][v] = pair(0.0f);
            // xi: the line's own rows against the columns of D
#pragma unroll
            for (int c = 0; c < RPL; ++c) {
                const float *row = W + n * (j + n * k) + 4 * c;
                float f[6][4];
#pragma unroll
                for (int v = 0; v < 4; ++v) *(float4 *)f[v] = *(const float4 *)(row + v * n3);
                *(float4 *)f[4] = *(const float4 *)(row + 12 * n3);
                *(float4 *)f[5] = *(const float4 *)(row + 13 * n3);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const float4 D = *(const float4 *)(sT + (4 * c + m) * n + 4 * h);
                    const float4 L = *(const float4 *)(sTl + (4 * c + m) * n + 4 * h);
                    const float2 D2[2] = {make_float2(D.x, D.y), make_float2(D.z, D.w)};
                    const float2 L2[2] = {make_float2(L.x, L.y), make_float2(L.z, L.w)};
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
#pragma unroll
                        for (int v = 0; v < 4; ++v) P[i][v] = __ffma2_rn(D2[i], pair(f[v][m]), P[i][v]);
                        if (c == 0 && m == 0) ff_mul2(Ch[i], Cl[i], D2[i], L2[i], pair(f[4][m]), pair(f[5][m]));
                        else ff_fma2(Ch[i], Cl[i], D2[i], L2[i], pair(f[4][m]), pair(f[5][m]));
                    }
                }
            }
            // eta and zeta: rows of four nodes
#pragma unroll
            for (int d = 1; d < 3; ++d) {
                const float *row = W + 4 * h + (d == 1 ? n2 * k : n * j);
                const int step = d == 1 ? n : n2, at = (d == 1 ? j : k) * n;
#pragma unroll
                for (int m = 0; m < n; ++m) {
                    const float2 D = pair(sD[at + m]), L = pair(sDl[at + m]);
                    const float4 mh = *(const float4 *)(row + (12 + 2 * d) * n3 + m * step);
                    const float4 ml = *(const float4 *)(row + (13 + 2 * d) * n3 + m * step);
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const float4 f = *(const float4 *)(row + (d * 4 + v) * n3 + m * step);
                        P[0][v] = __ffma2_rn(D, make_float2(f.x, f.y), P[0][v]);
                        P[1][v] = __ffma2_rn(D, make_float2(f.z, f.w), P[1][v]);
                    }
                    ff_fma2(Ch[0], Cl[0], D, L, make_float2(mh.x, mh.y), make_float2(ml.x, ml.y));
                    ff_fma2(Ch[1], Cl[1], D, L, make_float2(mh.z, mh.w), make_float2(ml.z, ml.w));
                }
            }
            // volume rows: mass = C, energy = Hbar mass + rest
            float V[4][5];   // [node][row]
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                V[2 * i][0] = Ch[i].x + Cl[i].x;
                V[2 * i + 1][0] = Ch[i].y + Cl[i].y;
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    V[2 * i][v + 1] = P[i][v].x;
                    V[2 * i + 1][v + 1] = P[i][v].y;
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) V[i][4] += Hb * V[i][0];
            // surface term: +-(1/w) G on the faces the nodes lie on
            const float iw = ops->iw0f;
            if (h == 0) {
                const float *F = face[0] + j + n * k;
#pragma unroll
                for (int v = 0; v < 5; ++v) V[0][v] += -iw * F[v * n2];
            }
            if (h == RPL - 1) {
                const float *F = face[1] + j + n * k;
#pragma unroll
                for (int v = 0; v < 5; ++v) V[3][v] += iw * F[v * n2];
            }
#pragma unroll
            for (int d = 1; d < 3; ++d) {
                const int i = d == 1 ? j : k;
                if (i != 0 && i != N) continue;
                const float sw = i == N ? iw : -iw;
                const float *F = (i == N ? face[2 * d + 1] : face[2 * d]) + 4 * h + n * (d == 1 ? k : j);
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                    const float4 f = *(const float4 *)(F + v * n2);
                    V[0][v] += sw * f.x;
                    V[1][v] += sw * f.y;
                    V[2][v] += sw * f.z;
                    V[3][v] += sw * f.w;
                }
            }
            const float ijf[4] = {ij.x, ij.y, ij.z, ij.w};
            if (stage < 0) {
                double *O = it.out + (size_t)e * 5 * n3 + p0;
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                    *(double2 *)(O + v * n3) = make_double2(f2d_exact(-V[0][v] * ijf[0]), f2d_exact(-V[1][v] * ijf[1]));
                    *(double2 *)(O + v * n3 + 2) = make_double2(f2d_exact(-V[2][v] * ijf[2]), f2d_exact(-V[3][v] * ijf[3]));
                }
            } else {
                // FP32 register, FP64 state (as volume_dev_tile)
                const float dtf = __double2float_rn(dtv);
                double *Up = it.u + (size_t)e * 5 * n3 + p0;
                float nf[4][5];
                double uc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};   // the centre node's new state
#pragma unroll
                for (int v = 0; v < 5; ++v) {
                    const double2 lo = *(const double2 *)(Up + v * n3), hi = *(const double2 *)(Up + v * n3 + 2);
                    double u[4] = {lo.x, lo.y, hi.x, hi.y};
                    const float gp[4] = {g4[v].x, g4[v].y, g4[v].z, g4[v].w};
                    float gv[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float inc = -V[i][v] * (dtf * ijf[i]);
                        gv[i] = (stage == 0) ? inc : fmaf(rkA, gp[i], inc);
                        u[i] = fma(rkB, f2d_exact(gv[i]), u[i]);
                        if (lam_slot >= 0) nf[i][v] = d2f_rn(u[i]);
                    }
                    *(float4 *)(Gp + v * n3) = make_float4(gv[0], gv[1], gv[2], gv[3]);
                    *(double2 *)(Up + v * n3) = make_double2(u[0], u[1]);
                    *(double2 *)(Up + v * n3 + 2) = make_double2(u[2], u[3]);
                    uc[v] = u[pc % 4];
                }
                // the reference state of the next stage
                if (r == pc / 4) write_anchor(it, e, uc);
                if (lam_slot >= 0) {
                    const float *JA = it.Jaf + (size_t)e * 9 * n3 + p0;
                    float jf[9][4];
#pragma unroll
                    for (int m = 0; m < 9; ++m) *(float4 *)jf[m] = *(const float4 *)(JA + m * n3);
                    bool bad = false;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const Prim<float> qn = prim_from_f(nf[i], it.gm1f);
                        if (!(qn.rho > 0.0f) || !(qn.p > 0.0f)) {
                            bad = true;
                            continue;
                        }
                        const float c = sqrtf(it.gammaf * qn.p / qn.rho);
                        float sc = 0.0f, sv = 0.0f;
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            const float a1 = jf[d * 3][i], a2 = jf[d * 3 + 1][i], a3 = jf[d * 3 + 2][i];
                            const float an = sqrtf(a1 * a1 + a2 * a2 + a3 * a3);
                            sc += (fabsf(a1 * qn.v1 + a2 * qn.v2 + a3 * qn.v3) + c * an) * ijf[i];
                            sv += (an * ijf[i]) * (an * ijf[i]);
                        }
                        lc = fmaxf(lc, sc);
                        if (NS) lv = fmaxf(lv, it.muf * sv / qn.rho);
                        lam_active = true;
                    }
                    if (bad) it.clk->bad = 1;
                }
            }
        }
        if (lam_slot >= 0 && stage >= 0) rates_to_clock<float>(b, itp, lam_slot, NS, lc, lv, lam_active);
        if (!PERSIST) break;
        __syncthreads();   // the staging is written again
    }
}

template <int N, bool NS>
static cudaError_t vol_row_launch(const Batch &b, int stage, float rkA, double rkB, int lam_slot, cudaStream_t s)
{
    using S = VolRow<N>;
    const unsigned tiles = (unsigned)b.total_elems;
    const Ops *ops = device_ops(N);
    if (!ops) return cudaErrorMemoryAllocation;
    const int slot = stage >= 0 ? lam_slot : -1;
    if (b.persistent)
        return launch_pdl(k_volume_row<N, NS, true>, persistent_grid(k_volume_row<N, NS, true>, S::TPE, S::SMEM, tiles),
                          S::TPE, S::SMEM, s, b, ops, stage, rkA, rkB, slot, (long long)tiles);
    return launch_pdl(k_volume_row<N, NS, false>, tiles, S::TPE, S::SMEM, s, b, ops, stage, rkA, rkB, slot,
                      (long long)tiles);
}

template <int N>
static cudaError_t vol_row_prep()
{
    cudaError_t e = prep_vol_dev_kernel(k_volume_row<N, false, false>);
    if (e == cudaSuccess) e = prep_vol_dev_kernel(k_volume_row<N, true, false>);
    if (e == cudaSuccess) e = prep_vol_dev_kernel(k_volume_row<N, false, true>);
    if (e == cudaSuccess) e = prep_vol_dev_kernel(k_volume_row<N, true, true>);
    return e;
}

}  // namespace hs3d
