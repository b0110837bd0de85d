// CUDA kernels of the FDLB solver for the simplified Enskog equation (sm_103a).
//
// One TVD-RK3 stage (Eq. rk3) is two kernels over a batch of independent channel problems:
//   k_nodal    per node: chi (Eq. chi), Pr (Eq. prandtl), tau (Eqs. viscosity, tau),
//              6th-order gradients (Sec. III B 3), the 13 monomial coefficients of
//              f^S + tau J1 (Sec. II A, Eq. j1) and their projections onto the
//              half-range (Sec. III A 2) and full-range (App. A) velocity sets (on x
//              either rule);
//              per instance: the wall densities n_w (Sec. III B);
//   k_update   per (velocity, node): WENO-5 fluxes (Sec. III B 2) with the
//              diffuse-reflection closure, the p_y-derivative force (App. A,
//              Eq. kernel_H), relaxation to the projected target and the RK3
//              combination; its epilogue reduces the new values to the moments
//              n, u, T, q, Pi of every node (Eq. macro_LB) for the next stage.
// After stage 3 the residual pass (per-step residual, status): blocks of the next step's first
// k_nodal, or k_resid.  k_moments computes the moments
// from scratch (creation, new profiles, a loaded state) with the epilogue's arithmetic.
// k_resident runs whole steps of one instance per thread-block cluster with the same item
// functions.
//
// Storage type S (double | float) holds f; compute type C of the per-velocity work is
// double for FDLB_FP64 and float for FDLB_FP32_STORAGE.  FP64 instances do all the rest in
// double (but for the WENO weights of smooth stencils, fdlb_weno.cuh); FP32-storage instances run the moment sums
// and their finalisation, the velocity projections and the closure chain in double-float (float
// pairs) and keep the gradients and the residual in double.
#include "fdlb_internal.h"
#include "fdlb_launch.h"
#include "fdlb_round.cuh"
#include "fdlb_weno.cuh"
#include "../../include/fdlb.h"

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math_constants.h>

#include <mutex>

namespace fdlb {

__constant__ int c_mono[NTERMS][3] = {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {2, 0, 0}, {0, 2, 0}, {0, 0, 2}, {1, 1, 0},
                                      {3, 0, 0}, {1, 2, 0}, {1, 0, 2}, {2, 1, 0}, {0, 3, 0}, {0, 1, 2}};

// Column `lane` of tile i0's projection table (rows TILE apart).
__device__ __forceinline__ size_t tab_col(const Inst& I, int i0, int lane) { return (size_t)(i0 / TILE) * I.ntab * TILE + lane; }

__device__ __forceinline__ double chi_cs(double eta) {
    const double om = 1.0 - eta;
    return (2.0 - eta) / (2.0 * om * om * om);
}

// ---------------------------------------------------------------------------
// projections of (p - u)^a g(p; u, T), a = 0..3
// ---------------------------------------------------------------------------

// Half-range axis (Sec. III A 2): value at node +p_k (half = 0) of
//   int_0^inf l_k(p) (p - u)^a g(p; u, T) dp,
// or at node -p_k (half = 1), which is (-1)^a times the same with u -> -u.  Evaluated in
// the orthonormal basis, value_k = w_k sum_l h_l(p_k) G_l, with
//   G_l = int_0^inf h_l(p) (p - u)^a g dp = sum_m W_m exp(q_m v - v^2/2) h_l(sqrt(T) q_m) y_m^a,
// p = sqrt(T) q, v = u/sqrt(T), y_m = sqrt(T) q_m - u, on the MX-point auxiliary rule.
// Full-range x axis (App. A, I.xfull): the integrals run over the whole line with the
// 2Q-node basis, G_l = sum_m W_m h_l(u + sqrt(T) y_m) (sqrt(T) y_m)^a on the Mx-point
// Gauss-Hermite rule (exact); the rule is symmetric, so the mirror relation for -p_k holds
// as well.
__device__ void proj_x(const Inst& I, double u, double T, int half, double* out, int stride) {
    const int Q = I.Q, Lx = I.Lx;
    const bool full = I.xfull;
    const double uu = half ? -u : u;
    const double sT = sqrt(T), v = uu / sT, ev = -0.5 * v * v;
    const int M = I.Mx;
    // the polynomials in blocks of QMAX; the H products continue one chain across blocks
    // (kept in out, signed at the end)
    for (int lb = 0; lb < Lx; lb += QMAX) {
        const int nl = min(QMAX, Lx - lb);
        double G[4][QMAX];
#pragma unroll
        for (int a = 0; a < 4; ++a)
            for (int l = 0; l < QMAX; ++l) G[a][l] = 0.0;
        for (int m = 0; m < M; ++m) {
            const double q = I.xq[m];
            const double x = full ? fma(sT, q, uu) : sT * q;
            const double E = full ? I.xw[m] : I.xw[m] * exp(fma(q, v, ev));
            const double y = full ? sT * q : x - uu;
            const double e1 = E * y, e2 = e1 * y, e3 = e2 * y;
            double hm = 0.0, h = I.x_h0;
            for (int l = 0; l < lb; ++l) {
                const double hn = ((x - I.xa[l]) * h - I.xb[l] * hm) * I.xib[l + 1];
                hm = h;
                h = hn;
            }
            for (int j = 0; j < nl; ++j) {
                const int l = lb + j;
                G[0][j] = fma(E, h, G[0][j]);
                G[1][j] = fma(e1, h, G[1][j]);
                G[2][j] = fma(e2, h, G[2][j]);
                G[3][j] = fma(e3, h, G[3][j]);
                const double hn = ((x - I.xa[l]) * h - I.xb[l] * hm) * I.xib[l + 1];
                hm = h;
                h = hn;
            }
        }
        const bool last = lb + nl == Lx;
        for (int a = 0; a < 4; ++a) {
            const double sgn = (half && (a & 1)) ? -1.0 : 1.0;
            for (int k = 0; k < Q; ++k) {
                double* o = out + (a * 2 * Q + half * Q + k) * stride;
                double s = lb == 0 ? 0.0 : *o;
                for (int j = 0; j < nl; ++j) s = fma(I.xH[(lb + j) * Q + k], G[a][j], s);
                *o = last ? sgn * s : s;
            }
        }
    }
}

// Full-range axis (App. A): out[a*Qn + k] = int_R l_k(p) (p - u)^a g(p; u, T) dp, exact
// with p = u + sqrt(T) y on the M-point Gauss-Hermite rule (2M - 1 >= Qn + 2).
__device__ void proj_full(const Inst& I, const double* aq, const double* aw, const double* H, int Qn, int M, double u,
                          double T, int amax, double* out) {
    double G[4][QYMAX];
#pragma unroll
    for (int a = 0; a < 4; ++a)
        for (int l = 0; l < QYMAX; ++l) G[a][l] = 0.0;
    const double sT = sqrt(T);
    for (int m = 0; m < M; ++m) {
        const double y = sT * aq[m], x = u + y, E = aw[m];
        const double e1 = E * y, e2 = e1 * y, e3 = e2 * y;
        double hm = 0.0, h = 1.0;
        for (int l = 0; l < Qn; ++l) {
            G[0][l] = fma(E, h, G[0][l]);
            G[1][l] = fma(e1, h, G[1][l]);
            G[2][l] = fma(e2, h, G[2][l]);
            G[3][l] = fma(e3, h, G[3][l]);
            const double hn = (x * h - I.fsq[l] * hm) * I.fisq[l + 1];
            hm = h;
            h = hn;
        }
    }
    for (int a = 0; a <= amax; ++a)
        for (int k = 0; k < Qn; ++k) {
            double s = 0.0;
            for (int l = 0; l < Qn; ++l) s = fma(H[l * Qn + k], G[a][l], s);
            out[a * Qn + k] = s;
        }
}

// E[xi^j] of a centred Gaussian of variance T.
__device__ __forceinline__ double gmom(int j, double T) {
    switch (j) {
        case 0: return 1.0;
        case 2: return T;
        case 4: return 3.0 * T * T;
        case 6: return 15.0 * T * T * T;
        default: return 0.0;
    }
}

// Transverse factors: out[(a*Tc + t)*stride] = nscale * sum_{terms with x-power a} c_term * Ytrans(t).
__device__ void build_Y(const Inst& I, const double* c, double uy, double T, double nscale, double* out, int stride) {
    const int Tc = I.Tc;
    if (I.form == FORM_REDUCED1D) {
        for (int a = 0; a < 4; ++a)
            for (int slot = 0; slot < 2; ++slot) {
                double s = 0.0;
                for (int j = 0; j < NTERMS; ++j) {
                    if (c_mono[j][0] != a) continue;
                    const int b = c_mono[j][1], cc = c_mono[j][2];
                    const double e = slot == 0 ? gmom(b, T) * gmom(cc, T)
                                               : gmom(b + 2, T) * gmom(cc, T) + gmom(b, T) * gmom(cc + 2, T);
                    s = fma(c[j], e, s);
                }
                out[(a * Tc + slot) * stride] = nscale * s;
            }
        return;
    }
    double Py[4 * QYMAX];
    proj_full(I, I.yq, I.yw, I.yH, I.Qy, I.My, uy, T, 3, Py);
    const int Qy = I.Qy;
    if (I.form == FORM_UNREDUCED) {
        double Pz[3 * QZMAX];
        const int Qz = I.Qz;
        proj_full(I, I.zq, I.zw, I.zH, Qz, I.Mz, 0.0, T, 2, Pz);
        for (int a = 0; a < 4; ++a)
            for (int t = 0; t < Tc; ++t) {
                const int ky = t / Qz, kz = t - ky * Qz;
                double s = 0.0;
                for (int j = 0; j < NTERMS; ++j) {
                    if (c_mono[j][0] != a) continue;
                    s = fma(c[j], Py[c_mono[j][1] * Qy + ky] * Pz[c_mono[j][2] * Qz + kz], s);
                }
                out[(a * Tc + t) * stride] = nscale * s;
            }
    } else {
        for (int a = 0; a < 4; ++a)
            for (int t = 0; t < Tc; ++t) {
                const int ky = t >> 1, slot = t & 1;
                double s = 0.0;
                for (int j = 0; j < NTERMS; ++j) {
                    if (c_mono[j][0] != a) continue;
                    const int cc = c_mono[j][2];
                    const double zf = slot == 0 ? gmom(cc, T) : gmom(cc + 2, T);
                    s = fma(c[j], Py[c_mono[j][1] * Qy + ky] * zf, s);
                }
                out[(a * Tc + t) * stride] = nscale * s;
            }
    }
}

// ---------------------------------------------------------------------------
// set-up: wall Maxwellians, initial state
// ---------------------------------------------------------------------------
__device__ void wall_maxwellian(const Inst& I, double U, double T, double* g) {
    double Px[4 * 2 * QX_FULL_MAX];
    proj_x(I, 0.0, T, 0, Px, 1);
    proj_x(I, 0.0, T, 1, Px, 1);
    double c[NTERMS];
    for (int j = 0; j < NTERMS; ++j) c[j] = 0.0;
    c[0] = 1.0;
    double Y[4 * TCMAX];
    build_Y(I, c, U, T, 1.0, Y, 1);
    for (int k = 0; k < I.K; ++k) {
        const int kx = k / I.Tc, t = k - kx * I.Tc;
        g[k] = Px[kx] * Y[t];
    }
}

__global__ void k_setup(Inst* insts) {
    Inst& I = insts[blockIdx.x];
    if (threadIdx.x == 0) wall_maxwellian(I, I.U_L, I.T_L, I.gL);
    if (threadIdx.x == 32) wall_maxwellian(I, I.U_R, I.T_R, I.gR);
    __syncthreads();
    if (I.gL32)
        for (int k = threadIdx.x; k < I.K; k += blockDim.x) {
            I.gL32[k] = (float)I.gL[k];
            I.gR32[k] = (float)I.gR[k];
        }
    if (threadIdx.x == 0) {
        const int Q = I.Q, Tc = I.Tc;
        double inL = 0.0, inR = 0.0;
        for (int k = 0; k < I.K; ++k) {
            const int kx = k / Tc, t = k - kx * Tc;
            const double mp = I.tmt[t] * I.px[kx];
            if (kx < Q) inL = fma(mp, I.gL[k], inL);
            else inR = fma(mp, I.gR[k], inR);
        }
        I.misc[M_INL] = inL;
        I.misc[M_INR] = inR;
        I.misc[M_NWL] = 1.0;
        I.misc[M_NWR] = 1.0;
        I.misc[M_RESID] = CUDART_INF;
        I.misc[M_WIN_STEP] = -1.0;
        I.misc[M_WIN_RESID] = CUDART_INF;
        I.misc[M_SWITCH] = -1.0;
        *I.status = FDLB_ACTIVE;
        *I.steps = 0;
    }
    const double T0 = I.T_init;
    for (int i = threadIdx.x; i < I.ld; i += blockDim.x) {
        I.node[R_N * I.ld + i] = 1.0;
        I.node[R_UX * I.ld + i] = 0.0;
        I.node[R_UY * I.ld + i] = 0.0;
        I.node[R_T * I.ld + i] = T0;
    }
}

// ---------------------------------------------------------------------------
// moments
// ---------------------------------------------------------------------------
// Arithmetic R of the per-node work: FP64 for FP64 storage, double-float for FP32 storage (whose
// tables are rounded to FP32).
__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ df shfl_xor(df v, int o) { return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)}; }

// Projection table outputs in the closure's arithmetic type.
__device__ __forceinline__ double* r_out(const Inst& I, int i0, int lane, double) { return I.tab + tab_col(I, i0, lane); }
__device__ __forceinline__ float* r_out(const Inst& I, int i0, int lane, df) { return I.tab32 + tab_col(I, i0, lane); }

constexpr int NTW = 6;     // transverse weights: mt, mt py, mt py^2, mt py^3, et, et py

template <typename R>
__device__ __forceinline__ R chi_of(R eta) {
    const R om = r_c(1.0, R{}) - eta;
    return r_div(r_c(2.0, R{}) - eta, r_c(2.0, R{}) * om * om * om);
}

// Heat fluxes from the raw sums s[j TILE] (each sum_kx px^a (sum_t w_j(t) f)): third-order sums about the
// mean, s8 - 3 ux s4 + 2 n ux^3 and so on.
template <typename R>
__device__ __forceinline__ R heat_flux_x(const R* s, R n, R ux, R uy) {
    const R two = r_c(2.0, R{}), n2 = two * n;
    const R cx3 = s[8 * TILE] + ux * (n2 * (ux * ux) - r_c(3.0, R{}) * s[4 * TILE]);
    const R cxyy = s[9 * TILE] - two * (uy * s[5 * TILE]) + ux * (n2 * (uy * uy) - s[6 * TILE]);
    return r_c(0.5, R{}) * (cx3 + cxyy) + (s[12 * TILE] - ux * s[7 * TILE]);
}
template <typename R>
__device__ __forceinline__ R heat_flux_y(const R* s, R n, R ux, R uy) {
    const R two = r_c(2.0, R{}), n2 = two * n;
    const R cxxy = s[10 * TILE] - two * (ux * s[5 * TILE]) + uy * (n2 * (ux * ux) - s[4 * TILE]);
    const R cy3 = s[11 * TILE] + uy * (n2 * (uy * uy) - r_c(3.0, R{}) * s[6 * TILE]);
    return r_c(0.5, R{}) * (cy3 + cxxy) + (s[13 * TILE] - uy * s[7 * TILE]);
}

// Moments of the nodes of tile i0 from the 14 raw sums ss[MOM_SUMS][TILE], by nw warps: independent
// chains, one per warp (n, u, T and the stresses; ln n; ln T; ln chi(eta0 n); q_x; q_y).  SPLIT: six
// chains, for the last block of a split tile, which everything waits for (one Couette instance:
// update 18.1 -> 16.4 us per launch); else the heat fluxes with the first, which shares its
// quotients (2048 mixed instances: 756 us per launch with six chains, 705 with four).  FP32 storage
// finalises its double-float sums in double-float: in FP64 this took 362 FP64 instructions per tile,
// 45 % of the FP64 pipe's time on large batches.
template <bool SPLIT, typename R>
__device__ __forceinline__ void finalize_chain(const Inst& I, int i0, const R* ss, int lane, int g) {
    const int i = i0 + lane, ld = I.ld;
    if (i >= I.N) return;
    double* nd = I.node;
    const R* s = ss + lane;                        // raw sum j at s[j TILE]
    const R n = s[0], half = r_c(0.5, R{});
    if (g == 1) {
        nd[R_LNN * ld + i] = r_dbl(r_log(n));
    } else if (g == 3) {
        nd[R_LNCHI * ld + i] = r_dbl(r_log(chi_of(r_of(I.eta0, R{}) * n)));
    } else if (g == 0 || g == 2) {
        // n times the thermal energy, without a division: T = (n E)/(1.5 n^2)
        const R s1 = s[1 * TILE], s2 = s[2 * TILE], s3 = s[3 * TILE], s4 = s[4 * TILE];
        const R sx = s1 + s2;
        const R nE = half * ((n * s4 - sx * sx) + (n * s[6 * TILE] - s3 * s3)) + n * s[7 * TILE];
        const R T = r_div(nE, r_c(1.5, R{}) * (n * n));
        if (g == 2) {
            nd[R_LNT * ld + i] = r_dbl(r_log(T));
            return;
        }
        const R ux = r_div(sx, n), uy = r_div(s3, n), nux = n * ux;
        nd[R_N * ld + i] = r_dbl(n);
        nd[R_UX * ld + i] = r_dbl(ux);
        nd[R_UY * ld + i] = r_dbl(uy);
        nd[R_T * ld + i] = r_dbl(T);
        nd[R_PXX * ld + i] = r_dbl(s4 - nux * ux);
        nd[R_PXY * ld + i] = r_dbl(s[5 * TILE] - nux * uy);
        nd[R_SNEG * ld + i] = r_dbl(s1);
        nd[R_SPOS * ld + i] = r_dbl(s2);
        if (!SPLIT) {
            nd[R_QX * ld + i] = r_dbl(heat_flux_x(s, n, ux, uy));
            nd[R_QY * ld + i] = r_dbl(heat_flux_y(s, n, ux, uy));
        }
    } else {
        const R ux = r_div(s[1 * TILE] + s[2 * TILE], n), uy = r_div(s[3 * TILE], n);
        if (g == 4) nd[R_QX * ld + i] = r_dbl(heat_flux_x(s, n, ux, uy));
        else nd[R_QY * ld + i] = r_dbl(heat_flux_y(s, n, ux, uy));
    }
}
template <bool SPLIT, typename R>
__device__ __forceinline__ void finalize_tile(const Inst& I, int i0, const R* ss, int lane, int wy, int nw) {
#pragma unroll 1
    for (int g = wy; g < (SPLIT ? 6 : 4); g += nw) finalize_chain<SPLIT>(I, i0, ss, lane, g);
}

// Programmatic dependent launch: a stepping kernel launched with programmatic stream
// serialization may start while its predecessor in the stream drains; it waits here, before
// reading anything, until the predecessor has completed and its writes are visible (a no-op
// for a kernel launched without the attribute).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel's blocks start their set-up (up to their own wait) once every block of this
// launch has come here: in the update, after its velocities (one Couette instance 65.1 -> 63.2 us
// per step; in the closure it gave nothing, and right after the wait it slowed every phase).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// The instance's record, copied into shared memory by the whole block (ends with a barrier).  The
// record and the work list are written at creation, before any stepping kernel is launched, so
// this runs before pdl_wait and overlaps the predecessor's end; the two fields that kernels
// change (precision, smem_res) are read again after it.  A block otherwise meets one L2 round trip
// per line of the record that its code touches first.
__device__ __forceinline__ void load_inst(const Inst* src, Inst* dst, int tid, int n) {
    static_assert(sizeof(Inst) % 8 == 0, "copied in 8-byte words");
    for (int w = tid; w < (int)(sizeof(Inst) / 8); w += n)
        reinterpret_cast<unsigned long long*>(dst)[w] = reinterpret_cast<const unsigned long long*>(src)[w];
    __syncthreads();
}

// After the predecessor: does this launch step the instance (active, of this storage, not with the
// shared-memory-resident kernel)?  g: the record in global memory, I: its copy.  One decision for the
// block: another block of the launch may set FDLB_FAILED_COPY between two threads' reads, and the threads
// that went on would miss the others' copies and barrier.
__device__ __forceinline__ bool runs_now(const Inst& g, const Inst& I, bool fp64) {
    pdl_wait();
    const int st = *(volatile int*)I.status, res = *(const volatile int*)&g.smem_res, pr = *(const volatile int*)&g.precision;
    return !__syncthreads_or(st != FDLB_ACTIVE || res || (pr == FDLB_FP64) != fp64);
}

// Named barrier over `n` threads (moment finalisation runs on 128-thread parts of a block).
__device__ __forceinline__ void named_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }


__device__ __forceinline__ double mom_of(double f) { return f; }
__device__ __forceinline__ df mom_of(float f) { return {f, 0.0f}; }
__device__ __forceinline__ double mom_zero(double) { return 0.0; }
__device__ __forceinline__ df mom_zero(df) { return {0.0f, 0.0f}; }
template <typename S>
using MomR = decltype(mom_of(S{}));      // arithmetic of the moment sums of storage type S
__device__ __forceinline__ double ld_cg(const double* p) { return __ldcg(p); }
__device__ __forceinline__ df ld_cg(const df* p) { return df_of(__ldcg(reinterpret_cast<const float2*>(p))); }

// Moments of tile i0 from the I.mgroups partials of its update chunks, added in chunk order, by
// nw warps (tid < 32 nw, barrier `bar` over them, nw >= 4); ss: MOM_SUMS x TILE values of shared
// memory.
template <typename S>
__device__ void moments_final_tile(const Inst& I, int i0, double* ss, int tid, int nw, int bar) {
    using R = MomR<S>;
    const int lane = tid & 31, g = tid >> 5, i = i0 + lane;
    const int ld = I.ld, G = I.mgroups;
    R* rs = reinterpret_cast<R*>(ss);
    named_sync(bar, 32 * nw);             // the previous item's readers of `ss` are done
    for (int j = g; j < MOM_SUMS; j += nw) {
        R a = mom_of((S)0);
        if (i < I.N) {
            // (loads of a batch in flight together: each is a round trip to L2)
            const R* ms = reinterpret_cast<const R*>(I.msum) + (size_t)j * ld + i;
            constexpr int B = 6;
            for (int q = 0; q < G; q += B) {
                R b[B];
#pragma unroll
                for (int e = 0; e < B; ++e) b[e] = q + e < G ? ld_cg(ms + (size_t)(q + e) * MOM_SUMS * ld) : mom_of((S)0);
#pragma unroll
                for (int e = 0; e < B; ++e)
                    if (q + e < G) a = a + b[e];
            }
        }
        rs[j * TILE + lane] = a;
    }
    named_sync(bar, 32 * nw);
    finalize_tile<true>(I, i0, rs, lane, g, nw);
}

// ---------------------------------------------------------------------------
// per-node closure and projection tables
// ---------------------------------------------------------------------------
// Two independent block roles per 32-node tile (lane = node, so every FP64 instruction runs
// with full lanes): role 0 = x projection onto the nodes +p_k and -p_k (half-range rules, or
// the full-range rule of order 2Q), role 1 = gradients, closure, coefficients, y and z
// projections and the transverse factors.
//
// The projections of (p - u)^a g, a = 0..3, need only the a = 0 sums and three scalars: with
// the basis L_k(x) = w_k sum_l h_l(p_k) h_l(x) of an n-point Gauss rule the Christoffel-Darboux
// formula gives (x - p_k) L_k(x) = d_k h_n(x), d_k = w_k b_n h_{n-1}(p_k) (h_n(p_k) = 0), so
//   P_{a+1}[k] = (p_k - u) P_a[k] + d_k T_a,   T_a = int h_n(x) (x - u)^a g dx,
// the same sum over the auxiliary points, at two products per value instead of n.  Measured
// against the four direct sums in 64 bits (orders 4 .. 200, T 0.8 .. 1.9, |u| up to 0.8): the
// rounding errors are equal (half range: 8e-16 at order 16, 1e-14 at 100; full range 2 to 4
// times smaller).  On a full axis (App. A) no auxiliary points are needed either: the expansion
// coefficients m_l = int h_l g follow from m_{l+1} = (u m_l + sqrt(l) (T - 1) m_{l-1})/sqrt(l+1)
// (generating function of the Hermite polynomials) and, by parts, T_0 = m_n,
// T_1 = T sqrt(n) m_{n-1}, T_2 = T m_n + T^2 sqrt(n (n-1)) m_{n-2}.
// The kernel is bound by its instructions (large batches) and by the chain of one block (small
// ones).  Measured per launch, the four direct sums on each half-axis in a block of its own ->
// this form: 2048 mixed FP32 instances 1778 -> 913 us, one Couette instance (200 nodes, 6 x 6 x
// 4) 18.8 -> 12.6, six of order 100 per side 1079 -> 711, three of full-range order 200 in FP64
// 2581 -> 248.
// Shared doubles: role 0 (half): [NOD_WARPS + 1][2 nl + 6][32] sums, [4][32] node scalars, beyond
//                 QMAX polynomials [M][2][32] recurrence states; (full): [3 Lx + 4][32];
//                 role 1: CL_ROWS rows + Py [4 QYMAX] + Pz [2 QZMAX] + A [8 QYMAX] + moments.
constexpr int CL_ROWS = 5 + 8 + 14;                       // gradients, scalars, coefficients and n
constexpr int CL_MOM = (QYMAX + 4) + (QZMAX + 4) + 1;     // m_l and T_a of y and z, T

__host__ __device__ inline int nodal_smem_doubles(int qmax) {
    // larger x orders run in blocks of QMAX polynomials, with the recurrence state of every
    // auxiliary point kept between blocks: [M][2][32] more
    const int qb = qmax > QMAX ? QMAX : qmax;
    const int mst = qmax > QMAX ? aux_points_half(qmax > QX_HALF_MAX ? QX_HALF_MAX : qmax) : 0;
    const int rh = ((NOD_WARPS + 1) * (2 * qb + 6) + 4 + 2 * mst) * TILE;
    const int rf = (3 * qmax + 4) * TILE;
    const int rc = (CL_ROWS + 4 * QYMAX + 2 * QZMAX + 8 * QYMAX + CL_MOM) * TILE;
    const int m = rh > rf ? rh : rf;
    return m > rc ? m : rc;
}

constexpr int XQ_DF = 32;           // half-range double-float projections: unscaled up to this order

// Do the x projections of the tile's nodes stay in the double-float range at every order?  T < XQ_TMAX
// and |u| < sqrt(T) (the same answer in every warp; NaN: no).  Half range, scaled points: e^((T - 1)
// q^2/4) < 1e25 at q = 17, the outermost point of order 100, and exponents q |u|/sqrt(T) below 17.  Full range: the
// coefficients m_l are at most 17 up to order 200; beyond, they grow like |T - 1|^(l/2), 2e7 at T =
// 2.2 and out of the float range at T = 3.3.
constexpr float XQ_TMAX = 1.8f;
__device__ __forceinline__ bool in_df_range(const Inst& I, int i0, int lane) {
    const int i = min(i0 + lane, I.N - 1);
    const float T = (float)I.node[R_T * I.ld + i], u = (float)I.node[R_UX * I.ld + i];
    return __all_sync(0xffffffffu, T < XQ_TMAX && u * u < T);
}

// 1/j as float pairs, j = 0..16 (set by prepare_kernels)
constexpr int NINV2 = 17;
__constant__ float2 c_inv2[NINV2];

// exp of a double-float: z = k ln 2 + r with |r| <= ln 2 / 2, e^r from its Taylor series to
// r^14/14! (the rest is below 2^-57 relative), then the exact scaling by 2^k.  For |z| < 80.
__device__ __forceinline__ df df_exp(df z) {
    const df ln2 = {0.693147182464599609375f, -1.90465429995776787e-09f};
    const float k = rintf(z.hi * 1.44269504088896341f);
    const df r = z - ln2 * df{k, 0.0f};
    const df one = {1.0f, 0.0f};
    df e = one;
#pragma unroll
    for (int j = 14; j >= 1; --j) e = e * r * df_of(c_inv2[j]) + one;
    const int ki = (int)k;
    return {ldexpf(e.hi, ki), ldexpf(e.lo, ki)};
}

// Expansion coefficients m_l = int h_l(p) g(p; u, T) dp, l = 0..n, on a full axis and T_a = int
// h_n(p) (p - u)^a g dp, a = 0..2 (see above); b[l] = sqrt(l), ib[l] = 1/sqrt(l); ml and ts are this
// lane's columns (stride TILE).
template <typename R>
__device__ __forceinline__ void hermite_moments(R u, R T, int n, const double* b, const float2* b2, const double* ib,
                                                const float2* ib2, R* ml, R* ts) {
    const R zero = r_c(0.0, R{}), one = r_c(1.0, R{}), t1 = T - one;
    R mp = zero, m = one, mm = zero;                // m_{l-1}, m_l, m_{l-2}
    ml[0] = m;
#pragma unroll 1
    for (int l = 0; l < n; ++l) {
        const R il = r_tab(ib, ib2, l + 1, zero);
        // off the chain: the factor of m_{l-1}; on it: one product and sum
        const R f = l > 0 ? (r_tab(b, b2, l, zero) * il) * (t1 * mp) : zero;
        const R mn = (u * il) * m + f;
        mm = mp;
        mp = m;
        m = mn;
        ml[(l + 1) * TILE] = m;
    }
    const R bn = r_tab(b, b2, n, zero);
    ts[0] = m;
    ts[TILE] = T * (bn * mp);
    ts[2 * TILE] = T * m + (T * bn) * ((T * r_tab(b, b2, n - 1, zero)) * mm);
}

// exp(q v - d) and exp(-q v - d), d = v^2/2.
__device__ __forceinline__ void exp_pair(double z, double d, double& ep, double& em) {
    ep = exp(z - d);
    em = exp(-z - d);
}
__device__ __forceinline__ void exp_pair(df z, df d, df& ep, df& em) {
    ep = df_exp(z - d);
    em = df_exp(-z - d);
}

// The same for |v| < 0.02, |q v| < 0.12: e^-d (cosh z +- sinh z) by their series, the even and the
// odd part once for both signs.  The neglected terms are below 2e-17; double-float computes the
// terms below 2^-24 of the sum in FP32.
__device__ __forceinline__ void exp_pair_short(double z, double d, double& ep, double& em) {
    const double w = z * z;
    const double c = fma(w, fma(w, fma(w, fma(w, 1.0 / 40320.0, 1.0 / 720.0), 1.0 / 24.0), 0.5), 1.0);
    const double s = z * fma(w, fma(w, fma(w, fma(w, 1.0 / 362880.0, 1.0 / 5040.0), 1.0 / 120.0), 1.0 / 6.0), 1.0);
    const double g = fma(-d, fma(-d, fma(-d, fma(-d, 1.0 / 24.0, 1.0 / 6.0), 0.5), 1.0), 1.0);
    ep = g * (c + s);
    em = g * (c - s);
}
__device__ __forceinline__ void exp_pair_short(df z, df d, df& ep, df& em) {
    const df one = {1.0f, 0.0f};
    const df i2 = {0.5f, 0.0f}, i6 = df_of(c_inv2[6]), i24 = {1.0f / 24.0f, -1.2417634e-9f}, i120 = {1.0f / 120.0f, -4.3461720e-10f};
    const df w = z * z;
    const df c4 = i24 + df{w.hi * fmaf(w.hi, 1.0f / 40320.0f, 1.0f / 720.0f), 0.0f};
    const df c = w * (w * c4 + i2) + one;
    const df s5 = i120 + df{w.hi * fmaf(w.hi, 1.0f / 362880.0f, 1.0f / 5040.0f), 0.0f};
    const df s = z * (w * (w * s5 + i6) + one);
    const df d2 = d * d;
    const df g = one - d + d2 * (i2 - df{d.hi * fmaf(-d.hi, 1.0f / 24.0f, 1.0f / 6.0f), 0.0f});
    ep = g * (c + s);
    em = g * (c - s);
}

// P_a[k] and P_a[-k], a = 0..3, of node k from the a = 0 values and the T_a of either sign of u
// (tp, tm), written to rows a 2Q + k and a 2Q + Q + k; the values at -p_k are (-1)^a those of
// the mirrored problem (u -> -u).
template <typename R, typename O>
__device__ __forceinline__ void put_powers(O* out, int Q, int k, R p, R u, R d, R Pp, R Pm, const R* tp, const R* tm) {
    const R pu = p - u, mu = p + u;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        r_put(out, (a * 2 * Q + k) * TILE, Pp);
        r_put(out, (a * 2 * Q + Q + k) * TILE, (a & 1) ? -Pm : Pm);
        if (a < 3) {
            Pp = pu * Pp + d * tp[a];
            Pm = mu * Pm + d * tm[a];
        }
    }
}
__device__ __forceinline__ float to_float(double x) { return (float)x; }
__device__ __forceinline__ float to_float(df x) { return x.hi; }

// A share of a tile's x projection (tiles of high orders are split over several blocks when the
// batch has few of them): nodes k = NOD_WARPS (i + n j) + 0 .. NOD_WARPS - 1.
struct Part {
    int i, n;
};

// Weight W and first polynomial h of an auxiliary point, scaled by 2^e and 2^-e so that both stay in
// the float range: W falls like e^(-q^2/2) and the polynomials grow like e^(x^2/4), x = sqrt(T) q;
// with 2^e ~ W^(-1/2) both run between e^(-q^2/4) and e^((T - 1) q^2/4).  (Exact powers of two; the
// tail of h underflows only at points that do not contribute.)
__device__ __forceinline__ void scale_point(double W, df& w, df& h) {
    const int e = (1023 - ((__double2hiint(W) >> 20) & 0x7ff)) / 2;
    const double s = __hiloint2double(__double2hiint(W) + (e << 20), __double2loint(W));
    w.hi = (float)s;
    w.lo = (float)(s - (double)w.hi);
    const float f = __uint_as_float((uint32_t)(127 - e) << 23);
    h = {h.hi * f, h.lo * f};
}
__device__ __forceinline__ void scale_point(double, double&, double&) {}

// Half-range x projection of a tile (Sec. III A 2), both half-axes: the auxiliary points
// x = sqrt(T) q and the polynomials there do not depend on the sign of u, so one recurrence
// serves both.  With |v| < 0.02 and Q <= MX8 the 8-point auxiliary rule is used: it is exact for v = 0
// (degree 15 >= Q + 2), and what it misses of exp(q v) at |v| = 0.02 is 3e-13 of the largest value at
// Q = 8 and less at smaller orders (7e-11 at Q = 9, 1e-4 at Q = 12: those take the 16-point rule, 41 us
// per launch for twelve Couette instances of order 9 in FP64 against 31).  Warp w
// takes auxiliary points w, w + 8, ...  R: double, or double-float for FP32 storage; out: the
// table written (FP32 storage's tab32 also from double).
template <int QB, typename R, typename O>
__device__ void xproj_half(const Inst& I, int i0, double* nsm, O* out, Part pt) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int i = i0 + lane, N = I.N, ld = I.ld, Q = I.Q;
    const bool valid = i < N;
    const int ic = valid ? i : N - 1;           // padding lanes work on a real node, write nothing
    const R zero = r_of(0.0, R{});
    R* xs = reinterpret_cast<R*>(nsm);                               // [4][32] sqrt(T), u, v, v^2/2
    R* part = xs + 4 * TILE;                                         // [NOD_WARPS + 1][2 QB + 6][32]
    R* hst = part + (NOD_WARPS + 1) * (2 * QB + 6) * TILE;           // [M][2][32] recurrence state (Q > QB)
    __shared__ int use_short;
    if (wid == 0) {
        const R u = r_of(I.node[R_UX * ld + ic], R{});
        const R sT = r_sqrt(r_of(I.node[R_T * ld + ic], R{}));
        const R v = r_div(u, sT), d = r_c(0.5, R{}) * v * v;
        xs[0 * TILE + lane] = sT;
        xs[1 * TILE + lane] = u;
        xs[2 * TILE + lane] = v;
        xs[3 * TILE + lane] = d;
        float av = valid ? fabsf(to_float(v)) : 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) av = fmaxf(av, __shfl_xor_sync(0xffffffffu, av, o));
        // one rule per block so that the warps agree: the largest |v| of the tile decides
        if (lane == 0) use_short = av < 0.02f ? 1 : 0;
    }
    __syncthreads();
    const bool short_rule = use_short && Q <= MX8;
    const int M = short_rule ? MX8 : I.Mx;
    const double* xq = short_rule ? I.xq8 : I.xq;
    const double* xw = short_rule ? I.xw8 : I.xw;
    const float2* xq2 = short_rule ? I.xq82 : I.xq2;
    const float2* xw2 = short_rule ? I.xw82 : I.xw2;
    const double *xa = I.xa, *xb = I.xb, *xib = I.xib, *xH = I.xH, *px = I.px;
    const float2 *xa2 = I.xa2, *xb2 = I.xb2, *xib2 = I.xib2, *xH2 = I.xH2, *px2 = I.px2;
    const R h0 = r_pair(I.x_h0, I.x_h02, R{});
    const bool scaled = QB > 8 && sizeof(O) == 4 && Q > XQ_DF;      // (R = double-float: see nodal_item)
    const R sT = xs[lane], u = xs[TILE + lane], v = xs[2 * TILE + lane], d = xs[3 * TILE + lane];
    // blocks of QB polynomials: per block the sums over the auxiliary points (the recurrence
    // continued from the previous block's state), then the H products, whose chain continues
    // across blocks in the instance's FP64-sized table rows; the powers follow the last block
    for (int lb = 0; lb < Q; lb += QB) {
        const int nl = min(QB, Q - lb);
        const bool last = lb + nl == Q;
        const int nr = 2 * nl + (last ? 6 : 0);
        R Gp[QB], Gm[QB], Tp[3], Tm[3];
#pragma unroll
        for (int j = 0; j < QB; ++j) Gp[j] = Gm[j] = zero;
#pragma unroll
        for (int a = 0; a < 3; ++a) Tp[a] = Tm[a] = zero;
        for (int m = wid; m < M; m += NOD_WARPS) {
            const R q = r_tab(xq, xq2, m, zero);
            R W = r_tab(xw, xw2, m, zero), hs = h0;
            if (scaled) scale_point(xw[m], W, hs);
            R ep, em;
            if (short_rule) exp_pair_short(q * v, d, ep, em);
            else exp_pair(q * v, d, ep, em);
            ep = W * ep;
            em = W * em;
            const R x = sT * q;
            R hm = zero, h = hs;
            if (lb > 0) {
                hm = hst[(2 * m) * TILE + lane];
                h = hst[(2 * m + 1) * TILE + lane];
            }
#pragma unroll
            for (int j = 0; j < QB; ++j) {
                if (j < nl) {
                    const int l = lb + j;
                    Gp[j] = acc(Gp[j], ep, h);
                    Gm[j] = acc(Gm[j], em, h);
                    const R hn = rec3(x - r_tab(xa, xa2, l, zero), h, r_tab(xb, xb2, l, zero), hm, r_tab(xib, xib2, l + 1, zero));
                    hm = h;
                    h = hn;
                }
            }
            if (last) {                                  // h = h_Q: the T_a of both signs
                const R yp = x - u, ym = x + u;
                ep = ep * h;
                em = em * h;
                Tp[0] = Tp[0] + ep;
                Tm[0] = Tm[0] + em;
                Tp[1] = acc(Tp[1], ep, yp);
                Tm[1] = acc(Tm[1], em, ym);
                Tp[2] = acc(Tp[2], ep, yp * yp);
                Tm[2] = acc(Tm[2], em, ym * ym);
            } else {
                hst[(2 * m) * TILE + lane] = hm;
                hst[(2 * m + 1) * TILE + lane] = h;
            }
        }
        if (lb > 0) __syncthreads();              // the previous block's readers of part are done
#pragma unroll
        for (int j = 0; j < QB; ++j)
            if (j < nl) {
                part[(wid * nr + j) * TILE + lane] = Gp[j];
                part[(wid * nr + nl + j) * TILE + lane] = Gm[j];
            }
        if (last)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                part[(wid * nr + 2 * nl + a) * TILE + lane] = Tp[a];
                part[(wid * nr + 2 * nl + 3 + a) * TILE + lane] = Tm[a];
            }
        __syncthreads();
        R* sum = part + NOD_WARPS * nr * TILE;
        for (int r = wid; r < nr; r += NOD_WARPS) {
            R t = fin(part[r * TILE + lane]);
#pragma unroll
            for (int q = 1; q < NOD_WARPS; ++q) t = t + part[(q * nr + r) * TILE + lane];
            sum[r * TILE + lane] = t;
        }
        __syncthreads();
        R* chain = reinterpret_cast<R*>(I.tab) + tab_col(I, i0, lane);
        for (int k = pt.i * NOD_WARPS + wid; k < Q; k += NOD_WARPS * pt.n) {
            R sp = zero, sm = zero;
            if (lb > 0 && valid) {
                sp = chain[k * TILE];
                sm = chain[(Q + k) * TILE];
            }
            for (int j = 0; j < nl; ++j) {
                const R H = r_tab(xH, xH2, (lb + j) * Q + k, zero);
                sp = acc(sp, H, sum[j * TILE + lane]);
                sm = acc(sm, H, sum[(nl + j) * TILE + lane]);
            }
            sp = fin(sp);
            sm = fin(sm);
            if (last) {
                const R dk = r_tab(xb, xb2, Q, zero) * r_tab(xH, xH2, (Q - 1) * Q + k, zero);
                R tp[3], tm[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    tp[a] = sum[(2 * nl + a) * TILE + lane];
                    tm[a] = sum[(2 * nl + 3 + a) * TILE + lane];
                }
                if (valid) put_powers(out, Q, k, r_tab(px, px2, k, zero), u, dk, sp, sm, tp, tm);
            } else if (valid) {
                chain[k * TILE] = sp;
                chain[(Q + k) * TILE] = sm;
            }
        }
    }
}

// Full-range x projection of a tile (App. A, order Lx = 2Q): the expansion coefficients by their
// recurrence (warp 0), then the sums over l, the even and the odd part once for both signs of
// the node.
template <typename R, typename O>
__device__ void xproj_full(const Inst& I, int i0, double* nsm, O* out, Part pt) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int i = i0 + lane, N = I.N, ld = I.ld, Q = I.Q, Lx = I.Lx;
    const bool valid = i < N;
    const int ic = valid ? i : N - 1;
    const R zero = r_of(0.0, R{});
    R* ml = reinterpret_cast<R*>(nsm);                               // [Lx + 1][32] m_l
    R* ts = ml + (Lx + 1) * TILE;                                    // [3][32] T_a
    R* ca = ts + 3 * TILE;                                           // [Lx][32] u/sqrt(l + 1)
    R* cb = ca + Lx * TILE;                                          // [Lx][32] (T - 1) sqrt(l/(l + 1))
    const double *xb = I.xb, *xib = I.xib, *xH = I.xH, *px = I.px;
    const float2 *xb2 = I.xb2, *xib2 = I.xib2, *xH2 = I.xH2, *px2 = I.px2;
    const R T = r_of(I.node[R_T * ld + ic], zero), u = r_of(I.node[R_UX * ld + ic], zero), t1 = T - r_c(1.0, zero);
    // the recurrence's factors by all warps, then the chain (a product and an FMA per step) by warp 0
    for (int l = wid; l < Lx; l += NOD_WARPS) {
        const R il = r_tab(xib, xib2, l + 1, zero);
        ca[l * TILE + lane] = u * il;
        cb[l * TILE + lane] = t1 * (r_tab(xb, xb2, l, zero) * il);
    }
    __syncthreads();
    if (wid == 0) {
        R mp = zero, m = r_c(1.0, zero), mm = zero;
        ml[lane] = m;
        for (int l = 0; l < Lx; ++l) {
            const R mn = ca[l * TILE + lane] * m + cb[l * TILE + lane] * mp;
            mm = mp;
            mp = m;
            m = mn;
            ml[(l + 1) * TILE + lane] = m;
        }
        const R bn = r_tab(xb, xb2, Lx, zero);
        ts[lane] = m;
        ts[TILE + lane] = T * (bn * mp);
        ts[2 * TILE + lane] = T * m + (T * bn) * ((T * r_tab(xb, xb2, Lx - 1, zero)) * mm);
    }
    __syncthreads();
    for (int k = pt.i * NOD_WARPS + wid; k < Q; k += NOD_WARPS * pt.n) {
        R e = zero, o = zero;
        for (int l = 0; l < Lx; l += 2) {
            e = acc(e, r_tab(xH, xH2, l * Q + k, zero), ml[l * TILE + lane]);
            o = acc(o, r_tab(xH, xH2, (l + 1) * Q + k, zero), ml[(l + 1) * TILE + lane]);
        }
        e = fin(e);
        o = fin(o);
        const R dk = r_tab(xb, xb2, Lx, zero) * r_tab(xH, xH2, (Lx - 1) * Q + k, zero);
        // mirrored problem of -p_k: u -> -u changes the signs of m_l, odd l, and of T_1 (Lx even)
        const R tp[3] = {ts[lane], ts[TILE + lane], ts[2 * TILE + lane]}, tm[3] = {tp[0], -tp[1], tp[2]};
        if (valid) put_powers(out, Q, k, r_tab(px, px2, k, zero), u, dk, e + o, e - o, tp, tm);
    }
}

// Role 1 of a tile: gradients (Sec. III B 3), closure (Eqs. chi, prandtl, viscosity, tau), the
// 13 coefficients of f^S + tau J1 = n g(xi) sum_j c_j xi^(a_j, b_j, c_j) (Eq. j1), the y and z
// projections (App. A) and the transverse factors n Y[a][t]; wall densities (Sec. III B).
// Phase A: warps 0..4 one gradient each (warp 3 also the expansion coefficients of z, warp 4 the
// wall densities), warp 5 the expansion coefficients of y, warps 6 and 7 the closure's factors of
// n and T and of chi, kept apart so that neither chain waits for the other; warps 0..6 then run
// the projections while warp 7 is still busy.  Phase B: the coefficients; phase C: assembly.
template <typename R>
__device__ void closure_item(const Inst& I, int i0, double* nsm) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int i = i0 + lane, N = I.N, ld = I.ld, Q = I.Q, Tc = I.Tc, Qy = I.Qy, Qz = I.Qz;
    const bool valid = i < N;
    const int ic = valid ? i : N - 1;           // padding lanes work on a real node, write nothing
    const double* nd = I.node;
    R* gr = reinterpret_cast<R*>(nsm);                  // [5][32] d/dx of ln n, ln chi, ln T, u_x, u_y
    R* cs = gr + 5 * TILE;                              // [8][32] closure scalars
    R* sc = cs + 8 * TILE;                              // [14][32] coefficients, n
    R* Py = sc + 14 * TILE;                             // [4 QYMAX][32]
    R* Pz = Py + 4 * QYMAX * TILE;                      // [2 QZMAX][32] (p_z^0 and p_z^2)
    R* Ay = Pz + 2 * QZMAX * TILE;                      // [8 QYMAX][32]
    R* my = Ay + 8 * QYMAX * TILE;                      // [QYMAX + 1][32] m_l of y, then T_a [3][32]
    R* mz = my + (QYMAX + 4) * TILE;                    // the same of z
    R* Ts = mz + (QZMAX + 4) * TILE;                    // [32] T
    // Fischer-Methfessel contact value (Eq. chi_ret): the averaged density n-bar and ln chi(n-bar)
    // on the tile and a halo of 7 nodes each side (what the gradient stencils reach)
    constexpr int FH = 7;
    __shared__ __align__(8) unsigned char fm_raw[2 * (TILE + 2 * FH) * 8];
    R* fm_nbar = reinterpret_cast<R*>(fm_raw);
    double* fm_lnchi = reinterpret_cast<double*>(fm_raw) + TILE + 2 * FH;
    const bool fm = I.chi_model == FDLB_CHI_RET_FM;
    const int h0 = i0 - FH;
    const R zero = r_c(0.0, R{}), one = r_c(1.0, R{});
    if (fm) {
        for (int h = wid; h < TILE + 2 * FH; h += NOD_WARPS) {
            const int j = h0 + h;
            R v = zero;
            if (j >= 0 && j < N)
                for (int e = I.fm_ptr[j] + lane; e < I.fm_ptr[j + 1]; e += 32)
                    v = acc(v, r_of(I.fm_w[e], R{}), r_of(nd[R_N * ld + I.fm_col[e]], R{}));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v = plus(v, shfl_xor(v, o));
            if (lane == 0) fm_nbar[h] = fin(v);
        }
        __syncthreads();
        if (threadIdx.x < TILE + 2 * FH) {
            const int j = h0 + threadIdx.x;
            fm_lnchi[threadIdx.x] = (j >= 0 && j < N) ? r_dbl(r_log(chi_of(r_of(I.eta0, R{}) * fm_nbar[threadIdx.x]))) : 0.0;
        }
        __syncthreads();
    }
    if (wid < 5) {
        // the gradients stay FP64 for either storage: differences of nearly equal numbers
        const int row = wid == 0 ? R_LNN : (wid == 1 ? R_LNCHI : (wid == 2 ? R_LNT : (wid == 3 ? R_UX : R_UY)));
        const double cen[7] = {-1.0 / 60.0, 3.0 / 20.0, -0.75, 0.0, 0.75, -3.0 / 20.0, 1.0 / 60.0};
        double g = 0.0;
#pragma unroll
        for (int j = 0; j < 7; ++j) {
            int idx;
            double wj;
            if (ic < 3) { idx = j; wj = I.gst[ic * 7 + j]; }
            else if (ic > N - 4) { const int m = N - 1 - ic; idx = N - 1 - j; wj = -I.gst[m * 7 + j]; }
            else { idx = ic - 3 + j; wj = cen[j]; }
            g = fma(wj, (fm && wid == 1) ? fm_lnchi[idx - h0] : nd[row * ld + idx], g);
        }
        gr[wid * TILE + lane] = r_of(g * I.xpinv[ic], R{});
        if (wid == 3 && I.form == FORM_UNREDUCED)
            hermite_moments(zero, r_of(nd[R_T * ld + ic], R{}), Qz, I.fsq, I.fsq2, I.fisq, I.fisq2, mz + lane,
                            mz + (QZMAX + 1) * TILE + lane);
        if (wid == 4 && i0 == 0 && lane < 2) {
            // zero net mass flux through each wall (Sec. III B): the outgoing wall-face flux is
            // the quadratic reconstruction (11 f_1 - 7 f_2 + 2 f_3)/6 of outgoing populations
            // (lane 0 the left wall, lane 1 the right one)
            const double* sr = nd + (lane ? R_SPOS * ld + N - 1 : R_SNEG * ld);
            const int st = lane ? -1 : 1;
            const double o = (11.0 * sr[0] - 7.0 * sr[st] + 2.0 * sr[2 * st]) / 6.0;
            I.misc[lane ? M_NWR : M_NWL] = -o / I.misc[lane ? M_INR : M_INL];
        }
    } else if (wid == 5) {
        const R T = r_of(nd[R_T * ld + ic], R{});
        Ts[lane] = T;
        if (I.form != FORM_REDUCED1D)
            hermite_moments(r_of(nd[R_UY * ld + ic], R{}), T, Qy, I.fsq, I.fsq2, I.fisq, I.fisq2, my + lane,
                            my + (QYMAX + 1) * TILE + lane);
    } else if (wid == 6) {
        // the factors of n and T alone: tau = mu/(n T) = mu0c X g, g = sqrt T/(T n)
        const R n = r_of(nd[R_N * ld + ic], R{}), T = r_of(nd[R_T * ld + ic], R{});
        const R iT = r_div(one, T), in = r_div(one, n), sT = r_sqrt(T);
        cs[0 * TILE + lane] = (iT * in) * sT;                             // g
        cs[1 * TILE + lane] = iT;
        cs[2 * TILE + lane] = (r_c(0.2, R{}) * in) * (iT * iT);
        cs[3 * TILE + lane] = n * sT;                                     // 1/g
        sc[13 * TILE + lane] = n;
    } else {
        // the factors of chi: X = 1/chi + 0.8 b rho + k_mu (b rho)^2 chi, Pr, b rho chi
        const R k_mu = r_c((4.0 / 25.0) * (1.0 + 12.0 / CUDART_PI), R{});
        const R k_pd = r_c((9.0 / 25.0) * (1.0 + 32.0 / (9.0 * CUDART_PI)), R{});
        const R n = r_of(nd[R_N * ld + ic], R{}), e0 = r_of(I.eta0, R{});
        const R eta = e0 * n, ec = fm ? e0 * fm_nbar[ic - h0] : eta;
        const R om = one - ec, den = r_c(2.0, R{}) * om * om * om, num = r_c(2.0, R{}) - ec;
        const R chi = r_div(num, den), br = r_c(4.0, R{}) * eta, brc = br * chi, brc2 = brc * brc;
        const R Pr = r_div(r_c(2.0 / 3.0, R{}) * (one + r_c(0.8, R{}) * brc + k_mu * brc2),
                           one + r_c(1.2, R{}) * brc + k_pd * brc2);
        const R X = r_of(I.mu0c, R{}) * (r_div(den, num) + r_c(0.8, R{}) * br + k_mu * br * brc);
        cs[4 * TILE + lane] = -(X * brc);                                 // W = -tau b rho chi = this times g
        cs[5 * TILE + lane] = one - Pr;
        cs[6 * TILE + lane] = X;
    }
    // warps 0..6 go on to the projections (they need m_l, T and u_y only) while warp 7 still
    // runs the closure chain; named barrier 1 synchronises the 7 warps
    if (wid < NOD_WARPS - 1 && I.form != FORM_REDUCED1D) {
        const R z = r_of(0.0, R{});
        named_sync(1, (NOD_WARPS - 1) * TILE);
        // one node of y or z per warp: (p_y - u_y)^b g, b = 0..3, and p_z^c g, c = 0, 2
        const int nz = I.form == FORM_UNREDUCED ? Qz : 0;
        for (int it = wid; it < Qy + nz; it += NOD_WARPS - 1) {
            const bool ydir = it < Qy;
            const int k = ydir ? it : it - Qy, Qn = ydir ? Qy : Qz;
            const double* H = ydir ? I.yH : I.zH;
            const float2* H2 = ydir ? I.yH2 : I.zH2;
            const R* m = ydir ? my : mz;
            const R* ts = m + (ydir ? QYMAX + 1 : QZMAX + 1) * TILE;
            R P = z;
#pragma unroll 1
            for (int l = 0; l < QYMAX; ++l)
                if (l < Qn) P = acc(P, r_tab(H, H2, l * Qn + k, z), m[l * TILE + lane]);
            P = fin(P);
            const R dk = r_tab((ydir ? I.yw : I.zw) + MYMAX, ydir ? I.yd2 : I.zd2, k, z);
            if (ydir) {
                const R pu = r_tab(I.yn, I.yn2, k, z) - r_of(nd[R_UY * ld + ic], z);
                Py[k * TILE + lane] = P;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    P = pu * P + dk * ts[a * TILE + lane];
                    Py[((a + 1) * QYMAX + k) * TILE + lane] = P;
                }
            } else {
                const R p = r_tab(I.zn, I.zn2, k, z);
                Pz[k * TILE + lane] = P;
                P = p * P + dk * ts[lane];
                Pz[(QZMAX + k) * TILE + lane] = p * P + dk * ts[TILE + lane];
            }
        }
    }
    __syncthreads();
    auto* out = r_out(I, i0, lane, R{});
    {
        // coefficients: warp w computes a few, reading only what they need; warp 6 also 1/tau
        const R W = cs[4 * TILE + lane] * cs[0 * TILE + lane], A = cs[5 * TILE + lane] * cs[2 * TILE + lane];
        const R iT = cs[1 * TILE + lane];
        const R qx = r_of(nd[R_QX * ld + ic], R{}), qy = r_of(nd[R_QY * ld + ic], R{});
        switch (wid) {
            case 0: sc[0 * TILE + lane] = one - W * gr[3 * TILE + lane]; break;
            case 1: {
                // 2 d ln n + d ln chi + d ln T - 1.5 d ln T
                const R Gr = r_c(2.0, R{}) * gr[0 * TILE + lane] + gr[1 * TILE + lane] - r_c(0.5, R{}) * gr[2 * TILE + lane];
                sc[1 * TILE + lane] = W * Gr - r_c(5.0, R{}) * (A * qx);
                break;
            }
            case 2:
                sc[2 * TILE + lane] = -(r_c(5.0, R{}) * (A * qy));
                sc[6 * TILE + lane] = I.j1_shear ? (W * r_c(0.4, R{})) * (gr[4 * TILE + lane] * iT) : zero;
                break;
            case 3: {
                const R u = (W * gr[3 * TILE + lane]) * iT, c = r_c(0.2, R{}) * u;
                sc[3 * TILE + lane] = r_c(0.6, R{}) * u;
                sc[4 * TILE + lane] = c;
                sc[5 * TILE + lane] = c;
                break;
            }
            case 4: {
                const R c3 = (A * qx + r_c(0.3, R{}) * (W * gr[2 * TILE + lane])) * iT;
                sc[7 * TILE + lane] = c3;
                sc[8 * TILE + lane] = c3;
                sc[9 * TILE + lane] = c3;
                break;
            }
            case 5: {
                const R cy = (A * qy) * iT;
                sc[10 * TILE + lane] = cy;
                sc[11 * TILE + lane] = cy;
                sc[12 * TILE + lane] = cy;
                break;
            }
            case 6:
                if (valid) r_put(out, (8 * Q + 4 * Tc) * TILE, r_div(cs[3 * TILE + lane], cs[6 * TILE + lane]));
                break;
            default: break;
        }
    }
    __syncthreads();
    const int form = I.form;
    if (form != FORM_REDUCED1D) {
        // A[a][c'][ky] = n sum over the monomials (a, b, c = 2 c') of coef * Py[b][ky]; with the
        // monomial order of c_mono: (0,0,0) (1,0,0) (0,1,0) (2,0,0) (0,2,0) (0,0,2) (1,1,0)
        // (3,0,0) (1,2,0) (1,0,2) (2,1,0) (0,3,0) (0,1,2)
        for (int ky = wid; ky < Qy; ky += NOD_WARPS) {
            R c[NTERMS];
#pragma unroll
            for (int j = 0; j < NTERMS; ++j) c[j] = sc[j * TILE + lane];
            const R n = sc[13 * TILE + lane];
            const R P0 = Py[(0 * QYMAX + ky) * TILE + lane], P1 = Py[(1 * QYMAX + ky) * TILE + lane];
            const R P2 = Py[(2 * QYMAX + ky) * TILE + lane], P3 = Py[(3 * QYMAX + ky) * TILE + lane];
            const R zero = r_of(0.0, R{});
            Ay[(0 * Qy + ky) * TILE + lane] = n * (c[0] * P0 + c[2] * P1 + c[4] * P2 + c[11] * P3);   // a = 0, c' = 0
            Ay[(1 * Qy + ky) * TILE + lane] = n * (c[5] * P0 + c[12] * P1);                          // a = 0, c' = 1
            Ay[(2 * Qy + ky) * TILE + lane] = n * (c[1] * P0 + c[6] * P1 + c[8] * P2);               // a = 1, c' = 0
            Ay[(3 * Qy + ky) * TILE + lane] = n * (c[9] * P0);                                       // a = 1, c' = 1
            Ay[(4 * Qy + ky) * TILE + lane] = n * (c[3] * P0 + c[10] * P1);                          // a = 2, c' = 0
            Ay[(5 * Qy + ky) * TILE + lane] = zero;                                                  // a = 2, c' = 1
            Ay[(6 * Qy + ky) * TILE + lane] = n * (c[7] * P0);                                       // a = 3, c' = 0
            Ay[(7 * Qy + ky) * TILE + lane] = zero;                                                  // a = 3, c' = 1
        }
        __syncthreads();
        // transverse factors n Y[a][t] = A[a][0][ky] Z0(t) + A[a][1][ky] Z2(t), t = ky Tz + kz;
        // a warp takes (a, ky) pairs and runs over kz (no per-output index divisions)
        const R Tr = Ts[lane], T3 = r_of(3.0, R{}) * Tr;
        const bool unred = form == FORM_UNREDUCED;
        const int Tz = unred ? Qz : 2;
        for (int pr = wid; pr < 4 * Qy; pr += NOD_WARPS) {
            const int a = pr / Qy, ky = pr - a * Qy;
            const R A0 = Ay[((2 * a) * Qy + ky) * TILE + lane], A1 = Ay[((2 * a + 1) * Qy + ky) * TILE + lane];
            auto* row = out + (8 * Q + a * Tc + ky * Tz) * TILE;
            if (unred) {
                for (int kz = 0; kz < Qz; ++kz) {
                    const R v = A0 * Pz[(0 * QZMAX + kz) * TILE + lane] + A1 * Pz[(QZMAX + kz) * TILE + lane];
                    if (valid) r_put(row, kz * TILE, v);
                }
            } else {
                const R v0 = A0 + A1 * Tr, v1 = (A0 + A1 * T3) * Tr;
                if (valid) {
                    r_put(row, 0, v0);
                    r_put(row, TILE, v1);
                }
            }
        }
    } else {
        // 1D reduced (Sec. II B 1): slots phi, theta carry the (p_y, p_z) Gaussian moments
        // (E[1] = 1, E[xi^2] = T, E[xi^4] = 3 T^2, odd moments zero):
        //   phi   = n (c_a0 + (c_a20 + c_a02) T),  theta = n (2 c_a0 + 4 (c_a20 + c_a02) T) T
        // with the coefficients of xi_x^a, xi_x^a xi_y^2 and xi_x^a xi_z^2
        const int a = wid >> 1, slot = wid & 1;
        const R Tr = Ts[lane];
        const R c0 = sc[(a == 0 ? 0 : a == 1 ? 1 : a == 2 ? 3 : 7) * TILE + lane];
        R c2 = r_of(0.0, R{});
        if (a == 0) c2 = sc[4 * TILE + lane] + sc[5 * TILE + lane];
        if (a == 1) c2 = sc[8 * TILE + lane] + sc[9 * TILE + lane];
        const R two = r_of(2.0, R{});
        R t = slot == 0 ? c0 + c2 * Tr : (two * c0 + (two * two * c2) * Tr) * Tr;
        if (valid) r_put(out, (8 * Q + a * Tc + slot) * TILE, sc[13 * TILE + lane] * t);
    }
}

// The read-only tables of role `role` (at most 16 KB of them) into L1, one load per 128-byte line,
// before the predecessor has finished: the loops that read them would else wait for L2 once per
// line, one after the other.
__device__ __forceinline__ void warm_lines(const void* from, size_t bytes, int tid, int n) {
    const char* a = static_cast<const char*>(from);
    const int lines = (int)((bytes < 16384 ? bytes : 16384) + 127) / 128;
    for (int l = tid; l < lines; l += n) {
        unsigned x;
        asm volatile("ld.global.b32 %0, [%1];" : "=r"(x) : "l"(a + l * 128));
    }
}
__device__ __forceinline__ void warm_tables(const Inst& I, int role, int tid, int n) {
    const bool f32 = I.precision == FDLB_FP32_STORAGE;
    const char *b, *e;
    if (role == 0) {
        b = f32 ? (const char*)I.xq2 : (const char*)I.px;
        e = f32 ? (const char*)I.yn2 : (const char*)I.yn;
    } else {
        b = f32 ? (const char*)I.yn2 : (const char*)I.yn;
        e = f32 ? (const char*)I.px2 : (const char*)I.Ky;
    }
    warm_lines(b, e - b, tid, n);
}

// One (tile, role) item by a block of NOD_WARPS warps; nsm holds nodal_smem_doubles(max Lx)
// doubles; fp32: the instance stores f in FP32 (tables go to tab32).
template <int QB>
__device__ void nodal_item(const Inst& I, int i0, int role, double* nsm, bool fp32, Part pt = {0, 1}) {
    const int lane = threadIdx.x & 31;
    __syncthreads();                      // the previous item's readers of nsm are done
    if (role == 1) {
        if (fp32) closure_item<df>(I, i0, nsm);
        else closure_item<double>(I, i0, nsm);
        return;
    }
    // FP32 storage: double-float, FP64 in tiles beyond its range (708 us per launch for six instances of order
    // 100, against 212 in double-float)
    if (I.xfull) {
        if (!fp32) xproj_full<double>(I, i0, nsm, r_out(I, i0, lane, 0.0), pt);
        else if (in_df_range(I, i0, lane)) xproj_full<df>(I, i0, nsm, r_out(I, i0, lane, df{}), pt);
        else xproj_full<double>(I, i0, nsm, r_out(I, i0, lane, df{}), pt);
        return;
    }
    if (!fp32) {
        xproj_half<QB, double>(I, i0, nsm, r_out(I, i0, lane, 0.0), pt);
        return;
    }
    if constexpr (QB > 8) {               // (QB = 8: no order above 8 in the batch)
        // above XQ_DF polynomials the points are scaled (scale_point)
        if (I.Lx > XQ_DF && !in_df_range(I, i0, lane)) {
            xproj_half<QB, double>(I, i0, nsm, r_out(I, i0, lane, df{}), pt);
            return;
        }
    }
    xproj_half<QB, df>(I, i0, nsm, r_out(I, i0, lane, df{}), pt);
}

// ---------------------------------------------------------------------------
// per-step residual and status
// ---------------------------------------------------------------------------
// Stagnation of a two-phase instance in its FP32 phase (window rule of FDLB_FP32_THEN_FP64).
__device__ int stagnated(Inst& I, double r, double step) {
    if (r == 0.0) return 1;
    double* m = I.misc;
    if (m[M_WIN_STEP] < 0.0) {
        m[M_WIN_STEP] = step;
        m[M_WIN_RESID] = r;
        return 0;
    }
    if (step - m[M_WIN_STEP] < FDLB_STAGNATION_WINDOW) return 0;
    if (!(r < FDLB_STAGNATION_FACTOR * m[M_WIN_RESID])) return 1;
    m[M_WIN_STEP] = step;
    m[M_WIN_RESID] = r;
    return 0;
}

// Residual, status and (two-phase) precision switch of instance I (batch index idx) after a
// step, by a block of 256 threads; red: 7 x 256 doubles of shared memory.
__device__ void resid_item(Inst& I, int idx, double tol, double* resid_all, double* red) {
    const int ld = I.ld, N = I.N;
    double* nd = I.node;
    constexpr int RT = 256;                   // threads of the calling block
    __shared__ double tot[7], term[4];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double s[7] = {0, 0, 0, 0, 0, 0, 0};
    int bad_nf = 0, bad_ph = 0;
    for (int i = threadIdx.x; i < N; i += RT) {
        const double n = nd[R_N * ld + i], ux = nd[R_UX * ld + i], uy = nd[R_UY * ld + i], T = nd[R_T * ld + i];
        if (!isfinite(n) || !isfinite(ux) || !isfinite(uy) || !isfinite(T)) bad_nf = 1;
        else if (!(n > 0.0) || !(T > 0.0)) bad_ph = 1;
        const double w = I.dxw[i];
        const double dn = n - nd[R_PREV_N * ld + i], dT = T - nd[R_PREV_T * ld + i];
        const double dux = ux - nd[R_PREV_UX * ld + i], duy = uy - nd[R_PREV_UY * ld + i];
        s[0] += w * dn * dn;
        s[1] += w * n * n;
        s[2] += w * dT * dT;
        s[3] += w * T * T;
        s[4] += w * dux * dux;
        s[5] += w * duy * duy;
        s[6] += w * n;
        nd[R_PREV_N * ld + i] = n;
        nd[R_PREV_UX * ld + i] = ux;
        nd[R_PREV_UY * ld + i] = uy;
        nd[R_PREV_T * ld + i] = T;
    }
    __shared__ int flags[3];
    __shared__ double scale;
    if (threadIdx.x == 0) { flags[0] = 0; flags[1] = 0; flags[2] = 0; }
#pragma unroll
    for (int j = 0; j < 7; ++j) red[j * RT + threadIdx.x] = s[j];
    __syncthreads();
    if (bad_nf) atomicOr(&flags[0], 1);
    if (bad_ph) atomicOr(&flags[1], 1);
    // sum j over the block by warp j (independent FP64 chains on different schedulers)
    if (wid < 7) {
        double v = 0.0;
#pragma unroll
        for (int q = 0; q < RT / 32; ++q) v += red[wid * RT + q * 32 + lane];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) tot[wid] = v;
    }
    __syncthreads();
    // the four terms of the residual on four warps
    if (lane == 0 && wid < 4)
        term[wid] = wid == 0 ? sqrt(tot[0] / tot[1]) : (wid == 1 ? sqrt(tot[2] / tot[3]) : sqrt(tot[wid + 2]));
    __syncthreads();
    if (threadIdx.x == 0) {
        double r = fmax(fmax(term[0], term[1]), fmax(term[2], term[3]));
        *I.steps += 1;
        I.misc[M_RESID] = r;
        resid_all[idx] = r;
        const bool fp32 = I.precision == FDLB_FP32_STORAGE;
        if (flags[0]) *I.status = FDLB_FAILED_NONFINITE;
        else if (flags[1]) *I.status = FDLB_FAILED_UNPHYSICAL;
        else if (fp32 && r == 0.0 && I.two_phase) flags[2] = 1;   // FP32 f stopped changing
        else if (fp32 && r == 0.0 && tol > 0.0) *I.status = FDLB_STAGNATED;
        else if (tol > 0.0 && r < tol) *I.status = FDLB_CONVERGED;
        else if (I.two_phase && fp32) flags[2] = stagnated(I, r, (double)*I.steps);
        scale = I.misc[M_MASS0] / tot[6];
    }
    __syncthreads();
    if (!flags[2]) return;
    // Up-cast f: floats of F -> doubles in the stage buffer A, then back into F (which holds
    // K ld doubles in a two-phase instance; A is free between steps), times the factor that
    // restores the channel mass of the last anchor.  The discrete scheme conserves mass, but
    // FP32 rounding near stagnation drops the same small updates step after step and lets the
    // mass drift, which would move the FP64 steady state.  The node rows are rescaled alike
    // (extensive rows by the factor, ln n and ln chi(eta0 n) anew; u and T are unchanged),
    // so the next stage sees the moments of the rescaled f.
    const double c = scale;
    const size_t nf = (size_t)I.K * ld;
    const float* src = static_cast<const float*>(I.f[0]);
    double* tmp = static_cast<double*>(I.f[1]);
    for (size_t e = threadIdx.x; e < nf; e += blockDim.x) tmp[e] = (double)src[e] * c;
    __syncthreads();
    double* dst = static_cast<double*>(I.f[0]);
    for (size_t e = threadIdx.x; e < nf; e += blockDim.x) dst[e] = tmp[e];
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const double n = nd[R_N * ld + i] * c;
        nd[R_N * ld + i] = n;
        nd[R_PREV_N * ld + i] *= c;
        nd[R_QX * ld + i] *= c;
        nd[R_QY * ld + i] *= c;
        nd[R_PXX * ld + i] *= c;
        nd[R_PXY * ld + i] *= c;
        nd[R_SNEG * ld + i] *= c;
        nd[R_SPOS * ld + i] *= c;
        nd[R_LNN * ld + i] = log(n);
        nd[R_LNCHI * ld + i] = log(chi_cs(I.eta0 * n));
    }
    if (threadIdx.x == 0) {
        I.precision = FDLB_FP64;
        I.misc[M_SWITCH] = (double)*I.steps;
    }
}


// The closure launch of a step's first stage can carry the residual pass of the step before it
// (blocks from n_nod on, one per instance): both only need that step's moments, and the pass, whose
// chain of one block takes ~5 us, no longer stands between two steps of a small batch (one Couette
// instance 74 -> 69 us per step).  Whether the instance goes on is decided by the status that the
// update kernels read; a closure block that still saw ACTIVE has only written tables that nothing
// reads.  Not with two-phase instances, whose residual pass may rewrite f and the moments.
template <int QB, int MB>
__global__ void __launch_bounds__(TILE * NOD_WARPS, MB) k_nodal(Inst* __restrict__ insts, const Work* __restrict__ work,
                                                                           int n_nod, double tol, double* resid_all) {
    extern __shared__ __align__(16) double nsm[];
    __shared__ Inst I;
    if ((int)blockIdx.x >= n_nod) {
        if (blockIdx.y) return;
        pdl_wait();
        Inst& g = insts[blockIdx.x - n_nod];
        if (*(volatile int*)g.status == FDLB_ACTIVE && !g.smem_res) resid_item(g, blockIdx.x - n_nod, tol, resid_all, nsm);
        return;
    }
    const Work w = work[blockIdx.x];
    if (blockIdx.y && w.k0 != 0) return;                // the x projections alone are split
    load_inst(insts + w.inst, &I, threadIdx.x, TILE * NOD_WARPS);
    warm_tables(I, w.k0, threadIdx.x, TILE * NOD_WARPS);
    pdl_wait();
    const Inst& g = insts[w.inst];
    const int st = *(volatile int*)I.status, res = *(const volatile int*)&g.smem_res, pr = *(const volatile int*)&g.precision;
    // (one decision for the block: the residual block of this launch may change the status meanwhile)
    if (__syncthreads_or(st != FDLB_ACTIVE || res)) return;
    nodal_item<QB>(I, w.i0, w.k0, nsm, pr == FDLB_FP32_STORAGE, {(int)blockIdx.y, (int)gridDim.y});
}

// Projected local equilibrium of the profile rows (n, u_x = 0, u_y, T) into F: one block per tile (the
// work list's x-projection items), with the x projection of the closure and the zeroth y and z projections, in FP64 for either storage; then a warp per
// velocity writes f, whole lines at a time.  (One block per instance with a thread per node took
// 1.0 ms for a 200-node instance of 288 velocities; this takes 20 us.)  A two-phase instance
// restarts in its FP32 phase.
template <int QB>
__global__ void __launch_bounds__(TILE * NOD_WARPS) k_profiles(Inst* insts, const Work* __restrict__ work) {
    extern __shared__ __align__(16) double nsm[];
    __shared__ double Yz[(QYMAX + 4 + QZMAX + 4) * TILE];            // m_l and T_a of y, then of z
    __shared__ double Yt[(QYMAX + QZMAX) * TILE];                    // P_0 of y, then of z
    const Work w = work[blockIdx.x];
    Inst& I = insts[w.inst];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, i0 = w.i0, i = i0 + lane, ld = I.ld, Q = I.Q, Tc = I.Tc;
    const bool valid = i < I.N;
    const int ic = valid ? i : I.N - 1;
    const bool fp32 = I.two_phase || I.precision == FDLB_FP32_STORAGE;
    double* col = I.tab + tab_col(I, i0, lane);
    if (I.xfull) xproj_full<double>(I, i0, nsm, col, Part{0, 1});
    else xproj_half<QB, double>(I, i0, nsm, col, Part{0, 1});
    const double n = I.node[R_N * ld + ic], T = I.node[R_T * ld + ic];
    const int form = I.form, Qy = I.Qy, Qz = form == FORM_UNREDUCED ? I.Qz : 0;
    double* mz = Yz + (QYMAX + 4) * TILE;
    if (wid == 0 && form != FORM_REDUCED1D)
        hermite_moments(I.node[R_UY * ld + ic], T, Qy, I.fsq, I.fsq2, I.fisq, I.fisq2, Yz + lane, Yz + (QYMAX + 1) * TILE + lane);
    if (wid == 1 && Qz)
        hermite_moments(0.0, T, Qz, I.fsq, I.fsq2, I.fisq, I.fisq2, mz + lane, mz + (QZMAX + 1) * TILE + lane);
    __syncthreads();
    for (int k = wid; form != FORM_REDUCED1D && k < Qy + Qz; k += NOD_WARPS) {
        const bool y = k < Qy;
        const int kk = y ? k : k - Qy, Qn = y ? Qy : Qz;
        const double *H = y ? I.yH : I.zH, *m = y ? Yz : mz;
        double s = 0.0;
        for (int l = 0; l < Qn; ++l) s = fma(H[l * Qn + kk], m[l * TILE + lane], s);
        Yt[k * TILE + lane] = s;
    }
    __syncthreads();
    // f = n P_0(p_x) times the transverse value (phi and theta slots carry the Gaussian's moments)
    for (int kx = wid; kx < 2 * Q; kx += NOD_WARPS) {
        const double px = valid ? n * col[kx * TILE] : 0.0;          // (written by this block)
        for (int t = 0; t < Tc; ++t) {
            double v;
            if (form == FORM_UNREDUCED) v = px * (Yt[(t / Qz) * TILE + lane] * Yt[(Qy + t % Qz) * TILE + lane]);
            else if (form == FORM_REDUCED2D) v = px * Yt[(t >> 1) * TILE + lane] * ((t & 1) ? T : 1.0);
            else v = px * (t ? 2.0 * T : 1.0);
            const size_t e = (size_t)(kx * Tc + t) * ld + i;
            if (fp32) static_cast<float*>(I.f[0])[e] = (float)v;
            else static_cast<double*>(I.f[0])[e] = v;
        }
    }
    if (threadIdx.x == 0) I.mcnt[i0 / TILE] = 0;
    if (threadIdx.x == 0 && i0 == 0) {
        if (I.two_phase) {
            I.precision = FDLB_FP32_STORAGE;
            I.misc[M_SWITCH] = -1.0;
        }
        *I.status = FDLB_ACTIVE;
        *I.steps = 0;
    }
}

__global__ void __launch_bounds__(256) k_resid(Inst* insts, int anchor, double tol, double* resid_all) {
    pdl_wait();
    Inst& I = insts[blockIdx.x];
    const int ld = I.ld, N = I.N;
    double* nd = I.node;
    __shared__ double red[7][8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (anchor >= -1) {
        if (anchor >= 0 && anchor != (int)blockIdx.x) return;
        double m = 0.0;
        for (int i = threadIdx.x; i < N; i += blockDim.x) {
            nd[R_PREV_N * ld + i] = nd[R_N * ld + i];
            nd[R_PREV_UX * ld + i] = nd[R_UX * ld + i];
            nd[R_PREV_UY * ld + i] = nd[R_UY * ld + i];
            nd[R_PREV_T * ld + i] = nd[R_T * ld + i];
            m = fma(I.dxw[i], nd[R_N * ld + i], m);
        }
        for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
        if (lane == 0) red[0][wid] = m;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += red[0][q];
            I.misc[M_MASS0] = t;
            I.misc[M_RESID] = CUDART_INF;
            I.misc[M_WIN_STEP] = -1.0;
            resid_all[blockIdx.x] = CUDART_INF;
        }
        return;
    }
    if (*I.status != FDLB_ACTIVE || I.smem_res) return;
    __shared__ double buf[7 * 256];
    resid_item(I, blockIdx.x, tol, resid_all, buf);
}

// ---------------------------------------------------------------------------
// update: WENO-5 advection + walls + force + relaxation + RK3 combination
// ---------------------------------------------------------------------------

constexpr int UPD_WARPS = 8;          // warps of an update block; the moment epilogue's partials
constexpr int UPD_WARPS_WIDE = 16;    // wide update blocks: the velocity loop on 16 warps

// ---------------------------------------------------------------------------
// stochastic rounding of FP32 storage
// ---------------------------------------------------------------------------
// With round-to-nearest, FP32 storage drops every per-step change below half an ulp of f, so a
// solve stalls at a distance ~ ulp / (2 eps) from the steady state (eps = decay per step of its
// slowest mode; ~5e-5 on the Couette sweep), and the dropped changes no longer sum to zero
// over the channel, which drifts the mass.  Rounding base + inc up or down at random, with the
// probabilities that make the expected stored value the exact sum (Connolly, Higham & Mary,
// SIAM J. Sci. Comput. 43, 2021), keeps small changes in expectation: no stall, and a mass
// error that only random-walks (sr_add, fdlb_round.cuh).  The random bits come from a counter-based hash of (the
// instance's parameters, step, stage, velocity, node), so runs are reproducible, both schedules
// round alike, and an instance rounds the same way whatever batch it is in.

// MurmurHash3's 32-bit finalizer (Appleby, public domain): a bijective avalanche mix.
__device__ __forceinline__ uint32_t fmix32(uint32_t h) {
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    return h;
}

// Per-launch seed of instance I for RK stage `stage` of the current step.
__device__ __forceinline__ uint32_t sr_seed(const Inst& I, int stage) {
    const unsigned long long step = (unsigned long long)*(volatile long long*)I.steps;
    return fmix32((uint32_t)(step * 3ull + (unsigned long long)stage) ^ fmix32(I.sr_key));
}

// Tables read by the update kernel in its compute type (FP32 copies for FP32 storage).
template <typename C>
struct Tabs;
template <>
struct Tabs<double> {
    __device__ static const double* tab(const Inst& I) { return I.tab; }
    __device__ static const double* px(const Inst& I) { return I.px; }
    __device__ static const double* gL(const Inst& I) { return I.gL; }
    __device__ static const double* gR(const Inst& I) { return I.gR; }
    __device__ static const double* xpinv(const Inst& I) { return I.xpinv; }
    __device__ static const double* Ky(const Inst& I) { return I.Ky; }
};
template <>
struct Tabs<float> {
    __device__ static const float* tab(const Inst& I) { return I.tab32; }
    __device__ static const float* px(const Inst& I) { return I.px32; }
    __device__ static const float* gL(const Inst& I) { return I.gL32; }
    __device__ static const float* gR(const Inst& I) { return I.gR32; }
    __device__ static const float* xpinv(const Inst& I) { return I.xpinv32; }
    __device__ static const float* Ky(const Inst& I) { return I.Ky32; }
};

// Shared memory of one update item: the transverse moment weights; the projection table and the
// staged source rows of the chunk (each with a 4-node halo on either side: 40 values per row),
// whose space the epilogue's per-warp sums reuse once both are consumed; and the step's F
// values, which the outputs replace (the epilogue reads them there).
constexpr size_t TW_BYTES = (size_t)NTW * TCMAX * sizeof(double);
constexpr int SW = 40;                // staged row: nodes i0 - 4 .. i0 + 35
__host__ __device__ inline size_t upd_table_bytes(int trows, size_t s) { return ((size_t)trows * TILE * s + 15) / 16 * 16; }
__host__ __device__ inline size_t upd_ex_bytes() { return (size_t)(UPD_WARPS + 1) * MOM_SUMS * TILE * sizeof(double); }
__host__ __device__ inline size_t upd_fo_offset(int trows, int ukc, size_t s) {
    const size_t rows = upd_table_bytes(trows, s) + (size_t)ukc * SW * s, ex = upd_ex_bytes();
    return TW_BYTES + ((rows > ex ? rows : ex) + 15) / 16 * 16;
}
__host__ __device__ inline size_t upd_smem_bytes(int trows, int ukc, size_t s) {
    return upd_fo_offset(trows, ukc, s) + (size_t)ukc * TILE * s;
}

// Transverse moment weights of the epilogue into shared memory (FP32 storage: float heads and, from
// TWL on, tails; FP64: doubles), by the whole block.
constexpr int TWL = NTW * TCMAX;
template <typename S>
__device__ __forceinline__ void load_tw(const Inst& I, void* tws, int tid, int nthreads) {
    const int n = NTW * I.Tc;
    if constexpr (sizeof(S) == 4) {
        float* h = static_cast<float*>(tws);
        for (int e = tid; e < n; e += nthreads) {
            h[e] = I.twh[e];
            h[TWL + e] = I.twl[e];
        }
    } else {
        double* d = static_cast<double*>(tws);
        for (int e = tid; e < n; e += nthreads) d[e] = I.tw[e];
    }
}

__device__ __forceinline__ double mom_w(const double* tw, int e, double) { return tw[e]; }
__device__ __forceinline__ df mom_w(const double* tw, int e, df) {
    const float* h = reinterpret_cast<const float*>(tw);
    return {h[e], h[TWL + e]};
}

// The 6 transverse sums of the velocities t in [t, tb) of one x-velocity, values *fr, TILE apart.
// The weights factor: over the p_z values of a p_y (or its two reduced slots) only A = sum f and
// B = sum e_z f are formed (the mass and the internal energy), then A, y A, y^2 A, y^3 A, B, y B
// once per p_y: 2 + 6/Q_z terms per value instead of 6 (3 for the reduced slots).
template <typename S, typename R>
__device__ __forceinline__ void transverse_sums(const double* tw, int Tc, int Tz, bool unred, bool ydep, int t, int tb,
                                                const S* fr, R* Sv) {
    const R zero = mom_of((S)0);
#pragma unroll
    for (int j = 0; j < NTW; ++j) Sv[j] = zero;
    int ty = t / Tz * Tz;                       // first index of t's p_y
    for (; t < tb; ty += Tz) {
        const int te = min(tb, ty + Tz);
        R A = zero, B = zero;
        if (unred) {
            A = mom_of(*fr);
            B = acc(zero, *fr, mom_w(tw, 4 * Tc + t, R{}));
            fr += TILE;
            for (++t; t < te; ++t, fr += TILE) {
                A = plus(A, *fr);
                B = acc(B, *fr, mom_w(tw, 4 * Tc + t, R{}));
            }
        } else {
            if (t == ty) {
                A = mom_of(*fr);
                fr += TILE;
                ++t;
            }
            if (t < te) {
                B = mom_of((S)0.5 * *fr);
                fr += TILE;
                ++t;
            }
        }
        Sv[0] = plus(Sv[0], A);
        Sv[4] = plus(Sv[4], B);
        if (ydep) {
            const R y = mom_w(tw, Tc + ty, R{});
            Sv[1] = acc(Sv[1], A, y);
            Sv[2] = acc(Sv[2], A, mom_w(tw, 2 * Tc + ty, R{}));
            Sv[3] = acc(Sv[3], A, mom_w(tw, 3 * Tc + ty, R{}));
            Sv[5] = acc(Sv[5], B, y);
        }
    }
}

// Epilogue of an update item: the 14 raw moment sums of the chunk's values fo[k - k0][lane],
// then the moments (one chunk per tile) or the chunk's partial sums in msum[grp].
// The chunk is cut into pieces of at most one x-velocity's length (whole x-velocities when there
// are at least UPD_WARPS of them, else an eighth of the chunk); a warp forms the transverse sums of
// a piece, one slot of shared memory per x-velocity it touches (at most two).  Then warps 0..5 add
// the 14 sums over the slots, times the power of p_x, each the sums that share a transverse sum
// (a value is read once, and the code has no index tables: those took as many instructions as the
// sums).  Against 14 sums per warp and a sum over the warps this takes 14 terms per slot once
// instead of per warp.  The pieces and the order of the slots depend on the chunk alone, not on
// the number of warps.
// Shared space ex: [2 UPD_WARPS][NTW][TILE] slots, [MOM_SUMS][TILE] sums, [2 UPD_WARPS][4] powers.

// Adds over the slots of up to UPD_WARPS pieces (sl: this lane's column), to v[0..n): x-velocity power E_j times transverse sum
// B (E_j < 0: none).  SIGN: v[0] takes the negative x-velocities, v[1] the positive ones.
struct Slots {
    int kx, t, Q, Tc, len, nk, q0;
};
template <typename R, int B, int E0, int E1 = -1, int E2 = -1, bool SIGN = false>
__device__ __forceinline__ void add_slots(const Slots& g, const R* sl, const R* pw, R* v) {
    int kx = g.kx, t = g.t;
    const R* x = sl + B * TILE;
    for (int r = 0, a = g.q0 * g.len; r < UPD_WARPS && a < g.nk; ++r, a += g.len, x += 2 * NTW * TILE, pw += 8) {
        const int n = min(g.len, g.nk - a);
        t += n;
        for (int seg = 0; seg < 2; ++seg) {
            if (seg && t <= g.Tc) break;
            const R xs = x[seg * NTW * TILE];
            const R* ps = pw + 4 * seg;
            if (SIGN) {
                const R y = acc(mom_zero(R{}), ps[1], xs);
                if (kx + seg >= g.Q) v[0] = plus(v[0], y);
                else v[1] = plus(v[1], y);
            } else {
                v[0] = E0 == 0 ? plus(v[0], xs) : acc(v[0], ps[E0], xs);
                if (E1 >= 0) v[1] = acc(v[1], ps[E1 < 0 ? 0 : E1], xs);
                if (E2 >= 0) v[2] = acc(v[2], ps[E2 < 0 ? 0 : E2], xs);
            }
        }
        if (t >= g.Tc) {
            t -= g.Tc;
            ++kx;
        }
    }
}

template <typename S>
__device__ void chunk_moments(const Inst& I, int i0, int k0, int k1, int grp, const S* fo, double* ex, const void* tws,
                              int lane, int wy) {
    using R = MomR<S>;
    const int i = i0 + lane, ld = I.ld, Tc = I.Tc, Q = I.Q, G = I.mgroups, nk = k1 - k0;
    const bool valid = i < I.N;
    const bool unred = I.form == FORM_UNREDUCED, ydep = I.form != FORM_REDUCED1D;
    const int Tz = unred ? I.Qz : 2;
    const double* tw = static_cast<const double*>(tws);
    R* sl = reinterpret_cast<R*>(ex);
    R* ss = sl + 2 * UPD_WARPS * NTW * TILE;
    R* pw = ss + MOM_SUMS * TILE;
    const int kx0 = k0 / Tc, t0 = k0 - kx0 * Tc;
    const int len = (t0 == 0 && nk >= UPD_WARPS * Tc && nk % Tc == 0) ? Tc : min(Tc, (nk + UPD_WARPS - 1) / UPD_WARPS);
    R v[3] = {mom_of((S)0), mom_of((S)0), mom_of((S)0)};
    Slots g = {kx0, t0, Q, Tc, len, nk, 0};           // kx, t: of the first velocity of piece q0
    for (int q0 = 0; q0 * len < nk; q0 += UPD_WARPS) {
        if (q0) __syncthreads();          // the slots' readers are done
        const int a = (q0 + wy) * len;
        if (wy < UPD_WARPS && a < nk) {
            int t = t0 + a, kx = kx0 + t / Tc;
            t -= (kx - kx0) * Tc;
            const int n = min(len, nk - a), n0 = min(n, Tc - t);
            const S* fr = fo + a * TILE + lane;
            for (int seg = 0; seg < 2; ++seg) {
                const int ta = seg ? 0 : t, tb = seg ? n - n0 : t + n0;
                if (ta < tb) {
                    R Sv[NTW];
                    transverse_sums(tw, Tc, Tz, unred, ydep, ta, tb, fr + (seg ? n0 * TILE : 0), Sv);
                    const int slot = 2 * wy + seg;
#pragma unroll
                    for (int j = 0; j < NTW; ++j) sl[(slot * NTW + j) * TILE + lane] = fin(Sv[j]);
                    if (lane == 0) {
                        const R p = r_tab(I.px, I.px2, kx + seg, R{}), p2 = p * p;
                        pw[slot * 4 + 1] = p;
                        pw[slot * 4 + 2] = p2;
                        pw[slot * 4 + 3] = p2 * p;
                    }
                }
            }
        }
        __syncthreads();
        g.q0 = q0;
        switch (wy) {
            case 0: add_slots<R, 0, 0, 2, 3>(g, sl + lane, pw, v); break;                 // raw sums 0, 4, 8
            case 1: add_slots<R, 0, 1, 1, -1, true>(g, sl + lane, pw, v); break;          // 1, 2
            case 2: if (ydep) add_slots<R, 1, 0, 1, 2>(g, sl + lane, pw, v); break;       // 3, 5, 10
            case 3: if (ydep) add_slots<R, 2, 0, 1>(g, sl + lane, pw, v); break;          // 6, 9
            case 4: add_slots<R, 4, 0, 1>(g, sl + lane, pw, v); break;                    // 7, 12
            case 5:
                if (ydep) {
                    add_slots<R, 3, 0>(g, sl + lane, pw, v);                              // 11
                    add_slots<R, 5, 0>(g, sl + lane, pw, v + 1);                          // 13
                }
                break;
            default: break;
        }
        if (q0 + UPD_WARPS < (nk + len - 1) / len) {
            const int t = g.t + UPD_WARPS * len;
            g.kx += t / Tc;
            g.t = t % Tc;
        }
    }
    const int j0 = wy == 0 ? 0 : wy == 1 ? 1 : wy == 2 ? 3 : wy == 3 ? 6 : wy == 4 ? 7 : 11;
    const int j1 = wy == 0 ? 4 : wy == 1 ? 2 : wy == 2 ? 5 : wy == 3 ? 9 : wy == 4 ? 12 : 13;
    const int j2 = wy == 0 ? 8 : wy == 2 ? 10 : -1;
    if (wy < 6) {
#pragma unroll
        for (int o = 0; o < 3; ++o) {
            const int j = o == 0 ? j0 : (o == 1 ? j1 : j2);
            if (j >= 0) {
                const R x = fin(v[o]);
                if (G > 1) {
                    if (valid) reinterpret_cast<R*>(I.msum)[((size_t)grp * MOM_SUMS + j) * ld + i] = x;
                } else {
                    ss[j * TILE + lane] = x;
                }
            }
        }
    }
    if (G > 1) return;
    __syncthreads();
    finalize_tile<false>(I, i0, ss, lane, wy, UPD_WARPS);
}

// Tiled schedule, tiles split into several chunks: the last chunk block of the tile to arrive
// (ticket) adds the chunks' partial sums in chunk order -- the result does not depend on the
// arrival order -- and resets the ticket.  (A chunk whose copies failed takes none; the tile's count then
// stays short until new profiles or a loaded state clear it.)  ss: MOM_SUMS x TILE shared doubles.
template <typename S>
__device__ void chunk_ticket_final(const Inst& I, int i0, double* ss, int nwb = UPD_WARPS) {
    __shared__ int last;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x, tile = i0 / TILE;
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(I.mcnt + tile, 1) == I.mgroups - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (tid == 0) I.mcnt[tile] = 0;
    moments_final_tile<S>(I, i0, ss, tid, nwb, 1);
}

// ---- bulk asynchronous copies into shared memory (cp.async.bulk with an mbarrier) ----
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// bytes (a multiple of 16) from global src to shared dst (both 16-byte aligned), completing on bar
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// 16 bytes from global src to shared dst (both 16-byte aligned), asynchronously
__device__ __forceinline__ void cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(smem_u32(dst)), "l"(src) : "memory");
}

// Phase `parity` of bar complete?  Each poll may suspend the thread for up to ~1 us.
__device__ __forceinline__ bool mbar_poll(uint64_t* bar, uint32_t parity) {
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return done != 0;
}

constexpr long COPY_WAIT_POLLS = 2000000;      // ~2 s at the suspend hint

// What an update item reads, into shared memory: rows [k0, k0 + nrows) of one tile -- the source
// stage's values of nodes i0 - 4 .. i0 + 35 (clipped to the row) into Sw[r][0..SW), and, beyond
// stage 1, the step's values of nodes i0 .. i0 + 31 into Fo[r][0..TILE) --, the compact projection
// table (rows of the NKX x-velocities from kx0 on, then the 4 Tc transverse rows and 1/tau) and the
// moment weights.  BULK (the tiled schedule): the table and the weights as cp.async.bulk copies (one
// to five and two, their completion counted in bytes on an mbarrier), the rows as 16-byte cp.async
// copies, all in flight together; a row is too short for a bulk copy of its own, whose operands go
// through uniform registers one lane at a time.  Otherwise (the resident schedules) plain loads.
// Both leave the same values in shared memory.  Window bounds are multiples of 4 nodes, so every
// copy starts on a 16-byte boundary.  Returns false if the bulk copies did not complete within
// the wait limit (the instance is then marked FDLB_FAILED_COPY).
template <typename S, bool BULK>
__device__ bool stage_item(const Inst& I, int i0, int k0, int nrows, int stage, int NKX, int kx0, S* Sw, S* Fo, S* stab,
                           void* tws, int lane, int wy, int nwb) {
    const int ld = I.ld, Q2 = 2 * I.Q, Tc = I.Tc;
    const int lo = max(0, i0 - 4), hi = min(ld, i0 + 36);
    const int off = lo - (i0 - 4);
    const S* src = static_cast<const S*>(I.f[stage - 1]);
    const S* F = static_cast<const S*>(I.f[0]);
    const bool withF = stage != 1;
    const S* tab = Tabs<S>::tab(I) + tab_col(I, i0, 0);
    const int nx = min(NKX, Q2 - kx0);                  // (the last chunk's x-velocities may be fewer)
    const int trest = 4 * Tc + 1;
    const int tid = wy * TILE + lane;
    if constexpr (BULK) {
        __shared__ __align__(8) uint64_t bar;
        const uint32_t rb = TILE * sizeof(S);           // a table row
        const bool whole = NKX == Q2;
        const uint32_t twb = ((uint32_t)(NTW * Tc) * (sizeof(S) == 4 ? 4 : 8) + 15) / 16 * 16;   // (tables are padded to 256 B)
        if (tid == 0) {
            mbar_init(&bar, 1);
            mbar_expect_tx(&bar, (4 * nx + trest) * rb + (sizeof(S) == 4 ? 2 : 1) * twb);
        }
        // earlier generic accesses of this shared memory come before the copies' writes
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        // table and weights: lane 0 of the first warps
        if (lane == 0 && wy < 7) {
            const int c = wy;
            if (c < 4) {
                if (whole) {
                    if (c == 0) bulk_g2s(stab, tab, (4 * nx + trest) * rb, &bar);
                } else {
                    bulk_g2s(stab + c * NKX * TILE, tab + (c * Q2 + kx0) * TILE, nx * rb, &bar);
                }
            } else if (c == 4) {
                if (!whole) bulk_g2s(stab + 4 * NKX * TILE, tab + 4 * Q2 * TILE, trest * rb, &bar);
            } else if constexpr (sizeof(S) == 4) {
                if (c == 5) bulk_g2s(tws, I.twh, twb, &bar);
                else bulk_g2s(static_cast<float*>(tws) + TWL, I.twl, twb, &bar);
            } else {
                if (c == 5) bulk_g2s(tws, I.tw, twb, &bar);
            }
        }
        // rows: 16 lanes each, 16 bytes per copy
        {
            constexpr int V = 16 / sizeof(S);
            const int nv = (hi - lo) / V;
            const S* g = src + (size_t)(k0 + (tid >> 4)) * ld + lo + (tid & 15) * V;
            const S* gf = F + (size_t)(k0 + (tid >> 4)) * ld + i0 + (tid & 15) * V;
            S* d = Sw + (tid >> 4) * SW + off + (tid & 15) * V;
            S* df_ = Fo + (tid >> 4) * TILE + (tid & 15) * V;
            const int dr = nwb * 2;                     // rows per pass of the block
            for (int r = tid >> 4; r < nrows; r += dr) {
                if ((tid & 15) < nv) cp16(d, g);
                if (sizeof(S) == 8 && (tid & 15) + 16 < nv) cp16(d + 16 * V, g + 16 * V);
                if (withF && (tid & 15) < TILE / V) cp16(df_, gf);
                g += (size_t)dr * ld;
                gf += (size_t)dr * ld;
                d += dr * SW;
                df_ += dr * TILE;
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
        }
        // warp 0 polls, the others wait at the barrier
        bool ok = wy != 0;
        for (long it = 0; it < COPY_WAIT_POLLS && !ok; ++it) ok = mbar_poll(&bar, 0);
        if (__syncthreads_or(!ok)) {          // the same decision in every thread of the block
            if (tid == 0) atomicExch(I.status, FDLB_FAILED_COPY);
            // give copies still in flight a second bounded wait before the block leaves
            for (long it = 0; it < COPY_WAIT_POLLS && !mbar_poll(&bar, 0); ++it) {
            }
            __syncthreads();
            return false;
        }
        if (tid == 0) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" :: "r"(smem_u32(&bar)) : "memory");
        return true;
    } else {
        __syncthreads();
        const int n = hi - lo;
        for (int r = wy; r < nrows; r += nwb) {
            const S* row = src + (size_t)(k0 + r) * ld + lo;
            for (int j = lane; j < n; j += TILE) Sw[r * SW + off + j] = row[j];
            if (withF) Fo[r * TILE + lane] = F[(size_t)(k0 + r) * ld + i0 + lane];
        }
        for (int a = 0; a < 4; ++a)
            for (int j = wy; j < nx; j += nwb) stab[(a * NKX + j) * TILE + lane] = tab[(a * Q2 + kx0 + j) * TILE + lane];
        for (int r = wy; r < trest; r += nwb) stab[(4 * NKX + r) * TILE + lane] = tab[(4 * Q2 + r) * TILE + lane];
        load_tw<S>(I, tws, tid, nwb * TILE);
        __syncthreads();
        return true;
    }
}

// RK3 combination of a new value (Eq. rk3) from f, the step's F and inc = cb dt L: FP64 cb f + inc
// + ca F, two roundings of the size of f; FP32 as an increment of F, F + cb ((f - F) + dt L)
// (stage 1: f + dt L).  In the printed form ca F + cb (f +
// dt L) the rounded weights (float) 1/3 + (float) 2/3 = 1 + 3e-8 scale a steady f up by half an
// ulp every step, a mass drift of ~1e-3 over a solve; the increment form has no such bias.  The
// FP32 sum is stored with stochastic rounding (sr_add).
struct Stage {
    double ca, cb;
    bool first;
    uint32_t seed;
};
__device__ __forceinline__ double rk_combine(const Stage& g, double fi, double F, double inc, uint32_t) {
    return g.first ? fi + inc : fma(g.ca, F, fma(g.cb, fi, inc));
}
__device__ __forceinline__ float rk_combine(const Stage& g, float fi, float F, float inc, uint32_t e) {
    const float cb = (float)g.cb;
    const float base = g.first ? fi : F;
    if (!g.first) inc = fmaf(cb, fi - F, inc);
    return sr_add(base, inc, fmix32(e ^ g.seed));
}

// What a lane (node) carries through its warp's velocities; the pointers are stepped from one
// velocity to the next.
template <typename S>
struct Lane {
    bool valid, at_wall, inner;    // inner: its right face is neither the wall's nor padding
    int lane, ld, TcS;
    S xp, invtau, Px[4];       // -cb dt p/(x' ds), cb dt/tau, the x projections of this p
    const S* row;              // staged row at this node
    const S* wall;             // staged row: [0] left face of the tile's first node, [SW - 1] wall face
    const S* Y;                // transverse factors n Y[a][t], a TcS apart
    S* fo;
    S* dst;
    uint32_t elem;             // k ld + i, for the stochastic rounding
};
template <typename S>
struct Force {
    const S* f;                // values of this x-velocity's velocities t, `stride` apart
    const S* K;
    int stride, Qy, Tz;
    S ay;
};

// Position of the k-th set bit (k from 0) of a mask with more than k.
__device__ __forceinline__ int nth_bit(unsigned mask, int k) {
    int at = 0;
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
        const int n = __popc(mask & ((1u << w) - 1u));
        if (k >= n) {
            k -= n;
            mask >>= w;
            at += w;
        }
    }
    return at;
}

// Right faces of nb <= FACE_BATCH velocities (one in FP32) from the staged rows r, r + SW, ...  FP64: the
// nodes whose stencil is rough (fdlb_weno.cuh: three to five next to a wall at start-up, rarely more) of all
// the batch's velocities are dealt out to the lanes, so that their 40 FP64 instructions run once a batch and
// not once a velocity.  Twelve Couette instances: update 96 us per launch, 104 with batches of two, 121
// one velocity at a time (93 with double-float weights everywhere); 900 nodes: 56, 56 and 65 (56).  A
// batch of four spills 296 bytes at the 80 registers of three blocks per SM; two blocks: 97 and 55, but
// full-range order 200 138 against 128.
constexpr int FACE_BATCH = 4;

template <bool POS>
__device__ __forceinline__ void upwind_faces(const float* r, int, const Lane<float>&, float* fb) {
    fb[0] = POS ? weno_face(r[-2], r[-1], r[0], r[1], r[2]) : weno_face(r[3], r[2], r[1], r[0], r[-1]);
}
template <bool POS>
__device__ __forceinline__ void upwind_faces(const double* r, int nb, const Lane<double>& c, double* fb) {
    unsigned mask[FACE_BATCH];
    int total = 0;
#pragma unroll
    for (int b = 0; b < FACE_BATCH; ++b) {
        bool rough = false;
        if (b < nb) {
            const double* q = r + b * SW;
            fb[b] = POS ? weno_face_smooth(q[-2], q[-1], q[0], q[1], q[2], rough)
                        : weno_face_smooth(q[3], q[2], q[1], q[0], q[-1], rough);
        }
        mask[b] = __ballot_sync(0xffffffffu, rough && c.inner);
        total += __popc(mask[b]);
    }
    // the rough ones, one per lane whichever velocity and node they belong to
    for (int base = 0; base < total; base += 32) {
        int k = base + c.lane, at = -1;
#pragma unroll
        for (int b = 0; b < FACE_BATCH; ++b) {
            const int nm = __popc(mask[b]);
            if (k >= 0 && k < nm) at = b * SW + 4 + nth_bit(mask[b], k);
            k -= nm;
        }
        double v = 0.0;
        if (base + c.lane < total) {
            const double* q = c.wall + at;
            v = POS ? weno_face_rough(q[-2], q[-1], q[0], q[1], q[2]) : weno_face_rough(q[3], q[2], q[1], q[0], q[-1]);
        }
        int first = -base;
#pragma unroll
        for (int b = 0; b < FACE_BATCH; ++b) {
            const int rank = first + __popc(mask[b] & ((1u << c.lane) - 1u));
            const double x = __shfl_sync(0xffffffffu, v, rank & 31);
            if ((mask[b] >> c.lane & 1) && rank >= 0 && rank < 32) fb[b] = x;
            first += __popc(mask[b]);
        }
    }
}

// n velocities t, t + 1, ... of one x-velocity; POS: p_x > 0.
template <typename S, bool POS, bool FORCE>
__device__ __forceinline__ void update_run(const Stage& g, Lane<S>& c, const Force<S>& fc, int t, int n) {
    const S *Kr = fc.K, *q0 = fc.f;              // FORCE: row p_y of the kernel, first of the p_y values
    int kz = 0;
    if (FORCE) {
        const int ky = t / fc.Tz;
        kz = t - ky * fc.Tz;
        Kr += ky * fc.Qy;
        q0 += (size_t)kz * fc.stride;
    }
    const size_t qs = FORCE ? (size_t)fc.Tz * fc.stride : 0;
    constexpr int B = sizeof(S) == 8 ? FACE_BATCH : 1;
    S fb[B];
    for (int m = 0; m < n; ++m) {
        // right faces (i + 1/2) from the five upwind nodes, of B velocities at a time
        const S* r = c.row;
        if (m % B == 0) upwind_faces<POS>(r, min(B, n - m), c, fb);
        const S fi = r[0];
        S fr = fb[0];
#pragma unroll
        for (int b = 1; b < B; ++b) fr = m % B == b ? fb[b] : fr;
        if (c.at_wall) fr = c.wall[SW - 1];
        S fl = __shfl_up_sync(0xffffffffu, fr, 1);
        if (c.lane == 0) fl = c.wall[0];
        S tgt = c.Px[0] * c.Y[0];
#pragma unroll
        for (int a = 1; a < 4; ++a) tgt += c.Px[a] * c.Y[a * c.TcS];
        S inc = c.xp * (fr - fl) + (tgt - fi) * c.invtau;
        if (FORCE) {
            const S* q = q0;
            S d = (S)0;
            for (int kp = 0; kp < fc.Qy; ++kp, q += qs) d += Kr[kp] * *q;
            q0 += fc.stride;
            if (++kz == fc.Tz) {
                kz = 0;
                q0 = fc.f;
                Kr += fc.Qy;
            }
            inc -= fc.ay * d;
        }
        const S out = rk_combine(g, fi, g.first ? (S)0 : *c.fo, inc, c.elem);
        if (c.valid) *c.dst = out;
        *c.fo = c.valid ? out : (S)0;
        c.row += SW;
        c.wall += SW;
        c.Y += TILE;
        c.fo += TILE;
        c.dst += c.ld;
        c.elem += (uint32_t)c.ld;
    }
}

// Velocities [k0, k1) of one tile for RK stage `stage`, by W warps (lane, warp wy; the moment
// partials on UPD_WARPS of them, so that W = 8 and 16 give the same results bit for bit);
// smem_raw holds upd_smem_bytes(trows, ukc, sizeof(S)).  The chunk's source rows (and F) are
// staged in shared memory first (stage_item).  Then, with one thread per velocity, the ghost cells
// of the diffuse walls are written into the rows and the faces computed that a node-per-lane loop
// cannot share (the left face of the tile's first node, and the wall face), so that the loop
// itself is the same for every tile: a contiguous range of velocities per warp, five stencil
// values, one face per lane, the left face from the neighbouring lane.  The epilogue
// computes the moments of the new values (chunk_moments).  Returns false when the staging copies
// failed.
// What bounds it: FP64 storage, the FP64 pipe (21 FP64 instructions per node-velocity and stage
// before the moments where the solution is smooth, from ~170: the first node's left face had cost a second whole face
// evaluation per warp, now one per 32 velocities, and see fdlb_weno.cuh); FP32 storage, the
// instructions issued.
template <typename S, bool BULK, int W = UPD_WARPS>
__device__ bool update_item(const Inst& I, int i0, int k0, int k1, int stage, unsigned char* smem_raw, int lane, int wy) {
    using C = S;
    const int N = I.N, ld = I.ld, Q = I.Q, Tc = I.Tc, trows = I.trows;
    void* tws = smem_raw;
    C* stab = reinterpret_cast<C*>(smem_raw + TW_BYTES);
    S* Sw = reinterpret_cast<S*>(smem_raw + TW_BYTES + upd_table_bytes(trows, sizeof(C)));
    double* ex = reinterpret_cast<double*>(stab);               // after table and rows are consumed
    S* fo = reinterpret_cast<S*>(smem_raw + upd_fo_offset(trows, I.ukc, sizeof(S)));
    const int i = i0 + lane;
    // compact table: the x-projection rows of the NKX x-velocities from kx0 on (the chunk's),
    // then the 4 Tc transverse rows and 1/tau; NKX = 2Q (kx0 = 0) is the whole table
    const int NKX = (trows - 4 * Tc - 1) / 4;
    const int kx0 = NKX == 2 * Q ? 0 : k0 / Tc;
    const bool valid = i < N;
    const C* pxc = Tabs<C>::px(I);
    __syncthreads();                      // the previous item's readers of shared memory are done
    if (!stage_item<S, BULK>(I, i0, k0, k1 - k0, stage, NKX, kx0, Sw, fo, stab, tws, lane, wy, W)) return false;
    const C nwL = (C)I.misc[M_NWL], nwR = (C)I.misc[M_NWR];
    const bool rwall = N <= i0 + TILE + 3;       // the stencil reaches the right wall
    // one thread per velocity; the left face goes into the row's first value and the wall face into
    // its last one (nodes i0 - 4 and i0 + 35, which no stencil reads)
    for (int r = wy * TILE + lane; r < k1 - k0; r += W * TILE) {
        const int k = k0 + r;
        const bool pos = k < Q * Tc;
        S* row = Sw + r * SW + 4 - i0;           // staged node j at row[j]
        C flv;
        // ghost cells and wall faces (Sec. III B): incoming populations take the wall Maxwellian
        // n_w g, outgoing ones the quadratic extrapolation of the three nodes next to the wall
        if (i0 == 0) {
            if (pos) {
                flv = nwL * Tabs<C>::gL(I)[k];
                row[-1] = row[-2] = row[-3] = flv;
            } else {
                const C f0 = row[0], f1 = row[1], f2 = row[2];
                row[-1] = 3 * f0 - 3 * f1 + f2;
                row[-2] = 6 * f0 - 8 * f1 + 3 * f2;
                row[-3] = 10 * f0 - 15 * f1 + 6 * f2;
                flv = (11 * f0 - 7 * f1 + 2 * f2) * (C)(1.0 / 6.0);
            }
        }
        if (rwall) {
            C g0, g1, g2, fwv;
            if (!pos) {
                fwv = nwR * Tabs<C>::gR(I)[k];
                g0 = g1 = g2 = fwv;
            } else {
                const C f0 = row[N - 1], f1 = row[N - 2], f2 = row[N - 3];
                g0 = 3 * f0 - 3 * f1 + f2;
                g1 = 6 * f0 - 8 * f1 + 3 * f2;
                g2 = 10 * f0 - 15 * f1 + 6 * f2;
                fwv = (11 * f0 - 7 * f1 + 2 * f2) * (C)(1.0 / 6.0);
            }
            // (stencils end at node i0 + 34)
            if (N < i0 + 35) row[N] = g0;
            if (N + 1 < i0 + 35) row[N + 1] = g1;
            if (N + 2 < i0 + 35) row[N + 2] = g2;
            Sw[r * SW + SW - 1] = fwv;
        }
        if (i0 != 0) {
            const S* q = row + (pos ? i0 - 3 : i0 + 2);
            const int d = pos ? 1 : -1;
            flv = weno_face(q[0], q[d], q[2 * d], q[3 * d], q[4 * d]);
        }
        Sw[r * SW] = flv;
    }
    const int per = (k1 - k0 + W - 1) / W;
    const int ka = min(k1, k0 + wy * per), nk = min(k1, ka + per) - ka;
    __syncthreads();
    const S* src = static_cast<const S*>(I.f[stage - 1]);
    S* dst = static_cast<S*>(I.f[stage % 3]);
    Stage g;
    g.first = stage == 1;
    g.ca = stage == 1 ? 0.0 : (stage == 2 ? 0.75 : 1.0 / 3.0);
    g.cb = stage == 1 ? 1.0 : (stage == 2 ? 0.25 : 2.0 / 3.0);
    g.seed = sizeof(S) == 4 ? sr_seed(I, stage) : 0u;
    // increments are in units of cb dt
    const C cdt = (C)(g.cb * I.dt);
    const C xpi = valid ? -cdt * Tabs<C>::xpinv(I)[i] : (C)0;
    const C invtau = cdt * stab[(4 * NKX + 4 * Tc) * TILE + lane];
    const bool force = I.accel_y != 0.0 && I.form != FORM_REDUCED1D;
    const int Qy = I.Qy, Tz = I.form == FORM_UNREDUCED ? I.Qz : 2;
    const C ay = cdt * (C)I.accel_y;
    const C* Kyc = Tabs<C>::Ky(I);
    // padding lanes read the last node's values and write nothing
    const int li = valid ? lane : N - 1 - i0;
    Lane<S> c;
    c.valid = valid;
    c.at_wall = i + 1 == N;
    c.inner = i + 1 < N;
    c.lane = lane;
    c.ld = ld;
    c.TcS = Tc * TILE;
    c.invtau = invtau;
    c.row = Sw + (ka - k0) * SW + 4 + li;
    c.wall = Sw + (ka - k0) * SW;
    c.fo = fo + (ka - k0) * TILE + lane;
    c.dst = dst + (size_t)ka * ld + i;
    c.elem = (uint32_t)ka * (uint32_t)ld + (uint32_t)i;
    int kx = ka / Tc, t = ka - kx * Tc;
    for (int left = nk; left > 0; ++kx) {
        const int nt = min(left, Tc - t);
        c.xp = xpi * pxc[kx];
#pragma unroll
        for (int a = 0; a < 4; ++a) c.Px[a] = stab[(a * NKX + kx - kx0) * TILE + lane];
        c.Y = stab + (4 * NKX + t) * TILE + lane;
        Force<S> fc;
        if (force) {
            // the rows of this x-velocity's other p_y: staged if the chunk has them all
            const bool in = kx * Tc >= k0 && (kx + 1) * Tc <= k1;
            fc.f = in ? Sw + (kx * Tc - k0) * SW + 4 + li : src + (size_t)kx * Tc * ld + i0 + li;
            fc.stride = in ? SW : ld;
            fc.K = Kyc;
            fc.ay = ay;
            fc.Qy = Qy;
            fc.Tz = Tz;
            if (kx < Q) update_run<S, true, true>(g, c, fc, t, nt);
            else update_run<S, false, true>(g, c, fc, t, nt);
        } else if (kx < Q) {
            update_run<S, true, false>(g, c, fc, t, nt);
        } else {
            update_run<S, false, false>(g, c, fc, t, nt);
        }
        left -= nt;
        t = 0;
    }
    __syncthreads();                      // every warp is done with table and rows (ex aliases them)
    if (BULK) pdl_trigger();
    chunk_moments<S>(I, i0, k0, k1, k0 / I.ukc, fo, ex, tws, lane, wy);
    return true;
}

template <typename S, int W>
__global__ void __launch_bounds__(TILE * W, W == UPD_WARPS ? (sizeof(S) == 4 ? 4 : 3) : 1) k_update(const Inst* __restrict__ insts, const Work* __restrict__ work, int stage) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Inst I;
    const Work w = work[blockIdx.x];
    load_inst(insts + w.inst, &I, threadIdx.y * TILE + threadIdx.x, W * TILE);
    if (!runs_now(insts[w.inst], I, sizeof(S) == 8)) return;
    if (!update_item<S, true, W>(I, w.i0, w.k0, w.k1, stage, smem_raw, threadIdx.x, threadIdx.y)) return;
    if (I.mgroups > 1)
        chunk_ticket_final<S>(I, w.i0, reinterpret_cast<double*>(smem_raw + TW_BYTES), W);
}

// Moments of buffer `buf` from scratch (creation, new profiles, a loaded state): one block per
// update chunk of a tile with exactly the arithmetic of the update epilogue, so that the
// moments of a state do not depend on how it was reached (restarts are bitwise).
template <typename S>
__global__ void __launch_bounds__(TILE * UPD_WARPS) k_moments(const Inst* __restrict__ insts, const Work* __restrict__ work, int buf) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Work w = work[blockIdx.x];
    const Inst& I = insts[w.inst];
    if (*I.status != FDLB_ACTIVE) return;
    if ((I.precision == FDLB_FP64) != (sizeof(S) == 8)) return;
    const int lane = threadIdx.x, wy = threadIdx.y, i = w.i0 + lane, ld = I.ld;
    const bool valid = i < I.N;
    void* tws = smem_raw;
    S* fo = reinterpret_cast<S*>(smem_raw + TW_BYTES);
    double* ex = reinterpret_cast<double*>(smem_raw + TW_BYTES + (size_t)I.ukc * TILE * sizeof(S));
    const S* f = static_cast<const S*>(I.f[buf]);
    for (int k = w.k0 + wy; k < w.k1; k += UPD_WARPS) fo[(k - w.k0) * TILE + lane] = valid ? f[(size_t)k * ld + i] : (S)0;
    load_tw<S>(I, tws, wy * TILE + lane, UPD_WARPS * TILE);
    __syncthreads();
    chunk_moments<S>(I, w.i0, w.k0, w.k1, w.k0 / I.ukc, fo, ex, tws, lane, wy);
    if (I.mgroups > 1) chunk_ticket_final<S>(I, w.i0, ex);
}

// ---------------------------------------------------------------------------
// resident schedule: one thread-block cluster per instance runs whole steps
// ---------------------------------------------------------------------------
// The phases of a step are the items of the tiled kernels (identical arithmetic), spread over
// the cluster's CTAs and separated by cluster barriers instead of kernel boundaries.  Every
// CTA of a cluster passes the same barriers: the trip counts depend only on the instance and
// on values broadcast from rank 0's shared memory.  Clusters never wait on each other.
namespace cg = cooperative_groups;

constexpr int RES_THREADS = TILE * NOD_WARPS;    // 256 = UPD_WARPS warps = two moment halves

__host__ __device__ inline size_t resident_smem_bytes(int qmax, size_t upd_max) {
    const size_t fin = (size_t)2 * MOM_SUMS * TILE * sizeof(double);
    const size_t nod = (size_t)nodal_smem_doubles(qmax) * sizeof(double);
    size_t m = fin > nod ? fin : nod;
    return m > upd_max ? m : upd_max;
}

// Moments of tiles whose update was split into chunks: the chunk partials, by 128-thread halves.
template <typename S>
__device__ void res_final(const Inst& I, int rank, int CS, unsigned char* sm, cg::cluster_group& cl) {
    const int tiles = (I.N + TILE - 1) / TILE, half = threadIdx.x >> 7;
    double* ss = reinterpret_cast<double*>(sm) + half * MOM_SUMS * TILE;
    for (int tl = 2 * rank + half; tl < tiles; tl += 2 * CS) moments_final_tile<S>(I, tl * TILE, ss, threadIdx.x & 127, 4, 1 + half);
    cl.sync();
}

template <int QB, typename S>
__device__ void res_step(Inst& I, int idx, double tol, double* resid_all, int rank, int CS, unsigned char* sm,
                         cg::cluster_group& cl) {
    const int tiles = (I.N + TILE - 1) / TILE, K = I.K, KC = I.ukc, nch = I.mgroups;
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    // the update items' epilogue computes the moments of each stage's result
    for (int stage = 1; stage <= 3; ++stage) {
        for (int it = rank; it < NODAL_ROLES * tiles; it += CS)
            nodal_item<QB>(I, (it / NODAL_ROLES) * TILE, it % NODAL_ROLES, reinterpret_cast<double*>(sm), sizeof(S) == 4);
        cl.sync();
        for (int it = rank; it < tiles * nch; it += CS) {
            const int tl = it / nch, c = it - tl * nch, k0 = c * KC;
            update_item<S, false>(I, tl * TILE, k0, min(K, k0 + KC), stage, sm, lane, wy);
        }
        cl.sync();
        if (nch > 1) res_final<S>(I, rank, CS, sm, cl);
    }
    if (rank == 0) resid_item(I, idx, tol, resid_all, reinterpret_cast<double*>(sm));
}

// Cluster c of the grid advances instance list[c] by up to nsteps steps (it stops early when
// the instance leaves ACTIVE).
template <int QB>
__global__ void __launch_bounds__(RES_THREADS, 1) k_resident(Inst* insts, const int* list, int nsteps, double tol, double* resid_all) {
    extern __shared__ __align__(16) unsigned char rsm[];
    __shared__ int bc[2];
    cg::cluster_group cl = cg::this_cluster();
    const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int idx = list[blockIdx.x / CS];
    Inst& I = insts[idx];
    for (int s = 0; s < nsteps; ++s) {
        if (rank == 0 && threadIdx.x == 0) {
            bc[0] = *(volatile int*)I.status;
            bc[1] = *(volatile int*)&I.precision;
        }
        cl.sync();
        const int* b0 = cl.map_shared_rank(bc, 0);
        const int st = b0[0], prec = b0[1];
        if (st != FDLB_ACTIVE) {
            cl.sync();                    // nobody reads rank 0's shared memory after it exits
            break;
        }
        if (prec == FDLB_FP64) res_step<QB, double>(I, idx, tol, resid_all, rank, CS, rsm, cl);
        else res_step<QB, float>(I, idx, tol, resid_all, rank, CS, rsm, cl);
    }
}

// ---------------------------------------------------------------------------
// shared-memory-resident schedule: one CTA per instance keeps f in shared memory
// ---------------------------------------------------------------------------
// The CTA runs whole steps of its instance with the items of the tiled kernels (identical
// arithmetic) on a block-local copy of the instance record whose three RK buffers point into
// dynamic shared memory: f crosses HBM only when the launch starts and ends.  Tables, node rows
// and partial sums stay in global memory (L2).  Stages are separated by block barriers.
__host__ __device__ inline size_t smemres_f_bytes(int K, int ld, size_t s) { return ((size_t)K * ld * s + 15) / 16 * 16; }

template <int QB, typename S>
__device__ void smem_step(Inst& I, int idx, double tol, double* resid_all, unsigned char* sm) {
    const int tiles = (I.N + TILE - 1) / TILE, K = I.K, KC = I.ukc, nch = I.mgroups;
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    for (int stage = 1; stage <= 3; ++stage) {
        for (int it = 0; it < NODAL_ROLES * tiles; ++it)
            nodal_item<QB>(I, (it / NODAL_ROLES) * TILE, it % NODAL_ROLES, reinterpret_cast<double*>(sm), sizeof(S) == 4);
        __syncthreads();
        for (int it = 0; it < tiles * nch; ++it) {
            const int tl = it / nch, c = it - tl * nch, k0 = c * KC;
            update_item<S, false>(I, tl * TILE, k0, min(K, k0 + KC), stage, sm, lane, wy);
        }
        __syncthreads();
        if (nch > 1) {
            // moments of chunked tiles from their partials, by 128-thread halves
            const int half = threadIdx.x >> 7;
            double* ss = reinterpret_cast<double*>(sm) + half * MOM_SUMS * TILE;
            for (int tl = half; tl < tiles; tl += 2) moments_final_tile<S>(I, tl * TILE, ss, threadIdx.x & 127, 4, 1 + half);
            __syncthreads();
        }
    }
    resid_item(I, idx, tol, resid_all, reinterpret_cast<double*>(sm));
    __syncthreads();
}

// Block b advances instance list[b] by up to nsteps steps; dynamic shared memory = scratch
// bytes for the items, then the three RK buffers.
template <int QB>
__global__ void __launch_bounds__(RES_THREADS, 1) k_smemres(Inst* insts, const int* list, int nsteps, double tol, double* resid_all,
                                                            size_t scratch) {
    extern __shared__ __align__(16) unsigned char rsm[];
    __shared__ Inst Is;
    const int idx = list[blockIdx.x];
    Inst& Ig = insts[idx];
    if (*(volatile int*)Ig.status != FDLB_ACTIVE) return;
    if (threadIdx.x == 0) Is = Ig;
    __syncthreads();
    const bool fp32 = Is.precision == FDLB_FP32_STORAGE;
    const size_t bytes = (size_t)Is.K * Is.ld * (fp32 ? 4 : 8);          // a multiple of 128
    const size_t fb = smemres_f_bytes(Is.K, Is.ld, fp32 ? 4 : 8);
    unsigned char* fs = rsm + scratch;
    uint4* gF = static_cast<uint4*>(Ig.f[0]);
    __syncthreads();
    if (threadIdx.x == 0)
        for (int b = 0; b < 3; ++b) Is.f[b] = fs + b * fb;
    uint4* sF = reinterpret_cast<uint4*>(fs);
    for (size_t e = threadIdx.x; e < bytes / 16; e += blockDim.x) sF[e] = gF[e];
    __syncthreads();
    for (int step = 0; step < nsteps; ++step) {
        if (*(volatile int*)Is.status != FDLB_ACTIVE) break;              // written by this block
        if (fp32) smem_step<QB, float>(Is, idx, tol, resid_all, rsm);
        else smem_step<QB, double>(Is, idx, tol, resid_all, rsm);
    }
    for (size_t e = threadIdx.x; e < bytes / 16; e += blockDim.x) gF[e] = sF[e];
}

// ---------------------------------------------------------------------------
// launch wrappers
// ---------------------------------------------------------------------------
// The stepping kernels (closure, update, residual) are launched with programmatic stream
// serialization: the next kernel of a step is set up while the previous one finishes.
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Kernel attributes (dynamic shared memory above 48 KB, non-portable cluster sizes) and the
// __constant__ tables are per device: each device keeps its own record of what was set, and
// a mutex serialises the updates.  Attributes only ever grow, so contexts created earlier on
// a device keep launching.
namespace {
constexpr int kMaxDevices = 64;
// Dynamic sizes above this are opted in: static and dynamic shared memory together may take 48 KB
// without it, and the kernels' static parts are below 16 KB.
constexpr size_t SMEM_OPTIN = 32 * 1024;
struct DevAttr {
    bool consts = false;
    int nodal = 0;
    size_t mom64 = 0, mom32 = 0, upd64 = 0, upd32 = 0;
    size_t res[2] = {0, 0};
    size_t smemres[2] = {0, 0};
    bool nonport[2] = {false, false};
};
std::mutex g_attr_mu;
DevAttr g_attr[kMaxDevices];

// Record of the current device (the caller holds g_attr_mu).
cudaError_t dev_attr(DevAttr** out) {
    int d = -1;
    cudaError_t e = cudaGetDevice(&d);
    if (e != cudaSuccess) return e;
    if (d < 0 || d >= kMaxDevices) return cudaErrorInvalidDevice;
    *out = &g_attr[d];
    return cudaSuccess;
}
}  // namespace

cudaError_t launch_setup(const Inst* d_inst, int count, cudaStream_t s) {
    k_setup<<<count, 128, 0, s>>>(const_cast<Inst*>(d_inst));
    return cudaGetLastError();
}

cudaError_t launch_profiles(const Inst* d_inst, const Work* d_nod, int n_nod, int qmax, cudaStream_t s) {
    const size_t smem = (size_t)nodal_smem_doubles(qmax) * sizeof(double);
    Inst* in = const_cast<Inst*>(d_inst);
    if (qmax <= 8) k_profiles<8><<<n_nod, TILE * NOD_WARPS, smem, s>>>(in, d_nod);
    else k_profiles<QMAX><<<n_nod, TILE * NOD_WARPS, smem, s>>>(in, d_nod);
    return cudaGetLastError();
}

size_t moments_smem_bytes(int ukc, size_t s) {
    return TW_BYTES + (size_t)ukc * TILE * s + (size_t)(UPD_WARPS + 1) * MOM_SUMS * TILE * sizeof(double);
}

size_t update_smem_bytes(int trows, int ukc, size_t s) { return upd_smem_bytes(trows, ukc, s); }

// The need that the chunk of the largest velocity sets and the set of shared-memory instances are
// chosen with: an upper bound of update_smem_bytes, kept apart from it so that a batch's layout
// and mix do not change with the kernel's own use.
size_t update_smem_bound(int trows, int ukc, size_t s) {
    const size_t rows = (size_t)ukc * SW * s, ex = upd_ex_bytes();
    return upd_table_bytes(trows, s) + TW_BYTES + ((rows > ex ? rows : ex) + 15) / 16 * 16 + (size_t)ukc * TILE * s;
}

cudaError_t launch_moments(const Inst* d_inst, const Work* d_upd, int n_upd, int buf, int ukc_max, bool f64, bool f32,
                           cudaStream_t s) {
    const size_t m64 = moments_smem_bytes(ukc_max, 8), m32 = moments_smem_bytes(ukc_max, 4);
    {
        std::lock_guard<std::mutex> lk(g_attr_mu);
        DevAttr* A = nullptr;
        cudaError_t e = dev_attr(&A);
        if (e == cudaSuccess && f64 && m64 > SMEM_OPTIN && m64 > A->mom64) {
            e = cudaFuncSetAttribute(k_moments<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)m64);
            if (e == cudaSuccess) A->mom64 = m64;
        }
        if (e == cudaSuccess && f32 && m32 > SMEM_OPTIN && m32 > A->mom32) {
            e = cudaFuncSetAttribute(k_moments<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)m32);
            if (e == cudaSuccess) A->mom32 = m32;
        }
        if (e != cudaSuccess) return e;
    }
    dim3 blk(TILE, UPD_WARPS);
    if (f64) k_moments<double><<<n_upd, blk, m64, s>>>(d_inst, d_upd, buf);
    if (f32) k_moments<float><<<n_upd, blk, m32, s>>>(d_inst, d_upd, buf);
    return cudaGetLastError();
}

cudaError_t launch_resid(const Inst* d_inst, int count, int anchor_inst, double freeze_tol, double* d_resid_all, cudaStream_t s) {
    if (anchor_inst != -2) {
        k_resid<<<count, 256, 0, s>>>(const_cast<Inst*>(d_inst), anchor_inst, freeze_tol, d_resid_all);
        return cudaGetLastError();
    }
    return launch_pdl(k_resid, dim3(count), dim3(256), 0, s, const_cast<Inst*>(d_inst), anchor_inst, freeze_tol, d_resid_all);
}

// (the caller holds g_attr_mu)
static cudaError_t set_smem(DevAttr* A, size_t smem64, size_t smem32) {
    cudaError_t e = cudaSuccess;
    if (smem64 > SMEM_OPTIN && smem64 > A->upd64) {
        e = cudaFuncSetAttribute(k_update<double, UPD_WARPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem64);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_update<double, UPD_WARPS_WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem64);
        if (e == cudaSuccess) A->upd64 = smem64;
    }
    if (e == cudaSuccess && smem32 > SMEM_OPTIN && smem32 > A->upd32) {
        e = cudaFuncSetAttribute(k_update<float, UPD_WARPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem32);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_update<float, UPD_WARPS_WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem32);
        if (e == cudaSuccess) A->upd32 = smem32;
    }
    return e;
}

cudaError_t launch_nodal(const Inst* d_inst, const Work* d_nod, int n_nod, int qmax, int xparts, bool one_wave, int n_resid,
                         double freeze_tol, double* d_resid_all, cudaStream_t s) {
    const size_t smem = (size_t)nodal_smem_doubles(qmax) * sizeof(double);
    const dim3 grid(n_nod + n_resid, xparts);
    Inst* in = const_cast<Inst*>(d_inst);
    if (qmax <= 8) {
        // three blocks per SM (80 registers, a few spilled) where blocks queue: 2048 mixed instances
        // 790 -> 720 us per launch against two; unconstrained (150 registers) when each block has an
        // SM to itself: one Couette instance 13.5 -> 12.2 us (and 12 instances 15.3 -> 20.3, so not there).
        // Whole steps of 1 to 10 instances (14 to 140 blocks) take 1 to 3 us less, 11 (154) take 106 us against 95.
        auto k = one_wave ? k_nodal<8, 1> : k_nodal<8, 3>;
        return launch_pdl(k, grid, dim3(TILE * NOD_WARPS), smem, s, in, d_nod, n_nod, freeze_tol, d_resid_all);
    }
    return launch_pdl(k_nodal<QMAX, 1>, grid, dim3(TILE * NOD_WARPS), smem, s, in, d_nod, n_nod, freeze_tol, d_resid_all);
}

cudaError_t prepare_kernels(size_t smem64, size_t smem32, int qmax) {
    std::lock_guard<std::mutex> lk(g_attr_mu);
    DevAttr* A = nullptr;
    cudaError_t ed = dev_attr(&A);
    if (ed != cudaSuccess) return ed;
    if (!A->consts) {
        float2 h[NINV2];
        h[0] = make_float2(0.0f, 0.0f);
        for (int j = 1; j < NINV2; ++j) {
            const double v = 1.0 / j;
            const float hi = (float)v;
            h[j] = make_float2(hi, (float)(v - (double)hi));
        }
        // synchronous copy: the table is in place before any kernel of this device uses it
        cudaError_t e = cudaMemcpyToSymbol(c_inv2, h, sizeof(h));
        if (e != cudaSuccess) return e;
        A->consts = true;
    }
    const int smem = nodal_smem_doubles(qmax) * (int)sizeof(double);
    if ((size_t)smem > SMEM_OPTIN && smem > A->nodal) {
        cudaError_t e = cudaFuncSetAttribute(k_nodal<8, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_nodal<8, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_nodal<QMAX, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_profiles<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_profiles<QMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        A->nodal = smem;
    }
    return set_smem(A, smem64, smem32);
}

// Attributes only ever grow, so that contexts created earlier keep launching; slot 0 records
// k_resident<8>, slot 1 k_resident<QMAX>.
template <int QB>
static cudaError_t resident_config(size_t smem, int cs) {
    std::lock_guard<std::mutex> lk(g_attr_mu);
    DevAttr* A = nullptr;
    cudaError_t e = dev_attr(&A);
    if (e != cudaSuccess) return e;
    const int slot = QB == 8 ? 0 : 1;
    if (smem > A->res[slot]) {
        e = cudaFuncSetAttribute(k_resident<QB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) A->res[slot] = smem;
    }
    if (e == cudaSuccess && cs > 8 && !A->nonport[slot]) {
        e = cudaFuncSetAttribute(k_resident<QB>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess) A->nonport[slot] = true;
    }
    return e;
}

cudaError_t prepare_resident(int qmax, size_t upd_max, int cs, size_t* smem) {
    *smem = resident_smem_bytes(qmax, upd_max);
    return qmax <= 8 ? resident_config<8>(*smem, cs) : resident_config<QMAX>(*smem, cs);
}

template <int QB>
static cudaError_t max_clusters(size_t smem, int cs, int* n) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(RES_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(n, k_resident<QB>, &cfg);
}

cudaError_t resident_max_clusters(int qmax, size_t smem, int cs, int* n) {
    return qmax <= 8 ? max_clusters<8>(smem, cs, n) : max_clusters<QMAX>(smem, cs, n);
}

cudaError_t launch_resident(Inst* d_inst, const int* d_list, int nclusters, int cs, int qmax, size_t smem, int nsteps,
                            double freeze_tol, double* d_resid_all, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(nclusters * cs);
    cfg.blockDim = dim3(RES_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (qmax <= 8) return cudaLaunchKernelEx(&cfg, k_resident<8>, d_inst, d_list, nsteps, freeze_tol, d_resid_all);
    return cudaLaunchKernelEx(&cfg, k_resident<QMAX>, d_inst, d_list, nsteps, freeze_tol, d_resid_all);
}

__global__ void k_set_smem_flags(Inst* insts, const int* list, int n, int on) {
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) insts[list[j]].smem_res = on;
}

cudaError_t launch_set_smem_flags(Inst* d_inst, const int* d_list, int n, int on, cudaStream_t s) {
    if (n > 0) k_set_smem_flags<<<(n + 255) / 256, 256, 0, s>>>(d_inst, d_list, n, on);
    return cudaGetLastError();
}

// The scratch is at least the bound that the set of shared-memory instances has always been
// chosen with, so that a batch keeps its mix when the closure's own need changes.
size_t smemres_scratch_bytes(int qmax, size_t upd_max) {
    const int qb = qmax > QMAX ? QMAX : qmax;
    const int states = qmax > QMAX ? (aux_points_half(qmax) > qmax / 2 + 2 ? aux_points_half(qmax) : qmax / 2 + 2) : 0;
    const int rows_x = (NOD_WARPS + 1) * 4 * qb + 2 * states;
    const int rows_c = 28 + 4 * QYMAX + 3 * QZMAX + 8 * QYMAX + 2 * MYMAX * (QYMAX + 1);
    const size_t bound = (size_t)(rows_x > rows_c ? rows_x : rows_c) * TILE * sizeof(double);
    const size_t need = resident_smem_bytes(qmax, upd_max);
    return need > bound ? need : bound;
}
size_t smemres_buffer_bytes(int K, int ld, size_t s) { return smemres_f_bytes(K, ld, s); }

// Dynamic shared memory available to k_smemres<QB>: the per-block maximum minus its static part.
cudaError_t smemres_dynamic_limit(int qmax, size_t* limit) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = qmax <= 8 ? cudaFuncGetAttributes(&fa, k_smemres<8>) : cudaFuncGetAttributes(&fa, k_smemres<QMAX>);
    if (e != cudaSuccess) return e;
    *limit = (size_t)optin > fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : 0;
    return cudaSuccess;
}

cudaError_t prepare_smemres(int qmax, size_t dyn) {
    std::lock_guard<std::mutex> lk(g_attr_mu);
    DevAttr* A = nullptr;
    cudaError_t e = dev_attr(&A);
    if (e != cudaSuccess) return e;
    const int slot = qmax <= 8 ? 0 : 1;
    if (dyn > A->smemres[slot]) {
        e = qmax <= 8 ? cudaFuncSetAttribute(k_smemres<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn)
                      : cudaFuncSetAttribute(k_smemres<QMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
        if (e == cudaSuccess) A->smemres[slot] = dyn;
    }
    return e;
}

cudaError_t launch_smemres(Inst* d_inst, const int* d_list, int n, int qmax, size_t scratch, size_t dyn, int nsteps,
                           double freeze_tol, double* d_resid_all, cudaStream_t s) {
    if (qmax <= 8) k_smemres<8><<<n, RES_THREADS, dyn, s>>>(d_inst, d_list, nsteps, freeze_tol, d_resid_all, scratch);
    else k_smemres<QMAX><<<n, RES_THREADS, dyn, s>>>(d_inst, d_list, nsteps, freeze_tol, d_resid_all, scratch);
    return cudaGetLastError();
}

cudaError_t launch_update(const Inst* d_inst, const Work* d_upd, int n_upd, int stage, size_t smem64, size_t smem32,
                          bool f64, bool f32, bool wide, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    if (wide) {
        const dim3 blk(TILE, UPD_WARPS_WIDE);
        if (f64) e = launch_pdl(k_update<double, UPD_WARPS_WIDE>, dim3(n_upd), blk, smem64, s, d_inst, d_upd, stage);
        if (e == cudaSuccess && f32)
            e = launch_pdl(k_update<float, UPD_WARPS_WIDE>, dim3(n_upd), blk, smem32, s, d_inst, d_upd, stage);
    } else {
        const dim3 blk(TILE, UPD_WARPS);
        if (f64) e = launch_pdl(k_update<double, UPD_WARPS>, dim3(n_upd), blk, smem64, s, d_inst, d_upd, stage);
        if (e == cudaSuccess && f32) e = launch_pdl(k_update<float, UPD_WARPS>, dim3(n_upd), blk, smem32, s, d_inst, d_upd, stage);
    }
    return e;
}

}  // namespace fdlb
