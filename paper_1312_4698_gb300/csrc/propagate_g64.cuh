// FP64 propagation by packed lane groups (Sec. III.A / III.B of arXiv:1312.4698).
//
// A group of G lanes owns one trajectory, a warp T = 32 / G of them.  The 2F columns of the
// monodromy matrix, the F modes and the P = F (F + 1) / 2 packed Hessian entries are dealt out
// over the group in rounds: NC = ceil(2F / G) columns, NM modes and NE entries to a lane, the
// state in registers, the Hessian and the coordinates exchanged through shared memory.  Steps
// run in chunks of C; the job (trajectory, step) of a chunk is a lane's own in the determinant
// of the Herman-Kluk matrix, the continuous phase and the amplitude.
//
// What bounds it: a warp's FP64 instruction holds its sub-partition's FP64 pipe for 64 cycles on
// GB300 whatever lanes are active (measured from 1 to 32 lanes; 76 with all four sub-partitions
// busy; conversions, comparisons and mma.f64 share the pipe), which is also its latency: one warp
// per sub-partition keeps the pipe busy, and the time is the number of FP64 instructions a warp
// executes.  So the group size follows the number of trajectories (choose_g64_lanes): few
// trajectories take wide groups (fewest rounds), many take narrow groups (at F = 6 four lanes hold
// exactly 3 columns each: every lane works in 98 % of the instructions, against 75 % with 16).
// The FP64 instructions themselves are cut down: coupling tensors and diagonal parameters staged
// with the factor -tau of their kick, V and its gradient from the rows of H q and H3 q,
// reciprocals in three multiply-adds from the hardware's approximation, exponentials from a
// 64-entry table, pivots and thresholds compared as integers, det M's pivots multiplied pairwise.
// Against the groups of 8 to 32 lanes without these, us per step: F = 6, 4096 trajectories: 103 -> 59;
// F = 3, 96: 17.0 -> 9.7 (6.6 with a recording warp).
#pragma once

#include <math_constants.h>
#include <cstddef>
#include <type_traits>
#include <utility>

#include "fp64_ops.cuh"
#include "scivr_internal.cuh"

namespace scivr {
namespace g64 {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kMaxWarps = 4;   // warps per CTA: one for each sub-partition of an SM

// Shared rows read with 16-byte loads by several groups at once: an even length, an odd number of
// 16-byte vectors, so that the groups' rows start in different bank groups.
__host__ __device__ constexpr int even(int n) { return (n + 1) & ~1; }
__host__ __device__ constexpr int row_len(int n) { return even(n) / 2 % 2 ? even(n) : even(n) + 2; }
__host__ __device__ constexpr int ilog2(int n) { return n < 2 ? 0 : 1 + ilog2(n / 2); }

template <int F, int G>
struct Geo {
    static constexpr int N2 = 2 * F, P = F * (F + 1) / 2, T = 32 / G;
    static constexpr int NC = (N2 + G - 1) / G, NM = (F + G - 1) / G, NE = (P + G - 1) / G;
    // Steps per chunk: a job for every lane.  At F = 9 half as many, so that four warps'
    // prefactor matrices (1.3 KB a job) fit an SM's shared memory.
    static constexpr int C = F > 8 ? G / 2 : G;
    static constexpr int JOBS = T * C;
    static constexpr int S3 = row_len(F), S4 = row_len(P), SH = even(F), HT = row_len(F * SH);
    static constexpr int AS = (F * F) | 1;

    // FP64 instructions of a warp per step, counted from the code below: the trajectory and its
    // monodromy, and the records (determinants, phase, amplitude).  The measure by which the group
    // size is chosen.
    static constexpr int kStepInstr =
        4 * (NC * F + 3 * NM) + 3 * (NE * (1 + F + P) + NM * (2 * F + 28) + NC * F * F) + ilog2(G);
    static constexpr int kRecordInstr =
        NC * (N2 * (N2 - 1) / 2) + N2 * (3 + NC) + NC + ilog2(G) + 4 * NM * F + 6 +
        (4 * (F * (F * F - 1)) / 3 + 11 * F + 4 * F * (F - 1) / 2 + 9 * F + 110) / C;
    static constexpr int kStateInstr = (9 * F + 75) / C;   // of a record, for every reference state but the first (counted at
                                                           // F = 1, where a step is little beside them)
    static constexpr int MAIL = NC * N2 + 2 * NM + 1;   // state of a step that its records need, per lane
};

// Constants of a CTA, staged once: the coupling tensors and diagonal parameters times -tau of each
// of the two kick lengths (k = 0 the outer kicks, 1 the middle one).
template <int F>
struct CtaShared {
    using E = Geo<F, 32>;
    alignas(16) double T3[2][E::P][E::S3];    // cubic rows of an entry
    alignas(16) double T4[2][E::P][E::S4];    // quartic rows of an entry
    alignas(16) double acoef[F * F][4];       // (1/2) {rg_a/rg_b, rg_b/rg_a, -rg_a rg_b, 1/(rg_a rg_b)}
    double kD[2][F], kDa[2][F], kDaa[2][F];   // -tau {D, 2 D a, 2 D a^2} (Morse), -tau {omega^2 / 2, omega^2, omega^2}
    double na[F];                             // -a
    double qw[F], pw[F];
    double p_eq[SCIVR_MAX_CHI][F], q_eq[SCIVR_MAX_CHI][F];
    alignas(16) double2 exp2t[64];
};

template <int F, int G>
struct WarpShared {
    using E = Geo<F, G>;
    alignas(16) double q[E::T][E::S3];        // zero-padded, as are qq, H and H3
    alignas(16) double qq[E::T][E::S4];
    alignas(16) double H[E::T][E::HT];        // -tau H
    alignas(16) double H3[E::T][E::HT];       // -tau times its cubic part
    double2 A[E::JOBS * E::AS];               // prefactor matrix per job
    double pj[F][E::JOBS], qj[F][E::JOBS];    // state per job (columns swizzled)
    double Sj[E::JOBS];                       // action per job
    double2 ov0[SCIVR_MAX_CHI][E::T];         // log of the Herman-Kluk summand's divisor
};

// A step's state on its way from the warp that propagates to the warp that records (two slots;
// a lane's values go to the same lane).
template <int F, int G>
struct Mail {
    double v[2][Geo<F, G>::MAIL][32];
};

// Named barriers of 64 threads: a pair of warps.
__device__ __forceinline__ void pair_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void pair_arrive(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }

// Column of job j in row r of the per-job arrays: a group's lanes store one job into different rows.
template <int JOBS>
__device__ __forceinline__ int swz(int r, int j) { return j ^ (r & (JOBS >= 16 ? 15 : JOBS - 1)); }

template <int N, typename Fn, int... Ks>
__device__ __forceinline__ void static_for_impl(Fn &&f, std::integer_sequence<int, Ks...>)
{
    (f(std::integral_constant<int, Ks>{}), ...);
}
template <int N, typename Fn>
__device__ __forceinline__ void static_for(Fn &&f)
{
    static_for_impl<N>(f, std::make_integer_sequence<int, N>{});
}

// w[s] for a run-time slot s < N (predicated moves; 0 past the end).
template <int N>
__device__ __forceinline__ double slot(const double (&w)[N], int s)
{
    double v = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i) v = s == i ? w[i] : v;
    return v;
}

// HELP: a second warp, on another sub-partition, makes the records (a quarter to a third of the
// instructions), for launches that leave half of the sub-partitions without a warp.  F = 3, 96
// trajectories x 400 steps, the whole FP64 run: 3.68 -> 2.93 ms (2.72 with the later Fourier step).
template <int F, int G, bool HELP>
__global__ void __launch_bounds__(32 * kMaxWarps, 1) k_propagate_g64(const PropLaunch L)
{
    using E = Geo<F, G>;
    constexpr int N2 = E::N2, P = E::P, T = E::T, C = E::C, JOBS = E::JOBS;
    constexpr int NC = E::NC, NM = E::NM, NE = E::NE, S3 = E::S3, S4 = E::S4, SH = E::SH;
    using Sh = WarpShared<F, G>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    CtaShared<F> &cs = *reinterpret_cast<CtaShared<F> *>(smem_raw);
    constexpr size_t cta_bytes = (sizeof(CtaShared<F>) + 15) & ~(size_t)15;

    const PesDev &pes = L.pes;
    const PropArgs &A = L.args;
    const bool use3 = pes.has3, use4 = pes.has4;
    for (int i = threadIdx.x; i < 2 * P * S3; i += blockDim.x) {
        const int kk = i / (P * S3), e = i / S3 % P, k = i % S3;
        (&cs.T3[0][0][0])[i] = use3 && k < F ? -A.tkick[kk] * pes.T3[k * P + e] : 0.0;
    }
    for (int i = threadIdx.x; i < 2 * P * S4; i += blockDim.x) {
        const int kk = i / (P * S4), e = i / S4 % P, kl = i % S4;
        (&cs.T4[0][0][0])[i] = use4 && kl < P ? -A.tkick[kk] * pes.T4[kl * P + e] : 0.0;
    }
    for (int i = threadIdx.x; i < 2 * F; i += blockDim.x) {
        const int kk = i / F, a = i % F;
        const double nt = -A.tkick[kk];
        const bool morse = pes.diag_kind == SCIVR_DIAG_MORSE;
        const double D = pes.D[a], al = pes.a[a], w2 = pes.omega[a] * pes.omega[a];
        cs.kD[kk][a] = nt * (morse ? D : 0.5 * w2);
        cs.kDa[kk][a] = nt * (morse ? 2.0 * D * al : w2);
        cs.kDaa[kk][a] = nt * (morse ? 2.0 * D * al * al : w2);
        cs.na[a] = -al;
        cs.qw[a] = A.qw[a];
        cs.pw[a] = A.pw[a];
    }
    for (int i = threadIdx.x; i < F * F; i += blockDim.x) {
        const int a = i / F, b = i % F;
        cs.acoef[i][0] = 0.5 * (A.rg[a] * A.irg[b]);
        cs.acoef[i][1] = 0.5 * (A.rg[b] * A.irg[a]);
        cs.acoef[i][2] = -0.5 * (A.rg[a] * A.rg[b]);
        cs.acoef[i][3] = 0.5 * (A.irg[a] * A.irg[b]);
    }
    for (int i = threadIdx.x; i < SCIVR_MAX_CHI * F; i += blockDim.x) {
        const bool on = i / F < A.n_chi;
        cs.p_eq[i / F][i % F] = on ? A.p_eq[i] : 0.0;
        cs.q_eq[i / F][i % F] = on ? A.q_eq[i] : 0.0;
    }
    for (int i = threadIdx.x; i < 64; i += blockDim.x) cs.exp2t[i] = kExp2Table[i];
    __syncthreads();

    const int warp = threadIdx.x >> 5, ln = threadIdx.x & 31;
    const int t = ln / G, g = ln % G, base = t * G;
    const int n_set = HELP ? blockDim.x >> 6 : blockDim.x >> 5;   // sets of T trajectories in the CTA
    const int set = HELP ? warp % n_set : warp;
    const bool advances = !HELP || warp < n_set, records = !HELP || warp >= n_set;
    Sh &sh = reinterpret_cast<Sh *>(smem_raw + cta_bytes)[set];
    Mail<F, G> &mail = reinterpret_cast<Mail<F, G> *>(smem_raw + cta_bytes + n_set * sizeof(Sh))[HELP ? set : 0];
    const int bar_full = 1 + 4 * set, bar_free = bar_full + 2;    // + slot
    if (advances) {
        // the rows' padding is multiplied by zero but never written: clear it once
        double *z = &sh.q[0][0];
        constexpr int nz = (int)(offsetof(Sh, A) / sizeof(double));
        for (int i = ln; i < nz; i += 32) z[i] = 0.0;
        __syncwarp();
    }
    const int64_t n = L.n_traj;
    const int64_t j_traj = ((int64_t)blockIdx.x * n_set + set) * T + t;
    const bool active = j_traj < n;
    const int64_t jl = active ? j_traj : n - 1;

    int ent[NE];   // this lane's Hessian entries e = g + i G as (a, b), a | b << 8
#pragma unroll
    for (int i = 0; i < NE; ++i) {
        int e = g + i * G, a = 0;
        if (e >= P) e = 0;
        while (e >= F - a) { e -= F - a; ++a; }
        ent[i] = a | ((a + e) << 8);
    }

    // modes g + s G: position and momentum; columns g + s G of M = d(p,q)/d(p0,q0), zero past 2F
    double p[NM], q[NM], S = 0.0;
    double Mp[NC][F], Mq[NC][F];
#pragma unroll
    for (int s = 0; s < NM; ++s) {
        const int a = g + s * G < F ? g + s * G : 0;
        p[s] = L.p0[a * n + jl];
        q[s] = L.q0[a * n + jl];
    }
#pragma unroll
    for (int s = 0; s < NC; ++s) {
        const int col = g + s * G;
#pragma unroll
        for (int a = 0; a < F; ++a) {
            Mp[s][a] = a == col ? 1.0 : 0.0;
            Mq[s][a] = a + F == col ? 1.0 : 0.0;
        }
    }
    bool good = true;
    double stab = 0.0, detM_last = 1.0, theta_last = 0.0, arg_last = 0.0;
    double2 detA_last = make_double2(1.0, 0.0);

    // amplitude at c = 0 (M = I, S = 0, theta = 0): a group's lanes take the reference states in turn
    if (records) {
        double re00 = 0.0;
        for (int x0 = 0; x0 < A.n_chi; x0 += G) {
            const int x = x0 + g, xc = x < A.n_chi ? x : 0;
            double re = 0.0, im = 0.0;
            for (int a = 0; a < F; ++a) {
                const double pa = L.p0[a * n + jl], qa = L.q0[a * n + jl];
                const double dq = cs.q_eq[xc][a] - qa, dp = cs.p_eq[xc][a] - pa;
                re = fma(-cs.qw[a] * dq, dq, re);
                re = fma(-cs.pw[a] * dp, dp, re);
                im = fma(0.5 * (cs.p_eq[xc][a] + pa), dq, im);
            }
            if (x0 == 0) re00 = __shfl_sync(FULL, re, base);
            // the Herman-Kluk summand divides by the initial overlap times the importance weight
            // of the sampling density, the first reference state's (chi_log_overlap0); at t = 0 it
            // is |<chi_x|p0 q0>|^2 / |<chi_0|p0 q0>|^2
            const double rdiv = x == 0 ? re : 2.0 * re00 - re;
            if (x < A.n_chi && active) {
                sh.ov0[x][t] = make_double2(rdiv, im);
                double sn, cs_;
                sincos(im, &sn, &cs_);
                const double mag = exp(re);
                const int64_t ia = x * L.chi_stride + jl * L.amp_ld;
                if (A.amplitude == SCIVR_AMP_HK) amp_store(L, ia, x == 0 ? 1.0 : exp(re - rdiv), 0.0);
                else amp_store(L, ia, mag * cs_, mag * sn);
            }
        }
        __syncwarp();
    }

    const int jc = g, jb = t * C + jc;   // this lane's job of a chunk: step jc of its trajectory
    for (int step0 = 0; step0 < A.n_steps; step0 += C) {
        const int cnt = min(C, A.n_steps - step0);
        for (int c = 0; c < cnt; ++c) {
            double dS = 0.0;   // this lane's share of the step's action increment
#pragma unroll 1
            for (int sub = advances ? 0 : 4; sub < 4; ++sub) {
                // drift: q += tau p, S += tau p.p / 2, M_q += tau M_p
                const double td = A.tdrift[sub], th = 0.5 * td;
#pragma unroll
                for (int s = 0; s < NM; ++s) {
                    q[s] = fma(td, p[s], q[s]);
                    if (g + s * G < F) dS = fma(th * p[s], p[s], dS);
                }
#pragma unroll
                for (int s = 0; s < NC; ++s)
#pragma unroll
                    for (int a = 0; a < F; ++a) Mq[s][a] = fma(td, Mp[s][a], Mq[s][a]);
                if (sub == 3) break;
                // kick at q, every force term times -tau
                const int kk = sub == 1;
                __syncwarp();   // the previous kick's readers of H are done
#pragma unroll
                for (int s = 0; s < NM; ++s)
                    if (g + s * G < F) sh.q[t][g + s * G] = q[s];
                __syncwarp();
                if (use3 || use4) {
#pragma unroll
                    for (int i = 0; i < NE; ++i)
                        if (g + i * G < P) sh.qq[t][g + i * G] = sh.q[t][ent[i] & 255] * sh.q[t][ent[i] >> 8];
                    __syncwarp();
                    double h[NE];
                    const double *r3[NE], *r4[NE];
#pragma unroll
                    for (int i = 0; i < NE; ++i) {
                        const int e = g + i * G < P ? g + i * G : 0;
                        r3[i] = cs.T3[kk][e];
                        r4[i] = cs.T4[kk][e];
                        h[i] = 0.0;
                    }
                    if (use3) {
#pragma unroll
                        for (int k = 0; k < F; k += 2) {
                            const double2 x = *reinterpret_cast<const double2 *>(&sh.q[t][k]);
#pragma unroll
                            for (int i = 0; i < NE; ++i) {
                                const double2 w = *reinterpret_cast<const double2 *>(r3[i] + k);
                                h[i] = fma(w.x, x.x, h[i]);
                                if (k + 1 < F) h[i] = fma(w.y, x.y, h[i]);
                            }
                        }
                    }
#pragma unroll
                    for (int i = 0; i < NE; ++i)
                        if (g + i * G < P) {
                            const int a = ent[i] & 255, b = ent[i] >> 8;
                            sh.H3[t][a * SH + b] = h[i];
                            sh.H3[t][b * SH + a] = h[i];
                        }
                    if (use4) {
#pragma unroll 4
                        for (int k = 0; k < P; k += 2) {
                            const double2 x = *reinterpret_cast<const double2 *>(&sh.qq[t][k]);
#pragma unroll
                            for (int i = 0; i < NE; ++i) {
                                const double2 w = *reinterpret_cast<const double2 *>(r4[i] + k);
                                h[i] = fma(w.x, x.x, h[i]);
                                if (P % 2 == 0 || k + 1 < P) h[i] = fma(w.y, x.y, h[i]);
                            }
                        }
                    }
#pragma unroll
                    for (int i = 0; i < NE; ++i)
                        if (g + i * G < P) {
                            const int a = ent[i] & 255, b = ent[i] >> 8;
                            sh.H[t][a * SH + b] = h[i];
                            sh.H[t][b * SH + a] = h[i];
                        }
                    __syncwarp();
                }
                // gradient, momentum and action (modes).  By Euler's theorem with s = H q and s3 = H3 q:
                // grad V_c = s / 3 + s3 / 6 and V_c = q.(s + s3) / 12.
#pragma unroll
                for (int s = 0; s < NM; ++s) {
                    const int a = g + s * G;
                    if (a < F) {
                        const double qa = q[s];
                        double gd, hd;   // the separable diagonal's gradient and Hessian
                        if (pes.diag_kind == SCIVR_DIAG_MORSE) {
                            const double u = exp_t(cs.na[a] * qa, cs.exp2t);
                            const double omu = 1.0 - u;
                            dS = fma(cs.kD[kk][a] * omu, omu, dS);
                            gd = cs.kDa[kk][a] * (u * omu);
                            hd = cs.kDaa[kk][a] * u * fma(2.0, u, -1.0);
                        } else {
                            dS = fma(cs.kD[kk][a] * qa, qa, dS);
                            gd = cs.kDa[kk][a] * qa;
                            hd = cs.kDaa[kk][a];
                        }
                        if (use3 || use4) {
                            double sa = 0.0, s3 = 0.0;
#pragma unroll
                            for (int b = 0; b < F; b += 2) {
                                const double2 x = *reinterpret_cast<const double2 *>(&sh.q[t][b]);
                                const double2 hv = *reinterpret_cast<const double2 *>(&sh.H[t][a * SH + b]);
                                const double2 h3 = *reinterpret_cast<const double2 *>(&sh.H3[t][a * SH + b]);
                                sa = fma(hv.x, x.x, sa);
                                s3 = fma(h3.x, x.x, s3);
                                if (b + 1 < F) {
                                    sa = fma(hv.y, x.y, sa);
                                    s3 = fma(h3.y, x.y, s3);
                                }
                            }
                            gd = fma(1.0 / 3.0, sa, fma(1.0 / 6.0, s3, gd));
                            dS = fma(qa * (1.0 / 12.0), sa + s3, dS);
                            sh.H[t][a * SH + a] += hd;
                        } else {
                            sh.H[t][a * SH + a] = hd;
                        }
                        p[s] += gd;
                    }
                }
                __syncwarp();   // H complete
                // monodromy kick: M_p -= tau H M_q
#pragma unroll
                for (int a = 0; a < F; ++a)
#pragma unroll
                    for (int b = 0; b < F; b += 2) {
                        const double2 hv = *reinterpret_cast<const double2 *>(&sh.H[t][a * SH + b]);
#pragma unroll
                        for (int s = 0; s < NC; ++s) {
                            Mp[s][a] = fma(hv.x, Mq[s][b], Mp[s][a]);
                            if (b + 1 < F) Mp[s][a] = fma(hv.y, Mq[s][b + 1], Mp[s][a]);
                        }
                    }
            }
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) dS += __shfl_xor_sync(FULL, dS, o);
            S += dS;
            if constexpr (HELP) {
                const int step = step0 + c, sl = step & 1;
                auto pass = [&](auto &&move) {
                    int k = 0;
#pragma unroll
                    for (int s = 0; s < NC; ++s)
#pragma unroll
                        for (int a = 0; a < F; ++a) {
                            move(Mp[s][a], mail.v[sl][k++][ln]);
                            move(Mq[s][a], mail.v[sl][k++][ln]);
                        }
#pragma unroll
                    for (int s = 0; s < NM; ++s) {
                        move(p[s], mail.v[sl][k++][ln]);
                        move(q[s], mail.v[sl][k++][ln]);
                    }
                    move(S, mail.v[sl][k][ln]);
                };
                if (advances) {
                    if (step >= 2) pair_sync(bar_free + sl);
                    pass([](double &x, double &m) { m = x; });
                    pair_arrive(bar_full + sl);
                    continue;
                }
                pair_sync(bar_full + sl);
                pass([](double &x, double &m) { x = m; });
                if (step + 2 < A.n_steps) pair_arrive(bar_free + sl);
            }
            // ---- stability: det M = det M^T by Gaussian elimination of M^T with partial pivoting ----
            // Column c of M is row c of M^T, held by lane c % G in slot c / G.  Stage k picks the unused
            // row of the largest |entry k| (keys: the leading bits of the magnitude, then the row), and
            // the other unused rows subtract their multiples of it.  Rows stay in place; the sign is the
            // parity of the order in which they are picked.
            {
                double W[NC][N2], pv[NC];
#pragma unroll
                for (int s = 0; s < NC; ++s) {
                    pv[s] = 1.0;
#pragma unroll
                    for (int a = 0; a < F; ++a) { W[s][a] = Mp[s][a]; W[s][F + a] = Mq[s][a]; }
                }
                unsigned unused = (1u << N2) - 1u, parity = 0u;
                static_for<N2>([&](auto kc) {
                    constexpr int k = decltype(kc)::value;
                    unsigned key = 0u;
#pragma unroll
                    for (int s = 0; s < NC; ++s) {
                        const int col = g + s * G;
                        const unsigned kv = ((unsigned)mag_key(W[s][k]) & ~31u) | (unsigned)(col + 1);
                        if (col < N2 && ((unused >> col) & 1u)) key = max(key, kv);
                    }
#pragma unroll
                    for (int o = 1; o < G; o <<= 1) key = max(key, __shfl_xor_sync(FULL, key, o));
                    const int pc = (int)(key & 31u) - 1;
                    const int pl = base + pc % G, ps = pc / G;
                    parity ^= (unsigned)__popc(unused & ((1u << pc) - 1u)) & 1u;
                    unused &= ~(1u << pc);
                    auto pivot_row = [&](int i) -> double {
                        double col_i[NC];
#pragma unroll
                        for (int s = 0; s < NC; ++s) col_i[s] = W[s][i];
                        return __shfl_sync(FULL, slot<NC>(col_i, ps), pl);
                    };
                    const double pk = pivot_row(k);
                    double l[NC];
                    if constexpr (k + 1 < N2) {
                        const double inv = recip(pk);
#pragma unroll
                        for (int s = 0; s < NC; ++s) l[s] = W[s][k] * inv;
                    }
#pragma unroll
                    for (int s = 0; s < NC; ++s) {
                        const int col = g + s * G;
                        if (col == pc) pv[s] = pk;
                    }
                    // (used rows are updated along: nothing reads them again)
#pragma unroll
                    for (int i = k + 1; i < N2; ++i) {
                        const double wp = pivot_row(i);
#pragma unroll
                        for (int s = 0; s < NC; ++s) W[s][i] = fma(-l[s], wp, W[s][i]);
                    }
                });
                double det = pv[0];
#pragma unroll
                for (int s = 1; s < NC; ++s) det *= pv[s];
#pragma unroll
                for (int o = 1; o < G; o <<= 1) det *= __shfl_xor_sync(FULL, det, o);
                if (parity) det = -det;
                // deviations are non-negative or NaN: ordered as integers (NaN above infinity)
                const double dev = finite_bits(det) ? fabs(fma(det, det, -1.0)) : CUDART_INF;
                if (__double_as_longlong(dev) > __double_as_longlong(stab)) stab = dev;
                if (dev > A.stab_tol) good = false;
                if (c == cnt - 1) detM_last = det;
            }
            // ---- Herman-Kluk matrix columns b = g + s G (each needs column F + b) ----
            const int job = t * C + c;
#pragma unroll
            for (int s = 0; s < NM; ++s) {
                // column F + b sits in lane (F + g) % G; a sending lane h is asked for it by one lane
                // only, the slot being one further where F % G wraps around
                constexpr int f0 = F / G, fr = F % G;
                const int src = base + (F + g) % G, from = s + f0 + (g < fr ? 1 : 0);
                const int b = g + s * G;
#pragma unroll
                for (int a = 0; a < F; ++a) {
                    double sp[NC], sq[NC];
#pragma unroll
                    for (int i = 0; i < NC; ++i) { sp[i] = Mp[i][a]; sq[i] = Mq[i][a]; }
                    const double mpq = __shfl_sync(FULL, slot<NC>(sp, from), src);
                    const double mqq = __shfl_sync(FULL, slot<NC>(sq, from), src);
                    if (b < F) {
                        const double2 k0 = *reinterpret_cast<const double2 *>(&cs.acoef[a * F + b][0]);
                        const double2 k1 = *reinterpret_cast<const double2 *>(&cs.acoef[a * F + b][2]);
                        sh.A[job * E::AS + a * F + b] = make_double2(fma(k0.x, mqq, k0.y * Mp[s][a]),
                                                                     fma(k1.x, Mq[s][a], k1.y * mpq));
                    }
                }
                if (b < F) {
                    sh.pj[b][swz<JOBS>(b, job)] = p[s];
                    sh.qj[b][swz<JOBS>(b, job)] = q[s];
                }
            }
            if (g == 0) sh.Sj[job] = S;
        }
        if (!records) continue;
        {
            // non-finite state persists, so testing once per chunk marks the same trajectories
            bool fin = true;
#pragma unroll
            for (int s = 0; s < NM; ++s) fin = fin && finite_bits(p[s]) && finite_bits(q[s]);
            const unsigned bad = __ballot_sync(FULL, !fin);
            if (bad & (G == 32 ? FULL : ((1u << (G & 31)) - 1u) << base)) good = false;
        }
        __syncwarp();
        // ---------------- det A per job: elimination in place, one lane per job ----------------
        const bool jvalid = jc < cnt;
        double argA = 0.0;
        double2 detA = make_double2(1.0, 0.0);
        if (jvalid) {
            double2 *Aj = &sh.A[jb * E::AS];
            double dr = 1.0, di = 0.0;
#pragma unroll 1
            for (int k = 0; k < F; ++k) {
                // pivot by max(|re|, |im|), within a factor sqrt(2) of |z|
                int piv = k, best = -1;
                for (int i = k; i < F; ++i) {
                    const double2 v = Aj[i * F + k];
                    const int m = max(mag_key(v.x), mag_key(v.y));
                    if (m > best) { best = m; piv = i; }
                }
                if (piv != k) {
                    for (int cc = k; cc < F; ++cc) {
                        const double2 v = Aj[piv * F + cc];
                        Aj[piv * F + cc] = Aj[k * F + cc];
                        Aj[k * F + cc] = v;
                    }
                    dr = -dr;
                    di = -di;
                }
                const double2 pk = Aj[k * F + k];
                const double nr = fma(dr, pk.x, -di * pk.y), ni = fma(dr, pk.y, di * pk.x);
                dr = nr;
                di = ni;
                const double rr = recip(fma(pk.x, pk.x, pk.y * pk.y));
                const double ir = pk.x * rr, ii = -pk.y * rr;
                for (int i = k + 1; i < F; ++i) {
                    const double2 v = Aj[i * F + k];
                    const double lr = fma(v.x, ir, -v.y * ii), li = fma(v.x, ii, v.y * ir);
#pragma unroll 2
                    for (int cc = k + 1; cc < F; ++cc) {
                        const double2 pr = Aj[k * F + cc];
                        double2 x = Aj[i * F + cc];
                        x.x = fma(-lr, pr.x, fma(li, pr.y, x.x));
                        x.y = fma(-lr, pr.y, fma(-li, pr.x, x.y));
                        Aj[i * F + cc] = x;
                    }
                }
            }
            detA = make_double2(dr, di);
            argA = atan2(di, dr);
        }
        // ---------------- continuous phase: segmented scan over the group's steps ----------------
        double arg_prev = __shfl_up_sync(FULL, argA, 1, G);
        if (g == 0) arg_prev = arg_last;
        double d = argA - arg_prev + A.ref_step;
        d = fma(-kTwoPi, rint(d * kInvTwoPi), d);
        double inc = jvalid ? d - A.ref_step : 0.0;
#pragma unroll
        for (int o = 1; o < C; o <<= 1) {
            const double v = __shfl_up_sync(FULL, inc, o, G);
            if (g >= o) inc += v;
        }
        const double theta = theta_last + inc;
        const int lastlane = base + cnt - 1;
        theta_last = __shfl_sync(FULL, theta, lastlane);
        arg_last = __shfl_sync(FULL, argA, lastlane);
        detA_last.x = __shfl_sync(FULL, detA.x, lastlane);
        detA_last.y = __shfl_sync(FULL, detA.y, lastlane);
        if (!finite_bits(theta_last)) good = false;
        // ---------------- amplitudes ----------------
        if (jvalid && active) {
            const double Sc = sh.Sj[jb];
            const double lnA = A.amplitude == SCIVR_AMP_HK ? 0.5 * log(hypot(detA.x, detA.y)) : 0.0;   // the same for every state
            for (int x = 0; x < A.n_chi; ++x) {
                double re = 0.0, im = 0.0;
#pragma unroll
                for (int a = 0; a < F; ++a) {
                    const double pa = sh.pj[a][swz<JOBS>(a, jb)], qa = sh.qj[a][swz<JOBS>(a, jb)];
                    const double dq = cs.q_eq[x][a] - qa, dp = cs.p_eq[x][a] - pa;
                    re = fma(-cs.qw[a] * dq, dq, re);
                    re = fma(-cs.pw[a] * dp, dp, re);
                    im = fma(0.5 * (cs.p_eq[x][a] + pa), dq, im);
                }
                double ph = im + Sc + 0.5 * theta;
                if (A.amplitude == SCIVR_AMP_HK) {
                    const double2 o = sh.ov0[x][t];
                    re = re - o.x + lnA;
                    ph -= o.y;
                }
                double sn, cs_;
                sincos(ph, &sn, &cs_);
                const double mag = exp_t(re, cs.exp2t);
                amp_store(L, x * L.chi_stride + jl * L.amp_ld + step0 + jc + 1, mag * cs_, mag * sn);
            }
        }
        if (!finite_bits(S)) good = false;
        __syncwarp();
    }

    if (!active || !records) return;
    if (g == 0) L.good[jl] = good ? 1 : 0;
    const FinalDev &fo = L.fin;
#pragma unroll
    for (int s = 0; s < NM; ++s) {
        const int a = g + s * G;
        if (a < F && fo.p) fo.p[a * n + jl] = p[s];
        if (a < F && fo.q) fo.q[a * n + jl] = q[s];
    }
    if (g == 0) {
        if (fo.S) fo.S[jl] = S;
        if (fo.theta) fo.theta[jl] = theta_last;
        if (fo.detM) fo.detM[jl] = detM_last;
        if (fo.stab) fo.stab[jl] = stab;
        if (fo.detA) { fo.detA[2 * jl] = detA_last.x; fo.detA[2 * jl + 1] = detA_last.y; }
    }
    if (fo.M) {
#pragma unroll
        for (int s = 0; s < NC; ++s) {
            const int col = g + s * G;
            if (col < N2) {
#pragma unroll
                for (int a = 0; a < F; ++a) {
                    fo.M[jl * N2 * N2 + a * N2 + col] = Mp[s][a];
                    fo.M[jl * N2 * N2 + (F + a) * N2 + col] = Mq[s][a];
                }
            }
        }
    }
}

// Sets of T trajectories per CTA: up to four warps, fewer where fewer spread over all SMs.
template <int F, int G, bool HELP>
cudaError_t launch(const PropLaunch &L, int n_sm, cudaStream_t s)
{
    using E = Geo<F, G>;
    constexpr int most = HELP ? kMaxWarps / 2 : kMaxWarps;
    const int64_t sets = (L.n_traj + E::T - 1) / E::T;
    const int W = sets >= (int64_t)most * n_sm ? most : (int)((sets + n_sm - 1) / n_sm);
    constexpr size_t cta_bytes = (sizeof(CtaShared<F>) + 15) & ~(size_t)15;
    constexpr size_t set_bytes = sizeof(WarpShared<F, G>) + (HELP ? sizeof(Mail<F, G>) : 0);
    static_assert(sizeof(WarpShared<F, G>) % 16 == 0 && sizeof(Mail<F, G>) % 16 == 0, "the sets' shared blocks stay aligned");
    static_assert(cta_bytes + most * set_bytes <= 227 * 1024, "four warps fit an SM");
    auto kern = k_propagate_g64<F, G, HELP>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(cta_bytes + most * set_bytes));
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((sets + W - 1) / W), (HELP ? 64 : 32) * W, cta_bytes + W * set_bytes, s>>>(L);
    return cudaGetLastError();
}

// The narrowest group a lane's registers allow (its columns and their copy for det M).
constexpr int min_lanes(int F) { return F <= 1 ? 2 : F <= 6 ? 4 : 8; }
// The widest that still saves instructions where a warp records (at F = 1 beyond two lanes only those of
// several reference states: eight states, 64 steps of 600 harmonic trajectories 0.61 -> 0.24 ms).
constexpr int max_lanes(int F) { return F <= 1 ? 8 : F == 2 ? 4 : F == 3 ? 8 : F <= 5 ? 16 : 32; }

}  // namespace g64

// Group size: the fewest FP64 instructions over the rounds of four warps per SM that the
// trajectories take; with a recording warp where two per SM suffice.
template <int F, int G = g64::min_lanes(F)>
void choose_g64_lanes(int64_t n_traj, int n_chi, int n_sm, double &best, int &lanes, bool &help)
{
    using E = g64::Geo<F, G>;
    const int64_t warps = (n_traj * G + 31) / 32, slots = (int64_t)g64::kMaxWarps * n_sm;
    const bool h = 2 * warps <= slots;
    const int step = E::kStepInstr, record = E::kRecordInstr + (F == 1 ? (n_chi - 1) * E::kStateInstr : 0);
    const int instr = !h ? step + record : step > record ? step : record;
    const double cost = (double)((warps + slots - 1) / slots) * instr;
    if (lanes == 0 || cost < best) { best = cost; lanes = G; help = h; }
    if constexpr (G < g64::max_lanes(F)) choose_g64_lanes<F, 2 * G>(n_traj, n_chi, n_sm, best, lanes, help);
}

template <int F, int G = g64::min_lanes(F)>
cudaError_t launch_g64_lanes(const PropLaunch &L, int lanes, bool help, int n_sm, cudaStream_t s)
{
    if (lanes == G) return help ? g64::launch<F, G, true>(L, n_sm, s) : g64::launch<F, G, false>(L, n_sm, s);
    if constexpr (G < g64::max_lanes(F)) return launch_g64_lanes<F, 2 * G>(L, lanes, help, n_sm, s);
    return cudaErrorInvalidValue;
}

template <int F> cudaError_t launch_group_fp64(const PropLaunch &L, cudaStream_t s)
{
    int dev = 0, n_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    double cost = 0.0;
    int lanes = 0;
    bool help = false;
    choose_g64_lanes<F>(L.n_traj, L.args.n_chi, n_sm, cost, lanes, help);
    return launch_g64_lanes<F>(L, lanes, help, n_sm, s);
}

}  // namespace scivr
