// Propagation on a potential with a learned residual (Sec. III.A schedule,
// split into stages so that every force evaluation of the network is one
// batched tensor-core evaluation over all trajectories).
//
// Per step of the fourth-order triple jump  D(c0) K(d0) D(c1) K(d1) D(c2) K(d2) D(c3):
//   network at q  ->  k_mlp_kick, stage 1: K(d0) D(c1)
//   network at q  ->  k_mlp_kick, stage 2: K(d1) D(c2)
//   network at q  ->  k_mlp_kick, stage 3: K(d2) D(c3), det M (stability), and D(c0) of
//                     the next step for q and S
//                     k_mlp_record: det A and the continuous phase, the amplitude of
//                     Eq. I(E)_discreto
// k_mlp_start (before the first step) sets M = I, records c = 0 and drifts q by D(c0); M
// is drifted by D(c0) when stage 1 reads it.  A kick uses V, grad V and the Hessian of the
// analytic surface (FP64, at q) plus those of the network (FP32, at q rounded to FP32).  State
// between stages lives in HBM: p, q, S, theta (FP64, structure of arrays) and M (FP32,
// element (r, c) of trajectory j at (r 2F + c) n + j).
#include "fp64_ops.cuh"
#include "propagate_tpt.cuh"

namespace scivr {
namespace pm {

struct State {
    double *p, *q;        // [F][n]
    float *M;             // [(2F)^2][n]
    double *S, *theta, *arg_old, *stab;
    double *qe, *Se;      // [F][n], [n]: q and S at the end of the step (q and S are a drift ahead)
    float *det;           // [n] det M
    float *qf;            // [n][F] network input
    const float *Vm, *gm, *Hm;   // network output at qf: [n], [n][F], [n][F][F]
    int *step;            // device step counter (column of the amplitude)
};

// Amplitude of step `step` for every reference state: the time-averaged summand,
// or with SCIVR_AMP_HK the Herman-Kluk summand (|det A|^{1/2} = sqrt(absA), divided
// by the initial overlap times the sampling weight, chi_log_overlap0).
template <int F>
__device__ __forceinline__ void record(const PropLaunch &L, int64_t j, int step, const double (&p)[F],
                                       const double (&q)[F], double S, double theta, double absA)
{
    const PropArgs &A = L.args;
    double re00 = 0.0;   // Re log <chi_0|p0 q0>, set by the x = 0 iteration (Herman-Kluk summand)
    for (int x = 0; x < A.n_chi; ++x) {
        double re = 0.0, im = 0.0;
#pragma unroll
        for (int a = 0; a < F; ++a) {
            const double dq = A.q_eq[x * F + a] - q[a];
            const double dp = A.p_eq[x * F + a] - p[a];
            re = fma(-A.qw[a] * dq, dq, re);
            re = fma(-A.pw[a] * dp, dp, re);
            im = fma(0.5 * (A.p_eq[x * F + a] + p[a]), dq, im);
        }
        double ph = im + S + 0.5 * theta;
        if (A.amplitude == SCIVR_AMP_HK) {
            double re0, im0;
            chi_log_overlap0<F>(A, L.p0, L.q0, L.n_traj, j, x, re00, re0, im0);
            re = re - re0 + 0.5 * log(absA);
            ph -= im0;
        }
        double sn, cs;
        sincos(ph, &sn, &cs);
        const double mag = exp(re);
        amp_store(L, x * L.chi_stride + j * L.amp_ld + step, mag * cs, mag * sn);
    }
}

// Set-up: M = I, the record of c = 0, the first drift of q and S.
template <int F>
__global__ void __launch_bounds__(128) k_mlp_start(const PropLaunch L, State st)
{
    constexpr int N2 = 2 * F;
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t n = L.n_traj;
    const PropArgs &A = L.args;
    if (j >= n) return;
    double p[F], q[F];
#pragma unroll
    for (int a = 0; a < F; ++a) {
        p[a] = L.p0[a * n + j];
        q[a] = L.q0[a * n + j];
    }
    st.theta[j] = 0.0;
    st.arg_old[j] = 0.0;
    st.stab[j] = 0.0;
    L.good[j] = 1;
    record<F>(L, j, 0, p, q, 0.0, 0.0, 1.0);
    for (int e = 0; e < N2 * N2; ++e) st.M[(int64_t)e * n + j] = e % (N2 + 1) == 0 ? 1.0f : 0.0f;
    double kin = 0.0;
#pragma unroll
    for (int a = 0; a < F; ++a) {
        kin = fma(0.5 * p[a], p[a], kin);
        const double qa = fma(A.tdrift[0], p[a], q[a]);
        st.p[a * n + j] = p[a];
        st.q[a * n + j] = qa;
        st.qf[j * F + a] = (float)qa;
    }
    st.S[j] = A.tdrift[0] * kin;
}

// One kick and the drift after it for 32 trajectories (a lane each) by F warps: warp b has mode b
// and columns b and F + b of M in registers.  LAST: the step's last stage, which forms det M and
// drifts q and S ahead by the next step's first drift.  COUPLED: the analytic part has coupling terms
// (else it is the separable diagonal alone).
//
// What bounded the thread-per-trajectory form: 512 warps at 16384 trajectories, each with 324
// dependent loads and stores of M, uncoalesced reads of the network's Hessian, 360 FP64 pipe slots,
// and at the last stage det M's 2109 updates through shared memory.  With a warp per mode the FP64
// work of a trajectory spreads over the SM's four pipes, all of a column is loaded at once, the
// Hessian arrives coalesced through shared memory and det M runs in registers, its pivot column
// passed through shared memory.
// F = 9, 16384 trajectories: 38 -> 24 us
// a kick, 39 with det M; three CTAs per SM (with two the det M stages' barriers take 18 us longer).
template <int F, bool COUPLED, bool LAST>
__global__ void __launch_bounds__(32 * F, 3) k_mlp_kick(const PropLaunch L, State st, int stage)
{
    constexpr int N2 = 2 * F, FF = F * F, P = F * (F + 1) / 2, NT = 32 * F;
    const int lane = threadIdx.x & 31, b = threadIdx.x >> 5;
    const int64_t n = L.n_traj, j0 = (int64_t)blockIdx.x * 32, j = j0 + lane;
    const bool on = j < n;
    const int64_t jl = on ? j : n - 1;
    const PropArgs &A = L.args;
    __shared__ float Hk[FF][33];                 // tau H
    __shared__ double inc[F][32], inc2[F][32];   // the modes' shares of the action
    __shared__ double2 exp2t[64];
    __shared__ double qs[COUPLED ? F : 1][32], gc[COUPLED ? P : 1][32];
    __shared__ unsigned keys[LAST ? F : 1][32];
    __shared__ float piv[LAST ? N2 : 1][32];
    if (stage == 1 && blockIdx.x == 0 && threadIdx.x == 0) *st.step += 1;   // read by k_mlp_record of this step

    float m[2][N2];   // columns b and F + b
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int r = 0; r < N2; ++r) m[s][r] = st.M[((int64_t)r * N2 + s * F + b) * n + jl];
    const double tk = A.tkick[stage - 1], td = A.tdrift[stage];
    const float tkf = A.tkick_f[stage - 1], tdf = A.tdrift_f[stage];
    double p = st.p[b * n + jl], q = st.q[b * n + jl];
    const float gm = st.gm[jl * F + b];
    {
        const int64_t total = n * FF;   // the tile's Hessians, contiguous: F values a thread
        float h[F];
#pragma unroll
        for (int k = 0; k < F; ++k) {
            const int64_t e = j0 * FF + threadIdx.x + k * NT;
            h[k] = e < total ? st.Hm[e] : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < F; ++k) {
            const int i = threadIdx.x + k * NT;
            Hk[i % FF][i / FF] = tkf * h[k];
        }
    }
    for (int i = threadIdx.x; i < 64; i += NT) exp2t[i] = kExp2Table[i];
    if constexpr (COUPLED) qs[b][lane] = q;
    __syncthreads();
    // the separable diagonal: value, gradient, Hessian of mode b
    double Va, ga, ha;
    if (L.pes.diag_kind == SCIVR_DIAG_MORSE) {
        const double Dm = __ldg(L.pes.D + b), am = __ldg(L.pes.a + b);
        const double u = exp_t(-am * q, exp2t);
        const double omu = 1.0 - u, c = 2.0 * Dm * am;
        Va = Dm * omu * omu;
        ga = c * (u * omu);
        ha = c * am * u * fma(2.0, u, -1.0);
    } else {
        const double w2 = __ldg(L.pes.omega + b) * __ldg(L.pes.omega + b);
        Va = 0.5 * w2 * q * q;
        ga = w2 * q;
        ha = w2;
    }
    if constexpr (COUPLED) {
        // coupling entries e = (b, b) and every F-th of the others
        auto entry = [&](int e, int r, int c) {
            double h3 = 0.0, h4 = 0.0;
            if (L.pes.has3)
                for (int k = 0; k < F; ++k) h3 = fma(__ldg(L.pes.T3 + k * P + e), qs[k][lane], h3);
            if (L.pes.has4) {
                int kl = 0;
                for (int k = 0; k < F; ++k) {
                    double t = 0.0;   // sum over l of T4[(k, l)][e] q_l
                    for (int l = k; l < F; ++l, ++kl) t = fma(__ldg(L.pes.T4 + kl * P + e), qs[l][lane], t);
                    h4 = fma(t, qs[k][lane], h4);
                }
            }
            gc[e][lane] = fma(0.5, h3, h4 * (1.0 / 3.0));
            const double vc = fma(1.0 / 6.0, h3, h4 * (1.0 / 12.0));
            Va = fma((r == c ? vc : 2.0 * vc) * qs[r][lane], qs[c][lane], Va);
            const double h = r == c ? h3 + h4 + ha : h3 + h4;
            const float hf = (float)(tk * h);
            Hk[r * F + c][lane] += hf;
            if (r != c) Hk[c * F + r][lane] += hf;
        };
        int turn = 0;
        for (int r = 0, e = 0; r < F; ++r)
            for (int c = r; c < F; ++c, ++e) {
                if (r == c) {
                    if (r == b) entry(e, r, c);
                } else {
                    if (turn == b) entry(e, r, c);
                    turn = turn + 1 == F ? 0 : turn + 1;
                }
            }
        __syncthreads();
        for (int c = 0; c < F; ++c) {
            const int lo = b < c ? b : c, hi = b < c ? c : b;
            ga = fma(gc[lo * F - lo * (lo - 1) / 2 + hi - lo][lane], qs[c][lane], ga);
        }
    } else {
        Hk[b * F + b][lane] += (float)(tk * ha);
    }
    p = fma(-tk, ga + widen(gm), p);
    const double kin = 0.5 * p * p;
    inc[b][lane] = fma(td, kin, -tk * Va);
    if constexpr (LAST) inc2[b][lane] = A.tdrift[0] * kin;
    q = fma(td, p, q);
    if (on) {
        st.p[b * n + j] = p;
        double qn = q;
        if constexpr (LAST) {
            st.qe[b * n + j] = q;
            qn = fma(A.tdrift[0], p, q);
        }
        st.q[b * n + j] = qn;
        st.qf[j * F + b] = (float)qn;
    }
    __syncthreads();
    if (b == 0 && on) {
        double d = -tk * widen(st.Vm[j]);
#pragma unroll
        for (int a = 0; a < F; ++a) d += inc[a][lane];
        double S = st.S[j] + d;
        if constexpr (LAST) {
            st.Se[j] = S;
            double d2 = 0.0;
#pragma unroll
            for (int a = 0; a < F; ++a) d2 += inc2[a][lane];
            S += d2;
        }
        st.S[j] = S;
    }
    // M: the step's first drift (stage 1), the kick M_p -= tk H M_q, the drift M_q += td M_p
    if (stage == 1) {
        const float td0 = A.tdrift_f[0];
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int a = 0; a < F; ++a) m[s][F + a] = fmaf(td0, m[s][a], m[s][F + a]);
    }
#pragma unroll 1
    for (int a = 0; a < F; ++a) {   // M_p turns by one place an iteration: F turns restore it
        float h0 = 0.0f, h1 = 0.0f;
#pragma unroll
        for (int c = 0; c < F; ++c) {
            const float h = Hk[a * F + c][lane];
            h0 = fmaf(h, m[0][F + c], h0);
            h1 = fmaf(h, m[1][F + c], h1);
        }
        const float n0 = m[0][0] - h0, n1 = m[1][0] - h1;
#pragma unroll
        for (int c = 0; c + 1 < F; ++c) {
            m[0][c] = m[0][c + 1];
            m[1][c] = m[1][c + 1];
        }
        m[0][F - 1] = n0;
        m[1][F - 1] = n1;
    }
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int a = 0; a < F; ++a) m[s][F + a] = fmaf(tdf, m[s][a], m[s][F + a]);
    if (on) {
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int r = 0; r < N2; ++r) st.M[((int64_t)r * N2 + s * F + b) * n + j] = m[s][r];
    }
    if constexpr (LAST) {
        // det M = det M^T by Gaussian elimination with partial pivoting: column c of M is row c of
        // M^T.  A stage picks the unused row of the largest leading entry (keys: the leading bits of the
        // magnitude, then the row); its entries reach the other warps through piv.  Rows move up by
        // one place a stage (the entries that come in are never part of the result).
        float det = 1.0f;
        unsigned unused = (1u << N2) - 1u, parity = 0u;
#pragma unroll 1
        for (int k = 0; k < N2; ++k) {
            unsigned key = 0u;
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int col = s * F + b;
                const unsigned kv = (__float_as_uint(fabsf(m[s][0])) & ~31u) | (unsigned)(col + 1);
                if ((unused >> col) & 1u) key = max(key, kv);
            }
            keys[b][lane] = key;
            __syncthreads();
#pragma unroll
            for (int a = 0; a < F; ++a) key = max(key, keys[a][lane]);
            const int pc = (int)(key & 31u) - 1;
            parity ^= (unsigned)__popc(unused & ((1u << pc) - 1u)) & 1u;
            unused &= ~(1u << pc);
#pragma unroll
            for (int s = 0; s < 2; ++s)
                if (pc == s * F + b) {
#pragma unroll
                    for (int i = 0; i < N2; ++i) piv[i][lane] = m[s][i];
                }
            __syncthreads();
            const float pk = piv[0][lane];
            det *= pk;
            const float inv = 1.0f / pk;
            const float l0 = m[0][0] * inv, l1 = m[1][0] * inv;
#pragma unroll
            for (int i = 1; i < N2; ++i) {   // (used rows are updated along: nothing reads them again)
                const float w = piv[i][lane];
                m[0][i - 1] = fmaf(-l0, w, m[0][i]);
                m[1][i - 1] = fmaf(-l1, w, m[1][i]);
            }
        }
        if (b == 0 && on) st.det[j] = parity ? -det : det;
    }
}

// The records of a step, a thread per trajectory: stability flag, det A (FP64, complex LU with
// partial pivoting in shared memory), the continuous phase, the amplitude.  Bounded by the FP64
// pipe: a warp's instructions there take 64 cycles each, about 1700 of them at F = 9 (1200 in the
// elimination, 324 to form A).  They were 3400 before the coefficients of A were formed once per
// CTA, FP32 entries widened and pivots compared as integers and divisions and atan2 replaced.  The
// loads of M are issued a row pair ahead (each waited for in turn, they took 130 us).
// Four warps per CTA, one for each sub-partition (single-warp CTAs share them unevenly).  F = 9, 16384
// trajectories: 74 us; the last kick, det M and the records together 178 -> 113 us.
constexpr int kRecThreads = 128;

template <int F>
__global__ void __launch_bounds__(kRecThreads) k_mlp_record(const PropLaunch L, State st)
{
    constexpr int N2 = 2 * F, NT = kRecThreads;
    extern __shared__ __align__(16) uint8_t rec_smem[];
    double4 *coef = reinterpret_cast<double4 *>(rec_smem);                       // [F * F]
    double2 *Z = reinterpret_cast<double2 *>(rec_smem + sizeof(double4) * F * F) + threadIdx.x;   // (a, b) at Z[(a F + b) NT]
    const int64_t j = blockIdx.x * (int64_t)NT + threadIdx.x;
    const int64_t n = L.n_traj;
    const PropArgs &A = L.args;
    for (int i = threadIdx.x; i < F * F; i += NT) {
        const int a = i / F, b = i % F;
        coef[i] = make_double4(0.5 * (A.rg[a] * A.irg[b]), 0.5 * (A.rg[b] * A.irg[a]), -0.5 * (A.rg[a] * A.rg[b]),
                               0.5 * (A.irg[a] * A.irg[b]));
    }
    __syncthreads();
    if (j >= n) return;
    const float *Mj = st.M + j;               // element (r, c) at Mj[(r 2F + c) n]
    const int step = *st.step;
    bool good = L.good[j] != 0;
    const float det = st.det[j];
    const float dev = isfinite(det) ? fabsf(fmaf(det, det, -1.0f)) : __int_as_float(0x7f800000);
    double stab = st.stab[j];
    {
        const double dv = widen(dev);         // non-negative: ordered as integers
        if (__double_as_longlong(dv) > __double_as_longlong(stab)) stab = dv;
        st.stab[j] = stab;
    }
    if (dev > A.stab_tol_f) good = false;
    {
        // rows a and F + a of M, the next pair in flight (all loads of a row ahead of widen's branches)
        float mp[N2], mq[N2], np[N2], nq[N2];
        auto load = [&](int a) {
#pragma unroll
            for (int c = 0; c < N2; ++c) {
                np[c] = Mj[((int64_t)a * N2 + c) * n];
                nq[c] = Mj[((int64_t)(F + a) * N2 + c) * n];
            }
        };
        load(0);
#pragma unroll 1
        for (int a = 0; a < F; ++a) {
#pragma unroll
            for (int c = 0; c < N2; ++c) {
                mp[c] = np[c];
                mq[c] = nq[c];
            }
            if (a + 1 < F) load(a + 1);
#pragma unroll
            for (int b = 0; b < F; ++b) {
                const double4 k = coef[a * F + b];
                Z[(a * F + b) * NT] = make_double2(fma(k.x, widen(mq[F + b]), k.y * widen(mp[b])),
                                                   fma(k.z, widen(mq[b]), k.w * widen(mp[F + b])));
            }
        }
    }
    tpt::cplx dA = {1.0, 0.0};
#pragma unroll 1
    for (int k = 0; k < F; ++k) {
        // pivot by max(|re|, |im|), within a factor sqrt(2) of |z|
        int piv = k, best = -1;
        for (int i = k; i < F; ++i) {
            const double2 v = Z[(i * F + k) * NT];
            const int key = max(mag_key(v.x), mag_key(v.y));
            if (key > best) { best = key; piv = i; }
        }
        double2 *rk = Z + k * F * NT, *rp = Z + piv * F * NT;
        if (piv != k) {
            for (int c = k; c < F; ++c) {
                const double2 v = rp[c * NT];
                rp[c * NT] = rk[c * NT];
                rk[c * NT] = v;
            }
            dA.re = -dA.re; dA.im = -dA.im;
        }
        const tpt::cplx pk = {rk[k * NT].x, rk[k * NT].y};
        dA = tpt::cmul(dA, pk);
        const double rr = recip(fma(pk.re, pk.re, pk.im * pk.im));
        const tpt::cplx inv = {pk.re * rr, -pk.im * rr};
#pragma unroll 1
        for (int i = k + 1; i < F; ++i) {
            double2 *ri = Z + i * F * NT;
            const tpt::cplx l = tpt::cmul({ri[k * NT].x, ri[k * NT].y}, inv);
#pragma unroll 4
            for (int c = k + 1; c < F; ++c) {
                const tpt::cplx y = tpt::cfnma(l, {rk[c * NT].x, rk[c * NT].y}, {ri[c * NT].x, ri[c * NT].y});
                ri[c * NT] = make_double2(y.re, y.im);
            }
        }
    }
    double arg_new;
    {
        const int e = max(mag_key(dA.re), mag_key(dA.im)) >> 20;   // to a larger part in [1, 2)
        if (e < 64 || e > 1980) {
            arg_new = atan2(dA.im, dA.re);
        } else {
            const double sc = __hiloint2double((2046 - e) << 20, 0);
            const double x = dA.re * sc, y = dA.im * sc;
            arg_new = arg_normal(x, y, (float)x, (float)y);
        }
    }
    double d = arg_new - st.arg_old[j] + A.ref_step;
    d = fma(-kTwoPi, rint(d * kInvTwoPi), d);
    const double theta = st.theta[j] + d - A.ref_step;
    st.theta[j] = theta;
    st.arg_old[j] = arg_new;
    double p[F], q[F];
    const double S = st.Se[j];
    bool finite = finite_bits(S) && finite_bits(theta);
#pragma unroll
    for (int a = 0; a < F; ++a) {
        p[a] = st.p[a * n + j];
        q[a] = st.qe[a * n + j];
        finite = finite && finite_bits(p[a]) && finite_bits(q[a]);
    }
    if (!finite) good = false;
    L.good[j] = good ? 1 : 0;
    record<F>(L, j, step, p, q, S, theta, A.amplitude == SCIVR_AMP_HK ? hypot(dA.re, dA.im) : 1.0);
    if (step == A.n_steps) {
        const FinalDev &fo = L.fin;
        if (fo.p) for (int a = 0; a < F; ++a) fo.p[a * n + j] = p[a];
        if (fo.q) for (int a = 0; a < F; ++a) fo.q[a * n + j] = q[a];
        if (fo.S) fo.S[j] = S;
        if (fo.theta) fo.theta[j] = theta;
        if (fo.detM) fo.detM[j] = (double)det;
        if (fo.stab) fo.stab[j] = stab;
        if (fo.detA) { fo.detA[2 * j] = dA.re; fo.detA[2 * j + 1] = dA.im; }
        if (fo.M)
            for (int r = 0; r < N2; ++r)
                for (int c = 0; c < N2; ++c) fo.M[j * N2 * N2 + r * N2 + c] = Mj[((int64_t)r * N2 + c) * n];
    }
}

inline size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

template <int F>
cudaError_t run(const PropLaunch &L, cudaStream_t s, int *n_launch)
{
    constexpr int N2 = 2 * F;
    const int64_t n = L.n_traj;
    size_t o = 0;
    const size_t oP = o; o += a256((size_t)F * n * 8);
    const size_t oQ = o; o += a256((size_t)F * n * 8);
    const size_t oM = o; o += a256((size_t)N2 * N2 * n * 4);
    const size_t oS = o; o += a256((size_t)n * 8);
    const size_t oT = o; o += a256((size_t)n * 8);
    const size_t oA = o; o += a256((size_t)n * 8);
    const size_t oB = o; o += a256((size_t)n * 8);
    const size_t oQe = o; o += a256((size_t)F * n * 8);
    const size_t oSe = o; o += a256((size_t)n * 8);
    const size_t oDet = o; o += a256((size_t)n * 4);
    const size_t oQf = o; o += a256((size_t)n * F * 4);
    const size_t oV = o; o += a256((size_t)n * 4);
    const size_t oG = o; o += a256((size_t)n * F * 4);
    const size_t oH = o; o += a256((size_t)n * F * F * 4);
    const size_t oStep = o; o += 256;
    const size_t oEval = o; o += mlp_eval_scratch_bytes(F, n, true);
    void *scr = nullptr;
    cudaError_t e = cudaMallocAsync(&scr, o, s);
    if (e != cudaSuccess) return e;
    char *b = static_cast<char *>(scr);
    State st{};
    st.p = reinterpret_cast<double *>(b + oP);
    st.q = reinterpret_cast<double *>(b + oQ);
    st.M = reinterpret_cast<float *>(b + oM);
    st.S = reinterpret_cast<double *>(b + oS);
    st.theta = reinterpret_cast<double *>(b + oT);
    st.arg_old = reinterpret_cast<double *>(b + oA);
    st.stab = reinterpret_cast<double *>(b + oB);
    st.qe = reinterpret_cast<double *>(b + oQe);
    st.Se = reinterpret_cast<double *>(b + oSe);
    st.det = reinterpret_cast<float *>(b + oDet);
    st.qf = reinterpret_cast<float *>(b + oQf);
    float *Vm = reinterpret_cast<float *>(b + oV), *gm = reinterpret_cast<float *>(b + oG);
    float *Hm = reinterpret_cast<float *>(b + oH);
    st.Vm = Vm; st.gm = gm; st.Hm = Hm;
    st.step = reinterpret_cast<int *>(b + oStep);
    int nl = 0;
    e = cudaMemsetAsync(st.step, 0, sizeof(int), s);
    if (e == cudaSuccess) e = mlp_prepare();
    const unsigned tiles = (unsigned)((n + 31) / 32);
    const size_t rec_smem = (size_t)(32 + 16 * kRecThreads) * F * F;   // A's coefficients, the threads' matrices
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_mlp_record<F>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rec_smem);
    if (e == cudaSuccess) {
        const bool cpl = L.pes.has3 || L.pes.has4;
        k_mlp_start<F><<<(unsigned)((n + 127) / 128), 128, 0, s>>>(L, st);
        nl += 1;
        for (int step = 1; step <= L.args.n_steps && e == cudaSuccess; ++step) {
            for (int stage = 1; stage <= 3; ++stage) {
                int ne = 0;
                e = mlp_eval(L.pes.mlp, F, n, st.qf, Vm, gm, Hm, b + oEval, s, &ne);
                nl += ne;
                if (e != cudaSuccess) break;
                if (stage < 3) {
                    if (cpl) k_mlp_kick<F, true, false><<<tiles, 32 * F, 0, s>>>(L, st, stage);
                    else k_mlp_kick<F, false, false><<<tiles, 32 * F, 0, s>>>(L, st, stage);
                } else {
                    if (cpl) k_mlp_kick<F, true, true><<<tiles, 32 * F, 0, s>>>(L, st, stage);
                    else k_mlp_kick<F, false, true><<<tiles, 32 * F, 0, s>>>(L, st, stage);
                    k_mlp_record<F><<<(unsigned)((n + kRecThreads - 1) / kRecThreads), kRecThreads, rec_smem, s>>>(L, st);
                    nl += 1;
                }
                nl += 1;
            }
            if (e == cudaSuccess) e = cudaGetLastError();
        }
    }
    cudaError_t e2 = cudaFreeAsync(scr, s);
    *n_launch = nl;
    return e != cudaSuccess ? e : e2;
}

}  // namespace pm

cudaError_t launch_propagate_mlp(const PropLaunch &L, cudaStream_t s, int *n_launch)
{
    switch (L.args.F) {
#define SCIVR_PM(FF) case FF: return pm::run<FF>(L, s, n_launch);
    SCIVR_PM(1) SCIVR_PM(2) SCIVR_PM(3) SCIVR_PM(4) SCIVR_PM(5) SCIVR_PM(6) SCIVR_PM(7) SCIVR_PM(8) SCIVR_PM(9)
#undef SCIVR_PM
    default: *n_launch = 0; return cudaErrorInvalidValue;
    }
}

}  // namespace scivr
