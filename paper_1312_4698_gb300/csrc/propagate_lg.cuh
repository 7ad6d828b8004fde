// Mixed-precision lane-group propagation kernel (Sec. III.A / III.B of arXiv:1312.4698); the
// FP64 lane groups are in propagate_g64.cuh.
//
// A group of G lanes (mixed_group_lanes) owns one trajectory; a warp holds T = 32/G
// trajectories.  Steps are processed in chunks of C (lg_chunk), and work is split by
// what parallelises:
//
//   phase 1 (per step, group-parallel):
//     lane g owns columns g, g + G < 2F of the monodromy matrix M (their p- and q-rows
//     in registers); lane a < F owns mode a: p_a, q_a and the
//     separable diagonal of the potential.  The Hessian's packed coupling
//     entries e(a,b) are spread over the group, reading the coupling tensors
//     staged in shared memory; above F = 13 the warps of a CTA form their
//     trajectories' Hessians together.  The Herman-Kluk matrix A of the step goes to
//     shared memory.
//   phase 2 (once per chunk): 32 / (T C) lanes take a job (trajectory, step) and compute det A
//     and its argument by an LU in place in shared memory; every kDetMEvery steps det M by
//     Gaussian elimination of M^T across the group.
//   phase 3: the continuous phase, a segmented prefix sum over each group.
//   phase 4 (job-parallel): overlap <chi|p q>, action, phase and the amplitude;
//     each group writes C consecutive samples of its row.
//
// FP32: monodromy, potential, det M, A, the overlap and each step's action
// increment; positions, momenta, the accumulated action and the elimination that gives det A
// in double-FP32; the continuous phase in FP64; the amplitude's phase is reduced modulo 2 pi
// in FP64 and its sine, cosine and magnitude are evaluated in FP32.
//
// On GB300 a warp-wide FP64 instruction holds a sub-partition's FP64 pipe for
// about 64 cycles, so phase 1 keeps off it altogether.
#pragma once

#include <math_constants.h>
#include <cstddef>
#include <algorithm>
#include <utility>
#include <type_traits>

#include "fp64_ops.cuh"
#include "scivr_internal.cuh"

namespace scivr {
namespace lg {

constexpr unsigned FULL = 0xffffffffu;

template <int F>
__host__ __device__ constexpr int pidx(int a, int b)
{
    return a * F - a * (a - 1) / 2 + (b - a);
}

// Storage of one entry of the Herman-Kluk matrix A during its elimination: a double-FP32
// complex (re.hi, im.hi, re.lo, im.lo) -- the entries are formed in FP32 and eliminated to
// FP64-class accuracy, the real and imaginary words side by side for packed FP32 arithmetic.
using AEntry = float4;

// ---- double-FP32 arithmetic (hi + lo, |lo| <= ulp(hi)/2): error-free sum and
// product of two floats (Knuth's TwoSum, the FMA form of Dekker's TwoProduct) and
// the compositions the elimination needs.  Accuracy about 2^-46 relative per
// operation, on the FP32 pipe.
struct ff { float hi, lo; };

__device__ __forceinline__ void ff_two_sum(float a, float b, float &s, float &e)
{
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

__device__ __forceinline__ ff ff_norm(float hi, float lo)    // |lo| well below |hi| or hi == 0
{
    ff r;
    r.hi = hi + lo;
    r.lo = lo - (r.hi - hi);
    return r;
}

__device__ __forceinline__ ff ff_mul(ff x, ff y)
{
    const float p = x.hi * y.hi;
    float e = fmaf(x.hi, y.hi, -p);
    e = fmaf(x.hi, y.lo, e);
    e = fmaf(x.lo, y.hi, e);
    return ff_norm(p, e);
}

__device__ __forceinline__ ff ff_add(ff x, ff y)
{
    float s, e;
    ff_two_sum(x.hi, y.hi, s, e);
    return ff_norm(s, e + (x.lo + y.lo));
}

// a - x u + y v for double-FP32 a, x, u, y, v (one real part of a complex
// multiply-subtract): both products exact to their double-FP32 width, both sums
// error-free in their leading words.
__device__ __forceinline__ ff ff_sub_mul_add_mul(ff a, ff x, ff u, ff y, ff v)
{
    const float p1 = x.hi * u.hi;
    float e1 = fmaf(x.hi, u.hi, -p1);
    e1 = fmaf(x.hi, u.lo, e1);
    e1 = fmaf(x.lo, u.hi, e1);
    const float p2 = y.hi * v.hi;
    float e2 = fmaf(y.hi, v.hi, -p2);
    e2 = fmaf(y.hi, v.lo, e2);
    e2 = fmaf(y.lo, v.hi, e2);
    float s1, t1, s2, t2;
    ff_two_sum(a.hi, -p1, s1, t1);
    ff_two_sum(s1, p2, s2, t2);
    return ff_norm(s2, ((a.lo - e1) + e2) + (t1 + t2));
}

// 1 / m for double-FP32 m > 0: the FP32 reciprocal refined by one Newton step on
// the exact FMA residual.
__device__ __forceinline__ ff ff_recip(ff m)
{
    const float y0 = __frcp_rn(m.hi);
    float r = fmaf(-m.hi, y0, 1.0f);   // 1 - m.hi y0, exact
    r = fmaf(-m.lo, y0, r);
    return ff_norm(y0, y0 * r);
}

// Positions, momenta and the action: double-FP32 pairs (FP64-class accuracy, about 2^-46
// relative per operation, on the FP32 pipe: on this GPU an FP64 instruction or conversion costs
// the FP64 pipe ~70 times the issue of an FP32 one).  coord_axpy: c + t x; coord_kick: c - t g
// for an FP32 force g; t is given as FP32 leading and trailing words (th, tl).
__device__ __forceinline__ void coord_set(ff &c, double x)
{
    c.hi = (float)x;
    c.lo = (float)(x - (double)c.hi);
}
__device__ __forceinline__ double coord_get(ff c) { return (double)c.hi + (double)c.lo; }
__device__ __forceinline__ float coord_f(ff c) { return c.hi; }
__device__ __forceinline__ bool coord_finite(ff c) { return isfinite(c.hi) && isfinite(c.lo); }
__device__ __forceinline__ ff coord_axpy(ff c, float th, float tl, ff x)
{
    const float p = th * x.hi;
    float e = fmaf(th, x.hi, -p);   // th x.hi - p, exact
    e = fmaf(th, x.lo, e);
    e = fmaf(tl, x.hi, e);
    float s, e2;
    ff_two_sum(c.hi, p, s, e2);
    return ff_norm(s, e2 + (c.lo + e));
}
__device__ __forceinline__ ff coord_kick(ff c, float th, float tl, float g)
{
    const float p = -th * g;
    float e = fmaf(-th, g, -p);
    e = fmaf(-tl, g, e);
    float s, e2;
    ff_two_sum(c.hi, p, s, e2);
    return ff_norm(s, e2 + (c.lo + e));
}
// the action increment (FP32 partial sums) joins the running action
__device__ __forceinline__ ff coord_add(ff c, float d)
{
    float s, e;
    ff_two_sum(c.hi, d, s, e);
    return ff_norm(s, e + c.lo);
}

// Complex double-FP32 numbers as packed pairs: hi = (re.hi, im.hi), lo = (re.lo, im.lo); each
// instruction does the real and the imaginary part at once.  Differences are multiply-adds by
// -1 (one rounding, the same result), so that no operand has to be negated first.
struct ff2 { float2 hi, lo; };

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }

__device__ __forceinline__ void ff2_two_sum(float2 a, float2 b, float2 &s, float2 &e)
{
    s = add2(a, b);
    const float2 bb = sub2(s, a);
    e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// A row's multiplier l = lr + i li, spread for the packed update: a - l p has the parts
// a.re - lr p.re + li p.im and a.im - lr p.im - li p.re, i.e. a - x u + y v with u = (p.re, p.im),
// v = (p.im, p.re), x = (lr, lr) and y = (li, -li).  Held: x, -x, y and -y in the signs the
// products need.
struct ElimRow {
    float2 xh, nxh, xl, y, ny, nyl;
    __device__ __forceinline__ ElimRow(ff lr, ff li)
        : xh(make_float2(lr.hi, lr.hi)), nxh(make_float2(-lr.hi, -lr.hi)), xl(make_float2(lr.lo, lr.lo)),
          y(make_float2(li.hi, -li.hi)), ny(make_float2(-li.hi, li.hi)), nyl(make_float2(-li.lo, li.lo)) {}
};

// a - l p for entries stored (re.hi, im.hi, re.lo, im.lo): both products exact to their
// double-FP32 width (d gathers minus their trailing parts: fma(x, u, -x u rounded) and the cross
// terms), both sums error-free in their leading words, the result normalised.
__device__ __forceinline__ float4 elim_update(const float4 &a, const ElimRow &l, const float4 &p)
{
    const float2 uh = make_float2(p.x, p.y), ul = make_float2(p.z, p.w);
    const float2 vh = make_float2(p.y, p.x), vl = make_float2(p.w, p.z);
    const float2 ah = make_float2(a.x, a.y), al = make_float2(a.z, a.w);
    const float2 p1 = __fmul2_rn(l.nxh, uh);
    float2 d = __ffma2_rn(l.xh, uh, p1);
    const float2 p2 = __fmul2_rn(l.y, vh);
    const float2 d2 = __ffma2_rn(l.ny, vh, p2);
    d = __ffma2_rn(l.xh, ul, d);
    d = __ffma2_rn(l.xl, uh, d);
    d = __ffma2_rn(l.ny, vl, d);
    d = __ffma2_rn(l.nyl, vh, d);
    float2 s1, t1, s2, t2;
    ff2_two_sum(ah, p1, s1, t1);
    ff2_two_sum(s1, p2, s2, t2);
    const float2 lo = add2(sub2(al, add2(d, d2)), add2(t1, t2));
    const float2 h = add2(s2, lo);
    const float2 r = sub2(lo, sub2(h, s2));
    return make_float4(h.x, h.y, r.x, r.y);
}

// Per-mode and per-reference-state constants, staged in shared memory so that
// lane- or chi-dependent indexing never touches the kernel-parameter space.
template <int F>
struct CtaConst {
    double qw[F], pw[F];
    double p_eq[SCIVR_MAX_CHI][F], q_eq[SCIVR_MAX_CHI][F];
    float Df[F], af[F], w2f[F];            // diagonal parameters
    float qwf[F], pwf[F];                  // overlap constants in FP32 (mixed path's overlap)
    float p_eqf[SCIVR_MAX_CHI][F], q_eqf[SCIVR_MAX_CHI][F];
};

// Column of job j in row r of the per-job arrays: the F mode lanes of a group
// store one job into F different rows, which a plain [row][job] layout puts
// into a single shared-memory bank; XOR-ing the job with the row spreads them
// over banks, and every row is still a permutation of the chunk's jobs.
template <int JOBS>
__device__ __forceinline__ int jswz(int r, int j) { return j ^ (r & (JOBS >= 16 ? 15 : JOBS - 1)); }

// Steps per chunk of a lane group.  Phases 2-4 work on T * C jobs (trajectory, step) per warp.
// The double-FP32 elimination keeps two FP32 words per real entry, so chunks are short (8 steps; 4
// at F = 9 and 13..15, 2 at 16, 1 above) and 32 / (T * C) lanes share a job's elimination by rows.
// CUBIC: the kernels for surfaces without quartic terms (cubic_schedule).
// Mixed path: steps between stability tests (a multiple of every mixed chunk length).
// The flag is sticky and a bad trajectory is dropped whole, so a coarser test differs
// from the per-step one only for a deviation that crosses the threshold and falls back
// below it between two tests (on the recipe surfaces, none: the good sets at 8- and
// 16-step cadences equal the per-step ones).
constexpr int kDetMEvery = 16;

template <int F, int G, bool CUBIC = false> __host__ __device__ constexpr int lg_chunk()
{
    if (CUBIC) return F > 23 ? 1 : (F > 16 ? 2 : 4);
    return G == 32 && F > 16 ? 1 : (G == 32 && F > 15 ? 2 : ((G == 32 && F > 12) || (G == 16 && F > 8) ? 4 : 8));
}

// Warps per CTA and the launch-bounds CTA count: above F = 13 one CTA of 8 warps per SM, whose
// warps form the Hessians of their trajectories together (CoopHessian); F = 10..13 staged tensors
// and a Hessian per warp, 8 warps up to F = 12 and 2 CTAs of 4 at F = 13 (the shared contraction's
// barriers cost more than its loads save there: 5.84 against 5.57 ms for 4000 x 100 steps).
template <int F, int G> __host__ __device__ constexpr int lg_warps() { return G < 32 ? 4 : (F <= 9 ? 2 : (F == 13 ? 4 : 8)); }
// Two-trajectory mixed warps (F = 6..9) hold the coupling tensors in registers (no
// shared-memory reads of them, more registers: lg_min_ctas) or read them from shared
// memory in the same half-split layout (TensorLayout::split).  Measured on the recipe
// surfaces: registers win at F = 7 (7 %) and F = 8 (10 %: the shared-memory schedule there
// is held to 128 registers by its four CTAs per SM); shared memory wins at F = 6 (6 %, four
// CTAs per SM against three) and at F = 9 (12 %, three against two).
template <int F> __host__ __device__ constexpr bool lg_tensor_regs() { return F == 7 || F == 8; }

template <int F, int G> __host__ __device__ constexpr int lg_min_ctas()
{
    // register-held tensors: two CTAs per SM at F = 8, 9 (up to 255 registers), three at F = 6, 7
    if constexpr (G == 16 && F >= 6 && lg_tensor_regs<F>()) return F >= 8 ? 2 : 3;
    return F > 9 ? 1 : (2 * F > G ? 3 : 4);
}

// Length of a row padded to whole 16-byte vectors.
__host__ __device__ constexpr int vec_len(int n) { return (n + 3) / 4 * 4; }

// Row stride for rows that different lanes read with 16-byte loads at the same
// time: whole vectors, an odd number of them, so that the 8 lanes served by one
// shared-memory wavefront start in 8 different groups of 4 banks.
__host__ __device__ constexpr int row_stride(int n) { return vec_len(n) / 4 % 2 == 0 ? vec_len(n) + 4 : vec_len(n); }

// Packed FP32 multiply-add on register pairs (one instruction, two lanes of work).
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 lo2(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4 &v) { return make_float2(v.z, v.w); }

// sum_{i < S} a[i] b[i] over 16-byte aligned shared rows (S a multiple of four) in packed pairs.
template <int S>
__device__ __forceinline__ float dot16(const float *a, const float *b)
{
    static_assert(S % 4 == 0, "padded length");
    float2 a0 = make_float2(0.0f, 0.0f), a1 = a0;
#pragma unroll
    for (int i = 0; i < S; i += 4) {
        const float4 x = *reinterpret_cast<const float4 *>(a + i);
        const float4 y = *reinterpret_cast<const float4 *>(b + i);
        a0 = ffma2(lo2(x), lo2(y), a0);
        a1 = ffma2(hi2(x), hi2(y), a1);
    }
    return (a0.x + a1.x) + (a0.y + a1.y);
}

// Coupling tensors staged per CTA, transposed so that one potential entry e
// reads one contiguous row: sT3[e][k] (k < F, stride S3), sT4[e][kl] (kl < P,
// stride S4), zero-padded.
template <int F, bool STAGED = (F <= 16), bool CUBIC = false>
struct TensorLayout {
    static constexpr int P = F * (F + 1) / 2;
    static constexpr int S3 = vec_len(F);   // short rows: fewer loads outweigh a 2-way conflict
    static constexpr int S4 = row_stride(P);
    // Above F = 16 the quartic tensor (P^2 entries, 360 KB at F = 24) does not fit shared
    // memory: both tensors are read from global memory (L2) and only the coefficients are staged.
    static constexpr bool staged = STAGED;
    // Two-trajectory mixed warps (F = 6..9) cut x = (q, zero pad to an even length F3E, the
    // pair products, zero pad) into two halves of KH elements; those that do not hold the
    // tensors in registers read them from shared memory cut the same way ("split"):
    // sTh[h][e][KHS] = the tensor row of entry e over half h of x, KHS an odd number of
    // 16-byte vectors so that 8 lanes reading 8 consecutive entries hit disjoint banks.
    static constexpr int F3E = (F + 1) & ~1;
    static constexpr int KH = (((F3E + P + 1) / 2) + 3) & ~3;
    static constexpr int KHS = (KH / 4) % 2 ? KH : KH + 4;
    static constexpr bool split = STAGED && F >= 6 && F <= 9 && !lg_tensor_regs<F>();
    // One-trajectory mixed warps above F = 13, and all that do not stage the tensors, contract them
    // together (CoopHessian): rows of P4
    // consecutive entries, the F cubic rows first.
    static constexpr bool coop = !CUBIC && (F > 13 || (F > 9 && !STAGED));
    static constexpr int P4 = (P + 3) & ~3;
    static constexpr size_t tensor_elems = !staged ? 0 : (coop ? (size_t)(F + P) * P4 : (split ? (size_t)2 * P * KHS : (size_t)P * S3 + (size_t)P * S4));
    // after the tensors: the Herman-Kluk matrix coefficients acoef[a][b][4] =
    // (1/2) {rg_a/rg_b, rg_b/rg_a, -rg_a rg_b, 1/(rg_a rg_b)}, rg = sqrt(gamma)
    static constexpr size_t bytes = ((sizeof(float) * (tensor_elems + (size_t)4 * F * F)) + 15) & ~(size_t)15;
};

// Hessian contraction of the wide mixed groups (F > 13, and all that do not stage the tensors),
// shared by the warps of a CTA: entry e of trajectory t is sum_k T[k][e] x_t[k] over the cubic rows
// (x = q) and over the quartic rows (x = q_k q_l).  A lane takes a quad of four entries and TT of
// the CTA's TRAJ trajectories, so that a 16-byte tensor load feeds 4 TT multiply-adds; alone, a
// warp's one trajectory used every loaded element once, and the loads bound the kernel (four or
// eight warps per SM, issue 18-22 %).  Staged tensors (F <= 16): four lanes share a quad, lane s
// summing the rows k = s mod 4, and the four sums are added as (s0 + s2) + (s1 + s3).  Otherwise the
// rows stream from L2 through a ring of tiles in shared memory (cp.async), one sum per entry in row
// order.  Either way each entry's multiply-adds keep the order they have in a single lane's loop,
// whatever the tile: the results do not depend on TRAJ.  TT is the smallest tile whose items fit one
// round of the CTA's lanes.  F = 15, 3001 trajectories x 501 steps: 37.0 -> 27.6 ms; F = 24,
// 2048 x 200: 79.3 -> 45.8 ms (with the later changes to the prefactor 24.9 and 37.2).
template <int F, int WARPS, int TRAJ, bool STAGED>
struct CoopHessian {
    static constexpr int P = F * (F + 1) / 2, P4 = (P + 3) & ~3, Q = P4 / 4;
    static constexpr int SUB = STAGED ? 4 : 1;                      // lanes that share a quad's rows
    static constexpr int groups(int tt) { return (TRAJ + tt - 1) / tt; }
    static constexpr bool fits(int tt) { return Q * SUB * groups(tt) <= 32 * WARPS; }
    static constexpr int TT = fits(1) ? 1 : fits(2) ? 2 : fits(3) ? 3 : fits(4) ? 4 : 8;
    static_assert(fits(TT), "one round of items");
    static constexpr int NG = groups(TT);
    static constexpr int TP = TT == 3 ? 4 : TT;                     // trajectory slots of a group, padded to a vector
    static constexpr int XW = NG * TP;                              // row length of the contracted vectors
    static constexpr int ITEMS = Q * SUB * NG;
    static constexpr int RT = WARPS >= 8 ? 16 : 8, ST = STAGED ? 0 : (WARPS >= 8 ? 3 : 2);   // ring tiles: rows, stages
    static constexpr size_t x_bytes = (sizeof(float) * (size_t)(F + P) * XW + 15) & ~(size_t)15;
    static constexpr size_t bytes = x_bytes + sizeof(float) * (size_t)ST * RT * P4;
    __device__ static __forceinline__ int slot(int traj) { return (traj / TT) * TP + traj % TT; }
};

__device__ __forceinline__ void cp_async16(float *dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int TP>
__device__ __forceinline__ void load_x(const float *p, float (&x)[TP])
{
    if constexpr (TP == 1) x[0] = *p;
    else if constexpr (TP == 2) { const float2 v = *reinterpret_cast<const float2 *>(p); x[0] = v.x; x[1] = v.y; }
    else {
#pragma unroll
        for (int i = 0; i < TP; i += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(p + i);
            x[i] = v.x; x[i + 1] = v.y; x[i + 2] = v.z; x[i + 3] = v.w;
        }
    }
}

template <int TT, int TP>
__device__ __forceinline__ void coop_fma(const float4 &t, const float (&x)[TP], float (&acc)[TT][4])
{
#pragma unroll
    for (int j = 0; j < TT; ++j) {
        acc[j][0] = fmaf(t.x, x[j], acc[j][0]);
        acc[j][1] = fmaf(t.y, x[j], acc[j][1]);
        acc[j][2] = fmaf(t.z, x[j], acc[j][2]);
        acc[j][3] = fmaf(t.w, x[j], acc[j][3]);
    }
}

template <int F, int G, bool CUBIC = false>
struct WarpShared {
    static constexpr int P = F * (F + 1) / 2;
    static constexpr int T = 32 / G;
    static constexpr int JOBS = T * lg_chunk<F, G, CUBIC>();   // jobs per chunk (phases 2-4)
    static constexpr int S3 = TensorLayout<F>::S3;   // q, zero-padded (also the Gc row stride)
    static constexpr int S4 = TensorLayout<F>::S4;   // pair products q_k q_l, zero-padded
    // H, read whole by every column lane with 16-byte broadcasts: rows of an even
    // length back to back, so that pairs stay aligned and no load is mostly padding (9 instead of 12
    // loads at F = 6, 23 instead of 27 at F = 9; at F = 10, one trajectory a warp, 0.9 % slower and
    // not used: rows of whole vectors there).
    static constexpr int SH = F != 10 ? (F + 1) & ~1 : vec_len(F);
    static constexpr int HV = vec_len(F * SH);
    alignas(16) float qr[T][S3];
    alignas(16) float qq[T][S4];
    // x = (q, zero pad to an even length, pair products, zero pad) in two halves of KH for the
    // half-split Hessian of two-trajectory warps (see TensorLayout and lg_body)
    static constexpr int F3E = TensorLayout<F>::F3E;
    static constexpr int KH = TensorLayout<F>::KH;
    // only two-trajectory mixed warps use it: elsewhere a stub, so that the shared memory
    // left to L1 (the wide groups read their tensors through it) does not shrink
    static constexpr bool kHalves = T == 2 && F >= 6 && F <= 9;
    alignas(16) float xs[T][kHalves ? 2 * KH : 4];
    alignas(16) float Gc[T][F][S3];          // gradient coefficients, full symmetric matrix (row a read by mode lane a)
    alignas(16) float Hs[T][HV];
    __device__ __forceinline__ float &H(int tr, int a, int b) { return Hs[tr][a * SH + b]; }
    // Prefactor matrix per job.  LPJ = 32 / JOBS lanes of a job read consecutive rows at
    // the same column with 16-byte accesses, eight lanes (8 / LPJ jobs) to a wavefront.  The row
    // stride RS and the jobs' bases spread those eight over the eight 16-byte bank groups: an odd
    // RS for eight rows of one job, bases 4 apart (mod 8) for two jobs of four rows, 2 apart for four
    // jobs of two rows -- or, at F = 6, where an odd RS would cost a CTA per SM, 0, 5, 4, 1.  (With
    // F = 24 entries a row all eight fell into one group; with 81 a job two at F = 9.)
    static constexpr int LPJ = JOBS >= 32 ? 1 : 32 / JOBS;
    static constexpr int RS = LPJ == 1 || F == 6 ? F : F | 1;
    static constexpr int up(int n, int r) { return n % 8 == r ? n : up(n + 1, r); }
    // (at least the det M workspace of 2F rows of 2F + 1 floats per trajectory)
    static constexpr int AS0 = (T * 2 * F * (2 * F + 1) + 4 * JOBS - 1) / (4 * JOBS);
    static constexpr int AS1 = AS0 > F * RS ? AS0 : F * RS;
    static constexpr int AS = LPJ == 1 || LPJ >= 8 ? AS1 | 1 : (F == 6 ? 38 : up(AS1, LPJ == 4 ? 4 : 2));
    static_assert(F != 6 || LPJ == 1 || (LPJ == 2 && AS1 <= 37), "the bases of F = 6");
    AEntry A[JOBS * AS];
    __device__ static __forceinline__ int a_base(int job) { return F == 6 && LPJ == 2 ? 38 * job - (job & 1) : AS * job; }
    __device__ __forceinline__ AEntry &a_at(int job, int row, int col) { return A[a_base(job) + row * RS + col]; }
    // cubic and quartic parts of the Hessian entries (wide mixed groups): in the storage of the
    // step's own prefactor matrix, which is written after the step's last kick
    static constexpr int HP = (P + 3) & ~3;
    static_assert(F <= 9 || 8 * HP <= 16 * F * F, "the Hessian parts fit a job's matrix");
    __device__ __forceinline__ float *h3_at(int job) { return reinterpret_cast<float *>(&A[a_base(job)]); }
    __device__ __forceinline__ float *h4_at(int job) { return h3_at(job) + HP; }
    float pj[F][JOBS], qj[F][JOBS];         // state per job, for the overlap (job column swizzled); FP32
                                           // in the mixed path, where the overlap is evaluated in FP32
    double Sj[JOBS];                        // action per job
    double lnA[JOBS];                       // log |det A|^{1/2} per job (Herman-Kluk summand only)
    double argj[JOBS];                      // arg det A per job (mixed path: from the elimination's lanes)
    double2 detAj[JOBS];                    // det A per job (mixed path)
    double2 ov0[SCIVR_MAX_CHI][T];          // log of the Herman-Kluk summand's divisor per trajectory
};

// One CTA's share of a propagation: trajectories (cta * TRAJ_WARPS + warp) * T + t, warp <
// TRAJ_WARPS; the other warps only share the Hessian contraction (wide mixed groups).
// Called by the per-molecule kernel (cta = blockIdx.x) and by the batched
// persistent kernel (cta = the work item's tile).  Stages the molecule's
// constants itself and leaves shared memory free for the next call.
template <int F, int G, int WARPS, bool STAGED = (F <= 16), int TRAJ_WARPS = WARPS, bool CUBIC = false>
__device__ __forceinline__ void lg_body(const PropLaunch &L, int64_t cta, unsigned char *smem_raw)
{
    constexpr int N2 = 2 * F;
    constexpr int P = F * (F + 1) / 2;
    constexpr int T = 32 / G;
    constexpr int C = lg_chunk<F, G, CUBIC>();  // steps per chunk
    constexpr int JOBS = T * C;                // jobs per chunk: job t * C + c is trajectory t's step c
    constexpr int EPL = (P + G - 1) / G;       // packed Hessian entries per lane
    constexpr int NCOL = (N2 + G - 1) / G;     // monodromy columns per lane: column c sits in lane c % G, slot c / G
    static_assert(F <= G && NCOL <= 2, "a group holds every mode and at most two columns per lane");
    using Sh = WarpShared<F, G, CUBIC>;

    using TL = TensorLayout<F, STAGED, CUBIC>;
    constexpr int S3 = TL::S3, S4 = TL::S4;
    float *sT3 = reinterpret_cast<float *>(smem_raw);
    float *sT4 = sT3 + ((TL::staged && !TL::split && !TL::coop) ? P * S3 : 0);
    float *sTh = sT3;                                  // the half-split layout (TL::split)
    float *sAc = sT3 + TL::tensor_elems;   // Herman-Kluk matrix coefficients [a][b][4] (16-byte aligned: the tensor block is a vector multiple)
    size_t off = TL::bytes;
    CtaConst<F> &cc = *reinterpret_cast<CtaConst<F> *>(smem_raw + off);
    off += (sizeof(CtaConst<F>) + 15) & ~(size_t)15;
    // wide mixed groups: the CTA's contracted vectors and the ring of tensor rows
    constexpr bool kCoop = TL::coop;
    using CH = CoopHessian<kCoop ? F : 16, kCoop ? WARPS : 8, kCoop ? TRAJ_WARPS : 8, kCoop ? STAGED : true>;
    float *xall = reinterpret_cast<float *>(smem_raw + off);
    float *ring = reinterpret_cast<float *>(smem_raw + off + CH::x_bytes);
    if constexpr (kCoop) off += CH::bytes;
    Sh *wsh_all = reinterpret_cast<Sh *>(smem_raw + off);

    const PesDev &pes = L.pes;
    const PropArgs &A = L.args;
    const bool use3 = pes.has3, use4 = pes.has4;
    // stage the coupling tensors once per CTA
    if constexpr (TL::staged) {
        const float *g3 = pes.T3f, *g4 = pes.T4f;
        if constexpr (kCoop) {
            const float4 *v3 = reinterpret_cast<const float4 *>(pes.T3p), *v4 = reinterpret_cast<const float4 *>(pes.T4p);
            float4 *dst = reinterpret_cast<float4 *>(sT3);
            for (int i = threadIdx.x; i < F * (TL::P4 / 4); i += blockDim.x) dst[i] = v3[i];
            for (int i = threadIdx.x; i < P * (TL::P4 / 4); i += blockDim.x) dst[F * (TL::P4 / 4) + i] = v4[i];
        } else if constexpr (TL::split) {
            constexpr int KH = TL::KH, KHS = TL::KHS, F3E = TL::F3E;
            for (int i = threadIdx.x; i < 2 * P * KHS; i += blockDim.x) {
                const int h = i / (P * KHS), e = (i / KHS) % P, kk = i % KHS, gk = h * KH + kk;
                float v = 0.0f;
                if (kk < KH) {
                    if (gk < F) v = use3 ? g3[gk * P + e] : 0.0f;
                    else if (gk >= F3E && gk - F3E < P) v = use4 ? g4[(gk - F3E) * P + e] : 0.0f;
                }
                sTh[i] = v;
            }
        } else {
            for (int i = threadIdx.x; i < P * S3; i += blockDim.x) {
                const int e = i / S3, k = i % S3;
                sT3[i] = (use3 && k < F) ? g3[k * P + e] : 0.0f;
            }
            for (int i = threadIdx.x; i < P * S4; i += blockDim.x) {
                const int e = i / S4, kl = i % S4;
                sT4[i] = (use4 && kl < P) ? g4[kl * P + e] : 0.0f;
            }
        }
    }
    if (threadIdx.x == 0) {
#pragma unroll
        for (int a = 0; a < F; ++a) {
            cc.qw[a] = A.qw[a];
            cc.pw[a] = A.pw[a];
            cc.qwf[a] = (float)A.qw[a];
            cc.pwf[a] = (float)A.pw[a];
            cc.Df[a] = pes.D_f[a];
            cc.af[a] = pes.a_f[a];
            cc.w2f[a] = pes.omega_f[a] * pes.omega_f[a];
        }
        // (rolled: thread 0 alone, and unrolling F^2 iterations starves the step loop of registers)
        for (int a = 0; a < F; ++a)
            for (int b = 0; b < F; ++b) {
                const float rga = (float)A.rg[a], irga = (float)A.irg[a], rgb = (float)A.rg[b], irgb = (float)A.irg[b];
                float *k = sAc + 4 * (a * F + b);
                k[0] = 0.5f * (rga * irgb);
                k[1] = 0.5f * (rgb * irga);
                k[2] = -0.5f * (rga * rgb);
                k[3] = 0.5f * (irga * irgb);
            }
#pragma unroll
        for (int x = 0; x < SCIVR_MAX_CHI; ++x)
#pragma unroll
            for (int a = 0; a < F; ++a) {
                cc.p_eq[x][a] = x < A.n_chi ? A.p_eq[x * F + a] : 0.0;
                cc.q_eq[x][a] = x < A.n_chi ? A.q_eq[x * F + a] : 0.0;
                cc.p_eqf[x][a] = (float)cc.p_eq[x][a];
                cc.q_eqf[x][a] = (float)cc.q_eq[x][a];
            }
    }
    __syncthreads();

    const int warp = threadIdx.x >> 5, ln = threadIdx.x & 31;
    const int t = ln / G, g = ln % G, base = t * G;
    constexpr int P4 = (P + 3) & ~3;
    // the CTA's share of one kick's Hessian contraction (CoopHessian): from the trajectories'
    // vectors in xall to the entries' parts h3, h4 of step c's job
    auto contract = [&](int c) {
        if constexpr (kCoop) {
            const int it = threadIdx.x;
            const int sub = it % CH::SUB, quad = (it / CH::SUB) % CH::Q, grp = it / (CH::SUB * CH::Q);
            const bool work = it < CH::ITEMS;
            constexpr int TT = CH::TT, TP = CH::TP;
            float a3[TT][4], a4[TT][4];
#pragma unroll
            for (int j = 0; j < TT; ++j)
#pragma unroll
                for (int c4 = 0; c4 < 4; ++c4) a3[j][c4] = a4[j][c4] = 0.0f;
            const float *xg = xall + grp * TP;
            if constexpr (STAGED) {
                if (work) {
                    const float4 *trow = reinterpret_cast<const float4 *>(sT3) + quad;
                    if (use3) {
#pragma unroll 2
                        for (int k = sub; k < F; k += 4) {
                            float x[TP];
                            load_x<TP>(xg + k * CH::XW, x);
                            coop_fma<TT, TP>(trow[k * CH::Q], x, a3);
                        }
                    }
                    if (use4) {
#pragma unroll 4
                        for (int k = F + sub; k < F + P; k += 4) {
                            float x[TP];
                            load_x<TP>(xg + k * CH::XW, x);
                            coop_fma<TT, TP>(trow[k * CH::Q], x, a4);
                        }
                    }
                }
                // the four row classes of a quad sit in adjacent lanes
#pragma unroll
                for (int j = 0; j < TT; ++j)
#pragma unroll
                    for (int c4 = 0; c4 < 4; ++c4) {
                        a3[j][c4] += __shfl_xor_sync(FULL, a3[j][c4], 2);
                        a3[j][c4] += __shfl_xor_sync(FULL, a3[j][c4], 1);
                        a4[j][c4] += __shfl_xor_sync(FULL, a4[j][c4], 2);
                        a4[j][c4] += __shfl_xor_sync(FULL, a4[j][c4], 1);
                    }
            } else {
                // rows r < n3 of T3p, then the rows of T4p (one array), in tiles of RT rows
                constexpr int RT = CH::RT, ST = CH::ST;
                const int n3 = use3 ? F : 0, nr = n3 + (use4 ? P : 0), n_tile = (nr + RT - 1) / RT;
                const float *xr = xg + (use3 ? 0 : F * CH::XW);
                const float *src = (use3 ? pes.T3p : pes.T4p) + 4 * threadIdx.x;
                auto fetch = [&](int tile) {
                    if (tile < n_tile) {
                        float *dst = ring + (tile % ST) * (RT * P4) + 4 * threadIdx.x;
                        const float *from = src + (size_t)tile * (RT * P4);
                        const int cnt4 = min(RT, nr - tile * RT) * (P4 / 4) - (int)threadIdx.x;
#pragma unroll
                        for (int i = 0; i < RT * P4 / 4; i += 32 * WARPS)
                            if (i < cnt4) cp_async16(dst + 4 * i, from + 4 * i);
                    }
                    cp_async_commit();
                };
#pragma unroll
                for (int s = 0; s < ST - 1; ++s) fetch(s);
                for (int tile = 0; tile < n_tile; ++tile) {
                    cp_async_wait<ST - 2>();
                    __syncthreads();   // the tile is in; the one fetched next was read a turn ago
                    fetch(tile + ST - 1);
                    if (work) {
                        const float4 *trow = reinterpret_cast<const float4 *>(ring + (tile % ST) * (RT * P4)) + quad;
                        const int r0 = tile * RT, r1 = min(r0 + RT, nr);
                        int r = r0;
                        for (; r < min(r1, n3); ++r) {
                            float x[TP];
                            load_x<TP>(xr + r * CH::XW, x);
                            coop_fma<TT, TP>(trow[(r - r0) * CH::Q], x, a3);
                        }
#pragma unroll 4
                        for (; r < r1; ++r) {
                            float x[TP];
                            load_x<TP>(xr + r * CH::XW, x);
                            coop_fma<TT, TP>(trow[(r - r0) * CH::Q], x, a4);
                        }
                    }
                }
                cp_async_wait<0>();
            }
            if (work) {
#pragma unroll
                for (int j = 0; j < TT; ++j) {
                    const int tr = grp * TT + j;
                    if (tr < TRAJ_WARPS && j % CH::SUB == sub) {
                        *reinterpret_cast<float4 *>(wsh_all[tr].h3_at(c) + 4 * quad) = make_float4(a3[j][0], a3[j][1], a3[j][2], a3[j][3]);
                        *reinterpret_cast<float4 *>(wsh_all[tr].h4_at(c) + 4 * quad) = make_float4(a4[j][0], a4[j][1], a4[j][2], a4[j][3]);
                    }
                }
            }
        } else {
            (void)c;
        }
    };
    if constexpr (TRAJ_WARPS < WARPS) {
        static_assert(kCoop, "only the shared contraction employs warps without a trajectory");
        if (warp >= TRAJ_WARPS) {
            for (int step0 = 0; step0 < A.n_steps; step0 += C)
                for (int c = 0; c < min(C, A.n_steps - step0); ++c)
                    for (int kick = 0; kick < 3; ++kick) {
                        __syncthreads();
                        contract(c);
                        __syncthreads();
                    }
            __syncthreads();   // the body's last
            return;
        }
    }
    Sh &sh = wsh_all[warp];
    {
        // padding entries of the vector rows are read (multiplied by zero or skipped) but never
        // written by the step loop: clear the warp's rows once
        float *z = &sh.qr[0][0];
        constexpr int nz = (int)((offsetof(Sh, Hs) + sizeof(Sh::Hs) - offsetof(Sh, qr)) / sizeof(float));
        for (int i = ln; i < nz; i += 32) z[i] = 0.0f;
        __syncwarp();
    }
    const int64_t n = L.n_traj;
    const int64_t j_traj = (cta * TRAJ_WARPS + warp) * T + t;
    const bool active = j_traj < n;
    const int64_t jl = active ? j_traj : n - 1;

    // packed entries handled by this lane
    int ea[EPL], eb[EPL];
#pragma unroll
    for (int i = 0; i < EPL; ++i) {
        int e = g + i * G, a = 0;
        if (e >= P) e = 0;
        while (e >= F - a) { e -= F - a; ++a; }
        ea[i] = a;
        eb[i] = a + e;
    }
    // two trajectories per warp (16-lane groups, mixed path, P <= 64): the coupling tensors
    // live in registers.  x = (q, qq) is cut into two halves of KH elements; lane ln holds,
    // for its half hx = ln / 16, the matching parts of the tensor rows of the entries
    // jx + 16 i (jx = ln % 16, i < EPH), and multiplies them by both trajectories' halves of
    // x (read as warp-broadcast 16-byte loads).  Lanes ln and ln ^ 16 then exchange partial
    // sums so that each ends with whole entries of its own trajectory.
    constexpr bool kPair = (T == 2) && TL::staged && (P <= 64) && (P > 16);
    constexpr bool kTreg = kPair && lg_tensor_regs<F>();
    // or the same cut with the tensor rows read from shared memory (TL::split)
    constexpr bool kSplit = kPair && !kTreg && TL::split;
    static_assert(kPair == (kTreg || kSplit), "two-trajectory warps take one of the two half-split schedules");
    static_assert(!kPair || Sh::kHalves, "the half-split schedules need the halves of x");
    constexpr int F3E = Sh::F3E, KH = Sh::KH, KHS = TL::KHS;
    constexpr int EPH = (kTreg || kSplit) ? (P + 15) / 16 : 1;
    const int hx = ln >> 4, jx = ln & 15;
    int ebA[EPH], ebB[EPH];
    float2 Tr[EPH][kTreg ? KH / 2 : 1];
    if constexpr (kSplit) {
#pragma unroll
        for (int i = 0; i < EPH; ++i) {
            const int e0 = jx + 16 * i;
            int e = e0 < P ? e0 : 0, a = 0;
            while (e >= F - a) { e -= F - a; ++a; }
            ebA[i] = a;
            ebB[i] = a + e;
        }
    }
    if constexpr (kTreg) {
#pragma unroll
        for (int i = 0; i < EPH; ++i) {
            const int e0 = jx + 16 * i;
            int e = e0 < P ? e0 : 0, a = 0;
            while (e >= F - a) { e -= F - a; ++a; }
            ebA[i] = a;
            ebB[i] = a + e;
#pragma unroll
            for (int k2 = 0; k2 < KH / 2; ++k2) {
                float v[2];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int gk = hx * KH + 2 * k2 + c;   // position in x
                    v[c] = 0.0f;
                    if (e0 < P) {
                        if (gk < F) v[c] = sT3[e0 * S3 + gk];
                        else if (gk >= F3E && gk - F3E < P) v[c] = sT4[e0 * S4 + gk - F3E];
                    }
                }
                Tr[i][k2] = make_float2(v[0], v[1]);
            }
        }
    }
    // tensors not staged: quads of consecutive entries 4 (g + i G) .. + 3, (a, b) packed as a | b << 8
    constexpr int NQ = TL::staged ? 1 : (P4 / 4 + G - 1) / G;
    int eq[TL::staged ? 1 : 4 * NQ];
    if constexpr (!TL::staged) {
#pragma unroll
        for (int i = 0; i < 4 * NQ; ++i) {
            int e = 4 * (g + (i / 4) * G) + i % 4, a = 0;
            if (e >= P) e = 0;
            while (e >= F - a) { e -= F - a; ++a; }
            eq[i] = a | ((a + e) << 8);
        }
    }

    // mode state (lane g < F)
    const int mode = g < F ? g : 0;
    using Coord = ff;
    Coord p, q;
    coord_set(p, L.p0[mode * n + jl]);
    coord_set(q, L.q0[mode * n + jl]);
    float pr = (float)coord_get(p);   // the momentum as seen by the FP32 bulk
    Coord S;                        // accumulated action (lane 0 of the group holds the total)
    coord_set(S, 0.0);
    // per-job action in the job table: the double-FP32 pair in the 8 bytes of a double (a phase: what a
    // denormal word adds is nothing)
    auto sj_put = [&](int j, Coord v) { reinterpret_cast<float2 *>(sh.Sj)[j] = make_float2(v.hi, v.lo); };
    auto sj_get = [&](int j) -> double {
        const float2 v = reinterpret_cast<const float2 *>(sh.Sj)[j];
        return widen_normal(v.x) + widen_normal(v.y);
    };
    // column state: slot s of lane g holds column c = g + s G of M = d(p,q)/d(p0,q0) (c < 2F;
    // a slot past 2F holds a zero column)
    float Mp[NCOL][F], Mq[NCOL][F];
#pragma unroll
    for (int s = 0; s < NCOL; ++s) {
        const int col = g + s * G;
#pragma unroll
        for (int a = 0; a < F; ++a) {
            Mp[s][a] = (col < F && a == col) ? 1.0f : 0.0f;
            Mq[s][a] = (col >= F && col < N2 && a == col - F) ? 1.0f : 0.0f;
        }
    }
    bool good = true;
    float stab = 0.0f;
    double detM_last = 1.0;
    double theta_last = 0.0, arg_last = 0.0;
    double2 detA_last = make_double2(1.0, 0.0);   // det A of the last step

    // amplitude at c = 0 (M = I, S = 0, theta = 0): lane 0 of each group
    if (g == 0 && active) {
        double re00 = 0.0;   // Re log <chi_0|p0 q0>
        for (int x = 0; x < A.n_chi; ++x) {
            double re = 0.0, im = 0.0;
            for (int a = 0; a < F; ++a) {
                const double pa = L.p0[a * n + jl], qa = L.q0[a * n + jl];
                const double dq = cc.q_eq[x][a] - qa, dp = cc.p_eq[x][a] - pa;
                re = fma(-cc.qw[a] * dq, dq, re);
                re = fma(-cc.pw[a] * dp, dp, re);
                im = fma(0.5 * (cc.p_eq[x][a] + pa), dq, im);
            }
            if (x == 0) re00 = re;
            // what the Herman-Kluk summand divides by: <chi_x|p0 q0> |<p0 q0|chi_0>|^2 / |<p0 q0|chi_x>|^2,
            // i.e. the initial overlap times the importance weight of the sampling density (the first
            // reference state's); its real logarithm 2 re00 - re equals re for x = 0
            const double rdiv = x == 0 ? re : 2.0 * re00 - re;
            sh.ov0[x][t] = make_double2(rdiv, im);
            double sn, cs;
            sincos(im, &sn, &cs);
            const double mag = exp(re);
            // the Herman-Kluk summand at t = 0 (C = 1, S = 0) is |<chi_x|p0 q0>|^2 / |<chi_0|p0 q0>|^2,
            // exactly 1 for x = 0
            if (A.amplitude == SCIVR_AMP_HK) amp_store(L, x * L.chi_stride + jl * L.amp_ld, x == 0 ? 1.0 : exp(re - rdiv), 0.0);
            else amp_store(L, x * L.chi_stride + jl * L.amp_ld, mag * cs, mag * sn);
        }
    }

    for (int step0 = 0; step0 < A.n_steps; step0 += C) {
        const int cnt = min(C, A.n_steps - step0);
        // ---------------- phase 1: cnt steps, group-parallel ----------------
        for (int c = 0; c < cnt; ++c) {
            float dS = 0.0f;   // this lane's share of the step's action increment
#pragma unroll 1
            for (int sub = 0; sub < 4; ++sub) {
                // drift: q += tau p, S += tau p.p/2, M_q += tau M_p
                {
                    const float rt = A.tdrift_f[sub];
                    if (g < F) {
                        q = coord_axpy(q, A.tdrift_f[sub], A.tdrift_lo[sub], p);
                        dS = fma(rt * 0.5f * pr, pr, dS);
                    }
                    const float2 rt2 = make_float2(rt, rt);
#pragma unroll
                    for (int s = 0; s < NCOL; ++s) {
#pragma unroll
                        for (int a = 0; a + 1 < F; a += 2) {
                            const float2 r = ffma2(rt2, make_float2(Mp[s][a], Mp[s][a + 1]), make_float2(Mq[s][a], Mq[s][a + 1]));
                            Mq[s][a] = r.x;
                            Mq[s][a + 1] = r.y;
                        }
                        if constexpr (F % 2) Mq[s][F - 1] = fmaf(rt, Mp[s][F - 1], Mq[s][F - 1]);
                    }
                }
                if (sub == 3) break;
                // kick: potential at q
                const float rtk = A.tkick_f[sub];
                __syncwarp();   // previous kick's readers of qr/H are done
                if (g < F) {
                    sh.qr[t][g] = (float)coord_f(q);
                    if constexpr (kTreg || kSplit) sh.xs[t][g] = (float)coord_f(q);
                    if constexpr (kCoop) xall[g * CH::XW + CH::slot(warp)] = (float)coord_f(q);
                }
                __syncwarp();
#pragma unroll
                for (int i = 0; i < EPL; ++i) {
                    const int e = g + i * G;
                    if (e < P) {
                        const float v = sh.qr[t][ea[i]] * sh.qr[t][eb[i]];
                        if constexpr (kTreg || kSplit) sh.xs[t][F3E + e] = v;
                        else sh.qq[t][e] = v;
                        if constexpr (kCoop) xall[(F + e) * CH::XW + CH::slot(warp)] = (float)v;
                    }
                }
                __syncwarp();
                float vpart = 0.0f;
                if constexpr (kCoop) {
                    __syncthreads();   // every warp's x is written; every warp has read its last h3, h4
                    contract(c);
                    __syncthreads();
                    const float *s3 = sh.h3_at(c), *s4 = sh.h4_at(c);
                    auto entry = [&](int e, int a, int b) {
                        const float h3 = s3[e], h4 = s4[e];
                        const float h = h3 + h4;
                        sh.H(t, a, b) = h;
                        sh.H(t, b, a) = h;
                        const float gce = fmaf(0.5f, h3, h4 * (1.0f / 3.0f));
                        sh.Gc[t][a][b] = gce;
                        sh.Gc[t][b][a] = gce;
                        const float vc = fmaf(1.0f / 6.0f, h3, h4 * (1.0f / 12.0f));
                        vpart = fmaf(a == b ? vc : 2.0f * vc, sh.qq[t][e], vpart);
                    };
                    if constexpr (STAGED) {
#pragma unroll
                        for (int i = 0; i < EPL; ++i)
                            if (g + i * G < P) entry(g + i * G, ea[i], eb[i]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 4 * NQ; ++i) {
                            const int e = 4 * (g + (i / 4) * G) + i % 4;
                            if (e < P) entry(e, eq[i] & 255, eq[i] >> 8);
                        }
                    }
                } else if constexpr (CUBIC) {
                    // a lane's quads of entries against the cubic rows in L2, 4 F multiply-adds each
                    const float4 *T3v = reinterpret_cast<const float4 *>(pes.T3p);
#pragma unroll
                    for (int i = 0; i < NQ; ++i) {
                        const int q4 = g + i * G;
                        if (4 * q4 < P) {
                            float4 h = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                            if (use3) {
#pragma unroll 8
                                for (int k = 0; k < F; ++k) {
                                    const float4 tv = __ldg(T3v + k * (P4 / 4) + q4);
                                    const float x = sh.qr[t][k];
                                    h.x = fmaf(tv.x, x, h.x); h.y = fmaf(tv.y, x, h.y);
                                    h.z = fmaf(tv.z, x, h.z); h.w = fmaf(tv.w, x, h.w);
                                }
                            }
                            const float hj[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int e = 4 * q4 + j;
                                if (e < P) {
                                    const int a = eq[4 * i + j] & 255, b = eq[4 * i + j] >> 8;
                                    sh.H(t, a, b) = hj[j];
                                    sh.H(t, b, a) = hj[j];
                                    sh.Gc[t][a][b] = 0.5f * hj[j];
                                    sh.Gc[t][b][a] = 0.5f * hj[j];
                                    const float vc = (1.0f / 6.0f) * hj[j];
                                    vpart = fmaf(a == b ? vc : 2.0f * vc, sh.qq[t][e], vpart);
                                }
                            }
                        }
                    }
                } else if constexpr (kTreg || kSplit) {
                    float2 aF[EPH][2], a4[EPH][2];   // packed partial sums per entry and trajectory
                    float sF[EPH][2];                // the first F3E elements of x (q in half 0)
#pragma unroll
                    for (int i = 0; i < EPH; ++i)
#pragma unroll
                        for (int tt = 0; tt < 2; ++tt) {
                            aF[i][tt] = a4[i][tt] = make_float2(0.0f, 0.0f);
                            sF[i][tt] = 0.0f;
                        }
                    const float *x0 = &sh.xs[0][hx * KH], *x1 = &sh.xs[1][hx * KH];
                    const float *trow[EPH];          // kSplit: this lane's rows (entries past P read row 0)
#pragma unroll
                    for (int i = 0; i < EPH; ++i) {
                        const int e = jx + 16 * i;
                        trow[i] = sTh + (hx * P + (e < P ? e : 0)) * KHS;
                    }
                    // a surface without couplings (uniform over the CTA) leaves every sum zero
                    if (use3 || use4)
#pragma unroll
                    for (int c = 0; c < KH; c += 4) {
                        const float4 u = *reinterpret_cast<const float4 *>(x0 + c);
                        const float4 w = *reinterpret_cast<const float4 *>(x1 + c);
                        float4 tv[EPH];
                        if constexpr (kSplit) {
#pragma unroll
                            for (int i = 0; i < EPH; ++i) tv[i] = *reinterpret_cast<const float4 *>(trow[i] + c);
                        }
#pragma unroll
                        for (int hp = 0; hp < 2; ++hp) {
                            const int kk = c + 2 * hp;
                            const float2 xu = hp ? hi2(u) : lo2(u), xw = hp ? hi2(w) : lo2(w);
#pragma unroll
                            for (int i = 0; i < EPH; ++i) {
                                float2 t2;
                                if constexpr (kSplit) t2 = hp ? hi2(tv[i]) : lo2(tv[i]);
                                else t2 = Tr[i][kk / 2];
                                if (kk < F3E) {
                                    aF[i][0] = ffma2(t2, xu, aF[i][0]);
                                    aF[i][1] = ffma2(t2, xw, aF[i][1]);
                                } else {
                                    a4[i][0] = ffma2(t2, xu, a4[i][0]);
                                    a4[i][1] = ffma2(t2, xw, a4[i][1]);
                                }
                            }
                            if (kk + 2 == F3E) {
#pragma unroll
                                for (int i = 0; i < EPH; ++i)
#pragma unroll
                                    for (int tt = 0; tt < 2; ++tt) sF[i][tt] = aF[i][tt].x + aF[i][tt].y;
                            }
                        }
                    }
                    // half 0 holds the cubic rows (h3) and the first pair products; half 1 only
                    // pair products.  Keep trajectory hx, pass the partner its trajectory's sums.
                    float vp = 0.0f;
#pragma unroll
                    for (int i = 0; i < EPH; ++i) {
                        float s3[2], s4[2];
#pragma unroll
                        for (int tt = 0; tt < 2; ++tt) {
                            const float r = a4[i][tt].x + a4[i][tt].y;
                            s3[tt] = hx == 0 ? sF[i][tt] : 0.0f;
                            s4[tt] = hx == 0 ? r : sF[i][tt] + r;
                        }
                        const float o3 = __shfl_xor_sync(FULL, hx ? s3[0] : s3[1], 16);
                        const float o4 = __shfl_xor_sync(FULL, hx ? s4[0] : s4[1], 16);
                        const float h3 = (hx ? s3[1] : s3[0]) + o3, h4 = (hx ? s4[1] : s4[0]) + o4;
                        const int e = jx + 16 * i;
                        if (e < P) {
                            const int a = ebA[i], b = ebB[i];
                            const float h = h3 + h4;
                            sh.H(hx, a, b) = h;
                            sh.H(hx, b, a) = h;
                            const float gce = fmaf(0.5f, h3, h4 * (1.0f / 3.0f));
                            sh.Gc[hx][a][b] = gce;
                            sh.Gc[hx][b][a] = gce;
                            const float vc = fmaf(1.0f / 6.0f, h3, h4 * (1.0f / 12.0f));
                            vp = fmaf(a == b ? vc : 2.0f * vc, sh.xs[hx][F3E + e], vp);
                        }
                    }
                    vpart = vp;   // lane ln belongs to group hx = t
                } else
#pragma unroll
                for (int i = 0; i < EPL; ++i) {
                    const int e = g + i * G;
                    if (e < P) {
                        const float h3 = use3 ? dot16<S3>(sT3 + e * S3, sh.qr[t]) : 0.0f;
                        const float h4 = use4 ? dot16<S4>(sT4 + e * S4, sh.qq[t]) : 0.0f;
                        const int a = ea[i], b = eb[i];
                        // coupling part only: the mode lanes add the diagonal term below
                        const float h = h3 + h4;
                        sh.H(t, a, b) = h;
                        sh.H(t, b, a) = h;
                        const float gce = fma(0.5f, h3, h4 * (1.0f / 3.0f));
                        sh.Gc[t][a][b] = gce;
                        sh.Gc[t][b][a] = gce;
                        const float vc = fma((1.0f / 6.0f), h3, h4 * (1.0f / 12.0f));
                        vpart = fma(a == b ? vc : 2.0f * vc, sh.qq[t][e], vpart);
                    }
                }
                __syncwarp();
                // gradient, p and action (mode lanes)
                float vlane = vpart;
                if (g < F) {
                    const float gr = dot16<S3>(sh.Gc[t][g], sh.qr[t]);
                    float Vd, gd, hd;   // the separable diagonal: value, gradient, Hessian
                    if (pes.diag_kind == SCIVR_DIAG_MORSE) {
                        const float Dm = cc.Df[g], am = cc.af[g];
                        const float u = expf(-am * sh.qr[t][g]);
                        const float omu = 1.0f - u;
                        Vd = Dm * omu * omu;
                        gd = 2.0f * Dm * am * u * omu;
                        hd = 2.0f * Dm * am * am * u * (2.0f * u - 1.0f);
                    } else {
                        const float w2 = cc.w2f[g];
                        Vd = 0.5f * w2 * sh.qr[t][g] * sh.qr[t][g];
                        gd = w2 * sh.qr[t][g];
                        hd = w2;
                    }
                    sh.H(t, g, g) += hd;
                    p = coord_kick(p, A.tkick_f[sub], A.tkick_lo[sub], gr + gd);
                    pr = (float)coord_f(p);
                    vlane += Vd;
                }
                __syncwarp();   // H complete before the monodromy kick reads it
                dS = fma(-rtk, vlane, dS);
                // monodromy kick: M_p -= tau H M_q (column lanes; rows of H by 16-byte broadcast loads)
                {
                    // packed pairs of H's row entries against pairs of the column's entries
                    constexpr int SH = Sh::SH;
                    float2 acc[NCOL];
#pragma unroll
                    for (int v0 = 0; v0 < F * SH; v0 += 4) {
                        const float4 v = *reinterpret_cast<const float4 *>(&sh.Hs[t][v0]);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int a = (v0 + 2 * h) / SH, b = (v0 + 2 * h) % SH;
                            if (a < F && b < F) {
                                const float2 hv = h ? hi2(v) : lo2(v);
#pragma unroll
                                for (int s = 0; s < NCOL; ++s) {
                                    if (b == 0) acc[s] = make_float2(0.0f, 0.0f);
                                    if (b + 1 < F) acc[s] = ffma2(hv, make_float2(Mq[s][b], Mq[s][b + 1]), acc[s]);
                                    else acc[s].x = fmaf(hv.x, Mq[s][b], acc[s].x);
                                    if (b + 2 >= F) Mp[s][a] = fmaf(-rtk, acc[s].x + acc[s].y, Mp[s][a]);
                                }
                            }
                        }
                    }
                }
            }
            // ---- Herman-Kluk matrix column b = g (needs column F + b) ----
            {
                // column F + g sits in lane (F + g) % G; a lane h sends column h (h >= F, slot 0)
                // or column h + G (h < F, slot 1) -- the only one any mode lane asks it for
                const int src = base + (F + (g < F ? g : 0)) % G;
                const int job = t * C + c;
#pragma unroll
                for (int a = 0; a < F; ++a) {
                    float sp, sq;
                    if constexpr (NCOL == 1) { sp = Mp[0][a]; sq = Mq[0][a]; }
                    else { sp = g >= F ? Mp[0][a] : Mp[1][a]; sq = g >= F ? Mq[0][a] : Mq[1][a]; }
                    const float mpq = __shfl_sync(FULL, sp, src);
                    const float mqq = __shfl_sync(FULL, sq, src);
                    if (g < F) {
                        const float4 k4 = *reinterpret_cast<const float4 *>(sAc + 4 * (a * F + g));
                        sh.a_at(job, a, g) = make_float4(fma(k4.x, mqq, k4.y * Mp[0][a]), fma(k4.z, Mq[0][a], k4.w * mpq), 0.0f, 0.0f);
                    }
                }
                if (g < F) {
                    sh.pj[g][jswz<JOBS>(g, job)] = pr;   // p did not change since the last kick set pr
                    sh.qj[g][jswz<JOBS>(g, job)] = (float)coord_f(q);
                }
                // the step's action increment, summed over the group, joins the running action
#pragma unroll
                for (int o = G / 2; o > 0; o >>= 1) dS += __shfl_xor_sync(FULL, dS, o, G);
                if (g == 0) {
                    S = coord_add(S, dS);
                    sj_put(job, S);
                }
            }
        }
        {
            // non-finite state persists, so testing once per chunk marks the same trajectories
            const unsigned bad_bits = __ballot_sync(FULL, (g < F) && !(coord_finite(p) && coord_finite(q)));
            const unsigned gmask = (G == 32 ? FULL : (((1u << G) - 1u) << base));
            if (bad_bits & gmask) good = false;
        }
        __syncwarp();
        // ---------------- phase 2: det A per job ----------------
        const int jc = g;                 // phases 3-4: this lane's step of its trajectory (job t * C + jc)
        const int jb = t * C + jc;
        const bool jvalid = jc < cnt;
        double argA = 0.0;                // arg det A of this lane's job (principal value)
        double2 detA = make_double2(1.0, 0.0);
        {
            // The entries of A are FP32 (formed from the FP32 monodromy) and the
            // elimination runs in double-FP32 on the FP32 pipe, so det A carries FP64-class
            // accuracy for those entries.  LPJ lanes share a job: the rows still to be
            // eliminated are dealt out over them through a permutation (a 4-bit field per row
            // up to F = 16, 5 bits above, in two 64-bit words; positions k.. are the active
            // rows), the pivot is an arg-max of
            // |a_ik|^2 over the job's lanes, and det A is the product of the pivots,
            // its sign flipped per exchange of the permutation.
            constexpr int LPJ = 32 / JOBS;
            static_assert(LPJ * JOBS == 32, "jobs must tile the warp");
            const int job = ln / LPJ, r = ln % LPJ;
            auto at = [&](int row, int col) -> float4 & { return sh.a_at(job, row, col); };
            constexpr int PB = F > 16 ? 5 : 4, PPW = 64 / PB;   // bits per field, fields per word
            constexpr unsigned long long PMASK = (1ull << PB) - 1ull;
            unsigned long long perm0 = 0ull, perm1 = 0ull;
#pragma unroll
            for (int i = 0; i < F; ++i) {
                if (i < PPW) perm0 |= (unsigned long long)i << (PB * i);
                else perm1 |= (unsigned long long)i << (PB * (i - PPW));
            }
            auto prow = [&](int pos) -> int {
                return pos < PPW ? (int)((perm0 >> (PB * pos)) & PMASK) : (int)((perm1 >> (PB * (pos - PPW))) & PMASK);
            };
            auto pset = [&](int pos, unsigned long long v) {
                if (pos < PPW) perm0 = (perm0 & ~(PMASK << (PB * pos))) | (v << (PB * pos));
                else perm1 = (perm1 & ~(PMASK << (PB * (pos - PPW)))) | (v << (PB * (pos - PPW)));
            };
            bool odd = false;   // parity of the exchanges
            // pivot candidate of the next column among this lane's rows: the largest |a_ik|^2
            // (leading words), taken here for column 0 and from the updates afterwards
            float best = -1.0f;
            int bpos = 0;
            auto candidate = [&](const float4 &v, int pos) {
                const float m = fmaf(v.x, v.x, v.y * v.y);
                if (m > best) { best = m; bpos = pos; }
            };
            for (int pos = r; pos < F; pos += LPJ) candidate(at(pos, 0), pos);
#pragma unroll 1
            for (int k = 0; k < F; ++k) {
#pragma unroll
                for (int o = 1; o < LPJ; o <<= 1) {
                    const float ob = __shfl_xor_sync(FULL, best, o);
                    const int op = __shfl_xor_sync(FULL, bpos, o);
                    if (ob > best || (ob == best && op < bpos)) { best = ob; bpos = op; }
                }
                if (bpos != k) {
                    const unsigned long long a = (unsigned long long)prow(k), b = (unsigned long long)prow(bpos);
                    pset(k, b);
                    pset(bpos, a);
                    odd = !odd;
                }
                const int pr = prow(k);
                const float4 pk4 = at(pr, k);
                const ff pre = {pk4.x, pk4.z}, pim = {pk4.y, pk4.w};
                // 1 / pivot = conj(pivot) / |pivot|^2
                const ff m2 = ff_add(ff_mul(pre, pre), ff_mul(pim, pim));
                const ff rm = ff_recip(m2);
                const ff ir = ff_mul(pre, rm);
                const ff nii = ff_mul(pim, rm);
                const ff ii = {-nii.hi, -nii.lo};
                // The rows below the pivot go to the job's lanes, or, once there are fewer rows than
                // lanes, 2^sp lanes to a row, which share its columns.  With eight or more lanes to a
                // job a lane's two rows are updated together, each pivot-row entry read once for both
                // (with four, 5 % slower at F = 9).
                const int m = F - 1 - k;
                int sp = 0;
                if constexpr (LPJ >= 4) {
                    if (m > 0) sp = max(0, (31 - __clz(LPJ)) - (32 - __clz(m - 1)));
                }
                const int c0 = k + 1 + (r & ((1 << sp) - 1)), cstep = 1 << sp, rstep = LPJ >> sp;
                const float4 *prow_p = &at(pr, 0);
                best = -1.0f;
                bpos = k + 1;
                auto multiplier = [&](const float4 *row) {
                    const float4 aik = row[k];
                    const ff ar = {aik.x, aik.z}, ai = {aik.y, aik.w};
                    const ff zero = {0.0f, 0.0f};
                    const ff lr = ff_sub_mul_add_mul(zero, ai, ii, ar, ir);                       // ar ir - ai ii
                    const ff li = ff_sub_mul_add_mul(zero, {-ar.hi, -ar.lo}, ii, ai, ir);         // ar ii + ai ir
                    return ElimRow(lr, li);
                };
                if constexpr (LPJ >= 8) {
                    for (int s0 = k + 1; s0 < F; s0 += 2 * rstep) {
                        const int p0 = s0 + (r >> sp), p1 = p0 + rstep;
                        if (s0 + rstep < F) {      // some lane has two rows (uniform over the warp)
                            const bool on = p1 < F;
                            float4 *r0 = &at(prow(p0), 0), *r1 = on ? &at(prow(p1), 0) : r0;
                            const ElimRow l0 = multiplier(r0), l1 = multiplier(r1);
                            for (int cc = c0; cc < F; cc += cstep) {
                                const float4 pv = prow_p[cc];
                                const float4 n0 = elim_update(r0[cc], l0, pv), n1 = elim_update(r1[cc], l1, pv);
                                if (on) r1[cc] = n1;
                                r0[cc] = n0;
                                if (cc == k + 1) {
                                    candidate(n0, p0);
                                    if (on) candidate(n1, p1);
                                }
                            }
                        } else if (p0 < F) {
                            float4 *r0 = &at(prow(p0), 0);
                            const ElimRow l0 = multiplier(r0);
#pragma unroll 2
                            for (int cc = c0; cc < F; cc += cstep) {
                                const float4 n0 = elim_update(r0[cc], l0, prow_p[cc]);
                                r0[cc] = n0;
                                if (cc == k + 1) candidate(n0, p0);
                            }
                        }
                    }
                } else {
                    for (int p0 = k + 1 + (r >> sp); p0 < F; p0 += rstep) {
                        float4 *r0 = &at(prow(p0), 0);
                        const ElimRow l0 = multiplier(r0);
#pragma unroll 2
                        for (int cc = c0; cc < F; cc += cstep) {
                            const float4 n0 = elim_update(r0[cc], l0, prow_p[cc]);
                            r0[cc] = n0;
                            if (cc == k + 1) candidate(n0, p0);
                        }
                    }
                }
                if (LPJ > 1) __syncwarp();   // rows updated by the job's other lanes feed the next pivot
            }
            // det A, the product of the pivots (left in place): double-FP32 (re, im) times 2^dexp,
            // renormalised by an exact power of two after every factor (the FP32 exponent range alone
            // could overflow); each lane multiplies its positions' pivots, then the lanes' products
            // meet pairwise
            ff dr = {1.0f, 0.0f}, di = {0.0f, 0.0f};
            int dexp = 0;
            auto factor = [&](ff fr, ff fi) {
                const ff a1 = ff_mul(dr, fr), a2 = ff_mul(di, fi), b1 = ff_mul(dr, fi), b2 = ff_mul(di, fr);
                dr = ff_add(a1, {-a2.hi, -a2.lo});
                di = ff_add(b1, b2);
                const float mx = fmaxf(fabsf(dr.hi), fabsf(di.hi));
                const int eb = (__float_as_int(mx) >> 23) & 255;   // biased exponent of the larger part
                if (eb > 0 && eb < 255) {
                    const float sc = __int_as_float((254 - eb) << 23);   // 2^(127 - eb): the larger part to [1, 2)
                    dr.hi *= sc; dr.lo *= sc; di.hi *= sc; di.lo *= sc;
                    dexp += eb - 127;
                }
            };
#pragma unroll 1
            for (int k = r; k < F; k += LPJ) {
                const float4 v = at(prow(k), k);
                factor({v.x, v.z}, {v.y, v.w});
            }
#pragma unroll
            for (int o = 1; o < LPJ; o <<= 1) {
                const ff fr = {__shfl_xor_sync(FULL, dr.hi, o), __shfl_xor_sync(FULL, dr.lo, o)};
                const ff fi = {__shfl_xor_sync(FULL, di.hi, o), __shfl_xor_sync(FULL, di.lo, o)};
                const int fe = __shfl_xor_sync(FULL, dexp, o);
                factor(fr, fi);
                dexp += fe;
            }
            if (odd) {
                dr = {-dr.hi, -dr.lo};
                di = {-di.hi, -di.lo};
            }
            if (r == 0) {
                const double mr = widen_normal(dr.hi) + widen_normal(dr.lo), mi = widen_normal(di.hi) + widen_normal(di.lo);
                // (the power of two does not change the argument; with atan2 and conversions the FP64 pipe was
                // busy 21 % of the time: F = 9, 65536 x 1000: 166.0 -> 161.1 ms, F = 15, 3001 x 501: 26.0 -> 24.9)
                sh.argj[job] = arg_normal(mr, mi, dr.hi, di.hi);
                if (step0 + cnt == A.n_steps) sh.detAj[job] = make_double2(ldexp(mr, dexp), ldexp(mi, dexp));
                if (A.amplitude == SCIVR_AMP_HK) sh.lnA[job] = 0.5 * (log(hypot(mr, mi)) + dexp * 0.69314718055994530942);
            }
            __syncwarp();
            if (jvalid) {
                argA = sh.argj[jb];
                detA = sh.detAj[jb];
            }
        }
        {
            // det M every kDetMEvery steps and at the last step (at a chunk end: M is unchanged
            // since): rows of M^T in the job matrices' storage, free once det A is done
            // (2F (2F + 1) words per trajectory fit in its 4 F^2 C words), row stride 2F + 1 so
            // that lanes reading one column of different rows hit different banks; a rolled
            // loop keeps the code and registers small
            static_assert(kDetMEvery % C == 0, "det M cadence falls on chunk ends");
            if ((step0 + cnt) % kDetMEvery == 0 || step0 + cnt == A.n_steps) {
                float (*Wm)[N2 + 1] = reinterpret_cast<float (*)[N2 + 1]>(&sh.A[0]) + t * N2;
                static_assert(sizeof(float) * T * N2 * (N2 + 1) <= sizeof(sh.A), "det M workspace");
#pragma unroll
                    for (int s = 0; s < NCOL; ++s) {
                        const int col = g + s * G;
                        if (col < N2) {
#pragma unroll
                            for (int a = 0; a < F; ++a) { Wm[col][a] = Mp[s][a]; Wm[col][F + a] = Mq[s][a]; }
                        }
                    }
                    __syncwarp();
                    float det = 1.0f;
                    unsigned long long unused = N2 == 64 ? ~0ull : (1ull << N2) - 1ull;
                    unsigned parity = 0u;
#pragma unroll 1
                    for (int k = 0; k < N2; ++k) {
                        unsigned key = 0u;
#pragma unroll
                        for (int s = 0; s < NCOL; ++s) {
                            const int col = g + s * G;
                            if (col < N2 && ((unused >> col) & 1ull)) {
                                const unsigned kk = (__float_as_uint(fabsf(Wm[col][k])) & ~63u) | (unsigned)(col + 1);
                                key = kk > key ? kk : key;
                            }
                        }
                        // one full-warp integer max per group (the other groups' lanes contribute 0)
                        unsigned kmax = 0u;
#pragma unroll
                        for (int tt = 0; tt < T; ++tt) {
                            const unsigned r = __reduce_max_sync(FULL, t == tt ? key : 0u);
                            kmax = (t == tt) ? r : kmax;
                        }
                        const int pc = (int)(kmax & 63u) - 1;
                        const float pk = Wm[pc][k];
                        const float inv = __fdividef(1.0f, pk);
                        parity ^= (unsigned)__popcll(unused & ((1ull << pc) - 1ull)) & 1u;
                        unused &= ~(1ull << pc);
                        det *= pk;
#pragma unroll
                        for (int s = 0; s < NCOL; ++s) {
                            const int col = g + s * G;
                            if (col < N2 && ((unused >> col) & 1ull)) {
                                const float l = Wm[col][k] * inv;
                                for (int i = k + 1; i < N2; ++i) Wm[col][i] = fmaf(-l, Wm[pc][i], Wm[col][i]);
                            }
                        }
                        __syncwarp();
                    }
                    if (parity) det = -det;
                    const float dev = isfinite(det) ? fabsf(fmaf(det, det, -1.0f)) : CUDART_INF_F;
                    stab = dev > stab ? dev : stab;
                    if (dev > A.stab_tol_f) good = false;
                    detM_last = (double)det;
            }
            __syncwarp();   // the next chunk's phase 1 refills the job matrices
        }
        // ---------------- phase 3: continuous phase (segmented scan) ----------------
        const double arg = argA;
        double arg_prev = __shfl_up_sync(FULL, arg, 1, G);
        if (g == 0) arg_prev = arg_last;
        double d = arg - arg_prev + A.ref_step;
        d = fma(-kTwoPi, rint(d * kInvTwoPi), d);
        double inc = jvalid ? d - A.ref_step : 0.0;
#pragma unroll
        for (int o = 1; o < C; o <<= 1) {
            const double v = __shfl_up_sync(FULL, inc, o, G);
            if (g >= o) inc += v;
        }
        const double theta = theta_last + inc;
        const int lastlane = base + cnt - 1;     // lane of the chunk's last step of this trajectory
        theta_last = __shfl_sync(FULL, theta, lastlane);
        arg_last = __shfl_sync(FULL, arg, lastlane);
        detA_last.x = __shfl_sync(FULL, detA.x, lastlane);
        detA_last.y = __shfl_sync(FULL, detA.y, lastlane);
        if (!finite_bits(theta_last)) good = false;
        // ---------------- phase 4: amplitudes (job-parallel) ----------------
        // a chunk of one step has one job: the group's lanes take its reference states instead (eight of
        // them, 40 steps of 4000 F = 24 trajectories: 16.9 -> 15.9 ms, uncoupled 10.1 -> 9.2)
        constexpr bool kStates = C == 1;
        const int jr = kStates ? t : jb;
        if ((kStates ? g < A.n_chi : jvalid) && active) {
            const double S = sj_get(jr), th = kStates ? theta_last : theta;
            for (int x = kStates ? g : 0; x < A.n_chi; x += kStates ? G : 1) {
                {
                    // the overlap's exponent and phase are O(1)-O(10) in size: FP32 from the FP32
                    // state copies; the action and the continuous phase join in FP64, and the
                    // total phase is reduced modulo 2 pi in FP64 before FP32 sine and cosine
                    float rf = 0.0f, imf = 0.0f;
#pragma unroll
                    for (int a = 0; a < F; ++a) {
                        const float pa = sh.pj[a][jswz<JOBS>(a, jr)], qa = sh.qj[a][jswz<JOBS>(a, jr)];
                        const float dq = cc.q_eqf[x][a] - qa, dp = cc.p_eqf[x][a] - pa;
                        rf = fmaf(-cc.qwf[a] * dq, dq, rf);
                        rf = fmaf(-cc.pwf[a] * dp, dp, rf);
                        imf = fmaf(0.5f * (cc.p_eqf[x][a] + pa), dq, imf);
                    }
                    double ph = fma(0.5, th, widen_normal(imf) + S);
                    if (A.amplitude == SCIVR_AMP_HK) {
                        // Herman-Kluk summand: |det A|^{1/2} and the division by the initial
                        // overlap times the sampling weight
                        const double2 o = sh.ov0[x][t];
                        rf = (float)((double)rf - o.x + sh.lnA[jr]);
                        ph -= o.y;
                    }
                    const double red = fma(-kTwoPi, rint(ph * kInvTwoPi), ph);   // FP64 reduction to [-pi, pi]
                    float sf, cf;
                    sincosf((float)red, &sf, &cf);
                    const float mag = expf(rf);
                    const int64_t ia = x * L.chi_stride + jl * L.amp_ld + step0 + (kStates ? 0 : jc) + 1;
                    if (L.amp_f32) reinterpret_cast<float2 *>(L.amp)[ia] = make_float2(mag * cf, mag * sf);
                    else L.amp[ia] = make_double2((double)(mag * cf), (double)(mag * sf));
                }
            }
        }
        {
            const float2 v = reinterpret_cast<const float2 *>(sh.Sj)[t * C + cnt - 1];
            if (!(isfinite(v.x) && isfinite(v.y))) good = false;
        }
        __syncwarp();
    }

    if (active) {
    if (g == 0) L.good[jl] = good ? 1 : 0;
    const FinalDev &fo = L.fin;
    if (g < F) {
        if (fo.p) fo.p[g * n + jl] = coord_get(p);
        if (fo.q) fo.q[g * n + jl] = coord_get(q);
    }
    if (g == 0) {
        if (fo.S) fo.S[jl] = sj_get(t * C + ((A.n_steps - 1) % C));
        if (fo.theta) fo.theta[jl] = theta_last;
        if (fo.detM) fo.detM[jl] = detM_last;
        if (fo.stab) fo.stab[jl] = (double)stab;
        if (fo.detA) { fo.detA[2 * jl] = detA_last.x; fo.detA[2 * jl + 1] = detA_last.y; }
    }
    if (fo.M) {
#pragma unroll
        for (int s = 0; s < NCOL; ++s) {
            const int col = g + s * G;
            if (col < N2) {
#pragma unroll
                for (int a = 0; a < F; ++a) {
                    fo.M[jl * N2 * N2 + a * N2 + col] = (double)Mp[s][a];
                    fo.M[jl * N2 * N2 + (F + a) * N2 + col] = (double)Mq[s][a];
                }
            }
        }
    }
    }
    __syncthreads();   // the caller may restage shared memory next
}

template <int F, int G, int WARPS, int TRAJ_WARPS, bool CUBIC>
__global__ void __launch_bounds__(32 * WARPS, lg_min_ctas<F, G>()) k_propagate_lg(const PropLaunch L)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    lg_body<F, G, WARPS, (F <= 16 && !CUBIC), TRAJ_WARPS, CUBIC>(L, blockIdx.x, smem_raw);
}

// Batched persistent kernel: CTAs pull (molecule, tile) work items from a
// list sorted by decreasing cost until it is exhausted.  items: device array
// of per-molecule launches (all of this F); work: (item, tile) pairs.
template <int F, int G, int WARPS, bool CUBIC>
__global__ void __launch_bounds__(32 * WARPS, lg_min_ctas<F, G>()) k_propagate_lg_batch(const PropLaunch *__restrict__ items,
                                                                       const int2 *__restrict__ work,
                                                                       int n_work, int *__restrict__ counter)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int next;
    for (;;) {
        if (threadIdx.x == 0) next = atomicAdd(counter, 1);
        __syncthreads();
        const int w = next;
        __syncthreads();
        if (w >= n_work) break;
        const int2 it = work[w];
        lg_body<F, G, WARPS, (F <= 16 && !CUBIC), WARPS, CUBIC>(items[it.x], it.y, smem_raw);
    }
}

// One persistent launch for molecules of several F: CTAs of four warps pull (molecule,
// tile) work items from one list (all molecules, sorted by decreasing cost) and run the
// body specialised for each item's F.  Above F = 9 the coupling tensors are read from L2
// here, so that no class's shared memory sets the whole launch's occupancy.
template <int... Fs>
__global__ void __launch_bounds__(128, 1) k_propagate_lg_multi(const PropLaunch *__restrict__ items,
                                                               const int2 *__restrict__ work, int n_work,
                                                               int *__restrict__ counter)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int next;
    for (;;) {
        if (threadIdx.x == 0) next = atomicAdd(counter, 1);
        __syncthreads();
        const int w = next;
        __syncthreads();
        if (w >= n_work) break;
        const int2 it = work[w];
        const int F = items[it.x].args.F;
        const bool ran = ((F == Fs ? (lg_body<Fs, mixed_group_lanes(Fs), 4, (Fs <= 9)>(items[it.x], it.y, smem_raw),
                                      true)
                                   : false) ||
                          ...);
        (void)ran;
    }
}

}  // namespace lg

template <int F, int G, int WARPS, bool STAGED = (F <= 16), int TRAJ_WARPS = WARPS, bool CUBIC = false>
size_t lg_smem_bytes()
{
    using namespace lg;
    using TL = TensorLayout<F, STAGED, CUBIC>;
    const size_t consts = (sizeof(CtaConst<F>) + 15) & ~(size_t)15;
    size_t coop = 0;
    if constexpr (TL::coop) coop = CoopHessian<F, WARPS, TRAJ_WARPS, STAGED>::bytes;
    return TL::bytes + consts + coop + TRAJ_WARPS * sizeof(WarpShared<F, G, CUBIC>);
}

template <int F, int G, int WARPS, bool CUBIC = false>
cudaError_t launch_lg_batch(const PropLaunch *items, const int2 *work, int n_work, int *counter, int n_sm,
                            cudaStream_t s)
{
    using namespace lg;
    const size_t bytes = lg_smem_bytes<F, G, WARPS, (F <= 16 && !CUBIC), WARPS, CUBIC>();
    auto kern = k_propagate_lg_batch<F, G, WARPS, CUBIC>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    // the largest shared-memory carveout, so that as many CTAs fit as the registers allow
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * WARPS, bytes);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    int grid = n_sm * per_sm;
    if (grid > n_work) grid = n_work;
    if (grid < 1) return cudaSuccess;
    kern<<<grid, 32 * WARPS, bytes, s>>>(items, work, n_work, counter);
    return cudaGetLastError();
}

template <int F, int G, int WARPS, int TRAJ_WARPS = WARPS, bool CUBIC = false>
cudaError_t launch_lg(const PropLaunch &L, cudaStream_t s)
{
    using namespace lg;
    constexpr int T = 32 / G;
    const size_t bytes = lg_smem_bytes<F, G, WARPS, (F <= 16 && !CUBIC), TRAJ_WARPS, CUBIC>();
    auto kern = k_propagate_lg<F, G, WARPS, TRAJ_WARPS, CUBIC>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    // the largest shared-memory carveout, so that as many CTAs fit as the registers allow
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    const int64_t per_cta = (int64_t)TRAJ_WARPS * T;
    const int64_t blocks = (L.n_traj + per_cta - 1) / per_cta;
    kern<<<(unsigned)blocks, 32 * WARPS, bytes, s>>>(L);
    return cudaGetLastError();
}

// Launchers instantiated by the prop_lg_*.cu units: lanes per trajectory by F
// (2F columns must fit), warps per CTA, and the batch variants the tuner may pick.

template <int F> cudaError_t launch_group_mixed(const PropLaunch &L, cudaStream_t s)
{
    constexpr int G = mixed_group_lanes(F);
    constexpr int W = lg::lg_warps<F, G>();
    if constexpr (F > 13) {
        // few trajectories: two or four per CTA, so that they spread over the SMs and the other
        // warps share their Hessians (F = 24: 50 steps of 64 trajectories take 3.6 ms two to a CTA,
        // of 600 3.9 ms four to a CTA, of 1216 5.0 ms eight to a CTA)
        int dev = 0, n_sm = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        if constexpr (cubic_schedule(F)) {
            if (!L.pes.has4 && (F < 24 || !L.pes.has3 || L.n_traj > 4 * (int64_t)n_sm)) return launch_lg<F, G, 4, 4, true>(L, s);
        }
        if (L.n_traj <= 2 * (int64_t)n_sm) return launch_lg<F, G, W, 2>(L, s);
        if (L.n_traj <= 4 * (int64_t)n_sm) return launch_lg<F, G, W, 4>(L, s);
    }
    return launch_lg<F, G, W>(L, s);
}

template <int F>
cudaError_t launch_group_batch_mixed_F(int warps, const PropLaunch *items, const int2 *work, int n_work,
                                      int *counter, int n_sm, cudaStream_t s)
{
    constexpr int G = mixed_group_lanes(F);
    if constexpr (G == 32 && F > 9) {
        constexpr int W = lg::lg_warps<F, G>();
        if (warps == W) return launch_lg_batch<F, G, W>(items, work, n_work, counter, n_sm, s);
        if constexpr (cubic_schedule(F)) {
            static_assert(W != 4, "four warps mark the class without quartic terms");
            if (warps == 4) return launch_lg_batch<F, G, 4, true>(items, work, n_work, counter, n_sm, s);
        }
    } else if constexpr (G == 32) {
        if (warps == 1) return launch_lg_batch<F, G, 1>(items, work, n_work, counter, n_sm, s);
        if (warps == 2) return launch_lg_batch<F, G, 2>(items, work, n_work, counter, n_sm, s);
    } else {
        if (warps == 2) return launch_lg_batch<F, G, 2>(items, work, n_work, counter, n_sm, s);
        if (warps == 4) return launch_lg_batch<F, G, 4>(items, work, n_work, counter, n_sm, s);
    }
    return cudaErrorInvalidValue;
}

// The classes one persistent launch can hold, and the trajectories per work tile of each.
template <int... Fs>
struct MultiLaunch {
    static constexpr bool holds(int F) { return ((F == Fs) || ...); }
    static size_t smem_bytes()
    {
        size_t m = 0;
        ((m = std::max(m, lg_smem_bytes<Fs, mixed_group_lanes(Fs), 4, (Fs <= 9)>())), ...);
        return m;
    }
    static cudaError_t launch(const PropLaunch *items, const int2 *work, int n_work, int *counter, int n_sm,
                              cudaStream_t s)
    {
        const size_t bytes = smem_bytes();
        auto kern = lg::k_propagate_lg_multi<Fs...>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 128, bytes);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
        int grid = n_sm * per_sm;
        if (grid > n_work) grid = n_work;
        if (grid < 1) return cudaSuccess;
        kern<<<grid, 128, bytes, s>>>(items, work, n_work, counter);
        return cudaGetLastError();
    }
};


}  // namespace scivr
