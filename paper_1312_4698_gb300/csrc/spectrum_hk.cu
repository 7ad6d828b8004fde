// Plain Herman-Kluk SC-IVR spectrum (Eq. I(E)_SCIVR of arXiv:1312.4698) from
// the per-trajectory Herman-Kluk summands that scivr_propagate records with
// SCIVR_AMP_HK: the survival amplitude C(c dt) is their mean over the good
// trajectories (a column sum of the amplitude matrix, one read of
// 16 n K bytes), then I(E_k) = (dt/pi) Re[C(0)/2 + sum_{c>=1} C(c dt) e^{i E_k c dt}].
// Column sums are deterministic: each block sums a fixed slice of rows for
// 256 consecutive columns (coalesced along the time axis), and the slices'
// partials are added in slice order.
#include <cmath>

#include "fp64_ops.cuh"
#include "scivr_internal.cuh"

namespace scivr {
namespace {

constexpr int kColThreads = 256;
constexpr int kMaxSliceRows = 4096;   // flags of one slice staged in shared memory
constexpr int kMinSliceRows = 16;
// Blocks wanted for the column sum, 8 CTAs of 256 threads on each of 152 SMs: with fixed slices
// of 4096 rows (64 blocks at 16384 x 4001 summands) most of the chip was idle.
constexpr int kColBlocks = 152 * 8;

// Rows per slice: enough slices to reach kColBlocks, none shorter than kMinSliceRows.
inline int slice_rows(int64_t n, int K)
{
    const int64_t cols = (K + kColThreads - 1) / kColThreads;
    const int64_t slices = (kColBlocks + cols - 1) / cols;
    int64_t rows = (n + slices - 1) / slices;
    if (rows < kMinSliceRows) rows = kMinSliceRows;
    if (rows > kMaxSliceRows) rows = kMaxSliceRows;
    return (int)rows;
}

// Sum of one column's real or imaginary parts as a 128-bit integer in units of 2^(top - 1023 - kLead):
// a summand with the window's largest biased exponent, top, has its leading bit at kLead = 126 - kHead,
// so that 2^kHead summands, all rows of a slice, cannot overflow it, and one up to 2^62 times smaller
// keeps all of its bits (a smaller one is cut at the unit).  The window opens kRoom binades above the first
// summand and moves on when a larger one arrives; the integer is then rounded, once and correctly,
// into FP64, as it is at the end.  So a slice's sum carries one rounding where FP64 additions carry
// one for every row, and a part keeps its own precision however large the other part is.
// top = -1: no window.
constexpr int kHead = 12, kLead = 126 - kHead, kRoom = 8;
static_assert(kMaxSliceRows <= 1 << kHead, "a slice's rows fit the integer");

struct WideSum {
    int top = -1;
    unsigned neg = 0;                     // negative summands: each has been added as its complement, one unit low
    unsigned long long lo = 0, hi = 0;
    double out = 0.0;                     // what has left the integer, and summands beyond any window

    __device__ __forceinline__ void put(double x)
    {
        const int h = __double2hiint(x);
        const unsigned l = (unsigned)__double2loint(x);
        // the mantissa with its leading bit at 63, then moved down 128 bits' worth (shifts past the width give zero)
        const unsigned long long m = ((unsigned long long)(__funnelshift_l(l, (unsigned)h, 11) | 0x80000000u) << 32) | (l << 11);
        const int s = top - ((h >> 20) & 0x7ff) + (127 - kLead);
        unsigned long long vh, v1, v2;
        asm("shr.u64 %0, %1, %2;" : "=l"(vh) : "l"(m), "r"(s));
        asm("shl.b64 %0, %1, %2;" : "=l"(v1) : "l"(m), "r"(64 - s));
        asm("shr.u64 %0, %1, %2;" : "=l"(v2) : "l"(m), "r"(s - 64));
        const unsigned long long sign = (long long)(h >> 31);
        const unsigned long long vl = (v1 | v2) ^ sign;
        vh ^= sign;
        neg += (unsigned)h >> 31;
        asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;" : "+l"(lo), "+l"(hi) : "l"(vl), "l"(vh));
    }
    __device__ __forceinline__ void flush()
    {
        if (top < 0) return;
        lo += neg;
        hi += lo < neg ? 1 : 0;
        const bool minus = (long long)hi < 0;
        if (minus) {
            lo = 0 - lo;
            hi = ~hi + (lo == 0 ? 1 : 0);
        }
        int down = 0;                     // binades by which the leading bit is below 127
        if (hi == 0) {
            hi = lo;
            lo = 0;
            down = 64;
        }
        if (hi != 0) {
            const int z = __clzll(hi);
            if (z > 0) hi = (hi << z) | (lo >> (64 - z));
            lo <<= z;
            down += z;
            const double v = __ull2double_rn(hi | (lo != 0 ? 1 : 0));   // (a bit below the 53 stands for all of them)
            const double unit = __hiloint2double((top - kLead + 64 - down) << 20, 0);
            out = fma(minus ? -v : v, unit, out);
        }
        lo = hi = 0;
        neg = 0;
    }
    // the summands x[0..U) (zero where skipped)
    template <int U>
    __device__ __forceinline__ void add(const double (&x)[U])
    {
        int key = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) key = max(key, __double2hiint(x[u]) & 0x7fffffff);
        const int e = key >> 20;
        if (e > top) {
            flush();
            top = e < 200 || e == 0x7ff ? -1 : min(e + kRoom, 2046);
            if (top < 0) {   // near the smallest numbers, or not finite: in FP64
#pragma unroll
                for (int u = 0; u < U; ++u) out += x[u];
                return;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) put(x[u]);
    }
};

// Two additions per summand on the FP64 pipe bounded this sum (248 us at 16384 x 4001, against 156 us for
// one read of the summands from HBM), so the integer units
// add in its place (WideSum).  A thread owns one column and keeps eight 16-byte loads in flight; bad
// rows are loaded too (their flags, from shared memory, only select), so that no load waits for a
// branch.  The three launches at 16384 x 4001 summands, 4000 energies: 373 us with FP64 additions, 310 now (with the transform below); the integer units are 80 % busy,
// HBM at 63 % of the copy rate.
__global__ void __launch_bounds__(kColThreads, 4) k_hk_colsum(const double2 *__restrict__ amp, int64_t amp_ld,
                                                           const uint8_t *__restrict__ good, int64_t n, int K,
                                                           int rows, double2 *__restrict__ part)
{
    __shared__ uint8_t ok[kMaxSliceRows];
    const int64_t r0 = (int64_t)blockIdx.y * rows;
    const int cnt = (int)(n - r0 < rows ? n - r0 : rows);
    for (int i = threadIdx.x; i < cnt; i += kColThreads) ok[i] = good[r0 + i];
    __syncthreads();
    const int c = blockIdx.x * kColThreads + threadIdx.x;
    if (c >= K) return;
    const double2 *src = amp + r0 * amp_ld + c;
    WideSum re, im;
    constexpr int U = 8;
    int i = 0;
    for (; i + U <= cnt; i += U) {
        double2 a[U];
#pragma unroll
        for (int u = 0; u < U; ++u) a[u] = __ldcs(src + (i + u) * amp_ld);
        double x[U], y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool take = ok[i + u];   // bad rows never reach the sum, whatever they hold
            x[u] = take ? a[u].x : 0.0;
            y[u] = take ? a[u].y : 0.0;
        }
        re.add(x);
        im.add(y);
    }
#pragma unroll 1
    for (; i < cnt; ++i) {
        double x[1] = {0.0}, y[1] = {0.0};
        if (ok[i]) {
            const double2 a = __ldcs(src + i * amp_ld);
            x[0] = a.x;
            y[0] = a.y;
        }
        re.add(x);
        im.add(y);
    }
    re.flush();
    im.flush();
    part[(int64_t)blockIdx.y * K + c] = make_double2(re.out, im.out);
}

// Slices' partials in a fixed order (a thread of row y adds slices y, y + 8, ...; the 8 sums in
// order of y), divided by the good count.  Every block counts the flags: n bytes from L2, cheaper
// than a launch of its own.
constexpr int kRedX = 32, kRedY = 8;

__global__ void __launch_bounds__(kRedX *kRedY) k_hk_reduce(const double2 *__restrict__ part, int n_slices, int K,
                                                            const uint8_t *__restrict__ good, int64_t n,
                                                            int64_t *__restrict__ ng_out, double2 *__restrict__ C)
{
    __shared__ double2 sums[kRedY][kRedX];
    __shared__ int64_t cnts[kRedY];
    const int tid = threadIdx.y * kRedX + threadIdx.x;
    int64_t cnt = 0;
#pragma unroll 8
    for (int64_t j = tid; j < n; j += kRedX * kRedY) cnt += good[j] ? 1 : 0;
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if (threadIdx.x == 0) cnts[threadIdx.y] = cnt;
    const int c = blockIdx.x * kRedX + threadIdx.x;
    double sr = 0.0, si = 0.0;
    if (c < K) {
#pragma unroll 8
        for (int s = threadIdx.y; s < n_slices; s += kRedY) {
            const double2 v = part[(int64_t)s * K + c];
            sr += v.x;
            si += v.y;
        }
    }
    sums[threadIdx.y][threadIdx.x] = make_double2(sr, si);
    __syncthreads();
    if (threadIdx.y != 0) return;
    int64_t ng = 0;
    for (int y = 0; y < kRedY; ++y) ng += cnts[y];
    if (ng_out && blockIdx.x == 0 && threadIdx.x == 0) ng_out[0] = ng;
    if (c >= K) return;
    sr = si = 0.0;
#pragma unroll
    for (int y = 0; y < kRedY; ++y) {
        sr += sums[y][threadIdx.x].x;
        si += sums[y][threadIdx.x].y;
    }
    const double inv = ng > 0 ? 1.0 / (double)ng : 0.0;
    C[c] = make_double2(sr * inv, si * inv);
}

// Re sum_{c} C_c e^{i E_k c dt} on the FP64 pipe, whose rate (one warp instruction per 64
// cycles and sub-partition) is the bound: a sine and cosine per term (about 45 instructions)
// took 4.2 ms for 4001 samples and 4000 energies.  The samples are cut into blocks of
// 2 R + 1 around centres c_m = (2 R + 1) m + R:
//   sum_c C_c z^c = sum_m z^{c_m} S_m,   S_m = C_{c_m} + sum_{r=1}^{R} A_{m,r} cos(r t) + B_{m,r} sin(r t),
//   t = E dt, z = e^{i t}, A = C_{c_m + r} + C_{c_m - r}, B = i (C_{c_m + r} - C_{c_m - r}),
// so that a term costs two multiply-adds; A and B do not depend on the energy.  A thread owns
// an energy, a warp G consecutive blocks at a time (its A and B in shared memory, read as
// broadcasts), the kFtWarps warps of a CTA share 32 energies' blocks.  The powers z^r and the z^{c_m} of
// a warp's G blocks are complex products of a sine and cosine at r = 1, 8, 16, 24 and at the
// first centre, at most seven on end.  Whatever error these factors have is shared by many samples and does
// not average out, so the phases' own rounding is put back (unit_phase) and the products are kept few.
// With rounded phases and 30 products on end, spectra of 200 to 4000 samples were up to five times less
// accurate than with a phase for every sample; they are as accurate now, or more.
// 4001 samples x 4000 energies: 4234 -> 97 us (6.4e7 multiply-adds; the FP64 pipe takes 61 us for them).
constexpr int kFtR = 31, kFtW = 2 * kFtR + 1, kFtG = 8, kFtWarps = 8;
constexpr int kFtAnew = 8;   // powers of z from one sine and cosine
// Few samples take a sine and cosine per term, shared out over the CTA's warps.  Blocks take 50 us
// whatever one warp's hold (up to 504 samples); terms 0.3 us a sample while each CTA has an SM to itself, and
// with more CTAs the instructions count, 50 a term against 1500 for the blocks.  The three launches,
// blocks / terms: 400 energies, 2 samples 61 / 9 us, 128 samples 62 / 48; 4900 energies, 64 samples
// 66 / 48; 30000 energies, 64 samples 184 / 149.
inline int few_samples(int n_E) { return n_E <= 32 * 152 ? 128 : 80; }

__device__ __forceinline__ double2 hk_cmul(double2 x, double2 y)
{
    return make_double2(fma(x.x, y.x, -x.y * y.y), fma(x.x, y.y, x.y * y.x));
}

__global__ void __launch_bounds__(32 * kFtWarps) k_hk_ft(const double2 *__restrict__ C, int K, int few, double dt,
                                                         double E_min, double dE, int n_E, double *__restrict__ I_out)
{
    extern __shared__ __align__(16) double2 ab_all[];   // [warp][r][g]{A, B}
    __shared__ double part[kFtWarps][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double2 *ab = ab_all + warp * (kFtR + 1) * kFtG * 2;
    const int k = blockIdx.x * 32 + lane;
    const double E = E_min + k * dE;
    const int n_blk = (K + kFtW - 1) / kFtW, n_grp = (n_blk + kFtG - 1) / kFtG;
    auto at = [&](int c) -> double2 {
        if (c >= K) return make_double2(0.0, 0.0);
        double2 v = __ldg(C + c);
        if (c == 0) { v.x *= 0.5; v.y *= 0.5; }   // the folded transform's half weight at t = 0
        return v;
    };
    double acc = 0.0;
    if (K <= few) {
        for (int c = warp; c < K; c += kFtWarps) {
            const double2 v = at(c), ph = unit_phase(E, c, dt);
            acc = fma(v.x, ph.x, fma(-v.y, ph.y, acc));
        }
    } else {
        const double2 z = unit_phase(E, 1.0, dt), step = unit_phase(E, kFtW, dt);
        for (int grp = warp; grp < n_grp; grp += kFtWarps) {
            __syncwarp();
            for (int i = lane; i < (kFtR + 1) * kFtG; i += 32) {
                const int r = i / kFtG, c = (grp * kFtG + i % kFtG) * kFtW + kFtR;
                const double2 u = at(c + r), v = r ? at(c - r) : make_double2(0.0, 0.0);
                ab[2 * i] = make_double2(u.x + v.x, u.y + v.y);
                ab[2 * i + 1] = make_double2(v.y - u.y, u.x - v.x);
            }
            __syncwarp();
            double2 S[kFtG];
#pragma unroll
            for (int g = 0; g < kFtG; ++g) S[g] = ab[2 * g];
            double2 zr = z;
#pragma unroll 1
            for (int r = 1; r <= kFtR; ++r) {
                const double2 *row = ab + 2 * r * kFtG;
#pragma unroll
                for (int g = 0; g < kFtG; ++g) {
                    const double2 A = row[2 * g], B = row[2 * g + 1];
                    S[g].x = fma(A.x, zr.x, fma(B.x, zr.y, S[g].x));
                    S[g].y = fma(A.y, zr.x, fma(B.y, zr.y, S[g].y));
                }
                zr = r % kFtAnew == kFtAnew - 1 ? unit_phase(E, r + 1, dt) : hk_cmul(zr, z);
            }
            double2 ph = unit_phase(E, grp * kFtG * kFtW + kFtR, dt);
#pragma unroll
            for (int g = 0; g < kFtG; ++g) {
                acc = fma(S[g].x, ph.x, fma(-S[g].y, ph.y, acc));
                ph = hk_cmul(ph, step);
            }
        }
    }
    part[warp][lane] = acc;
    __syncthreads();
    if (warp == 0 && k < n_E) {
        double s = part[0][lane];
#pragma unroll
        for (int w = 1; w < kFtWarps; ++w) s += part[w][lane];
        I_out[k] = dt / 3.141592653589793238462643383280 * s;
    }
}

constexpr size_t kFtSmem = sizeof(double2) * kFtWarps * (kFtR + 1) * kFtG * 2;

}  // namespace

size_t spectrum_hk_scratch_bytes(int64_t n_traj, int n_steps)
{
    const int64_t K = n_steps + 1;
    const int rows = slice_rows(n_traj, (int)K);
    const int64_t slices = (n_traj + rows - 1) / rows;
    return (size_t)(slices * K + K) * sizeof(double2);
}

cudaError_t launch_spectrum_hk(const double2 *amp, int64_t amp_ld, const uint8_t *good, int64_t n_traj, int n_steps,
                               double dt, double E_min, double E_max, int n_E, double *I_out, double2 *C_out,
                               int64_t *n_good_out, void *scratch, cudaStream_t s, int *n_launch)
{
    const int K = n_steps + 1;
    const int rows = slice_rows(n_traj, K);
    const int slices = (int)((n_traj + rows - 1) / rows);
    double2 *part = static_cast<double2 *>(scratch);
    double2 *C = C_out ? C_out : part + (size_t)slices * K;
    const unsigned cols = (unsigned)((K + kColThreads - 1) / kColThreads);
    *n_launch = 0;
    cudaError_t e = cudaFuncSetAttribute(k_hk_ft, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFtSmem);
    if (e != cudaSuccess) return e;
    k_hk_colsum<<<dim3(cols, slices), kColThreads, 0, s>>>(amp, amp_ld, good, n_traj, K, rows, part);
    k_hk_reduce<<<(K + kRedX - 1) / kRedX, dim3(kRedX, kRedY), 0, s>>>(part, slices, K, good, n_traj, n_good_out, C);
    const double dE = n_E > 1 ? (E_max - E_min) / (n_E - 1) : 0.0;
    k_hk_ft<<<(n_E + 31) / 32, 32 * kFtWarps, kFtSmem, s>>>(C, K, few_samples(n_E), dt, E_min, dE, n_E, I_out);
    *n_launch = 3;
    return cudaGetLastError();
}

}  // namespace scivr
