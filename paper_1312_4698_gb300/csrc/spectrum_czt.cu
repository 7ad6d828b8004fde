// Time -> energy Fourier step of the time-averaged spectrum (Eq. I(E)_discreto of
// arXiv:1312.4698) in FP64 by the chirp-z transform: the same sums
//   X_j(E_k) = sum_{c=0}^{K-1} a_j(c) exp(i E_k c dt),  E_k = E_min + k dE,
// evaluated through Bluestein's identity k c = (k^2 + c^2 - (k - c)^2) / 2:
//   X_j(E_k) = exp(i w k^2/2) sum_c u_c v_{k-c},  w = dE dt,
//   u_c = a_j(c) exp(i (E_min c dt + w c^2/2)),  v_m = exp(-i w m^2/2),
// a linear convolution computed by FFTs of length L >= K + n_E - 1.  The output chirp
// has modulus one, so |X_j(E_k)|^2 = |(u * v)_k|^2.  Per trajectory this costs about
// 10 L log2 L FP64 flops instead of the direct sum's 8 K n_E: on GB300, whose FP64
// rate is 1/64 of FP32, the transform runs in O(L log L) on the FP64 pipe and keeps
// FP64 rounding (about log2(L) * 2^-53 of the largest |X|).
//
// Layout: the CTAs of a persistent grid loop over trajectories, one at a time, the whole
// length-L complex vector in shared memory.  Both transforms use the butterfly a +- w b, six
// FP64 instructions (a + w b by four multiply-adds, a - w b = 2 a - (a + w b) by two; the
// add-then-multiply form takes eight): the forward one splits the polynomial sum_c u_c z^c
// modulo z^h -+ r from the top (natural order in, bit-reversed out, one twiddle per block of
// a stage), the inverse one is decimation in time (bit-reversed in, natural out) of the
// conjugated product with V = FFT(v), conj(FFT(conj(.))) / L.  Three or four stages run in
// registers between two passes over shared memory: the first three take u from global memory
// as it is formed, the last four of the forward transform, the product with V and the first
// four of the inverse one share one pass over 16 contiguous points, and the last three of the
// inverse one go straight into the weighted |X|^2 sums.  Twiddles 1 and -i cost no products,
// the upper half of u is often zero (K <= L / 2) and the upper outputs unused.
// The FP64 pipe bounds it (85 % busy with radix-2 stages over shared memory too, but 223
// butterfly equivalents of L / 2 instructions per trajectory against 155 now).
// L is the shortest of 1024 .. 8192 points that is cheapest over the blocks of energies it
// needs (energies beyond L - K + 1 go to another block with its own input chirp): a water-sized
// run of 2001 samples and 2000 energies takes 4096 points.  1024 trajectories x 3001 samples x
// 2000 energies: 1903 -> 1199 us (95 % of the FP64 pipe), the four launches 2128 -> 1242 us;
// 4096 x 2001 x 4000: 7.13 -> 4.56 ms.
// Each CTA keeps its weighted |X|^2 sums in shared memory; a fixed-order reduction over CTAs
// follows (deterministic).
#include "scivr_internal.cuh"
#include "spectrum_reduce.cuh"

namespace scivr {
namespace {

constexpr int kLog2Max = 13, kLog2Min = 10;     // 8192 points: 128 KB of FP64 complex
constexpr int kVParts = 16;                     // CTAs that share the transform of the kernel chirp

__device__ __forceinline__ double2 cmul(double2 x, double2 y)
{
    return make_double2(fma(x.x, y.x, -x.y * y.y), fma(x.x, y.y, x.y * y.x));
}

// Shared-memory place of point i: the low three bits XOR bits 4..6, so that the 8 lanes of a
// 16-byte access wavefront hit different banks both with consecutive points and with points 16 apart.
__device__ __forceinline__ int place(int i) { return i ^ ((i >> 4) & 7); }

// (a, b) -> (a + w b, a - w b), w = 1, -i, w and -i w
__device__ __forceinline__ void bf_one(double2 &a, double2 &b)
{
    const double2 s = make_double2(a.x + b.x, a.y + b.y);
    b = make_double2(a.x - b.x, a.y - b.y);
    a = s;
}
__device__ __forceinline__ void bf_mi(double2 &a, double2 &b)
{
    const double2 s = make_double2(a.x + b.y, a.y - b.x);
    b = make_double2(a.x - b.y, a.y + b.x);
    a = s;
}
__device__ __forceinline__ void bf_w(double2 &a, double2 &b, double2 w)
{
    const double2 s = make_double2(fma(-w.y, b.y, fma(w.x, b.x, a.x)), fma(w.y, b.x, fma(w.x, b.y, a.y)));
    b = make_double2(fma(2.0, a.x, -s.x), fma(2.0, a.y, -s.y));
    a = s;
}
__device__ __forceinline__ void bf_miw(double2 &a, double2 &b, double2 w) { bf_w(a, b, make_double2(w.y, -w.x)); }

// R stages of the forward transform on the 2^R points of one block i of stage t, spaced by the
// last stage's span.  W[i] = exp(-i pi sum_j bit_j(i) 2^-(j+1)) is block i's twiddle at every
// stage that has it; W[2 i + 1] = -i W[2 i].  TOP: block 0 of stage 0 (twiddles 1 and -i free),
// HALF: its upper half is zero.
template <int R, bool TOP>
__device__ __forceinline__ void fwd_group(double2 (&x)[1 << R], const double2 *__restrict__ W, int i, bool half)
{
#pragma unroll
    for (int s = 0; s < R; ++s) {
        const int h = 1 << (R - 1 - s);
#pragma unroll
        for (int b = 0; b < (1 << s); ++b) {
            if (TOP && s == 0) {
#pragma unroll
                for (int j = 0; j < h; ++j) {
                    if (half) x[h + j] = x[j];
                    else bf_one(x[j], x[h + j]);
                }
                continue;
            }
            double2 w;
            if (!(TOP && b < 2)) w = __ldg(W + (i << s) + (b & ~1));
#pragma unroll
            for (int j = 0; j < h; ++j) {
                double2 &u = x[2 * b * h + j], &v = x[2 * b * h + h + j];
                if (TOP && b == 0) bf_one(u, v);
                else if (TOP && b == 1) bf_mi(u, v);
                else if (s > 0 && (b & 1)) bf_miw(u, v, w);
                else bf_w(u, v, w);
            }
        }
    }
}

// R stages of the inverse transform on 2^R points p + j h (h the first stage's span, p < h);
// T[k] = exp(-2 pi i k / L).  UNIT: h = 1, p = 0.
template <int R, int LOGL, bool UNIT>
__device__ __forceinline__ void inv_group(double2 (&x)[1 << R], const double2 *__restrict__ T, int p, int log2h)
{
#pragma unroll
    for (int s = 0; s < R; ++s) {
        const int q = 1 << s;   // span in units of h
#pragma unroll
        for (int j = 0; j < q; ++j) {
            const bool turn = s > 0 && j >= q / 2;             // exp(-i pi (j + q/2) / q) = -i exp(-i pi j / q)
            const int jj = turn ? j - q / 2 : j;
            double2 w;
            if (!(UNIT && jj == 0)) w = __ldg(T + ((p + (jj << log2h)) << (LOGL - 1 - s - log2h)));
#pragma unroll
            for (int g = 0; g < (1 << R); g += 2 * q) {
                double2 &u = x[g + j], &v = x[g + q + j];
                if (UNIT && jj == 0) {
                    if (turn) bf_mi(u, v); else bf_one(u, v);
                } else if (turn) bf_miw(u, v, w);
                else bf_w(u, v, w);
            }
        }
    }
}

// A pass of R stages over shared memory: forward stages t .. t + R - 1, or the inverse stages
// that undo them.  Spans run from L / 2^(t+1) down to H = L / 2^(t+R).
template <int LOGL, int t, int R>
__device__ __forceinline__ void fwd_pass(double2 *xs, const double2 *__restrict__ W)
{
    constexpr int L = 1 << LOGL, LH = LOGL - t - R, H = 1 << LH, NT = L / 16;
#pragma unroll 1
    for (int u = threadIdx.x; u < (L >> R); u += NT) {
        const int i = u >> LH, lo = u & (H - 1), base = (i << (LH + R)) + lo;
        double2 x[1 << R];
#pragma unroll
        for (int j = 0; j < (1 << R); ++j) x[j] = xs[place(base + (j << LH))];
        fwd_group<R, false>(x, W, i, false);
#pragma unroll
        for (int j = 0; j < (1 << R); ++j) xs[place(base + (j << LH))] = x[j];
    }
    __syncthreads();
}

template <int LOGL, int t, int R>
__device__ __forceinline__ void inv_pass(double2 *xs, const double2 *__restrict__ T)
{
    constexpr int L = 1 << LOGL, LH = LOGL - t - R, H = 1 << LH, NT = L / 16;
#pragma unroll 1
    for (int u = threadIdx.x; u < (L >> R); u += NT) {
        const int i = u >> LH, lo = u & (H - 1), base = (i << (LH + R)) + lo;
        double2 x[1 << R];
#pragma unroll
        for (int j = 0; j < (1 << R); ++j) x[j] = xs[place(base + (j << LH))];
        inv_group<R, LOGL, false>(x, T, lo, LH);
#pragma unroll
        for (int j = 0; j < (1 << R); ++j) xs[place(base + (j << LH))] = x[j];
    }
    __syncthreads();
}

struct CztTables {
    int64_t *ng;          // good trajectories
    double2 *W, *T;       // [L / 2] forward and inverse twiddles
    double2 *v, *V;       // [L] kernel chirp, and its transform (point 16 g + j at j L / 16 + g)
    double2 *chirp;       // [n_blk][K] input chirps
    double *part;         // [CTA][n_E]
};

// Twiddles, the kernel chirp v_m = exp(-i w m^2/2) at index m mod L (m in [-(K-1), nb - 1]),
// the input chirps chirp[b][c] = exp(i (E_b c dt + w c^2/2)), and (block 0) the good count.
__global__ void __launch_bounds__(256) k_czt_tables(CztTables tb, int log2L, int K, int n_blk, int nb, double E_min,
                                                    double dE, double dt, const uint8_t *__restrict__ good,
                                                    int64_t n_traj, int64_t *__restrict__ n_good_out)
{
    const int L = 1 << log2L;
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const double w = dE * dt;
    double s, co;
    if (idx < L / 2) {
        sincospi(-2.0 * idx / L, &s, &co);
        tb.T[idx] = make_double2(co, s);
        sincospi(-(double)__brev((unsigned)idx) * 0x1p-32, &s, &co);   // bit j of idx weighs 2^-(j+1)
        tb.W[idx] = make_double2(co, s);
    }
    if (idx < L) {
        const int m = idx < nb ? (int)idx : (int)idx - L;
        double2 v = make_double2(0.0, 0.0);
        if (m < nb && m > -K) {
            sincos(-0.5 * w * ((double)m * (double)m), &s, &co);
            v = make_double2(co, s);
        }
        tb.v[idx] = v;
    }
    if (idx < (int64_t)n_blk * K) {
        const int b = (int)(idx / K), c = (int)(idx % K);
        const double Eb = E_min + (double)b * nb * dE;
        // phase modulo 2 pi in FP64 (c^2 is exact); sincos keeps full accuracy for these arguments
        const double ph = Eb * (c * dt) + 0.5 * w * ((double)c * (double)c);
        sincos(ph, &s, &co);
        tb.chirp[idx] = make_double2(co, s);
    }
    if (blockIdx.x == 0) {
        __shared__ long long red[256];
        long long acc = 0;
#pragma unroll 8
        for (int64_t i = threadIdx.x; i < n_traj; i += 256) acc += good[i] ? 1 : 0;
        red[threadIdx.x] = acc;
        __syncthreads();
        for (int o = 128; o > 0; o >>= 1) {
            if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            tb.ng[0] = red[0];
            if (n_good_out) n_good_out[0] = red[0];
        }
    }
}

// V = FFT(v), one of kVParts blocks of the transform's fourth stage per CTA: the residue of
// v modulo z^(L/16) - rho (15 multiply-adds a point instead of the first four stages), then the
// remaining stages on L / 16 points.  One CTA for the whole transform took 190 us.  The powers of rho are
// each rounded once: Horner's rule multiplies rho's rounding by up to 15, and V, which every trajectory
// shares, came out 3 to 8 times less accurate than by the stages.
__global__ void __launch_bounds__(256) k_czt_kernel_fft(CztTables tb, int log2L)
{
    __shared__ double2 x[(1 << kLog2Max) / kVParts], rho[kVParts];
    const int L = 1 << log2L, n = L / kVParts, part = blockIdx.x;
    if (threadIdx.x < kVParts) {
        // rho = exp(-2 pi i r / 16), r the bits of part from the other end
        const int r = (int)(__brev((unsigned)part) >> 28) * (int)threadIdx.x % kVParts;
        double s, c;
        sincospi(-2.0 * r / kVParts, &s, &c);
        rho[threadIdx.x] = make_double2(c, s);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        double2 y = tb.v[k];
#pragma unroll
        for (int j = 1; j < kVParts; ++j) {
            const double2 u = tb.v[k + j * n], w = rho[j];
            y = make_double2(fma(-w.y, u.y, fma(w.x, u.x, y.x)), fma(w.y, u.x, fma(w.x, u.y, y.y)));
        }
        x[k] = y;
    }
    __syncthreads();
    for (int h = n / 2, blocks = 1; h >= 1; h >>= 1, blocks <<= 1) {
        for (int u = threadIdx.x; u < n / 2; u += blockDim.x) {
            const int i = u / h, a = 2 * h * i + u % h;
            bf_w(x[a], x[a + h], __ldg(tb.W + part * blocks + i));
        }
        __syncthreads();
    }
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int at = part * n + k;
        tb.V[(at & 15) * (L / 16) + (at >> 4)] = x[k];
    }
}

// Weighted |X|^2 of the CTA's good trajectories for every energy block; per-CTA sums.
template <int LOGL>
__global__ void __launch_bounds__((1 << LOGL) / 16, LOGL == 13 ? 1 : (LOGL == 12 ? 2 : 4))
    k_czt(const AmpRef amp, int64_t amp_ld, const double *__restrict__ w, const uint8_t *__restrict__ good,
          int64_t n_traj, int K, int n_E, int n_blk, int nb, CztTables tb)
{
    constexpr int L = 1 << LOGL, NT = L / 16, MID = LOGL - 7;   // middle stages between the first 3 and the last 4
    constexpr int R1 = (MID + 1) / 2, R2 = MID - R1;            // 13: 3 + 3, 12: 3 + 2, 11: 2 + 2, 10: 2 + 1
    extern __shared__ __align__(16) double2 xs[];
    double *Ip = reinterpret_cast<double *>(xs + L);   // [n_E]
    for (int k = threadIdx.x; k < n_E; k += NT) Ip[k] = 0.0;
    const double inv_L2 = 1.0 / ((double)L * (double)L);
    const double2 *__restrict__ W = tb.W, *__restrict__ T = tb.T, *__restrict__ V = tb.V;
    const bool half = K <= L / 2;
    for (int64_t j = blockIdx.x; j < n_traj; j += gridDim.x) {
        if (!good[j]) continue;                       // uniform over the CTA
        const AmpRef a = amp.offset(j * amp_ld);
        const double wj = w[j] * inv_L2;
        for (int b = 0; b < n_blk; ++b) {
            const double2 *ch = tb.chirp + (int64_t)b * K;
#pragma unroll 1
            for (int u = threadIdx.x; u < L / 8; u += NT) {
                double2 x[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int c = u + e * (L / 8);
                    x[e] = c < K ? cmul(a[c], __ldg(ch + c)) : make_double2(0.0, 0.0);
                }
                fwd_group<3, true>(x, W, 0, half);
#pragma unroll
                for (int e = 0; e < 8; ++e) xs[place(u + e * (L / 8))] = x[e];
            }
            __syncthreads();
            fwd_pass<LOGL, 3, R1>(xs, W);
            fwd_pass<LOGL, 3 + R1, R2>(xs, W);
            {
                double2 x[16];
                const int g = threadIdx.x;
#pragma unroll
                for (int e = 0; e < 16; ++e) x[e] = xs[place(16 * g + e)];
                fwd_group<4, false>(x, W, g, false);
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const double2 p = cmul(x[e], __ldg(V + e * NT + g));
                    x[e] = make_double2(p.x, -p.y);
                }
                inv_group<4, LOGL, true>(x, T, 0, 0);
#pragma unroll
                for (int e = 0; e < 16; ++e) xs[place(16 * g + e)] = x[e];
            }
            __syncthreads();
            inv_pass<LOGL, 3 + R1, R2>(xs, T);
            inv_pass<LOGL, 3, R1>(xs, T);
            const int k0 = b * nb, nk = min(nb, n_E - k0);
#pragma unroll 1
            for (int u = threadIdx.x; u < L / 8; u += NT) {
                if (u >= nk) break;
                double2 x[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] = xs[place(u + e * (L / 8))];
                inv_group<3, LOGL, false>(x, T, u, LOGL - 3);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int k = u + e * (L / 8);
                    if (k < nk) Ip[k0 + k] = fma(wj, fma(x[e].x, x[e].x, x[e].y * x[e].y), Ip[k0 + k]);
                }
            }
            __syncthreads();
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n_E; k += NT) tb.part[(int64_t)blockIdx.x * n_E + k] = Ip[k];
}

inline size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

struct CztLayout {
    int K, nb, n_blk, n_cta, log2L;
    size_t smem, off_W, off_T, off_v, off_V, off_chirp, off_part, total;
};

// The transform length: the cheapest of n_blk blocks of L (log2 L + 3) (butterflies, chirps and
// products) over L = 1024 .. 8192 with at least L / 8 energies a block; up to four CTAs per SM.
CztLayout czt_layout(int n_steps, int n_E, int n_sm)
{
    CztLayout Y{};
    Y.K = n_steps + 1;
    int64_t best = -1;
    for (int lg = kLog2Min; lg <= kLog2Max; ++lg) {
        const int L = 1 << lg, nb = L - Y.K + 1;
        if (nb < L / 8) continue;
        const int n_blk = (n_E + nb - 1) / nb;
        const int64_t cost = (int64_t)n_blk * L * (lg + 3);
        if (best < 0 || cost < best) {
            best = cost;
            Y.log2L = lg;
            Y.nb = nb;
            Y.n_blk = n_blk;
        }
    }
    const int L = 1 << Y.log2L;
    Y.smem = sizeof(double2) * (size_t)L + sizeof(double) * (size_t)n_E;
    int per_sm = (int)(227 * 1024 / (Y.smem + 1024));
    const int most = Y.log2L == 13 ? 1 : (Y.log2L == 12 ? 2 : 4);
    per_sm = per_sm < 1 ? 1 : (per_sm > most ? most : per_sm);
    Y.n_cta = n_sm * per_sm;
    Y.off_W = a256(sizeof(int64_t));
    Y.off_T = Y.off_W + a256(sizeof(double2) * L / 2);
    Y.off_v = Y.off_T + a256(sizeof(double2) * L / 2);
    Y.off_V = Y.off_v + a256(sizeof(double2) * L);
    Y.off_chirp = Y.off_V + a256(sizeof(double2) * L);
    Y.off_part = Y.off_chirp + a256(sizeof(double2) * (size_t)Y.n_blk * Y.K);
    Y.total = Y.off_part + a256(sizeof(double) * (size_t)Y.n_cta * n_E);
    return Y;
}

int sm_count()
{
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 1;
    return n > 0 ? n : 1;
}

template <int LOGL>
cudaError_t launch_czt(const CztLayout &Y, AmpRef amp, int64_t amp_ld, const double *w, const uint8_t *good,
                       int64_t n_traj, int n_E, const CztTables &tb, cudaStream_t s)
{
    // the largest size any grid needs: the limit is the kernel's, shared by all host threads, and one
    // set to this call's size could be lowered by another thread before the launch
    constexpr size_t most = sizeof(double2) * ((size_t)1 << LOGL) + sizeof(double) * kCztMaxEnergies;
    static_assert(most <= 227 * 1024, "the vector and the sums fit an SM's shared memory");
    const cudaError_t e = cudaFuncSetAttribute(k_czt<LOGL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (e != cudaSuccess) return e;
    k_czt<LOGL><<<Y.n_cta, (1 << LOGL) / 16, Y.smem, s>>>(amp, amp_ld, w, good, n_traj, Y.K, n_E, Y.n_blk, Y.nb, tb);
    return cudaGetLastError();
}

}  // namespace

// Largest K = n_steps + 1 the chirp-z mode takes: an energy block of the longest transform
// holds at least 1024 energies (L - K + 1 >= 1024).
int spectrum_czt_max_samples() { return (1 << kLog2Max) - 1023; }

size_t spectrum_czt_scratch_bytes(int64_t n_traj, int n_steps, int n_E)
{
    (void)n_traj;
    return czt_layout(n_steps, n_E, sm_count()).total;
}

cudaError_t launch_spectrum_czt(AmpRef amp, int64_t amp_ld, const double *w, const uint8_t *good,
                                int64_t n_traj, int n_steps, double dt, double E_min, double E_max, int n_E,
                                double *I_out, int64_t *n_good_out, void *scratch, cudaStream_t s, int *n_launch)
{
    *n_launch = 0;
    if (n_steps + 1 > spectrum_czt_max_samples()) return cudaErrorInvalidValue;
    const CztLayout Y = czt_layout(n_steps, n_E, sm_count());
    char *base = static_cast<char *>(scratch);
    auto at = [&](size_t off) { return reinterpret_cast<double2 *>(base + off); };
    const CztTables tb{reinterpret_cast<int64_t *>(base), at(Y.off_W), at(Y.off_T), at(Y.off_v), at(Y.off_V),
                       at(Y.off_chirp), reinterpret_cast<double *>(base + Y.off_part)};
    const double dE = (E_max - E_min) / (n_E - 1);
    const double scale = dt * dt / (kTwoPi * (n_steps * dt));
    const int64_t L = 1 << Y.log2L, nch = (int64_t)Y.n_blk * Y.K;
    const int64_t items = L > nch ? L : nch;
    cudaError_t e;
    k_czt_tables<<<(unsigned)((items + 255) / 256), 256, 0, s>>>(tb, Y.log2L, Y.K, Y.n_blk, Y.nb, E_min, dE, dt, good,
                                                                 n_traj, n_good_out);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_czt_kernel_fft<<<kVParts, 256, 0, s>>>(tb, Y.log2L);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    switch (Y.log2L) {
    case 10: e = launch_czt<10>(Y, amp, amp_ld, w, good, n_traj, n_E, tb, s); break;
    case 11: e = launch_czt<11>(Y, amp, amp_ld, w, good, n_traj, n_E, tb, s); break;
    case 12: e = launch_czt<12>(Y, amp, amp_ld, w, good, n_traj, n_E, tb, s); break;
    default: e = launch_czt<13>(Y, amp, amp_ld, w, good, n_traj, n_E, tb, s); break;
    }
    if (e != cudaSuccess) return e;
    *n_launch = 4;
    return launch_reduce_rows(tb.part, Y.n_cta, n_E, tb.ng, scale, I_out, s);
}

}  // namespace scivr
