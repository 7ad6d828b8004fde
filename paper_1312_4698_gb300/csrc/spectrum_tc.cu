// Time -> energy Fourier step (Eq. I(E)_discreto of arXiv:1312.4698) on the
// 5th-generation tensor cores (tcgen05, sm_103a).
//
// The complex contraction X = a . tw (n_traj x K times K x n_E) is written
// as one real GEMM  [Re a | Im a] . [[cos, sin], [-sin, cos]]  with
// M = n_traj, N = 2 n_E (each 256-column tile holds the real parts of 128
// energies followed by their imaginary parts), K' = 2K.  Each FP64/FP32
// operand is split into ND BF16 digits (x ~ d0 + d1 + d2, d_i = bf16 of the
// remainder) and the digit products with d_a + d_b < ND are accumulated in
// one FP32 TMEM accumulator: ND = 1 is plain BF16, ND = 2 keeps ~16 bits
// (3 products), ND = 3 keeps FP32-level accuracy (6 products).
//
// Operands are pre-tiled in HBM in the tensor core's canonical K-major
// no-swizzle layout (8-row x 16-byte core matrices), so each pipeline stage
// is one contiguous bulk copy (cp.async.bulk) per operand.  One CTA per
// 128 x 256 output tile: warp 0 lane 0 issues the copies, warp 1 lane 0
// issues tcgen05.mma from one elected thread, and all four warps read the
// accumulator back with tcgen05.ld and reduce w_j |X_jk|^2 over the tile's
// rows.  Every mbarrier wait is bounded; an expired wait records
// SCIVR_ETIMEOUT in a device status word and the CTA winds down.
#include <cuda_bf16.h>

#include <cstdint>

#include "spectrum_reduce.cuh"
#include "tc_common.cuh"

namespace scivr {
namespace tc {

template <int ND>
__device__ __forceinline__ void split_digits(float x, __nv_bfloat16 (&d)[ND])
{
    float r = x;
#pragma unroll
    for (int i = 0; i < ND; ++i) {
        d[i] = __float2bfloat16_rn(r);
        r -= __bfloat162float(d[i]);
    }
}

// ---- operand tiles.  A' row: [Re a(0..K-1), Im a(0..K-1), 0 ...]; rows of bad or missing
// trajectories are zero.  B' rows of tile nt: rows 0..127 are Re rows of energies nt*128 + i,
// [cos(E c dt), -sin(E c dt)], rows 128..255 Im rows, [sin(E c dt), cos(E c dt)].
//
// A block of either operand takes 8 rows (trajectories, energies: one 8-row group of core
// matrices) and C samples, plus SP_HALO before them, as (re, im) pairs in shared memory, and
// writes all places they have: an amplitude is read from HBM once (a thread per output chunk read
// every row twice, half of each sector at a time), a twiddle's phase -- five FP64 instructions on
// a pipe that takes 64 cycles for each -- is formed once instead of four times.  The halo lets a
// block own whole 16-byte chunks of the second half, whose samples start K mod 8 off a chunk
// boundary.  16384 trajectories x 5001 samples, 4000 energies, two digits: amplitudes 288 ->
// 243 us, twiddles 1066 -> 228 us.  C = 248, but 56 for the amplitudes of up to 224 samples, whose blocks
// of 256 threads had few of them at work or a second block that was nearly empty: the whole step for
// 65536 trajectories and 100 energies, 248 / 56: 50 samples 158 / 107 us, 113 172 / 148, 168 159 / 143,
// 224 166 / 164, 248 174 / 183.
constexpr int SP_ROWS = 8, SP_C = 248, SP_FEW = 56, SP_HALO = 8;
static_assert(SP_C % 8 == 0 && SP_FEW % 8 == 0, "whole chunks");

template <int C>
struct SplitTile {
    static constexpr int W = C + SP_HALO;   // samples, and threads of a block
    float2 v[SP_ROWS][W + 1];               // odd row length: the 8 rows of a chunk in different banks
};

template <int ND>
__device__ __forceinline__ void put_chunk(uint8_t *dst, int64_t digit_stride, const float (&v)[8])
{
    __nv_bfloat16 dg[ND][8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        __nv_bfloat16 d[ND];
        split_digits<ND>(v[i], d);
#pragma unroll
        for (int q = 0; q < ND; ++q) dg[q][i] = d[q];
    }
#pragma unroll
    for (int q = 0; q < ND; ++q) *reinterpret_cast<uint4 *>(dst + q * digit_stride) = *reinterpret_cast<const uint4 *>(&dg[q][0]);
}

// The output chunks (8 columns kp) of sample block cb: of the first half (kp = c) and of the second
// (kp = K + c); the last block also has the zero columns past 2 K and the chunk that holds the end
// of one half and the start of the other.  put(row, kp0, x, second): the 8 samples of one chunk;
// edge(row, c): sample c from memory, for that last chunk.
template <int C, typename Put, typename Edge>
__device__ __forceinline__ void split_chunks(const SplitTile<C> &t, int cb, int n_c, int K, int n_kt, Put &&put, Edge &&edge)
{
    const bool last = cb == n_c - 1;
    const int c0 = cb * C;                                         // first owned sample
    const int lo1 = c0, hi1 = min(c0 + C, K / 8 * 8);              // whole chunks of the first half
    const int up = (K + 7) / 8 * 8;                                   // first whole chunk of the second
    const int lo2 = max(up, (K + c0) / 8 * 8), hi2 = last ? n_kt * BK : (K + c0 + C) / 8 * 8;
    const int n1 = hi1 > lo1 ? (hi1 - lo1) / 8 : 0, n2 = hi2 > lo2 ? (hi2 - lo2) / 8 : 0;
    const int n3 = last && K % 8 ? 1 : 0;
    for (int i = threadIdx.x; i < (n1 + n2 + n3) * SP_ROWS; i += SplitTile<C>::W) {
        const int row = i % SP_ROWS, ch = i / SP_ROWS;
        float2 x[8];
        if (ch < n1 + n2) {
            const bool second = ch >= n1;
            const int kp0 = second ? lo2 + 8 * (ch - n1) : lo1 + 8 * ch;
            const int at = kp0 - (second ? K : 0) - c0 + SP_HALO;
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = at + u < SplitTile<C>::W ? t.v[row][at + u] : make_float2(0.0f, 0.0f);
            put(row, kp0, x, second ? 0 : 8);
        } else {
            const int kp0 = K / 8 * 8, first = K - kp0;   // first columns of the chunk are of the first half
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int c = u < first ? kp0 + u : u - first;
                x[u] = c < K ? edge(row, c) : make_float2(0.0f, 0.0f);
            }
            put(row, kp0, x, first);
        }
    }
}

template <int ND, int C>
__global__ void __launch_bounds__(SplitTile<C>::W)
    k_split_amp(const AmpRef amp, int64_t amp_ld, const uint8_t *__restrict__ good, int64_t n_traj, int K, int n_kt,
                int n_c, uint8_t *__restrict__ At)
{
    __shared__ SplitTile<C> t;
    const int cb = (int)(blockIdx.x % n_c);
    const int64_t row0 = (int64_t)(blockIdx.x / n_c) * SP_ROWS;
    const int ci = threadIdx.x, c = cb * C - SP_HALO + ci;
    // a thread's eight loads go out together: bad rows are read too, their flags only select
    float2 v[SP_ROWS];
    bool ok[SP_ROWS];
#pragma unroll
    for (int el = 0; el < SP_ROWS; ++el) {
        const int64_t r = row0 + el;
        const bool in = c >= 0 && c < K && r < n_traj;
        v[el] = in ? amp.f(r * amp_ld + c) : make_float2(0.0f, 0.0f);
        ok[el] = in && good[r];
    }
#pragma unroll
    for (int el = 0; el < SP_ROWS; ++el) t.v[el][ci] = ok[el] ? v[el] : make_float2(0.0f, 0.0f);
    __syncthreads();
    uint8_t *tile = At + (row0 / BM) * n_kt * (int64_t)(ND * TILE_A);
    split_chunks(
        t, cb, n_c, K, n_kt,
        [&](int row, int kp0, const float2 (&x)[8], int first) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = u < first ? x[u].x : x[u].y;
            put_chunk<ND>(tile + (kp0 / BK) * (int64_t)(ND * TILE_A) + canon_off((int)(row0 % BM) + row, kp0 % BK), TILE_A, v);
        },
        [&](int row, int cc) {
            const int64_t r = row0 + row;
            return r < n_traj && good[r] ? amp.f(r * amp_ld + cc) : make_float2(0.0f, 0.0f);
        });
}

__device__ __forceinline__ float2 twiddle(double E, double cdt)   // (cos, sin) of E c dt
{
    const double turns = E * cdt * kInvTwoPi;
    const float fr = (float)(turns - rint(turns));
    float2 r;
    sincospif(2.0f * fr, &r.y, &r.x);
    return r;
}

template <int ND>
__global__ void __launch_bounds__(SplitTile<SP_C>::W)
    k_split_tw(int K, int n_kt, int n_E, int n_c, double E_min, double dE, double dt, uint8_t *__restrict__ Bt)
{
    __shared__ SplitTile<SP_C> t;
    __shared__ double Es[SP_ROWS];
    const int cb = blockIdx.x % n_c, e0 = blockIdx.x / n_c * SP_ROWS;
    if (threadIdx.x < SP_ROWS) Es[threadIdx.x] = E_min + (e0 + (int)threadIdx.x) * dE;
    __syncthreads();
    const int ci = threadIdx.x, c = cb * SP_C - SP_HALO + ci;
    const double cdt = c * dt;
#pragma unroll 4
    for (int el = 0; el < SP_ROWS; ++el)
        t.v[el][ci] = e0 + el < n_E && c >= 0 && c < K ? twiddle(Es[el], cdt) : make_float2(0.0f, 0.0f);
    __syncthreads();
    uint8_t *tile = Bt + (e0 / EPT) * n_kt * (int64_t)(ND * TILE_B);
    split_chunks(
        t, cb, n_c, K, n_kt,
        [&](int row, int kp0, const float2 (&x)[8], int first) {
            float re[8], im[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                re[u] = u < first ? x[u].x : -x[u].y;
                im[u] = u < first ? x[u].y : x[u].x;
            }
            uint8_t *dst = tile + (kp0 / BK) * (int64_t)(ND * TILE_B);
            put_chunk<ND>(dst + canon_off(e0 % EPT + row, kp0 % BK), TILE_B, re);
            put_chunk<ND>(dst + canon_off(EPT + e0 % EPT + row, kp0 % BK), TILE_B, im);
        },
        [&](int row, int cc) { return e0 + row < n_E ? twiddle(Es[row], cc * dt) : make_float2(0.0f, 0.0f); });
}

template <int ND>
__global__ void __launch_bounds__(128, 1)
    k_ft_tc(const uint8_t *__restrict__ At, const uint8_t *__restrict__ Bt, const double *__restrict__ w,
            const uint8_t *__restrict__ good, int64_t n_traj, int n_kt, int n_E, double *__restrict__ part)
{
    using CF = Cfg<ND>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t full_bar[CF::STAGES], empty_bar[CF::STAGES], done_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nt = blockIdx.x;
    const int64_t mt = blockIdx.y;

    if (threadIdx.x == 0) {
        for (int s = 0; s < CF::STAGES; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(&done_bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_slot)),
                     "r"(256)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    const uint8_t *Ablk = At + (size_t)mt * n_kt * CF::A_BYTES;
    const uint8_t *Bblk = Bt + (size_t)nt * n_kt * CF::B_BYTES;

    if (warp == 0 && lane == 0) {
        // producer: one bulk copy per operand per stage
        int issued = 0;
        for (int kt = 0; kt < n_kt; ++kt) {
            const int s = kt % CF::STAGES, use = kt / CF::STAGES;
            if (use > 0 && !mbar_wait(&empty_bar[s], (use - 1) & 1, kWaitLimitCycles)) {
                atomicExch(&abort_flag, 1);
                break;
            }
            if (*(volatile int *)&abort_flag) break;
            uint8_t *sa = smem + s * CF::STAGE;
            uint8_t *sb = sa + CF::A_BYTES;
            mbar_expect_tx(&full_bar[s], CF::A_BYTES + CF::B_BYTES);
            bulk_g2s(sa, Ablk + (size_t)kt * CF::A_BYTES, CF::A_BYTES, &full_bar[s]);
            bulk_g2s(sb, Bblk + (size_t)kt * CF::B_BYTES, CF::B_BYTES, &full_bar[s]);
            issued = kt + 1;
        }
        // never leave with copies in flight: wait (bounded) for the last use of each stage
        for (int kt = issued - CF::STAGES > 0 ? issued - CF::STAGES : 0; kt < issued; ++kt)
            mbar_wait(&full_bar[kt % CF::STAGES], (kt / CF::STAGES) & 1, kWaitLimitCycles);
    } else if (warp == 1 && lane == 0) {
        // MMA issuer
        constexpr uint32_t idesc = idesc_bf16(BM, BN);
        constexpr int pa[6] = {0, 0, 1, 0, 1, 2};
        constexpr int pb[6] = {0, 1, 0, 2, 1, 0};
        bool ok = true;
        for (int kt = 0; kt < n_kt && ok; ++kt) {
            const int s = kt % CF::STAGES;
            if (!mbar_wait(&full_bar[s], (kt / CF::STAGES) & 1, kWaitLimitCycles) || *(volatile int *)&abort_flag) {
                atomicExch(&abort_flag, 1);
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t sa = su32(smem + s * CF::STAGE);
            const uint32_t sb = sa + CF::A_BYTES;
#pragma unroll
            for (int ks = 0; ks < BK / 16; ++ks) {
#pragma unroll
                for (int p = 0; p < CF::NPAIR; ++p) {
                    const uint64_t ad = sdesc(sa + pa[p] * TILE_A + ks * 2 * LBO);
                    const uint64_t bd = sdesc(sb + pb[p] * TILE_B + ks * 2 * LBO);
                    umma(tmem, ad, bd, idesc, (kt | ks | p) != 0);
                }
            }
            umma_commit(&empty_bar[s]);
        }
        umma_commit(&done_bar);
    }
    __syncwarp();
    // epilogue: all 128 threads, row = 32 * warp + lane
    const bool done_ok = mbar_wait(&done_bar, 0, kWaitLimitCycles) && !*(volatile int *)&abort_flag;
    tc_fence_after();
    __syncwarp();
    float *stg = reinterpret_cast<float *>(smem);   // [BM][EPT + 1], reuses the stage buffers
    const int row = warp * 32 + lane;
    const int64_t grow = mt * BM + row;
    const bool ok = done_ok && grow < n_traj && good[grow];
    const float wr = ok ? (float)w[grow] : 0.0f;
#pragma unroll 1
    for (int ch = 0; ch < EPT / 32; ++ch) {
        float re[32], im[32];
        const uint32_t base = tmem + ((uint32_t)(warp * 32) << 16);
        tmem_ld32(base + ch * 32, re);
        tmem_ld32(base + EPT + ch * 32, im);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const float m2 = fmaf(re[i], re[i], im[i] * im[i]);
            stg[row * (EPT + 1) + ch * 32 + i] = ok ? wr * m2 : 0.0f;
        }
    }
    tc_fence_before();
    __syncthreads();
    {
        const int e = nt * EPT + threadIdx.x;
        double s = 0.0;
#pragma unroll 8
        for (int r = 0; r < BM; ++r) s += (double)stg[r * (EPT + 1) + threadIdx.x];
        if (e < n_E) part[mt * n_E + e] = s;
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256) : "memory");
    }
}

__global__ void k_tc_count_good(const uint8_t *__restrict__ good, int64_t n, int64_t *__restrict__ out,
                                int64_t *__restrict__ out2)
{
    __shared__ long long red[1024];
    long long acc = 0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) acc += good[i] ? 1 : 0;
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = red[0];
        if (out2) out2[0] = red[0];
    }
}

// Waits on an mbarrier that nothing completes, with a short limit: the
// bounded-wait path must set SCIVR_ETIMEOUT and return.
__global__ void k_wait_selftest(long long limit)
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_wait(&bar, 0, limit);
}

inline size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

struct TcLayout {
    int K, n_kt, n_nt;
    int64_t n_mt, rows_pad;
    size_t off_ng, off_part, off_A, off_B, total;
};

inline TcLayout tc_layout(int nd, int64_t n_traj, int n_steps, int n_E)
{
    TcLayout L{};
    L.K = n_steps + 1;
    L.n_kt = (2 * L.K + BK - 1) / BK;
    L.n_mt = (n_traj + BM - 1) / BM;
    L.rows_pad = L.n_mt * BM;
    L.n_nt = (n_E + EPT - 1) / EPT;
    L.off_ng = 0;
    L.off_part = a256(sizeof(int64_t));
    L.off_A = L.off_part + a256(sizeof(double) * (size_t)L.n_mt * n_E);
    L.off_B = L.off_A + a256((size_t)L.n_mt * L.n_kt * nd * TILE_A);
    L.total = L.off_B + a256((size_t)L.n_nt * L.n_kt * nd * TILE_B);
    return L;
}

template <int ND>
cudaError_t run(AmpRef amp, int64_t amp_ld, const double *w, const uint8_t *good, int64_t n_traj,
                int n_steps, double dt, double E_min, double E_max, int n_E, double *I_out,
                int64_t *n_good_out, void *scratch, cudaStream_t s, int *n_launch)
{
    using CF = Cfg<ND>;
    const TcLayout L = tc_layout(ND, n_traj, n_steps, n_E);
    uint8_t *base = static_cast<uint8_t *>(scratch);
    int64_t *ng = reinterpret_cast<int64_t *>(base + L.off_ng);
    double *part = reinterpret_cast<double *>(base + L.off_part);
    uint8_t *At = base + L.off_A;
    uint8_t *Bt = base + L.off_B;
    const double dE = (E_max - E_min) / (n_E - 1);
    const double scale = dt * dt / (kTwoPi * (n_steps * dt));
    cudaError_t e;
    *n_launch = 0;
    k_tc_count_good<<<1, 1024, 0, s>>>(good, n_traj, ng, n_good_out);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int n_c = (L.K + SP_C - 1) / SP_C;
    const int64_t row_groups = L.rows_pad / SP_ROWS;
    if (L.K <= 4 * SP_FEW) {
        const int n_f = (L.K + SP_FEW - 1) / SP_FEW;
        k_split_amp<ND, SP_FEW><<<(unsigned)(row_groups * n_f), SplitTile<SP_FEW>::W, 0, s>>>(amp, amp_ld, good, n_traj, L.K,
                                                                                             L.n_kt, n_f, At);
    } else {
        k_split_amp<ND, SP_C><<<(unsigned)(row_groups * n_c), SplitTile<SP_C>::W, 0, s>>>(amp, amp_ld, good, n_traj, L.K,
                                                                                         L.n_kt, n_c, At);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_split_tw<ND><<<(unsigned)(L.n_nt * (EPT / SP_ROWS) * n_c), SplitTile<SP_C>::W, 0, s>>>(L.K, L.n_kt, n_E, n_c, E_min, dE, dt,
                                                                                    Bt);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_ft_tc<ND>, cudaFuncAttributeMaxDynamicSharedMemorySize, CF::SMEM);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)L.n_nt, (unsigned)L.n_mt);
    k_ft_tc<ND><<<grid, 128, CF::SMEM, s>>>(At, Bt, w, good, n_traj, L.n_kt, n_E, part);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    *n_launch = 5;
    return launch_reduce_rows(part, (int)L.n_mt, n_E, ng, scale, I_out, s);
}

}  // namespace tc

int ft_tc_digits(int ft_mode)
{
    switch (ft_mode) {
    case SCIVR_FT_TC_BF16: return 1;
    case SCIVR_FT_TC_BF16X3: return 2;
    case SCIVR_FT_TC_BF16X6: return 3;
    default: return 0;
    }
}

size_t spectrum_tc_scratch_bytes(int ft_mode, int64_t n_traj, int n_steps, int n_E)
{
    return tc::tc_layout(ft_tc_digits(ft_mode), n_traj, n_steps, n_E).total;
}

cudaError_t launch_spectrum_tc(int ft_mode, AmpRef amp, int64_t amp_ld, const double *w,
                               const uint8_t *good, int64_t n_traj, int n_steps, double dt, double E_min,
                               double E_max, int n_E, double *I_out, int64_t *n_good_out, void *scratch,
                               cudaStream_t s, int *n_launch)
{
    switch (ft_tc_digits(ft_mode)) {
    case 1: return tc::run<1>(amp, amp_ld, w, good, n_traj, n_steps, dt, E_min, E_max, n_E, I_out, n_good_out, scratch, s, n_launch);
    case 2: return tc::run<2>(amp, amp_ld, w, good, n_traj, n_steps, dt, E_min, E_max, n_E, I_out, n_good_out, scratch, s, n_launch);
    case 3: return tc::run<3>(amp, amp_ld, w, good, n_traj, n_steps, dt, E_min, E_max, n_E, I_out, n_good_out, scratch, s, n_launch);
    default: *n_launch = 0; return cudaErrorInvalidValue;
    }
}

cudaError_t launch_wait_selftest(double seconds, cudaStream_t s)
{
    const long long limit = (long long)(seconds * 2.0e9);   // SM clock cycles at about 2 GHz
    tc::k_wait_selftest<<<1, 32, 0, s>>>(limit);
    return cudaGetLastError();
}

cudaError_t read_and_clear_status(int *status)
{
    int zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(status, g_device_status, sizeof(int));
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbol(g_device_status, &zero, sizeof(int));
}

}  // namespace scivr
