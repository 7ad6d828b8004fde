// Time -> energy Fourier step of the time-averaged spectrum, Eq. I(E)_discreto
// of arXiv:1312.4698, as a direct FP64 sum with a fused epilogue:
//
//   X[j][k] = sum_c amp[j][c] exp(i E_k c dt)
//   part[m][k] = sum_{j in row tile m, good} w_j |X[j][k]|^2
//   I[k] = dt^2 / (2 pi T n_good) sum_m part[m][k]     (fixed order, deterministic)
//
// The samples are cut into blocks of 2 B + 1 around centres c_b, and the two samples at
// distance m from the centre meet before the energies come in:
//
//   X = sum_b e^{i E c_b dt} [ a_{c_b} + sum_{m=1..B} cos(E m dt) u_m + sin(E m dt) v_m ],
//   u_m = a_{c_b + m} + a_{c_b - m},   v_m = i (a_{c_b + m} - a_{c_b - m}),
//
// four multiply-adds per pair of samples and energy instead of eight (and four per block),
// with B + n_blocks instead of K sines and cosines per energy.
//
// X is never written to memory.  The paper's design writes a private
// n_traj x k buffer per trajectory and reduces its columns in a second
// kernel (Sec. III.B); here the per-column weighted reduction happens in the
// epilogue and only one partial row per row tile reaches global memory.
#include "fp64_ops.cuh"
#include "scivr_internal.cuh"
#include "spectrum_reduce.cuh"

namespace scivr {
namespace {

constexpr int B = 16, BLOCK = 2 * B + 1;         // samples on each side of a block's centre
constexpr int WARPS = 4, COLS = 32;              // a CTA: 32 energies (a lane's own), four warps of rows
constexpr int kMaxGridY = 65535;                 // energy tiles beyond it go to the grid's z

__global__ void k_count_good(const uint8_t *__restrict__ good, int64_t n, int64_t *__restrict__ out,
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

// tab[m - 1][k] = (cos, sin)(E_k m dt), m = 1..B, then rot[b][k] = (cos, sin)(E_k c_b dt).  33 samples share a
// rotation and all blocks the table, so the phases' rounding, which would not average out, is put back
// (unit_phase): without that, spectra were up to 3.3 times less accurate than with a phase for every sample.
__global__ void k_twiddles(double2 *__restrict__ tab, int n_blocks, int n_E, double E_min, double dE, double dt)
{
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (idx >= (int64_t)(B + n_blocks) * n_E) return;
    const int r = (int)(idx / n_E), k = (int)(idx % n_E);
    const int c = r < B ? r + 1 : (r - B) * BLOCK + B;
    const double E = E_min + k * dE;
    tab[idx] = unit_phase(E, c, dt);
}

// X of WARPS * RPT rows x 32 energies.  What bounds it: the FP64 pipe, whose instructions take 64
// to 76 cycles of a sub-partition each; beside them the shared-memory reads (one table pair per
// RPT rows, two broadcasts per row) and the loads of the next block's samples, which are in
// flight while this block's are summed, cost nothing, so that a small tile runs as fast as a large
// one: RPT = 8 rows per lane where the tiles fill the chip several times over, 2 where they would
// leave SMs idle (fp64_rows).  The whole step,
// 96 x 401 samples x 300 energies (10 CTAs before): 1728 -> 120 us; 1024 x 3001 x 2000: 48.3 ->
// 23.4 ms (the two-samples-at-once form; 92 % of the FP64 pipe).
template <int RPT>
__global__ void __launch_bounds__(32 * WARPS) k_ft_fp64(const AmpRef amp, int64_t amp_ld,
                                                        const double2 *__restrict__ tab, const double *__restrict__ w,
                                                        const uint8_t *__restrict__ good, int64_t n_traj, int K,
                                                        int n_blocks, int n_E, double *__restrict__ part)
{
    constexpr int ROWS = WARPS * RPT, NT = 32 * WARPS;
    constexpr int ITEMS = ROWS * (B + 1), NI = (ITEMS + NT - 1) / NT;   // (row, m) pairs of a block; per thread
    __shared__ double2 tcs[B][COLS];
    __shared__ double2 su[ROWS][B + 1], sv[ROWS][B + 1];                // u_m, v_m; u_0 = the centre
    __shared__ double red[WARPS][COLS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t row0 = (int64_t)blockIdx.x * ROWS;
    const int tile = blockIdx.z * kMaxGridY + blockIdx.y;   // of energies
    if ((int64_t)tile * COLS >= n_E) return;
    const int col = tile * COLS + lane;
    const bool on = col < n_E;
    const int colc = on ? col : n_E - 1;

    for (int m = warp; m < B; m += WARPS) tcs[m][lane] = tab[(int64_t)m * n_E + colc];
    const double2 *rot = tab + (int64_t)B * n_E + colc;

    double2 hi[NI], lo[NI], rb;   // the next block's samples and rotation
    auto fetch = [&](int b) {
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int it = threadIdx.x + i * NT, r = it / (B + 1), m = it % (B + 1);
            const int cp = b * BLOCK + B + m, cm = cp - 2 * m;
            const bool row = it < ITEMS && row0 + r < n_traj;
            hi[i] = lo[i] = make_double2(0.0, 0.0);
            if (row && cp < K) hi[i] = amp[(row0 + r) * amp_ld + cp];
            if (row && m > 0 && cm < K) lo[i] = amp[(row0 + r) * amp_ld + cm];
        }
        rb = rot[(int64_t)b * n_E];
    };
    double2 X[RPT];
#pragma unroll
    for (int r = 0; r < RPT; ++r) X[r] = make_double2(0.0, 0.0);
    fetch(0);
    for (int b = 0; b < n_blocks; ++b) {
        __syncthreads();   // the previous block's readers are done
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int it = threadIdx.x + i * NT, r = it / (B + 1), m = it % (B + 1);
            if (it < ITEMS) {
                su[r][m] = make_double2(hi[i].x + lo[i].x, hi[i].y + lo[i].y);
                sv[r][m] = make_double2(lo[i].y - hi[i].y, hi[i].x - lo[i].x);
            }
        }
        const double2 rot_b = rb;
        __syncthreads();
        if (b + 1 < n_blocks) fetch(b + 1);
        double2 acc[RPT];
#pragma unroll
        for (int r = 0; r < RPT; ++r) acc[r] = su[warp * RPT + r][0];
#pragma unroll 4
        for (int m = 1; m <= B; ++m) {
            const double2 t = tcs[m - 1][lane];
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                const double2 u = su[warp * RPT + r][m], v = sv[warp * RPT + r][m];
                acc[r].x = fma(t.x, u.x, acc[r].x);
                acc[r].y = fma(t.x, u.y, acc[r].y);
                acc[r].x = fma(t.y, v.x, acc[r].x);
                acc[r].y = fma(t.y, v.y, acc[r].y);
            }
        }
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            X[r].x = fma(rot_b.x, acc[r].x, fma(-rot_b.y, acc[r].y, X[r].x));
            X[r].y = fma(rot_b.x, acc[r].y, fma(rot_b.y, acc[r].x, X[r].y));
        }
    }
    // epilogue: weighted |X|^2 summed over the tile's good rows
    double sum = 0.0;
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        const int64_t row = row0 + warp * RPT + r;
        if (row < n_traj && good[row]) sum += w[row] * fma(X[r].x, X[r].x, X[r].y * X[r].y);
    }
    red[warp][lane] = sum;
    __syncthreads();
    if (warp == 0 && on) {
        double s = red[0][lane];
#pragma unroll
        for (int t = 1; t < WARPS; ++t) s += red[t][lane];
        part[(int64_t)blockIdx.x * n_E + col] = s;
    }
}

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Rows per lane: 8 once such tiles fill the 152 SMs four times over, else 2 (tiles a quarter the
// size; with 8, 608 tiles of 32 x 32 are where an uneven last round costs at most a fifth).
int fp64_rows(int64_t n_traj, int n_E)
{
    const int64_t tiles = ((n_traj + 8 * WARPS - 1) / (8 * WARPS)) * (((int64_t)n_E + COLS - 1) / COLS);
    return tiles >= 4 * 152 ? 8 : 2;
}

int64_t row_tiles(int64_t n_traj, int n_E)
{
    const int rows = WARPS * fp64_rows(n_traj, n_E);
    return (n_traj + rows - 1) / rows;
}

int sample_blocks(int n_steps) { return (n_steps + BLOCK) / BLOCK; }   // of n_steps + 1 samples

}  // namespace

size_t spectrum_fp64_scratch_bytes(int64_t n_traj, int n_steps, int n_E)
{
    return align256(sizeof(int64_t)) + align256(sizeof(double2) * (size_t)(B + sample_blocks(n_steps)) * n_E) +
           align256(sizeof(double) * row_tiles(n_traj, n_E) * n_E);
}

cudaError_t launch_spectrum_fp64(AmpRef amp, int64_t amp_ld, const double *w,
                                 const uint8_t *good, int64_t n_traj, int n_steps, double dt,
                                 double E_min, double E_max, int n_E, double *I_out,
                                 int64_t *n_good_out, void *scratch, cudaStream_t s, int *n_launch)
{
    const int K = n_steps + 1, n_blocks = sample_blocks(n_steps);
    const int64_t n_mt = row_tiles(n_traj, n_E), n_tab = (int64_t)(B + n_blocks) * n_E;
    char *base = static_cast<char *>(scratch);
    int64_t *ng = reinterpret_cast<int64_t *>(base);
    double2 *tab = reinterpret_cast<double2 *>(base + align256(sizeof(int64_t)));
    double *part = reinterpret_cast<double *>(base + align256(sizeof(int64_t)) + align256(sizeof(double2) * (size_t)n_tab));
    const double dE = (E_max - E_min) / (n_E - 1);
    const double T = n_steps * dt;
    const double scale = dt * dt / (kTwoPi * T);
    cudaError_t e;
    k_count_good<<<1, 1024, 0, s>>>(good, n_traj, ng, n_good_out);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_twiddles<<<(unsigned)((n_tab + 255) / 256), 256, 0, s>>>(tab, n_blocks, n_E, E_min, dE, dt);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const unsigned tiles = (unsigned)(((int64_t)n_E + COLS - 1) / COLS);
    const dim3 grid((unsigned)n_mt, tiles < kMaxGridY ? tiles : kMaxGridY, (tiles + kMaxGridY - 1) / kMaxGridY);
    if (fp64_rows(n_traj, n_E) == 8)
        k_ft_fp64<8><<<grid, 32 * WARPS, 0, s>>>(amp, amp_ld, tab, w, good, n_traj, K, n_blocks, n_E, part);
    else
        k_ft_fp64<2><<<grid, 32 * WARPS, 0, s>>>(amp, amp_ld, tab, w, good, n_traj, K, n_blocks, n_E, part);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    *n_launch = 4;
    return launch_reduce_rows(part, (int)n_mt, n_E, ng, scale, I_out, s);
}

}  // namespace scivr
