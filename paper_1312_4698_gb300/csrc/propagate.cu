// Propagation dispatch: picks the kernel instantiation for (F, precision, schedule).
#include "scivr_internal.cuh"

namespace scivr {

template <int F> cudaError_t launch_tpt_fp64(const PropLaunch &L, cudaStream_t s);
template <int F> cudaError_t launch_group_mixed(const PropLaunch &L, cudaStream_t s);
template <int F> cudaError_t launch_group_fp64(const PropLaunch &L, cudaStream_t s);
template <int F>
cudaError_t launch_group_batch_mixed_F(int warps, const PropLaunch *items, const int2 *work, int n_work,
                                      int *counter, int n_sm, cudaStream_t s);

int batch_warp_candidates(int F, bool has4, int *out)
{
    if (F < 1 || F > 24) return 0;
    if (!has4 && cubic_schedule(F)) { out[0] = 4; return 1; }
    if (F > 9) { out[0] = F == 13 ? 4 : 8; return 1; }   // wide groups: one shape each (lg_warps)
    if (mixed_group_lanes(F) == 32) { out[0] = 1; out[1] = 2; }
    else { out[0] = 2; out[1] = 4; }
    return 2;
}

cudaError_t launch_group_batch_mixed(int F, int warps, const PropLaunch *items, const int2 *work, int n_work,
                                     int *counter, int n_sm, cudaStream_t s)
{
    switch (F) {
#define SCIVR_B(FF) case FF: return launch_group_batch_mixed_F<FF>(warps, items, work, n_work, counter, n_sm, s);
    SCIVR_B(1) SCIVR_B(2) SCIVR_B(3) SCIVR_B(4) SCIVR_B(5) SCIVR_B(6) SCIVR_B(7) SCIVR_B(8) SCIVR_B(9)
    SCIVR_B(10) SCIVR_B(11) SCIVR_B(12) SCIVR_B(13) SCIVR_B(14) SCIVR_B(15) SCIVR_B(16)
    SCIVR_B(17) SCIVR_B(18) SCIVR_B(19) SCIVR_B(20) SCIVR_B(21) SCIVR_B(22) SCIVR_B(23) SCIVR_B(24)
#undef SCIVR_B
    default: return cudaErrorInvalidValue;
    }
}

namespace {

constexpr int kMaxThreadF = 9;   // thread-per-trajectory FP64 kernel
constexpr int kMaxGroupF = 9;    // FP64 lane-group kernel
constexpr int kMaxMixedF = 24;   // mixed lane-group kernel (one trajectory per warp above F = 9, two columns per lane above F = 16)

// Schedule choice when the caller leaves it to the library: the lane groups, but in FP64 at F <= 2
// beyond the numbers of trajectories where the thread kernel passes them.  Measured on GB300, us
// per step, groups / thread: F = 1: 6.3 / 9.8 at 8192 trajectories, 11.4 / 11.0 at 19456,
// 39.8 / 36.8 at 65536; F = 2: 15.7 / 23.5, 31.3 / 26.1, 109 / 90; F = 3: 26.6 / 49.8, 51.8 / 54.3,
// 169 / 199; F = 6: 117 / 252, 236 / 297, 821 / 1005; F = 9: 458 / 1005, 803 / 1106 at 16384.  The
// lines are where the groups' rounds of four warps per SM (9728 trajectories a round at F = 1, 4864
// at F = 2) add up to the thread kernel's one flat round.  That round is also the shorter one while the
// groups take four at F = 3 without couplings or with both kinds (64 steps of 16384: 2.59 / 2.52 and
// 3.44 / 3.29 ms; cubic alone 3.14 / 3.31, quartic alone 3.29 / 3.30) and at F = 5 without (6.62 / 6.37; with
// both 9.51 / 10.47).  And a chunk's records cost the groups as much for one step as for a chunk: one
// step of 16384 takes them 1.0 to 1.5 times as long at F = 3..9, two steps 1.0 to 1.2 times up to F = 7.
int choose(const PropLaunch &L)
{
    const int F = L.args.F;
    const int64_t n = L.n_traj;
    if (L.args.precision == SCIVR_MIXED) return SCIVR_KERNEL_GROUP;
    if (F > kMaxGroupF) return SCIVR_KERNEL_THREAD;
    const bool has3 = L.pes.has3, has4 = L.pes.has4;
    if (n > 14592 && n <= 19456 && ((F == 3 && has3 == has4) || (F == 5 && !has3 && !has4))) return SCIVR_KERNEL_THREAD;
    if (L.args.n_steps == 1 && n > (F <= 7 ? 9728 : 14592)) return SCIVR_KERNEL_THREAD;
    if (L.args.n_steps == 2 && n > 14592 && F <= 7) return SCIVR_KERNEL_THREAD;
    if (F > 2) return SCIVR_KERNEL_GROUP;
    return n > (F == 1 ? 9728 : 14592) ? SCIVR_KERNEL_THREAD : SCIVR_KERNEL_GROUP;
}

}  // namespace

bool propagate_supported(int F, int precision, int kernel)
{
    if (F < 1) return false;
    if (precision == SCIVR_MIXED) return kernel != SCIVR_KERNEL_THREAD && F <= kMaxMixedF;
    if (precision != SCIVR_FP64) return false;
    if (kernel == SCIVR_KERNEL_THREAD) return F <= kMaxThreadF;
    if (kernel == SCIVR_KERNEL_GROUP) return F <= kMaxGroupF;
    return F <= kMaxThreadF;
}

#define SCIVR_CASES(M, X) \
    case 1: return M<1>(X, s); case 2: return M<2>(X, s); case 3: return M<3>(X, s); \
    case 4: return M<4>(X, s); case 5: return M<5>(X, s); case 6: return M<6>(X, s); \
    case 7: return M<7>(X, s); case 8: return M<8>(X, s);

cudaError_t launch_propagate(const PropLaunch &L, cudaStream_t s, int *n_launch)
{
    *n_launch = 1;
    const int kern = L.args.kernel == SCIVR_KERNEL_AUTO ? choose(L) : L.args.kernel;
    if (L.args.precision == SCIVR_MIXED) {
        switch (L.args.F) {
            SCIVR_CASES(launch_group_mixed, L)
            case 9: return launch_group_mixed<9>(L, s);
            case 10: return launch_group_mixed<10>(L, s);
            case 11: return launch_group_mixed<11>(L, s);
            case 12: return launch_group_mixed<12>(L, s);
            case 13: return launch_group_mixed<13>(L, s);
            case 14: return launch_group_mixed<14>(L, s);
            case 15: return launch_group_mixed<15>(L, s);
            case 16: return launch_group_mixed<16>(L, s);
            case 17: return launch_group_mixed<17>(L, s);
            case 18: return launch_group_mixed<18>(L, s);
            case 19: return launch_group_mixed<19>(L, s);
            case 20: return launch_group_mixed<20>(L, s);
            case 21: return launch_group_mixed<21>(L, s);
            case 22: return launch_group_mixed<22>(L, s);
            case 23: return launch_group_mixed<23>(L, s);
            case 24: return launch_group_mixed<24>(L, s);
            default: break;
        }
    } else if (kern == SCIVR_KERNEL_GROUP) {
        switch (L.args.F) { SCIVR_CASES(launch_group_fp64, L) case 9: return launch_group_fp64<9>(L, s); default: break; }
    } else {
        switch (L.args.F) {
            SCIVR_CASES(launch_tpt_fp64, L)
            case 9: return launch_tpt_fp64<9>(L, s);
            default: break;
        }
    }
    *n_launch = 0;
    return cudaErrorInvalidValue;
}

}  // namespace scivr
