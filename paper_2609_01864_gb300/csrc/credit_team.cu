// credit_team.cu -- instantiates the team kernels for one input
// dtype (compiled with -DCREDIT_TIN=0, 1 and 2, like credit_kernels.cu; with
// -DCREDIT_TRACED=1 once more for the kernels that write trace stamps).
#include "credit_row_team.cuh"

#ifndef CREDIT_TIN
#error "CREDIT_TIN must be defined (0 = FP32, 1 = BF16, 2 = FP8-E4M3)"
#endif

#ifndef CREDIT_TRACED
#define CREDIT_TRACED 0
#endif
#define CREDIT_CAT2(a, b) a##b
#define CREDIT_CAT(a, b) CREDIT_CAT2(a, b)
#if CREDIT_TRACED
#define CREDIT_TEAM_KERNEL CREDIT_CAT(team_kernel_traced_tin, CREDIT_TIN)
#else
#define CREDIT_TEAM_KERNEL CREDIT_CAT(team_kernel_tin, CREDIT_TIN)
#endif

namespace credit {

// Clusters: rows at any phase, gamma / beta always in shared memory.
template <int OP, int TOUT>
static const void *team_fn(bool grid, bool aff, bool cluster) {
    constexpr bool N = OP == OP_LN || OP == OP_RMS, R = CREDIT_TRACED != 0;
    if (cluster) return reinterpret_cast<const void *>(&k_row_team<OP, CREDIT_TIN, TOUT, false, N, true, R>);
    if (N && aff)
        return grid ? reinterpret_cast<const void *>(&k_row_team<OP, CREDIT_TIN, TOUT, true, N, false, R>)
                    : reinterpret_cast<const void *>(&k_row_team<OP, CREDIT_TIN, TOUT, false, N, false, R>);
    return grid ? reinterpret_cast<const void *>(&k_row_team<OP, CREDIT_TIN, TOUT, true, false, false, R>)
                : reinterpret_cast<const void *>(&k_row_team<OP, CREDIT_TIN, TOUT, false, false, false, R>);
}

template <int OP>
static const void *team_out(int tout, bool grid, bool aff, bool cluster) {
    switch (tout) {
    case DT_F32: return team_fn<OP, DT_F32>(grid, aff, cluster);
    case DT_BF16: return team_fn<OP, DT_BF16>(grid, aff, cluster);
    case DT_E4M3: return team_fn<OP, DT_E4M3>(grid, aff, cluster);
    default: return nullptr;
    }
}

const void *CREDIT_TEAM_KERNEL(int op, int tout, bool grid, bool aff, bool cluster) {
    switch (op) {
    case OP_SOFTMAX: return team_out<OP_SOFTMAX>(tout, grid, aff, cluster);
    case OP_LSE: return team_fn<OP_LSE, DT_F32>(grid, aff, cluster);
    case OP_LN: return team_out<OP_LN>(tout, grid, aff, cluster);
    case OP_RMS: return team_out<OP_RMS>(tout, grid, aff, cluster);
#if CREDIT_TIN != 2
    case OP_Q8: return tout == DT_I8 ? team_fn<OP_Q8, DT_I8>(grid, aff, cluster) : nullptr;
#endif
    default: return nullptr;
    }
}

}  // namespace credit
