// credit_warps.cu -- k_row_warps for rows of one width: softmax, log-sum-exp
// and int8 quantisation of FP32 and BF16 rows (plans with CREDIT_RETAIN_WARPS).
// Compiled twice: with -DCREDIT_TRACED=1 for the kernels that write trace
// stamps alone.
#include <cuda_runtime.h>

#include "../../include/credit.h"
#include "credit_host.h"
#include "credit_row_warps.cuh"

namespace credit {

template <int W, bool TR>
static const void *kernel_of(int op, int tin) {
    const bool f32 = tin == DT_F32;
    switch (op) {
    case OP_SOFTMAX:
        return f32 ? reinterpret_cast<const void *>(&k_row_warps<OP_SOFTMAX, DT_F32, W, TR>)
                   : reinterpret_cast<const void *>(&k_row_warps<OP_SOFTMAX, DT_BF16, W, TR>);
    case OP_LSE:
        return f32 ? reinterpret_cast<const void *>(&k_row_warps<OP_LSE, DT_F32, W, TR>)
                   : reinterpret_cast<const void *>(&k_row_warps<OP_LSE, DT_BF16, W, TR>);
    case OP_Q8:
        return f32 ? reinterpret_cast<const void *>(&k_row_warps<OP_Q8, DT_F32, W, TR>)
                   : reinterpret_cast<const void *>(&k_row_warps<OP_Q8, DT_BF16, W, TR>);
    default: return nullptr;
    }
}

const void *row_warps_kernel_traced(int op, int tin, int W);

#if CREDIT_TRACED
const void *row_warps_kernel_traced(int op, int tin, int W) {
    return W == kWWarps ? kernel_of<kWWarps, true>(op, tin) : kernel_of<kWWarps / 2, true>(op, tin);
}
#else
bool row_warps_config(const DeviceInfo &di, int op, int tin, int tout, long long rows, long long cols, int P, int W,
                      RowWarpsCfg *out) {
    if (tin != DT_F32 && tin != DT_BF16) return false;
    if (op == OP_SOFTMAX ? tout != tin : op == OP_Q8 ? tout != DT_I8 : op != OP_LSE) return false;
    if (!team_cluster(di, P) || (W != kWWarps && W != kWWarps / 2)) return false;
    if (rows > (1LL << 30) || cols > (1LL << 24) || warps_smem(W) > di.smem_optin) return false;
    const long long groups = cols * dtype_size(tin) / 16 + 1;
    int lu = 0;
    while ((1 << lu) < P) ++lu;
    while (((groups - 1) >> lu) + 1 > 2 * kWHalf)
        if ((1 << ++lu) > P * W) return false;
    *out = {P, W, lu, warps_smem(W), W == kWWarps ? kernel_of<kWWarps, false>(op, tin) : kernel_of<kWWarps / 2, false>(op, tin)};
    return out->fn != nullptr;
}

credit_status run_row_warps(int device, const credit_args *a, const RowWarpsCfg &cfg, cudaStream_t s) {
    WarpArgs w{};
    w.trace = trace_buffer(&w.trace_rows);
    const void *fn = w.trace != nullptr ? row_warps_kernel_traced(a->op, a->in_dtype, cfg.W) : cfg.fn;
    credit_status st = prepare_staged_kernel(device, fn);
    if (st != CREDIT_OK) return st;
    const int most = staged_max_clusters(device, fn, cfg.P, 32 * cfg.W, cfg.smem, false);
    if (most <= 0) return CREDIT_ERR_UNSUPPORTED;
    const long long per = static_cast<long long>(cfg.P) * cfg.W >> cfg.lu;  // rows a cluster works on at a time
    const long long want = (a->rows + per - 1) / per;
    const int ncl = static_cast<int>(want < most ? want : most);
    w.in = static_cast<const unsigned char *>(a->in);
    w.out = static_cast<unsigned char *>(a->out);
    w.n_classes = 1;
    w.cls[0].lu = cfg.lu;
    while ((1 << w.cls[0].lw) < cfg.P) ++w.cls[0].lw;
    w.cls[0].row_end = static_cast<int>(a->rows);
    w.cls[0].k_end = static_cast<int>((a->rows + ncl * per - 1) / (ncl * per));
    w.err = device_error_word(device);
    w.ld_in = a->ld_in ? a->ld_in : a->cols;
    w.ld_out = a->op == OP_LSE ? 1 : a->ld_out ? a->ld_out : a->cols;
    w.cols = static_cast<int>(a->cols);
    w.out_scale = a->out_scale;
    void *args[] = {&w};
    const cudaError_t e = launch_kernel(fn, dim3(static_cast<unsigned>(cfg.P * ncl)), dim3(32 * cfg.W),
                                        static_cast<size_t>(cfg.smem), cfg.P, s, args);
    return e == cudaSuccess ? CREDIT_OK : CREDIT_ERR_CUDA;
}
#endif

}  // namespace credit
