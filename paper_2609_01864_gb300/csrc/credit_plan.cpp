// credit_plan.cpp -- plan selection (CREDIT Sec. III-D).
//
// Candidates for a shape: the one-CTA staged path (P = 1), the cluster path
// for every P in {2, 4, 8, 16} that passes the capacity check of Eq. 3 and
// can be scheduled (max active clusters > 0), and the two-pass global-reread
// path.  Without calibration data the built-in heuristic below is used; the
// analytic model of Eq. 7-9 and the learned model plug in through
// credit_model.cpp.
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <initializer_list>
#include <mutex>
#include <unordered_map>

#include "credit_host.h"
#include "credit_model.h"

namespace credit {

// Plans chosen by credit_plan_ex, per (device, op, rows, cols, dtypes): the
// learned planner evaluates every candidate through the network ensemble on
// the host, which costs more than a short launch, so a call without a plan
// reuses the choice made for the same shape.  Emptied when the calibration or
// the model changes; bypassed while CREDIT_FORCE_PATH or CREDIT_MODEL select
// a planner by environment.
namespace {
struct PlanKey {
    int dev, op, tin, tout;
    long long rows, cols;
    bool operator==(const PlanKey &o) const {
        return dev == o.dev && op == o.op && tin == o.tin && tout == o.tout && rows == o.rows && cols == o.cols;
    }
};
struct PlanKeyHash {
    size_t operator()(const PlanKey &k) const {
        uint64_t h = 1469598103934665603ull;
        const long long v[6] = {k.dev, k.op, k.tin, k.tout, k.rows, k.cols};
        for (long long x : v) h = (h ^ static_cast<uint64_t>(x)) * 1099511628211ull;
        return static_cast<size_t>(h);
    }
};
std::mutex g_plan_mu;
std::unordered_map<PlanKey, credit_plan_t, PlanKeyHash> g_plan_cache;
std::atomic<unsigned long long> g_plan_gen{0};
unsigned long long g_cache_gen = 0;
constexpr size_t kPlanCacheMax = 4096;
}  // namespace

void bump_plan_generation() { g_plan_gen.fetch_add(1); }

static bool env_force(const DeviceInfo *di, credit_plan_t *p, long long cols, int tin) {
    const char *fp = std::getenv("CREDIT_FORCE_PATH");
    if (!fp || !*fp) return false;
    std::memset(p, 0, sizeof(*p));
    const char *fP = std::getenv("CREDIT_FORCE_P");
    const char *fG = std::getenv("CREDIT_FORCE_G");
    const char *fT = std::getenv("CREDIT_FORCE_THREADS");
    const char *fR = std::getenv("CREDIT_FORCE_RING");
    const char *fC = std::getenv("CREDIT_FORCE_CHUNK");
    const char *fRd = std::getenv("CREDIT_FORCE_REDUCERS");
    p->threads = fT ? std::atoi(fT) : 0;
    p->ring_chunks = fR ? std::atoi(fR) : 0;
    p->chunk_bytes = fC ? std::atoi(fC) : 0;
    p->reducer_threads = fRd ? std::atoi(fRd) : 0;
    p->source = 2;
    if (!std::strcmp(fp, "one_cta") || !std::strcmp(fp, "cluster")) {
        const bool one = !std::strcmp(fp, "one_cta");
        p->path = one ? CREDIT_PATH_ONE_CTA : CREDIT_PATH_CLUSTER;
        p->cluster_size = one ? 1 : (fP ? std::atoi(fP) : 4);
        p->ctas_per_row = p->cluster_size;
        RingCfg rc;
        if (di && ring_config(*di, cols, dtype_size(tin), p->cluster_size, p->ring_chunks, p->chunk_bytes,
                              p->threads, p->reducer_threads, 0, &rc))
            p->smem_bytes = rc.smem;
    } else if (!std::strcmp(fp, "two_pass")) {
        p->path = CREDIT_PATH_TWO_PASS;
        p->cluster_size = 1;
        p->ctas_per_row = fG ? std::atoi(fG) : 1;
    } else {
        return false;
    }
    return true;
}

// Split factor for the two-pass path: enough CTAs to cover the GPU several
// times over, but no CTA with fewer than ~1024 16-byte groups.
int two_pass_split(int sm_count, long long rows, long long cols, int isz) {
    const long long target = 4LL * sm_count;
    if (rows >= target) return 1;
    long long G = (target + rows - 1) / rows;
    const long long groups = (cols * isz) / 16;
    long long gmax = groups / 1024;
    if (gmax < 1) gmax = 1;
    if (G > gmax) G = gmax;
    if (G > 1024) G = 1024;
    return static_cast<int>(G < 1 ? 1 : G);
}

// Widest rows that row_plan gives to one CTA's teams, and to a cluster's.
constexpr long long kTeamRowBytes = 96 << 10, kTeamClusterBytes = 1 << 20;

// Rows (or slices of rows) of one CTA's teams that fit shared memory beside the op's gamma / beta.
static long long team_room(const DeviceInfo &di, long long cols, int isz, int nab, int P) {
    const long long V = 16 / isz, groups = (cols / V + P - 1) / P;
    const long long aff = nab * (groups + 3) * V * 4, room = di.smem_optin - (20 << 10) - aff;
    return groups < 1 ? 16 : room < 0 ? 0 : room / (groups * 16);
}

// Rows for k_row_team: whole rows in one CTA (P = 1), or split over a cluster.
// Measured on GB300 against the learned model's picks (us, the model's pick ->
// this one).
// P = 1, rows of 256 B to 96 KiB, 96 to 16384 of them, on and off the 16-byte
// grid:
//   16384 x 4096 BF16 RMSNorm 80 -> 47, 65536 x 1024 FP32 softmax 252 -> 92,
//   20325 x 3616 BF16 softmax 130 -> 50, 16384 x 8192 BF16 -> FP8 RMSNorm
//   167 -> 81, FP8 LayerNorm 332 -> 115, 10800 x 4096 BF16 int8 93 -> 26,
//   1000 rows of 24 KiB: 5-60% faster for every op and type but FP8 softmax.
// Its limits: norms of rows on the 16-byte grid go to the tensor-memory path
// from 48 KiB (1000 x 64 KiB BF16 RMSNorm 29 against 38), off the grid, where
// that path loses its staged gamma / beta, only above 96 KiB; E4M3 softmax and
// log-sum-exp have their code tables (24 KiB rows of FP8 log-sum-exp 11
// against 15, 32 KiB of FP8 softmax 13 against 15); log-sum-exp has no output
// for the second look at the row to save, in BF16 it draws level at 32 KiB.
// P > 1, where the other paths are weak: rows off the grid, and norms with FP8
// rows or outputs.  The smallest P that leaves an SM room for three teams with
// gamma / beta (1500 rows; with two teams the copies show: 300 KiB BF16
// LayerNorm P = 8 580, P = 16 296, 504 before): LayerNorm 140 KiB FP32 128 ->
// 110, BF16 252 -> 140, FP8 1359 -> 436, RMSNorm 200 KiB BF16 217 -> 146, 140
// KiB BF16 -> FP8 252 -> 126 (on the grid 208 -> 120), FP8 726 -> 267, softmax
// 300 KiB BF16 222 -> 194, int8 200 KiB BF16 234 -> 102; without gamma P = 2
// stays behind P = 4 (140 KiB int8 84 against 71).  Few rows keep P = 1 up to
// 96 KiB (100 x 48 KiB FP32 LayerNorm 9 against 12) unless they are FP8, whose
// arithmetic is worth more CTAs (100 x 64 KiB LayerNorm 40 -> 24; not RMSNorm on
// the grid, 300 x 60 KiB 26 against 33).  With fewer
// than four rows per SM the two-pass paths find the rows in L2: softmax (150 x
// 200 KiB FP32 16 against 19) and FP32 norms of 56 to 280 KiB (600 x 80 KiB
// RMSNorm 23 against 28, 150 x 140 KiB 13 against 17; 300 KiB 32 -> 29) stay
// there.  Softmax is split from
// 128 KiB (1300 x 96 KiB BF16 60 against 64) to 256 KiB in FP32 (1300 x 300
// KiB 156 against 173), 512 KiB in BF16 (600 x 420 KiB 136 -> 112, 960 KiB 279
// against 319).
static bool row_plan(const DeviceInfo &di, int op, long long rows, long long cols, int tin, int tout,
                     credit_plan_t *p) {
    const int isz = dtype_size(tin), nab = op == CREDIT_OP_LAYERNORM ? 2 : op == CREDIT_OP_RMSNORM ? 1 : 0;
    const bool grid = cols * isz % 16 == 0, fp8 = tin == 2 || tout == 2, sm8 = op == CREDIT_OP_SOFTMAX && tin == 2;
    const long long bytes = cols * isz;
    const bool many = rows >= 4LL * di.sm_count;
    long long limit = kTeamRowBytes;
    if (op == CREDIT_OP_LOGSUMEXP) limit = tin == 0 ? limit : tin == 1 ? 32 << 10 : 8 << 10;
    else if (sm8) limit = 24 << 10;
    else if (nab && !fp8 && grid) limit = 48 << 10;
    else if (nab && tin == 0 && tout == 0 && !many) limit = 56 << 10;
    int P = bytes <= limit ? 1 : 0;
    const bool pays = op == CREDIT_OP_SOFTMAX ? many && bytes > 128 << 10 && bytes <= (tin == 0 ? 256 << 10 : 512 << 10)
                      : nab && tin == 0 && tout == 0 ? many || (bytes > 280 << 10 && bytes <= 512 << 10 &&
                                                              (nab > 1 || rows >= di.sm_count))
                                                     : true;
    const bool split = op != CREDIT_OP_LOGSUMEXP && !sm8 && pays && (!grid || (nab && fp8)) &&
                       bytes <= (grid ? 450LL << 10 : kTeamClusterBytes);
    if (split && (P == 0 || (nab && (many || (tin == 2 && !(op == CREDIT_OP_RMSNORM && grid && bytes <= 64 << 10)))))) {
        int q = nab || P ? 1 : 4;
        while (q <= 16 && team_room(di, cols, isz, nab, q) < 3) q *= 2;
        if (q <= 16 && (q > 1 || P)) P = q;
    }
    TeamCfg tc;
    if (P == 0 || !team_config(di, rows, cols, isz, nab, P, 0, &tc)) return false;
    std::memset(p, 0, sizeof(*p));
    p->source = 3;
    p->path = P == 1 ? CREDIT_PATH_ONE_CTA : CREDIT_PATH_CLUSTER;
    p->cluster_size = P;
    p->ctas_per_row = P;
    p->retain = CREDIT_RETAIN_ROW;
    p->smem_bytes = tc.smem;
    return true;
}

// Rows over warps (k_row_warps), for softmax, log-sum-exp and int8 of FP32 and
// BF16 rows.  u is the number of warps whose buffers of 880 16-byte groups hold
// a row, fill the part of them that it fills.  Clusters of CTAs of 8 warps, two
// to an SM, of which a row takes four warps each (rows of 128 KiB 104 us, 107
// with its 16 warps in one CTA), eight of 8 CTAs from u = 64 (512 KiB 408, over
// 16 CTAs 436), and eight CTAs of 16 warps at u = 128; one CTA while that holds
// the row (but for many rows of u = 8, 2600 FP32 of 96 KiB 94 us against 80
// over four), or there is hardly a row per SM (150 rows of 128 KiB 11 against
// 13).
// Where it pays, the other plans' time over this one's for 200, 400, 600, 1300
// and 2600 rows (u = 8 .. 128 at six fills and 24 widths in whole KiB, on and
// off the 16-byte grid):
//   - half-full buffers keep half the bytes in flight.  FP32 softmax u = 32 and
//     64 above fill 0.6 1.02-1.46, at 0.5-0.58 0.86-1.18 (448 KiB 0.87, 512 KiB
//     0.92); u = 128 0.81-1.2 at all.  BF16 softmax, whose other path reads the
//     row twice, 1.05-1.53 from u = 16 on, u = 128 0.95-1.16.
//   - u = 8 (55 to 110 KiB) competes with whole rows in one CTA up to 96 KiB
//     (kTeamRowBytes): beyond, FP32 softmax 1.0-1.26, BF16 1.02-1.43, int8
//     1.9-2.7 (0.88-1.45 off the grid); within, BF16 softmax off the grid
//     1.0-1.31, on it 0.97-1.2, but with more than 8 rows per SM 0.90-0.95 from
//     fill 0.65 on; FP32 softmax and int8 0.78-1.0, log-sum-exp 0.95-1.35.
//   - u = 16: FP32 softmax above two rows per SM 0.96-1.42, below 0.91-1.09;
//     BF16 int8 off the grid below two rows per SM 0.72-1.01.  Int8 from u = 16
//     on 1.0-2.9 else; FP32 u = 128 behind eight CTAs' rings of whole 16 KiB
//     chunks (896 and 1024 KiB 0.86-0.95), 1.5-1.7 at other widths of that fill.
//   - log-sum-exp, with no output to save a second look for: u = 8 0.95-1.53,
//     BF16 u = 4 from fill 0.72 1.0-1.41; FP32 u = 16 above 8 rows per SM
//     1.13-1.3, below 0.83-1.16; wider 0.54-1.25.
static bool warps_plan(const DeviceInfo &di, int op, long long rows, long long cols, int tin, int tout,
                       credit_plan_t *p) {
    if (tin > 1) return false;
    RowWarpsCfg c;
    if (!row_warps_config(di, op, tin, tout, rows, cols, 1, 16, &c) &&
        !row_warps_config(di, op, tin, tout, rows, cols, 16, 16, &c))
        return false;
    const long long bytes = cols * dtype_size(tin);
    const bool f32 = tin == 0, grid = bytes % 16 == 0, many = rows >= 8LL * di.sm_count, two = rows > 2LL * di.sm_count;
    const int u = 1 << c.lu;
    const float fill = static_cast<float>(bytes / 16) / static_cast<float>(880 * u);
    bool pays = false;
    if (op == CREDIT_OP_SOFTMAX) {
        if (u == 8)
            pays = bytes > kTeamRowBytes || (!f32 && fill > 0.54f && (!grid || !many || fill < 0.65f));
        else if (u == 16)
            pays = !f32 || two;
        else
            pays = f32 ? (u == 32 || u == 64) && fill > 0.6f : u >= 32;
    } else if (op == CREDIT_OP_QUANT_INT8) {
        const bool ring8 = bytes / 16 * 16 % (8 * 16384) == 0 && (grid || bytes > kTeamClusterBytes);
        pays = u == 8    ? bytes > kTeamRowBytes
               : u == 16 ? f32 || grid || two
                         : u > 16 && !(f32 && u == 128 && fill < 0.6f && ring8);
    } else if (op == CREDIT_OP_LOGSUMEXP) {
        pays = f32 ? (u == 8 && fill > 0.54f) || (u == 16 && many) : u == 8 || (u == 4 && fill > 0.72f);
    }
    if (!pays) return false;
    int P = u < 8 ? 1 : u <= 8 ? (op != CREDIT_OP_LOGSUMEXP && rows >= 8LL * di.sm_count ? 4 : 1) : u <= 32 ? u / 4 : 8;
    int W = u <= 64 ? 8 : 16;
    if (u == 16 && rows < 2LL * di.sm_count) {
        P = 1;
        W = 16;
    }
    if (!row_warps_config(di, op, tin, tout, rows, cols, P, W, &c)) return false;
    std::memset(p, 0, sizeof(*p));
    p->source = 3;
    p->path = P == 1 ? CREDIT_PATH_ONE_CTA : CREDIT_PATH_CLUSTER;
    p->cluster_size = p->ctas_per_row = P;
    p->threads = 32 * W;
    p->retain = CREDIT_RETAIN_WARPS;
    p->smem_bytes = c.smem;
    return true;
}

// Rule for int8 quantisation (measured on GB300, 4096 rows of 16K-256K FP32
// columns): the smallest cluster whose slices fit the tensor-memory tier
// (128 KiB); the fewest CTAs per row keeps the most rows in flight and the
// exchange shortest.  Two-pass when no staged plan fits.
static bool quant_plan(const DeviceInfo &di, int device, long long rows, long long cols, int tin, credit_plan_t *p) {
    const int isz = dtype_size(tin);
    for (int P : {1, 2, 4, 8, 16}) {
        RingCfg rc;
        if (!ring_config_tm(di, cols, isz, P, 0, 0, 0, &rc)) continue;
        if (ring_max_clusters(device, CREDIT_OP_QUANT_INT8, tin, CREDIT_INT8, P, rc.threads, rc.smem, true) <= 0) continue;
        p->path = P == 1 ? CREDIT_PATH_ONE_CTA : CREDIT_PATH_CLUSTER;
        p->cluster_size = P;
        p->ctas_per_row = P;
        p->retain = CREDIT_RETAIN_TMEM;
        p->smem_bytes = rc.smem;
        return true;
    }
    p->path = CREDIT_PATH_TWO_PASS;
    p->cluster_size = 1;
    p->ctas_per_row = two_pass_split(di.sm_count, rows, cols, isz);
    return true;
}

// Staged cluster plans whose rows lie off the 16-byte grid, where int8 codes
// are stored byte by byte from the writer warps and LayerNorm's gamma / beta
// are read element by element: the two-pass path is ahead (300 rows, this <-
// the plan): 280001 FP32 int8 128 us <- 196, 600001 BF16 int8 166 <- 346 (from
// 16 CTAs on: eight are ahead, 262145 FP32 94 against 112),
// 400001 FP32 LayerNorm 286 <- 872, 400001 FP8 LayerNorm (70 rows) 127 <- 249.
// RMSNorm and softmax, with one or no such array, stay (1500 x 280001 FP32 787
// against 892, 611 against 805).
static void off_grid_plan(const DeviceInfo &di, int op, long long rows, long long cols, int tin, credit_plan_t *p) {
    const int isz = dtype_size(tin);
    if (p->path != CREDIT_PATH_CLUSTER || p->retain == CREDIT_RETAIN_ROW || p->retain == CREDIT_RETAIN_WARPS || cols * isz % 16 == 0 ||
        (!(op == CREDIT_OP_LAYERNORM && p->cluster_size >= 8) && !(op == CREDIT_OP_QUANT_INT8 && p->cluster_size == 16)))
        return;
    std::memset(p, 0, sizeof(*p));
    p->source = 3;
    p->path = CREDIT_PATH_TWO_PASS;
    p->cluster_size = 1;
    p->ctas_per_row = two_pass_split(di.sm_count, rows, cols, isz);
}

void heuristic_plan(const DeviceInfo &di, int device, int op, long long rows, long long cols, int tin, int tout,
                    credit_plan_t *p) {
    if (warps_plan(di, op, rows, cols, tin, tout, p) || row_plan(di, op, rows, cols, tin, tout, p)) return;
    std::memset(p, 0, sizeof(*p));
    p->source = 3;
    if (op == CREDIT_OP_QUANT_INT8 && quant_plan(di, device, rows, cols, tin, p)) return;
    const int isz = dtype_size(tin);
    if (op != 1) {
        // Smallest P whose slice is <= 64 KiB, else the smallest P that fits.
        int pick = 0;
        RingCfg best{};
        for (int pass = 0; pass < 2 && !pick; ++pass) {
            for (int P : {1, 2, 4, 8, 16}) {
                RingCfg rc;
                if (!ring_config(di, cols, isz, P, 0, 0, 0, 0, 0, &rc)) continue;
                if (pass == 0 && rc.body_max > 65536) continue;
                if (ring_max_clusters(device, op, tin, tout, P, rc.threads, rc.smem) <= 0) continue;
                pick = P;
                best = rc;
                break;
            }
        }
        if (pick) {
            p->path = pick == 1 ? CREDIT_PATH_ONE_CTA : CREDIT_PATH_CLUSTER;
            p->cluster_size = pick;
            p->ctas_per_row = pick;
            p->smem_bytes = best.smem;
            return;
        }
    }
    p->path = CREDIT_PATH_TWO_PASS;
    p->cluster_size = 1;
    p->ctas_per_row = two_pass_split(di.sm_count, rows, cols, isz);
}

}  // namespace credit

using namespace credit;

extern "C" {

credit_status credit_plan_ex(credit_op op, int64_t rows, int64_t cols, credit_dtype in_dtype, credit_dtype out_dtype,
                             credit_plan_t *out) {
    const bool q8 = op == CREDIT_OP_QUANT_INT8;
    if (!out || ((op < 0 || op > 3) && !q8) || in_dtype < 0 || in_dtype > 2 || out_dtype < 0 || out_dtype > 3)
        return CREDIT_ERR_INVALID_ARG;
    if (q8 != (out_dtype == CREDIT_INT8)) return CREDIT_ERR_INVALID_ARG;
    if (q8 && in_dtype == CREDIT_FP8_E4M3) return CREDIT_ERR_UNSUPPORTED;
    if (rows < 0 || cols <= 0) return CREDIT_ERR_INVALID_ARG;
    const int tout = op == CREDIT_OP_LOGSUMEXP ? 0 : out_dtype;
    int dev = 0;
    credit_status st = ensure_init(&dev, nullptr);
    if (st != CREDIT_OK) return st;
    const DeviceInfo *di = device_info(dev);
    if (!di) return CREDIT_ERR_NOT_INITIALIZED;
    if (env_force(di, out, cols, in_dtype)) return CREDIT_OK;
    const char *menv = std::getenv("CREDIT_MODEL");
    const bool cache = !(menv && *menv);
    const PlanKey key{dev, static_cast<int>(op), static_cast<int>(in_dtype), tout, rows, cols};
    const unsigned long long gen = g_plan_gen.load();
    if (cache) {
        std::lock_guard<std::mutex> lk(g_plan_mu);
        if (g_cache_gen != gen) {
            g_plan_cache.clear();
            g_cache_gen = gen;
        }
        const auto it = g_plan_cache.find(key);
        if (it != g_plan_cache.end()) {
            *out = it->second;
            return CREDIT_OK;
        }
    }
    // narrow rows take the rule unless CREDIT_MODEL asks for a model's own choice; the calibration and the
    // learned model cover the four ops of Sec. III-B; the quantiser takes the rule
    if (!(cache && (warps_plan(*di, op, rows, cols, in_dtype, tout, out) ||
                    row_plan(*di, op, rows, cols, in_dtype, tout, out))) &&
        (q8 || !model_plan(*di, dev, op, rows, cols, in_dtype, tout, out)))
        heuristic_plan(*di, dev, op, rows, cols, in_dtype, tout, out);
    if (cache) off_grid_plan(*di, op, rows, cols, in_dtype, out);
    if (cache) {
        std::lock_guard<std::mutex> lk(g_plan_mu);
        if (g_cache_gen == gen) {
            if (g_plan_cache.size() >= kPlanCacheMax) g_plan_cache.clear();
            g_plan_cache[key] = *out;
        }
    }
    return CREDIT_OK;
}

credit_status credit_plan(credit_op op, int64_t rows, int64_t cols, credit_dtype dtype, credit_plan_t *out) {
    return credit_plan_ex(op, rows, cols, dtype, op == CREDIT_OP_LOGSUMEXP ? CREDIT_F32 : dtype, out);
}

}  // extern "C"
