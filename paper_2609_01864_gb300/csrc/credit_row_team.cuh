// credit_row_team.cuh -- whole rows in shared memory, several per SM at once: rows of one CTA (up to ~100 KiB), or the
// slices of rows split over a cluster (up to 1 MiB as planned).
//
// k_row_team is the staged method (one HBM read and one write, Eq. 4) without
// roles: one persistent CTA of up to 1024 threads per SM is split into teams of
// T threads (four to eight 16-byte groups of the row per thread); a team walks
// rows g, g + teams, ...  Over a cluster the teams of one number hold a row's
// slices and exchange their partials over DSMEM (Eq. 5).
//
//   - bulk-async copies bring rows into the team's S shared-memory stages;
//     a stage takes its next row as soon as the team is done with it (at the
//     first reduction of the following row, whose barrier shows that), so the
//     copy runs behind the team's work;
//   - the row statistics take one or two reductions of one float over the
//     team, the row being read again from shared memory for each step;
//   - the outputs are written from shared memory.
//
// The teams of an SM overlap one another's copies, reductions and stores.
// k_ring spends warps on roles and a chunk ring that narrow rows do not need,
// and k_tp_fused waits for its loads once per CTA and row.
//
// gamma / beta sit in shared memory once per SM when they fit beside the
// stages (any row phase: they are indexed by column; a cluster's CTA holds its
// slice's).  Rows off the 16-byte grid are cut as everywhere (Eq. 2); their
// head and tail elements are held one per thread and loaded one row ahead.  A
// row without a whole group asks for no copy and waits for none, while the
// stages' phases go on with the rows: rows of one team all have a group or all
// have none, since rows that short make 32 teams wherever a team has a second
// row, and a team's rows then lie a multiple of 32 apart, at one phase.
//
// A second look at the row is a shared-memory read, so the statistics take two
// local steps: softmax the maximum first and then each exponential, LayerNorm
// the mean about the row's first group's first element and then the squared
// deviations.
#pragma once

#include "credit_rows.cuh"

namespace credit {

constexpr int kTeamGroups = 4;         // 16-byte groups per thread and row
constexpr int kTeamMaxThreads = 1024;  // threads of a CTA, and of the largest team
constexpr int kTeamMaxTeams = 32;
constexpr int kTeamMaxStages = 4;
// Shared memory: [0, 1024) mbarriers [team][stage], [1024, 1024 + teams * 512)
// reduction scratch [team][4][32 floats], gamma, beta (16-byte
// multiples plus one pad group each), then the stages.
constexpr int kTeamXchBytes = 544;  // cluster exchange of one team: 512 bytes of slots, four mbarriers
__host__ __device__ constexpr int team_ctrl_bytes(int teams, bool cluster) {
    return kTeamMaxTeams * kTeamMaxStages * 8 + teams * (512 + (cluster ? kTeamXchBytes : 0));
}

// gamma / beta in shared memory, in planes: float4 number j = i / 4 of the
// array lies in plane j % NP at position j / NP, NP = V / 4 float4s per
// 16-byte group of data.  The lanes of a warp work on consecutive groups, so
// each of their reads covers consecutive float4s of one plane (in plain order
// they would be NP float4s apart: a 2- or 4-way bank conflict).  A plane has
// np float4s, one more than the array fills, so that the read past the last
// value of a shifted group (below) stays inside.
struct AffinePlanes {
    const float *p;  // shared memory, 16-byte aligned
    int np;
};
template <int NP>
__host__ __device__ constexpr int affine_np(int N) { return ((N + 3) / 4 + NP - 1) / NP + 1; }

// Where one row's groups find their values: group gi, starting at column
// i0 + gi * V of the array, reads float4s k = 0, 1, ... at a[k] + 16 gi (a
// group is NP float4s, so float4 k of every group lies in one plane).  i0 may
// lie anywhere: q = i0 % 4 values of float4 0 belong to the group before.
template <int NP>
struct AffineRow {
    uint32_t a[NP + 1];
    int q;
    __device__ __forceinline__ AffineRow(const AffinePlanes &p, int i0) : q(i0 & 3) {
        const int j0 = i0 >> 2;
#pragma unroll
        for (int k = 0; k <= NP; ++k)
            a[k] = smem_addr(p.p) + 16u * static_cast<uint32_t>((j0 + k) % NP * p.np + (j0 + k) / NP);
    }
};
// SV values from element hv of group gi on, Q = r.q known at compile time: the float4s that cover them, whole
// (one more than SV / 4 where Q > 0), `array` bytes after the first array (beta after gamma).
template <int Q, int NP, int SV>
__device__ __forceinline__ void affine_load(const AffineRow<NP> &r, uint32_t array, int gi, int hv, float (&v)[SV]) {
    constexpr int n = SV / 4 + (Q > 0 ? 1 : 0);
    float f[4 * n];
#pragma unroll
    for (int k = 0; k < n; ++k)
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(f[4 * k]), "=f"(f[4 * k + 1]), "=f"(f[4 * k + 2]), "=f"(f[4 * k + 3])
                     : "r"(r.a[hv / 4 + k] + array + 16u * static_cast<uint32_t>(gi)));
#pragma unroll
    for (int j = 0; j < SV; ++j) v[j] = f[j + Q];
}

template <int NP>
__device__ __forceinline__ void planes_fill(float *dst, int np, const float *src, float dflt, int N, int first, int step) {
    for (int i = first; i < N; i += step) {
        const int j = i >> 2;
        dst[((j % NP) * np + j / NP) * 4 + (i & 3)] = src ? __ldg(src + i) : dflt;
    }
}

// SV floats from i0 on.  i0 may lie anywhere (rows off the 16-byte grid start
// at any column): the vectors that cover the values are read whole and shifted
// (SV / 4 + 1 reads instead of SV).
template <int NP, int SV>
__device__ __forceinline__ void affine_shift(const AffinePlanes &a, int i0, float (&v)[SV]) {
    const int q = i0 & 3, j0 = i0 >> 2;
    auto ld = [&](int k, float *f) {
        const int j = j0 + k;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(f[0]), "=f"(f[1]), "=f"(f[2]), "=f"(f[3])
                     : "r"(smem_addr(a.p) + 16u * static_cast<uint32_t>((j % NP) * a.np + j / NP)));
    };
    if (q == 0) {
#pragma unroll
        for (int k = 0; k < SV / 4; ++k) ld(k, v + 4 * k);
        return;
    }
    float f[SV + 4];
#pragma unroll
    for (int k = 0; k < SV / 4 + 1; ++k) ld(k, f + 4 * k);
    const bool q1 = (q & 1) != 0, q2 = (q & 2) != 0;
#pragma unroll
    for (int k = 0; k < SV + 2; ++k) f[k] = q1 ? f[k + 1] : f[k];
#pragma unroll
    for (int k = 0; k < SV; ++k) v[k] = q2 ? f[k + 2] : f[k];
}

// gamma and, with TWO, beta of part of a group (b: beta's planes), the row's phase q tested here.  BF16 rows
// (NP = 2) have one copy of the reads per phase: the selects of affine_shift cost them 5 of some 30 instructions
// per element (16384 x 4095 LayerNorm 79 -> 73 us); FP32 and FP8 rows measure better with the selects (4096 x
// 6001 FP32 LayerNorm 50 against 55, where the copies spill).
template <bool GRID, bool TWO, int NP, int SV>
__device__ __forceinline__ void affine_pair(const AffineRow<NP> &r, const AffinePlanes &pg, const AffinePlanes &pb,
                                            int i0, int gi, int hv, float (&g)[SV], float (&b)[SV]) {
    const uint32_t at = TWO ? smem_addr(pb.p) - smem_addr(pg.p) : 0u;
    if (GRID || (NP == 2 && r.q == 0)) {
        affine_load<0>(r, 0u, gi, hv, g);
        if constexpr (TWO) affine_load<0>(r, at, gi, hv, b);
    } else if constexpr (NP != 2) {
        affine_shift<NP>(pg, i0, g);
        if constexpr (TWO) affine_shift<NP>(pb, i0, b);
    } else if (r.q == 1) {
        affine_load<1>(r, 0u, gi, hv, g);
        if constexpr (TWO) affine_load<1>(r, at, gi, hv, b);
    } else if (r.q == 2) {
        affine_load<2>(r, 0u, gi, hv, g);
        if constexpr (TWO) affine_load<2>(r, at, gi, hv, b);
    } else {
        affine_load<3>(r, 0u, gi, hv, g);
        if constexpr (TWO) affine_load<3>(r, at, gi, hv, b);
    }
}

// All-reduce over the T threads of a team (T > 32: through red, one float per
// warp, and named barrier `bar`).  Every warp merges the warps' values with
// the same shuffle tree, so every thread returns the same value.
template <bool MAX>
__device__ __forceinline__ float team_reduce(float v, float *red, int bar, int T) {
    v = MAX ? warp_max_redux(v) : warp_sum(v);
    if (T == 32) return v;
    const int lane = threadIdx.x & 31, nw = T >> 5;
    if (lane == 0) red[threadIdx.x >> 5] = v;
    named_bar_sync(bar, T);
    const float t = lane < nw ? red[lane] : (MAX ? -INFINITY : 0.0f);
    return MAX ? warp_max_redux(t) : warp_sum(t);
}

// Elements hv .. hv + SV - 1 of one 16-byte group (E4M3 groups are worked on in two halves of 8).
template <int TIN, int SV>
__device__ __forceinline__ void decode_part(const uint4 &w, int hv, float scale, float (&f)[SV]) {
    if constexpr (SV == Fmt<TIN>::V) {
        decode_group<TIN>(w, f, scale);
    } else {
        const uint32_t u[2] = {hv == 0 ? w.x : w.z, hv == 0 ? w.y : w.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const __half2_raw hr = __nv_cvt_fp8x2_to_halfraw2(
                static_cast<__nv_fp8x2_storage_t>((u[k >> 1] >> (16 * (k & 1))) & 0xFFFFu), __NV_E4M3);
            const float2 ff = __fmul2_rn(__half22float2(*reinterpret_cast<const __half2 *>(&hr)),
                                         make_float2(scale, scale));
            f[2 * k] = ff.x;
            f[2 * k + 1] = ff.y;
        }
    }
}

// Running maximum over the elements of a group (|.| with ABS), in the elements' own format: FP32 pairs, packed
// BF16 pairs, or E4M3 codes as packed halves (E4M3 is a subset of FP16).  Maxima are exact in any of them, and
// NaNs are passed over as fmaxf does.
template <int TIN, bool ABS>
struct GroupMax {
    using T2 = std::conditional_t<TIN == DT_F32, float2, std::conditional_t<TIN == DT_BF16, __nv_bfloat162, __half2>>;
    T2 m;
    __device__ __forceinline__ GroupMax() {
        if constexpr (TIN == DT_F32) m = make_float2(-INFINITY, -INFINITY);
        else if constexpr (TIN == DT_BF16) m = __bfloat162bfloat162(__ushort_as_bfloat16(0xFF80u));
        else m = __half2half2(__ushort_as_half(0xFC00u));
    }
    __device__ __forceinline__ void add(const uint4 &w) {
        const uint32_t u[4] = {w.x, w.y, w.z, w.w};
        if constexpr (TIN == DT_F32) {
#pragma unroll
            for (int k = 0; k < 4; k += 2) {
                const float x = __uint_as_float(u[k]), y = __uint_as_float(u[k + 1]);
                m.x = fmaxf(m.x, ABS ? fabsf(x) : x);
                m.y = fmaxf(m.y, ABS ? fabsf(y) : y);
            }
        } else if constexpr (TIN == DT_BF16) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t v = ABS ? u[k] & 0x7FFF7FFFu : u[k];
                m = __hmax2(m, *reinterpret_cast<const __nv_bfloat162 *>(&v));
            }
        } else {
            m = __hmax2(m, e4m3_group_hmax(w));
        }
    }
    __device__ __forceinline__ float value() const {
        if constexpr (TIN == DT_F32) return fmaxf(m.x, m.y);
        else return fmaxf(__low2float(m), __high2float(m));
    }
};

// The exponents (x - m) log2 e + c of part of a group, two per packed op (E4M3: x = a q from the sign-folded
// codes, the difference a q - m rounded once).
template <int TIN, int SV>
__device__ __forceinline__ void exp_args(const uint4 &w, int hv, float a, float m, float c, float (&t)[SV]) {
    float f[SV];
    decode_part<TIN>(w, hv, 1.0f, f);
#pragma unroll
    for (int j = 0; j < SV; j += 2) {
        const float2 x = make_float2(f[j], f[j + 1]);
        const float2 d = TIN == DT_E4M3 ? __ffma2_rn(x, make_float2(a, a), make_float2(-m, -m))
                                        : __fadd2_rn(x, make_float2(-m, -m));
        const float2 r = __ffma2_rn(d, make_float2(kLog2e, kLog2e), make_float2(c, c));
        t[j] = r.x;
        t[j + 1] = r.y;
    }
}

// GRID: every row of both tensors starts on the 16-byte grid and ends on it
// (no head or tail elements, one geometry for all rows); otherwise each row is
// cut on the grid of its own address.  AFF: gamma / beta (ones / zeros where
// null) in shared memory; otherwise read through L1.  TR: with the stamps of
// credit_set_trace (kernels of their own: in the others the test for a buffer
// costs up to 3%, 4096 x 30001 BF16 LayerNorm 150 us against 146).
template <int OP, int TIN, int TOUT, bool GRID, bool AFF, bool CL, bool TR = false>
__global__ void __launch_bounds__(kTeamMaxThreads, 1) k_row_team(const RowArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int isz = Fmt<TIN>::size, V = Fmt<TIN>::V, osz = Fmt<TOUT>::size, NP = V / 4;
    constexpr int SV = V < 8 ? V : 8;
    constexpr bool kNormOp = OP == OP_LN || OP == OP_RMS, kSm = OP == OP_SOFTMAX || OP == OP_LSE;
    constexpr bool kFp8Stage = TOUT == DT_E4M3 && kNormOp;
    // exponentials of FP32 / BF16 softmax outputs are raised by 2^24 (exp_sub's lift: subnormal results)
    constexpr bool kLift = OP == OP_SOFTMAX && TOUT != DT_E4M3;
    constexpr int vec_bytes = V * osz < 16 ? V * osz : 16;

    const int T = blockDim.x, t = threadIdx.x, team = threadIdx.y, teams = blockDim.y, S = a.ring;
    const int N = static_cast<int>(a.cols);
    const int P = CL ? static_cast<int>(cluster_nctarank()) : 1, c = CL ? static_cast<int>(cluster_ctarank()) : 0;
    const int lp = CL ? 31 - __clz(P) : 0;           // P is a power of two
    const int gmax = (N / V + P - 1) >> lp;          // groups of a row's slice are at most this many
    const int cb = CL ? ((N / V - 1) * c >> lp) * V : 0;  // no slice of this CTA starts before this column
    const int cn = CL ? min(N - cb, gmax * V + 3 * V) : N;  // columns of gamma / beta any slice needs
    uint64_t *full = reinterpret_cast<uint64_t *>(smem) + team * kTeamMaxStages;
    float *red = reinterpret_cast<float *>(smem + kTeamMaxTeams * kTeamMaxStages * 8) + team * 128;
    const bool has_g = kNormOp && a.gamma != nullptr, has_b = OP == OP_LN && a.beta != nullptr;
    const int np = affine_np<NP>(cn);
    float *gsm = reinterpret_cast<float *>(smem + team_ctrl_bytes(teams, CL));
    float *bsm = gsm + (AFF ? NP * np * 4 : 0);
    const AffinePlanes gp{gsm, np}, bp{bsm, np};
    unsigned char *stages = reinterpret_cast<unsigned char *>(bsm + (AFF && OP == OP_LN ? NP * np * 4 : 0)) +
                            static_cast<size_t>(team) * S * gmax * 16;
    // cluster exchange (CL): slots [stage][row parity][16 sources][2 floats] and mbarriers [stage][parity] of the team
    unsigned char *xch = smem + team_ctrl_bytes(teams, false) + team * kTeamXchBytes;
    uint64_t *xbar = reinterpret_cast<uint64_t *>(xch + 512);
    const long long stride = static_cast<long long>(gridDim.x >> lp) * teams;
    const long long row_first = static_cast<long long>(blockIdx.x >> lp) * teams + team;
    const float inv_n = 1.0f / static_cast<float>(N);

    // a row's head, groups and tail, and the groups lo .. lo + n - 1 of this CTA's slice
    struct Geo {
        int h0, G, t0, lo, n;
    };
    auto geo = [&](const unsigned char *row) {
        if constexpr (GRID) return Geo{0, gmax, 0, 0, gmax};
        Geo g;
        g.h0 = min(static_cast<int>((0u - static_cast<uint32_t>(reinterpret_cast<uintptr_t>(row))) & 15u) / isz, N);
        g.G = (N - g.h0) / V;
        g.t0 = (N - g.h0) % V;
        g.lo = CL ? g.G * c >> lp : 0;
        g.n = CL ? (g.G * (c + 1) >> lp) - g.lo : g.G;
        return g;
    };
    auto in_row = [&](long long row) { return a.in + row * a.ld_in * isz; };
    // thread 0: request a row's groups into stage slot
    auto issue = [&](long long row, int slot) {
        const unsigned char *p = in_row(row);
        const Geo g = geo(p);
        if (!GRID && g.n == 0) return;
        const uint32_t bytes = static_cast<uint32_t>(g.n) * 16u;
        unsigned char *dst = stages + static_cast<uint32_t>(slot) * (gmax * 16u);
        const unsigned char *src = p + g.h0 * isz + g.lo * 16;
        mbar_arrive_expect_tx(&full[slot], bytes);
        for (uint32_t o = 0; o < bytes; o += kMaxChunkBytes)
            bulk_g2s(dst + o, src + o, min(bytes - o, static_cast<uint32_t>(kMaxChunkBytes)), &full[slot]);
    };
    // edge elements, one per thread (fewer than 16 of each; a team has at least 32 threads)
    auto edge_index = [&](const Geo &g) -> int {
        if constexpr (GRID) return -1;
        if ((!CL || c == 0) && t < g.h0) return t;
        return (!CL || c == P - 1) && T - 1 - t < g.t0 ? g.h0 + g.G * V + (T - 1 - t) : -1;
    };

    // the first rows are requested before anything else; only this thread uses the barriers before the block's
    // barrier below
    if (t == 0) {
        for (int k = 0; k < S; ++k) mbar_init(&full[k], 1);
        if constexpr (CL) {
            for (int k = 0; k < 4; ++k) mbar_init(&xbar[k], 1);
        }
        fence_mbar_init();
        for (int k = 0; k < S; ++k)
            if (row_first + k * stride < a.rows) issue(row_first + k * stride, k);
    }
    if constexpr (AFF) {  // gamma / beta, once for every row of this SM
        planes_fill<NP>(gsm, np, has_g ? a.gamma + cb : nullptr, 1.0f, cn, team * T + t, T * teams);
        if constexpr (OP == OP_LN)
            planes_fill<NP>(bsm, np, has_b ? a.beta + cb : nullptr, 0.0f, cn, team * T + t, T * teams);
    }
    __syncthreads();
    if constexpr (CL) {  // every peer's exchange barriers exist before the first push
        cluster_arrive_release();
        cluster_wait_acquire();
    }
    // Push all-gather of two floats per CTA among the cluster's teams of one number (Eq. 5): each CTA's partial
    // goes to slot c of every CTA, its own included.  Slots and barriers alternate with the row: a CTA pushes into
    // a parity again only after its exchange of the row between, which needed a push that each peer made after it
    // had read this parity's slots.  Lane q < P returns CTA q's partial.
    auto exchange = [&](int stage, float p0, float p1, uint32_t k) -> float2 {
        const uint32_t par = k & 1u;
        float *slots = reinterpret_cast<float *>(xch) + (stage * 2 + par) * 32;
        uint64_t *bar = &xbar[stage * 2 + par];
        if (t < P) {
            fence_release_smem_cluster();
            st_async_v2f32(mapa_shared(smem_addr(slots + 2 * c), t), p0, p1, mapa_shared(smem_addr(bar), t));
        }
        if (t == 0) mbar_arrive_expect_tx(bar, static_cast<uint32_t>(P) * 8u);
        mbar_wait_bounded_cluster(bar, (k >> 1) & 1u, a.err);
        const int q = t & 31;
        return q < P ? make_float2(slots[2 * q], slots[2 * q + 1]) : make_float2(0.0f, 0.0f);
    };

    float rawn = 0.0f, scn = 1.0f;  // the next row's edge element (unscaled) and input scale
    auto fetch_next = [&](long long row) {
        if constexpr (!GRID) {
            const unsigned char *p = in_row(row);
            const int i = edge_index(geo(p));
            if (i >= 0) rawn = decode_one<TIN>(p + i * isz, 1.0f);
        }
        if constexpr (TIN == DT_E4M3) scn = a.in_scale[row];
    };
    if (row_first < a.rows) fetch_next(row_first);

    unsigned char *out_p = a.out + row_first * a.ld_out * osz;
    const long long out_step = stride * a.ld_out * osz;
    int slot = 0;
    uint32_t lap = 0;
    bool odd = false;  // row parity: reductions that are a row's only one alternate between two arrays
    uint32_t it = 0;   // rows done (CL)
    auto stamp = [&](int field) {
        if constexpr (TR) {
            if (team == 0 && t == 0) trace_stamp(a, static_cast<int>(lap) * S + slot, field);
        }
    };
    for (long long row = row_first; row < a.rows; row += stride, out_p += out_step, odd = !odd) {
        stamp(0);
        const Geo g = geo(GRID ? nullptr : in_row(row));
        const int ie = edge_index(g);
        const bool edge = !GRID && ie >= 0;
        const float in_sc = scn, xe = rawn * (TIN == DT_E4M3 ? in_sc : 1.0f);
        if (row + stride < a.rows) fetch_next(row + stride);
        const unsigned char *stage = stages + static_cast<uint32_t>(slot) * (gmax * 16u);

        // ---- the row in shared memory
        if (GRID || g.n > 0) mbar_wait_bounded(&full[slot], lap & 1u, a.err);
        stamp(5);
        const uint32_t neg = TIN == DT_E4M3 && kSm ? e4m3_sign_mask(in_sc) : 0u;
        auto lds = [&](int gi) {
            const uint4 x = *reinterpret_cast<const uint4 *>(stage + 16 * gi);
            if constexpr (TIN == DT_E4M3 && kSm) return e4m3_fold_sign(x, neg);
            else return x;
        };
        auto each = [&](auto &&fn) {  // this thread's groups
#pragma unroll 1
            for (int gi = t; gi < g.n; gi += T) fn(gi, lds(gi));
        };
        float K = 0.0f;
        if constexpr (OP == OP_LN) K = decode_one<TIN>(GRID || g.n > 0 ? stage : in_row(row), in_sc);
        const float a1 = fabsf(in_sc);
        // after the row's first reduction: every thread is done with the previous row, whose stage takes its next
        // row (one stage: at the end of the row instead)
        auto refill = [&]() {
            if (T == 32) __syncwarp();
            const long long nr = row + (S - 1) * stride;
            if (t == 0 && S > 1 && row != row_first && nr < a.rows) {
                fence_proxy_async_smem();
                issue(nr, (slot ? slot : S) - 1);
            }
        };

        // ---- statistics
        Stats st;
        st.b = 0.0f;
        if constexpr (kSm) {
            GroupMax<TIN, false> gm;
            each([&](int, const uint4 &x) { gm.add(x); });
            float m = gm.value();
            if (TIN == DT_E4M3 && m != -INFINITY) m *= a1;
            if (edge) m = fmaxf(m, xe);
            st.a = team_reduce<true>(m, red, team, T);
            refill();
            const float mz = st.a == -INFINITY ? 0.0f : st.a;  // a row of -inf: every term 0
            constexpr float lift = kLift ? kExpLift : 0.0f;
            float sum = 0.0f;
            each([&](int gi, const uint4 &x) {
#pragma unroll
                for (int hv = 0; hv < V; hv += SV) {
                    float e[SV];
                    exp_args<TIN>(x, hv, a1, mz, lift, e);
#pragma unroll
                    for (int j = 0; j < SV; ++j) e[j] = ex2_ftz(e[j]);
                    sum += sum_tree<SV>(e);
                }
            });
            if (edge) sum += ex2_ftz(fmaf(xe - mz, kLog2e, lift));
            st.b = team_reduce<false>(sum, red + 32, team, T);
            if constexpr (CL) {  // (max, sum) of every slice about the row's maximum
                const float2 p = exchange(0, st.a, st.b, it);
                const bool mine = (t & 31) < P;
                st.a = warp_max_redux(mine ? p.x : -INFINITY);
                // an all -inf slice has the sum 0 about 0; a NaN sum stays NaN
                st.b = warp_sum(mine ? (p.x == -INFINITY ? p.y : p.y * ex2_ftz((p.x - st.a) * kLog2e)) : 0.0f);
            }
        } else if constexpr (OP == OP_LN) {
            float2 s2 = make_float2(0.0f, 0.0f);
            each([&](int gi, const uint4 &x) {
#pragma unroll
                for (int hv = 0; hv < V; hv += SV) {
                    float f[SV];
                    decode_part<TIN>(x, hv, in_sc, f);
#pragma unroll
                    for (int j = 0; j < SV; j += 2)
                        s2 = __fadd2_rn(s2, __fadd2_rn(make_float2(f[j], f[j + 1]), make_float2(-K, -K)));
                }
            });
            float s1 = s2.x + s2.y;
            if (edge) s1 += xe - K;
            s1 = team_reduce<false>(s1, red, team, T);
            refill();
            // the slice's count, mean and squared deviations (the row's where it is not split)
            const float n_c = CL ? static_cast<float>(g.n * V + (c == 0 ? g.h0 : 0) + (c == P - 1 ? g.t0 : 0)) : 1.0f;
            st.a = CL ? K + s1 / n_c : fmaf(s1, inv_n, K);
            float2 q2 = make_float2(0.0f, 0.0f);
            each([&](int gi, const uint4 &x) {
#pragma unroll
                for (int hv = 0; hv < V; hv += SV) {
                    float f[SV];
                    decode_part<TIN>(x, hv, in_sc, f);
#pragma unroll
                    for (int j = 0; j < SV; j += 2) {
                        const float2 d = __fadd2_rn(make_float2(f[j], f[j + 1]), make_float2(-st.a, -st.a));
                        q2 = __ffma2_rn(d, d, q2);
                    }
                }
            });
            float m2 = q2.x + q2.y;
            if (edge) m2 = fmaf(xe - st.a, xe - st.a, m2);
            m2 = team_reduce<false>(m2, red + 32, team, T);
            if constexpr (CL) {
                // mean = m_0 + sum n_q (m_q - m_0) / N, M2 = sum (M2_q + n_q (m_q - mean)^2)
                const float2 p = exchange(0, st.a, m2, it);
                const int q = t & 31;
                const float n_q = q < P ? static_cast<float>(((g.G * (q + 1) >> lp) - (g.G * q >> lp)) * V +
                                                             (q == 0 ? g.h0 : 0) + (q == P - 1 ? g.t0 : 0))
                                        : 0.0f;
                const float m_0 = __shfl_sync(0xffffffffu, p.x, 0);
                st.a = fmaf(warp_sum(n_q * (p.x - m_0)), inv_n, m_0);
                const float d = p.x - st.a;
                m2 = warp_sum(fmaf(n_q * d, d, p.y));
            }
            st.b = rsqrtf(fmaf(m2, inv_n, a.eps));
        } else if constexpr (OP == OP_RMS) {
            float2 q2 = make_float2(0.0f, 0.0f);
            each([&](int gi, const uint4 &x) {
#pragma unroll
                for (int hv = 0; hv < V; hv += SV) {
                    float f[SV];
                    decode_part<TIN>(x, hv, in_sc, f);
#pragma unroll
                    for (int j = 0; j < SV; j += 2) {
                        const float2 d = make_float2(f[j], f[j + 1]);
                        q2 = __ffma2_rn(d, d, q2);
                    }
                }
            });
            float ss = q2.x + q2.y;
            if (edge) ss = fmaf(xe, xe, ss);
            ss = team_reduce<false>(ss, red + (odd ? 32 : 0), team, T);
            refill();
            if constexpr (CL) ss = warp_sum(exchange(0, ss, 0.0f, it).x);
            st.a = rsqrtf(fmaf(ss, inv_n, a.eps));
        } else {
            GroupMax<TIN, true> gm;
            each([&](int, const uint4 &x) { gm.add(x); });
            float am = fmaxf(gm.value(), 0.0f);
            if (edge) am = fmaxf(am, fabsf(xe));
            am = team_reduce<true>(am, red + (odd ? 32 : 0), team, T);
            refill();
            if constexpr (CL) am = warp_max_redux(exchange(0, am, 0.0f, it).x);
            const float p[2] = {am, 0.0f};
            st = combine_partials<OP>(p, 2, 1, RowSlice{}, V, N, a.eps);
        }

        stamp(3);
        // ---- outputs
        if constexpr (OP == OP_LSE) {
            if (c == 0 && t == 0) reinterpret_cast<float *>(a.out)[row] = st.a + logf(st.b);
        } else {
            // the norms' outputs hv .. hv + SV - 1 of group u, before the FP8 scaling
            const AffineRow<NP> ar(gp, GRID || !AFF ? 0 : g.h0 + g.lo * V - cb);
            auto norm_part = [&](int gi, const uint4 &x, int hv, float (&y)[SV]) {
                float gg[SV], bb[SV];
                decode_part<TIN>(x, hv, in_sc, y);
                if constexpr (AFF) {
                    affine_pair<GRID, OP == OP_LN>(ar, gp, bp, g.h0 + (g.lo + gi) * V + hv - cb, gi, hv, gg, bb);
                } else {
                    ldg_shift<SV>(a.gamma, g.h0 + (g.lo + gi) * V + hv, N, 1.0f, gg);
                    if constexpr (OP == OP_LN) ldg_shift<SV>(a.beta, g.h0 + (g.lo + gi) * V + hv, N, 0.0f, bb);
                }
#pragma unroll
                for (int j = 0; j < SV; j += 2) {  // norm_h, two elements per packed op
                    float2 v = make_float2(y[j], y[j + 1]);
                    const float2 gm = make_float2(gg[j], gg[j + 1]);
                    if constexpr (OP == OP_LN) {
                        v = __fmul2_rn(__fadd2_rn(v, make_float2(-st.a, -st.a)), make_float2(st.b, st.b));
                        v = __ffma2_rn(v, gm, make_float2(bb[j], bb[j + 1]));
                    } else {
                        v = __fmul2_rn(__fmul2_rn(v, make_float2(st.a, st.a)), gm);
                    }
                    y[j] = v.x;
                    y[j + 1] = v.y;
                }
            };
            auto norm_edge = [&]() -> float {
                return norm_h<OP>(xe, st, has_g ? a.gamma[ie] : 1.0f, has_b ? a.beta[ie] : 0.0f);
            };
            float mul = 1.0f, cL = 0.0f;
            if constexpr (kFp8Stage) {
                float am = 0.0f;
                each([&](int gi, const uint4 &x) {
#pragma unroll
                    for (int hv = 0; hv < V; hv += SV) {
                        float y[SV];
                        norm_part(gi, x, hv, y);
#pragma unroll
                        for (int j = 0; j < SV; ++j) am = fmaxf(am, fabsf(y[j]));
                    }
                });
                if (edge) am = fmaxf(am, fabsf(norm_edge()));
                am = team_reduce<true>(am, red + 64 + (odd ? 32 : 0), team, T);
                if constexpr (CL) am = warp_max_redux(exchange(1, am, 0.0f, it).x);
                mul = am > 0.0f ? 448.0f / am : 1.0f;
                if (c == 0 && t == 0) a.out_scale[row] = am > 0.0f ? am / 448.0f : 1.0f;
            } else if constexpr (OP == OP_SOFTMAX) {
                mul = TOUT == DT_E4M3 ? 448.0f : 1.0f / st.b;
                cL = TOUT == DT_E4M3 ? 8.807354922057604f /* log2 448 */ : kExpLift - log2f(st.b);
                if constexpr (TOUT == DT_E4M3) {
                    if (c == 0 && t == 0) a.out_scale[row] = (1.0f / st.b) * (1.0f / 448.0f);
                }
            } else if constexpr (OP == OP_Q8) {
                if (c == 0 && t == 0) a.out_scale[row] = st.a;
            }
            unsigned char *out_body = out_p + (g.h0 + g.lo * V) * osz;
            const bool out_vec = GRID || (reinterpret_cast<uintptr_t>(out_body) % vec_bytes) == 0;
            each([&](int gi, const uint4 &x) {
                uint32_t ow[V * osz / 4];
#pragma unroll
                for (int hv = 0; hv < V; hv += SV) {
                    float y[SV];
                    if constexpr (OP == OP_SOFTMAX) {
                        // the term again, lifted as exp_sub's (E4M3 codes need no lift)
                        exp_args<TIN>(x, hv, a1, st.a, TOUT == DT_E4M3 ? cL : cL + kExpLift, y);
#pragma unroll
                        for (int j = 0; j < SV; ++j) y[j] = TOUT == DT_E4M3 ? ex2_ftz(y[j]) : ex2_ftz(y[j]) * kExpDrop;
                    } else if constexpr (OP == OP_Q8) {
                        float f[SV];
                        decode_part<TIN>(x, hv, 1.0f, f);
                        q8_codes<SV>(f, st.a, st.b, y);
                    } else {
                        norm_part(gi, x, hv, y);
                        if constexpr (kFp8Stage) {
#pragma unroll
                            for (int j = 0; j < SV; ++j) y[j] *= mul;
                        }
                    }
                    uint32_t pw[SV * osz / 4];
                    pack_words<TOUT, SV>(y, pw);
#pragma unroll
                    for (int j = 0; j < SV * osz / 4; ++j) ow[hv * osz / 4 + j] = pw[j];
                }
                store_words<TOUT, V>(out_body + gi * (V * osz), ow, out_vec);
            });
            if (edge) {
                float y;
                if constexpr (OP == OP_SOFTMAX) {
                    y = TOUT == DT_E4M3 ? ex2_ftz(fmaf(xe - st.a, kLog2e, cL)) : exp_sub(xe, st.a, cL);
                } else if constexpr (OP == OP_Q8) {
                    y = q8_code(xe, st.a, st.b);
                } else {
                    y = norm_edge() * mul;
                }
                store_one<TOUT>(out_p + ie * osz, y);
            }
        }
        stamp(4);
        if (S == 1 && row + stride < a.rows) {
            if (T == 32) __syncwarp();
            else named_bar_sync(team, T);
            if (t == 0) {
                fence_proxy_async_smem();
                issue(row + stride, 0);
            }
        }
        if (++slot == S) {
            slot = 0;
            ++lap;
        }
        if constexpr (CL) ++it;
    }
    if constexpr (CL) {  // no CTA leaves while a peer may still push into it
        cluster_arrive_release();
        cluster_wait_acquire();
    }
}

}  // namespace credit
