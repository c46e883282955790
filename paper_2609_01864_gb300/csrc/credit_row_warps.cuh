// credit_row_warps.cuh -- rows over warps: k_row_warps, for ragged batches
// (credit_ragged.cu) and for rows of one width (credit_warps.cu).
//
// Persistent CTAs, 16 warps to an SM.  A row takes u = 1, 2, 4, ... warps, the
// fewest whose segments fit their buffers of 14 KiB: of one CTA, or u / P of
// each CTA of a cluster.  A warp loads its own segments, two turns ahead where
// two fit, and has nothing to wait for but its own copy and one reduction per
// row: no barrier of the CTA per chunk and none of the cluster per item, and
// the rows of an SM are at different stages, so that its loads, arithmetic and
// stores overlap.  The row in shared memory can be looked at twice: the
// maximum first, then the sum about it.
// Rows are sorted widest first; the classes of one u follow each other, and
// the CTA's warps meet between them.  Within a class partials lie in two sets
// by parity: a warp writes the next but one only when every member of its
// group has read this one.  The exchange barriers and slots of a group are its
// first warp's; groups only get smaller while rows span CTAs, so a warp's new
// first one has either been its own before or no one's.  Named barriers are
// numbered by the first warp as well.
// k_ragged, with its online maxima, chunk and item barriers, took 20
// instructions per element and 59% of the issue slots.  Measured (GB300,
// k_ragged -> this): 20000 BF16 rows of 1K to 1M columns 2640 us -> 2180 (the
// copy rate's 1765), 8000 of 8K to 40K 167 -> 114 (94), 4000 of 1K to 4K 33 ->
// 12, 3000 FP32 rows of 8K to 200K 295 -> 236 (210), 64 of 16K to 500K 29 ->
// 22.  Segments of all 14 KiB (half as many warps per row) are worth more than
// a second one in flight (20000 rows 2670 -> 2260), four groups per loop step
// 7% over one; 32 warps of 7 KiB or 8 of 28 KiB are slower (8000 rows 128 and
// 135 against 117).
#pragma once

#include "credit_row_team.cuh"

namespace credit {

constexpr int kWWarps = 16;  // warps of an SM: one CTA, or two of half as many
constexpr int kWHalf = 440;  // 16-byte groups of half a warp's buffer
// shared memory of a CTA of W warps: mbarriers (full [W][2], exchange [W][2], meet), partials [2][W], slots
// [W][2][16 CTAs], buffers
__host__ __device__ constexpr int warps_ctrl(int W) { return (W * 32 + 16 + W * 16 + W * 256 + 127) / 128 * 128; }
__host__ __device__ constexpr int warps_smem(int W) { return warps_ctrl(W) + W * 2 * kWHalf * 16; }
constexpr int kWClasses = 10;

struct WClass {
    int lu, lw;       // 2^lu warps per row, over 2^lw CTAs (one, or all the cluster's)
    int k_end;        // turns of a warp up to the class's end
    int row0, row_end;
};
// A row of a ragged batch (element offsets from the bases).
struct alignas(16) RRow {
    long long in_off, out_off, cols;
    int op;
    int pad;
};
struct WarpArgs {
    const unsigned char *in;
    unsigned char *out;
    const RRow *rows;
    int n_classes;
    WClass cls[kWClasses];
    float eps;
    unsigned *err;
    long long ld_in, ld_out;  // rows of one width and op: strides (elements), columns, int8 scales
    int cols;
    float *out_scale;
    unsigned long long *trace;  // as in RowArgs (TR)
    int trace_rows;
};
constexpr int OP_ROWS = -1;  // k_row_warps: the op is the row's

// Running minimum over the elements of a group, as GroupMax.
template <int TIN>
struct GroupMin {
    std::conditional_t<TIN == DT_F32, float2, __nv_bfloat162> m;
    __device__ __forceinline__ GroupMin() {
        if constexpr (TIN == DT_F32) m = make_float2(INFINITY, INFINITY);
        else m = __bfloat162bfloat162(__ushort_as_bfloat16(0x7F80u));
    }
    __device__ __forceinline__ void add(const uint4 &w) {
        const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if constexpr (TIN == DT_F32) {
                if (k & 1) m.y = fminf(m.y, __uint_as_float(u[k]));
                else m.x = fminf(m.x, __uint_as_float(u[k]));
            } else {
                m = __hmin2(m, *reinterpret_cast<const __nv_bfloat162 *>(&u[k]));
            }
        }
    }
    __device__ __forceinline__ float value() const {
        if constexpr (TIN == DT_F32) return fminf(m.x, m.y);
        else return fminf(__low2float(m), __high2float(m));
    }
};

// 2^t b, t <= 0, the exponential never flushed: scaled by 2^64 where it would be subnormal.
__device__ __forceinline__ float exp_scaled(float t, float b) {
    const bool low = t < -100.0f;
    return ex2_ftz(low ? t + 64.0f : t) * (low ? b * 0x1p-64f : b);
}

// The outputs exp(x - st.a) st.b (softmax), x st.b (RMSNorm) or the int8 codes of a warp's n groups.
// LOW: some exponentials are below the normal numbers (or the stores are not vectors; one loop for both).
template <int OP, int TIN, bool VEC, bool LOW>
__device__ __forceinline__ void write_segment(const unsigned char *d, unsigned char *o, int n, int lane, const Stats &st) {
    constexpr int V = Fmt<TIN>::V;
    constexpr bool SM = OP == OP_SOFTMAX;
#pragma unroll 4
    for (int g = lane; g < n; g += 32) {
        float f[V];
        decode_group<TIN>(*reinterpret_cast<const uint4 *>(d + 16 * g), f, 1.0f);
        if constexpr (OP == OP_Q8) {
            float y[V];
            q8_codes<V>(f, st.a, st.b, y);
            store_group<DT_I8, V>(o + V * g, y, VEC);
            continue;
        }
#pragma unroll
        for (int j = 0; j < V; j += 2) {
            const float2 x = make_float2(f[j], f[j + 1]);
            const float2 e = SM ? __fmul2_rn(__fadd2_rn(x, make_float2(-st.a, -st.a)), make_float2(kLog2e, kLog2e)) : x;
            f[j] = e.x;
            f[j + 1] = e.y;
        }
        if constexpr (SM && !LOW) {
#pragma unroll
            for (int j = 0; j < V; ++j) f[j] = ex2_ftz(f[j]);
        } else if constexpr (SM) {
#pragma unroll
            for (int j = 0; j < V; ++j) f[j] = exp_scaled(f[j], st.b);
        }
#pragma unroll
        for (int j = 0; j < V && !(SM && LOW); j += 2) {
            const float2 e = __fmul2_rn(make_float2(f[j], f[j + 1]), make_float2(st.b, st.b));
            f[j] = e.x;
            f[j + 1] = e.y;
        }
        store_group<TIN, V>(o + 16 * g, f, VEC);
    }
}

template <int OP, int TIN, int W, bool TR = false>  // TR: with the stamps of credit_set_trace
__global__ void __launch_bounds__(32 * W, kWWarps / W) k_row_warps(const WarpArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int isz = Fmt<TIN>::size, V = Fmt<TIN>::V, osz = OP == OP_Q8 ? 1 : isz;
    constexpr bool AM = OP == OP_Q8;  // the statistic is a maximum alone
    constexpr bool LO = OP == OP_SOFTMAX || OP == OP_ROWS;
    const int P = static_cast<int>(cluster_nctarank()), c = P > 1 ? static_cast<int>(cluster_ctarank()) : 0;
    const int ncl = gridDim.x / P, cl = blockIdx.x / P;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gw = c * W + warp;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem) + 2 * warp;     // of this warp's halves
    uint64_t *xbars = reinterpret_cast<uint64_t *>(smem + W * 16);      // exchange [first warp][parity]
    uint64_t *meet = reinterpret_cast<uint64_t *>(smem + W * 32);       // all warps, between classes
    float2 *red = reinterpret_cast<float2 *>(smem + W * 32 + 16);       // [parity][warp]
    float2 *slots = red + 2 * W;                                        // [first warp][parity][16 CTAs]
    unsigned char *buf = smem + warps_ctrl(W) + warp * (2 * kWHalf * 16);
    if (lane == 0) {
        mbar_init(&full[0], 1);
        mbar_init(&full[1], 1);
        mbar_init(&xbars[2 * warp], 1);
        mbar_init(&xbars[2 * warp + 1], 1);
        if (warp == 0) mbar_init(meet, W);
        fence_mbar_init();
    }
    __syncthreads();
    if (P > 1) {
        cluster_arrive_release();
        cluster_wait_acquire();
    }

    // this warp's rows, turn by turn
    struct Turn {
        int k, cls, k_end, lu, lw, n, row, row_end;  // n: groups of warps, the step from one turn's row to the next's
    };
    auto enter = [&](Turn &t) {  // the first turn of class t.cls
        const WClass &w = a.cls[t.cls];
        t.lu = w.lu;
        t.lw = w.lw;
        t.n = ncl * (P * W >> w.lu);
        const int g = ((w.lw ? warp : gw) >> (w.lu - w.lw)) * ncl + cl;
        // every other class deals its rows from the far end: the groups with one row more differ
        t.row = w.row0 + (t.cls & 1 ? t.n - 1 - g : g);
        t.row_end = w.row_end;
        t.k_end = w.k_end;
    };
    auto step = [&](Turn &t) {  // false past the last turn
        t.row += t.n;
        if (++t.k < t.k_end) return true;
        if (++t.cls == a.n_classes) return false;
        enter(t);
        return true;
    };
    struct Seg {  // the row cut on the 16-byte grid, and this warp's groups lo .. lo + n - 1
        int h0, G, t0, lo, n;
    };
    // number of this warp among a row's
    auto member = [&](int lu, int lw) { return (lw ? c << (lu - lw) : 0) + (warp & ((1 << (lu - lw)) - 1)); };
    auto row_at = [&](int r) {
        if constexpr (OP == OP_ROWS) return a.rows[r];
        else return RRow{r * a.ld_in, r * a.ld_out, a.cols, OP, 0};
    };
    auto segment = [&](const RRow &rw, int lu, int lw) {
        Seg s;
        const int N = static_cast<int>(rw.cols), m = member(lu, lw);
        const uint32_t at = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(a.in)) + static_cast<uint32_t>(rw.in_off) * isz;
        s.h0 = min(static_cast<int>((0u - at) & 15u) / isz, N);
        s.G = (N - s.h0) / V;
        s.t0 = (N - s.h0) % V;
        s.lo = s.G * m >> lu;  // G m < 2^18 2^9
        s.n = (s.G * (m + 1) >> lu) - s.lo;
        return s;
    };
    Turn next{};      // the next turn to load
    bool more = true;  // there is one
    int single = -1;  // the last turn whose segment takes both halves
    enter(next);
    // Loads after turn k is written: turn k + 1 and, where both segments fit a half, k + 2.
    auto load_ahead = [&](int k) {
        while (more && next.k <= k + 2) {
            if (next.row < next.row_end) {
                const RRow rw = row_at(next.row);
                const Seg s = segment(rw, next.lu, next.lw);
                if (next.k == k + 2 && (s.n > kWHalf || single == k + 1)) return;
                if (s.n > kWHalf) single = next.k;
                if (lane == 0 && s.n > 0) {
                    const int h = s.n > kWHalf ? 0 : next.k & 1;
                    const uint32_t bytes = static_cast<uint32_t>(s.n) * 16u;
                    fence_proxy_async_smem();
                    mbar_arrive_expect_tx(&full[h], bytes);
                    bulk_g2s_hint(buf + h * (kWHalf * 16), a.in + (rw.in_off + s.h0) * isz + s.lo * 16ll, bytes,
                                  &full[h], l2_evict_first_policy());
                }
            }
            more = step(next);
        }
    };
    // (maximum, sum about it), (unused, sum) or (maximum, unused) of the lanes below n
    auto merge = [&](bool sm, float2 v, int n) {
        if constexpr (AM) {
            v.x = warp_max_redux(lane < n ? v.x : 0.0f);
            return v;
        }
        if (sm) {
            const float m = warp_max_redux(lane < n ? v.x : -INFINITY);
            v.y = lane < n && v.x != m ? v.y * ex2_ftz((v.x - m) * kLog2e) : v.y;
            v.x = m;
        }
        v.y = warp_sum(lane < n ? v.y : 0.0f);
        return v;
    };

    load_ahead(-1);
    uint32_t phase = 0, reds = 0, xchs = 0, meets = 0;
    int was_first = 0;
    Turn turn{};
    enter(turn);
    auto stamp = [&](int field) {
        if constexpr (TR) {
            if (warp == 0 && lane == 0) trace_stamp(a, turn.k, field);
        }
    };
    for (int last = 0;;) {
        const int lu = turn.lu, lw = turn.lw, k = turn.k, wl = 1 << (lu - lw), first = warp & ~(wl - 1);
        if (turn.cls != last) {
            if (lane == 0) mbar_arrive(meet);
            mbar_wait_bounded(meet, meets++ & 1u, a.err);
            last = turn.cls;
            reds = 0;
            if (first != was_first) xchs = 0;  // barriers that no wider group has used
        }
        was_first = first;
        if (turn.row < turn.row_end) {
            stamp(0);
            const RRow rw = row_at(turn.row);
            const Seg s = segment(rw, lu, lw);
            const bool sm = OP == OP_ROWS ? rw.op == OP_SOFTMAX : true;  // a maximum (and a sum about it)
            const unsigned char *row = a.in + rw.in_off * isz;
            // edge elements, one per lane: the head's by the row's first warp, the tail's by its last
            const int m = member(lu, lw);
            const bool edges = (m == 0 && s.h0 > 0) || (m == (1 << lu) - 1 && s.t0 > 0);
            const int ie = m == 0 && lane < s.h0 ? lane
                           : m == (1 << lu) - 1 && 31 - lane < s.t0 ? s.h0 + s.G * V + (31 - lane) : -1;
            const float xe = ie >= 0 ? decode_one<TIN>(row + static_cast<long long>(ie) * isz, 1.0f) : 0.0f;
            const int h = s.n > kWHalf ? 0 : k & 1;
            const unsigned char *d = buf + h * (kWHalf * 16);
            if (s.n > 0) {
                mbar_wait_bounded(&full[h], phase >> h & 1u, a.err);
                phase ^= 1u << h;
            }
            stamp(5);
            float2 v = make_float2(-INFINITY, 0.0f);
            float lo = 0.0f;  // the segment's smallest element (softmax)
            float2 s2 = make_float2(0.0f, 0.0f);
            if (sm) {
                GroupMax<TIN, AM> gm;
                GroupMin<TIN> gl;
#pragma unroll 4
                for (int g = lane; g < s.n; g += 32) {
                    const uint4 x = *reinterpret_cast<const uint4 *>(d + 16 * g);
                    gm.add(x);
                    if constexpr (LO) gl.add(x);
                }
                if constexpr (LO) lo = -warp_max_redux(-gl.value());
                v.x = gm.value();
                if (edges) v.x = fmaxf(v.x, ie >= 0 ? (AM ? fabsf(xe) : xe) : -INFINITY);
                v.x = warp_max_redux(v.x);
                if constexpr (!AM) {
                    const float mz = v.x == -INFINITY ? 0.0f : v.x;
#pragma unroll 4
                    for (int g = lane; g < s.n; g += 32) {
                        float f[V];
                        decode_group<TIN>(*reinterpret_cast<const uint4 *>(d + 16 * g), f, 1.0f);
#pragma unroll
                        for (int j = 0; j < V; j += 2) {
                            const float2 t = __fmul2_rn(__fadd2_rn(make_float2(f[j], f[j + 1]), make_float2(-mz, -mz)),
                                                        make_float2(kLog2e, kLog2e));
                            s2 = __fadd2_rn(s2, make_float2(ex2_ftz(t.x), ex2_ftz(t.y)));
                        }
                    }
                    v.y = s2.x + s2.y;
                    if (ie >= 0) v.y += ex2_ftz((xe - mz) * kLog2e);
                }
            } else {
#pragma unroll 4
                for (int g = lane; g < s.n; g += 32) {
                    float f[V];
                    decode_group<TIN>(*reinterpret_cast<const uint4 *>(d + 16 * g), f, 1.0f);
#pragma unroll
                    for (int j = 0; j < V; j += 2) {
                        const float2 x = make_float2(f[j], f[j + 1]);
                        s2 = __ffma2_rn(x, x, s2);
                    }
                }
                v.y = s2.x + s2.y;
                if (ie >= 0) v.y = fmaf(xe, xe, v.y);
            }
            if constexpr (!AM) v.y = warp_sum(v.y);
            if (wl > 1) {  // over the row's warps of this CTA
                float2 *rd = red + (reds++ & 1u) * W;
                if (lane == 0) rd[warp] = v;
                named_bar_sync(first >> 1, wl * 32);
                v = merge(sm, rd[first + (lane & (wl - 1))], wl);
            }
            if (lw > 0) {  // over the cluster's CTAs: push all-gather among the groups of one number
                const uint32_t x = xchs & 1u;
                uint64_t *bar = &xbars[2 * first + x];
                float2 *sl = slots + (2 * first + x) * 16;
                if (warp == first && lane < P) {
                    fence_release_smem_cluster();  // this CTA's earlier reads of the slots first
                    st_async_v2f32(mapa_shared(smem_addr(sl + c), lane), v.x, v.y, mapa_shared(smem_addr(bar), lane));
                }
                if (warp == first && lane == 0) mbar_arrive_expect_tx(bar, static_cast<uint32_t>(P) * 8u);
                mbar_wait_bounded_cluster(bar, xchs >> 1 & 1u, a.err);
                ++xchs;
                v = merge(sm, sl[lane & (P - 1)], P);
            }
            stamp(3);
            unsigned char *orow = a.out + rw.out_off * (OP == OP_LSE ? 4 : osz);
            Stats st{v.x, v.y};
            if constexpr (OP == OP_LSE) {
                if (m == 0 && lane == 0) *reinterpret_cast<float *>(orow) = v.x + logf(v.y);
            } else {
                if constexpr (OP == OP_Q8) {
                    st.a = v.x > 0.0f ? __fdiv_rn(v.x, 127.0f) : 1.0f;  // the row scale
                    st.b = __frcp_rn(st.a);
                    if (m == 0 && lane == 0) a.out_scale[turn.row] = st.a;
                } else {
                    st.b = sm ? 1.0f / v.y : rsqrtf(v.y / static_cast<float>(rw.cols) + a.eps);
                }
                unsigned char *o = orow + (static_cast<long long>(s.h0) + s.lo * V) * osz;
                const bool vec = (reinterpret_cast<uintptr_t>(o) & (V * osz - 1)) == 0;
                auto one = [&](float x) {
                    if constexpr (OP == OP_Q8) return q8_code(x, st.a, st.b);
                    else return sm ? exp_scaled((x - st.a) * kLog2e, st.b) : x * st.b;
                };
                constexpr int OS = OP == OP_ROWS ? OP_SOFTMAX : OP;
                if (OP == OP_ROWS && !sm) {
                    if constexpr (OP == OP_ROWS) {
                        if (vec) write_segment<OP_RMS, TIN, true, false>(d, o, s.n, lane, st);
                        else write_segment<OP_RMS, TIN, false, false>(d, o, s.n, lane, st);
                    }
                } else if (vec && (AM || (lo - st.a) * kLog2e >= -126.0f)) {
                    write_segment<OS, TIN, true, false>(d, o, s.n, lane, st);
                } else if (vec) {
                    write_segment<OS, TIN, true, true>(d, o, s.n, lane, st);
                } else {
                    write_segment<OS, TIN, false, true>(d, o, s.n, lane, st);
                }
                if (ie >= 0) store_one<OP == OP_Q8 ? DT_I8 : TIN>(orow + static_cast<long long>(ie) * osz, one(xe));
            }
            stamp(4);
            __syncwarp();  // the segment is done with: its half takes a later turn's
        }
        load_ahead(k);
        if (!step(turn)) break;
    }
    __syncwarp();
    if (P > 1) {
        cluster_arrive_release();  // nobody exits while a peer may still push into it
        cluster_wait_acquire();
    }
}

}  // namespace credit
