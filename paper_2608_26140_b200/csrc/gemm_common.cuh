// Parts shared by the projection kernels (gemm_rows.cu, gemm_tc.cu, gemm_wm.cu): the row preparation in front of a contraction
// with its grid-wide barrier, and the epilogues on adjacent fp32 accumulator columns of one row.
#pragma once
#include "common.cuh"
#include "kernels.h"
#include "rows.cuh"
#include "tc_ptx.cuh"

namespace acache {

constexpr uint32_t GRID_WAIT_LIMIT = 1u << 21;

// Grid-wide barrier on a pair of counters in global memory: every CTA adds to bar[0] and waits for gridDim.x arrivals;
// those who have passed add to bar[1], and the last of them re-arms both words for the next launch.  One round trip to L2
// for the arrival and its view of the others: the arrival releases what the CTA wrote (the threads met at the block barrier
// before), the polls acquire, and the re-arming is left to a thread that has nothing to do until the epilogue (with fences
// around an atomic and the re-arming at the kernel's end, 1-2 us more per launch).  Bounded; returns false (and raises the CTA's abort flag) if the others do not arrive.
// self_test: the failure-detection self-test (acache_debug_expire_next_wait): the target is one arrival more than
// the grid can deliver and the poll limit is short, so the wait runs out and the abort path below is taken.
__device__ __forceinline__ bool grid_barrier(unsigned int* bar, volatile int* abort_flag, bool self_test = false) {
    __syncthreads();
    if (threadIdx.x == 0 && !*abort_flag) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        const unsigned int target = gridDim.x + (self_test ? 1u : 0u);
        const uint32_t limit = self_test ? (1u << 12) : GRID_WAIT_LIMIT;
        bool ok = false;
        for (uint32_t i = 0; i < limit; ++i) {
            unsigned int v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if (v >= target) { ok = true; break; }
            if (i >= 64) __nanosleep(100);
        }
        if (!ok) *abort_flag = 1;
    }
    __syncthreads();
    const bool passed = !*abort_flag;
    if (passed && threadIdx.x == 64 && atomicAdd(&bar[1], 1u) == gridDim.x - 1) {
        bar[0] = 0u;
        __threadfence();
        bar[1] = 0u;
    }
    return passed;
}

__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ uint4 pack8(const float* v) {
    return make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
}

// 16 bf16 of one row: one 32-byte store (a whole sector per lane) where the address allows it.
__device__ __forceinline__ void store16(__nv_bfloat16* o, const float* v) {
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = pack_bf16(v[2 * i], v[2 * i + 1]);
    if ((reinterpret_cast<uintptr_t>(o) & 31u) == 0) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                     ::"l"(o), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                     : "memory");
    } else {
        reinterpret_cast<uint4*>(o)[0] = make_uint4(w[0], w[1], w[2], w[3]);
        reinterpret_cast<uint4*>(o)[1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
}

// ---- epilogues on W adjacent fp32 accumulator columns of one row (W = 16 or 32) ----------------
// Every store is W*2 bytes of one row: whole 32-byte sectors, no partial-sector writes.

// x / (1 + exp(-x)).  The quotient by Markstein's scheme (IBM J. Res. Dev. 34, 1990): an approximate reciprocal, one Newton step
// for it, the quotient, one correction by its remainder.  Compared over all fp32 values it is the division operator's result,
// but for a last bit where that is denormal.  The operator checks for special operands with a branch that kept a thread from
// working on more than one element at a time (one warp per scheduler: a 256-column tile's SwiGLU took 10 us).  Divisor and
// dividend are quartered, so that the reciprocal of the largest finite divisor is not flushed to zero; an infinite one is
// replaced by a number whose reciprocal is, and the remainder of an infinite quotient (no number) is left out.
// Epilogue of a 128 x 256 tile: 10 -> 4.5 us, of the last one, which nothing hides, 9.5 -> 3.4.
__device__ __forceinline__ float silu(float x) {
    const float d = fminf(0.25f + 0.25f * __expf(-x), 3e38f), n = 0.25f * x;
    float r = __fdividef(1.f, d);
    r = fmaf(fmaf(-d, r, 1.f), r, r);
    const float q = n * r, rest = fmaf(-q, d, n);
    return rest == rest ? fmaf(rest, r, q) : q;
}

// out[grow, col..col+W) = bf16(silu(gate) * up)
template <int W>
__device__ __forceinline__ void out_swiglu(const GemmArgs& g, int grow, int col, float (&gate)[W], const float (&up)[W]) {
    __nv_bfloat16* o = static_cast<__nv_bfloat16*>(g.c) + (int64_t)grow * g.n[0] + col;
#pragma unroll
    for (int i = 0; i < W; ++i) gate[i] = silu(gate[i]) * up[i];
#pragma unroll
    for (int j = 0; j < W / 16; ++j) store16(o + 16 * j, gate + 16 * j);
}

// cos and sin of the row's position for W pairs from j0 on.
template <int W>
__device__ __forceinline__ void load_rope(const GemmArgs& g, int pos, int j0, float (&c)[W], float (&sn)[W]) {
    const int64_t at = (int64_t)(pos < 0 ? 0 : pos) * (g.head_dim >> 1) + j0;
    const float4* c4 = reinterpret_cast<const float4*>(g.rope_cos + at);
    const float4* s4 = reinterpret_cast<const float4*>(g.rope_sin + at);
#pragma unroll
    for (int j = 0; j < W / 4; ++j) {
        const float4 x = c4[j], y = s4[j];
        c[4 * j] = x.x; c[4 * j + 1] = x.y; c[4 * j + 2] = x.z; c[4 * j + 3] = x.w;
        sn[4 * j] = y.x; sn[4 * j + 1] = y.y; sn[4 * j + 2] = y.z; sn[4 * j + 3] = y.w;
    }
}

// q/k/v: bias, rotary embedding with the pairing (i, i + d/2) at the row's position, bf16 store
// to the compact output and, for k/v, straight into the cache row (scatter fused).
// lo/hi: W columns of each rotary half; col: column of lo[0] inside segment seg; c/sn: load_rope (rotary segments).
template <int W>
__device__ __forceinline__ void rope_qkv(const GemmArgs& g, int seg, int col, float (&lo)[W], float (&hi)[W], const float (&c)[W],
                                         const float (&sn)[W]) {
    const int half = g.head_dim >> 1;
    const __nv_bfloat16* bias = static_cast<const __nv_bfloat16*>(g.bias[seg]);
    if (bias) {
#pragma unroll
        for (int i = 0; i < W; ++i) {
            lo[i] += __bfloat162float(bias[col + i]);
            hi[i] += __bfloat162float(bias[col + half + i]);
        }
    }
    if (seg < g.rope_segments) {
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const float x = lo[i], y = hi[i];
            lo[i] = x * c[i] - y * sn[i];
            hi[i] = y * c[i] + x * sn[i];
        }
    }
}
template <int W>
__device__ __forceinline__ void store_qkv(const GemmArgs& g, int grow, int pos, int seg, int col, const float (&lo)[W],
                                          const float (&hi)[W]) {
    const int half = g.head_dim >> 1;
    const int nseg = g.n[seg];
    __nv_bfloat16* cache = seg == 1 ? static_cast<__nv_bfloat16*>(g.cache_k)
                         : seg == 2 ? static_cast<__nv_bfloat16*>(g.cache_v) : nullptr;
    int64_t orow = grow;
    bool o1_ok = g.out[seg] != nullptr;
    if (seg >= 1 && g.kv_out_rows && o1_ok) {          // the row's place in its request's private slot array
        const int r = __ldg(g.kv_out_rows + grow);
        if ((unsigned)r >= (unsigned)g.kv_out_stride) {
            atomicOr(g.status, kFlagBadIndex);
            o1_ok = false;
        }
        orow = (int64_t)(grow / g.rows_per_req) * g.kv_out_stride + r;
    }
    __nv_bfloat16* o1 = o1_ok ? static_cast<__nv_bfloat16*>(g.out[seg]) + orow * nseg + col : nullptr;
    __nv_bfloat16* o2 = (cache && pos >= 0)
                            ? cache + (int64_t)(grow / g.rows_per_req) * g.kv_batch_stride + (int64_t)pos * nseg + col
                            : nullptr;
#pragma unroll
    for (int j = 0; j < W / 16; ++j) {
        if (o1) { store16(o1 + 16 * j, lo + 16 * j); store16(o1 + half + 16 * j, hi + 16 * j); }
        if (o2) { store16(o2 + 16 * j, lo + 16 * j); store16(o2 + half + 16 * j, hi + 16 * j); }
    }
}

// Segment and in-segment column of the 128-wide column unit u128 of a q/k/v projection.
__device__ __forceinline__ void qkv_unit(const GemmArgs& g, int u128, int& seg, int& c0) {
    seg = 0; c0 = u128 * 128;
    while (seg < 2 && c0 >= g.n[seg]) { c0 -= g.n[seg]; ++seg; }
}

// Where row `row` of the A operand comes from (element offset inside rp.x); `writer` (one thread per
// row) records the row's position and source for the later kernels and raises the bad-index flag.
__device__ __forceinline__ int64_t prep_row_source(const GemmArgs& g, int row, bool writer, int* position = nullptr) {
    const RowPrep& rp = g.prep;
    const int rows_per_req = rp.k + rp.e;
    int64_t src = (int64_t)row * g.K;
    if (rp.enabled == 3) {       // compact rows picked by index
        const int b = row / rows_per_req;
        const int ci = rp.compact_idx[row];
        if (ci < 0 || ci >= rp.compact_rows) {
            if (writer) atomicOr(g.status, kFlagBadIndex);
        }
        src = ((int64_t)b * rp.compact_rows + (ci < 0 || ci >= rp.compact_rows ? 0 : ci)) * g.K;
    }
    if (rp.enabled == 1) {       // rows of R: position from the anchor / extra-row lists
        const int b = row / rows_per_req, i = row - b * rows_per_req;
        const int pos = row_position(rp.anchor_idx, rp.k, rp.extra_rows, rp.e, b, i, rp.affix_start,
                                     rp.affix_len, rp.ctx_len);
        if (!rp.x_is_compact) {
            if (rp.token_ids) {       // x is an embedding table: the row of the token at that position
                int id = rp.token_ids[(int64_t)b * rp.ctx_len + (pos < 0 ? 0 : pos)];
                if (id < 0 || id >= rp.table_rows) {
                    if (writer) atomicOr(g.status, kFlagBadIndex);
                    id = 0;
                }
                src = (int64_t)id * g.K;
            } else {
                src = (int64_t)b * rp.x_batch_stride + (int64_t)(pos < 0 ? 0 : pos) * g.K;
            }
        } else if (rp.compact_idx) {
            const int ci = rp.compact_idx[row];
            src = ((int64_t)b * rp.compact_rows + (ci < 0 ? 0 : ci)) * g.K;
        }
        if (position) *position = pos;
        if (writer) {
            rp.row_pos[row] = pos;
            rp.row_src[row] = src;
            if (pos < 0) atomicOr(g.status, kFlagBadIndex);
        }
    }
    return src;
}

// out = bf16(x * rsqrt(mean(x^2) + eps) * g) for one row, by one warp: rows of up to 4096 values in one pass from
// registers; longer ones in two passes with eight independent 16-byte loads in flight per lane (the second pass hits
// L1 / L2).
// GAIN_EARLY: the first half of the gain is asked for beside the row, in 32 more registers, where there are few rows per warp and
// the trip for it would follow the row's (615 rows: layer-step 384.7 -> 381.6 us, 5 x 203 rows 530.7 -> 527.7; the whole gain
// spills, see gemm_tc2_kernel).
template <bool GAIN_EARLY>
__device__ __forceinline__ void rmsnorm_row_warp(const uint4* __restrict__ xr, const uint4* __restrict__ gn,
                                                 uint4* __restrict__ out, int hidden, float eps, int lane,
                                                 uint4* __restrict__ raw) {
    const int nchunk = hidden >> 3;
    if (nchunk <= 512) {
        // rows of up to 4096 values: one pass, the row stays in registers (sixteen 16-byte loads in flight per lane,
        // one trip to memory per row instead of two), the gain is requested before the warp-wide sum
        uint4 u[16], early[GAIN_EARLY ? 8 : 1];
        float s1 = 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int c = i * 32 + lane;
            u[i] = c < nchunk ? __ldcg(xr + c) : make_uint4(0, 0, 0, 0);
        }
        if (GAIN_EARLY) {
#pragma unroll
            for (int i = 0; i < 8; ++i) early[GAIN_EARLY ? i : 0] = i * 32 + lane < nchunk ? __ldg(gn + i * 32 + lane) : make_uint4(0, 0, 0, 0);
        }
        if (raw) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int c = i * 32 + lane;
                if (c < nchunk) raw[c] = u[i];
            }
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const uint32_t w[4] = {u[i].x, u[i].y, u[i].z, u[i].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) { const float a = bf16_lo(w[e]), b = bf16_hi(w[e]); s1 += a * a + b * b; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        const float rstd1 = rsqrtf(s1 / (float)hidden + eps);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int c = i * 32 + lane;
            if (c < nchunk) {
                const uint4 gg = GAIN_EARLY && i < 8 ? early[GAIN_EARLY ? i & 7 : 0] : __ldg(gn + c);
                const uint32_t w[4] = {u[i].x, u[i].y, u[i].z, u[i].w};
                const uint32_t gw[4] = {gg.x, gg.y, gg.z, gg.w};
                uint32_t r[4];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    r[e] = pack_bf16(bf16_lo(w[e]) * rstd1 * bf16_lo(gw[e]), bf16_hi(w[e]) * rstd1 * bf16_hi(gw[e]));
                out[c] = make_uint4(r[0], r[1], r[2], r[3]);
            }
        }
        return;
    }
    float ss = 0.f;
    for (int c0 = 0; c0 < nchunk; c0 += 256) {
        uint4 u[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int c = c0 + i * 32 + lane;
            u[i] = c < nchunk ? __ldcg(xr + c) : make_uint4(0, 0, 0, 0);
            if (raw && c < nchunk) raw[c] = u[i];
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t w[4] = {u[i].x, u[i].y, u[i].z, u[i].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) { const float a = bf16_lo(w[e]), b = bf16_hi(w[e]); ss += a * a + b * b; }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const float rstd = rsqrtf(ss / (float)hidden + eps);
    for (int c0 = 0; c0 < nchunk; c0 += 256) {
        uint4 u[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int c = c0 + i * 32 + lane;
            u[i] = c < nchunk ? __ldcg(xr + c) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int c = c0 + i * 32 + lane;
            if (c < nchunk) {
                const uint4 gg = __ldg(gn + c);
                const uint32_t w[4] = {u[i].x, u[i].y, u[i].z, u[i].w};
                const uint32_t gw[4] = {gg.x, gg.y, gg.z, gg.w};
                uint32_t r[4];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    r[e] = pack_bf16(bf16_lo(w[e]) * rstd * bf16_lo(gw[e]), bf16_hi(w[e]) * rstd * bf16_hi(gw[e]));
                out[c] = make_uint4(r[0], r[1], r[2], r[3]);
            }
        }
    }
}

// Phase 0 of the projection kernels: the rows of R (or compact rows) -> RMSNorm -> the A operand,
// then a grid-wide barrier; the rows are read back through TMA.  With no more rows than CTAs (cta_rows) a
// whole CTA takes a row (shortest latency); with many rows every warp takes rows of its own, which
// keeps six rows in flight per SM instead of one.
template <bool GAIN_EARLY = false>
__device__ __forceinline__ void prep_phase(const GemmArgs& g, float* red, volatile int* abort_flag, int cta_rows) {
    const RowPrep& rp = g.prep;
    const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(rp.x);
    __nv_bfloat16* a_out = static_cast<__nv_bfloat16*>(const_cast<void*>(g.a));
    __nv_bfloat16* raw = static_cast<__nv_bfloat16*>(rp.raw_out);
    if (g.M <= cta_rows) {
        for (int row = blockIdx.x; row < g.M; row += gridDim.x) {
            const int64_t src = prep_row_source(g, row, threadIdx.x == 0);
            rmsnorm_row(reinterpret_cast<const uint4*>(x + src), reinterpret_cast<const uint4*>(rp.gain),
                        reinterpret_cast<uint4*>(a_out + (int64_t)row * g.K), g.K, rp.eps, red,
                        raw ? reinterpret_cast<uint4*>(raw + (int64_t)row * g.K) : nullptr);
        }
    } else {
        const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        // the source of the next row (index lookups: a dependent trip to memory) is asked for before this row is read
        int row = blockIdx.x * nw + warp;
        int64_t src = row < g.M ? prep_row_source(g, row, lane == 0) : 0;
        while (row < g.M) {
            const int next = row + gridDim.x * nw;
            const int64_t src_next = next < g.M ? prep_row_source(g, next, lane == 0) : 0;
            rmsnorm_row_warp<GAIN_EARLY>(reinterpret_cast<const uint4*>(x + src), reinterpret_cast<const uint4*>(rp.gain),
                             reinterpret_cast<uint4*>(a_out + (int64_t)row * g.K), g.K, rp.eps, lane,
                             raw ? reinterpret_cast<uint4*>(raw + (int64_t)row * g.K) : nullptr);
            row = next;
            src = src_next;
        }
    }
    asm volatile("fence.proxy.async;" ::: "memory");   // the rows are read back through TMA
    grid_barrier(g.grid_bar, abort_flag, g.debug_expire != 0);
    asm volatile("fence.proxy.async;" ::: "memory");
}

// Order of the whole tiles of the two-SM kernels, see kTileGroupN in gemm_tc.cu: groups of group_n weight tiles (nt), inside a
// group row pairs (mp, or chunks of rows) with the weight tiles innermost.
__device__ __forceinline__ void tile_coords(int t, int m_pairs, int n_tiles, int group_n, int& nt, int& mp) {
    const int full = n_tiles / group_n, per_group = group_n * m_pairs;
    if (t < full * per_group) {
        const int grp = t / per_group, r = t - grp * per_group;
        mp = r / group_n;
        nt = grp * group_n + (r - mp * group_n);
    } else {
        const int r = t - full * per_group, gn = n_tiles - full * group_n;
        mp = r / gn;
        nt = full * group_n + (r - mp * gn);
    }
}

// TMA load into this CTA's shared memory that completes on a barrier of the CTA pair's leader
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar_cluster,
                                                 uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1, {%2, %3}], [%4], %5;"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar_cluster), "l"(policy)
        : "memory");
}
// Tensor map over bf16 [rows, cols] row-major with the panel of 64 columns as a dimension: box = 64 columns x box_rows rows x
// `panels` panels, 128-byte swizzle, zero fill out of bounds.  half > 0: the rows in groups of `half`, box = box_rows rows of
// two consecutive groups (the two halves of rotary pairs).  Cached by (pointer, shape, box).  Host side, defined in
// gemm_tc.cu; the returned pointer is good until the next lookup (copy the map), under g_map_mutex.
const CUtensorMap* get_panel_map(const void* ptr, int rows, int cols, int box_rows, int panels, int half);
extern std::mutex g_map_mutex;
// box = 64 columns x box_rows rows of a bf16 [rows, cols] matrix, like above.
const CUtensorMap* get_rows_map(const void* ptr, int rows, int cols, int box_rows);
// Weights for gemm_wm.cu: box = 64 columns x 128 rows, the rows of unit c4 (coordinate of the last dimension) in the order in which
// the 32 lanes of each quarter want them.  Plain: rows 128 c4 + i.  Rope: 16 rows of the first half of a head, then their partners
// (head dimension 64: c4 counts heads, two per box).  Pairs: 16 rows of the matrix at ptr, then the same rows of the one `step`
// bytes further, 64 + 64 rows per unit.
enum WeightOrder : int { kWeightsPlain = 1, kWeightsRope128, kWeightsRope64, kWeightsPairs };
const CUtensorMap* get_weight_map(const void* ptr, int rows, int cols, WeightOrder order, int64_t step);

// gemm_wm.cu: projections of more than 128 rows, weights as the product's M.  own_us: what the caller's own kernel would take, as
// pair_tile_us has it.  0 = not taken (the caller launches its own), 1 = launched, -1 = the launch failed.
int launch_gemm_wm(const GemmArgs& g, double own_us, int group_n, cudaStream_t stream);
// Time from one tile of a two-SM kernel to the next: its main loop, k_blocks of 64 one after the other, `columns` wide, or the epilogue
// of the tile before it, if that is longer, and about 1 us for the change of tiles.  Measured at 615 rows (gate/up, 256 K blocks in a
// row): 0.33 us a K block at 256 columns, 0.285 at 208, 0.24 at 128; the instructions alone would take 0.27, 0.22, 0.14.
inline double pair_tile_us(int k_blocks, int columns, double epilogue_us) {
    const double loop_us = k_blocks * (columns + 200) * 0.0007;
    return 1.0 + (loop_us > epilogue_us ? loop_us : epilogue_us);
}

// gemm_rows.cu: projections of at most 128 rows whose tiles fit the SMs at once; 0 = not applicable (the caller then uses
// the kernels of gemm_tc.cu), else the number of kernels launched, -1 if a launch failed.
int launch_gemm_rows(const GemmArgs& g, cudaStream_t stream);

}  // namespace acache
