// C[M, N] = A[M, K] * B[N, K]^T (bf16 in, fp32 accumulate) on the 5th-generation tensor
// cores for the projections of the selective recomputation (Section 3.3).
//
// Projections of at most 128 rows run on gemm_rows.cu where their tiles fit the SMs at once; larger ones on gemm_wm.cu where chunks
// of rows fill the rounds better than 256-row pairs; here, the rest of both (the LM head, very wide ones, cut tiles).
//
// gemm_tc_kernel (at most one CTA per SM):
//   phase 0 (optional)  gather the rows of R (or take compact rows) and RMSNorm them into the
//                       A operand, then a grid-wide barrier
//   phase 1             the contraction: work = (output tiles of 128 x 256) x (K blocks of 64),
//                       the flat list of (tile, k-block) iterations cut into equal contiguous
//                       ranges, one per CTA, so every SM streams the same number of weight
//                       bytes whatever N and K are.  One thread issues TMA loads into a 4-stage
//                       128-byte-swizzled ring (weights evict-first, activations evict-last in
//                       L2), one thread issues tcgen05.mma (128 x 256 x 16) into one of two TMEM
//                       accumulators, four warps drain TMEM with tcgen05.ld and write fp32
//                       partial tiles
// gemm_tc2_kernel (two or more 128-row tiles): a cluster of two CTAs per 256 x 256 tile,
//   tcgen05.mma.cta_group::2; whole tiles walked round-robin, or, when the tiles fill less than
//   two thirds of a wave, equal contiguous (tile, k-block) ranges per cluster like the kernel above.
// gemm_finish_kernel: sums the partial tiles of every output element in ascending CTA order
//   (bitwise reproducible) and applies the epilogue: bias + RoPE + KV scatter, residual add,
//   or SwiGLU.  It is a kernel of its own because it is bound by L2 latency and wants far
//   more threads in flight than one CTA per SM provides (measured: fused into the contraction
//   kernel behind a second grid barrier it was ~10 us slower per projection).
//
// Every wait (mbarrier or grid barrier) is bounded: on expiry the CTA raises kFlagWaitExpired
// in the status word, stops issuing work, lets its in-flight copies land, frees its TMEM and
// returns.  The grid never exceeds the SM count, so all CTAs are resident for the barrier.
#include <cuda.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "gemm_common.cuh"
#include "kernels.h"
#include "launch.h"
#include "rows.cuh"
#include "tc_ptx.cuh"

namespace acache {

constexpr int TC_BM = 128, TC_BN = 256, TC_BK = 64, TC_STAGES = 4;
constexpr int TC_A_BYTES = TC_BM * TC_BK * 2;          // 16 KB
constexpr int TC_HALF_BYTES = 128 * TC_BK * 2;         // 16 KB: one 128-row half of the B tile
constexpr int TC_STAGE_BYTES = TC_A_BYTES + 2 * TC_HALF_BYTES;
constexpr int TC_THREADS = 192;                        // warp 0: TMA, warp 1: MMA, warps 2-5: drain; all six warps do phase 0
constexpr int TC_SMEM = TC_STAGES * TC_STAGE_BYTES + 1024 /*alignment slack*/ + 256 /*barriers*/;
static_assert(TC_SMEM >= kAloneBytes);
constexpr int TC_SLOT_FLOATS = TC_BM * TC_BN;          // one fp32 partial tile

struct TcPlan {
    int m_tiles, n_tiles, KB, tiles, U, ctas;
    int prefill;          // ring stages whose weight halves are loaded before the dependency wait
    int pair_u;           // two-SM kernel, stream-K mode: (pair tile, K block) iterations per cluster (0: whole tiles)
    int m_pairs;          // 256-row tile rows of the two-SM kernel
    int units;            // 128-row B halves over all segments (non-SwiGLU) or ffn/128 (SwiGLU)
    int group_n;          // two-SM kernel, whole tiles: weight tiles per group of the tile order
    int w_keep;           // weights loaded with the evict-last policy (every row tile re-reads them from L2) instead of evict-first
};

// Which weight matrix and row the 128-row half `h` of N tile `nt` starts at; -1 if past the end.
__device__ __forceinline__ int half_source(const GemmArgs& g, const TcPlan& p, int nt, int h, int& row) {
    if (g.epilogue == kEpiSwiGLU) {
        row = nt * 128;
        return h;                      // half 0: gate rows, half 1: up rows
    }
    int u = nt * 2 + h;
    if (u >= p.units) return -1;
    int r = u * 128, seg = 0;
    while (seg < 2 && r >= g.n[seg]) { r -= g.n[seg]; ++seg; }
    row = r;
    return seg;
}

// ---- split tiles: partial slots and their ordered sum -------------------------------------------
// A tile whose K range is cut between CTAs is accumulated through fp32 partial tiles.  Each CTA owns
// two slots: slot 0 for its first segment, slot 1 for its last (segments in between are whole tiles
// and never need one).  Tile t's contributors are CTAs c_first..c_last; CTA c's part of it is that
// CTA's first segment exactly when the CTA starts inside the tile.
// In the two-SM kernel's stream-K mode the contributors are clusters, the tile that is cut is the
// 256-row pair tile tp = nt * m_pairs + mt / 2, and each CTA of a cluster (rank = mt & 1) has its own
// pair of slots: slot = (cluster * 2 + segment) * 2 + rank.
__device__ __forceinline__ void tile_cover(const TcPlan& p, int t, int& c_first, int& c_last) {
    if (p.pair_u) {
        const int nt = t / p.m_tiles, mt = t - nt * p.m_tiles;
        t = nt * p.m_pairs + (mt >> 1);
    }
    const int U = p.pair_u ? p.pair_u : p.U;
    c_first = (int)(((int64_t)t * p.KB) / U);
    c_last = (int)(((int64_t)(t + 1) * p.KB - 1) / U);
}
__device__ __forceinline__ int64_t slot_of(const TcPlan& p, int t, int c) {
    if (p.pair_u) {
        const int nt = t / p.m_tiles, mt = t - nt * p.m_tiles;
        const int tp = nt * p.m_pairs + (mt >> 1);
        return ((int64_t)c * 2 + ((int64_t)c * p.pair_u >= (int64_t)tp * p.KB ? 0 : 1)) * 2 + (mt & 1);
    }
    return (int64_t)c * 2 + ((int64_t)c * p.U >= (int64_t)t * p.KB ? 0 : 1);
}

// Ordered sums over the contributing CTAs' partial tiles of one row for 16 adjacent columns
// starting at column group pc0 and, if pc1 >= 0, 16 more starting at pc1.  Loads are issued two
// CTAs at a time for all eight column groups (16 independent 16-byte loads in flight per thread)
// and added in ascending CTA order, which keeps the result bitwise reproducible.
__device__ __forceinline__ void sum_slots16(const float* __restrict__ partial, const TcPlan& p, int t, int c_first,
                                            int c_last, int pc0, int pc1, int row, float (&lo)[16], float (&hi)[16]) {
#pragma unroll
    for (int i = 0; i < 16; ++i) { lo[i] = 0.f; hi[i] = 0.f; }
    constexpr int NC = 2;      // contributing CTAs per round of loads
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const int o0 = pc0 * TC_BM + row, o1 = (pc1 < 0 ? pc0 : pc1) * TC_BM + row;
    for (int c = c_first; c <= c_last; c += NC) {
        float4 a[NC][4], b[NC][4];
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            const bool in = c + i <= c_last;
            const float4* src = reinterpret_cast<const float4*>(partial) + slot_of(p, t, in ? c + i : c) * (TC_SLOT_FLOATS / 4);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                a[i][j] = in ? __ldcg(src + o0 + j * TC_BM) : zero;
                b[i][j] = (in && pc1 >= 0) ? __ldcg(src + o1 + j * TC_BM) : zero;
            }
        }
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            if (c + i <= c_last) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    lo[4 * j] += a[i][j].x; lo[4 * j + 1] += a[i][j].y; lo[4 * j + 2] += a[i][j].z; lo[4 * j + 3] += a[i][j].w;
                    hi[4 * j] += b[i][j].x; hi[4 * j + 1] += b[i][j].y; hi[4 * j + 2] += b[i][j].z; hi[4 * j + 3] += b[i][j].w;
                }
            }
        }
    }
}

// Entry of the softmax statistics of one row in vocabulary tile nt: rows contiguous, so that a warp (a row per lane) writes
// whole lines.
__device__ __forceinline__ float4* logit_entry(const GemmArgs& g, int nt, int entry, int row) {
    return g.logit_stats + ((int64_t)nt * 16 + entry) * g.M + row;
}

// Softmax statistics of W logits starting at vocabulary index col: running (max, sum exp(z - max),
// arg max with the lowest index on ties).
template <int W>
__device__ __forceinline__ void logit_stats_update(const float (&v)[W], int col, float& m, float& s, int& arg) {
    float cm = v[0];
    int ca = 0;
#pragma unroll
    for (int i = 1; i < W; ++i)
        if (v[i] > cm) { cm = v[i]; ca = i; }
    if (cm > m) {
        s *= __expf(m - cm);
        m = cm;
        arg = col + ca;
    }
#pragma unroll
    for (int i = 0; i < W; ++i) s += __expf(v[i] - m);
}

// The same for one group of 16 columns, four CTAs at a time (the registers the second group would take hold
// two more CTAs' loads): epilogues without a second group (residual, logits) have nine or ten contributors per
// tile on the narrow projections, and every round of loads is a trip to L2.
__device__ __forceinline__ void sum_slots16_single(const float* __restrict__ partial, const TcPlan& p, int t, int c_first,
                                                   int c_last, int pc0, int row, float (&lo)[16]) {
#pragma unroll
    for (int i = 0; i < 16; ++i) lo[i] = 0.f;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const int o0 = pc0 * TC_BM + row;
    for (int c = c_first; c <= c_last; c += 4) {
        float4 a[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool in = c + i <= c_last;
            const float4* src = reinterpret_cast<const float4*>(partial) + slot_of(p, t, in ? c + i : c) * (TC_SLOT_FLOATS / 4);
#pragma unroll
            for (int j = 0; j < 4; ++j) a[i][j] = in ? __ldcg(src + o0 + j * TC_BM) : zero;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (c + i <= c_last) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    lo[4 * j] += a[i][j].x; lo[4 * j + 1] += a[i][j].y; lo[4 * j + 2] += a[i][j].z; lo[4 * j + 3] += a[i][j].w;
                }
            }
        }
    }
}

// Work items of the finish per output tile: 16 output columns each (q/k/v: 16 of each rotary half).
__host__ __device__ __forceinline__ int finish_items_per_tile(int epilogue) {
    return (epilogue == kEpiResidual || epilogue == kEpiLogits) ? 16 : 8;
}

// Finish of one work item of split tile t = nt * m_tiles + mt for tile row `row`.
// The row's 32 bytes of residual under an item's 16 columns (kEpiResidual).
__device__ __forceinline__ void load_residual16(const GemmArgs& g, int grow, int col, uint4 (&res)[2]) {
    const int64_t roff = g.resid_off ? __ldcg(g.resid_off + grow) : (int64_t)grow * g.n[0];
    const uint4* rp = reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(g.resid) + roff + col);
    res[0] = __ldcg(rp); res[1] = __ldcg(rp + 1);
}

// Tiles whose K range is cut, each listed once.
struct SplitTiles {
    int n;
    int tile[160];     // one per CTA boundary that cuts a tile (at most SM count - 1)
};

// Where an item of the finish lives: everything that can be worked out before the projection has finished.
struct FinishItem {
    int nt, grow, c_first, c_last, pc0, pc1, u128, lo_col;
    bool skip;
};
__device__ __forceinline__ FinishItem finish_plan(const GemmArgs& g, const TcPlan& p, int t, int item, int row) {
    FinishItem f;
    f.nt = t / p.m_tiles;
    f.grow = (t - f.nt * p.m_tiles) * TC_BM + row;
    tile_cover(p, t, f.c_first, f.c_last);
    const int half = g.head_dim >> 1;
    f.pc1 = -1; f.u128 = 0; f.lo_col = 0; f.skip = false;
    if (g.epilogue == kEpiResidual || g.epilogue == kEpiLogits) {
        f.pc0 = item * 4;
        f.skip = f.nt * 2 + (item >> 3) >= p.units;                           // the tile's second half is past the last column
    } else if (g.epilogue == kEpiSwiGLU) {
        f.pc0 = item * 4; f.pc1 = 32 + f.pc0;
    } else {
        const int h = item >> 2, r = item & 3;
        f.u128 = f.nt * 2 + h;
        if (f.u128 >= p.units) f.skip = true;                                 // the tile's second half is past the end
        f.lo_col = g.head_dim == 128 ? 16 * r : 64 * (r >> 1) + 16 * (r & 1);   // column inside the 128-wide unit
        f.pc0 = 32 * h + (f.lo_col >> 2);
        f.pc1 = f.pc0 + (half >> 2);
    }
    return f;
}

// res: the residual, loaded by the caller (kEpiResidual only).
__device__ __forceinline__ void finish_item(const GemmArgs& g, const TcPlan& p, int t, int item, int row, const FinishItem& f,
                                            const uint4 (&res)[2]) {
    if (f.skip) return;
    const int nt = f.nt, grow = f.grow, c_first = f.c_first, c_last = f.c_last, pc0 = f.pc0, pc1 = f.pc1, u128 = f.u128,
              lo_col = f.lo_col;
    const int half = g.head_dim >> 1;
    int pos = 0;
    if (g.epilogue == kEpiQKV) pos = __ldcg(g.row_pos + grow);     // independent of the sums: overlaps their loads
    float lo[16], hi[16];
    if (pc1 < 0) sum_slots16_single(g.partial, p, t, c_first, c_last, pc0, row, lo);
    else sum_slots16(g.partial, p, t, c_first, c_last, pc0, pc1, row, lo, hi);
    if (g.epilogue == kEpiResidual) {
        const uint32_t rw[8] = {res[0].x, res[0].y, res[0].z, res[0].w, res[1].x, res[1].y, res[1].z, res[1].w};
#pragma unroll
        for (int i = 0; i < 8; ++i) { lo[2 * i] += bf16_lo(rw[i]); lo[2 * i + 1] += bf16_hi(rw[i]); }
        store16(static_cast<__nv_bfloat16*>(g.c) + (int64_t)grow * g.n[0] + nt * TC_BN + item * 16, lo);
    } else if (g.epilogue == kEpiLogits) {
        float m = -INFINITY, sm = 0.f;
        int arg = 0;
        logit_stats_update<16>(lo, nt * TC_BN + item * 16, m, sm, arg);
        *logit_entry(g, nt, item, grow) = make_float4(m, sm, __int_as_float(arg), 16.f);
    } else if (g.epilogue == kEpiSwiGLU) {
        out_swiglu<16>(g, grow, nt * 128 + item * 16, lo, hi);
    } else {
        int seg, c0;
        qkv_unit(g, u128, seg, c0);
        float c[16], sn[16];
        if (seg < g.rope_segments) load_rope<16>(g, pos, lo_col & (half - 1), c, sn);
        rope_qkv<16>(g, seg, c0 + lo_col, lo, hi, c, sn);
        store_qkv<16>(g, grow, pos, seg, c0 + lo_col, lo, hi);
    }
}

// Epilogue of one half (128 accumulator columns) of a whole tile straight from TMEM: thread = one row, 32 columns per
// tcgen05.ld.  The last tile's epilogue is the tail of the launch, and with four warps taking a tile's 256 columns and asking
// for the residual (the rotary table) chunk by chunk it lasted 10-16 us.  So eight warps share a tile, and what does not
// depend on the accumulator is requested before the wait for it: the half's 256 bytes of residual, or the first 32 pairs'
// cosines and sines.  Last tile of a 1015-row down projection: 13.1 -> 3.0 us, of a q/k/v projection 14.3 -> 10.1.
struct HalfPre {
    uint32_t w[64];
    int pos;
};
__device__ __forceinline__ void half_prefetch(const GemmArgs& g, int nt, int hf, int grow, bool valid, HalfPre& pre) {
    pre.pos = 0;
    if (!valid) return;
    if (g.epilogue == kEpiResidual) {
        const int64_t roff = g.resid_off ? __ldcg(g.resid_off + grow) : (int64_t)grow * g.n[0];
        const uint4* rp = reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(g.resid) + roff + nt * TC_BN + hf * 128);
        if (nt * TC_BN + hf * 128 < g.n[0]) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const uint4 u = __ldcg(rp + j);
                pre.w[4 * j] = u.x; pre.w[4 * j + 1] = u.y; pre.w[4 * j + 2] = u.z; pre.w[4 * j + 3] = u.w;
            }
        }
    } else if (g.epilogue == kEpiQKV) {
        pre.pos = __ldcg(g.row_pos + grow);
        int seg, c0;
        qkv_unit(g, nt * 2 + hf, seg, c0);
        if (seg < g.rope_segments) {
            float (&c)[32] = reinterpret_cast<float (&)[32]>(pre.w[0]);
            float (&sn)[32] = reinterpret_cast<float (&)[32]>(pre.w[32]);
            load_rope<32>(g, pre.pos, 0, c, sn);
        }
    }
}
__device__ __forceinline__ void half_epilogue(const GemmArgs& g, const TcPlan& p, uint32_t taddr, int nt, int hf, int n_halves,
                                              int grow, bool valid, HalfPre& pre) {
    if (g.epilogue == kEpiResidual) {
        __nv_bfloat16* o = static_cast<__nv_bfloat16*>(g.c) + (int64_t)grow * g.n[0] + nt * TC_BN + hf * 128;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float v[32];
            tc_ld32(taddr + hf * 128 + c * 32, v);
#pragma unroll
            for (int i = 0; i < 16; ++i) { v[2 * i] += bf16_lo(pre.w[16 * c + i]); v[2 * i + 1] += bf16_hi(pre.w[16 * c + i]); }
            if (valid) { store16(o + c * 32, v); store16(o + c * 32 + 16, v + 16); }
        }
    } else if (g.epilogue == kEpiLogits) {
        // one entry per half; w: how many entries the tile has
        float m = -INFINITY, sm = 0.f;
        int arg = 0;
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
            float v[32];
            tc_ld32(taddr + hf * 128 + c * 32, v);
            logit_stats_update<32>(v, nt * TC_BN + hf * 128 + c * 32, m, sm, arg);
        }
        if (valid) *logit_entry(g, nt, hf, grow) = make_float4(m, sm, __int_as_float(arg), (float)n_halves);
    } else if (g.epilogue == kEpiSwiGLU) {
#pragma unroll 1
        for (int c = hf * 2; c < hf * 2 + 2; ++c) {
            float gate[32], up[32];
            tc_ld32(taddr + c * 32, gate);
            tc_ld32(taddr + 128 + c * 32, up);
            if (valid) out_swiglu<32>(g, grow, nt * 128 + c * 32, gate, up);
        }
    } else {
        const int half = g.head_dim >> 1;
        int seg, c0;
        qkv_unit(g, nt * 2 + hf, seg, c0);
        float (&c)[32] = reinterpret_cast<float (&)[32]>(pre.w[0]);
        float (&sn)[32] = reinterpret_cast<float (&)[32]>(pre.w[32]);
#pragma unroll 1
        for (int r = 0; r < 2; ++r) {
            // d = 128: chunks (r, r + 2) of the unit; d = 64: chunks (2r, 2r + 1)
            const int cl = g.head_dim == 128 ? r : 2 * r, ch = g.head_dim == 128 ? r + 2 : 2 * r + 1;
#pragma unroll
            for (int w = 0; w < 32; w += 16) {
                float lo[16], hi[16];
                tc_ld16(taddr + hf * 128 + cl * 32 + w, lo);
                tc_ld16(taddr + hf * 128 + ch * 32 + w, hi);
                if (valid) {
                    rope_qkv<16>(g, seg, c0 + cl * 32 + w, lo, hi, reinterpret_cast<float (&)[16]>(c[w]), reinterpret_cast<float (&)[16]>(sn[w]));
                    store_qkv<16>(g, grow, pre.pos, seg, c0 + cl * 32 + w, lo, hi);
                }
            }
            if (valid && r == 0 && half == 64 && seg < g.rope_segments) load_rope<32>(g, pre.pos, 32, c, sn);
        }
    }
}

// The same row preparation as a kernel of its own, for many rows: inside the projection kernel only the CTA's six warps
// work on it (one CTA per SM: 14 752 rows took 88-95 us per launch, 2.5 TB/s); here sixteen warps per SM do, and the
// projection starts without the grid-wide barrier.
__global__ void __launch_bounds__(256, 2) prep_rows_kernel(const GemmArgs g) {
    pdl_wait();
    pdl_launch_dependents();
    const RowPrep& rp = g.prep;
    const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(rp.x);
    __nv_bfloat16* a_out = static_cast<__nv_bfloat16*>(const_cast<void*>(g.a));
    __nv_bfloat16* raw = static_cast<__nv_bfloat16*>(rp.raw_out);
    const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int row = blockIdx.x * nw + warp;
    int64_t src = row < g.M ? prep_row_source(g, row, lane == 0) : 0;
    while (row < g.M) {
        const int next = row + gridDim.x * nw;
        const int64_t src_next = next < g.M ? prep_row_source(g, next, lane == 0) : 0;
        rmsnorm_row_warp<false>(reinterpret_cast<const uint4*>(x + src), reinterpret_cast<const uint4*>(rp.gain),
                         reinterpret_cast<uint4*>(a_out + (int64_t)row * g.K), g.K, rp.eps, lane,
                         raw ? reinterpret_cast<uint4*>(raw + (int64_t)row * g.K) : nullptr);
        row = next;
        src = src_next;
    }
}

__global__ void __launch_bounds__(TC_THREADS, 1)
gemm_tc_kernel(const GemmArgs g, const TcPlan p, const __grid_constant__ CUtensorMap mapA,
               const __grid_constant__ CUtensorMap mapB0, const __grid_constant__ CUtensorMap mapB1,
               const __grid_constant__ CUtensorMap mapB2) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ float red[TC_THREADS / 32];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char* base_ptr = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t bars = base + TC_STAGES * TC_STAGE_BYTES;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + TC_STAGES * TC_STAGE_BYTES + 192);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + TC_STAGES * TC_STAGE_BYTES + 200);
    auto full_bar = [&](int s) { return bars + 8 * s; };
    auto empty_bar = [&](int s) { return bars + 8 * (TC_STAGES + s); };
    auto tfull_bar = [&](int i) { return bars + 8 * (2 * TC_STAGES + i); };
    auto tempty_bar = [&](int i) { return bars + 8 * (2 * TC_STAGES + 2 + i); };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < TC_STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(tfull_bar(i), 1); mbar_init(tempty_bar(i), 4); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;"
                     ::"r"(smem_u32(const_cast<uint32_t*>(tmem_slot))) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const int it0 = blockIdx.x * p.U;
    const int it1 = min(it0 + p.U, p.tiles * p.KB);
    // The weights are constant inputs (no earlier kernel writes them), so their loads may start
    // before the previous kernel has finished: fill the ring's weight halves now.  The activation halves
    // follow once the producer kernel is done.
    int prefilled = 0;
    if (warp == 0 && lane == 0) {
        const CUtensorMap* maps[3] = {&mapB0, &mapB1, &mapB2};
        const uint64_t pol_w = g.keep_weights ? policy_evict_last() : policy_evict_first();
        for (int i = 0; i < p.prefill && it0 + i < it1; ++i) {
            const int it = it0 + i, t = it / p.KB, kb = it - t * p.KB, nt = t / p.m_tiles;
            int row0, row1;
            const int s0 = half_source(g, p, nt, 0, row0), s1 = half_source(g, p, nt, 1, row1);
            const uint32_t sB = base + i * TC_STAGE_BYTES + TC_A_BYTES;
            mbar_expect_tx(full_bar(i), TC_A_BYTES + TC_HALF_BYTES * (1 + (s1 >= 0)));
            tma_load_2d(sB, maps[s0], kb * TC_BK, row0, full_bar(i), pol_w);
            if (s1 >= 0) tma_load_2d(sB + TC_HALF_BYTES, maps[s1], kb * TC_BK, row1, full_bar(i), pol_w);
            prefilled = i + 1;
        }
    }
    // everything above overlaps the previous kernel's tail; its outputs are touched only below
    pdl_wait();
    pdl_launch_dependents();

    // ---------------- phase 0: gather the rows of R and RMSNorm them into A ----------------
    if (g.prep.enabled) prep_phase(g, red, abort_flag, gridDim.x);

    // ---------------- phase 1: the contraction ----------------

    if (warp == 0 && lane == 0) {
        // TMA producer
        const CUtensorMap* maps[3] = {&mapB0, &mapB1, &mapB2};
        int stage = 0;
        uint32_t phase = 0;
        bool ok = !*abort_flag;
        const uint64_t pol_a = policy_evict_last(), pol_w = g.keep_weights ? pol_a : policy_evict_first();
        for (int it = it0; it < it1 && ok;) {
            const int t = it / p.KB, kb0 = it - t * p.KB;
            const int kb1 = min(p.KB, kb0 + (it1 - it));
            const int nt = t / p.m_tiles, mt = t - nt * p.m_tiles;
            int row0, row1;
            const int s0 = half_source(g, p, nt, 0, row0), s1 = half_source(g, p, nt, 1, row1);
            const uint32_t bytes = TC_A_BYTES + TC_HALF_BYTES * (1 + (s1 >= 0));
            for (int kb = kb0; kb < kb1; ++kb) {
                const uint32_t sA = base + stage * TC_STAGE_BYTES, sB = sA + TC_A_BYTES;
                if (prefilled > 0) {          // this stage's weight halves are already on their way
                    --prefilled;
                    tma_load_2d(sA, &mapA, kb * TC_BK, mt * TC_BM, full_bar(stage), pol_a);
                } else {
                    if (!(ok = mbar_poll(empty_bar(stage), phase ^ 1, abort_flag))) break;
                    mbar_expect_tx(full_bar(stage), bytes);
                    tma_load_2d(sA, &mapA, kb * TC_BK, mt * TC_BM, full_bar(stage), pol_a);
                    tma_load_2d(sB, maps[s0], kb * TC_BK, row0, full_bar(stage), pol_w);
                    if (s1 >= 0) tma_load_2d(sB + TC_HALF_BYTES, maps[s1], kb * TC_BK, row1, full_bar(stage), pol_w);
                }
                if (++stage == TC_STAGES) { stage = 0; phase ^= 1; }
            }
            it += kb1 - kb0;
        }
    } else if (warp == 1 && lane == 0) {
        // MMA issuer
        int stage = 0, acc = 0;
        uint32_t phase = 0, acc_phase = 0;
        bool ok = !*abort_flag;
        for (int it = it0; it < it1 && ok;) {
            const int t = it / p.KB, kb0 = it - t * p.KB;
            const int kb1 = min(p.KB, kb0 + (it1 - it));
            const int nt = t / p.m_tiles;
            int row1;
            const uint32_t idesc = idesc_bf16(half_source(g, p, nt, 1, row1) >= 0 ? 256 : 128);
            if (!(ok = mbar_poll(tempty_bar(acc), acc_phase ^ 1, abort_flag))) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + acc * TC_BN;
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!(ok = mbar_poll(full_bar(stage), phase, abort_flag))) break;
                tc_fence_after();
                const uint32_t sA = base + stage * TC_STAGE_BYTES, sB = sA + TC_A_BYTES;
                const uint64_t da = smem_desc_sw128(sA), db = smem_desc_sw128(sB);
#pragma unroll
                for (int k = 0; k < TC_BK / 16; ++k)
                    tc_mma(d_tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc, (kb > kb0 || k > 0) ? 1u : 0u);
                tc_commit(empty_bar(stage));      // the stage is free once these MMAs have read it
                if (++stage == TC_STAGES) { stage = 0; phase ^= 1; }
            }
            if (!ok) break;
            tc_commit(tfull_bar(acc));            // accumulator complete
            if (++acc == 2) { acc = 0; acc_phase ^= 1; }
            it += kb1 - kb0;
        }
    } else if (warp >= 2 && warp < 6) {
        // drain: whole tiles get their epilogue straight from TMEM; a tile whose K range is split
        // between CTAs goes to this CTA's fp32 partial slot, layout [column / 4][row][4]
        const int q = warp & 3;                   // TMEM lane quarter this warp may read
        const int row = q * 32 + lane;
        int acc = 0;
        uint32_t acc_phase = 0;
        bool ok = !*abort_flag;
        const uint64_t pol_p = policy_evict_last();
        for (int it = it0; it < it1 && ok;) {
            const int t = it / p.KB, kb0 = it - t * p.KB;
            const int kb1 = min(p.KB, kb0 + (it1 - it));
            const int nt = t / p.m_tiles, mt = t - nt * p.m_tiles;
            int row1;
            const int nchunks = half_source(g, p, nt, 1, row1) >= 0 ? 8 : 4;
            if (!(ok = mbar_wait(tfull_bar(acc), acc_phase, abort_flag))) break;
            tc_fence_after();
            const bool valid = mt * TC_BM + row < g.M;
            const uint32_t taddr = tmem_base + acc * TC_BN + ((uint32_t)(q * 32) << 16);
            if (kb0 == 0 && kb1 == p.KB) {
                for (int hf = 0; hf < nchunks / 4; ++hf) {
                    HalfPre pre;
                    half_prefetch(g, nt, hf, mt * TC_BM + row, valid, pre);
                    half_epilogue(g, p, taddr, nt, hf, nchunks / 4, mt * TC_BM + row, valid, pre);
                }
            } else {
                float4* dst = reinterpret_cast<float4*>(g.partial) +
                              ((int64_t)blockIdx.x * 2 + (it == it0 ? 0 : 1)) * (TC_SLOT_FLOATS / 4);
                for (int c = 0; c < nchunks; ++c) {
                    float v[32];
                    tc_ld32(taddr + c * 32, v);
                    if (valid) {
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            st_hint_f4(&dst[(c * 8 + i) * TC_BM + row], make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]), pol_p);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty_bar(acc));
            if (++acc == 2) { acc = 0; acc_phase ^= 1; }
            it += kb1 - kb0;
        }
    }
    tc_fence_before();
    __syncthreads();
    // ---------------- teardown ----------------
    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0) {
            atomicOr(g.status, kFlagWaitExpired);
            // Ring stages whose weight halves were requested before the dependency wait but whose activation tile
            // never was (the wait that ran out came first): send that tile now, so that the stage's full barrier
            // completes exactly when all of its copies have landed, and wait for it.  No copy may still be on its
            // way into this CTA's shared memory when the CTA returns.
            const uint64_t pol = policy_evict_last();
            for (int i = 0; i < prefilled; ++i)
                tma_load_2d(base + i * TC_STAGE_BYTES, &mapA, 0, 0, full_bar(i), pol);
            for (int i = 0; i < prefilled; ++i)
                for (uint32_t n = 0; n < TC_WAIT_LIMIT && !mbar_try_wait(full_bar(i), 0); ++n) __nanosleep(40);
            for (int i = 0; i < 4096; ++i) __nanosleep(64);   // copies of stages that were complete when a role gave up
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

// ---- cta_group::2: two SMs on one 256 x 256 output tile (many-row problems) -----------------------
// A cluster of two CTAs owns a tile: CTA r holds rows [128 r, 128 r + 128) of A and the r-th
// 128-row half of the weight tile in its own shared memory, so each SM moves half of the weight
// bytes per flop that the one-CTA kernel moves; the leader CTA's MMA thread issues
// tcgen05.mma.cta_group::2 (M = 256) and each CTA's TMEM receives its 128 rows of the result.
// Whole tiles: clusters walk the tile list round-robin in groups of weight tiles (tile_coords).  Too few tiles for that: every cluster
// takes an equal contiguous range of (tile, K block) iterations, and the cut tiles go through the finish kernel (plan_gemm).
// Barriers: the leader's full[s] counts both CTAs' TMA bytes (announced by the leader's producer); empty[s] and tmem_full[a] live in
// each CTA and are signalled by a tcgen05.commit multicast to both; the leader's tmem_empty[a]
// collects the drain warps of both CTAs.
constexpr int TC2_THREADS = 320;                                // warp 0: TMA, warp 1: MMA, warps 2-9: drain
constexpr int TC2_STAGES = 6;
constexpr int TC2_STAGE_BYTES = TC_A_BYTES + TC_HALF_BYTES;     // 32 KB per CTA and stage
constexpr int TC2_SMEM = TC2_STAGES * TC2_STAGE_BYTES + 1024 + 256;
static_assert(TC2_SMEM >= kAloneBytes);

// Tile order of the two-SM kernel: groups of kTileGroupN weight tiles; inside a group the row
// pairs are walked with the group's weight tiles innermost.  The ~74 clusters running at any
// moment then cover a few row pairs x the group's weight tiles, whose A and B blocks (tens of MB) stay in
// L2 while they are reused, instead of streaming the whole A matrix from HBM once per weight tile.
// With three or more row pairs the weight tiles are loaded with the evict-last policy like the rows: every row
// pair re-reads them, and with evict-first (right for the few-row launches, whose weights pass through once) they
// left L2 between two uses.  Measured on the 32-layer step of 14 752 rows per layer under the power cap: 209-216 ms
// -> 191-197 ms at a 100-150 MHz higher SM clock (gate/up moved 8.6 GB through HBM per launch for 0.5 GB of
// operands; the saved traffic is power the tensor cores get); groups of 16 weight tiles then beat 8 by 1-2 %
// (4, 24, 32, 48 are slower), and cutting the row pairs into L2-sized blocks as well changes nothing more.
constexpr int kTileGroupN = 16;
constexpr int kKeepWeightsFromPairs = 3;
constexpr double kPairEpilogueUs = 9;     // epilogue of a 256 x 256 tile (1024 columns of K, rounds 1 to 3 of gate/up: 19, 28, 37 us)
constexpr int kWholeTilesFromKB = 56;     // K blocks from which whole tiles were measured against cut ones (plan_gemm)
constexpr int kSmallHeadPairs = 3, kSmallHeadBlocks = 24;   // an LM head stays on the one-SM kernel up to: row pairs, K blocks per CTA
constexpr int kPrepKernelRows = 4096;     // from this many rows the row preparation is a kernel of its own
// Ten warps leave a thread 168 registers.  With the rotary pairs finished 32 at a time and the whole gain requested early, 300
// bytes were spilled; 16 at a time and half of the gain, 52: layer-step of 615 rows 369.5 -> 366.4 us, 5 x 203 rows 515 -> 509,
// 64 x 103 rows 2666 -> 2629, refresh of 14 752 rows 12 286 -> 12 181.
__global__ void __launch_bounds__(TC2_THREADS, 1)
gemm_tc2_kernel(const GemmArgs g, const TcPlan p, const int clusters, const __grid_constant__ CUtensorMap mapA,
                const __grid_constant__ CUtensorMap mapB0, const __grid_constant__ CUtensorMap mapB1,
                const __grid_constant__ CUtensorMap mapB2) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ float red[TC2_THREADS / 32];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char* base_ptr = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t bars = base + TC2_STAGES * TC2_STAGE_BYTES;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + TC2_STAGES * TC2_STAGE_BYTES + 192);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + TC2_STAGES * TC2_STAGE_BYTES + 200);
    auto full_bar = [&](int s) { return bars + 8 * s; };
    auto empty_bar = [&](int s) { return bars + 8 * (TC2_STAGES + s); };
    auto tfull_bar = [&](int i) { return bars + 8 * (2 * TC2_STAGES + i); };
    auto tempty_bar = [&](int i) { return bars + 8 * (2 * TC2_STAGES + 2 + i); };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int cluster_id = blockIdx.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < TC2_STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(tfull_bar(i), 1); mbar_init(tempty_bar(i), 16); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;"
                     ::"r"(smem_u32(const_cast<uint32_t*>(tmem_slot))) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();          // the peer's barriers are initialised before anyone signals them
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_wait();
    pdl_launch_dependents();

    if (g.prep.enabled) prep_phase<true>(g, red, abort_flag, gridDim.x);

    const int m_pairs = (p.m_tiles + 1) >> 1;
    const int tiles = m_pairs * p.n_tiles;

    if (warp == 0) {
        // TMA producer of this CTA: its 128 rows of A and its half of the weight tile
        int stage = 0, issued = 0;
        uint32_t phase = 0;
        bool ok = __all_sync(0xffffffffu, !*abort_flag);
        const uint64_t pol_a = policy_evict_last();
        const uint64_t pol_w = (g.keep_weights || p.w_keep) ? pol_a : policy_evict_first();
        // work list: whole tiles round-robin (pair_u == 0), or this cluster's contiguous range of
        // (tile, K block) iterations, tiles in weight-tile-major order (stream-K)
        const long long it_end = p.pair_u ? min((long long)(cluster_id + 1) * p.pair_u, (long long)tiles * p.KB) : 0;
        long long it = p.pair_u ? (long long)cluster_id * p.pair_u : 0;
        for (int t = p.pair_u ? (int)(it / p.KB) : cluster_id; ok && (p.pair_u ? it < it_end : t < tiles);) {
            int nt, mp;
            if (p.pair_u) { nt = t / m_pairs; mp = t - nt * m_pairs; } else tile_coords(t, m_pairs, p.n_tiles, p.group_n, nt, mp);
            const int kb0 = p.pair_u ? (int)(it - (long long)t * p.KB) : 0;
            const int kb1 = p.pair_u ? (int)min((long long)p.KB, (long long)(kb0 + (it_end - it))) : p.KB;
            int brow;
            const int bs = half_source(g, p, nt, (int)rank, brow);
            const CUtensorMap* map_b = bs == 0 ? &mapB0 : bs == 1 ? &mapB1 : &mapB2;
            const int arow = (mp * 2 + (int)rank) * TC_BM;
            for (int kb = kb0; kb < kb1; ++kb) {
                // The first round of the ring and the first two accumulators are free: polled all the same, by the whole warp, they cost
                // a launch of a few K blocks 0.05-0.1 us (refresh of 4 x 307 rows of 256 columns, 4 layers, 313.8 -> 312.8).
                if (issued >= TC2_STAGES && !(ok = __all_sync(0xffffffffu, mbar_poll(empty_bar(stage), phase ^ 1, abort_flag)))) break;
                if (elect_lane()) {
                    const uint32_t sA = base + stage * TC2_STAGE_BYTES, sB = sA + TC_A_BYTES;
                    const uint32_t lead_full = mapa_u32(full_bar(stage), 0);
                    // the leader announces the bytes of both CTAs; the peer's copies only report completion
                    if (rank == 0) mbar_expect_tx(full_bar(stage), 2 * TC2_STAGE_BYTES);
                    tma_load_2d_pair(sA, &mapA, kb * TC_BK, arow, lead_full, pol_a);
                    tma_load_2d_pair(sB, map_b, kb * TC_BK, brow, lead_full, pol_w);
                }
                __syncwarp();
                ++issued;
                if (++stage == TC2_STAGES) { stage = 0; phase ^= 1; }
            }
            if (p.pair_u) { it += kb1 - kb0; ++t; } else t += clusters;
        }
        // wait until the MMAs have consumed everything this CTA loaded, so that no signal from the
        // leader can arrive after this CTA has left
        if (issued < TC2_STAGES) { stage = 0; phase = 1; }
        for (int i = 0; i < min(issued, TC2_STAGES) && ok; ++i) {
            ok = __all_sync(0xffffffffu, mbar_poll(empty_bar(stage), phase ^ 1, abort_flag));
            if (++stage == TC2_STAGES) { stage = 0; phase ^= 1; }
        }
    } else if (warp == 1 && rank == 0) {
        // MMA issuer (leader CTA only): the whole warp runs the loop, an elected lane issues, and the full barrier is polled at
        // CTA scope (a poll that acquires at cluster scope costs more than the data's own proxy needs).  With one lane in the loop
        // a K block took 540-630 cycles whatever the tile's width, of which the four instructions need 512: what bounded the loop was
        // the issue.  Back to back: 64 x 103 rows 2693 -> 2574 us, refresh of 14 752 rows 12 468 -> 12 112 (q/k/v 1209 -> 1043,
        // output 442 -> 375 a launch), probe of 20 480 rows 16 876 -> 16 341, 615 rows 374.7 -> 368.0; cluster-scope polls in the
        // same loop: refresh 12 400.
        int stage = 0, acc = 0, started = 0;
        uint32_t phase = 0, acc_phase = 0;
        bool ok = __all_sync(0xffffffffu, !*abort_flag);
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(256 >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
        const long long it_end = p.pair_u ? min((long long)(cluster_id + 1) * p.pair_u, (long long)tiles * p.KB) : 0;
        long long it = p.pair_u ? (long long)cluster_id * p.pair_u : 0;
        for (int t = p.pair_u ? (int)(it / p.KB) : cluster_id; ok && (p.pair_u ? it < it_end : t < tiles);) {
            const int kb0 = p.pair_u ? (int)(it - (long long)t * p.KB) : 0;
            const int kb1 = p.pair_u ? (int)min((long long)p.KB, (long long)(kb0 + (it_end - it))) : p.KB;
            if (started++ >= 2 && !(ok = __all_sync(0xffffffffu, mbar_poll_cluster(tempty_bar(acc), acc_phase ^ 1, abort_flag)))) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + acc * TC_BN;
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!(ok = __all_sync(0xffffffffu, mbar_poll(full_bar(stage), phase, abort_flag)))) break;
                tc_fence_after();
                if (elect_lane()) {
                    const uint32_t sA = base + stage * TC2_STAGE_BYTES, sB = sA + TC_A_BYTES;
                    const uint64_t da = smem_desc_sw128(sA), db = smem_desc_sw128(sB);
#pragma unroll
                    for (int k = 0; k < TC_BK / 16; ++k)
                        tc2_mma(d_tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc, (kb > kb0 || k > 0) ? 1u : 0u);
                    tc2_commit_both(empty_bar(stage));
                    if (kb + 1 == kb1) tc2_commit_both(tfull_bar(acc));
                }
                __syncwarp();
                if (++stage == TC2_STAGES) { stage = 0; phase ^= 1; }
            }
            if (!ok) break;
            if (++acc == 2) { acc = 0; acc_phase ^= 1; }
            if (p.pair_u) { it += kb1 - kb0; ++t; } else t += clusters;
        }
    } else if (warp >= 2) {
        // drain: this CTA's 128 rows of the tile, epilogue straight from TMEM; two warps per lane quarter, 128 columns each
        const int q = warp & 3, hf = (warp - 2) >> 2;
        const int row = q * 32 + lane;
        int acc = 0;
        uint32_t acc_phase = 0;
        bool ok = !*abort_flag;
        const long long it_end = p.pair_u ? min((long long)(cluster_id + 1) * p.pair_u, (long long)tiles * p.KB) : 0;
        long long it = p.pair_u ? (long long)cluster_id * p.pair_u : 0;
        const long long it_first = it;
        const uint64_t pol_p = policy_evict_last();
        for (int t = p.pair_u ? (int)(it / p.KB) : cluster_id; ok && (p.pair_u ? it < it_end : t < tiles);) {
            int nt, mp;
            if (p.pair_u) { nt = t / m_pairs; mp = t - nt * m_pairs; } else tile_coords(t, m_pairs, p.n_tiles, p.group_n, nt, mp);
            const int kb0 = p.pair_u ? (int)(it - (long long)t * p.KB) : 0;
            const int kb1 = p.pair_u ? (int)min((long long)p.KB, (long long)(kb0 + (it_end - it))) : p.KB;
            const int grow = (mp * 2 + (int)rank) * TC_BM + row;
            const bool is_whole = kb0 == 0 && kb1 == p.KB;
            HalfPre pre;
            if (is_whole) half_prefetch(g, nt, hf, grow, grow < g.M, pre);
            if (!(ok = mbar_wait(tfull_bar(acc), acc_phase, abort_flag))) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + acc * TC_BN + ((uint32_t)(q * 32) << 16);
            if (is_whole) {
                half_epilogue(g, p, taddr, nt, hf, 2, grow, grow < g.M, pre);
            } else {
                // a tile whose K range is cut between clusters: this CTA's 128 rows to its fp32 partial slot
                float4* dst = reinterpret_cast<float4*>(g.partial) +
                              (((int64_t)cluster_id * 2 + (it == it_first ? 0 : 1)) * 2 + rank) * (TC_SLOT_FLOATS / 4);
                for (int c = hf * 4; c < hf * 4 + 4; ++c) {
                    float v[32];
                    tc_ld32(taddr + c * 32, v);
                    if (grow < g.M) {
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            st_hint_f4(&dst[(c * 8 + i) * TC_BM + row], make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]), pol_p);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(mapa_u32(tempty_bar(acc), 0));
            if (++acc == 2) { acc = 0; acc_phase ^= 1; }
            if (p.pair_u) { it += kb1 - kb0; ++t; } else t += clusters;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0) {
            atomicOr(g.status, kFlagWaitExpired);
            for (int i = 0; i < 4096; ++i) __nanosleep(64);
        }
        __syncthreads();
    }
    cluster_sync_all();          // neither CTA leaves while its peer may still signal it
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

// Finish of the split tiles: grid row y finishes tile split.tile[y]; blockIdx.x * 256 +
// threadIdx.x -> (item, row).

__global__ void __launch_bounds__(256, 2) gemm_finish_kernel(const GemmArgs g, const TcPlan p, const SplitTiles split) {
    const int t = split.tile[blockIdx.y];
    const int mt = t % p.m_tiles;
    const int rows_per = p.m_tiles == 1 ? ((g.M + 31) & ~31) : TC_BM;
    const int w = blockIdx.x * 256 + threadIdx.x;
    const int row = w % rows_per, item = w / rows_per;
    const bool active = item < finish_items_per_tile(g.epilogue) && mt * TC_BM + row < g.M;
    // The residual rows and their offsets are outputs of kernels that had completed before the projection
    // whose tiles are finished here passed its own dependency wait, and this kernel starts after that: they can
    // be requested while the projection is still running.
    uint4 res[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
    FinishItem f{};
    if (active) {
        f = finish_plan(g, p, t, item, row);
        if (g.epilogue == kEpiResidual && !f.skip) load_residual16(g, f.grow, f.nt * TC_BN + item * 16, res);
    }
    pdl_wait();
    pdl_launch_dependents();
    if (!active) return;
    finish_item(g, p, t, item, row, f, res);
}

// ---- predict and commit (Eq. 2-3): confidence and arg max per row, commit rule per request ------
struct LogitAcc { float m, s; int arg; };
// Branch-free (lanes hold different tiles); an empty entry is m = -FLT_MAX, s = 0.  The lowest index wins a tie.
__device__ __forceinline__ void logit_merge(LogitAcc& a, float m, float s, int arg) {
    const float nm = fmaxf(a.m, m);
    a.s = a.s * __expf(a.m - nm) + s * __expf(m - nm);
    a.arg = m > a.m || (m == a.m && arg < a.arg) ? arg : a.arg;
    a.m = nm;
}
__device__ __forceinline__ void logit_merge_warp(LogitAcc& a, int width) {
#pragma unroll 1
    for (int o = width >> 1; o > 0; o >>= 1) {
        const float m = __shfl_xor_sync(0xffffffffu, a.m, o), sm = __shfl_xor_sync(0xffffffffu, a.s, o);
        logit_merge(a, m, sm, __shfl_xor_sync(0xffffffffu, a.arg, o));
    }
}

// One CTA per row: merges the per-tile statistics (16 entries for a tile whose K range was split between CTAs, one or two
// otherwise; the first one's w says how many) in a fixed order.  Bound by the latency of L2 and the instructions per entry:
// a thread takes a tile's first entry (and second); then half a warp takes one of the cut tiles, which the launch lists, a lane
// per entry.  32 rows x 126 464 logits with 147 cut tiles: 17.5 -> 9.7 us against reading sixteen entries of every tile.
constexpr int LR_THREADS = 512;
__global__ void __launch_bounds__(LR_THREADS) logit_reduce_kernel(const GemmArgs g, const TcPlan p, const SplitTiles split,
                                                                  int32_t* __restrict__ token, float* __restrict__ confidence) {
    __shared__ LogitAcc part[32];
    const int row = blockIdx.x, mt = row / TC_BM, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, entry = lane & 15;
    const LogitAcc empty{-3.402823466e38f, 0.f, 0x7fffffff};
    if (threadIdx.x < 32) part[threadIdx.x] = empty;
    pdl_wait();
    pdl_launch_dependents();
    LogitAcc a = empty;
#pragma unroll 1
    for (int nt = threadIdx.x; nt < p.n_tiles; nt += LR_THREADS) {
        const float4 v = __ldcg(logit_entry(g, nt, 0, row)), u = __ldcg(logit_entry(g, nt, 1, row));
        const bool one = v.w <= 2.f, two = v.w == 2.f;
        logit_merge(a, one ? v.x : empty.m, one ? v.y : 0.f, one ? __float_as_int(v.z) : empty.arg);
        logit_merge(a, two ? u.x : empty.m, two ? u.y : 0.f, two ? __float_as_int(u.z) : empty.arg);
    }
#pragma unroll 4
    for (int i = threadIdx.x >> 4; i < split.n; i += LR_THREADS / 16) {
        const int nt = split.tile[i] / p.m_tiles;
        const bool use = nt * p.m_tiles + mt == split.tile[i] && nt * 2 + (entry >> 3) < p.units;
        const float4 v = __ldcg(logit_entry(g, nt, entry, row));
        logit_merge(a, use ? v.x : empty.m, use ? v.y : 0.f, use ? __float_as_int(v.z) : empty.arg);
    }
    logit_merge_warp(a, 32);
    __syncthreads();
    if (lane == 0) part[warp] = a;
    __syncthreads();
    if (warp == 0) {
        a = part[lane];
        logit_merge_warp(a, LR_THREADS / 32);
        if (lane == 0) {
            token[row] = a.arg;
            confidence[row] = 1.f / a.s;       // softmax probability of the arg max
        }
    }
}

// One warp per request: commit the rows above the threshold, or the single most confident row
// (lowest index on ties) if there is none.
__global__ void __launch_bounds__(32) commit_kernel(const float* __restrict__ confidence, int n_blk, float threshold,
                                                    int32_t* __restrict__ commit) {
    pdl_wait();
    pdl_launch_dependents();
    const int b = blockIdx.x, lane = threadIdx.x;
    const float* c = confidence + (int64_t)b * n_blk;
    int32_t* out = commit + (int64_t)b * n_blk;
    int any = 0, best = 0x7fffffff;
    float bestc = -INFINITY;
    for (int i = lane; i < n_blk; i += 32) {
        const float v = __ldcg(c + i);
        const int f = v > threshold;
        out[i] = f;
        any |= f;
        if (v > bestc) { bestc = v; best = i; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        any |= __shfl_xor_sync(0xffffffffu, any, o);
        const float oc = __shfl_xor_sync(0xffffffffu, bestc, o);
        const int ob = __shfl_xor_sync(0xffffffffu, best, o);
        if (oc > bestc || (oc == bestc && ob < best)) { bestc = oc; best = ob; }
    }
    if (!any && lane == 0 && best < n_blk) out[best] = 1;
}

// ---- host side ------------------------------------------------------------------------------
namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

struct MapKey { const void* ptr; int rows, cols, box_rows, panels, half; int64_t step = 0; };
struct MapEntry { MapKey key; CUtensorMap map; };
// A weight matrix has an entry for each kernel that has read it (up to 128 rows, cut tiles, weights as M, where gate and up share one):
// some 640 for a 32-layer model at mixed row counts; an input has one per row count and box.  A miss encodes the map again.  Host
// time of a launch (32 layers, 228 launches, 300 calls of 40 to 932 rows): 2.7 us, as without the weights-as-M maps.
constexpr int kMapCache = 1024;
MapEntry g_maps[kMapCache];
int g_map_count = 0, g_map_next = 0;

const CUtensorMap* lookup_map(const MapKey& want, int rank, const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box) {
    for (int i = 0; i < g_map_count; ++i) {
        const MapKey& k = g_maps[i].key;
        if (k.ptr == want.ptr && k.rows == want.rows && k.cols == want.cols && k.box_rows == want.box_rows &&
            k.panels == want.panels && k.half == want.half && k.step == want.step)
            return &g_maps[i].map;
    }
    EncodeTiledFn fn = encode_fn();
    if (!fn) return nullptr;
    MapEntry& e = g_maps[g_map_next];
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    if (fn(&e.map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(want.ptr), dims, strides, box, estr,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return nullptr;
    e.key = want;
    g_map_next = (g_map_next + 1) % kMapCache;
    if (g_map_count < kMapCache) ++g_map_count;
    return &e.map;
}

}  // namespace

std::mutex g_map_mutex;

// bf16 [rows, cols] row-major, box = box_rows rows x 64 cols, 128-byte swizzle, zero fill out of bounds; like every lookup here,
// the pointer is only good until the next one (a miss may replace any entry): callers copy the map.
const CUtensorMap* get_rows_map(const void* ptr, int rows, int cols, int box_rows) {
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows}, strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    return lookup_map(MapKey{ptr, rows, cols, box_rows, 0, 0}, 2, dims, strides, box);
}

const CUtensorMap* get_weight_map(const void* ptr, int rows, int cols, WeightOrder order, int64_t step) {
    const cuuint64_t row = (cuuint64_t)cols * 2, k = (cuuint64_t)cols, n = (cuuint64_t)rows;
    const MapKey key{ptr, rows, cols, 128, -(int)order, 0, step};
    struct Shape { cuuint64_t dims[5], strides[4]; cuuint32_t box[5]; };
    const Shape s = order == kWeightsPlain   ? Shape{{k, 128, 1, 1, n / 128}, {row, row * 128, row * 128, row * 128}, {64, 128, 1, 1, 1}}
                  : order == kWeightsRope128 ? Shape{{k, 16, 2, 4, n / 128}, {row, row * 64, row * 16, row * 128}, {64, 16, 2, 4, 1}}
                  : order == kWeightsRope64  ? Shape{{k, 16, 2, 2, n / 64}, {row, row * 32, row * 16, row * 64}, {64, 16, 2, 2, 2}}
                                             : Shape{{k, 16, 2, 4, n / 64}, {row, (cuuint64_t)step, row * 16, row * 64}, {64, 16, 2, 4, 1}};
    return lookup_map(key, 5, s.dims, s.strides, s.box);
}

const CUtensorMap* get_panel_map(const void* ptr, int rows, int cols, int box_rows, int panels, int half) {
    const cuuint64_t row = (cuuint64_t)cols * 2;
    const MapKey key{ptr, rows, cols, box_rows, panels, half};
    if (half) {
        const cuuint64_t dims[4] = {64, (cuuint64_t)half, (cuuint64_t)(rows / half), (cuuint64_t)(cols / 64)};
        const cuuint64_t strides[3] = {row, row * half, 128};
        const cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 2, (cuuint32_t)panels};
        return lookup_map(key, 4, dims, strides, box);
    }
    const cuuint64_t dims[3] = {64, (cuuint64_t)rows, (cuuint64_t)(cols / 64)};
    const cuuint64_t strides[2] = {row, 128};
    const cuuint32_t box[3] = {64, (cuuint32_t)box_rows, (cuuint32_t)panels};
    return lookup_map(key, 3, dims, strides, box);
}

int sm_count() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 148;
    }
    return n;
}

namespace {

TcPlan make_plan(int M, int K, int units, bool swiglu) {
    TcPlan p{};
    p.units = units;
    p.m_tiles = (M + TC_BM - 1) / TC_BM;
    p.n_tiles = swiglu ? units : (units + 1) / 2;
    p.KB = K / TC_BK;
    p.tiles = p.m_tiles * p.n_tiles;
    const int64_t total = (int64_t)p.tiles * p.KB;
    const int g = (int)(total < sm_count() ? total : sm_count());
    p.U = (int)((total + g - 1) / g);
    p.ctas = (int)((total + p.U - 1) / p.U);
    // measured: 174.9 us per layer-step of 103 rows with no stage prefilled, 169.1 with two, 167.9-168.6 with three or four
    p.prefill = TC_STAGES;
    return p;
}

// How a projection is launched: kernel, work split and the tiles that the finish kernel completes.
struct GemmLaunch {
    TcPlan p;
    bool pair;                // gemm_tc2_kernel
    int clusters, max_clusters;
    SplitTiles split;
};

cudaLaunchConfig_t pair_config(cudaLaunchAttribute* at, int clusters, cudaStream_t stream) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(clusters * 2);
    cfg.blockDim = dim3(TC2_THREADS);
    cfg.dynamicSmemBytes = TC2_SMEM;
    cfg.stream = stream;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cfg;
}

// Clusters of the two-SM kernel that are resident at once (phase 0 ends in a grid-wide barrier); 0: none fits.
int pair_max_clusters() {
    static const int n = [] {
        cudaFuncSetAttribute(gemm_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
        cudaFuncSetAttribute(gemm_tc2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TC2_SMEM);
        cudaLaunchAttribute at[2];
        const cudaLaunchConfig_t cfg = pair_config(at, sm_count() / 2, nullptr);
        int c = 0;
        if (cudaOccupancyMaxActiveClusters(&c, gemm_tc2_kernel, &cfg) != cudaSuccess || c < 0) {
            (void)cudaGetLastError();
            c = 0;
        }
        return std::min(c, sm_count() / 2);
    }();
    return n;
}

GemmLaunch plan_gemm(const GemmArgs& g) {
    const bool swiglu = g.epilogue == kEpiSwiGLU;
    const int n_total = swiglu ? g.n[0] : g.n[0] + g.n[1] + g.n[2];
    GemmLaunch gl{};
    gl.p = make_plan(g.M, g.K, n_total / 128, swiglu);
    TcPlan& p = gl.p;
    // Two or more row tiles: two SMs per 256 x 256 tile.  With many tiles per cluster every tile is whole
    // and the clusters walk them round-robin; with few, the (tile, K block) iterations are cut into equal
    // contiguous ranges, one per cluster (stream-K), and the cut tiles go through the finish kernel.
    // The LM head comes here as well: on the one-SM kernel, which reads every weight tile once per 128 rows and moves twice
    // the shared-memory bytes per flop, 512 rows x 126 464 x 4096 took 670 us with its finish, here 379 us (decode
    // pass of 16 requests, 4 layers: 2349 -> 2025 us).  Except a small one, whose tiles would be cut here, over few rows
    // (us with its row preparation and reduction, one SM | two: 512 rows x 2048 x 256 21.5 | 24.2, 129 x 2560 x 2048
    // 22.2 | 27.3, 700 x 2048 x 1024 32.2 | 36.4, 700 x 2048 x 4096 (21 K blocks per CTA) 41.5 | 44.7; but 512 x 4096 x 4096
    // (28) 43.9 | 42.4, 1300 x 2048 x 256 (six row pairs) 43.7 | 35.4, and whole tiles, 160 x 16384 x 4096, 59.0 | 42.4).
    static const int pair_min_tiles = [] { const char* e = getenv("ACACHE_GEMM_PAIR_MIN_MTILES"); return e ? atoi(e) : 2; }();
    const int max_clusters = pair_max_clusters();
    static const int stream_k_pct = [] { const char* e = getenv("ACACHE_GEMM_PAIR_STREAMK_PCT"); return e ? atoi(e) : 66; }();
    const int m_pairs = (p.m_tiles + 1) / 2;
    const int tiles = m_pairs * p.n_tiles;
    const bool below_cut = tiles * 100 <= stream_k_pct * max_clusters;
    const bool small_head = g.epilogue == kEpiLogits && below_cut && m_pairs <= kSmallHeadPairs && p.U <= kSmallHeadBlocks;
    if (p.m_tiles >= pair_min_tiles && (p.units % 2 == 0 || swiglu) && max_clusters >= 1 && !small_head) {
        gl.pair = true;
        p.m_pairs = m_pairs;
        static const int group_n = [] { const char* e = getenv("ACACHE_GEMM_GROUP_N"); return e && atoi(e) > 0 ? atoi(e) : kTileGroupN; }();
        p.group_n = group_n;
        static const int w_keep_from = [] { const char* e = getenv("ACACHE_GEMM_WKEEP_PAIRS"); return e ? atoi(e) : kKeepWeightsFromPairs; }();
        gl.clusters = std::min(max_clusters, tiles);
        gl.max_clusters = max_clusters;
        // Cutting tiles pays up to about two thirds of a wave, unless K is so short that the finish costs what the shorter main
        // loop gains: of a whole tile's time the cut loop took 0.66-0.70 at 0.44 of its K blocks and 0.83-0.90 at 0.65 (partial
        // tiles included), the finish that of about 20 K blocks.  (us, whole | cut + finish: 512 rows output 32.0 | 22.3 + 7.3,
        // down 67.1 | 43.0 + 7.1; 615 rows output 31.3 | 27.9 + 9.3, down 73.5 | 61.0 + 9.5.)  Below half a wave always: whole tiles
        // leave too few CTAs for the row preparation (refresh of 166 rows of 256 columns 199.8 us cut, 203.3 whole).
        // Below 3584 columns (kWholeTilesFromKB) always too, although whole tiles are faster there (refresh of 1100 rows of 256
        // columns, 4 layers: 299 us whole, 324 cut): whole tiles add the K blocks in another order, no less precise, but narrow
        // models predict from near ties (1-2.5 % of the tokens of such passes changed).  (Not the LM head: its logits stay fp32, and
        // 780 rows x 2560 x 2048 took 35.8 us whole, 41.3 cut.)
        const int64_t total = (int64_t)tiles * p.KB;
        if (below_cut &&
            ((p.KB < kWholeTilesFromKB && g.epilogue != kEpiLogits) || tiles * 2 < max_clusters || 1.05 * tiles / max_clusters + 20.0 / p.KB < 0.8)) {
            gl.clusters = (int)std::min<int64_t>(max_clusters, total);
            p.pair_u = (int)((total + gl.clusters - 1) / gl.clusters);
            gl.clusters = (int)((total + p.pair_u - 1) / p.pair_u);
            // pair tiles cut by a boundary between two clusters: both of their 128-row tiles go to the finish
            int last = -1;
            for (int c = 1; c < gl.clusters; ++c) {
                const int64_t cut = (int64_t)c * p.pair_u;
                if (cut % p.KB == 0) continue;
                const int tp = (int)(cut / p.KB);
                if (tp == last) continue;
                last = tp;
                const int nt = tp / m_pairs, mp = tp - nt * m_pairs;
                for (int r = 0; r < 2; ++r)
                    if (mp * 2 + r < p.m_tiles && gl.split.n < 160) gl.split.tile[gl.split.n++] = nt * p.m_tiles + mp * 2 + r;
            }
            if (gl.split.n >= 159) { p.pair_u = 0; gl.split.n = 0; gl.clusters = std::min(max_clusters, tiles); }
        }
        p.w_keep = (m_pairs >= w_keep_from && p.pair_u == 0) ? 1 : 0;      // whole tiles, walked by three or more row pairs
        return gl;
    }
    // tiles whose K range is cut by a boundary between two CTAs, each listed once
    for (int c = 1; c < p.ctas && gl.split.n < 160; ++c) {
        const int64_t cut = (int64_t)c * p.U;
        if (cut % p.KB == 0) continue;
        const int t = (int)(cut / p.KB);
        if (gl.split.n == 0 || gl.split.tile[gl.split.n - 1] != t) gl.split.tile[gl.split.n++] = t;
    }
    return gl;
}

}  // namespace

size_t gemm_partial_bytes(int M, int K, int n_total, bool swiglu) {
    (void)M; (void)K; (void)n_total; (void)swiglu;
    // two fp32 partial tiles per CTA, at most one CTA per SM, whatever the problem size
    return (size_t)sm_count() * 2 * TC_SLOT_FLOATS * sizeof(float);
}

static int launch_gemm_impl(const GemmArgs& g, cudaStream_t stream);

int launch_gemm(const GemmArgs& g, cudaStream_t stream) {
    if (g.M == 0) return 0;
    // many rows: the row preparation runs as a kernel of its own (ACACHE_GEMM_PREP_KERNEL_ROWS: from how many rows; 0: never)
    static const int prep_rows = [] { const char* e = getenv("ACACHE_GEMM_PREP_KERNEL_ROWS"); return e ? atoi(e) : kPrepKernelRows; }();
    if (g.prep.enabled && prep_rows > 0 && g.M >= prep_rows) {
        const int blocks = std::min((g.M + 7) / 8, sm_count() * 2);
        if (launch_pdl(prep_rows_kernel, dim3(blocks), dim3(256), 0, stream, g) != cudaSuccess) return -1;
        GemmArgs g2 = g;
        g2.prep.enabled = 0;
        const int nl = launch_gemm_impl(g2, stream);
        return nl < 0 ? nl : nl + 1;
    }
    return launch_gemm_impl(g, stream);
}

static int launch_gemm_impl(const GemmArgs& g, cudaStream_t stream) {
    if (const int n = launch_gemm_rows(g, stream)) return n;
    const bool swiglu = g.epilogue == kEpiSwiGLU;
    const GemmLaunch gl = plan_gemm(g);
    const TcPlan& p = gl.p;
    if (gl.pair && !p.pair_u) {
        // whole tiles, which are the same sums with the weights as the product's M, where that takes less time
        const int tiles = p.m_pairs * p.n_tiles, rounds = (tiles + gl.max_clusters - 1) / gl.max_clusters;
        if (const int n = launch_gemm_wm(g, rounds * pair_tile_us(p.KB, 256, kPairEpilogueUs), p.group_n, stream)) return n;
    }
    std::lock_guard<std::mutex> lock(g_map_mutex);
    CUtensorMap map_a, map_b[3];
    {
        const CUtensorMap* m = get_rows_map(g.a, g.M, g.K, TC_BM);
        if (!m) return -1;
        map_a = *m;
    }
    bool have_b[3] = {false, false, false};
    for (int i = 0; i < 3; ++i)
        if (g.b[i]) {
            const CUtensorMap* m = get_rows_map(g.b[i], swiglu ? g.n[0] : g.n[i], g.K, 128);
            if (m) { map_b[i] = *m; have_b[i] = true; }
        }
    if (!have_b[0]) return -1;
    const CUtensorMap* mA = &map_a;
    const CUtensorMap* mB[3] = {&map_b[0], have_b[1] ? &map_b[1] : &map_b[0], have_b[2] ? &map_b[2] : &map_b[0]};
    if (gl.pair) {
        cudaLaunchAttribute at[2];
        const cudaLaunchConfig_t cfg = pair_config(at, gl.clusters, stream);
        if (cudaLaunchKernelEx(&cfg, gemm_tc2_kernel, g, p, gl.clusters, *mA, *mB[0], *mB[1], *mB[2]) != cudaSuccess) return -1;
        if (gl.split.n == 0) return 1;
        const int per_tile = finish_items_per_tile(g.epilogue) * TC_BM;
        if (launch_pdl(gemm_finish_kernel, dim3((per_tile + 255) / 256, gl.split.n), dim3(256), 0, stream, g, p, gl.split) !=
            cudaSuccess)
            return -1;
        return 2;
    }
    // a plain launch: a cooperative one measured ~2.5 us slower and cannot overlap the previous
    // kernel's tail; the grid never exceeds the SM count at one CTA per SM and the barrier is bounded
    if (launch_pdl(gemm_tc_kernel, dim3(p.ctas), dim3(TC_THREADS), TC_SMEM, stream, g, p, *mA, *mB[0], *mB[1], *mB[2]) !=
        cudaSuccess)
        return -1;
    if (gl.split.n == 0) return 1;
    const int rows_per = p.m_tiles == 1 ? ((g.M + 31) & ~31) : TC_BM;
    const int per_tile = finish_items_per_tile(g.epilogue) * rows_per;
    if (launch_pdl(gemm_finish_kernel, dim3((per_tile + 255) / 256, gl.split.n), dim3(256), 0, stream, g, p, gl.split) != cudaSuccess)
        return -1;
    return 2;
}

int launch_predict_commit(const GemmArgs& g, int batch, int n_blk, float threshold, int32_t* token, float* confidence,
                          int32_t* commit, cudaStream_t stream) {
    if (g.M == 0) return 0;
    const GemmLaunch gl = plan_gemm(g);
    if (launch_pdl(logit_reduce_kernel, dim3(g.M), dim3(LR_THREADS), 0, stream, g, gl.p, gl.split, token, confidence) != cudaSuccess) return -1;
    if (launch_pdl(commit_kernel, dim3(batch), dim3(32), 0, stream, (const float*)confidence, n_blk, threshold, commit) !=
        cudaSuccess)
        return -1;
    return 2;
}

}  // namespace acache
