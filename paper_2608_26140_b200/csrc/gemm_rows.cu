// Projections of few rows (C[M, N] = A[M, K] B[N, K]^T with M <= 128) as one launch without partial tiles in global memory.
//
// At these sizes the weights' stream from HBM is the floor and everything around it is latency.  The general one-SM kernel
// (gemm_tc.cu) cuts (tile, K block) ranges so that every SM streams the same bytes, and pays with fp32 partial tiles through
// L2 and a finish kernel behind every projection.  Here a tile of TN weight rows (TN chosen from N, not fixed) belongs to
// one CTA or to a cluster of S = 2 or 4 CTAs that split K; every CTA sends its partial accumulators to the CTA that finishes
// their columns (asynchronous stores into its shared memory, counted by an mbarrier there), and the epilogue follows in the same
// kernel.
//
// Small projections (the general kernel would give every CTA one K block) keep its order of sums: every block of 64 K columns
// has an accumulator of its own in tensor memory, and they are added in ascending order, a CTA of a cluster handing over its
// blocks one by one.  A row's result is then what the general kernel gives, whatever the tile, the split and the number of
// rows: narrow models predict from near ties (2-4 % of the rows of a 256-column model with 2048 tokens have a second choice
// within 0.02 of the first), which another order of sums, though no less precise, decides differently.  Price: layer-step of
// 58 rows of 256 columns 51.2 -> 53.1 us (the sums' code is a loop over the blocks: unrolled by four, its instructions' way
// from L2 made that 54.3).
//
// A ring stage holds CP panels of 64 K columns, loaded by one TMA instruction per operand box (3-d and 4-d tensor maps: the
// panel is a dimension of the box), so that a stage's fixed cost of waits and issue is shared by more bytes.
//
// Roles of the 256 threads: warp 0 TMA producer, warp 1 tcgen05.mma issuer, then all eight warps the epilogue (warp = TMEM
// lane quarter x column half).  All eight take part in the row preparation before (prep_phase).  Every wait on an mbarrier
// or the grid barrier is bounded as in gemm_tc.cu; the cluster barriers are passed by every CTA whatever happened before.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "gemm_common.cuh"
#include "kernels.h"
#include "launch.h"
#include "tc_ptx.cuh"

namespace acache {

constexpr int RW_THREADS = 256;
constexpr int RW_MAX_STAGES = 16;
constexpr int RW_MAX_UNITS = 4;

struct RowsPlan {
    int TN, n_tiles;
    int CP, blocks;           // K panels (64 columns) per ring stage, stages' worth of K in all
    int S;                    // CTAs per tile, splitting K
    int rows_pad;             // M rounded up to 8: rows of an A panel
    int R, n_units;           // weight rows per box, boxes per stage
    int mma_n, mma_count;     // columns per instruction, instructions per 16 K columns (one panel: the boxes lie side by side)
    int KB, apart;            // K blocks of 64; 1: an accumulator per K block, added in order
    int cta_rows;             // row preparation: a whole CTA per row up to this many rows, a warp above (rows of more than 256
                              // columns are then summed in another order: apart, as many as the general kernel would take)
    int stages, stage_bytes;
    int tmem_cols;
    int groups;               // q/k/v: groups of 32 rotary pairs over all segments
    int own_rows;             // every CTA prepares all rows itself, straight into its ring (own_row_prep)
    int recv_off, recv_late;  // where the peers' partial accumulators arrive, from the ring's start on; 1: in the ring itself
    int smem_bytes;
};

__device__ __forceinline__ void tc_ld8x2(uint32_t ta, uint32_t tb, float (&a)[8], float (&b)[8]) {
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(ta)
                 : "memory");
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(tb)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) { a[i] = __uint_as_float(r[i]); b[i] = __uint_as_float(r[8 + i]); }
}
__device__ __forceinline__ float4 ld_shared_f4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
// Four floats into another CTA's shared memory; its mbarrier counts the bytes as they arrive.
__device__ __forceinline__ void send_f4(uint32_t cluster_addr, const float* v, uint32_t cluster_bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(cluster_addr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "r"(cluster_bar)
                 : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c1, int c2, uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1, {%2, %3, %4}], [%5], %6;"
        ::"r"(dst), "l"(map), "r"(0), "r"(c1), "r"(c2), "r"(bar), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c1, int c2, int c3, uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
        ::"r"(dst), "l"(map), "r"(0), "r"(c1), "r"(c2), "r"(c3), "r"(bar), "l"(policy)
        : "memory");
}

// q/k/v: segment of the grp-th group of 32 rotary pairs, row of its first pair inside the segment (the partners sit
// head_dim / 2 rows further).
__device__ __forceinline__ int pair_group(const GemmArgs& g, int grp, int& row) {
    int r = g.head_dim == 128 ? (grp >> 1) * 128 + (grp & 1) * 32 : grp * 64;
    int seg = 0;
    while (seg < 2 && r >= g.n[seg]) { r -= g.n[seg]; ++seg; }
    row = r;
    return seg;
}

// The boxes of weight rows of tile `nt`.  q/k/v: a box is the two halves of a group, 32 rows each (past the last group the
// last one is loaded again and ignored); SwiGLU: gate rows, then as many up rows; residual: the tile's rows.  Rows past a
// matrix's end read as zero.
template <int EPI>
struct WeightBoxes {
    int seg[RW_MAX_UNITS], row[RW_MAX_UNITS];
    __device__ __forceinline__ WeightBoxes(const GemmArgs& g, const RowsPlan& p, int nt) {
#pragma unroll
        for (int u = 0; u < RW_MAX_UNITS; ++u) {
            if (EPI == kEpiQKV) seg[u] = pair_group(g, min(nt * p.n_units + u, p.groups - 1), row[u]);
            else { seg[u] = EPI == kEpiSwiGLU ? u : 0; row[u] = nt * p.R; }
        }
    }
};

// K blocks of 64 that rank r of a cluster multiplies.
template <int S>
__device__ __forceinline__ int rank_panels(const RowsPlan& p, int r) {
    return min((r + 1) * p.blocks / S * p.CP, p.KB) - r * p.blocks / S * p.CP;
}

// 16 adjacent accumulator columns of this thread's row, summed over the cluster: own tensor memory first, then the peers' parts in
// rank order (fixed, hence bitwise reproducible).  slice_col: the columns' place inside the slice this CTA finishes; recv: where
// the first peer's part of it lies in shared memory, `region` bytes from one peer to the next.
template <int S>
__device__ __forceinline__ void sum_cluster16(uint32_t taddr, uint32_t recv, int region, int slice_col, int rows_pad, int row,
                                              float (&v)[16]) {
    tc_ld16(taddr, v);
    const int r = min(row, rows_pad - 1);
#pragma unroll
    for (int i = 0; i < S - 1; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 t = ld_shared_f4(recv + i * region + ((((slice_col >> 2) + j) * rows_pad + r) << 4));
            v[4 * j] += t.x; v[4 * j + 1] += t.y; v[4 * j + 2] += t.z; v[4 * j + 3] += t.w;
        }
}

// The same 16 columns where every K block has its own accumulator: all blocks of the tile in ascending order, rank by rank.
// per_block: bytes between a peer's blocks.
template <int S>
__device__ __forceinline__ void sum_apart16(const RowsPlan& p, int rank, uint32_t taddr, uint32_t recv, int region, int slice_col,
                                            int per_block, int row, float (&v)[16]) {
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = 0.f;
    const int r = min(row, p.rows_pad - 1);
#pragma unroll
    for (int c = 0; c < S; ++c) {
        const int nb = rank_panels<S>(p, c);
        if (c == rank) {
#pragma unroll 1
            for (int i = 0; i < nb; ++i) {
                float t[16];
                tc_ld16(taddr + i * p.TN, t);
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] += t[j];
            }
        } else if (S > 1) {
            const uint32_t src = recv + (c < rank ? c : c - 1) * region + (((slice_col >> 2) * p.rows_pad + r) << 4);
#pragma unroll 1
            for (int i0 = 0; i0 < nb; i0 += 4) {
                float4 t[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) t[i][j] = ld_shared_f4(src + min(i0 + i, nb - 1) * per_block + ((j * p.rows_pad) << 4));
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (i0 + i < nb) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            v[4 * j] += t[i][j].x; v[4 * j + 1] += t[i][j].y; v[4 * j + 2] += t[i][j].z; v[4 * j + 3] += t[i][j].w;
                        }
                    }
            }
        }
    }
}

// The shared preparation of the usual case (a CTA per row, a row of up to three 16-byte pieces a thread) and, out of the way of its
// instructions, the rest: a launch runs most of its instructions once, from L2, and waits for them.  With all of it inline the
// kernels had 228-252 registers; those with one accumulator per tile now have 48-210, those with one per block keep it inline and
// have 230-252 (layer-step of 103 rows 142.6 -> 139.1 us, decode pass of 32 rows over 4 layers 638 -> 631).  The call gets a copy of the
// arguments, made on that way only: it takes their address, and a kernel whose parameter has one (as __grid_constant__) reads it more
// slowly everywhere (decode pass of 78 rows of 256 columns over 2 layers 89.4 -> 88.2 us, layer-step of 58 such rows 46.6 -> 46.0, of
// 103 rows of 4096 columns 134.8 -> 134.3; one that copies it at its start: the last 138.6).
__device__ __forceinline__ void prep_phase_short(const GemmArgs& g, float* red, volatile int* abort_flag) {
    const RowPrep& rp = g.prep;
    for (int row = blockIdx.x; row < g.M; row += gridDim.x) {
        const int64_t src = prep_row_source(g, row, threadIdx.x == 0);
        rmsnorm_row_short(reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(rp.x) + src), static_cast<const uint4*>(rp.gain),
                          reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(const_cast<void*>(g.a)) + (int64_t)row * g.K), g.K, rp.eps, red,
                          rp.raw_out ? reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(rp.raw_out) + (int64_t)row * g.K) : nullptr);
    }
    asm volatile("fence.proxy.async;" ::: "memory");   // the rows are read back through TMA
    grid_barrier(g.grid_bar, abort_flag, g.debug_expire != 0);
    asm volatile("fence.proxy.async;" ::: "memory");
}
__device__ __noinline__ void prep_phase_long(const GemmArgs& g, float* red, volatile int* abort_flag, int cta_rows) {
    prep_phase(g, red, abort_flag, cta_rows);
}

// Few rows of narrow models (up to 256 columns, 16 bytes a lane): every CTA gathers and normalises all rows itself and writes
// them into the ring where the TMA would put them.  The rows are 32 KB at most, from L2, and nobody waits for anybody: prepared
// once for all behind a grid-wide barrier, a row's way was a store to global memory, the barrier (1.5-2.1 us) and the TMA's load
// of it (0.8).  Layer-step of 58 rows of 256 columns 53.5 -> 46.2 us.  The sum of a row's squares is the shared preparation's, in its order.
__device__ __forceinline__ void own_row_prep(const GemmArgs& g, const RowsPlan& p, uint32_t base, int* s_pos) {
    const RowPrep& rp = g.prep;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nchunk = g.K >> 3;
    constexpr int NW = RW_THREADS / 32;
    // warp w takes rows w, w + 8, ..; lane i looks up the place of its i-th
    int64_t src = 0;
    const int mine = warp + lane * NW;
    if (mine < g.M) {
        int pos = 0;
        src = prep_row_source(g, mine, blockIdx.x == 0, &pos);
        s_pos[mine] = pos;
    }
    const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(rp.x);
    const bool in = lane < nchunk;
    const uint4 gain = in ? __ldg(static_cast<const uint4*>(rp.gain) + lane) : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t gw[4] = {gain.x, gain.y, gain.z, gain.w};
    const int panel = lane >> 3;                              // 64 columns, as eight chunks
    const uint32_t dst = base + panel / p.CP * p.stage_bytes + panel % p.CP * p.rows_pad * 128;
    auto at = [&](int row) { return dst + row * 128 + (((lane & 7) ^ (row & 7)) << 4); };
    // All rows of the warp are asked for at once, each lane's 16 bytes to where its result goes.  Loops rather than registers: the
    // instructions come from L2 on a first pass (eight rows unrolled took 1.9 us after the loads).
#pragma unroll 1
    for (int i = 0; warp + i * NW < g.M; ++i) {
        const int64_t from = __shfl_sync(0xffffffffu, src, i);
        if (in) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(at(warp + i * NW)), "l"(x + from + lane * 8) : "memory");
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll 2
    for (int row = warp; row < g.M; row += NW) {
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        if (in) asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(at(row)) : "memory");
        float ss = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) { const float a = bf16_lo(w[e]), b = bf16_hi(w[e]); ss += a * a + b * b; }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        const float rstd = rsqrtf(ss / (float)g.K + rp.eps);
        uint32_t r[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) r[e] = pack_bf16(bf16_lo(w[e]) * rstd * bf16_lo(gw[e]), bf16_hi(w[e]) * rstd * bf16_hi(gw[e]));
        if (in) asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at(row)), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the tensor core reads them
    __syncthreads();
}

// OWN: own_row_prep instead of the shared preparation, in a kernel of its own (with both in one, calls that take the shared one were
// 3 % slower, their instructions come from further away).
template <int S, int EPI, bool APART, bool OWN>
__device__ __forceinline__ void rows_body(const GemmArgs& g, const RowsPlan& p, const CUtensorMap& mapA, const CUtensorMap& mapB0,
                                          const CUtensorMap& mapB1, const CUtensorMap& mapB2) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint64_t bar_s[2 * RW_MAX_STAGES + 2];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_s;
    __shared__ float red[RW_THREADS / 32];
    __shared__ int s_pos[OWN ? 128 : 1];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    volatile int* abort_flag = &abort_s;
    const uint32_t bars = smem_u32(bar_s);
    auto full_bar = [&](int s) { return bars + 8 * s; };
    auto empty_bar = [&](int s) { return bars + 8 * (RW_MAX_STAGES + s); };
    const uint32_t done_bar = bars + 8 * 2 * RW_MAX_STAGES, recv_bar = done_bar + 8;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = S > 1 ? (int)cluster_ctarank() : 0;
    const int nt = blockIdx.x / S;
    const int blk0 = rank * p.blocks / S, blk1 = (rank + 1) * p.blocks / S;
    const int n_blk = blk1 - blk0;
    // the columns this CTA finishes: items of 16 + 16 rotary pairs (q/k/v), of 16 columns (residual), of 8 + 8 (SwiGLU)
    constexpr int UNIT = EPI == kEpiQKV ? 32 : 16;
    const int items = p.TN / UNIT, item0 = rank * items / S, item1 = (rank + 1) * items / S;
    // a peer's part of them: [block (one if not APART)][column / 4][row][4]
    const int per_block = (items + S - 1) / S * UNIT * p.rows_pad * 4;
    const int region = per_block * (APART ? (p.blocks + S - 1) / S * p.CP : 1);
    const uint32_t recv = base + p.recv_off;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        mbar_init(done_bar, 1);
        if (S > 1) mbar_init(recv_bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (S > 1) {              // what the peers will send
            int from = S - 1;
            if (APART) {
                from = 0;
                for (int c = 0; c < S; ++c) from += c == rank ? 0 : rank_panels<S>(p, c);
            }
            mbar_expect_tx(recv_bar, from * (item1 - item0) * UNIT * p.rows_pad * 4);
        }
    }
    // The weights are constant inputs: the ring's weight halves are requested before the previous kernel has finished; the
    // activation rows follow once they are there.
    const uint64_t pol_a = policy_evict_last(), pol_w = g.keep_weights ? pol_a : policy_evict_first();
    const uint32_t a_bytes = p.CP * p.rows_pad * 128, box_bytes = p.CP * p.R * 128;
    const WeightBoxes<EPI> boxes(g, p, nt);
    auto load_weights = [&](int stage, int blk) {
        const uint32_t dst = base + stage * p.stage_bytes + a_bytes;
#pragma unroll
        for (int u = 0; u < RW_MAX_UNITS; ++u) {
            if (u >= p.n_units) break;
            const CUtensorMap* map = boxes.seg[u] == 0 ? &mapB0 : boxes.seg[u] == 1 ? &mapB1 : &mapB2;
            if (EPI == kEpiQKV) {
                const int half = g.head_dim >> 1;
                const int h = boxes.row[u] / half;
                tma_load_4d(dst + u * box_bytes, map, boxes.row[u] - h * half, h, blk * p.CP, full_bar(stage), pol_w);
            } else {
                tma_load_3d(dst + u * box_bytes, map, boxes.row[u], blk * p.CP, full_bar(stage), pol_w);
            }
        }
    };
    int prefilled = 0;
    if (threadIdx.x == 0) {
        for (; prefilled < p.stages && prefilled < n_blk; ++prefilled) {
            mbar_expect_tx(full_bar(prefilled), OWN ? p.stage_bytes - a_bytes : p.stage_bytes);
            load_weights(prefilled, blk0 + prefilled);
        }
    }
    __syncwarp();
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_slot)), "r"(p.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (S > 1) cluster_arrive_relaxed();                   // the peers may send once all have come this far
    const uint32_t tmem_base = tmem_slot;
    pdl_wait();
    pdl_launch_dependents();

    if constexpr (OWN) own_row_prep(g, p, base, s_pos);
    else if (EPI != kEpiResidual && g.prep.enabled) {
        if constexpr (APART) prep_phase(g, red, abort_flag, p.cta_rows);     // (few tiles: mostly the long way, 3-5 % slower as a call)
        else if (g.M <= p.cta_rows && g.K <= 3 * RW_THREADS * 8) prep_phase_short(g, red, abort_flag);
        else {
            const GemmArgs args = g;
            prep_phase_long(args, red, abort_flag, p.cta_rows);
        }
    }

    // ---------------- the contraction ----------------
    if (threadIdx.x == 0) {
        bool ok = !*abort_flag;
        int stage = 0;
        uint32_t phase = 0;
        for (int i = 0; i < n_blk && ok && !OWN; ++i) {           // (OWN: the whole of K is in the ring)
            if (prefilled > 0) {
                --prefilled;              // this stage's weights are already on their way
            } else {
                if (!(ok = mbar_poll(empty_bar(stage), phase ^ 1, abort_flag))) break;
                mbar_expect_tx(full_bar(stage), p.stage_bytes);
                load_weights(stage, blk0 + i);
            }
            tma_load_3d(base + stage * p.stage_bytes, &mapA, 0, (blk0 + i) * p.CP, full_bar(stage), pol_a);
            if (++stage == p.stages) { stage = 0; phase ^= 1; }
        }
    } else if (warp == 1) {
        // What bounds a stage here is this warp, not the data: 4 to 32 instructions of 60-100 cycles (they read A and B from
        // shared memory, which the TMA fills meanwhile), then about 400 cycles until the next stage's first.  With one thread
        // in the loop, whose descriptors are no warp-uniform values, the instructions took 94-121 cycles: masked rows' queries
        // 2030 -> 1590 cycles a stage, layer-step of 103 rows 145.9 -> 144.2 us, of 8 rows 53.1 -> 51.6, decode pass of
        // 32 rows over 4 layers 656 -> 646.  The next stage's barrier tested before the instructions or before the commit:
        // 1 us slower.
        bool ok = __all_sync(0xffffffffu, !*abort_flag);
        int stage = 0;
        uint32_t phase = 0;
        const uint32_t idesc = idesc_bf16(p.mma_n);
        for (int i = 0; i < n_blk && ok; ++i) {
            if (!(ok = __all_sync(0xffffffffu, mbar_poll(full_bar(stage), phase, abort_flag)))) break;
            tc_fence_after();
            if (elect_lane()) {
                const uint32_t sA = base + stage * p.stage_bytes, sB = sA + a_bytes;
                const int panels = APART ? min(p.CP, p.KB - (blk0 + i) * p.CP) : p.CP;     // past K a panel has no accumulator
                for (int c = 0; c < panels; ++c) {
                    const uint32_t acc = tmem_base + (APART ? (i * p.CP + c) * p.TN : 0);
                    const uint64_t da = smem_desc_sw128(sA + c * p.rows_pad * 128);
                    for (int u = 0; u < p.mma_count; ++u) {
                        const uint64_t db = smem_desc_sw128(sB + u * box_bytes + c * p.R * 128);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            tc_mma(acc + u * p.mma_n, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc,
                                   (k > 0 || (!APART && (i > 0 || c > 0))) ? 1u : 0u);
                    }
                }
                tc_commit(empty_bar(stage));
                if (i + 1 == n_blk) tc_commit(done_bar);
            }
            __syncwarp();
            if (++stage == p.stages) { stage = 0; phase ^= 1; }
        }
    }
    __syncwarp();

    // ---------------- epilogue: thread = one row, warp = lane quarter x column half ----------------
    const int q = warp & 3, hf = warp >> 2, row = q * 32 + lane;
    const bool live = q * 32 < p.rows_pad;                 // warp-uniform: the tensor-memory accesses are collective
    const bool valid = row < g.M;
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16);
    // what does not depend on the sums is requested while the weights stream
    int pos = 0;
    uint4 res[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
    const uint4* res_row = nullptr;
    if (EPI == kEpiResidual && valid) {
        const int64_t roff = g.resid_off ? __ldcg(g.resid_off + row) : (int64_t)row * g.n[0];
        res_row = reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(g.resid) + roff);
        const int col = nt * p.TN + (item0 + hf) * UNIT;
        if (item0 + hf < item1 && col < g.n[0]) { res[0] = __ldcg(res_row + (col >> 3)); res[1] = __ldcg(res_row + (col >> 3) + 1); }
    }
    float c[16] = {}, sn[16] = {};         // the first item's waited 1.2 us for memory where they were asked for after the sums
    auto item_rope = [&](int u) {          // cosines and sines of item u's pairs
        int col;
        const int seg = pair_group(g, min(nt * p.n_units + (u >> 1), p.groups - 1), col);
        if (u < item1 && seg < g.rope_segments) load_rope<16>(g, pos, (col + (u & 1) * 16) & ((g.head_dim >> 1) - 1), c, sn);
    };
    if (EPI == kEpiQKV && valid) {
        pos = OWN ? s_pos[OWN ? row : 0] : __ldcg(g.row_pos + row);
        item_rope(item0 + hf);
    }

    bool ok = !*abort_flag;
    if (ok) ok = mbar_wait(done_bar, 0, abort_flag);
    ok = __all_sync(0xffffffffu, ok);
    tc_fence_after();
    if (S > 1) {
        // Every other CTA's columns straight from tensor memory into its shared memory; it waits for the bytes alone.  With the
        // parts staged here, a cluster barrier and loads from the peers: layer-step of 103 rows 145.7 -> 143.3 us, decode pass of
        // 32 rows over 4 layers 622 -> 618; a launch of 103 rows ended 3.0 us after its last MMA, now 2.0.
        cluster_wait();
        if (p.recv_late) {                                 // every CTA's MMAs have read its ring
            cluster_arrive_relaxed();
            cluster_wait();
        }
        if (ok && live) {
            const int nb = APART ? rank_panels<S>(p, rank) : 1;
            for (int d = 0; d < S; ++d) {
                if (d == rank) continue;
                const int u0 = d * items / S, u1 = (d + 1) * items / S;
                const uint32_t dst = mapa_u32(recv + (rank < d ? rank : rank - 1) * region, d), bar = mapa_u32(recv_bar, d);
                for (int u = u0 + hf; u < u1; u += 2) {
#pragma unroll
                    for (int part = 0; part < UNIT / 16; ++part) {
                        const int col = EPI == kEpiQKV ? (u >> 1) * 64 + (u & 1) * 16 + part * 32 : u * 16;
                        const int sc = ((u - u0) * UNIT + part * 16) >> 2;
#pragma unroll 1
                        for (int blk = 0; blk < nb; ++blk) {
                            float v[16];
                            tc_ld16(taddr + blk * p.TN + col, v);
                            if (row < p.rows_pad) {
#pragma unroll
                                for (int j = 0; j < 4; ++j) send_f4(dst + blk * per_block + (((sc + j) * p.rows_pad + row) << 4), v + 4 * j, bar);
                            }
                        }
                    }
                }
            }
        }
        __syncwarp();
        cluster_arrive_relaxed();                          // the last word to the peers: they may leave when they have theirs
        if (live) ok = __all_sync(0xffffffffu, ok && mbar_wait_cluster(recv_bar, 0, abort_flag));
    }
    auto sum16 = [&](int col, int slice_col, float (&v)[16]) {
        if (APART) sum_apart16<S>(p, rank, taddr + col, recv, region, slice_col, per_block, row, v);
        else sum_cluster16<S>(taddr + col, recv, region, slice_col, p.rows_pad, row, v);
    };
    if (ok && live) {
        for (int u = item0 + hf; u < item1; u += 2) {
            const int sc = (u - item0) * UNIT;
            if (EPI == kEpiResidual) {
                const int col = nt * p.TN + u * 16;
                float v[16];
                sum16(u * 16, sc, v);
                if (valid && col < g.n[0]) {
                    if (u != item0 + hf) { res[0] = __ldcg(res_row + (col >> 3)); res[1] = __ldcg(res_row + (col >> 3) + 1); }
                    const uint32_t rw[8] = {res[0].x, res[0].y, res[0].z, res[0].w, res[1].x, res[1].y, res[1].z, res[1].w};
#pragma unroll
                    for (int i = 0; i < 8; ++i) { v[2 * i] += bf16_lo(rw[i]); v[2 * i + 1] += bf16_hi(rw[i]); }
                    store16(static_cast<__nv_bfloat16*>(g.c) + (int64_t)row * g.n[0] + col, v);
                }
            } else if (EPI == kEpiSwiGLU) {
                const int col = nt * (p.TN >> 1) + u * 8;
                float gate[8], up[8];
                tc_ld8x2(taddr + u * 8, taddr + (p.TN >> 1) + u * 8, gate, up);
                if (APART) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) { gate[i] += 0.f; up[i] += 0.f; }        // -0 becomes 0, as in a sum from 0
#pragma unroll 1
                    for (int blk = 1; blk < p.KB; ++blk) {
                        float a[8], b[8];
                        tc_ld8x2(taddr + blk * p.TN + u * 8, taddr + blk * p.TN + (p.TN >> 1) + u * 8, a, b);
#pragma unroll
                        for (int i = 0; i < 8; ++i) { gate[i] += a[i]; up[i] += b[i]; }
                    }
                }
                if (valid && col < g.n[0]) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) gate[i] = silu(gate[i]) * up[i];
                    *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(g.c) + (int64_t)row * g.n[0] + col) = pack8(gate);
                }
            } else {
                const int grp = nt * p.n_units + (u >> 1);
                int col;
                const int seg = pair_group(g, min(grp, p.groups - 1), col);
                col += (u & 1) * 16;
                float lo[16], hi[16];
                sum16((u >> 1) * 64 + (u & 1) * 16, sc, lo);
                sum16((u >> 1) * 64 + (u & 1) * 16 + 32, sc + 16, hi);
                if (valid && grp < p.groups) {
                    rope_qkv<16>(g, seg, col, lo, hi, c, sn);
                    item_rope(u + 2);
                    store_qkv<16>(g, row, pos, seg, col, lo, hi);
                }
            }
        }
    }
    __syncwarp();
    // ---------------- teardown ----------------
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0) {
            atomicOr(g.status, kFlagWaitExpired);
            // ring stages whose weights were requested before the dependency wait but whose activation rows never were:
            // send those now, so that each stage's full barrier completes when all of its copies have landed
            for (int i = 0; i < prefilled && !OWN; ++i) tma_load_3d(base + i * p.stage_bytes, &mapA, 0, 0, full_bar(i), pol_a);
            for (int i = 0; i < prefilled; ++i)
                for (uint32_t n = 0; n < TC_WAIT_LIMIT && !mbar_try_wait(full_bar(i), 0); ++n) __nanosleep(40);
            for (int i = 0; i < 4096; ++i) __nanosleep(64);   // copies of stages that were complete when a role gave up
        }
        __syncthreads();
    }
    __syncwarp();
    if (S > 1) cluster_wait();                                // no CTA leaves before its peers have sent what they will send
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(p.tmem_cols) : "memory");
    }
}

template <int S, int EPI, bool APART>
__global__ void __launch_bounds__(RW_THREADS, 1)
gemm_rows_kernel(const GemmArgs g, const RowsPlan p, const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB0,
                 const __grid_constant__ CUtensorMap mapB1, const __grid_constant__ CUtensorMap mapB2) {
    rows_body<S, EPI, APART, false>(g, p, mapA, mapB0, mapB1, mapB2);
}
template <int S, int EPI, bool APART>
__global__ void __launch_bounds__(RW_THREADS, 1)
own_gemm_rows_kernel(const GemmArgs g, const RowsPlan p, const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB0,
                 const __grid_constant__ CUtensorMap mapB1, const __grid_constant__ CUtensorMap mapB2) {
    rows_body<S, EPI, APART, true>(g, p, mapA, mapB0, mapB1, mapB2);
}

// ---- host side ------------------------------------------------------------------------------
namespace {

constexpr int kSmemBytes = 226 * 1024;
template <int S, int EPI, bool APART, bool OWN = false>
cudaError_t launch_rows(const GemmArgs& g, const RowsPlan& p, const CUtensorMap& a, const CUtensorMap* b, cudaStream_t stream) {
    const auto kernel = [] {
        if constexpr (OWN) return own_gemm_rows_kernel<S, EPI, APART>;
        else return gemm_rows_kernel<S, EPI, APART>;
    }();
    static const cudaError_t attr = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (attr != cudaSuccess) return attr;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(p.n_tiles * S);
    cfg.blockDim = dim3(RW_THREADS);
    cfg.dynamicSmemBytes = p.smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = S; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = S > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, g, p, a, b[0], b[1], b[2]);
}

// Clusters of S CTAs that are resident at once with one CTA per SM (the SM counts of the GPCs are not multiples of S).
template <int S>
int resident_clusters() {
    static const int n = [] {
        if (S == 1) return sm_count();
        cudaFuncSetAttribute(gemm_rows_kernel<S, kEpiResidual, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(sm_count() / S * S);
        cfg.blockDim = dim3(RW_THREADS);
        cfg.dynamicSmemBytes = 200 * 1024;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = S; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int c = 0;
        if (cudaOccupancyMaxActiveClusters(&c, gemm_rows_kernel<S, kEpiResidual, false>, &cfg) != cudaSuccess) { (void)cudaGetLastError(); c = 0; }
        return c;
    }();
    return n;
}

// Tile width and K split: the least estimated time of one wave.  The weights cannot stream faster than HBM delivers them
// (6.5 TB/s); a CTA not faster than about 60 GB/s (its weight rows and, once per tile, all rows of A; measured 45-60 with
// this ring); a split costs an exchange per doubling, 1.5 us where rotary pairs are finished and 1 us otherwise.  A stage
// takes as many panels as leave three stages in the ring (fewer, larger stages lost, two stages of any size did too).
// Measured when it replaced that kernel, at 103 rows (us per launch, finish included | here): q/k/v 30.2 | 29.6, output
// 16.3 | 13.0, gate/up 47.7 | 43, down 25.7 | 23.4; at 32 rows output 14.3 | 10.9, down 25.0 | 20.4.
// With an accumulator per K block the tile is at most what 256 columns of tensor memory hold, as the widest tile does.  A split
// costs 2.5 us there, for every block is exchanged (58 rows, 1024 -> 256 columns in the chain above: over two CTAs 1.4 us slower
// than in one); it is taken for rotary pairs alone, whose tiles of 64 columns hold four blocks to a CTA.
constexpr int kRingBytes = 200 * 1024, kApartColumns = 256;
bool plan_rows(const GemmArgs& g, RowsPlan& best) {
    if (g.M > 128 || g.epilogue == kEpiLogits || g.K < 64) return false;
    const bool qkv = g.epilogue == kEpiQKV, swiglu = g.epilogue == kEpiSwiGLU;
    const int n_total = swiglu ? 2 * g.n[0] : g.n[0] + g.n[1] + g.n[2];
    const int KB = g.K / 64, rows_pad = (g.M + 7) & ~7;
    const int general_iterations = (swiglu ? g.n[0] / 128 : (n_total / 128 + 1) / 2) * KB;      // of the general kernel
    const bool apart = general_iterations <= sm_count();
    const int step = qkv ? 64 : swiglu || apart ? 16 : 32;
    const int limit[3] = {resident_clusters<1>(), resident_clusters<2>(), resident_clusters<4>()};
    double t_best = 1e30;
    for (int si = 0; si < (swiglu || (apart && !qkv) ? 1 : apart ? 2 : 3); ++si) {
        const int S = 1 << si;
        for (int TN = step; TN <= 256; TN += step) {
            const int items = TN / (qkv ? 32 : 16);
            const int n_tiles = (n_total + TN - 1) / TN;
            if (items < S || n_tiles > limit[si]) continue;
            const int panel = (rows_pad + TN) * 128;
            int CP = 1;         // an instruction spans 16 columns' multiples: half a SwiGLU tile has to be one to take more panels
            while (CP < 8 && (!swiglu || TN % 32 == 0) && 2 * CP * 3 * panel <= kRingBytes && 2 * CP * S <= KB) CP *= 2;
            const int blocks = (KB + CP - 1) / CP;
            if (blocks < S) continue;
            const int my_blocks = (blocks + S - 1) / S;
            const int accs = apart ? my_blocks * CP : 1;        // accumulators of a CTA
            if (apart && accs * TN > kApartColumns) continue;
            const int stages = std::min(std::min(kRingBytes / (CP * panel), RW_MAX_STAGES), my_blocks);
            const int region = (items + S - 1) / S * (qkv ? 32 : 16) * rows_pad * 4 * accs;
            const double t_hbm = 2.0 * n_total * g.K / 6.5e6, t_sm = (double)my_blocks * CP * panel / 60e3;
            const double t = std::max(std::max(t_hbm, t_sm), my_blocks * 0.15) + si * (apart ? 2.5 : qkv ? 1.5 : 1.0);
            if (t >= t_best * 0.999) continue;
            t_best = t;
            best = RowsPlan{};
            best.TN = TN; best.n_tiles = n_tiles; best.CP = CP; best.blocks = blocks; best.S = S; best.rows_pad = rows_pad;
            best.R = qkv ? 64 : swiglu ? TN / 2 : TN;
            best.n_units = TN / best.R;
            best.mma_n = CP == 1 ? TN : best.R;
            best.mma_count = CP == 1 ? 1 : best.n_units;
            best.stages = stages; best.stage_bytes = CP * panel;
            best.KB = KB; best.apart = apart;
            // Own rows up to eight a warp, where the whole of K is in the ring, and not from host memory (decode pass over 4 layers of
            // 256 columns, us, shared preparation | own: 16 rows 140 | 116, 32 142 | 120, 64 149 | 136; with both in one kernel, 78
            // 151 | 151, 96 153 | 157, 128 166 | 172).  The self-test of the grid barrier wants the barrier.
            best.own_rows = apart && S == 1 && g.prep.enabled && !g.prep.x_far && !g.debug_expire && g.K <= 256 && g.M <= 64 &&
                            stages == my_blocks && KB % CP == 0;
            best.cta_rows = apart && g.K > 256 ? general_iterations : n_tiles * S;
            best.tmem_cols = accs * TN <= 32 ? 32 : accs * TN <= 64 ? 64 : accs * TN <= 128 ? 128 : 256;
            best.groups = n_total / 64;
            // the MMA reads 128 rows of A whatever M is: the last panel's read may run past the ring
            const int ring = std::max(stages * CP * panel, (stages - 1) * CP * panel + (CP - 1) * rows_pad * 128 + 128 * 128);
            // The peers' parts arrive behind the ring, or where they do not fit there (more than 112 rows of tiles of 128 columns over
            // four CTAs) in it, once everyone is done with it: a ring of two stages less made the down projection of 124
            // rows of 18 944 columns 30.5 -> 33.1 us.
            best.recv_late = S > 1 && ring + (S - 1) * region + 1024 > kSmemBytes;
            best.recv_off = best.recv_late ? 0 : ring;
            best.smem_bytes = (best.recv_late ? std::max(ring, (S - 1) * region) : ring + (S - 1) * region) + 1024;
            if (!best.own_rows) best.smem_bytes = std::max(best.smem_bytes, kAloneBytes);    // (own rows wait for nobody)
        }
    }
    return t_best < 1e29;
}

}  // namespace

int launch_gemm_rows(const GemmArgs& g, cudaStream_t stream) {
    RowsPlan p;
    if (!plan_rows(g, p)) return 0;
    CUtensorMap map_a, map_b[3];
    {
        std::lock_guard<std::mutex> lock(g_map_mutex);
        const CUtensorMap* m = get_panel_map(g.a, g.M, g.K, p.rows_pad, p.CP, 0);
        if (!m) return -1;
        map_a = *m;
        const bool qkv = g.epilogue == kEpiQKV;
        for (int i = 0; i < 3; ++i) {
            if (!g.b[i]) { if (i == 0) return -1; map_b[i] = map_b[0]; continue; }
            if (!(m = get_panel_map(g.b[i], g.n[i], g.K, qkv ? 32 : p.R, p.CP, qkv ? g.head_dim / 2 : 0))) return -1;
            map_b[i] = *m;
        }
    }
    cudaError_t e = cudaErrorInvalidValue;
    auto launch = [&](auto epi, auto apart) {
        constexpr int EPI = decltype(epi)::value;
        constexpr bool APART = decltype(apart)::value;
        if constexpr (APART && EPI != kEpiResidual)
            if (p.own_rows) return launch_rows<1, EPI, APART, true>(g, p, map_a, map_b, stream);
        if constexpr (EPI == kEpiSwiGLU || (APART && EPI == kEpiResidual)) return launch_rows<1, EPI, APART>(g, p, map_a, map_b, stream);
        else if constexpr (APART)
            return p.S == 1 ? launch_rows<1, EPI, APART>(g, p, map_a, map_b, stream) : launch_rows<2, EPI, APART>(g, p, map_a, map_b, stream);
        else
            return p.S == 1 ? launch_rows<1, EPI, APART>(g, p, map_a, map_b, stream)
                 : p.S == 2 ? launch_rows<2, EPI, APART>(g, p, map_a, map_b, stream)
                            : launch_rows<4, EPI, APART>(g, p, map_a, map_b, stream);
    };
    auto launch_epi = [&](auto epi) { return p.apart ? launch(epi, std::true_type{}) : launch(epi, std::false_type{}); };
    if (g.epilogue == kEpiSwiGLU) e = launch_epi(std::integral_constant<int, kEpiSwiGLU>{});
    else if (g.epilogue == kEpiResidual) e = launch_epi(std::integral_constant<int, kEpiResidual>{});
    else e = launch_epi(std::integral_constant<int, kEpiQKV>{});
    return e == cudaSuccess ? 1 : -1;
}

}  // namespace acache
