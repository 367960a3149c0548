// Projections of more than 128 rows with the weights as the product's M and the rows as its N (D = W X^T).
//
// gemm_tc2_kernel (gemm_tc.cu) gives the rows the M side of its instruction: they come in pairs of 128-row tiles, 615 rows cost
// what 768 do, and a launch is a whole number of rounds of 256 x 256 tiles.  Here a cluster of two CTAs multiplies 256 rows of the
// weights by a chunk of NC rows of the input, NC a multiple of 16 from 64 to 256 (in use up to 240: chunks of 256 save nothing), chosen
// with the number of chunks so that rounds x time of a chunk is least (launch_wm).  Everything else is that kernel's: cta_group::2, one
// producer and one issuing warp, two accumulators, eight epilogue warps, whole tiles walked in groups of weight tiles; and so are the
// results, bit for bit.
//
// us per launch, gemm_tc2_kernel | this: 615 rows (three chunks of 208) q/k/v 60.6 | 55.0, gate/up 101 | 92, output (four chunks of 160)
// 26.9 | 25.4; 512 rows (three of 176) q/k/v 59.6 | 56.4, which the kernels behind it pay back; 1015 rows of a 3584-column model (five
// chunks of 208 for four row pairs) down 113 | 95; 1639 rows gate/up 239 | 230, down 140 | 118.
// Bound at these sizes by no unit: gate/up of 615 rows has the tensor pipe busy 66 % of the launch, L2 at 41 % and HBM at 33 % of their
// peaks (1.57 GHz); what is left is the launch's edges and waits for operands in the ring.  From about 1500 rows by power.
//
// The accumulator lies the other way round (tensor-memory lane = output column, column = row of the input), so the epilogue turns
// 32 x 32 pieces round in shared memory and then works on one row per thread like the others.  Which weight rows a warp's 32 lanes are
// is the tensor map's choice: of a rotary head 16 pairs (i and i + d/2 side by side), of gate/up 16 columns of each (the two matrices
// are one map whose third dimension steps from one to the other), else 32 adjacent columns.
#include <algorithm>

#include "common.cuh"
#include "gemm_common.cuh"
#include "kernels.h"
#include "launch.h"
#include "tc_ptx.cuh"

namespace acache {

constexpr int WM_THREADS = 320;                       // warp 0: TMA, warp 1: MMA, warps 2-9: epilogue
constexpr int WM_W_BYTES = 128 * 64 * 2;              // a CTA's 128 weight rows of one K block
constexpr int WM_MAX_STAGES = 8;
constexpr int WM_PIECE = 32 * 33 * 4;                 // a 32 x 32 piece in shared memory, rows of 33 words
constexpr int WM_STAGING = 8 * WM_PIECE;
constexpr int WM_SMEM_DYN = 227 * 1024 - 512;         // beside the barriers and reduction words
constexpr double kRowEpilogueUs = 0.05, kBehindUs = 0.75;   // the rule's, see launch_wm

struct WmPlan {
    int NC, chunks;           // rows per chunk (a multiple of 16), chunks
    int w_tiles, KB;
    int stages, stage_bytes, smem_bytes;
    int clusters, group_n;
    int keep;                 // weights evict-last (several chunks re-read them from L2)
    int up_first;             // gate/up: w_up lies below w_gate in memory, so a warp's lanes are 16 up, then 16 gate columns
};

__device__ __forceinline__ void wm_load_w(uint32_t dst, const CUtensorMap* map, int c0, int c4, uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1, {%2, %3, %4, %5, %6}], [%7], %8;"
        ::"r"(dst), "l"(map), "r"(c0), "r"(0), "r"(0), "r"(0), "r"(c4), "r"(bar), "l"(policy)
        : "memory");
}

template <int EPI>
__global__ void __launch_bounds__(WM_THREADS, 1)
gemm_wm_kernel(const GemmArgs g, const WmPlan p, const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapW0,
               const __grid_constant__ CUtensorMap mapW1, const __grid_constant__ CUtensorMap mapW2) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ float red[WM_THREADS / 32];
    __shared__ uint64_t bar_s[2 * WM_MAX_STAGES + 4];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_s;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    volatile int* abort_flag = &abort_s;
    const uint32_t bars = smem_u32(bar_s);
    auto full_bar = [&](int s) { return bars + 8 * s; };
    auto empty_bar = [&](int s) { return bars + 8 * (WM_MAX_STAGES + s); };
    auto tfull_bar = [&](int i) { return bars + 8 * (2 * WM_MAX_STAGES + i); };
    auto tempty_bar = [&](int i) { return bars + 8 * (2 * WM_MAX_STAGES + 2 + i); };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_ctarank();
    const int cluster_id = blockIdx.x >> 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(tfull_bar(i), 1); mbar_init(tempty_bar(i), 16); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();          // the peer's barriers are initialised before anyone signals them
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;
    pdl_wait();
    pdl_launch_dependents();

    if (g.prep.enabled) prep_phase<true>(g, red, abort_flag, gridDim.x);

    const int tiles = p.w_tiles * p.chunks;
    if (warp == 0) {
        // producer: this CTA's 128 weight rows and its half of the chunk's rows; both CTAs' bytes count on the leader's barrier
        int stage = 0, issued = 0;
        uint32_t phase = 0;
        bool ok = __all_sync(0xffffffffu, !*abort_flag);
        const uint64_t pol_x = policy_evict_last(), pol_w = g.keep_weights || p.keep ? pol_x : policy_evict_first();
        for (int t = cluster_id; ok && t < tiles; t += p.clusters) {
            int wt, rc;
            tile_coords(t, p.chunks, p.w_tiles, p.group_n, wt, rc);
            const int xrow = rc * p.NC + rank * (p.NC >> 1);
            int seg = 0, at = wt * 2 + rank;             // unit of 128 weight rows (gate/up: of 64 + 64)
            if (EPI == kEpiQKV) { qkv_unit(g, at, seg, at); at = g.head_dim == 128 ? at >> 7 : at >> 6; }
            const CUtensorMap* map = seg == 0 ? &mapW0 : seg == 1 ? &mapW1 : &mapW2;
            for (int kb = 0; kb < p.KB; ++kb) {
                if (!(ok = __all_sync(0xffffffffu, mbar_poll(empty_bar(stage), phase ^ 1, abort_flag)))) break;
                if (elect_lane()) {
                    const uint32_t sW = base + stage * p.stage_bytes, sX = sW + WM_W_BYTES;
                    const uint32_t lead_full = mapa_u32(full_bar(stage), 0);
                    if (rank == 0) mbar_expect_tx(full_bar(stage), 2 * p.stage_bytes);
                    wm_load_w(sW, map, kb * 64, at, lead_full, pol_w);
                    tma_load_2d_pair(sX, &mapX, kb * 64, xrow, lead_full, pol_x);
                }
                __syncwarp();
                ++issued;
                if (++stage == p.stages) { stage = 0; phase ^= 1; }
            }
        }
        // wait until the MMAs have consumed everything this CTA loaded, so that no signal from the leader can arrive after
        // this CTA has left
        if (issued < p.stages) { stage = 0; phase = 1; }
        for (int i = 0; i < min(issued, p.stages) && ok; ++i) {
            ok = __all_sync(0xffffffffu, mbar_poll(empty_bar(stage), phase ^ 1, abort_flag));
            if (++stage == p.stages) { stage = 0; phase ^= 1; }
        }
    } else if (warp == 1 && rank == 0) {
        int stage = 0, acc = 0;
        uint32_t phase = 0, acc_phase = 0;
        bool ok = __all_sync(0xffffffffu, !*abort_flag);
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.NC >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
        for (int t = cluster_id; ok && t < tiles; t += p.clusters) {
            if (!(ok = __all_sync(0xffffffffu, mbar_poll_cluster(tempty_bar(acc), acc_phase ^ 1, abort_flag)))) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + acc * 256;
            for (int kb = 0; kb < p.KB; ++kb) {
                if (!(ok = __all_sync(0xffffffffu, mbar_poll(full_bar(stage), phase, abort_flag)))) break;
                tc_fence_after();
                if (elect_lane()) {
                    const uint32_t sW = base + stage * p.stage_bytes;
                    const uint64_t da = smem_desc_sw128(sW), db = smem_desc_sw128(sW + WM_W_BYTES);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        tc2_mma(d_tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc, (kb > 0 || k > 0) ? 1u : 0u);
                    tc2_commit_both(empty_bar(stage));
                    if (kb + 1 == p.KB) tc2_commit_both(tfull_bar(acc));
                }
                __syncwarp();
                if (++stage == p.stages) { stage = 0; phase ^= 1; }
            }
            if (++acc == 2) { acc = 0; acc_phase ^= 1; }
        }
    } else if (warp >= 2) {
        // epilogue: two warps per lane quarter, alternate blocks of 32 rows of the chunk
        const int q = warp & 3, hf = (warp - 2) >> 2;
        const uint32_t stg = base + p.stages * p.stage_bytes + (warp - 2) * WM_PIECE;
        const int n_blk = (p.NC + 31) >> 5;
        const int half = g.head_dim >> 1;
        int acc = 0;
        uint32_t acc_phase = 0;
        bool ok = !*abort_flag;
        for (int t = cluster_id; ok && t < tiles; t += p.clusters) {
            int wt, rc;
            tile_coords(t, p.chunks, p.w_tiles, p.group_n, wt, rc);
            int seg = 0, col = 0, lo_col = 0;            // columns of this warp: segment, first column inside it
            if (EPI == kEpiQKV) {
                qkv_unit(g, wt * 2 + rank, seg, col);
                lo_col = g.head_dim == 128 ? 16 * q : 64 * (q >> 1) + 16 * (q & 1);
                col += lo_col;
            } else if (EPI == kEpiSwiGLU) {
                col = wt * 128 + rank * 64 + q * 16;
            } else {
                col = wt * 256 + rank * 128 + q * 32;
            }
            // What does not depend on the sums is requested before the wait for them: the residual of all of the thread's rows (at
            // most four), 64 bytes each, or their positions and the first two rows' cosines and sines (then two blocks ahead).
            uint4 res[EPI == kEpiResidual ? 4 : 1][4];
            int pos[EPI == kEpiQKV ? 4 : 1];
            float cs[EPI == kEpiQKV ? 2 : 1][2][16];
            const bool rotary = EPI == kEpiQKV && seg < g.rope_segments;
            auto row_of = [&](int i) {                   // row of the thread's i-th block; -1: none
                const int in = (hf + 2 * i) * 32 + lane, grow = rc * p.NC + in;
                return in < p.NC && grow < g.M ? grow : -1;
            };
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int grow = row_of(i);
                if (EPI == kEpiResidual && grow >= 0) {
                    const int64_t roff = g.resid_off ? __ldcg(g.resid_off + grow) : (int64_t)grow * g.n[0];
                    const uint4* rp = reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(g.resid) + roff + col);
#pragma unroll
                    for (int j = 0; j < 4; ++j) res[EPI == kEpiResidual ? i : 0][j] = __ldcg(rp + j);
                }
                if (EPI == kEpiQKV) pos[EPI == kEpiQKV ? i : 0] = grow >= 0 ? __ldcg(g.row_pos + grow) : 0;
            }
            if (rotary) {
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    if (row_of(i) >= 0) load_rope<16>(g, pos[i], lo_col & (half - 1), cs[EPI == kEpiQKV ? i : 0][0], cs[EPI == kEpiQKV ? i : 0][1]);
            }
            if (!(ok = __all_sync(0xffffffffu, mbar_wait(tfull_bar(acc), acc_phase, abort_flag)))) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + acc * 256 + ((uint32_t)(q * 32) << 16);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int blk = hf + 2 * i, grow = row_of(i);
                if (blk >= n_blk) break;
                const bool valid = grow >= 0;
                float v[32];
                tc_ld32(taddr + blk * 32, v);
                // turn the 32 columns x 32 rows round (rows 33 words apart: no two lanes meet in a bank)
#pragma unroll
                for (int r = 0; r < 32; ++r)
                    asm volatile("st.shared.f32 [%0], %1;" ::"r"(stg + lane * 4 + r * 132), "f"(v[r]) : "memory");
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 32; ++r)
                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[r]) : "r"(stg + lane * 132 + r * 4) : "memory");
                __syncwarp();
                float (&lo)[16] = reinterpret_cast<float (&)[16]>(v[0]);
                float (&hi)[16] = reinterpret_cast<float (&)[16]>(v[16]);
                if (EPI == kEpiResidual) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint4 u = res[EPI == kEpiResidual ? i : 0][j];
                        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) { v[8 * j + 2 * e] += bf16_lo(w[e]); v[8 * j + 2 * e + 1] += bf16_hi(w[e]); }
                    }
                    __nv_bfloat16* o = static_cast<__nv_bfloat16*>(g.c) + (int64_t)grow * g.n[0] + col;
                    if (valid) { store16(o, lo); store16(o + 16, hi); }
                } else if (EPI == kEpiSwiGLU) {
                    if (valid) {
                        if (p.up_first) out_swiglu<16>(g, grow, col, hi, lo);
                        else out_swiglu<16>(g, grow, col, lo, hi);
                    }
                } else {
                    const int ci = EPI == kEpiQKV ? i & 1 : 0;
                    if (valid) rope_qkv<16>(g, seg, col, lo, hi, cs[ci][0], cs[ci][1]);
                    if (rotary && i < 2 && row_of(i + 2) >= 0) load_rope<16>(g, pos[EPI == kEpiQKV ? i + 2 : 0], lo_col & (half - 1), cs[ci][0], cs[ci][1]);
                    if (valid) store_qkv<16>(g, grow, pos[EPI == kEpiQKV ? i : 0], seg, col, lo, hi);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(mapa_u32(tempty_bar(acc), 0));
            if (++acc == 2) { acc = 0; acc_phase ^= 1; }
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

// ---- host side ------------------------------------------------------------------------------
namespace {

template <int EPI>
cudaLaunchConfig_t wm_config(cudaLaunchAttribute* at, int clusters, int smem, cudaStream_t stream) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(clusters * 2);
    cfg.blockDim = dim3(WM_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cfg;
}

// Clusters that are resident at once (the row preparation ends in a grid-wide barrier); 0: none fits.
template <int EPI>
int wm_max_clusters() {
    static const int n = [] {
        cudaFuncSetAttribute(gemm_wm_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, WM_SMEM_DYN);
        cudaLaunchAttribute at[2];
        const cudaLaunchConfig_t cfg = wm_config<EPI>(at, sm_count() / 2, WM_SMEM_DYN, nullptr);
        int c = 0;
        if (cudaOccupancyMaxActiveClusters(&c, gemm_wm_kernel<EPI>, &cfg) != cudaSuccess || c < 0) { (void)cudaGetLastError(); c = 0; }
        return std::min(c, sm_count() / 2);
    }();
    return n;
}

template <int EPI>
int launch_wm(const GemmArgs& g, double own_us, int group_n, cudaStream_t stream) {
    const int max_clusters = wm_max_clusters<EPI>();
    if (max_clusters < 1) return 0;
    WmPlan p{};
    p.KB = g.K / 64;
    p.w_tiles = EPI == kEpiSwiGLU ? g.n[0] / 128 : (g.n[0] + g.n[1] + g.n[2]) / 256;
    p.group_n = group_n;
    // The least time, if it is 2 % and kBehindUs less than the caller's (behind this kernel a finish kernel takes 0.5-1 us longer, the
    // attention up to 0.8).  An epilogue takes 0.05 us a row here (1024 columns of K, a round of 208 rows of gate/up: 8-10 us for 4.6
    // of main loop) and 9 us a tile there; by main loops alone gate/up of short contractions came here and lost (us of a layer-step,
    // there | here: 2045 rows of 256 columns 83.6 | 87.5, 2700 of 1024 165 | 178, 800 of 2048 160 | 168).  With it, all projections
    // there | as chosen, 4096 columns: 129 rows 159.7 | 150.6, 300 218.9 | 203.7, 512 232.8 | 232.7, 615 291.5 | 281.0, 800 356 | 332,
    // 1200 508 | 477, 2045 729 | 727; 3584 columns: 129 146.4 | 143.6, 300 217 | 206, 615 299 | 288, 800 373 | 342, 1200 474 | 459,
    // 2045 755 | 727.  What is left on the wrong side: down projection of 3496 rows of a 1024-column model 169.5 | 173.0.
    const int first = (g.M + 255) / 256;
    double best = 0.98 * own_us - kBehindUs;
    for (int chunks = first; chunks <= first + 6; ++chunks) {
        const int NC = ((g.M + chunks - 1) / chunks + 15) & ~15;
        if (NC < 64) break;
        const int tiles = p.w_tiles * chunks, rounds = (tiles + max_clusters - 1) / max_clusters;
        const double t = rounds * pair_tile_us(p.KB, NC, NC * kRowEpilogueUs);
        if (t >= best) continue;
        best = t;
        p.NC = NC; p.chunks = chunks;
        p.clusters = std::min(max_clusters, tiles);
    }
    if (!p.NC) return 0;
    p.stage_bytes = WM_W_BYTES + p.NC * 64;
    p.stages = std::min(WM_MAX_STAGES, (WM_SMEM_DYN - 1024 - WM_STAGING) / p.stage_bytes);
    p.smem_bytes = std::max(kAloneBytes, 1024 + p.stages * p.stage_bytes + WM_STAGING);
    // From four chunks on the next round reads the weights again (16 weight tiles of a group x 4 chunks are a round).  Layer-step, us,
    // kept | not: one chunk (129 rows) 165 | 151, two (300) 213 | 204, three (615) 283 | 281; four (800) 332 | 333, 3584 columns 342 | 345;
    // six and nine (1200) 477 | 480, (1800) 648 | 663.
    p.keep = p.chunks >= 4;
    CUtensorMap map_x, map_w[3];
    {
        std::lock_guard<std::mutex> lock(g_map_mutex);
        // a map that cannot be made leaves the projection to the caller's kernel, whose maps have two dimensions
        const CUtensorMap* m = get_rows_map(g.a, g.M, g.K, p.NC / 2);
        if (!m) return 0;
        map_x = *m;
        const char *gate = static_cast<const char*>(g.b[0]), *up = static_cast<const char*>(g.b[1]);
        p.up_first = EPI == kEpiSwiGLU && up < gate;
        const int64_t step = p.up_first ? gate - up : up - gate;
        if (EPI == kEpiSwiGLU && (step <= 0 || step >= ((int64_t)1 << 40))) return 0;
        for (int i = 0; i < 3; ++i) {
            if (EPI == kEpiSwiGLU && i == 0) m = get_weight_map(p.up_first ? up : gate, g.n[0], g.K, kWeightsPairs, step);   // both matrices
            else if (EPI != kEpiSwiGLU && g.b[i])
                m = get_weight_map(g.b[i], g.n[i], g.K, EPI != kEpiQKV ? kWeightsPlain : g.head_dim == 128 ? kWeightsRope128 : kWeightsRope64, 0);
            if (!m) return 0;
            map_w[i] = *m;
        }
    }
    cudaLaunchAttribute at[2];
    const cudaLaunchConfig_t cfg = wm_config<EPI>(at, p.clusters, p.smem_bytes, stream);
    return cudaLaunchKernelEx(&cfg, gemm_wm_kernel<EPI>, g, p, map_x, map_w[0], map_w[1], map_w[2]) == cudaSuccess ? 1 : -1;
}

}  // namespace

int launch_gemm_wm(const GemmArgs& g, double own_us, int group_n, cudaStream_t stream) {
    if (g.epilogue == kEpiSwiGLU) return launch_wm<kEpiSwiGLU>(g, own_us, group_n, stream);
    if (g.epilogue == kEpiQKV) return launch_wm<kEpiQKV>(g, own_us, group_n, stream);
    if (g.epilogue == kEpiResidual) return launch_wm<kEpiResidual>(g, own_us, group_n, stream);
    return 0;
}

}  // namespace acache
