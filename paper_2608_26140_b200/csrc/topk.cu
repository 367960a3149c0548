// Top-K anchor selection, Eq. 6: A = TopK({s_j}, K).  One CTA per request.  The K-th largest score is found by
// histograms over ever narrower key ranges and, once few candidates are left, by ranking them; one ordered pass over
// the positions emits the anchors ascending, ties going to the lower position.
#include "common.cuh"
#include "kernels.h"
#include "launch.h"

namespace acache {

constexpr int kTopkThreads = 1024;
constexpr int kTopkSmemKeys = 16384;   // keys cached in shared memory up to this L
constexpr int kTopkBins = 2 * kTopkThreads;
constexpr int kTopkRank = 256;         // candidates ranked directly

// Order-preserving map fp32 -> uint32 (larger float <=> larger key).
__device__ __forceinline__ uint32_t score_key(float f) {
    uint32_t u = __float_as_uint(f);
    if (u == 0x80000000u) u = 0u;   // -0 and +0 compare equal
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Bound by latency: block barriers, dependent trips to shared memory, and instructions, which 32 warps each run once
// (loops over a thread's keys are not unrolled: an unrolled form of this kernel took 20 us for 512 scores).  The bins of a
// histogram divide [smallest, largest] in 2048, which sorts out more than the leading bits of the keys do (the scores of a
// request share their exponents), so one pass mostly leaves few candidates.  Warp w owns the keys of [w seg, (w + 1) seg):
// loads are coalesced and the ordered output needs ballots and one sum over the warps.  Against a radix select over four
// bytes with two block scans per 1024 positions (launches back to back, one request): 512 scores 7.8 | 8.0 us, 2048 7.8 | 8.0,
// 8192 19.2 | 8.0, 16 requests of them 19.5 | 8.6.
__global__ void __launch_bounds__(kTopkThreads) topk_kernel(float* scores, int L, int K,
                                                            int32_t* __restrict__ anchor_idx, int use_smem,
                                                            const float* __restrict__ head_partial, int n_heads,
                                                            int accumulate) {
    extern __shared__ uint32_t keys_s[];
    __shared__ uint32_t hist[kTopkBins];
    __shared__ uint32_t cand_key[kTopkRank];
    __shared__ int cand_pos[kTopkRank];
    __shared__ uint32_t warp_cnt[32];
    __shared__ uint32_t s_min, s_max, s_bin, s_want, s_tau;
    __shared__ int s_cand, s_slots, s_tau_pos;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) { s_min = 0xffffffffu; s_max = 0u; s_slots = 0; }
    hist[tid] = 0u;
    hist[tid + kTopkThreads] = 0u;
    __syncthreads();
    pdl_wait();
    pdl_launch_dependents();
    const int b = blockIdx.x;
    float* s = scores + (int64_t)b * L;
    int32_t* out = anchor_idx + (int64_t)b * K;
    const int seg = (L + kTopkThreads - 1) / kTopkThreads * 32;
    const int j0 = min(warp * seg, L), j1 = min(j0 + seg, L);

    uint32_t mn = 0xffffffffu, mx = 0u;
#pragma unroll 4
    for (int j = j0 + lane; j < j1; j += 32) {
        float v;
        if (head_partial) {   // Eq. 5: ordered sum over heads, fused in front of the selection
            v = 0.f;
            const float* hp = head_partial + (int64_t)b * n_heads * L + j;
            int h = 0;
#pragma unroll 1
            for (; h + 32 <= n_heads; h += 32) {    // 32 loads in flight (one trip to L2), added in head order
                float t[32];
#pragma unroll
                for (int u = 0; u < 32; ++u) t[u] = __ldcg(hp + (int64_t)(h + u) * L);
#pragma unroll
                for (int u = 0; u < 32; ++u) v += t[u];
            }
#pragma unroll 4
            for (; h < n_heads; ++h) v += __ldcg(hp + (int64_t)h * L);
            if (accumulate) v += s[j];
            s[j] = v;
        } else {
            v = s[j];
        }
        const uint32_t kk = score_key(v);
        if (use_smem) keys_s[j] = kk;
        mn = min(mn, kk);
        mx = max(mx, kk);
    }
    if (K == 0) return;
    auto key_at = [&](int j) -> uint32_t { return use_smem ? keys_s[j] : score_key(s[j]); };
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0 && j0 < j1) { atomicMin(&s_min, mn); atomicMax(&s_max, mx); }
    __syncthreads();
    uint32_t lo = s_min, width_m1 = s_max - s_min;            // the K-th largest key lies in [lo, lo + width_m1]
    uint32_t want = (uint32_t)K;                              // its rank (from 1) among the keys of that range, largest first
    int n_cand = L;
    while (n_cand > kTopkRank && width_m1 > 0u) {
        const int shift = max(0, 21 - __clz(width_m1));       // at most 2048 bins
#pragma unroll 1
        for (int j = j0 + lane; j < j1; j += 32) {
            const uint32_t d = key_at(j) - lo;
            if (d <= width_m1) atomicAdd(&hist[d >> shift], 1u);
        }
        __syncthreads();
        // descending scan over the bins: thread t owns bins top and top - 1
        const int top = kTopkBins - 1 - 2 * tid;
        const uint32_t h0 = hist[top], h1 = hist[top - 1];
        uint32_t inc = h0 + h1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) warp_cnt[warp] = inc;
        __syncthreads();
        const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? warp_cnt[lane] : 0u) + inc - h0 - h1;
        if (before < want && want <= before + h0 + h1) {      // exactly one thread
            const bool first = want <= before + h0;
            s_bin = (uint32_t)(first ? top : top - 1);
            s_want = want - before - (first ? 0u : h0);
            s_cand = (int)(first ? h0 : h1);
        }
        hist[top] = 0u;
        hist[top - 1] = 0u;
        __syncthreads();
        lo += s_bin << shift;
        width_m1 = min(width_m1 - (s_bin << shift), (1u << shift) - 1u);
        want = s_want;
        n_cand = s_cand;
        __syncthreads();
    }
    if (n_cand <= kTopkRank) {
        // rank the candidates, a warp each: by key, then by position
#pragma unroll 1
        for (int j = j0 + lane; j < j1; j += 32) {
            const uint32_t kk = key_at(j);
            if (kk - lo <= width_m1) {
                const int at = atomicAdd(&s_slots, 1);
                cand_key[at] = kk;
                cand_pos[at] = j;
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int c = warp; c < n_cand; c += 32) {
            const uint32_t kk = cand_key[c];
            const int jj = cand_pos[c];
            uint32_t better = 0;
#pragma unroll 1
            for (int u = lane; u < n_cand; u += 32) better += cand_key[u] > kk || (cand_key[u] == kk && cand_pos[u] < jj);
            if (__reduce_add_sync(0xffffffffu, better) + 1u == want && lane == 0) { s_tau = kk; s_tau_pos = jj; }
        }
    } else {
        // many equal keys: the want-th of them by position
        uint32_t mine = 0;
#pragma unroll 1
        for (int j = j0 + lane; j < j1; j += 32) mine += key_at(j) == lo;
        mine = __reduce_add_sync(0xffffffffu, mine);
        if (lane == 0) warp_cnt[warp] = mine;
        __syncthreads();
        uint32_t seen = __reduce_add_sync(0xffffffffu, lane < warp ? warp_cnt[lane] : 0u);
#pragma unroll 1
        for (int i = j0; i < j1 && seen < want; i += 32) {
            const bool eq = i + lane < j1 && key_at(i + lane) == lo;
            const uint32_t eqs = __ballot_sync(0xffffffffu, eq);
            if (eq && seen + __popc(eqs & ((1u << lane) - 1u)) + 1u == want) { s_tau = lo; s_tau_pos = i + lane; }
            seen += __popc(eqs);
        }
    }
    __syncthreads();
    const uint32_t tau = s_tau;
    const int tau_pos = s_tau_pos;
    auto taken = [&](int j) {
        if (j >= j1) return false;
        const uint32_t kk = key_at(j);
        return kk > tau || (kk == tau && j <= tau_pos);
    };
    // ordered output: positions ascending
    uint32_t mine = 0;
#pragma unroll 1
    for (int i = j0; i < j1; i += 32) mine += taken(i + lane);
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) warp_cnt[warp] = mine;
    __syncthreads();
    int at = (int)__reduce_add_sync(0xffffffffu, lane < warp ? warp_cnt[lane] : 0u);
#pragma unroll 1
    for (int i = j0; i < j1; i += 32) {
        const bool sel = taken(i + lane);
        const uint32_t sels = __ballot_sync(0xffffffffu, sel);
        const int o = at + __popc(sels & ((1u << lane) - 1u));
        if (sel && o < K) out[o] = i + lane;
        at += __popc(sels);
    }
}

void launch_topk(float* scores, int batch, int affix_len, int k, int32_t* anchor_idx, const float* head_partial,
                 int n_heads, int accumulate, cudaStream_t stream) {
    if (batch == 0 || (k == 0 && !head_partial)) return;
    const int use_smem = affix_len <= kTopkSmemKeys;
    const size_t smem = use_smem ? (size_t)affix_len * sizeof(uint32_t) : 0;
    if (smem > 32 * 1024)
        cudaFuncSetAttribute(topk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kTopkSmemKeys * (int)sizeof(uint32_t));
    launch_pdl(topk_kernel, batch, kTopkThreads, smem, stream, scores, affix_len, k, anchor_idx, use_smem, head_partial,
               n_heads, accumulate);
}

}  // namespace acache
